"""Calls from several threads: a thread whose first CUDA work is a call of the library, and two threads, each on its own stream, whose
calls need different amounts of shared memory of the same kernel (neither changes what the other may use)."""
import threading

import pytest
import torch

from tests._util import HC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


def test_first_call_of_a_thread(b):
    """Nothing has bound a CUDA context to the thread: tensor maps are encoded all the same."""
    g = torch.Generator(device="cuda").manual_seed(3)
    T, d_in, d_out, r = 300, 64, 72, 40
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()  # noqa: E731
    X, Q, P, z = rand(T, d_in), rand(r, d_in), rand(d_out, r), torch.rand(r, generator=g, device="cuda")
    Y, H, want, want_H = (torch.zeros(T, n, dtype=torch.bfloat16, device="cuda") for n in (d_out, r, d_out, r))
    b.gated_lowrank_fwd(X, Q, P, z, want, want_H)
    torch.cuda.synchronize()
    errors = []

    def body():
        try:
            b.gated_lowrank_fwd(X, Q, P, z, Y, H)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    thread = threading.Thread(target=body)
    thread.start()
    thread.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    assert torch.equal(Y, want) and torch.equal(H, want_H)
    assert b.device_status() == b.OK


def _together(works):
    errors, start = [], threading.Barrier(len(works))

    def body(work):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(1500):
                    work()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=body, args=(w,)) for w in works]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


def test_long_and_short_rows_of_p(b):
    works, checks = [], []
    for r in (14000, 50000):                    # 56 and 200 KB of a row of P in shared memory
        gates = torch.linspace(-3.0, 3.0, r, device="cuda")
        P, Q = torch.randn(3, r, device="cuda"), torch.randn(r, 4, device="cuda")
        idx, kd, zd = torch.zeros(r, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(r, device="cuda")
        Pc, Qc = torch.zeros(3, r, device="cuda"), torch.zeros(r, 4, device="cuda")
        works.append(lambda a=(gates, 0, HC, idx, kd, zd, P, Q, Pc, Qc): b.compact_ranks(*a))
        checks.append((P, idx, kd, Pc))
    torch.cuda.synchronize()
    _together(works)
    for P, idx, kd, Pc in checks:
        k = int(kd.item())
        assert 0 < k < P.shape[1] and torch.equal(Pc[:, :k], P[:, idx[:k].long()])
    assert b.device_status() == b.OK


def test_wide_and_narrow_embeddings(b):
    works, checks = [], []
    T, n, d = 64, 50, 8
    for d_i in (1600, 6400):                    # 50 and 200 KB of partial sums
        g = torch.Generator(device="cuda").manual_seed(d_i)
        rand = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()  # noqa: E731
        ids = torch.arange(T, dtype=torch.int32, device="cuda") % n
        E, O, dY, H = rand(n, d_i), rand(d_i, d), rand(T, d), rand(T, d_i)
        z, dz = torch.rand(d_i, device="cuda"), torch.rand(d_i, device="cuda")
        dE, dO, dla = torch.zeros(n, d_i, device="cuda"), torch.zeros(d_i, d, dtype=torch.bfloat16, device="cuda"), torch.zeros(d_i, device="cuda")
        ws = b.alloc_workspace(b.workspace_bytes(b.OP_EMBEDDING_BWD, T, 0, 0, d_i, b.BF16))
        works.append(lambda a=(dY, ids, E, O, z, dz, H, dE, dO, dla, ws): b.gated_embedding_bwd(*a))
        checks.append((dY, H, dO))
    torch.cuda.synchronize()
    _together(works)
    for dY, H, dO in checks:
        want = H.double().T @ dY.double()
        # T products in fp32, then one rounding to bf16
        bound = want.abs() * 2.0 ** -8 + (H.double().abs().T @ dY.double().abs()) * (T * 2.0 ** -23)
        assert torch.all((dO.double() - want).abs() <= bound)
    assert b.device_status() == b.OK
