"""Calls from several threads: a thread whose first CUDA work is a call of the library."""
import threading

import pytest
import torch

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
