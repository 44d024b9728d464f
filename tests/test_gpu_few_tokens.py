"""The few-token forward kernel at the edges of its blocks (8, 16, 32, 64 tokens; 16 and 32 weight rows; 32-wide steps of K dealt
out over its warps) and on both sides of the rules that send a product to it and cut its K, compact and gated, against the oracle.
Columns beyond K of every operand hold NaN: they must not be read as numbers.

Bound: H' is rounded to bf16 (2^-8) before the second product and Y once more; sums are fp32: the element-wise bf16 bound of
tests/_util.py."""
import numpy as np
import pytest
import torch

from oracle import flop_oracle as O
from tests._util import assert_close, empty_dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


def _mat(g, rows, cols, scale):
    v = empty_dev(rows, cols, torch.bfloat16)                       # the padding of every row stays NaN
    v.copy_(torch.from_numpy((g.standard_normal((rows, cols)) * scale).astype(np.float32)))
    return v


@pytest.mark.parametrize("T", [1, 7, 8, 9, 16, 17, 32, 33, 64, 65, 200])
@pytest.mark.parametrize("d_in,r,d_out", [(1, 1, 1), (30, 17, 33), (264, 250, 15), (1025, 99, 410), (520, 31, 2401)])
def test_pairs_of_products(b, T, d_in, r, d_out):
    g = np.random.default_rng(T + d_in)
    X, Q, P = _mat(g, T, d_in, 1.0), _mat(g, r, d_in, d_in ** -0.5), _mat(g, d_out, r, r ** -0.5)
    z = torch.from_numpy(np.where(g.random(r) < 0.3, 0.0, g.uniform(0.1, 1.0, r)).astype(np.float32)).cuda()
    H, Y, Yc = empty_dev(T, r, torch.bfloat16), empty_dev(T, d_out, torch.bfloat16), empty_dev(T, d_out, torch.bfloat16)
    for _ in range(2):                                                # twice: the second call starts while the first one drains
        b.gated_lowrank_fwd(X, Q, P, z, Y, H, None)
        b.compact_fwd(X, Q, P, Yc, r, b.alloc_workspace(b.workspace_bytes(b.OP_COMPACT_FWD, T, d_in, d_out, r, b.BF16)).fill_(0xFF))
    _, Hp, _ = O.gated_lowrank_fwd(host(X), host(Q), host(P), host(z))
    assert_close(H, Hp, "bf16", "H")
    assert_close(Y, host(H) @ host(P).T, "bf16", "Y")                # from the H' that was stored
    Hc = host((X.double() @ Q.double().T).float().to(torch.bfloat16))
    assert_close(Yc, Hc @ host(P).T, "bf16", "Yc")
    assert b.device_status() == b.OK


@pytest.mark.parametrize("T", [1, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("d_in,r,d_out", [(24, 33, 4737), (40, 33, 7105), (72, 150, 14210), (16, 31, 28420), (16, 640, 16384), (8, 1030, 40000)])
def test_wide_outputs(b, T, d_in, r, d_out):
    """Outputs so wide that K is cut over fewer warps, or that tcgen05 tiles take the product: one row above each line."""
    g = np.random.default_rng(T + d_out)
    X, Q, P = _mat(g, T, d_in, 1.0), _mat(g, r, d_in, d_in ** -0.5), _mat(g, d_out, r, r ** -0.5)
    Y = empty_dev(T, d_out, torch.bfloat16)
    b.compact_fwd(X, Q, P, Y, r, b.alloc_workspace(b.workspace_bytes(b.OP_COMPACT_FWD, T, d_in, d_out, r, b.BF16)).fill_(0xFF))
    H = host((X.double() @ Q.double().T).float().to(torch.bfloat16))
    assert_close(Y, H @ host(P).T, "bf16", "Y")
    assert b.device_status() == b.OK


@pytest.mark.parametrize("T", [1, 16, 32])
def test_weights_written_by_the_launch_before(b, T):
    """The second product asks for its weights before it waits; here they come from compact_ranks right before the pair, other ones
    every time."""
    g = np.random.default_rng(T)
    d_in, r, d_out = 1024, 1024, 4096
    P, Q, X = _mat(g, d_out, r, r ** -0.5), _mat(g, r, d_in, d_in ** -0.5), _mat(g, T, d_in, 1.0)
    Pc, Qc, Y = empty_dev(d_out, r, torch.bfloat16), empty_dev(r, d_in, torch.bfloat16), [empty_dev(T, d_out, torch.bfloat16) for _ in range(8)]
    idx, kd = torch.zeros(r, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws, k = b.alloc_workspace(b.workspace_bytes(b.OP_COMPACT_FWD, T, d_in, d_out, r, b.BF16)), 300
    gates = []
    for i in range(8):
        z = np.zeros(r, np.float32)
        z[np.sort(g.permutation(r)[:k])] = g.uniform(0.1, 1.0, k)
        gates.append(torch.from_numpy(z).cuda())
    for z, y in zip(gates, Y):
        b.compact_ranks(z, 1, (1.0, -0.1, 1.1), idx, kd, None, P, Q, Pc, Qc)
        b.compact_fwd(X, Qc[:k], Pc[:, :k], y, k, ws)
    for z, y in zip(gates, Y):
        keep = (z > 0).nonzero().flatten()
        H = (X.double() @ (Q[keep].float() * z[keep, None]).to(torch.bfloat16).double().T).float().to(torch.bfloat16)
        assert_close(y, host(H) @ host(P[:, keep]).T, "bf16", "Y")
    assert b.device_status() == b.OK
