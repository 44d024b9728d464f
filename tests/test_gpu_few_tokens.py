"""The few-token forward kernel at the edges of its blocks (8, 16, 32, 64 tokens; 16 and 32 weight rows; 32-wide steps of K dealt
out over eight warps) and on both sides of the rule that sends a product to it, compact and gated, against the oracle.
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
