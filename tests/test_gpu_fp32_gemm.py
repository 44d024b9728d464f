"""The fp32 FMA products at the edges of their 64 x 64 x 32 tiles, with K cut over clusters of 1, 2, 4 and 8 CTAs, with
rows that are 16-byte aligned and rows that are not (4-byte copies and stores), against the fp64 oracle.

Bound: an fp32 sum of K products in any order is off by at most K 2^-24 sum |a b|; rounding errors of random sign give
about sqrt(K) 2^-24 of the norm, and a chained product (H' then Y) twice that: 1e-5 (ELEMENT_BOUNDS["f32"]) covers K <= 1100."""
import numpy as np
import pytest
import torch

from oracle import flop_oracle as O
from tests._util import assert_close, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("T,d_in,d_out,r", [
    (1, 1, 1, 1), (3, 33, 5, 31), (64, 64, 64, 64), (65, 63, 129, 66), (130, 257, 100, 97),
    (520, 128, 256, 128), (1030, 96, 72, 40), (700, 768, 640, 640),
])
@pytest.mark.parametrize("odd_ld", [False, True])
@pytest.mark.parametrize("accumulate", [False, True])
def test_forward_and_backward_at_tile_edges(b, T, d_in, d_out, r, odd_ld, accumulate):
    g = np.random.default_rng(T + d_in + r)

    def mat(rows, cols, scale=1.0, fill=None):
        ld = cols + 1 if odd_ld and cols % 2 == 0 else cols if odd_ld else (cols + 7) // 8 * 8     # odd: no row but the first is aligned
        v = torch.full((rows, ld), float("nan") if fill is None else fill, device="cuda")[:, :cols]
        if fill is None and scale:
            v.copy_(torch.from_numpy((g.standard_normal((rows, cols)) * scale).astype(np.float32)))
        return v

    X, dY, Q, P = mat(T, d_in), mat(T, d_out), mat(r, d_in, d_in ** -0.5), mat(d_out, r, r ** -0.5)
    z = torch.from_numpy(np.where(g.random(r) < 0.4, 0.0, g.uniform(0.1, 1.0, r)).astype(np.float32)).cuda()
    dz = torch.from_numpy(g.uniform(0.0, 0.5, r).astype(np.float32)).cuda()
    init = 0.5 if accumulate else float("nan")
    H, Y, dX = mat(T, r, 0), mat(T, d_out, 0), mat(T, d_in, 0)
    dP, dQ, dla = mat(d_out, r, fill=init), mat(r, d_in, fill=init), torch.full((r,), init, device="cuda")
    ws = b.alloc_workspace(b.workspace_bytes(b.OP_BWD, T, d_in, d_out, r, b.F32))
    ws.fill_(0xFF)
    b.gated_lowrank_fwd(X, Q, P, z, Y, H, None)
    b.gated_lowrank_bwd(dY, X, Q, P, z, dz, H, dX, dP, dQ, dla, ws, accumulate)
    assert b.device_status() == b.OK
    zh = host(z)
    _, Hp, Yo = O.gated_lowrank_fwd(host(X), host(Q), host(P), zh)
    G = O.gated_lowrank_bwd(host(dY), host(X), host(Q), host(P), zh, host(dz))
    off = 0.5 if accumulate else 0.0
    for name, got, want in (("H", H, Hp), ("Y", Y, Yo), ("dX", dX, G["dX"]), ("dP", dP, G["dP"] + off), ("dQ", dQ, G["dQ"] + off)):
        assert_close(got, want, "f32", name)
    # dlog_alpha sums products of both signs: its error is measured against the sum of their magnitudes
    M = host(dY) @ host(P)
    size = np.sum(np.abs(host(Q)) * (np.abs(M).T @ np.abs(host(X))), axis=1) * host(dz) + off
    assert np.all(np.abs(host(dla) - (G["dlog_alpha"] + off)) <= 1e-5 * size + 1e-12)
    dla2 = torch.full((r,), init, device="cuda")                 # only dlog_alpha wanted: the product runs for its row dots
    b.gated_lowrank_bwd(dY, X, Q, P, z, dz, H, None, None, None, dla2, ws, accumulate)
    assert torch.equal(dla, dla2)
