"""Backward calls of few tokens or few tiles on both sides of the rule that runs them as two shared launches: ragged sizes,
fp32 and bf16 weight gradients, accumulated or not, optional outputs absent, single and grouped, against the oracle
(bf16 bounds of tests/_util.py)."""
import numpy as np
import pytest
import torch

from oracle import flop_oracle as O
from tests._util import assert_close, empty_dev, host, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("T,d_in,d_out,r", [(1, 40, 24, 16), (130, 257, 300, 129), (1000, 256, 520, 256), (515, 72, 1030, 72), (4100, 136, 264, 130)])
@pytest.mark.parametrize("wdt,accumulate", [("bf16", False), ("bf16", True), ("f32", False), ("f32", True)])
@pytest.mark.parametrize("skip", ["", "dX", "dP", "dQ"])
def test_backward_forms(b, T, d_in, d_out, r, wdt, accumulate, skip):
    g = np.random.default_rng(T + r)
    X, dY = to_dev(g.standard_normal((T, d_in)), "bf16"), to_dev(g.standard_normal((T, d_out)), "bf16")
    Q, P = to_dev(g.standard_normal((r, d_in)) * d_in ** -0.5, "bf16"), to_dev(g.standard_normal((d_out, r)) * r ** -0.5, "bf16")
    z = torch.from_numpy(np.where(g.random(r) < 0.4, 0.0, g.uniform(0.1, 1.0, r)).astype(np.float32)).cuda()
    dz = torch.from_numpy(g.uniform(0.05, 0.5, r).astype(np.float32)).cuda()
    H, Y = empty_dev(T, r, torch.bfloat16), empty_dev(T, d_out, torch.bfloat16)
    b.gated_lowrank_fwd(X, Q, P, z, Y, H, None)
    zh = host(z)
    G = O.gated_lowrank_bwd(host(dY), host(X), host(Q), host(P), zh, host(dz))
    # dlog_alpha: the row sums cancel, so the bf16 rounding of dH' (2^-8) is measured against the magnitudes summed
    size = np.sqrt(np.sum((np.abs(host(Q)) @ np.abs(host(X)).T) ** 2 * (host(dY) @ host(P)).T ** 2, axis=1)) * host(dz)
    off, tdt = (0.5 if accumulate else 0.0), torch.float32 if wdt == "f32" else torch.bfloat16
    for grouped in (False, True):
        init = 0.5 if accumulate else float("nan")
        o = dict(dX=empty_dev(T, d_in, torch.bfloat16), dP=empty_dev(d_out, r, tdt, init), dQ=empty_dev(r, d_in, tdt, init),
                 dla=torch.full((r,), init, device="cuda"))
        give = {k: None if k == skip else v for k, v in o.items()}
        ws = b.alloc_workspace(b.workspace_bytes(b.OP_BWD, T, d_in, d_out, r, b.BF16)).fill_(0xFF)
        if grouped:
            pr = [b.bwd_problem(dY, X, Q, P, z, dz, H, give["dX"], give["dP"], give["dQ"], give["dla"], ws)]
            b.gated_lowrank_bwd_grouped(pr, accumulate=accumulate, wgrad_dt=b.F32 if wdt == "f32" else b.BF16)
        else:
            b.gated_lowrank_bwd(dY, X, Q, P, z, dz, H, give["dX"], give["dP"], give["dQ"], give["dla"], ws, accumulate)
        for k, want in (("dX", G["dX"]), ("dP", G["dP"] + off), ("dQ", G["dQ"] + off)):
            if k == skip:
                assert torch.isnan(o[k]).all() or torch.all(o[k] == init)          # not written
            else:
                assert_close(o[k], want, "bf16", f"{k} grouped={grouped}")
        assert np.all(np.abs(host(o["dla"]) - (G["dlog_alpha"] + off)) <= 2.0 ** -6 * size + 1e-6)
        assert b.device_status() == b.OK
