"""Backward calls whose outputs take the place of inputs that a launch per product has finished reading: dX on X, dP on P.  The two
shared launches would overwrite them while other tiles still read; such calls run one product after another.  Against the
oracle, bf16 bounds of tests/_util.py."""
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


@pytest.mark.parametrize("T,d,r", [(130, 264, 136), (1000, 768, 768), (2100, 520, 400)])
@pytest.mark.parametrize("n", [0, 1, 2])                 # 0: the single call; else a grouped call of n problems
def test_dx_on_x_and_dp_on_p(b, T, d, r, n):
    g = np.random.default_rng(T)
    for rep in range(5):
        probs = []
        for _ in range(max(n, 1)):
            X, dY = to_dev(g.standard_normal((T, d)), "bf16"), to_dev(g.standard_normal((T, d)), "bf16")
            Q, P = to_dev(g.standard_normal((r, d)) * d ** -0.5, "bf16"), to_dev(g.standard_normal((d, r)) * r ** -0.5, "bf16")
            z = torch.from_numpy(np.where(g.random(r) < 0.4, 0.0, g.uniform(0.1, 1.0, r)).astype(np.float32)).cuda()
            dz, H, Y = torch.ones(r, device="cuda"), empty_dev(T, r, torch.bfloat16), empty_dev(T, d, torch.bfloat16)
            b.gated_lowrank_fwd(X, Q, P, z, Y, H, None)
            G = O.gated_lowrank_bwd(host(dY), host(X), host(Q), host(P), host(z), host(dz))
            dQ, dla = empty_dev(r, d, torch.bfloat16), torch.zeros(r, device="cuda")
            ws = b.alloc_workspace(b.workspace_bytes(b.OP_BWD, T, d, d, r, b.BF16))
            probs.append((G, dQ, X, P, (dY, X, Q, P, z, dz, H, X, P, dQ, dla, ws)))
        if n:
            b.gated_lowrank_bwd_grouped([b.bwd_problem(*p[4]) for p in probs], wgrad_dt=b.BF16)
        else:
            b.gated_lowrank_bwd(*probs[0][4])
        for G, dQ, X, P, _ in probs:
            assert_close(X, G["dX"], "bf16", "dX")
            assert_close(P, G["dP"], "bf16", "dP")
            assert_close(dQ, G["dQ"], "bf16", "dQ")
    assert b.device_status() == b.OK


@pytest.mark.parametrize("kind,T,d,r", [("f32", 200, 96, 64), ("bf16", 200, 96, 64), ("bf16", 1000, 768, 768)])
def test_dx_on_the_gates_derivatives(b, kind, T, d, r):
    """dX takes the place of d z / d log_alpha, which a launch per product has read by then."""
    dt, f32 = (torch.float32, True) if kind == "f32" else (torch.bfloat16, False)
    g = np.random.default_rng(T + d)
    X, dY = to_dev(g.standard_normal((T, d)), kind), to_dev(g.standard_normal((T, d)), kind)
    Q, P = to_dev(g.standard_normal((r, d)) * d ** -0.5, kind), to_dev(g.standard_normal((d, r)) * r ** -0.5, kind)
    z = torch.from_numpy(g.uniform(0.1, 1.0, r).astype(np.float32)).cuda()
    H, Y = empty_dev(T, r, dt), empty_dev(T, d, dt)
    b.gated_lowrank_fwd(X, Q, P, z, Y, H, None)
    dX = empty_dev(T, d, dt)
    dz = dX.flatten().view(torch.float32)[:r]
    assert dz.data_ptr() == dX.data_ptr()
    dz.copy_(torch.from_numpy(g.uniform(0.5, 1.5, r).astype(np.float32)))
    dz_host = host(dz)
    G = O.gated_lowrank_bwd(host(dY), host(X), host(Q), host(P), host(z), dz_host)
    dP, dQ, dla = empty_dev(d, r, dt), empty_dev(r, d, dt), torch.zeros(r, device="cuda")
    b.gated_lowrank_bwd(dY, X, Q, P, z, dz, H, dX, dP, dQ, dla, b.alloc_workspace(b.workspace_bytes(b.OP_BWD, T, d, d, r, b.F32 if f32 else b.BF16)))
    for got, name in ((dX, "dX"), (dP, "dP"), (dQ, "dQ")):
        assert_close(got, G[name], kind, name)
    # dlog_alpha sums products of both signs: its error is measured against the sum of their magnitudes
    size = np.sum(np.abs(host(Q)) * (np.abs(host(dY) @ host(P)).T @ np.abs(host(X))), axis=1) * dz_host
    assert np.all(np.abs(host(dla) - G["dlog_alpha"]) <= (1e-5 if f32 else 2.0 ** -6) * size + 1e-6)
    assert b.device_status() == b.OK
