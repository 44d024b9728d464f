"""Backward calls in workspaces smaller than the query's: the query sizes rows of dH' on 128-byte lines, a vector of dz partials per
32 tokens and slices for dO; a call that is given less lays dH' out in 16-byte pieces, takes a vector per 64 tokens and
leaves dO unsplit.  Smaller still is refused.  bf16 bounds of tests/_util.py."""
import numpy as np
import pytest
import torch

from oracle import flop_oracle as O
from tests._util import assert_close, empty_dev, host, rel_fro, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("form", ["single", "grouped", "deferred"])
@pytest.mark.parametrize("T,d_in,d_out,r", [(512, 256, 304, 130), (4096, 768, 768, 72)])
def test_layer_backward(b, form, T, d_in, d_out, r):
    g = np.random.default_rng(T)
    X, dY = to_dev(g.standard_normal((T, d_in)), "bf16"), to_dev(g.standard_normal((T, d_out)), "bf16")
    Q, P = to_dev(g.standard_normal((r, d_in)) * d_in ** -0.5, "bf16"), to_dev(g.standard_normal((d_out, r)) * r ** -0.5, "bf16")
    z, dz = torch.from_numpy(g.uniform(0.1, 1.0, r).astype(np.float32)).cuda(), torch.ones(r, device="cuda")
    H, Y = empty_dev(T, r, torch.bfloat16), empty_dev(T, d_out, torch.bfloat16)
    b.gated_lowrank_fwd(X, Q, P, z, Y, H, None)
    G = O.gated_lowrank_bwd(host(dY), host(X), host(Q), host(P), host(z), host(dz))
    size = np.sqrt(np.sum((np.abs(host(Q)) @ np.abs(host(X)).T) ** 2 * (host(dY) @ host(P)).T ** 2, axis=1))
    full = b.workspace_bytes(b.OP_BWD, T, d_in, d_out, r, b.BF16)
    pieces = full - 2 * T * ((r + 63) // 64 * 64 - (r + 7) // 8 * 8)

    def run(nbytes):
        ws = b.alloc_workspace(nbytes + 256).fill_(0xFF)[:nbytes]
        o = (empty_dev(T, d_in, torch.bfloat16), empty_dev(d_out, r, torch.float32), empty_dev(r, d_in, torch.float32), torch.full((r,), float("nan"), device="cuda"))
        if form == "single":
            b.gated_lowrank_bwd(dY, X, Q, P, z, dz, H, *o, ws)
        else:
            pr = [b.bwd_problem(dY, X, Q, P, z, dz, H, *o, ws, defer_dlog_alpha=form == "deferred")]
            b.gated_lowrank_bwd_grouped(pr, wgrad_dt=b.F32)
            if form == "deferred":
                b.dlog_alpha_finish_grouped(pr)
        for name, got in zip(("dX", "dP", "dQ"), o):
            assert_close(got, G[name], "bf16", name)
        assert np.all(np.abs(host(o[3]) - G["dlog_alpha"]) <= 2.0 ** -6 * size + 1e-6)
        assert b.device_status() == b.OK

    run(full)
    run(pieces)
    with pytest.raises(b.FlopError) as e:
        run(2 * T * r)                                    # not even dH'
    assert e.value.code == b.ERR_WORKSPACE


@pytest.mark.parametrize("T,d_i,d", [(1, 64, 40), (65, 300, 96), (2500, 256, 128), (4096, 7, 64)])
def test_embedding_backward(b, T, d_i, d):
    g = np.random.default_rng(T)
    n_rows = 50
    E, Om, dY = to_dev(g.standard_normal((n_rows, d_i)), "bf16"), to_dev(g.standard_normal((d_i, d)) / np.sqrt(d_i), "bf16"), to_dev(g.standard_normal((T, d)), "bf16")
    ids = torch.from_numpy((g.random(T) ** 3 * n_rows).astype(np.int32)).cuda()
    z, dz = torch.from_numpy(g.uniform(0.2, 1.0, d_i).astype(np.float32)).cuda(), torch.from_numpy(g.uniform(0.1, 0.5, d_i).astype(np.float32)).cuda()
    Y, H = empty_dev(T, d, torch.bfloat16), empty_dev(T, d_i, torch.bfloat16)
    b.gated_embedding_fwd(ids, E, Om, z, Y, H)
    up = lambda v: (v + 255) // 256 * 256
    dh = up(2 * T * ((d_i + 7) // 8 * 8))
    per32, per64 = dh + up(4 * d_i * ((T + 31) // 32)), dh + up(4 * d_i * ((T + 63) // 64))
    idn = ids.cpu().numpy()
    dH = host(dY) @ host(Om).T
    want, sums, size = np.zeros((n_rows, d_i)), np.sum(host(E)[idn] * dH, axis=0) * host(dz), np.sum(np.abs(host(E)[idn] * dH), axis=0) * host(dz)
    np.add.at(want, idn, dH * host(z))

    def run(nbytes):
        ws = b.alloc_workspace(nbytes + 256).fill_(0xFF)[:nbytes]
        dE, dO, dla = torch.zeros(n_rows, (d_i + 7) // 8 * 8, device="cuda")[:, :d_i], empty_dev(d_i, d, torch.float32), torch.full((d_i,), float("nan"), device="cuda")
        b.gated_embedding_bwd(dY, ids, E, Om, z, dz, H, dE, dO, dla, ws)
        assert rel_fro(host(dO), host(H).T @ host(dY)) < 1e-5
        assert rel_fro(host(dE), want) < 4e-3                                # dH' is rounded to bf16 before it is summed
        assert np.all(np.abs(host(dla) - sums) <= 2.0 ** -7 * size + 1e-6)
        assert b.device_status() == b.OK

    for nbytes in (b.workspace_bytes(b.OP_EMBEDDING_BWD, T, 0, 0, d_i, b.BF16), per32, per64):
        run(nbytes)
    with pytest.raises(b.FlopError) as e:
        run(dh)
    assert e.value.code == b.ERR_WORKSPACE
