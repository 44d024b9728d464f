"""Gated embedding backward at the sizes where its kernels change form: 8, 16 and 32 lanes per token (widths around 64 and
128, ragged and odd ones), token counts around a block of 32, dO with and without split slices (few / many tokens), fp32
and bf16 dO, accumulate.  dE sums in no fixed order; every tolerance is the element-wise bf16 bound of tests/_util.py
(H', dH' are rounded to bf16; fp32 sums)."""
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


@pytest.mark.parametrize("d_i", [7, 64, 65, 128, 129, 300])
@pytest.mark.parametrize("T,d", [(1, 40), (31, 130), (33, 64), (2500, 96)])
@pytest.mark.parametrize("wdt,accumulate", [("bf16", False), ("f32", True)])
def test_widths_and_token_counts(b, d_i, T, d, wdt, accumulate):
    g = np.random.default_rng(d_i + T)
    n_rows, bf = 50, torch.bfloat16
    E, Om, dY = to_dev(g.standard_normal((n_rows, d_i)), "bf16"), to_dev(g.standard_normal((d_i, d)) / np.sqrt(d_i), "bf16"), to_dev(g.standard_normal((T, d)), "bf16")
    ids = torch.from_numpy((g.random(T) ** 3 * n_rows).astype(np.int32)).cuda()
    z = torch.from_numpy(np.where(g.random(d_i) < 0.3, 0.0, g.uniform(0.2, 1.0, d_i)).astype(np.float32)).cuda()
    dz = torch.from_numpy(g.uniform(0.1, 0.5, d_i).astype(np.float32)).cuda()
    Y, H = empty_dev(T, d, bf), empty_dev(T, d_i, bf)
    b.gated_embedding_fwd(ids, E, Om, z, Y, H)
    init = 0.5 if accumulate else float("nan")
    tdt = torch.float32 if wdt == "f32" else bf
    dE, dO, dla = torch.zeros(n_rows, (d_i + 7) // 8 * 8, device="cuda")[:, :d_i], empty_dev(d_i, d, tdt, init), torch.full((d_i,), init, device="cuda")
    ws = b.alloc_workspace(b.workspace_bytes(b.OP_EMBEDDING_BWD, T, 0, 0, d_i, b.BF16))
    ws.fill_(0xFF)
    b.gated_embedding_bwd(dY, ids, E, Om, z, dz, H, dE, dO, dla, ws, accumulate)
    assert b.device_status() == b.OK
    idn, zh, Eh, Oh, dYh, Hh = ids.cpu().numpy(), host(z), host(E), host(Om), host(dY), host(H)
    rows = Eh[idn] * zh
    assert np.all(np.abs(Hh - rows) <= 2.0 ** -8 * np.abs(rows))                   # one rounding to 8 bits
    assert_close(Y, Hh @ Oh, "bf16", "Y")
    dH = dYh @ Oh.T
    off = 0.5 if accumulate else 0.0
    assert rel_fro(host(dO), Hh.T @ dYh + off) < (4e-3 if wdt == "bf16" else 1e-5)
    want = np.zeros((n_rows, d_i))
    np.add.at(want, idn, dH * zh)
    assert rel_fro(host(dE), want) < 4e-3                                            # dH' is rounded to bf16 before it is summed
    size = np.sum(np.abs(Eh[idn] * dH), axis=0) * host(dz)
    assert np.all(np.abs(host(dla) - (np.sum(Eh[idn] * dH, axis=0) * host(dz) + off)) <= 2.0 ** -7 * size + 1e-6)


@pytest.mark.parametrize("d_i,line", [(40, 4736), (100, 2368), (300, 1184), (2048, 1184)])
@pytest.mark.parametrize("over", [0, 1])
def test_lookup_on_both_sides_of_one_round(b, d_i, line, over):
    """One token per lane group while that is one round of blocks over 148 SMs, four in flight beyond: one rounding to 8 bits."""
    T, n_rows, d = line + over, 70, 24
    g = np.random.default_rng(T)
    E, Om = to_dev(g.standard_normal((n_rows, d_i)), "bf16"), to_dev(g.standard_normal((d_i, d)) / np.sqrt(d_i), "bf16")
    ids = torch.from_numpy(g.integers(-3, n_rows + 3, T).astype(np.int32)).cuda()
    z = torch.from_numpy(g.uniform(0.2, 1.0, d_i).astype(np.float32)).cuda()
    Y, H = empty_dev(T, d, torch.bfloat16), empty_dev(T, d_i, torch.bfloat16)
    b.gated_embedding_fwd(ids, E, Om, z, Y, H)
    rows = host(E)[np.clip(ids.cpu().numpy(), 0, n_rows - 1)] * host(z)
    assert np.all(np.abs(host(H) - rows) <= 2.0 ** -8 * np.abs(rows))
    assert_close(Y, host(H) @ host(Om), "bf16", "Y")
    assert b.device_status() == b.OK
