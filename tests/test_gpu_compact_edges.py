"""Selection and gathers in one launch (ranks up to 1024) and in three: ranks at word, block and route edges, odd numbers of survivors, outputs whose rows allow no paired stores, ties at the cut.  A gather moves values: exact."""
import numpy as np
import pytest
import torch

from oracle import flop_oracle as O
from tests._util import HC, empty_dev, host, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("r", [1, 31, 256, 257, 1023, 1024, 1025, 4097])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("odd_ld", [False, True])
@pytest.mark.parametrize("ties", [False, True])
def test_mask_and_compact_factors(b, r, dtype, odd_ld, ties):
    g = np.random.default_rng(r)
    a = g.normal(0.0, 2.5, r).astype(np.float32)
    if ties:
        a = g.choice(np.array([-1.5, -0.0, 0.0, 0.75], np.float32), size=r)
    d_in, d_out, tdt = 27, 13, torch.bfloat16 if dtype == "bf16" else torch.float32
    P, Q = to_dev(g.standard_normal((d_out, r)), dtype), to_dev(g.standard_normal((r, d_in)), dtype)
    out = (lambda rows, cols: torch.full((rows, cols | 1), float("nan"), dtype=tdt, device="cuda")[:, :cols]) if odd_ld else \
        (lambda rows, cols: empty_dev(rows, cols, tdt))
    Pc, Qc, zd = out(d_out, r), out(r, d_in), torch.full((r,), float("nan"), device="cuda")
    idx, kd = torch.full((r,), -1, dtype=torch.int32, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda")
    b.compact_ranks(torch.from_numpy(a).cuda(), 0, HC, idx, kd, zd, P, Q, Pc, Qc)
    k, idxo, zo = O.deterministic_mask(a, *HC)
    assert int(kd.item()) == k and np.array_equal(idx.cpu().numpy()[:k], idxo) and np.all(idx.cpu().numpy()[k:] == -1)
    assert np.max(np.abs(host(zd) - zo)) < 1e-7
    Pco, Qco = O.compact_ranks(host(P), host(Q), idxo, host(zd))
    assert np.array_equal(host(Pc)[:, :k], Pco) and np.all(np.isnan(host(Pc)[:, k:])) and np.all(np.isnan(host(Qc)[k:]))
    if k:      # one rounding of each product to 8 (bf16) or 24 (fp32) significant bits: at most 2^-8 or 2^-24 relative
        assert np.all(np.abs(host(Qc)[:k] - Qco) <= (2.0 ** -8 if dtype == "bf16" else 2.0 ** -24) * np.abs(Qco))
    assert b.device_status() == b.OK


@pytest.mark.parametrize("d_in", [4095, 4096, 4097, 8193, 30001])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("odd_ld", [False, True])
def test_rows_of_q_in_pieces(b, d_in, dtype, odd_ld):
    """Rows longer than 4096 elements are gathered in pieces; with and without 16-byte vectors."""
    g = np.random.default_rng(d_in)
    r, d_out, tdt = 100, 5, torch.bfloat16 if dtype == "bf16" else torch.float32
    z = np.where(g.random(r) < 0.4, g.uniform(0.05, 1.0, r), 0.0).astype(np.float32)
    P, Q = to_dev(g.standard_normal((d_out, r)), dtype), to_dev(g.standard_normal((r, d_in)), dtype)
    Pc, Qc = empty_dev(d_out, r, tdt), torch.full((r, d_in + (9 if odd_ld else 24)), float("nan"), dtype=tdt, device="cuda")[:, :d_in]
    if not odd_ld:
        Qc = empty_dev(r, d_in, tdt)
    idx, kd = torch.full((r,), -1, dtype=torch.int32, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda")
    b.compact_ranks(torch.from_numpy(z).cuda(), 1, HC, idx, kd, None, P, Q, Pc, Qc)
    k, idxo = O.active_ranks(z)
    assert int(kd.item()) == k and np.array_equal(idx.cpu().numpy()[:k], idxo)
    Pco, Qco = O.compact_ranks(host(P), host(Q), idxo, z.astype(np.float64))
    got = host(Qc)
    assert np.array_equal(host(Pc)[:, :k], Pco) and np.all(np.isnan(got[k:]))
    assert np.all(np.abs(got[:k] - Qco) <= (2.0 ** -8 if dtype == "bf16" else 2.0 ** -24) * np.abs(Qco))      # one rounding of each product
    assert b.device_status() == b.OK
