"""Compaction whose results take the place of its inputs: the gates become z_det, P its own surviving columns.  Selection and gather
by a single launch would read what another block has already overwritten; such calls run as separate launches.  Exact."""
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


@pytest.mark.parametrize("r,d_in,d_out", [(1, 8, 8), (768, 768, 3072), (1000, 24, 700), (1024, 1024, 4096)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_outputs_over_inputs(b, r, d_in, d_out, dtype):
    g = np.random.default_rng(r)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    for rep in range(20):
        a = g.normal(0.3, 2.0, r).astype(np.float32)
        gates = torch.from_numpy(a).cuda()
        P, Q = to_dev(g.standard_normal((d_out, r)), dtype), to_dev(g.standard_normal((r, d_in)), dtype)
        Ph, Qh, Qc = host(P), host(Q), empty_dev(r, d_in, tdt)
        idx, kd = torch.full((r,), -1, dtype=torch.int32, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda")
        b.compact_ranks(gates, 0, HC, idx, kd, gates, P, Q, P, Qc)
        k, idxo, zo = O.deterministic_mask(a, *HC)
        assert int(kd.item()) == k and np.array_equal(idx.cpu().numpy()[:k], idxo)
        assert np.max(np.abs(host(gates) - zo)) < 1e-7
        Pco, Qco = O.compact_ranks(Ph, Qh, idxo, host(gates))
        got = host(P)
        assert np.array_equal(got[:, :k], Pco) and np.array_equal(got[:, k:], Ph[:, k:])       # columns from k on stay untouched
        assert np.all(np.abs(host(Qc)[:k] - Qco) <= (2.0 ** -8 if dtype == "bf16" else 2.0 ** -24) * np.abs(Qco))
    assert b.device_status() == b.OK
