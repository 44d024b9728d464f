"""Survivors chosen inside the one-launch compaction, whatever the gates ask of its bins (one pass over them or several, gates ranked or
equal, k from fp32 or fp64 probabilities), against the oracle and against the separate launches (which a call takes when z_det overwrites the gates).  Indices and values are exact."""
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


def _gates(kind, r):
    g = np.random.default_rng([r, len(kind)])
    a = g.normal(0.0, 2.0, r)
    if kind == "bimodal":
        a = np.where(g.random(r) < 0.3, 4.0, -4.0) + 0.1 * g.standard_normal(r)
    elif kind == "far":             # one distant gate: all others share a bin, more of them than are ranked against one another
        a = 1e-3 * g.standard_normal(r)
        a[r // 2] = 1e30
    elif kind == "ties":            # the cut falls inside a class of equal gates, small and large ones
        a = np.round(a * 20) / 20
    elif kind == "equal":
        a = np.full(r, 0.3)
    elif kind == "half":            # the expected count is a half within 1e-6: only fp64 decides
        thr = HC[0] * np.log(-HC[1] / HC[2])
        p = lambda x: 1.0 / (1.0 + np.exp(-(x - thr)))  # noqa: E731
        a = a.astype(np.float32).astype(np.float64)
        rest = p(a[1:]).sum()
        want = np.floor(rest) + 0.5 - rest
        want += want < 0.02
        a[0] = thr + np.log(want / (1.0 - want)) if want < 1.0 else a[0]
    elif kind == "none":
        a = np.full(r, -30.0) - g.random(r)
    elif kind == "every":
        a = 30.0 + g.random(r)
    elif kind == "wide":            # differences beyond the largest finite number
        a = np.where(g.random(r) < 0.5, 3e38, -3e38) * g.random(r)
    elif kind == "infinite":
        a[:: 5], a[1:: 7] = np.inf, -np.inf
    elif kind == "clamped":         # two classes of equal gates
        a = np.where(g.random(r) < 0.4, 4.0, -4.0)
    elif kind == "scales":          # distances over 76 decades: several passes over the bins
        a = np.sign(a) * 10.0 ** g.uniform(-38.0, 38.0, r)
    elif kind == "steps":           # neighbouring numbers, many of them equal
        a = 1.0 + np.round(40.0 * g.random(r)) * 2.0 ** -23
    elif kind == "masked":          # hard-pruned gates
        a = np.where(g.random(r) < 0.5, -np.inf, a)
    elif kind == "signs":           # equal to the selection
        a = np.where(g.random(r) < 0.5, 0.0, -0.0)
    elif kind == "nan":
        a[r // 3] = np.nan
    return a.astype(np.float32)


@pytest.mark.parametrize("kind", ["normal", "bimodal", "far", "ties", "equal", "half", "none", "every", "wide", "infinite", "clamped", "scales", "steps", "masked",
                                  "signs", "nan"])
@pytest.mark.parametrize("r", [1, 2, 65, 511, 513, 768, 1024])
def test_survivors(b, kind, r):
    a, d_in, d_out = _gates(kind, r), 24, 40
    P, Q = to_dev(np.random.default_rng(1).standard_normal((d_out, r)), "bf16"), to_dev(np.random.default_rng(2).standard_normal((r, d_in)), "bf16")

    def call(in_place):
        gates = torch.from_numpy(a.copy()).cuda()
        zd = gates if in_place else torch.full((r,), float("nan"), device="cuda")
        idx, kd = torch.full((r,), -1, dtype=torch.int32, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda")
        Pc, Qc = empty_dev(d_out, r, torch.bfloat16), empty_dev(r, d_in, torch.bfloat16)
        b.compact_ranks(gates, 0, HC, idx, kd, zd, P, Q, Pc, Qc)
        return int(kd.item()), idx.cpu().numpy(), host(zd), host(Pc), host(Qc)

    one, three = call(False), call(True)
    assert one[0] == three[0]
    for x, y in zip(one[1:], three[1:]):
        assert np.array_equal(x, y, equal_nan=x.dtype.kind == "f")
    if kind != "nan":
        k, idx, _ = O.deterministic_mask(a, *HC)
        assert one[0] == k and np.array_equal(one[1][:k], idx)
    assert b.device_status() == b.OK


def _count_gates(hc, r, units):
    """fp32 gates around the constants' threshold whose fp64 probabilities sum to a half plus about `units` * 2^-20."""
    thr = hc[0] * np.log(-hc[1] / hc[2])
    p = lambda x: 1.0 / (1.0 + np.exp(-(x.astype(np.float64) - thr)))  # noqa: E731
    a = (thr + np.random.default_rng([r, int(hc[0])]).normal(0.0, 0.3, r)).astype(np.float32)
    rest = p(a[1:]).sum()
    want = (0.5 + units * 2.0 ** -20 - rest) % 1.0
    a[0] = thr + np.log(want / (1.0 - want))
    return a


# k = floor(sum + 1/2) must be the fp64 one wherever the fp32 sum is taken for certain: it declines within r + 16 units of 2^-20
@pytest.mark.parametrize("beta,gamma,zeta", [HC, (1.0, -0.5, 1.5), (20.0, -0.1, 1.1), (100.0, -0.1, 1.1), (100.0, -1.1, 1.1), (1000.0, -0.1, 1.1),
                                             (1e5, -0.1, 1.1), (1e7, -0.1, 1.1)])
def test_count_near_a_half(b, beta, gamma, zeta):
    hc = tuple(float(np.float32(v)) for v in (beta, gamma, zeta))
    for r in (300, 1024):
        for units in (0.0, 0.02 * r, 0.25 * r, 0.5 * r, 0.75 * r, r + 20.0, r + 200.0, 1.5 * r, 3.0 * r):
            for sign in (1.0, -1.0):
                a = _count_gates(hc, r, sign * units)
                gates = torch.from_numpy(a).cuda()
                idx, kd = torch.full((r,), -1, dtype=torch.int32, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda")
                b.compact_ranks(gates, 0, hc, idx, kd, torch.empty(r, device="cuda"))
                k, want, _ = O.deterministic_mask(a, *hc)
                assert int(kd.item()) == k and np.array_equal(idx.cpu().numpy()[:k], want), (r, sign * units)
    assert b.device_status() == b.OK
