"""The one-launch expected-L0 call on both sides of its limit (65 536 gates), with empty and uneven segments, segments that cross
the runs its warps take and tables of mostly empty segments, against the oracle.  out4 is formed in fp64 from probabilities good to a few fp32 ulp, the gradient adds one fp32
product to what is there: relative 2e-6."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import flop_oracle as O
from tests._util import HC, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("sizes", [[1], [31, 0, 33], [256], [2048], [2049], [768] * 72, [0, 5000, 1, 0, 7], [512] * 128, [512] * 128 + [1], [3] * 4000,
                                   [65000] + [1] * 31, [1] * 31 + [65000], [0] * 4000 + [40000] + [0] * 90, [20000, 0, 1, 30000, 0], [511, 513, 512, 1, 3000],
                                   [65536], [33, 0, 4063] * 16])
@pytest.mark.parametrize("noalloc", [False, True])
def test_against_the_oracle(b, sizes, noalloc):
    g = np.random.default_rng(len(sizes))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n, a, size = int(off[-1]), g.normal(0.5, 2.0, int(off[-1])).astype(np.float32), g.uniform(100, 3000, len(sizes)).astype(np.float32)
    dev = lambda v: torch.from_numpy(np.asarray(v)).cuda()
    out4, seg, dla = torch.full((4,), float("nan"), device="cuda"), torch.full((len(sizes),), float("nan"), device="cuda"), dev(np.linspace(-1, 1, n).astype(np.float32))
    args = (dev(a), dev(off), dev(size), HC, dev(np.float32([0.4])), dev(np.float32([0.3, 1.7])), out4, seg, dla)
    if noalloc:
        b.expected_l0_lagrangian_noalloc(*args)
    else:
        b.expected_l0_lagrangian(*args, b.alloc_workspace(b.workspace_bytes(b.OP_L0, n, 0, 0, len(sizes), b.F32)))
    assert b.device_status() == b.OK
    want = O.expected_l0_lagrangian(a, off, size, *HC, float(np.float32(0.4)), float(np.float32(0.3)), float(np.float32(1.7)))
    ref = np.array([want["s"], want["g"], want["dg_dlambda1"], want["dg_dlambda2"]])
    assert np.all(np.abs(host(out4) - ref) <= 2e-6 * np.maximum(np.abs(ref), want["s"]))
    assert np.all(np.abs(host(seg) - want["seg_expected"]) <= 2e-6 * np.maximum(want["seg_expected"], 1.0))
    base = np.linspace(-1, 1, n).astype(np.float32).astype(np.float64)
    assert np.all(np.abs(host(dla) - (base + want["dlog_alpha"])) <= 1e-6 * (np.abs(base) + np.abs(want["dlog_alpha"])) + 2e-6 * np.abs(want["dlog_alpha"]) + 1e-12)


@pytest.mark.parametrize("at", [0, 2, 3])
def test_results_over_the_multipliers(b, at):
    """out4 on the same memory as lambda (and target): every block has read them before the results are written."""
    sizes = [768] * 72
    g = np.random.default_rng(7)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    a, size = g.normal(0.5, 2.0, int(off[-1])).astype(np.float32), g.uniform(100, 3000, len(sizes)).astype(np.float32)
    want = O.expected_l0_lagrangian(a, off, size, *HC, float(np.float32(0.4)), float(np.float32(0.3)), float(np.float32(1.7)))
    dev = lambda v: torch.from_numpy(np.asarray(v)).cuda()
    ws = b.alloc_workspace(b.workspace_bytes(b.OP_L0, a.size, 0, 0, len(sizes), b.F32))
    la, offd, sized = dev(a), dev(off), dev(size)
    for _ in range(50):
        buf, dla = dev(np.float32([9, 9, 0.3, 1.7, 0.4, 9, 9, 9])), torch.zeros(a.size, device="cuda")
        b.expected_l0_lagrangian(la, offd, sized, HC, buf[4:5], buf[2:4], buf[at:at + 4], None, dla, ws)
        assert abs(float(buf[at]) - want["s"]) <= 2e-6 * want["s"]
        assert np.all(np.abs(host(dla) - want["dlog_alpha"]) <= 3e-6 * np.abs(want["dlog_alpha"]) + 1e-12)
    assert b.device_status() == b.OK


def _time_us(b, sizes):
    off = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]), device="cuda")
    n, zeros = int(off[-1]), lambda k: torch.zeros(k, device="cuda")
    args = (zeros(n), off, torch.ones(len(sizes), device="cuda"), HC, zeros(1), zeros(2), zeros(4), zeros(len(sizes)), zeros(n),
            b.alloc_workspace(b.workspace_bytes(b.OP_L0, n, 0, 0, len(sizes), b.F32)))
    best = float("inf")
    for _ in range(5):
        a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            b.expected_l0_lagrangian(*args)
        e.record()
        e.synchronize()
        best = min(best, a.elapsed_time(e) * 50)
    return best


@pytest.mark.parametrize("sizes", [[65000] + [1] * 31, [32000, 32000] + [1] * 40, [1] * 100 + [32768]])
def test_an_uneven_table_costs_about_what_an_even_one_does(b, sizes):
    """One long segment took sixteen times as long when a warp walked a whole segment; three times leaves room for noise."""
    assert _time_us(b, sizes) < 3 * _time_us(b, [sum(sizes) // 64] * 64)


CAPTURE_AFTER_SMALL = """
import torch
from paper_1910_04732_b200 import binding as b
hc = (2.0 / 3.0, -0.1, 1.1)
def table(sizes):
    n = sum(sizes)
    off = torch.cumsum(torch.tensor([0] + sizes), 0).cuda()
    return (torch.linspace(-3, 3, n, device="cuda"), off, torch.full((len(sizes),), 100.0, device="cuda"), hc, torch.tensor([0.5], device="cuda"),
            torch.tensor([0.3, 1.7], device="cuda"), torch.zeros(4, device="cuda"), torch.zeros(len(sizes), device="cuda"), torch.zeros(n, device="cuda"))
small, large = table([64]), table([2048] * 40)
b.expected_l0_lagrangian_noalloc(*small)
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    b.expected_l0_lagrangian_noalloc(*large)
g.replay()
torch.cuda.synchronize()
want = table([2048] * 40)
b.expected_l0_lagrangian(*want, b.alloc_workspace(b.workspace_bytes(b.OP_L0, 81920, 0, 0, 40, b.F32)))
assert torch.equal(large[6], want[6]) and torch.equal(large[8], want[8]) and float(large[6][0]) > 0
assert b.device_status() == b.OK
print("captured")
"""


def test_first_call_small_then_a_larger_one_captured(b):
    """The first call on a device looks up the built-in scratch even when it needs none, so that a later call may be captured.
    In a process of its own: the lookup happens once per process."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CAPTURE_AFTER_SMALL], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "captured", r.stderr[-2000:]
