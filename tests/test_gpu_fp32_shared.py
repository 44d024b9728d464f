"""fp32 backward products that share a launch, each with its own cut of K (1 to 8 slices, in clusters that hold several tiles of the
product with fewer slices, and tiles missing from the last cluster): the bits of the separate launches, which a call whose
gradients overwrite its inputs keeps."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


# 64 x 64 tiles x slices of (dH', dP, dX, dQ) for 148 SMs in the comments
@pytest.mark.parametrize("T,d_in,d_out,r", [
    (64, 64, 768, 64),       # 1 x 8, 12 x 1, 1 x 1, 1 x 1
    (1100, 100, 60, 60),     # 18 x 1, 1 x 8, 36 x 1, 2 x 8
    (200, 320, 256, 192),    # 12 x 4, 12 x 2, 20 x 2, 15 x 2
    (200, 320, 300, 192),    # 12 x 4, 15 x 2 in clusters of four (half of the last one empty), 20 x 2, 15 x 2
    (300, 130, 1400, 130),   # 15 x 8, 66 x 4 in clusters of eight, 15 x 2 in clusters of four (half of the last one empty), 9 x 4
    (520, 128, 256, 128),    # 18 x 4, 8 x 8, 18 x 2, 4 x 8
    (2048, 200, 700, 130),   # 96 x 2, 33 x 8, 128 x 2, 12 x 8
    (1500, 640, 640, 640),   # 240 x 1, 100 x 2 of both: more tiles than SMs
])
@pytest.mark.parametrize("accumulate", [False, True])
def test_shared_launch_has_the_bits_of_separate_ones(b, T, d_in, d_out, r, accumulate):
    g = torch.Generator(device="cuda").manual_seed(T + r)
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    X, dY, Q, P, H = rand(T, d_in), rand(T, d_out), rand(r, d_in), rand(d_out, r), rand(T, r)
    z, dz = torch.rand(r, generator=g, device="cuda"), torch.rand(r, generator=g, device="cuda")
    ws = b.alloc_workspace(b.workspace_bytes(b.OP_BWD, T, d_in, d_out, r, b.F32))

    def run(in_place):
        x, dP, dQ, dla = X.clone(), torch.full((d_out, r), 0.25, device="cuda"), torch.full((r, d_in), 0.25, device="cuda"), torch.full((r,), 0.25, device="cuda")
        dX = x if in_place else torch.empty_like(X)
        before = b.launch_count()
        b.gated_lowrank_bwd(dY, x, Q, P, z, dz, H, dX, dP, dQ, dla, ws, accumulate)
        return (dX, dP, dQ, dla), b.launch_count() - before

    shared, n_shared = run(False)
    separate, n_separate = run(True)
    assert (n_shared, n_separate) == (3, 5)
    for a, c in zip(shared, separate):
        assert torch.equal(a, c)
    assert b.device_status() == b.OK


@pytest.mark.parametrize("T,d,launches", [(100, 768, 5), (160, 768, 5), (2048, 768, 5), (128, 700, 3), (200, 768, 3), (554, 512, 3)])
def test_products_that_fill_the_sms_keep_their_launches(b, T, d, launches):
    """The line of the shared launches on 148 SMs: each alone with nearly two blocks per SM (5) or not (3)."""
    rand = lambda *s: torch.randn(*s, device="cuda")  # noqa: E731
    ws = b.alloc_workspace(b.workspace_bytes(b.OP_BWD, T, d, d, d, b.F32))
    before = b.launch_count()
    b.gated_lowrank_bwd(rand(T, d), rand(T, d), rand(d, d), rand(d, d), rand(d), rand(d), rand(T, d), rand(T, d), rand(d, d), rand(d, d), rand(d), ws)
    assert b.launch_count() - before == launches
    assert b.device_status() == b.OK
