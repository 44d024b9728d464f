"""Launches that give a persistent unit more work items than its table in shared memory holds (32): single products on one-CTA and
pair tiles, and grouped calls whose rank only the device knows, where the items beyond the table are decoded by each role and
must come out as active or empty for all of them alike.  Against fp32 products of the same operands on the device (bf16 outputs
of 72- to 1024-term sums: the element-wise bf16 bound of tests/_util.py)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
BF = torch.bfloat16


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


def _rand(rows, cols, scale=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(rows + cols)
    return (torch.randn(rows, cols, generator=g, device="cuda") * scale).to(BF)


def _close(got, A, B, rows=8192):
    """got = A B^T, in slabs of rows; per element 2^-7 of the value and 2 % of the row's rms, as in tests/_util.py, and what two fp32
    sums of K terms in different orders can differ by, 2 K 2^-24 sum |a b|: a row of one column can cancel to nearly nothing, and
    its rms with it."""
    for r in range(0, got.shape[0], rows):
        want = A[r:r + rows].float() @ B.float().T
        err = (got[r:r + rows].float() - want).abs()
        bound = 2.0 ** -7 * want.abs() + 2.0e-2 * want.square().mean(1, keepdim=True).sqrt()
        bound += 2 * A.shape[1] * 2.0 ** -24 * (A[r:r + rows].float().abs() @ B.float().abs().T)
        assert bool((err <= bound).all()), (r, float((err / bound.clamp_min(1e-30)).max()))


@pytest.fixture(autouse=True)
def exact_reference():
    before = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    yield
    torch.backends.cuda.matmul.allow_tf32 = before


@pytest.mark.parametrize("cta2", [0, 1])
@pytest.mark.parametrize("b_mn", [False, True])
def test_one_product(b, cta2, b_mn):
    M, N, K = 79500, 2040, 72          # 622 x 8 tiles of 128 x 256 on 148 CTAs (33.6 each), 311 x 8 of 256 x 256 on 74 pairs
    A, B, D = _rand(M, K), _rand(N, K, K ** -0.5), torch.full((M, N), float("nan"), dtype=BF, device="cuda")
    b.tc_gemm(A, False, B.T.contiguous() if b_mn else B, b_mn, M, N, K, D=D, bn=256, cta2=cta2)
    _close(D, A, B)
    assert b.device_status() == b.OK


@pytest.mark.parametrize("k", [1, 300, 1024])
def test_grouped_calls_with_a_rank_on_the_device(b, k):
    T, d, r = 157000, 72, 1024         # 614 x 4 pair tiles of H' and of Y: 33.2 per pair
    X, Q, P, z = _rand(T, d), _rand(r, d, d ** -0.5), _rand(r, r, k ** -0.5), torch.linspace(0.1, 1.0, r, device="cuda")
    kd = torch.tensor([k], dtype=torch.int32, device="cuda")
    Qk, Pk = Q.clone(), P.clone()
    Qk[k:], Pk[:, k:] = 0, 0           # what a gather leaves beyond the rank, up to the next multiple of 64 at least
    H, Y = torch.zeros(T, r, dtype=BF, device="cuda"), torch.full((T, r), float("nan"), dtype=BF, device="cuda")
    b.gated_lowrank_fwd_grouped([b.fwd_problem(X, Qk, Pk, z, Y, H, r_dev=kd)])
    _close(H[:, :k], X, (Q[:k].float() * z[:k, None]))
    _close(Y, H[:, :k], P[:, :k])
    assert b.device_status() == b.OK
