"""Few-token products whose rows end inside a 16-byte piece: padding full of NaN does not reach the result, and the end of a matrix's last
row, whose padding may not exist, is put together from smaller loads for each remainder.  (That these stay inside the row is not
tested: a 16-byte load across its end would neither fault nor change the result.)  Against fp64 products of the same bf16 operands, H' rounded to bf16 in between."""
import pytest
import torch

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


@pytest.fixture(scope="module")
def b():
    from paper_1910_04732_b200 import build, binding
    build.build()
    binding.load_library()
    return binding


def _matrix(g, rows, cols, scale):
    """Rows padded with NaN; the buffer ends with the last element of the last row."""
    ld = (cols + 7) // 8 * 8
    flat = torch.full(((rows - 1) * ld + cols,), float("nan"), dtype=BF16, device="cuda")
    m = flat.as_strided((rows, cols), (ld, 1))
    m.copy_(torch.randn(rows, cols, generator=g, device="cuda") * scale)
    return m


@pytest.mark.parametrize("T", [17, 32, 33, 64, 65, 150])
@pytest.mark.parametrize("k", [1, 7, 15, 33, 35, 100, 255, 358])
@pytest.mark.parametrize("d_in,d_out", [(410, 410), (33, 1000), (301, 97)])
def test_ragged_rows(b, T, k, d_in, d_out):
    g = torch.Generator(device="cuda").manual_seed(T * k)
    X, Q, P = _matrix(g, T, d_in, 1.0), _matrix(g, k, d_in, d_in ** -0.5), _matrix(g, d_out, k, k ** -0.5)
    Y = torch.full((T, (d_out + 7) // 8 * 8), float("nan"), dtype=BF16, device="cuda")[:, :d_out]
    b.compact_fwd(X, Q, P, Y, k, b.alloc_workspace(b.workspace_bytes(b.OP_COMPACT_FWD, T, d_in, d_out, k, b.BF16)))
    exact = X.double() @ Q.double().T
    want = exact.to(BF16).double() @ P.double().T
    # the result is rounded to 8 significant bits, half a step of at most 2^-7 of it; a value of H' whose fp32 sum falls on the other
    # side of a rounding is off by a whole step, and the worst case is that all are
    moved = (exact.abs() * 2.0 ** -7) @ P.double().abs().T
    assert torch.all((Y.double() - want).abs() <= want.abs() * 2.0 ** -8 + moved * (1.0 + 2.0 ** -8) + 1e-6)
    assert b.device_status() == b.OK


@pytest.mark.parametrize("T,k,d_out", [
    (100, 40, 4096), (256, 40, 4096), (1000, 61, 600),          # 64 and 128 weight rows per block, K over two warps or one
    (100, 100, 4096), (1023, 127, 512), (40, 128, 9000),
    (150, 160, 1024), (150, 255, 2048), (64, 129, 6000), (256, 256, 1500),   # K over four warps, 32 and 64 rows
    (150, 257, 1000), (150, 264, 1000), (64, 300, 900),         # all warps on K, 32 rows and 16
    (257, 160, 2048), (100, 257, 4096),                         # just beyond: tcgen05 tiles
    (17, 348, 5478), (18, 73, 4855), (32, 99, 9000),            # up to 32 tokens, more than two rounds of blocks: rows not clipped
])
def test_block_shapes(b, T, k, d_out):
    """Every block shape above 32 tokens, ragged and whole, and wide outputs of fewer tokens."""
    d_in, g = 72, torch.Generator(device="cuda").manual_seed(T + k)
    X, Q, P = _matrix(g, T, d_in, 1.0), _matrix(g, k, d_in, d_in ** -0.5), _matrix(g, d_out, k, k ** -0.5)
    Y = torch.full((T, (d_out + 15) // 8 * 8), float("nan"), dtype=BF16, device="cuda")[:, :d_out]
    b.compact_fwd(X, Q, P, Y, k, b.alloc_workspace(b.workspace_bytes(b.OP_COMPACT_FWD, T, d_in, d_out, k, b.BF16)))
    exact = X.double() @ Q.double().T
    want = exact.to(BF16).double() @ P.double().T
    moved = (exact.abs() * 2.0 ** -7) @ P.double().abs().T      # as above
    assert torch.all((Y.double() - want).abs() <= want.abs() * 2.0 ** -8 + moved * (1.0 + 2.0 ** -8) + 1e-6)
    assert b.device_status() == b.OK
