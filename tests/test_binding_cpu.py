"""Argument checks of the native binding that need no GPU: they come before the check that the tensors are on the device."""
import pytest
import torch


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_11021_b200 import build
    build.build()
    import paper_2603_11021_b200 as P
    return P.Context(2, 2, device=-1)


def test_a_leading_dimension_that_wraps_is_too_long_for_the_output(ctx):
    import paper_2603_11021_b200 as P
    rows, ld = 1 << 13, 1 << 51                            # (rows - 1) * ld + 1 = -2^51 + 1 modulo 2^64
    idx = torch.zeros(ctx.index_bytes(rows), dtype=torch.uint8)
    gain, w = torch.zeros(rows, dtype=torch.half), torch.zeros(rows, dtype=torch.bfloat16)
    with pytest.raises(AssertionError):
        P.llvq_dequant_matrix(ctx, idx, gain, rows, 1, P.LLVQ_LAYOUT_ROWWISE, w, ld)
    with pytest.raises(AssertionError):
        P.llvq_dequant_matrix_sg(ctx, idx, 0, torch.ones(1), None, rows, 1, w, ld)


def test_the_type_of_an_output_is_not_asked_for_where_the_output_is_given(ctx):
    import paper_2603_11021_b200 as P
    idx, gain = torch.zeros(ctx.index_bytes(8), dtype=torch.uint8), torch.zeros(8, dtype=torch.half)
    x, y = torch.zeros(24, dtype=torch.bfloat16), torch.zeros(8)
    with pytest.raises(TypeError, match="contiguous CUDA tensor"):       # as far as a CPU tensor gets
        P.llvq_gemv(ctx, idx, gain, 8, 24, x, y, y_dtype=None)
    with pytest.raises(TypeError, match="contiguous CUDA tensor"):
        P.llvq_gemv_sg(ctx, idx, 0, torch.ones(1), None, 8, 24, x, y, y_dtype=None)
    with pytest.raises(TypeError, match="torch.dtype"):
        P.llvq_gemv(ctx, idx, gain, 8, 24, x, y_dtype="float32")


@pytest.mark.parametrize("sorted_layout", [False, True])
@pytest.mark.parametrize("dtype", [torch.int8, torch.float16, torch.float64])
def test_outputs_of_several_products_are_binary32_or_bf16(ctx, dtype, sorted_layout):
    # anything else was written as bf16, two bytes per element whatever its width
    import paper_2603_11021_b200 as P
    idx, gain = torch.zeros(ctx.index_bytes(8), dtype=torch.uint8), torch.zeros(8, dtype=torch.half)
    mat = (idx, gain, 8, 24, torch.zeros(24, dtype=torch.bfloat16), torch.zeros(8, dtype=dtype))
    with pytest.raises(AssertionError):
        (P.llvq_gemv_sorted_multi if sorted_layout else P.llvq_gemv_multi)(ctx, [mat], y_dtype=dtype)
