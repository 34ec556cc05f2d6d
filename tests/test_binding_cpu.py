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
