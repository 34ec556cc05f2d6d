"""The native binding's answers to calls that fail."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_an_output_that_does_not_fit_raises_what_torch_raises():
    import paper_2603_11021_b200 as P
    ctx, none = P.Context(2, 2, device=0), torch.empty(0, dtype=torch.uint8, device="cuda")
    with pytest.raises(torch.OutOfMemoryError):            # 8 TB; no block is read: the matrix has no columns
        P.llvq_dequant_matrix(ctx, none, none.half(), 1 << 20, 0, P.LLVQ_LAYOUT_ROWWISE, ld=1 << 22)
    with pytest.raises(RuntimeError):                      # a negative size
        P.llvq_decode_blocks(ctx, none, -1)
    assert P.llvq_last_error(ctx) == (0, 0)
