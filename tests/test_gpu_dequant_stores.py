"""Dequantized rows that start at every alignment of a weight and end at every kind of remainder, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import llvq_inputs as gen
from gpu_util import bf16_bits, to_dev_f16, to_dev_u8

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code", [(2, 13), (2, 53)])
@pytest.mark.parametrize("cols,ld", [(1, 1), (23, 23), (24, 25), (40, 48), (47, 49), (49, 50), (100, 108), (120, 124), (775, 775)])
def test_rows_at_every_alignment(oracle_mod, code, cols, ld):
    # odd leading dimensions pass through all eight places inside 16 bytes, the even ones through the multiples of 4 and 8 bytes
    import paper_2603_11021_b200 as P
    ctx, o, rows = P.Context(*code, device=0), oracle_mod.Code(*code), 19
    stream, gain, _ = gen.make_layer(o.N, o.W, rows, cols, 1, seed=cols)
    want = o.dequant_matrix(stream, gain, rows, cols, 1)
    w = torch.full((rows, ld), 7.0, dtype=torch.bfloat16, device="cuda")
    P.llvq_dequant_matrix(ctx, to_dev_u8(stream), to_dev_f16(gain), rows, cols, P.LLVQ_LAYOUT_ROWWISE, w, ld)
    torch.cuda.synchronize()
    got = bf16_bits(w)
    assert np.array_equal(got[:, :cols], np.asarray(want).reshape(rows, cols))
    assert (got[:, cols:] == 0x40e0).all()                 # nothing written past a row
    assert P.llvq_last_error(ctx) == (0, 0)
