"""Products on stored fields of 49 to 64 bits of codes whose class tables fit shared memory, against the oracle.

Tolerance: products accumulate in binary32, against the oracle's binary64: 1e-3 of an output, floored at 1e-3 of the largest, plus the
rounding to 8 significand bits of a bf16 output (at most 2^-8 of it)."""
import os

import numpy as np
import pytest
import torch

import llvq_inputs as gen
from gpu_util import gemm_error, to_dev_bf16, to_dev_f16, to_dev_u8

pytestmark = pytest.mark.gpu

TOL_BF16_OUT = 1e-3 + 2.0 ** -8


# 50 and 51 bits of index; an index of 48 bits with 1 and 8 bits of gain; 53 + 8 bits.  Small and large padded batches, ragged tiles
@pytest.mark.parametrize("code,bits", [((2, 14), None), ((2, 15), None), ((2, 13), 1), ((2, 13), 8), ((17, 18), 8)])
@pytest.mark.parametrize("n_out,k_in,batch", [(5, 40, 1), (129, 200, 16), (300, 584, 33), (127, 1000, 64)])
def test_batched_product_of_wide_fields(oracle_mod, code, bits, n_out, k_in, batch):
    import paper_2603_11021_b200 as P
    ctx, o = P.Context(*code, device=0), oracle_mod.Code(*code)
    assert 48 < ctx.index_bits + (bits or 0) <= 64
    X, threads = gen.normal_bf16((batch, k_in), seed=4), os.cpu_count() or 1
    if bits is None:
        stream, gain, _ = gen.make_layer(o.N, o.W, n_out, k_in, 1, seed=n_out)
        want = o.gemm(stream, gain, n_out, k_in, X, threads=threads)
        y = P.llvq_gemm_small_batch(ctx, to_dev_u8(stream), to_dev_f16(gain), n_out, k_in, to_dev_bf16(X))
    else:
        stream, _ = gen.make_layer_sg(o.N, o.W, bits, n_out, k_in, seed=n_out)
        cb, rs = np.linspace(3.0, 7.0, 1 << bits, dtype=np.float32), gen.row_scales_f32(n_out, seed=3)
        want = o.gemm_sg(stream, bits, cb, rs, n_out, k_in, X, threads=threads)
        y = P.llvq_gemm_small_batch_sg(ctx, to_dev_u8(stream), bits, torch.from_numpy(cb).cuda(), torch.from_numpy(rs).cuda(), n_out, k_in,
                                       to_dev_bf16(X))
    assert gemm_error(y.float().cpu().numpy(), want, k_in) <= TOL_BF16_OUT
    assert P.llvq_last_error(ctx) == (0, 0)
