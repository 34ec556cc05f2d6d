"""The end of a row tile of the batched products: accumulators carried out by a warp per 16 columns and quarter of the rows, tiles shared by thread
blocks converted four values at a time, at batches around both steps and ragged last tiles; repeated, so that scratch left behind shows."""
import pytest
import torch

import llvq_inputs as gen
import paper_2603_11021_b200 as P
from gpu_util import gemm_error, to_dev_bf16, to_dev_f16, to_dev_u8

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code", [(2, 13), (3, 3)])
@pytest.mark.parametrize("n_out,k_in", [(129, 4800), (300, 808), (19000, 96)])
@pytest.mark.parametrize("batch", [1, 8, 15, 16, 17, 32, 33, 40, 48, 49, 64])
def test_batched_products_at_the_end_of_a_tile(oracle_mod, code, n_out, k_in, batch):
    o, ctx = oracle_mod.Code(*code), P.Context(*code, device=0)
    stream, gain, _ = gen.make_layer(o.N, o.W, n_out, k_in, 1, seed=n_out)
    d_s, d_g, d_x = to_dev_u8(stream), to_dev_f16(gain), to_dev_bf16(gen.normal_bf16((batch, k_in), seed=batch))
    w = P.llvq_dequant_matrix(ctx, d_s, d_g, n_out, k_in, P.LLVQ_LAYOUT_ROWWISE).double()
    want = (d_x.double() @ w.T).cpu().numpy()
    srt = P.llvq_sort_blocks_gemm(ctx, d_s, n_out, k_in)
    for _ in range(2):
        assert gemm_error(P.llvq_gemm_small_batch(ctx, d_s, d_g, n_out, k_in, d_x).float().cpu().numpy(), want, k_in) <= 1e-3 + 2.0 ** -8
        assert gemm_error(P.llvq_gemm_small_batch_sorted(ctx, srt, d_g, n_out, k_in, d_x).float().cpu().numpy(), want, k_in) <= 1e-3 + 2.0 ** -8
    assert P.llvq_last_error(ctx) == (0, 0)
