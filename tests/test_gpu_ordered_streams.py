"""The products that order a stored stream inside the kernel, at the edges of their pieces, domains and tiles, against the oracle.

Tolerance: products accumulate in binary32, against the oracle's binary64: 1e-3 of an output, floored at 1e-3 of the largest; outputs in
bf16 add the rounding to 8 significand bits (at most 2^-8 of the output)."""
import os

import numpy as np
import pytest
import torch

import llvq_inputs as gen
from gpu_util import gemm_error, gemv_error, to_dev_bf16, to_dev_f16, to_dev_u8

pytestmark = pytest.mark.gpu

TOL = 1e-3
TOL_BF16_OUT = 1e-3 + 2.0 ** -8


def _f32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _layer(o, bits, n_out, k_in, X):
    """The call's arguments behind the context, and the exact product, of the stored-gain (bits None) or shape-gain form."""
    if bits is None:
        stream, gain, _ = gen.make_layer(o.N, o.W, n_out, k_in, 1, seed=n_out)
        return (to_dev_u8(stream), to_dev_f16(gain)), o.gemm(stream, gain, n_out, k_in, X, threads=os.cpu_count() or 1)
    from oracle.gain_codebook import chi_codebook
    stream, _ = gen.make_layer_sg(o.N, o.W, bits, n_out, k_in, seed=n_out)
    cb, rs = chi_codebook(bits).astype(np.float32), gen.row_scales_f32(n_out, seed=3)
    return (to_dev_u8(stream), bits, _f32(cb), _f32(rs)), o.gemm_sg(stream, bits, cb, rs, n_out, k_in, X, threads=os.cpu_count() or 1)


# a piece of the GEMV is 32 units of 8 rows x 4 blocks, and 256 units per thread block are the most that the kernel which orders its whole
# range takes: one unit more than that, with rows, columns and the last piece ragged; the same with one block per row (every unit a row group
# of its own, several passes); many pieces per team
@pytest.mark.parametrize("code,bits", [((2, 13), None), ((2, 12), 1)])
@pytest.mark.parametrize("shape", ["wide", "narrow", "long"])
def test_gemv_of_more_units_than_one_segment(oracle_mod, code, bits, shape):
    import paper_2603_11021_b200 as P
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_out, k_in = {"wide": (8 * (256 * sms // 38 + 4) - 7, 24 * 4 * 37 + 8), "narrow": (8 * 257 * sms + 3, 8), "long": (8 * 11 * sms + 1, 24 * 4 * 60 - 8)}[shape]
    ctx, o = P.Context(*code, device=0), oracle_mod.Code(*code)
    x = gen.normal_bf16((1, k_in), seed=1)
    args, want = _layer(o, bits, n_out, k_in, x)
    gemv = P.llvq_gemv if bits is None else P.llvq_gemv_sg
    y = gemv(ctx, *args, n_out, k_in, to_dev_bf16(x[0]))
    yb = gemv(ctx, *args, n_out, k_in, to_dev_bf16(x[0]), y_dtype=torch.bfloat16)
    torch.cuda.synchronize()
    assert gemv_error(y.cpu().numpy(), want[0]) <= TOL
    assert gemv_error(yb.float().cpu().numpy(), want[0]) <= TOL_BF16_OUT
    assert P.llvq_last_error(ctx) == (0, 0)


# a domain of the batched product is 128 rows x 8 blocks, and two teams take the domains of a thread block in turn: one block; one domain; two
# and three domains of ragged rows; several tiles per thread block that start with either team.  Batches at the edges of the padding
# to 16 and of the two forms of the X buffers.  Shells 2..20: class tables in global memory with an index below 64 bits
@pytest.mark.parametrize("code,bits", [((2, 13), None), ((2, 12), 1), ((2, 10), 4), ((2, 53), None), ((2, 20), None)])
@pytest.mark.parametrize("n_out,k_in,batch", [(1, 8, 1), (128, 192, 16), (129, 200, 17), (300, 400, 33), (127, 584, 48), (128 * 150 + 1, 400, 64)])
def test_gemm_of_a_stored_stream_by_two_teams(oracle_mod, code, bits, n_out, k_in, batch):
    import paper_2603_11021_b200 as P
    ctx, o = P.Context(*code, device=0), oracle_mod.Code(*code)
    X = gen.normal_bf16((batch, k_in), seed=2)
    args, want = _layer(o, bits, n_out, k_in, X)
    gemm = P.llvq_gemm_small_batch if bits is None else P.llvq_gemm_small_batch_sg
    for _ in range(2):                                     # the counters and histograms are left as they were found
        y = gemm(ctx, *args, n_out, k_in, to_dev_bf16(X))
        torch.cuda.synchronize()
        assert gemm_error(y.float().cpu().numpy(), want, k_in) <= TOL_BF16_OUT
    assert P.llvq_last_error(ctx) == (0, 0)
