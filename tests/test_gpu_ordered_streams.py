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


# several matrices on their stored streams, one of them with more units per thread block than a segment, so that the ordering kernel takes
# all: short shares before it and longer rows behind it carry the teams' histograms from matrix to matrix
@pytest.mark.parametrize("y_dtype", [torch.float32, torch.bfloat16])
def test_several_products_of_more_units_than_one_segment(oracle_mod, y_dtype):
    import paper_2603_11021_b200 as P
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx, o = P.Context(2, 13, device=0), oracle_mod.Code(2, 13)
    shapes = [(8 * (sms // 5) + 3, 24 * 4 * 5 + 17), (8 * (256 * sms // 38 + 4) - 7, 24 * 4 * 37 + 8), (8 * (sms // 60 + 1) + 1, 24 * 4 * 60 - 8), (8 * sms, 24)]
    mats, want = [], []
    for n_out, k_in in shapes:
        x = gen.normal_bf16((1, k_in), seed=n_out)
        args, w = _layer(o, None, n_out, k_in, x)
        mats.append((*args, n_out, k_in, to_dev_bf16(x[0]), torch.empty(n_out, dtype=y_dtype, device="cuda")))
        want.append(w[0])
    for _ in range(2):                                     # the scratch and the counters are left as they were found
        for m in mats:
            m[5].fill_(float("nan"))
        P.llvq_gemv_multi(ctx, mats, y_dtype=y_dtype)
        for m, w in zip(mats, want):
            assert gemv_error(m[5].float().cpu().numpy(), w) <= (TOL if y_dtype == torch.float32 else TOL_BF16_OUT)
    assert P.llvq_last_error(ctx) == (0, 0)


# a band of more units per thread block than a segment (narrow rows keep it small) and a small one behind it, each written into both copies
def test_row_sharded_gemv_of_more_units_than_one_segment(oracle_mod):
    import paper_2603_11021_b200 as P
    from paper_2603_11021_b200.rowshard import band_of_stream
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx, o, k_in = P.Context(2, 13, device=0), oracle_mod.Code(2, 13), 8
    bands = [(0, 8 * 257 * sms), (8 * 257 * sms, 13)]
    n_out = bands[1][0] + bands[1][1]
    stream, gain, _ = gen.make_layer(o.N, o.W, n_out, k_in, 1, seed=9)
    x = gen.normal_bf16(k_in, seed=9)
    want = o.gemv(stream, gain, n_out, k_in, x, threads=4)
    copies = [torch.full((n_out,), float("nan"), device="cuda") for _ in bands]
    flags = [torch.zeros(2, dtype=torch.int32, device="cuda") for _ in bands]
    for r, (row0, n) in enumerate(bands):
        s, g = band_of_stream(stream, gain, k_in, o.W, row0, n)
        P.llvq_gemv_rowshard(ctx, to_dev_u8(s), to_dev_f16(g), n, k_in, to_dev_bf16(x), copies, r, row0, torch.float32,
                             flag_words=[f.data_ptr() + 4 * r for f in flags], epoch=3)
    torch.cuda.synchronize()
    assert [f.tolist() for f in flags] == [[0, 3], [3, 0]]
    for y in copies:
        assert gemv_error(y.cpu().numpy(), want) <= TOL
    assert P.llvq_last_error(ctx) == (0, 0)


@pytest.mark.parametrize("batch", [16, 64])
def test_row_sharded_batched_product_of_the_72_bit_code(oracle_mod, batch):
    import paper_2603_11021_b200 as P
    from paper_2603_11021_b200.rowshard import band_of_stream, row_bands
    ctx, o, n_out, k_in = P.Context(2, 53, device=0), oracle_mod.Code(2, 53), 300, 584
    stream, gain, _ = gen.make_layer(o.N, o.W, n_out, k_in, 1, seed=10)
    X = gen.normal_bf16((batch, k_in), seed=10)
    want = o.gemm(stream, gain, n_out, k_in, X, threads=os.cpu_count() or 1)
    copies = [torch.full((batch, n_out), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    flags = [torch.zeros(2, dtype=torch.int32, device="cuda") for _ in range(2)]
    for r, (row0, n) in enumerate(row_bands(n_out, 2)):
        s, g = band_of_stream(stream, gain, k_in, o.W, row0, n)
        P.llvq_gemm_small_batch_rowshard(ctx, to_dev_u8(s), to_dev_f16(g), n, k_in, to_dev_bf16(X), copies, r, row0, n_out,
                                         flag_words=[f.data_ptr() + 4 * r for f in flags], epoch=4)
    torch.cuda.synchronize()
    assert [f.tolist() for f in flags] == [[0, 4], [4, 0]]
    for y in copies:
        assert gemm_error(y.float().cpu().numpy(), want, k_in) <= TOL_BF16_OUT
    assert P.llvq_last_error(ctx) == (0, 0)
