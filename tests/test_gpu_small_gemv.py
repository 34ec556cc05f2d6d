"""Products of small matrices: row groups shared by one to many thread blocks (whole groups, one exchange, trees of exchanges, scratch and
counter), at most one unit per warp and just beyond, repeated so that a slot left behind by one call shows in the next."""
import numpy as np
import pytest
import torch

import llvq_inputs as gen
import paper_2603_11021_b200 as P
from gpu_util import gemv_error, to_dev_bf16, to_dev_f16, to_dev_u8

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code", [(2, 13), (3, 3)])
@pytest.mark.parametrize("n_out,k_in", [(8, 24), (16, 4100), (133, 500), (160, 8000), (240, 8000), (400, 480), (500, 3100), (1000, 1000), (1184, 768), (1192, 770),
                                        (3800, 480)])
def test_small_products_by_how_a_row_group_is_shared(oracle_mod, code, n_out, k_in):
    o, ctx = oracle_mod.Code(*code), P.Context(*code, device=0)
    stream, gain, _ = gen.make_layer(o.N, o.W, n_out, k_in, 1, seed=n_out)
    x = gen.normal_bf16(k_in, seed=k_in)
    want = o.gemv(stream, gain, n_out, k_in, x)
    d_s, d_g, d_x = to_dev_u8(stream), to_dev_f16(gain), to_dev_bf16(x)
    srt = P.llvq_sort_blocks(ctx, d_s, n_out, k_in)
    for _ in range(3):
        assert gemv_error(P.llvq_gemv(ctx, d_s, d_g, n_out, k_in, d_x).cpu().numpy(), want) <= 1e-3
        assert gemv_error(P.llvq_gemv_sorted(ctx, srt, d_g, n_out, k_in, d_x).cpu().numpy(), want) <= 1e-3
    assert P.llvq_last_error(ctx) == (0, 0)


def test_small_shape_gain_products(oracle_mod):
    from oracle.gain_codebook import chi_codebook
    o, ctx = oracle_mod.Code(2, 12), P.Context(2, 12, device=0)
    for n_out, k_in in [(133, 500), (1000, 1000), (240, 8000)]:
        bpr = (k_in + 23) // 24
        lo, hi = gen.random_indices(o.N, o.W, n_out * bpr, seed=n_out)
        k = gen.gain_indices(n_out * bpr, 1, seed=n_out)
        d_s = to_dev_u8(gen.pack_indices(lo | (k << np.uint64(o.W)), hi, o.W + 1))
        cb = torch.tensor(chi_codebook(1), dtype=torch.float32, device="cuda")
        scale = torch.linspace(0.01, 0.03, n_out, device="cuda")
        x = to_dev_bf16(gen.normal_bf16(k_in, seed=1))
        w = P.llvq_dequant_matrix_sg(ctx, d_s, 1, cb, scale, n_out, k_in).double()
        want = (w @ x.double()).cpu().numpy()
        for _ in range(2):
            assert gemv_error(P.llvq_gemv_sg(ctx, d_s, 1, cb, scale, n_out, k_in, x).cpu().numpy(), want) <= 1e-3
    assert P.llvq_last_error(ctx) == (0, 0)


@pytest.mark.parametrize("blocks", [31, 32, 33])          # units per thread block where every group of 8 rows has one: the two kernels' border lies at 32
@pytest.mark.parametrize("gain_bits", [None, 1])
def test_out_of_range_blocks_add_nothing_whatever_they_meet(oracle_mod, blocks, gain_bits):
    code = (2, 13) if gain_bits is None else (2, 12)
    o, ctx = oracle_mod.Code(*code), P.Context(*code, device=0)
    n_out, k_in = 8 * torch.cuda.get_device_properties(0).multi_processor_count, 96 * blocks
    bpr, row = k_in // 24, 777
    lo, hi = gen.random_indices(o.N, o.W, n_out * bpr, seed=blocks)
    x = gen.normal_bf16(k_in, seed=1)
    for at in (3, bpr - 1):
        lo[row * bpr + at] = o.N                          # the first index that is out of range ...
    d_x = to_dev_bf16(x)
    d_x[24 * 3 + 5], d_x[24 * (bpr - 1)] = float("inf"), float("nan")       # ... meets what is not finite
    x[24 * 3:24 * 4] = x[24 * (bpr - 1):] = 0
    if gain_bits is None:
        gain = gen.make_layer(o.N, o.W, n_out, k_in, 1, seed=2)[1]
        gain[row * bpr + 3] = 0x7c00
        d_s, d_g = to_dev_u8(gen.pack_indices(lo, hi, o.W)), to_dev_f16(gain)
        y = P.llvq_gemv(ctx, d_s, d_g, n_out, k_in, d_x)
        w = P.llvq_dequant_matrix(ctx, d_s, d_g, n_out, k_in, P.LLVQ_LAYOUT_ROWWISE)
    else:
        k = gen.gain_indices(n_out * bpr, gain_bits, seed=2)
        d_s = to_dev_u8(gen.pack_indices(lo | (k << np.uint64(o.W)), hi, o.W + gain_bits))
        cb, scale = torch.tensor([4.3, 5.4], device="cuda"), torch.full((n_out,), 0.02, device="cuda")
        y = P.llvq_gemv_sg(ctx, d_s, gain_bits, cb, scale, n_out, k_in, d_x)
        w = P.llvq_dequant_matrix_sg(ctx, d_s, gain_bits, cb, scale, n_out, k_in)
    terms = torch.where(to_dev_bf16(x) == 0, 0.0, w[row].double() * to_dev_bf16(x).double())
    assert abs(y[row].item() - terms.sum().item()) <= 100 * 2.0 ** -24 * terms.abs().sum().item()      # a term goes through fewer than 100 binary32 additions
    assert P.llvq_last_error(ctx)[0] == 4                 # two blocks, counted by the product and by the dequantizer


def test_groups_shared_by_many_and_by_two_in_one_launch(oracle_mod):
    # the trees of slots serve the first and the last of these matrices, the pairs of slots the other one
    o, ctx = oracle_mod.Code(2, 13), P.Context(2, 13, device=0)
    mats, want = [], []
    for n_out, k_in in [(240, 8000), (4096, 480), (1000, 1000)]:
        stream, gain, _ = gen.make_layer(o.N, o.W, n_out, k_in, 1, seed=n_out)
        x = gen.normal_bf16(k_in, seed=k_in)
        want.append(o.gemv(stream, gain, n_out, k_in, x))
        mats.append((to_dev_u8(stream), to_dev_f16(gain), n_out, k_in, to_dev_bf16(x)))
    y = [torch.empty(m[2], dtype=torch.float32, device="cuda") for m in mats]
    stored = [m + (out,) for m, out in zip(mats, y)]
    srt = [(P.llvq_sort_blocks(ctx, m[0], m[2], m[3]),) + m[1:] for m in stored]
    for multi, args in [(P.llvq_gemv_multi, stored), (P.llvq_gemv_sorted_multi, srt), (P.llvq_gemv_sorted_multi, srt[:2]), (P.llvq_gemv_multi, stored)]:
        for out in y:
            out.fill_(-1)
        multi(ctx, args)
        for out, w in zip(y[:len(args)], want):
            assert gemv_error(out.cpu().numpy(), w) <= 1e-3
    assert P.llvq_last_error(ctx) == (0, 0)
