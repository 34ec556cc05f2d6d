"""Batched products whose rows are so long that the bits, the blocks or the columns of a row tile leave 32 bits."""
import pytest
import torch

from gpu_util import gemm_error

pytestmark = pytest.mark.gpu

# binary32 accumulation (1e-3 of an output, floored at 1e-3 of the largest) and the rounding of the bf16 output
TOL_BF16_OUT = 1e-3 + 2.0 ** -8


def _random_stream(P, ctx, nblocks, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    gain = (torch.randn(nblocks, generator=g, device="cuda").abs() * 0.02).half()
    if ctx.index_bits <= 64:
        index = torch.randint(0, ctx.num_points, (nblocks,), generator=g, dtype=torch.int64, device="cuda")
        return P.llvq_pack_fields(ctx, index), gain
    assert ctx.index_bits == 72
    out = torch.randint(0, 256, (nblocks, 9), generator=g, dtype=torch.uint8, device="cuda")
    out[:, 8] %= ctx.num_points >> 64                       # below N whatever the low 64 bits are
    return torch.cat([out.reshape(-1), torch.zeros(-nblocks * 9 % 16, dtype=torch.uint8, device="cuda")]), gain


@pytest.mark.parametrize("code", [(2, 13), (2, 53)])
def test_rows_of_a_tile_beyond_2_to_the_32_bits(code):
    # the first bit of row 127 lies 2^32 bits behind that of row 0; rows of whole 16 bytes, so that the last eight can be dequantized alone
    import paper_2603_11021_b200 as P
    ctx, n_out, batch = P.Context(*code, device=0), 128, 2
    bpr = -(-2 ** 32 // (127 * ctx.index_bits) // 16) * 16
    assert 127 * bpr * ctx.index_bits >= 2 ** 32
    k_in = 24 * bpr
    stream, gain = _random_stream(P, ctx, n_out * bpr, seed=5)
    x = torch.randn((batch, k_in), generator=torch.Generator(device="cuda").manual_seed(6), device="cuda").bfloat16()
    y = P.llvq_gemm_small_batch(ctx, stream, gain, n_out, k_in, x)
    first = n_out - 8
    w = P.llvq_dequant_matrix(ctx, stream[first * bpr * ctx.index_bits // 8:], gain[first * bpr:], 8, k_in, P.LLVQ_LAYOUT_ROWWISE)
    want = (x.double() @ w.double().T).cpu().numpy()
    # every thread block sums its share of the columns in an accumulator of its own
    share = k_in // torch.cuda.get_device_properties(0).multi_processor_count
    assert gemm_error(y[:, first:].float().cpu().numpy(), want, share) <= TOL_BF16_OUT
    assert P.llvq_last_error(ctx) == (0, 0)


def test_gains_of_a_tile_beyond_2_to_the_32_blocks():
    # field 0 is the point (4, 4, 0, ..), so a row is known from its gains: zero but for the last rows, whose gains lie 2^32 behind those of
    # row 0.  A code of few classes, one of many, one with class tables in global memory
    import paper_2603_11021_b200 as P
    n_out, bpr = 128, 2 ** 32 // 127 // 8 * 8 + 8
    assert 127 * bpr >= 2 ** 32
    k_in = 24 * bpr
    gain = torch.zeros(n_out * bpr, dtype=torch.half, device="cuda")
    gain[125 * bpr:] = 0.5
    x = torch.zeros((1, k_in), dtype=torch.bfloat16, device="cuda")
    x[0, ::24 * 1024] = 1.0                                # whole numbers: exact in binary32 whatever the order of the sums
    want = 2.0 * x.count_nonzero().item()
    for code in [(2, 2), (2, 8), (2, 53)]:
        ctx = P.Context(*code, device=0)
        stream = torch.zeros(ctx.index_bytes(n_out * bpr), dtype=torch.uint8, device="cuda")
        y = P.llvq_gemm_small_batch(ctx, stream, gain, n_out, k_in, x).float()
        assert y[0, 125:].tolist() == pytest.approx([want] * 3, rel=2.0 ** -8), code      # the rounding of the bf16 output
        assert not y[0, :125].any(), code
        assert P.llvq_last_error(ctx) == (0, 0)
        del stream


def test_columns_beyond_2_to_the_31():
    # the column coordinates of a TMA copy are signed 32-bit numbers
    import paper_2603_11021_b200 as P
    k_in = 2 ** 31 + 4800
    nblocks = -(-k_in // 24)
    x = torch.zeros((1, k_in), dtype=torch.bfloat16, device="cuda")
    x[0, 0], x[0, 24 * (nblocks - 100)] = 3.0, 5.0
    gain = torch.full((nblocks,), 0.5, dtype=torch.half, device="cuda")
    for code in [(2, 2), (2, 8)]:
        ctx = P.Context(*code, device=0)
        stream = torch.zeros(ctx.index_bytes(nblocks), dtype=torch.uint8, device="cuda")      # field 0: the point (4, 4, 0, ..)
        assert P.llvq_gemm_small_batch(ctx, stream, gain, 1, k_in, x).item() == 16.0
        assert P.llvq_last_error(ctx) == (0, 0)


def test_rows_too_long_for_the_kernels_that_copy_x_by_tma_are_refused():
    # refused by the size alone, before anything is launched
    import paper_2603_11021_b200 as P
    k_in, some = 2 ** 30 + 8, torch.zeros(64, device="cuda").data_ptr()
    L = P.load_library()
    for code in [(2, 2), (2, 8), (2, 53)]:
        ctx = P.Context(*code, device=0)
        args = (ctx._h, some, some, 1, k_in, some, 1, some, None)
        assert L.llvq_gemm_small_batch_sorted(*args) == 3
        if code == (2, 53):
            assert L.llvq_gemm_small_batch(*args) == 3
            assert L.llvq_gemv_sorted(ctx._h, some, some, 1, k_in, some, some, P.LLVQ_F32, None) == 3
