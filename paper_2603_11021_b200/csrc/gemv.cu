// The fused dequant + GEMV entry points of the C ABI (see include/llvq.h): stored stream, sorted layout, shape-gain
// form and the row-sharded variants, with the kernels they launch (gemv_kernels.cuh).
#include "kernels_common.cuh"

int llvq_internal_gemv_domains(const llvq_ctx* ctx, const void* d_sorted, const uint16_t* d_gain_f16, int64_t n_out, int64_t k_in,
                               const uint16_t* d_x_bf16, void* d_y, int y_dtype, void* stream);      // gemm.cu

namespace {

#include "order.cuh"
#include "gemv_kernels.cuh"

constexpr size_t kSmemLimit = 227 * 1024;

// Shared memory of gemv_bin_kernel, and whether the table of small subsets still fits.  acc_floats = room for the row sums, cut down to one
// copy per row where rows are so long that x needs the space.
void bin_smem(const llvq_ctx* ctx, int64_t nq, size_t& bytes, bool& ext, uint32_t& acc_floats)
{
    const size_t rest = 16 + (size_t)nq * 48 * 4 + 16 + 2 * 1024 * 4 + (size_t)kBinSegUnits * 32 * (8 + 2);
    acc_floats = kSortAccFloats;
    while (acc_floats > kGemvGroupsPerPass * kGemvGroupRows && ctx->fl.total + rest + acc_floats * 4 > kSmemLimit) acc_floats /= 2;
    ext = ctx->fl.total_ext + rest + acc_floats * 4 <= kSmemLimit;
    bytes = (ext ? ctx->fl.total_ext : ctx->fl.total) + rest + acc_floats * 4;
}

// Whether gemv_bin_kernel takes a matrix; order = gemv_order_kernel takes it too, which is preferred to cut row sums.
bool bin_kernel_serves(const llvq_ctx* ctx, int64_t nq, const SgArgs* sg, bool order)
{
    size_t bytes; bool ext; uint32_t acc_floats;
    bin_smem(ctx, nq, bytes, ext, acc_floats);
    return (!sg || sg->bits <= 5) && ctx->fast && ctx->d_sort_rank && ctx->host.desc.size() >= 64 && ctx->host.W <= 48 && bytes <= kSmemLimit &&
           nq < (1ll << 24) && (acc_floats == kSortAccFloats || !order);
}

// Stored streams of codes with many classes: gemv_bin_kernel while a CTA's range is one of its segments (it orders the whole range at
// once, so the warps share classes best), else gemv_order_kernel, whose teams order small pieces and unrank others meanwhile.  Rows of
// 4096, shells 2..13, gemv_bin_kernel / gemv_order_kernel in us by units per CTA: 19 11.7 / 13.8, 74 16.2 / 16.6, 149 23.7 / 26.9, 205 30.0 /
// 30.2, 256 35.2 / 33.9, 298 43.8 / 41.8, 400 54.5 / 53.7, 521 70.9 / 67.1; 595 (8192 x 8192) 82.8 / 71.9.
bool one_segment(int64_t units_per_cta) { return units_per_cta <= kBinSegUnits; }

// Whether gemv_order_kernel takes a matrix of nq units per row group; its shared memory, and whether the table of small subsets
// still fits.
bool order_smem(const llvq_ctx* ctx, int64_t nq, int gain_bits, OrderArgs& oa, size_t& bytes, bool& ext)
{
    // (the GEMV of codes with class tables in global memory is no faster ordered: 4096 x 4096, 72 bits: 49.7 us against 44.2)
    if (!ctx->fast || nq >= (1ll << 24) || !order_args(ctx, gain_bits, &oa)) return false;
    const size_t rest = 16 + (size_t)nq * 48 * 4 + kSortAccFloats * 4 + gemv_order_bytes(oa);
    ext = ctx->fl.total_ext + rest <= kSmemLimit;
    bytes = (ext ? ctx->fl.total_ext : ctx->fl.total) + rest;
    return bytes <= kSmemLimit;
}

// The shared memory of gemv_sorted_kernel; acc_floats = room for the row sums, cut down to one copy per row where rows are so long that x
// needs the space.
void sorted_smem(const llvq_ctx* ctx, int64_t nq, size_t& bytes, bool& ext, uint32_t& acc_floats)
{
    const size_t rest = 16 + (size_t)nq * 48 * 4 + 16;
    acc_floats = kSortAccFloats;
    while (acc_floats > kGemvGroupsPerPass * kGemvGroupRows && ctx->fl.total + rest + acc_floats * 4 > kSmemLimit) acc_floats /= 2;
    ext = ctx->fl.total_ext + rest + acc_floats * 4 <= kSmemLimit;
    bytes = (ext ? ctx->fl.total_ext : ctx->fl.total) + rest + acc_floats * 4;
}

// Where every unit of a matrix has a warp of its own, codes with many classes have nothing to gain from ordering their blocks first: the direct kernel with
// binary32 FMAs.  Shells 2..13, us for gemv_bin_kernel / the direct kernel by units per CTA (of 148): 1 10.4 / 6.2, 5 10.2 / 6.6, 10 9.9 / 6.4, 13 9.0 / 7.0,
// 19 10.7 / 7.3, 27 10.0 / 8.3; with two rounds 37 13.1 / 13.2.
constexpr int64_t kOneRound = 32;
// With two CTAs per row group, or one, a row's sum takes one exchange or none instead of a tree of them: about 1 us, which some ten units more per CTA cost
// (512 x 1024 7.9 -> 6.7 us, 1000 x 1000 8.0 -> 6.4).  The same cut serves the codes that stay with the direct kernel as it was, us without / with it:
// 72 bits 600 x 1000 9.5 / 8.5, 304 x 2880 10.2 / 9.9, 1100 x 2900 12.8 / 11.9; shells 3 600 x 1920 5.2 / 4.8, 1000 x 2000 5.7 / 4.9; shells 2..11 with two gain
// bits 640 x 1900 7.4 / 6.9.  Six more units per CTA and no row whole is where it loses most: 400 x 4000 7.9 / 8.0, 72 bits 10.4 / 10.9.
constexpr int64_t kMoreUnits = 10;

// Shared by llvq_gemv, llvq_gemv_sg and llvq_gemv_rowshard: exactly one of d_gain_f16 / sg is used.
int gemv_common(const llvq_ctx* ctx, const void* d_idx, const uint16_t* d_gain_f16, const SgArgs* sg, int64_t n_out, int64_t k_in,
                       const uint16_t* d_x_bf16, const YOut& yo, int y_dtype, void* stream)
{
    if (!d_x_bf16 || n_out < 0 || k_in < 0) return LLVQ_EINVAL;
    if (int e = check_yout(yo, y_dtype)) return e;
    if (!aligned(d_x_bf16, 2)) return LLVQ_EALIGN;
    if (n_out == 0) return LLVQ_OK;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return LLVQ_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    if (k_in == 0) {
        const size_t bytes = (size_t)n_out * (y_dtype == LLVQ_F32 ? 4 : 2);
        if (cudaMemsetAsync(yo.y, 0, bytes, st) != cudaSuccess) return LLVQ_ECUDA;
        for (int p = 0; p < yo.n_peer; ++p)
            if (cudaMemsetAsync(yo.peer[p], 0, bytes, st) != cudaSuccess) return LLVQ_ECUDA;
        return LLVQ_OK;
    }
    const int64_t bpr = (k_in + 23) / 24;
    const int64_t nq = (bpr + 3) / 4;
    const size_t kSmemMax = 227 * 1024;
    // row groups per pass: the row sums take 32 bytes each beside x, so rows too long for 128 of them get passes of 8
    const size_t rest_x = 16 + (size_t)nq * 48 * 4 + 16;
    const uint32_t per_pass = ctx->fl.total + rest_x + kGemvGroupsPerPass * kGemvGroupRows * 4 <= kSmemMax ? kGemvGroupsPerPass : 8;
    const size_t rest = rest_x + per_pass * kGemvGroupRows * 4;
    // room for the table of small subsets (not for the 72-bit code: its warps hold 32 unrelated classes that almost never take it together)
    const bool ext_direct = ctx->fast && ctx->fl.total_ext + rest <= kSmemMax;
    const size_t smem = (ext_direct ? ctx->fl.total_ext : ctx->fl.total) + rest;
    if (smem > kSmemMax || n_out > 64ll * kMaxScratchRows) return LLVQ_EUNSUPPORTED;
    const int64_t units = ((n_out + kGemvGroupRows - 1) / kGemvGroupRows) * nq;
    unsigned g = (unsigned)std::min<int64_t>(units, ctx->sm_count);
    const bool one_round = units <= kOneRound * g;
    if (one_round) {
        const int64_t groups = units / nq, per_group = std::min<int64_t>(ctx->sm_count / groups, 2);
        if (per_group > 0) {
            const int64_t most = (nq + per_group - 1) / per_group;
            if (most <= kOneRound && most <= (units + g - 1) / g + kMoreUnits) g = (unsigned)std::min(groups * per_group, units);
        }
    }
    const Split sp = make_gemv_split(units, nq, g, n_out);
    // warps per CTA: the count in [28, 32] that wastes the fewest warp slots on the units of one CTA
    const int64_t upc = (units + g - 1) / g;
    int warps = 32; double best_eff = 0.0;
    for (int w = 32; w >= 28; --w) {
        const double eff = (double)upc / (double)(((upc + w - 1) / w) * w);
        if (eff > best_eff + 1e-9) { best_eff = eff; warps = w; }
    }
    const unsigned threads = 32u * (unsigned)warps;
    const uint32_t* idx = static_cast<const uint32_t*>(d_idx);
    const SgArgs sga = sg ? *sg : SgArgs{};
    const bool shard = yo.n_peer > 0 || yo.n_flag > 0;                  // row-sharded launch: stored-gain form only
    if (shard && sg) return LLVQ_EUNSUPPORTED;
    // codes with many classes (a warp of unrelated blocks is what costs there): the kernels that order the blocks before they unrank
    // them; the others, and rows too long for their buffers, go to the direct kernel
    size_t smem_bin; bool ext_bin; uint32_t acc_floats;
    bin_smem(ctx, nq, smem_bin, ext_bin, acc_floats);
    OrderArgs oa;
    size_t smem_order; bool ext_order;
    const bool order = order_smem(ctx, nq, sg ? sg->bits : 0, oa, smem_order, ext_order);
    const bool bin = bin_kernel_serves(ctx, nq, sg, order) && (one_segment(upc) || !order);
    const size_t rest_fma = rest_x + kSortAccFloats * 4;
    const bool ext_fma = ctx->fl.total_ext + rest_fma <= kSmemLimit, fma = one_round && (bin || order) && ctx->fl.total + rest_fma <= kSmemLimit;
    const size_t smem_fma = (ext_fma ? ctx->fl.total_ext : ctx->fl.total) + rest_fma;
    if (bin && !fma) {
        const FastArgs fa = fast_args(ctx, ext_bin);
#define LLVQ_LAUNCH_BIN_T(BF16, SG, SH, TREES)                                                                             \
    do {                                                                                                                   \
        if (!set_smem<gemv_bin_kernel<BF16, SG, SH, TREES>>(ctx, smem_bin)) return LLVQ_ECUDA;                                   \
        if (launch_pdl(gemv_bin_kernel<BF16, SG, SH, TREES>, g, (unsigned)kSortThreads, smem_bin, st, fa, idx, ctx->d_sort_rank, d_gain_f16, sga, sp, n_out, k_in, \
                       bpr, acc_floats, d_x_bf16, yo, ctx->d_scratch, ctx->d_counters) != cudaSuccess) return LLVQ_ECUDA; \
    } while (0)
#define LLVQ_LAUNCH_BIN(BF16, SG, SH) do { if (sp.trees) LLVQ_LAUNCH_BIN_T(BF16, SG, SH, true); else LLVQ_LAUNCH_BIN_T(BF16, SG, SH, false); } while (0)
        if (shard)   { if (y_dtype == LLVQ_BF16) LLVQ_LAUNCH_BIN(true, false, true); else LLVQ_LAUNCH_BIN(false, false, true); }
        else if (sg) { if (y_dtype == LLVQ_BF16) LLVQ_LAUNCH_BIN(true, true, false); else LLVQ_LAUNCH_BIN(false, true, false); }
        else         { if (y_dtype == LLVQ_BF16) LLVQ_LAUNCH_BIN(true, false, false); else LLVQ_LAUNCH_BIN(false, false, false); }
#undef LLVQ_LAUNCH_BIN
#undef LLVQ_LAUNCH_BIN_T
        return launch_status();
    }
    if (order && !fma) {
        const FastArgs fa = fast_args(ctx, ext_order);
#define LLVQ_LAUNCH_ORDER_T(BF16, SG, SH, TREES)                                                                      \
    do {                                                                                                                   \
        if (!set_smem<gemv_order_kernel<BF16, SG, SH, TREES>>(ctx, smem_order)) return LLVQ_ECUDA;                   \
        if (launch_pdl(gemv_order_kernel<BF16, SG, SH, TREES>, g, (unsigned)kSortThreads, smem_order, st, fa, idx, oa, d_gain_f16, sga, sp, n_out, k_in, \
                       bpr, d_x_bf16, yo, ctx->d_scratch, ctx->d_counters) != cudaSuccess) return LLVQ_ECUDA;              \
    } while (0)
        const bool bf16 = y_dtype == LLVQ_BF16;
#define LLVQ_LAUNCH_ORDER(BF16, SG, SH) do { if (sp.trees) LLVQ_LAUNCH_ORDER_T(BF16, SG, SH, true); else LLVQ_LAUNCH_ORDER_T(BF16, SG, SH, false); } while (0)
        if (shard)   { if (bf16) LLVQ_LAUNCH_ORDER(true, false, true); else LLVQ_LAUNCH_ORDER(false, false, true); }
        else if (sg) { if (bf16) LLVQ_LAUNCH_ORDER(true, true, false); else LLVQ_LAUNCH_ORDER(false, true, false); }
        else         { if (bf16) LLVQ_LAUNCH_ORDER(true, false, false); else LLVQ_LAUNCH_ORDER(false, false, false); }
#undef LLVQ_LAUNCH_ORDER
#undef LLVQ_LAUNCH_ORDER_T
        return launch_status();
    }
    const FastArgs fa = fast_args(ctx, fma ? ext_fma : ext_direct);
#define LLVQ_LAUNCH_GEMV_T(BIG, BF16, SG, SH, FMA, TREES)                                                          \
    do {                                                                                                           \
        if (!set_smem<gemv_fast_kernel<BIG, BF16, SG, SH, FMA, TREES>>(ctx, FMA ? smem_fma : smem)) return LLVQ_ECUDA;                          \
        if (launch_pdl(gemv_fast_kernel<BIG, BF16, SG, SH, FMA, TREES>, g, FMA ? fma_threads : threads, FMA ? smem_fma : smem, st, fa, idx, d_gain_f16, sga, sp, FMA ? (uint32_t)kGemvGroupsPerPass : per_pass, n_out, k_in, bpr, \
                       d_x_bf16, yo, ctx->d_scratch, ctx->d_counters) != cudaSuccess) return LLVQ_ECUDA;           \
    } while (0)
#define LLVQ_LAUNCH_GEMV(BIG, BF16, SG, SH, FMA)                                                                   \
    do { if (sp.trees) LLVQ_LAUNCH_GEMV_T(BIG, BF16, SG, SH, FMA, true); else LLVQ_LAUNCH_GEMV_T(BIG, BF16, SG, SH, FMA, false); } while (0)
    const unsigned fma_threads = 32u * (unsigned)std::max<int64_t>(upc, 16);        // a warp per unit
    const bool bf16 = y_dtype == LLVQ_BF16;
    if (fma && shard)       { if (bf16) LLVQ_LAUNCH_GEMV(false, true, false, true, true);   else LLVQ_LAUNCH_GEMV(false, false, false, true, true); }
    else if (fma && sg)     { if (bf16) LLVQ_LAUNCH_GEMV(false, true, true, false, true);   else LLVQ_LAUNCH_GEMV(false, false, true, false, true); }
    else if (fma)           { if (bf16) LLVQ_LAUNCH_GEMV(false, true, false, false, true);  else LLVQ_LAUNCH_GEMV(false, false, false, false, true); }
    else if (shard && ctx->fast) { if (bf16) LLVQ_LAUNCH_GEMV(false, true, false, true, false); else LLVQ_LAUNCH_GEMV(false, false, false, true, false); }
    else if (shard)         { if (bf16) LLVQ_LAUNCH_GEMV(true, true, false, true, false);   else LLVQ_LAUNCH_GEMV(true, false, false, true, false); }
    else if (sg)            { if (bf16) LLVQ_LAUNCH_GEMV(false, true, true, false, false);  else LLVQ_LAUNCH_GEMV(false, false, true, false, false); }
    else if (ctx->fast)     { if (bf16) LLVQ_LAUNCH_GEMV(false, true, false, false, false); else LLVQ_LAUNCH_GEMV(false, false, false, false, false); }
    else                    { if (bf16) LLVQ_LAUNCH_GEMV(true, true, false, false, false);  else LLVQ_LAUNCH_GEMV(true, false, false, false, false); }
#undef LLVQ_LAUNCH_GEMV
#undef LLVQ_LAUNCH_GEMV_T
    return launch_status();
}

// Sorted layout (see the comment at sort_blocks_kernel).  Available for fast-path codes whose indices fit 48 bits
// with 2^48 - 1 left over as the "no block" marker.
bool sortable(const llvq_ctx* ctx, int64_t k_in)
{
    if (!ctx->fast || !ctx->d_sort_rank || ctx->host.W > 48 || ctx->host.N >= (u128)kSortIndexMask) return false;
    const int64_t nq = ((k_in + 23) / 24 + 3) / 4;
    size_t smem; bool ext; uint32_t acc_floats;
    sorted_smem(ctx, nq, smem, ext, acc_floats);
    return smem <= kSmemLimit && nq < (1ll << 24);
}

}  // namespace

extern "C" {

int llvq_gemv(const llvq_ctx* ctx, const void* d_idx, const uint16_t* d_gain_f16, int64_t n_out, int64_t k_in,
              const uint16_t* d_x_bf16, void* d_y, int y_dtype, void* stream)
{
    if (ctx && ctx->device >= 0 && n_out == 0) return LLVQ_OK;                     // nothing to do: pointers may be null
    if (int e = check_common(ctx, d_idx)) return e;
    if (!d_gain_f16) return LLVQ_EINVAL;
    if (!aligned(d_gain_f16, 2)) return LLVQ_EALIGN;
    return gemv_common(ctx, d_idx, d_gain_f16, nullptr, n_out, k_in, d_x_bf16, single_y(d_y), y_dtype, stream);
}

int llvq_gemv_sg(const llvq_ctx* ctx, const void* d_fields, int gain_bits, const float* d_codebook_f32, const float* d_row_scale_f32,
                 int64_t n_out, int64_t k_in, const uint16_t* d_x_bf16, void* d_y, int y_dtype, void* stream)
{
    if (ctx && ctx->device >= 0 && n_out == 0) return LLVQ_OK;                     // nothing to do: pointers may be null
    if (int e = check_sg(ctx, d_fields, gain_bits, d_codebook_f32, d_row_scale_f32)) return e;
    const SgArgs sg{d_codebook_f32, d_row_scale_f32, gain_bits};
    return gemv_common(ctx, d_fields, nullptr, &sg, n_out, k_in, d_x_bf16, single_y(d_y), y_dtype, stream);
}

size_t llvq_sorted_bytes(const llvq_ctx* ctx, int64_t n_out, int64_t k_in)
{
    if (ctx && !ctx->fast) return llvq_sorted_gemm_bytes(ctx, n_out, k_in);      // one sorted layout serves both products of these codes
    if (!ctx || ctx->device < 0 || n_out <= 0 || k_in <= 0 || !sortable(ctx, k_in)) return 0;
    const int64_t nq = ((k_in + 23) / 24 + 3) / 4;
    return (size_t)(((n_out + kGemvGroupRows - 1) / kGemvGroupRows) * nq) * 32 * 8;
}

static int sort_blocks_common(const llvq_ctx* ctx, const void* d_fields, int gain_bits, int64_t n_out, int64_t k_in, void* d_sorted, void* stream)
{
    if (int e = check_common(ctx, d_fields)) return e;
    if (!d_sorted || n_out <= 0 || k_in <= 0 || gain_bits < 0 || gain_bits > 8) return LLVQ_EINVAL;
    if (!aligned(d_sorted, 16)) return LLVQ_EALIGN;
    if (!sortable(ctx, k_in) || ctx->host.W + gain_bits > 48 || n_out > 64ll * kMaxScratchRows) return LLVQ_EUNSUPPORTED;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return LLVQ_ECUDA;
    const int64_t bpr = (k_in + 23) / 24, nq = (bpr + 3) / 4;
    const int64_t units = ((n_out + kGemvGroupRows - 1) / kGemvGroupRows) * nq;
    const unsigned g = (unsigned)std::min<int64_t>(units, ctx->sm_count);
    const size_t smem = ctx->fl.total + 16;
    if (!set_smem<sort_blocks_kernel>(ctx, smem)) return LLVQ_ECUDA;
    sort_blocks_kernel<<<g, kSortThreads, smem, (cudaStream_t)stream>>>(fast_args(ctx), static_cast<const uint32_t*>(d_fields), ctx->d_sort_rank, gain_bits,
                                                                       make_split(units, nq, g), n_out, bpr, static_cast<unsigned long long*>(d_sorted));
    return launch_status();
}

int llvq_sort_blocks(const llvq_ctx* ctx, const void* d_idx, int64_t n_out, int64_t k_in, void* d_sorted, void* stream)
{
    if (ctx && !ctx->fast) return llvq_sort_blocks_gemm(ctx, d_idx, n_out, k_in, d_sorted, stream);
    return sort_blocks_common(ctx, d_idx, 0, n_out, k_in, d_sorted, stream);
}

int llvq_sort_blocks_sg(const llvq_ctx* ctx, const void* d_fields, int gain_bits, int64_t n_out, int64_t k_in, void* d_sorted, void* stream)
{
    return sort_blocks_common(ctx, d_fields, gain_bits, n_out, k_in, d_sorted, stream);
}

// Exactly one of d_gain_f16 / sg is used.
static int gemv_sorted_common(const llvq_ctx* ctx, const void* d_sorted, const uint16_t* d_gain_f16, const SgArgs* sg, int64_t n_out, int64_t k_in,
                              const uint16_t* d_x_bf16, const YOut& yo, int y_dtype, void* stream)
{
    if (!d_x_bf16 || n_out < 0 || k_in <= 0) return LLVQ_EINVAL;
    if (int e = check_yout(yo, y_dtype)) return e;
    if (!aligned(d_x_bf16, 2)) return LLVQ_EALIGN;
    if (!sortable(ctx, k_in) || n_out > 64ll * kMaxScratchRows) return LLVQ_EUNSUPPORTED;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return LLVQ_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t bpr = (k_in + 23) / 24, nq = (bpr + 3) / 4;
    const int64_t units = ((n_out + kGemvGroupRows - 1) / kGemvGroupRows) * nq;
    const unsigned g = (unsigned)std::min<int64_t>(units, ctx->sm_count);
    size_t smem; bool ext; uint32_t acc_floats;
    sorted_smem(ctx, nq, smem, ext, acc_floats);
    const FastArgs fa = fast_args(ctx, ext);
    const Split split = make_gemv_split(units, nq, g, n_out);
    const unsigned long long* sp = static_cast<const unsigned long long*>(d_sorted);
    const SgArgs sga = sg ? *sg : SgArgs{};
#define LLVQ_LAUNCH_SORTED(BF16, SG, SH)                                                                                \
    do {                                                                                                                \
        if (!set_smem<gemv_sorted_kernel<BF16, SG, SH>>(ctx, smem)) return LLVQ_ECUDA;                                        \
        if (launch_pdl(gemv_sorted_kernel<BF16, SG, SH>, g, (unsigned)kSortThreads, smem, st, fa, sp, d_gain_f16, sga, split, n_out, k_in, bpr, \
                       acc_floats, d_x_bf16, yo, ctx->d_scratch, ctx->d_counters) != cudaSuccess) return LLVQ_ECUDA;          \
    } while (0)
    const bool shard = yo.n_peer > 0 || yo.n_flag > 0;                  // row-sharded launch: stored-gain form only
    if (shard && sg) return LLVQ_EUNSUPPORTED;
    if (shard)   { if (y_dtype == LLVQ_BF16) LLVQ_LAUNCH_SORTED(true, false, true); else LLVQ_LAUNCH_SORTED(false, false, true); }
    else if (sg) { if (y_dtype == LLVQ_BF16) LLVQ_LAUNCH_SORTED(true, true, false); else LLVQ_LAUNCH_SORTED(false, true, false); }
    else         { if (y_dtype == LLVQ_BF16) LLVQ_LAUNCH_SORTED(true, false, false); else LLVQ_LAUNCH_SORTED(false, false, false); }
#undef LLVQ_LAUNCH_SORTED
    return launch_status();
}

int llvq_gemv_sorted(const llvq_ctx* ctx, const void* d_sorted, const uint16_t* d_gain_f16, int64_t n_out, int64_t k_in,
                     const uint16_t* d_x_bf16, void* d_y, int y_dtype, void* stream)
{
    if (ctx && ctx->device >= 0 && n_out == 0) return LLVQ_OK;
    if (int e = check_common(ctx, d_sorted)) return e;
    if (!d_gain_f16) return LLVQ_EINVAL;
    if (!aligned(d_gain_f16, 2)) return LLVQ_EALIGN;
    if (!ctx->fast) {
        if (!d_x_bf16 || n_out < 0 || k_in <= 0) return LLVQ_EINVAL;
        if (int e = check_yout(single_y(d_y), y_dtype)) return e;
        return llvq_internal_gemv_domains(ctx, d_sorted, d_gain_f16, n_out, k_in, d_x_bf16, d_y, y_dtype, stream);
    }
    return gemv_sorted_common(ctx, d_sorted, d_gain_f16, nullptr, n_out, k_in, d_x_bf16, single_y(d_y), y_dtype, stream);
}

int llvq_gemv_sorted_sg(const llvq_ctx* ctx, const void* d_sorted, int gain_bits, const float* d_codebook_f32, const float* d_row_scale_f32,
                        int64_t n_out, int64_t k_in, const uint16_t* d_x_bf16, void* d_y, int y_dtype, void* stream)
{
    if (ctx && ctx->device >= 0 && n_out == 0) return LLVQ_OK;
    if (int e = check_sg(ctx, d_sorted, gain_bits, d_codebook_f32, d_row_scale_f32)) return e;
    if (ctx->host.W + gain_bits > 48) return LLVQ_EUNSUPPORTED;
    const SgArgs sg{d_codebook_f32, d_row_scale_f32, gain_bits};
    return gemv_sorted_common(ctx, d_sorted, nullptr, &sg, n_out, k_in, d_x_bf16, single_y(d_y), y_dtype, stream);
}

// llvq_gemv_multi / llvq_gemv_sorted_multi: checks, then one launch that walks the matrices.
static int gemv_multi_common(const llvq_ctx* ctx, const llvq_gemv_desc* descs, int n_mats, int y_dtype, bool sorted, void* stream)
{
    if (!ctx || ctx->device < 0 || !descs || n_mats < 1) return LLVQ_EINVAL;
    if (y_dtype != LLVQ_F32 && y_dtype != LLVQ_BF16) return LLVQ_EINVAL;
    if (n_mats > kMaxMultiMats) return LLVQ_EUNSUPPORTED;
    GemvMulti mm{};
    mm.n = n_mats;
    uint32_t acc_floats = kSortAccFloats;
    int64_t slot = 0, max_nq = 0;
    bool bin = true;                                     // stored streams: which of the two kernels (see one_segment)
    for (int i = 0; i < n_mats; ++i) {
        const llvq_gemv_desc& d = descs[i];
        if (int e = check_common(ctx, d.d_weights)) return e;
        if (!d.d_gain_f16 || !d.d_x_bf16 || !d.d_y || d.n_out <= 0 || d.k_in <= 0) return LLVQ_EINVAL;
        if (!aligned(d.d_gain_f16, 2) || !aligned(d.d_x_bf16, 2) || !aligned(d.d_y, y_dtype == LLVQ_F32 ? 4 : 2)) return LLVQ_EALIGN;
        const int64_t bpr = (d.k_in + 23) / 24, nq = (bpr + 3) / 4;
        const int64_t units = ((d.n_out + kGemvGroupRows - 1) / kGemvGroupRows) * nq;
        // every matrix must give every CTA work: the sorted layout was made for that many CTAs
        if (units < ctx->sm_count) return LLVQ_EUNSUPPORTED;
        if (sorted && !sortable(ctx, d.k_in)) return LLVQ_EUNSUPPORTED;
        bin = bin && one_segment((units + ctx->sm_count - 1) / ctx->sm_count);
        max_nq = std::max(max_nq, nq);
        GemvMat& m = mm.m[i];
        m.weights = d.d_weights; m.gain = d.d_gain_f16; m.x = d.d_x_bf16; m.y = d.d_y;
        m.n_out = d.n_out; m.k_in = d.k_in; m.slot0 = slot;
        m.sp = make_split(units, nq, (unsigned)ctx->sm_count); m.bpr = (int32_t)bpr;
        slot += (d.n_out + kGemvGroupRows - 1) / kGemvGroupRows * kGemvGroupRows;
    }
    if (slot > 64ll * kMaxScratchRows) return LLVQ_EUNSUPPORTED;
    bool trees = false;
    for (int i = 0; i < n_mats; ++i) {
        mm.m[i].sp.trees = tree_rows(mm.m[i].sp, mm.m[i].slot0, mm.m[i].n_out, slot);
        trees = trees || mm.m[i].sp.trees;
    }
    size_t smem; bool ext;                               // the longest rows decide for the whole launch
    OrderArgs oa{};
    if (sorted) sorted_smem(ctx, max_nq, smem, ext, acc_floats);
    else {
        const bool order = order_smem(ctx, max_nq, 0, oa, smem, ext);
        bin = bin_kernel_serves(ctx, max_nq, nullptr, order) && (bin || !order);
        if (!bin && !order) return LLVQ_EUNSUPPORTED;
        if (bin) bin_smem(ctx, max_nq, smem, ext, acc_floats);
    }
    if (smem > kSmemLimit) return LLVQ_EUNSUPPORTED;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return LLVQ_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    const FastArgs fa = fast_args(ctx, ext);
    const unsigned g = (unsigned)ctx->sm_count;
    const bool bf16 = y_dtype == LLVQ_BF16;
#define LLVQ_LAUNCH_MULTI_T(K, BYTES, ...)                                                                                                      \
    do {                                                                                                                                        \
        if (!set_smem<K>(ctx, BYTES)) return LLVQ_ECUDA;                                                                                        \
        if (launch_pdl(K, g, (unsigned)kSortThreads, BYTES, st, fa, __VA_ARGS__, ctx->d_scratch, ctx->d_counters) != cudaSuccess) return LLVQ_ECUDA; \
    } while (0)
#define LLVQ_LAUNCH_MULTI(K, BYTES, ...)                                                                                    \
    do {                                                                                                                    \
        if (trees) { if (bf16) LLVQ_LAUNCH_MULTI_T((K<true, true>), BYTES, __VA_ARGS__); else LLVQ_LAUNCH_MULTI_T((K<false, true>), BYTES, __VA_ARGS__); } \
        else { if (bf16) LLVQ_LAUNCH_MULTI_T((K<true, false>), BYTES, __VA_ARGS__); else LLVQ_LAUNCH_MULTI_T((K<false, false>), BYTES, __VA_ARGS__); } \
    } while (0)
    if (sorted && n_mats >= 2) {
        // the kernel without a barrier between the matrices, when every CTA's share of every matrix is one segment and
        // one pass and three sets of (x, row sums) fit beside the tables
        int64_t max_groups = 0;
        bool one_pass = true;
        for (int i = 0; i < n_mats; ++i) {
            // a CTA's share is at most ceil(U / g) units, hence at most that many + nq - 2 units' worth of row groups, cut at both ends
            const Split& sp = mm.m[i].sp;
            const int64_t most = sp.each + (sp.rest ? 1 : 0), nq = sp.per_row;
            one_pass = one_pass && most <= kSortSegUnits;
            max_groups = std::max(max_groups, (most + nq - 2) / nq + 1);
        }
        const int xs_words = (int)(max_nq * 48), acc_rows = (int)(max_groups * kGemvGroupRows);
        uint32_t shift = 4;                              // copies of every row sum: up to sixteen (one warp alone sums them up), at least four
        auto ov_bytes = [&] {
            return fa.image_bytes + 16 + (size_t)kOverlapSets * ((size_t)xs_words + ((size_t)acc_rows << shift)) * 4 + kOverlapSets * sizeof(OverlapSet);
        };
        while (shift > 2 && ov_bytes() > kSmemLimit) --shift;
        const size_t smem_ov = ov_bytes();
        if (one_pass && max_groups <= kGemvGroupsPerPass && smem_ov <= kSmemLimit) {
            LLVQ_LAUNCH_MULTI(gemv_sorted_overlap_kernel, smem_ov, mm, xs_words, acc_rows, shift);
            return launch_status();
        }
    }
    if (sorted) { if (bf16) LLVQ_LAUNCH_MULTI_T(gemv_sorted_multi_kernel<true>, smem, mm, acc_floats); else LLVQ_LAUNCH_MULTI_T(gemv_sorted_multi_kernel<false>, smem, mm, acc_floats); }
    else if (bin) LLVQ_LAUNCH_MULTI(gemv_bin_multi_kernel, smem, ctx->d_sort_rank, mm, acc_floats);
    else LLVQ_LAUNCH_MULTI(gemv_order_multi_kernel, smem, oa, mm, (uint32_t)max_nq);
#undef LLVQ_LAUNCH_MULTI
#undef LLVQ_LAUNCH_MULTI_T
    return launch_status();
}

int llvq_gemv_multi(const llvq_ctx* ctx, const llvq_gemv_desc* descs, int n_mats, int y_dtype, void* stream)
{
    return gemv_multi_common(ctx, descs, n_mats, y_dtype, false, stream);
}

int llvq_gemv_sorted_multi(const llvq_ctx* ctx, const llvq_gemv_desc* descs, int n_mats, int y_dtype, void* stream)
{
    return gemv_multi_common(ctx, descs, n_mats, y_dtype, true, stream);
}

int llvq_gemv_rowshard(const llvq_ctx* ctx, const void* d_idx, const uint16_t* d_gain_f16, int64_t n_rows, int64_t k_in,
                       const uint16_t* d_x_bf16, void* const* d_y_all, int n_dest, int own_slot, int64_t row0, int y_dtype,
                       uint32_t* const* d_flag_words, uint32_t epoch, void* stream)
{
    YOut yo;
    if (int e = shard_yout(ctx, d_y_all, n_dest, own_slot, row0, y_dtype, d_flag_words, epoch, &yo)) return e;
    if (n_rows == 0) return signal_only(ctx, yo, stream);
    if (int e = check_common(ctx, d_idx)) return e;
    if (!d_gain_f16) return LLVQ_EINVAL;
    if (!aligned(d_gain_f16, 2)) return LLVQ_EALIGN;
    if (k_in == 0) {                                   // y = 0 by copies, no kernel to raise the flags
        if (int e = gemv_common(ctx, d_idx, d_gain_f16, nullptr, n_rows, k_in, d_x_bf16, yo, y_dtype, stream)) return e;
        return signal_only(ctx, yo, stream);
    }
    return gemv_common(ctx, d_idx, d_gain_f16, nullptr, n_rows, k_in, d_x_bf16, yo, y_dtype, stream);
}

int llvq_gemv_sorted_rowshard(const llvq_ctx* ctx, const void* d_sorted, const uint16_t* d_gain_f16, int64_t n_rows, int64_t k_in,
                              const uint16_t* d_x_bf16, void* const* d_y_all, int n_dest, int own_slot, int64_t row0, int y_dtype,
                              uint32_t* const* d_flag_words, uint32_t epoch, void* stream)
{
    YOut yo;
    if (int e = shard_yout(ctx, d_y_all, n_dest, own_slot, row0, y_dtype, d_flag_words, epoch, &yo)) return e;
    if (n_rows == 0) return signal_only(ctx, yo, stream);
    if (int e = check_common(ctx, d_sorted)) return e;
    if (!d_gain_f16) return LLVQ_EINVAL;
    if (!aligned(d_gain_f16, 2)) return LLVQ_EALIGN;
    return gemv_sorted_common(ctx, d_sorted, d_gain_f16, nullptr, n_rows, k_in, d_x_bf16, yo, y_dtype, stream);
}

}  // extern "C"
