// The fused dequant + small-batch GEMM kernels (tcgen05, accumulator in tensor memory): the kernel with two thread
// groups on alternating stages, the kernels that make the sorted layouts, the pipeline kernel that consumes them (and stored streams of few
// classes), and the kernel whose two teams order a stored stream of many classes.  Included by gemm.cu inside its unnamed
// namespace, after kernels_common.cuh, order.cuh and gemv_kernels.cuh (shard_arrive).
#pragma once

// ===========================================================================
// llvq_gemm_small_batch: Y[b][i] = sum_k X[b][k] W[i][k] on the tensor cores.
// A work item is a tile of 128 output rows x a range of K stages (96 columns = 4 blocks of 24 per row).
// Per stage every thread of a 512-thread group dequantizes one block into the group's shared-memory A tile
// (bf16, K-major core-matrix layout), the matching slice of X goes into its B tile, and one thread issues
// six tcgen05 MMAs (M = 128, N = padded batch, K = 16) into the group's accumulator in tensor memory.
// The two groups of a CTA take alternate stages, so two stages are in flight.
// Split-K partial sums are added into a zero-initialised binary32 scratch [npad][n_out]; the last item
// of a row tile converts it to bf16 and clears it again.
// ===========================================================================
constexpr int kGemmThreads = 1024;
constexpr int kGemmGroupThreads = 512;
constexpr int kStageBlocks = 4;                       // column blocks per stage
constexpr int kStageK = kStageBlocks * 24;            // 96
constexpr uint32_t kTmemCols = 128;

struct GemmArgs {
    int64_t n_out, k_in, bpr;
    int batch, npad;
    int nstages, split;        // gemm_kernel: 96-column stages and pieces of K
    Split sp;                  // the kernels on domains: which CTA works on which
    uint32_t gain_row;         // bytes of gains per row of blocks (below 2^32: k_in <= kMaxMapColumns)
    const uint16_t* x;
    uint16_t* y;               // Y [batch][y_ld] bf16, at the first row of this launch's rows
    int64_t y_ld;
    const YOut* shard;         // row-sharded launch: the peers' copies and flags (device memory), else null
    float* scratch;            // [npad][scratch_ld] binary32, all zero on entry and on exit
    int64_t scratch_ld;        // row tiles * 128
    uint32_t* counters;        // [row tiles], zero on entry and on exit
    int y_f32;                 // Y holds binary32 instead of bf16 (the batch-1 product behind llvq_gemv_sorted of the 72-bit code)
};

__global__ void put_shard_kernel(YOut yo, YOut* dst)
{
    if (threadIdx.x == 0) *dst = yo;
}

// One element of Y; a row-sharded launch also writes it into the peers' copies (their description sits in device
// memory so that the ordinary launch's parameters stay as small as they were).
template <bool kShard>
__device__ __forceinline__ void gemm_store(const GemmArgs& ga, int n, int64_t orow, float v)
{
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    const int64_t at = (int64_t)n * ga.y_ld + orow;
    if (!kShard && ga.y_f32) { reinterpret_cast<float*>(ga.y)[at] = v; return; }
    reinterpret_cast<__nv_bfloat16*>(ga.y)[at] = h;
    if (kShard) {
        const int np = ga.shard->n_peer;
        for (int p = 0; p < np; ++p) reinterpret_cast<__nv_bfloat16*>(ga.shard->peer[p])[at] = h;
    }
}

// Carries a finished accumulator of row tile rt out, a quarter of its rows and 16 of its columns per warp (a warp reaches the rows 32 (warp & 3) on): into the
// scratch where CTAs share the tile, else to Y.  second = the accumulator 64 columns on belongs to the same tile.  With four warps taking all columns one
// after the other, and the shared tile then read, converted and cleared value by value, a tile's end grew with the batch: sorted, shells 2..13, batch 64,
// 512 x 1024 17.2 -> 12.8 us, 4096 x 4096 39.8 -> 31.6, 8192 x 8192 87.6 -> 79.5; batch 16 30.3 -> 30.1 and 77.0 -> 76.8.
template <bool kShard>
__device__ __forceinline__ void carry_out(const GemmArgs& ga, uint32_t tmem, bool second, bool shared_tile, uint32_t rt, int warp, int lane)
{
    const int c0 = (warp >> 2) * 16;
    const uint32_t from = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
    const int64_t orow = (int64_t)rt * kGemmRows + (warp & 3) * 32 + lane;
    float v[16];
    tmem_ld16(from, v);
    if (second) {
        float v1[16];
        tmem_ld16(from + 64u, v1);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] += v1[i];
    }
    if (orow < ga.n_out) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int n = c0 + i;
            if (n < ga.batch) {
                if (!shared_tile) gemm_store<kShard>(ga, n, orow, v[i]);
                else atomicAdd(ga.scratch + (int64_t)n * ga.scratch_ld + orow, v[i]);
            }
        }
    }
}

// Y of row tile rt from the scratch, which is left at zero; all threads of the CTA that arrived last.  Four of a thread's values are asked for together (all
// eight of a batch of 64 in one go cost the main loop registers: batch 16 1 to 4 % slower).
template <bool kShard>
__device__ __forceinline__ void convert_tile(const GemmArgs& ga, uint32_t rt)
{
    static_assert(kGemmThreads % kGemmRows == 0, "a thread has one row of the tile");
    constexpr int kAhead = 4, kStep = kGemmThreads / kGemmRows;
    const int64_t orow = (int64_t)rt * kGemmRows + threadIdx.x % kGemmRows;
    if (orow >= ga.n_out) return;
    float* at = ga.scratch + (int64_t)(threadIdx.x / kGemmRows) * ga.scratch_ld + orow;
    const int64_t step = (int64_t)kStep * ga.scratch_ld;
#pragma unroll 1
    for (int n = (int)(threadIdx.x / kGemmRows); n < ga.batch; n += kAhead * kStep, at += kAhead * step) {
        float v[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) v[j] = n + j * kStep < ga.batch ? __ldcg(at + j * step) : 0.f;
#pragma unroll
        for (int j = 0; j < kAhead; ++j)
            if (n + j * kStep < ga.batch) {
                gemm_store<kShard>(ga, n + j * kStep, orow, v[j]);
                __stcg(at + j * step, 0.f);
            }
    }
}

// Gain of the block in row r of a row tile and column block cb.  A tile may hold more than 2^32 blocks.
__device__ __forceinline__ const uint16_t* gain_at(const GemmArgs& ga, const uint16_t* gain_tile, uint32_t r, uint32_t cb)
{
    return reinterpret_cast<const uint16_t*>(reinterpret_cast<const uint8_t*>(gain_tile + cb) + (uint64_t)r * ga.gain_row);
}

__device__ __forceinline__ void group_barrier(int group)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kGemmGroupThreads) : "memory");
}

template <bool kSg = false, bool kShard = false>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_kernel(FastArgs fa, const uint32_t* __restrict__ stream, const uint16_t* __restrict__ gain, SgArgs sg, GemmArgs ga)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t img_bytes = fa.image_bytes;
    uint64_t* bar_img = reinterpret_cast<uint64_t*>(smem + img_bytes);
    uint64_t* bar_free = bar_img + 1;                                     // [2]: the MMAs reading group h's buffers are done
    uint64_t* bar_done = bar_img + 3;                                     // [2]: group h's accumulator of this item is complete
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_img + 5);
    uint32_t* last_flag = tmem_slot + 1;
    const uint32_t a_off = (img_bytes + 64 + 1023) & ~1023u;
    uint8_t* a_buf = smem + a_off;                                        // [2 groups] x 24576
    uint8_t* b_buf = a_buf + 2 * kGemmRows * kStageK * 2;                  // [2 groups] x npad * 192
    const uint32_t b_stage = (uint32_t)ga.npad * kStageK * 2;

    pdl_launch_dependents();
    const bool image_ok = fast_load_image(smem, fa.image, fa.image_bytes, bar_img, fa.flags);
    pdl_wait();                                        // also when the image did not arrive: the dependents of this launch rely on it
    if (!image_ok) {
        if (kShard) shard_arrive(*ga.shard);           // the peers must not wait for this rank
        return;
    }
    const FastSmem T = fast_view(smem, fa.L);
    // Two groups of 512 threads fill alternate stages, each into its own buffers and its own accumulator
    // (TMEM columns [64 h, 64 h + npad)); the epilogue adds the two accumulators.
    const int group = threadIdx.x / kGemmGroupThreads, gtid = threadIdx.x % kGemmGroupThreads;
    const int gwarp = gtid >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        mbar_init(&bar_free[0], 1); mbar_init(&bar_free[1], 1); mbar_init(&bar_done[0], 1); mbar_init(&bar_done[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t idesc = instr_desc_bf16_m128((uint32_t)ga.npad);
    uint8_t* const a_mine = a_buf + group * (kGemmRows * kStageK * 2);
    uint8_t* const b_mine = b_buf + group * b_stage;

    const int64_t row_tiles = (ga.n_out + kGemmRows - 1) / kGemmRows;
    const int64_t items = row_tiles * ga.split;
    uint32_t uses = 0;                                  // stages this group has filled so far
    uint32_t done[2] = {0, 0};                          // completed accumulations per group
    bool timeout = false;
    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const int64_t rt = item / ga.split;
        const int f = (int)(item % ga.split);
        const int s_begin = (int)((int64_t)f * ga.nstages / ga.split), s_end = (int)((int64_t)(f + 1) * ga.nstages / ga.split);
        const int64_t row = (int64_t)rt * kGemmRows + gwarp * 8 + (lane & 7);
        for (int s = s_begin + group; s < s_end; s += 2, ++uses) {
            // ---- A: dequantize one block of 24 weights
            const int64_t cb = (int64_t)s * kStageBlocks + (lane >> 3);
            const bool in = row < ga.n_out && cb < ga.bpr;
            const uint64_t b = in ? (uint64_t)(row * ga.bpr + cb) : 0ull;
            uint32_t w[12];
            const RawBlock<false> raw = request_block<false>(stream, kSg ? nullptr : gain, fa.dc.W + (kSg ? sg.bits : 0), b, in);
            if constexpr (kSg) block_pairs_sg(fa, T, raw.field, sg, row, in, w);
            else block_pairs<false>(fa, T, raw, in, w);
            // the MMAs of this group's previous stage read its buffers: wait for them only now, with the block already unranked
            if (uses > 0 && !mbar_wait(&bar_free[group], (uses - 1u) & 1u)) timeout = true;
            uint8_t* a_dst = a_mine + gwarp * 128 + (lane & 7) * 16;
#pragma unroll
            for (int j = 0; j < 3; ++j)
                *reinterpret_cast<uint4*>(a_dst + (3 * (lane >> 3) + j) * 2048) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            // ---- B: the slice of X, 16-byte chunks (8 values along K)
            for (int i = gtid; i < ga.npad * (kStageK / 8); i += kGemmGroupThreads) {
                const int kc = i / ga.npad, n = i % ga.npad;
                const int64_t k = (int64_t)s * kStageK + kc * 8;
                uint4 v = make_uint4(0, 0, 0, 0);
                if (n < ga.batch && k < ga.k_in) v = __ldg(reinterpret_cast<const uint4*>(ga.x + (int64_t)n * ga.k_in + k));
                *reinterpret_cast<uint4*>(b_mine + (uint32_t)kc * ga.npad * 16 + n * 16) = v;
            }
            fence_async_smem();
            group_barrier(group);
            if (gtid == 0) {
                tc_fence_after();
                const uint32_t a_addr = smem_u32(a_mine), b_addr = smem_u32(b_mine);
#pragma unroll
                for (int j = 0; j < kStageK / 16; ++j)
                    umma_bf16(tmem + 64u * group, smem_desc(a_addr + j * 4096, 2048, 128),
                              smem_desc(b_addr + j * 2 * ga.npad * 16, ga.npad * 16, 128), idesc, (s > s_begin + group || j > 0) ? 1u : 0u);
                umma_commit(&bar_free[group]);
                if (s + 2 >= s_end) umma_commit(&bar_done[group]);
            }
        }
        // ---- epilogue: accumulators -> scratch (split-K) or Y
        const bool has0 = s_end > s_begin, has1 = s_end > s_begin + 1;
        if (has0 && (warp >> 2) * 16 < ga.npad) {
            if (!mbar_wait(&bar_done[0], done[0] & 1u)) timeout = true;
            if (has1 && !mbar_wait(&bar_done[1], done[1] & 1u)) timeout = true;
            tc_fence_after();
            carry_out<kShard>(ga, tmem, has1, ga.split > 1, (uint32_t)rt, warp, lane);
            tc_fence_before();
        }
        done[0] += has0; done[1] += has1;
        if (ga.split > 1) {
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) *last_flag = (atomicAdd(ga.counters + rt, 1u) == (uint32_t)ga.split - 1u);
            __syncthreads();
            if (*last_flag) {
                __threadfence();
                convert_tile<kShard>(ga, (uint32_t)rt);
                if (threadIdx.x == 0) ga.counters[rt] = 0u;
            }
        }
        __syncthreads();
    }
    if (timeout) atomicOr(fa.flags, 1u);
    if (kShard) {
        __threadfence_system();                           // this thread's stores to the peers' copies, before the CTA counts itself in
        shard_arrive(*ga.shard);
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

// ===========================================================================
// Sorted layout for the small-batch GEMM (llvq_sort_blocks_gemm / llvq_gemm_small_batch_sorted).
// A domain is 128 rows x 8 column blocks (1024 blocks, two 96-column MMA stages); the stream holds the domains
// row tile major, each domain's blocks ordered like the GEMV's sorted layout (decoder form, unranking steps,
// class), one 64-bit entry per block: the stored index unchanged (48 bits) + position in the domain (row * 8 +
// column block, 10 bits, stored in the high 16).  gemm_pipe_kernel unranks them, writing the bf16 weights straight to
// their place in the K-major A tiles.
// ===========================================================================
constexpr int kDomBlocks = 8;                          // column blocks per domain
constexpr int kDomEntries = kGemmRows * kDomBlocks;    // 1024
constexpr int kDomStages = 2;                          // 96-column MMA stages per domain
// The slice of X that goes with a domain, 192 columns x the padded batch: three panels of 64 columns, each one TMA box with the
// 128-byte swizzle (rows and columns outside X come as zeros).  One thread asks for them; copied by a warp, 16 bytes per lane and
// row, the slices took 85 of the 212 passes per chunk through the load / store pipe that bounds the kernel at batch 64
// (28672 x 8192: 308 -> 250 us).
constexpr int kXPanels = kDomBlocks * 24 / 64;

__device__ __forceinline__ void request_x(uint32_t dst, const CUtensorMap* map, int domain, int npad, uint64_t* bar)
{
    mbar_expect(bar, (uint32_t)(kXPanels * npad * 128));
#pragma unroll
    for (int i = 0; i < kXPanels; ++i) tma_load_2d(dst + (uint32_t)(i * npad * 128), map, domain * (kDomBlocks * 24) + i * 64, 0, bar);
}

// The 12 MMAs of a domain: A tile at a_addr (two 96-column stages), X slice at b_addr; fresh = the accumulator starts at zero.
__device__ __forceinline__ void domain_mmas(uint32_t tmem, uint32_t a_addr, uint32_t b_addr, int npad, uint32_t idesc, bool fresh)
{
#pragma unroll
    for (int t = 0; t < kDomBlocks * 24 / 16; ++t)
        umma_bf16(tmem, smem_desc(a_addr + (uint32_t)t * 4096u, 2048, 128), smem_desc_sw128(b_addr + (uint32_t)((t >> 2) * npad * 128 + (t & 3) * 32)), idesc,
                  !fresh || t > 0 ? 1u : 0u);
}

__global__ void __launch_bounds__(kDomEntries, 1)
sort_blocks_gemm_kernel(FastArgs fa, const uint32_t* __restrict__ stream, const uint16_t* __restrict__ sort_rank, int gain_bits, int64_t n_out,
                        int64_t bpr, int64_t ndomains, unsigned long long* __restrict__ out)
{
    FAST_PROLOGUE();
    __shared__ uint32_t hist[1024], cursor[1024];
    const int64_t nd = (bpr + kDomBlocks - 1) / kDomBlocks;
    for (int64_t dom = blockIdx.x; dom < ndomains; dom += gridDim.x) {
        hist[threadIdx.x] = 0; cursor[threadIdx.x] = 0;
        __syncthreads();
        const int64_t rt = dom / nd, d = dom - rt * nd;
        const int i = threadIdx.x;
        const int64_t row = (int64_t)rt * kGemmRows + (i >> 3), cb = d * kDomBlocks + (i & 7);
        unsigned long long field = kSortIndexMask;
        uint32_t key = 1023u;
        if (row < n_out && cb < bpr) {
            const uint64_t f = load_field(stream, (uint64_t)(row * bpr + cb), (int)fa.L.W + gain_bits);   // shape index | gain index << W
            const uint64_t I = f & ((1ull << fa.L.W) - 1ull);
            if (I < fa.n_points) {
                uint64_t local;
                field = f;
                key = __ldg(sort_rank + fast_find_class(T, I, local));
            } else {
                atomicAdd(fa.bad_index, 1ull);
            }
        }
        atomicAdd(&hist[key], 1u);
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t run = 0;
            for (int k = 0; k < 1024; ++k) { const uint32_t c = hist[k]; hist[k] = run; run += c; }
        }
        __syncthreads();
        const uint32_t slot = hist[key] + atomicAdd(&cursor[key], 1u);
        out[dom * kDomEntries + slot] = field | (unsigned long long)i << 48;
        __syncthreads();
    }
}

// The same layout for codes whose class tables live in global memory (72-bit indices): 96-bit entries (three 32-bit
// words).  An index is stored as its two digits in the mixed radix of the class table (App. A step 2, taken when the
// layout is made): words 0-1 = the class-local index I - offset[class] (class sizes fit 63 bits; bit 63 set marks "no
// block": ragged edge or index out of range), word 2 = class (17 bits) | position in the domain << 17 (10 bits).  The
// kernel then needs neither the bucket table nor the 128-bit offsets, and the class record can be requested as soon as
// the entry is there.  The blocks of a domain are ordered by the shape of their unranking: parity (odd first), number of
// steps (most first), which of the steps take at most three slots, steps of the first group; the lanes of a warp then
// run the same trip counts over similar slot counts and mostly agree on the cheap form of a step.
// Inside the kernels an entry travels as two 64-bit words: x = the class-local index (stored stream: index bits 0..63),
// y = class << 8 | position << 32, bit 63 = no block (stored stream: index bits 64..71 in the low byte).
constexpr unsigned long long kBigNoBlock = 1ull << 63;
constexpr int kBigEntryWords = 3;
constexpr int kBigClassBits = 17;

// Entry `at` of a sorted stream of 96-bit entries, in the two-word form the kernels use.
__device__ __forceinline__ ulonglong2 load_big_entry(const void* sorted, int64_t at)
{
    const uint32_t* p = static_cast<const uint32_t*>(sorted) + at * kBigEntryWords;
    const uint32_t w0 = __ldg(p), w1 = __ldg(p + 1), w2 = __ldg(p + 2);
    const unsigned long long pos = w2 >> kBigClassBits, cls = w2 & ((1u << kBigClassBits) - 1u);
    return make_ulonglong2((unsigned long long)(w1 & 0x7fffffffu) << 32 | w0,
                           ((unsigned long long)(w1 >> 31) << 63) | cls << 8 | pos << 32);
}

__global__ void __launch_bounds__(kDomEntries, 1)
sort_blocks_gemm_big_kernel(FastArgs fa, const uint32_t* __restrict__ stream, int64_t n_out, int64_t bpr, int64_t ndomains,
                            uint32_t* __restrict__ out)
{
    __shared__ uint32_t keys[kDomEntries];
    __shared__ unsigned long long ex[kDomEntries], ey[kDomEntries];
    const int64_t nd = (bpr + kDomBlocks - 1) / kDomBlocks;
    const int i = threadIdx.x;
    for (int64_t dom = blockIdx.x; dom < ndomains; dom += gridDim.x) {
        const int64_t rt = dom / nd, d = dom - rt * nd;
        const int64_t row = (int64_t)rt * kGemmRows + (i >> 3), cb = d * kDomBlocks + (i & 7);
        unsigned long long x = kBigNoBlock, y = (unsigned long long)i << kBigClassBits;   // words 0-1 and word 2 of an entry
        uint32_t key = 0x7ffffc00u | (uint32_t)i;                   // no block: after everything else
        if (row < n_out && cb < bpr) {
            uint64_t lo, hi;
            load_index(stream, (uint64_t)(row * bpr + cb), fa.dc.W, lo, hi);
            if (hi < fa.dc.n_hi || (hi == fa.dc.n_hi && lo < fa.dc.n_lo)) {
                uint64_t local;
                const uint32_t cls = (uint32_t)big_find_class(fa.dc, lo, hi, local);
                const uint32_t* rec = reinterpret_cast<const uint32_t*>(fa.dc.big + cls);
                const uint32_t h = __ldg(rec), small_k = __ldg(rec + 6) >> 24;
                const uint32_t nlev = h >> 28, nlev1 = (h >> 24) & 7u, parity = (h >> 16) & 1u;
                x = local;
                y = (unsigned long long)cls | (unsigned long long)i << kBigClassBits;
                // odd classes first (their steps choose among up to 24 slots, the even classes' among at most 16), then by steps
                key = (1u - parity) << 24 | (7u - min(nlev, 7u)) << 21 | (small_k & 0x7fu) << 14 | nlev1 << 11 | (uint32_t)i;
            } else {
                atomicAdd(fa.bad_index, 1ull);
            }
        }
        keys[i] = key; ex[i] = x; ey[i] = y;
        __syncthreads();
        for (int k = 2; k <= kDomEntries; k <<= 1)                   // bitonic sort of the 1024 keys
            for (int j = k >> 1; j > 0; j >>= 1) {
                const int o = i ^ j;
                if (o > i) {
                    const uint32_t a = keys[i], b = keys[o];
                    if ((a > b) == ((i & k) == 0)) { keys[i] = b; keys[o] = a; }
                }
                __syncthreads();
            }
        const uint32_t src = keys[i] & 1023u;
        uint32_t* o = out + (dom * kDomEntries + i) * kBigEntryWords;
        o[0] = (uint32_t)ex[src]; o[1] = (uint32_t)(ex[src] >> 32); o[2] = (uint32_t)ey[src];
        __syncthreads();
    }
}

// The product from a sorted layout: two buffer sets alternate between consecutive domains (two A tiles; two X slices, or one where
// shared memory has room for no more) and nobody waits for the whole CTA.  Warps 1..31 unrank: the chunks of 32 sorted entries of a
// row tile are handed out by a ticket counter (ticket t = chunk t % 32 of the tile's domain t / 32, so from expensive
// to cheap inside a domain), a warp always holding its next ticket with that chunk's entries already requested.
// It unranks the chunk, waits (rarely) until the MMAs that read this buffer two domains ago are done, writes its
// part of A and arrives on the buffer's "full" barrier.  The first thread of warp 0 asks for the X slice of the next domain, whose
// bytes that barrier counts too, and issues the MMAs of a domain as soon as it completes.
// kStored: the same structure on the stored stream (`sorted` then points at it): a chunk is 32 consecutive blocks of the
// domain in natural order (4 rows x 8 column blocks), unranked by the any-class decoder.
template <bool kBig, bool kSg = false, bool kShard = false, bool kStored = false>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_pipe_kernel(FastArgs fa, const unsigned long long* __restrict__ sorted, const uint16_t* __restrict__ gain, SgArgs sg, GemmArgs ga,
                 int b_double, const __grid_constant__ CUtensorMap xmap)
{
    static_assert(!(kStored && kBig), "the stored streams of codes with tables in global memory go to gemm_team_kernel");
    extern __shared__ __align__(1024) uint8_t smem_1k[];
    uint8_t* const smem = smem_1k;
    const uint32_t img_bytes = fa.image_bytes;
    uint64_t* bar_img = reinterpret_cast<uint64_t*>(smem + img_bytes);
    uint64_t* bar_full = bar_img + 1;                                     // [2] 32 chunks of A and the X slice are in the buffer
    uint64_t* bar_free = bar_img + 3;                                     // [2] the MMAs reading the buffer are done
    uint64_t* bar_done = bar_img + 5;                                     // the accumulator of this row tile is complete
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_img + 6);
    uint32_t* last_flag = tmem_slot + 1;
    uint32_t* ticket = tmem_slot + 2;                                     // next chunk ticket of the row tile in progress
    const uint32_t a_off = (img_bytes + 64 + 1023) & ~1023u;
    constexpr uint32_t kAStage = kGemmRows * kStageK * 2;                  // 24576
    uint8_t* a_buf = smem + a_off;                                        // [2 buffers][2 stages] x 24576
    const uint32_t b_stage = (uint32_t)ga.npad * kStageK * 2;
    uint8_t* b_buf = a_buf + 2u * kDomStages * kAStage;                    // [2 buffers, or 1][2 stages] x npad * 192
    constexpr uint32_t kWorkers = kGemmThreads / 32 - 1;                   // 31 unranking warps

    pdl_launch_dependents();
    const bool image_ok = fast_load_image(smem, fa.image, fa.image_bytes, bar_img, fa.flags);
    pdl_wait();                                        // also when the image did not arrive: the dependents of this launch rely on it
    if (!image_ok) {
        if (kShard) shard_arrive(*ga.shard);           // the peers must not wait for this rank
        return;
    }
    const FastSmem T = fast_view(smem, fa.L);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        mbar_init(bar_full, 33); mbar_init(bar_full + 1, 33);             // 32 chunks + the X slice
        mbar_init(bar_free, 1); mbar_init(bar_free + 1, 1); mbar_init(bar_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t idesc = instr_desc_bf16_m128((uint32_t)ga.npad);
    const uint32_t nd = ga.sp.per_row;                                     // domains per row tile
    const uint32_t dom_begin = split_begin(ga.sp, blockIdx.x), dom_end = split_begin(ga.sp, blockIdx.x + 1u);
    uint32_t g_base = 0, done = 0;                                         // domains this CTA has finished (domain g uses buffer g & 1 for the (g >> 1)-th time)
    bool timeout = false;
    const ulonglong2 no_entry = make_ulonglong2(kSortIndexMask, kBigNoBlock);
    auto arrive_full = [&](uint32_t b) {
        fence_async_smem();
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar_full + b)) : "memory");
    };

    for (uint32_t rt = split_row(ga.sp, dom_begin); rt * nd < dom_end; ++rt) {
        const uint32_t tile0 = rt * nd, tile1 = tile0 + nd;
        const int d_begin = (int)(max(dom_begin, tile0) - tile0), d_end = (int)(min(dom_end, tile1) - tile0);
        // CTAs that share this row tile
        const uint32_t parts = dom_begin <= tile0 && tile1 <= dom_end ? 1u : split_owner(ga.sp, tile1 - 1u) - split_owner(ga.sp, tile0) + 1u;
        const uint32_t n_dom = (uint32_t)(d_end - d_begin), n_tickets = n_dom * 32u;
        if (threadIdx.x == 0) *ticket = kWorkers;                          // the first tickets are the workers' own numbers
        __syncthreads();
        if (warp == 0) {
            // ---- X slices and MMAs
            // With two X buffers a domain's slice may be written once the MMAs of two domains ago are done; with one (wide batches: no
            // room for two), only after the previous domain's
            if (lane == 0) {
                auto stage_b = [&](uint32_t j) {
                    const uint32_t gd = g_base + j, b = gd & 1u, bx = b_double ? b : 0u;
                    if (b_double) { if (gd >= 2u && !mbar_wait(bar_free + b, ((gd >> 1) - 1u) & 1u)) timeout = true; }
                    else if (gd >= 1u && !mbar_wait(bar_free + ((gd - 1u) & 1u), ((gd - 1u) >> 1) & 1u)) timeout = true;
                    request_x(smem_u32(b_buf) + bx * kDomStages * b_stage, &xmap, d_begin + (int)j, ga.npad, bar_full + b);
                };
                if (n_dom > 0) stage_b(0);
                for (uint32_t j = 0; j < n_dom; ++j) {
                    if (b_double && j + 1 < n_dom) stage_b(j + 1);
                    const uint32_t gd = g_base + j, b = gd & 1u, bx = b_double ? b : 0u;
                    if (!mbar_wait_copies(bar_full + b, (gd >> 1) & 1u)) timeout = true;
                    tc_fence_after();
                    domain_mmas(tmem, smem_u32(a_buf) + b * kDomStages * kAStage, smem_u32(b_buf) + bx * kDomStages * b_stage, ga.npad, idesc, j == 0);
                    umma_commit(bar_free + b);
                    if (j + 1 == n_dom) umma_commit(bar_done);
                    if (!b_double && j + 1 < n_dom) stage_b(j + 1);
                }
            }
            __syncwarp();
        } else {
            // ---- A: unrank chunks until the tile's tickets are gone
            const int64_t entry0 = (int64_t)(tile0 + d_begin) * kDomEntries + lane;
            const uint32_t bpr = (uint32_t)ga.bpr;
            const uint16_t* gain_tile = gain + (int64_t)rt * kGemmRows * ga.bpr;
            auto entry_of = [&](uint32_t t) {
                if (t >= n_tickets) return no_entry;
                if (kBig) return load_big_entry(sorted, entry0 + t * 32u);     // chunk t % 32 of domain t / 32
                return make_ulonglong2(__ldg(sorted + entry0 + t * 32u), 0ull);
            };
            // stored stream: the words of this lane's block of chunk t (position t % 32 * 32 + lane of domain t / 32)
            const int wbits = fa.dc.W + (kSg ? sg.bits : 0);
            auto stored_of = [&](uint32_t t, bool& in) {
                const uint32_t pos = (t & 31u) * 32u + lane, c0 = ((uint32_t)d_begin + (t >> 5)) * kDomBlocks + (pos & 7u), r0 = pos >> 3;
                in = t < n_tickets && (int64_t)rt * kGemmRows + r0 < ga.n_out && c0 < bpr;
                return request_field<kBig>(reinterpret_cast<const uint32_t*>(sorted), ((uint64_t)rt * kGemmRows + r0) * bpr + c0, wbits, in);
            };
            uint32_t tk = (uint32_t)warp - 1u;
            ulonglong2 e = no_entry;
            RawField<kBig> raw{};
            bool in = false;
            if (kStored) raw = stored_of(tk, in); else e = entry_of(tk);
            // sorted 96-bit entries name their class: its record is requested while the previous chunk is still being expanded
            uint4 rec0 = make_uint4(0u, 0u, 0u, 0u), rec1 = rec0;
            if (kBig) big_load_record(fa.dc, (int)((uint32_t)(e.y >> 8) & 0xffffffu), !(e.y >> 63), rec0, rec1);
            while (tk < n_tickets) {
                uint32_t tk_next = 0;
                if (lane == 0) tk_next = atomicAdd(ticket, 1u);
                tk_next = __shfl_sync(kFullMask, tk_next, 0);
                ulonglong2 e_next = no_entry;                               // requested a chunk ahead (it comes from DRAM)
                RawField<kBig> raw_next{};
                bool in_next = false;
                if (kStored) raw_next = stored_of(tk_next, in_next); else e_next = entry_of(tk_next);
                if (kStored) {                                              // a field may take all 64 bits: its position is known from the ticket
                    uint64_t lo, none;
                    field_value(raw, wbits, lo, none);
                    e.x = lo;
                }
                const uint32_t j = tk >> 5, gd = g_base + j, b = gd & 1u;
                const int d = d_begin + (int)j;
                const uint64_t field = kStored ? (uint64_t)e.x : e.x & kSortIndexMask;
                const uint64_t I = kSg ? field & ((1ull << fa.L.W) - 1ull) : field;     // shape-gain form: gain index above the shape index
                const uint32_t pos = kBig ? (uint32_t)(e.y >> 32) & 1023u : kStored ? (tk & 31u) * 32u + lane : (uint32_t)(e.x >> 48);
                const bool there = kStored ? in : field != kSortIndexMask;
                const bool valid = kBig ? !(e.y >> 63) : (there && I < fa.n_points);
                const uint32_t r = pos >> 3, c = pos & 7u;
                uint16_t gbits = 0;
                if (!kSg && valid) gbits = ldg_u16_here(gain_at(ga, gain_tile, r, (uint32_t)d * kDomBlocks + c));
                float gn = 0.f;                                               // the gain is converted once the block is unranked
                uint32_t w[12];
                if (kBig) {
                    DecodedBig dec{};
                    big_decode_record(T, rec0, rec1, valid ? e.x : 0ull, valid, kFullMask, dec);
                    // the next chunk's entries were requested a whole chunk ago: they are here, and their records have the
                    // rest of this iteration to arrive
                    big_load_record(fa.dc, (int)((uint32_t)(e_next.y >> 8) & 0xffffffu), !(e_next.y >> 63), rec0, rec1);
                    gn = gain_to_float(gbits);
                    expand_bf16(dec.d, gn, w);
                    patch_id8_bf16(dec, gn, w);
                } else {
                    Decoded dec{};
                    uint32_t cls;
                    if (kStored) {
                        if (there && !valid) atomicAdd(fa.bad_index, 1ull);
                        uint64_t local = 0;
                        cls = valid ? fast_find_class(T, I, local) : 0u;
                        fast_decode_local<-1>(T, cls, local, valid, kFullMask, dec);
                    } else {
                        cls = decode_sorted_entry(fa, T, I, valid, dec);
                    }
                    if (!kSg) gn = gain_to_float(gbits);
                    if (kSg && valid) {
                        const float scale = sg.row_scale ? __ldg(sg.row_scale + (int64_t)rt * kGemmRows + r) : 1.f;
                        gn = __fmul_rn(__fmul_rn(scale, __ldg(sg.codebook + (uint32_t)(field >> fa.L.W))),
                                       __uint_as_float(T.desc[cls * kFastDescStride + kFastDescRnorm]));
                    }
                    expand_bf16(dec, gn, w);
                }
                // the MMAs of two domains ago read this buffer: wait for them only now, with the chunk already unranked
                if (gd >= 2u && !mbar_wait(bar_free + b, ((gd >> 1) - 1u) & 1u)) timeout = true;
                uint8_t* a_dst = a_buf + (b * kDomStages + (c >> 2)) * kAStage + (r >> 3) * 128u + (r & 7u) * 16u + 3u * (c & 3u) * 2048u;
#pragma unroll
                for (int jj = 0; jj < 3; ++jj)
                    *reinterpret_cast<uint4*>(a_dst + jj * 2048) = make_uint4(w[4 * jj], w[4 * jj + 1], w[4 * jj + 2], w[4 * jj + 3]);
                arrive_full(b);
                tk = tk_next;
                if (kStored) { raw = raw_next; in = in_next; use_field_from_here(raw); }
                else {
                    e = e_next;
                    use_from_here(e.x);
                    if (kBig) use_from_here(e.y);
                }
            }
        }
        g_base += n_dom;
        const bool has = d_end > d_begin;
        // ---- epilogue: accumulator -> scratch (split-K) or Y
        if (has && (warp >> 2) * 16 < ga.npad) {
            if (!mbar_wait(bar_done, done & 1u)) timeout = true;
            tc_fence_after();
            carry_out<kShard>(ga, tmem, false, parts > 1u, rt, warp, lane);
            tc_fence_before();
        }
        done += has;
        if (parts > 1u) {
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) *last_flag = (atomicAdd(ga.counters + rt, 1u) == parts - 1u);
            __syncthreads();
            if (*last_flag) {
                __threadfence();
                convert_tile<kShard>(ga, (uint32_t)rt);
                if (threadIdx.x == 0) ga.counters[rt] = 0u;
            }
        }
        __syncthreads();
    }
    if (timeout) atomicOr(fa.flags, 1u);
    if (kShard) {
        __threadfence_system();                           // this thread's stores to the peers' copies, before the CTA counts itself in
        shard_arrive(*ga.shard);
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

// The product on the stored stream of codes with many classes: two teams of 16 warps take the domains of a row tile in turn.  A team orders
// its domain's 1024 blocks (order.cuh; the entries lie in its own A buffer, which its previous MMAs have left by then), every
// warp takes two chunks of them into registers, unranks them, writes its part of A, and the team's first thread issues the MMAs
// into the team's own accumulator.  The teams meet only at the end of a row tile: while one orders, which leaves most issue slots
// empty, the other unranks.  x_double: an X buffer per team, asked for ahead; else one that the teams use in turn (wide batches).
constexpr int kGemmTeams = 2;
constexpr int kGemmTeamThreads = kGemmThreads / kGemmTeams;

template <bool kBig, bool kSg = false, bool kShard = false>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_team_kernel(FastArgs fa, const uint32_t* __restrict__ stream, OrderArgs oa, const uint16_t* __restrict__ gain, SgArgs sg, GemmArgs ga, int x_double,
                 const __grid_constant__ CUtensorMap xmap)
{
    extern __shared__ __align__(1024) uint8_t smem_1k[];
    uint8_t* const smem = smem_1k;
    const uint32_t img_bytes = fa.image_bytes;
    uint64_t* bar_img = reinterpret_cast<uint64_t*>(smem + img_bytes);
    uint64_t* bar_free = bar_img + 1;                                     // [2] the MMAs of the team's last domain are done (its A buffer and X are free)
    uint64_t* bar_x = bar_img + 3;                                        // [2] the X slice of the team's domain has arrived
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_img + 5);
    uint32_t* last_flag = tmem_slot + 1;
    const uint32_t a_off = (img_bytes + 64 + 1023) & ~1023u;
    constexpr uint32_t kASet = kDomStages * kGemmRows * kStageK * 2;       // 49152
    uint8_t* a_buf = smem + a_off;                                        // [2 teams] x 49152
    const uint32_t x_set = (uint32_t)ga.npad * kDomStages * kStageK * 2;
    uint8_t* b_buf = a_buf + kGemmTeams * kASet;                          // [2 teams, or 1]
    uint32_t* hists = reinterpret_cast<uint32_t*>(b_buf + (x_double ? 2u : 1u) * x_set);      // [2 teams][2][words]

    pdl_launch_dependents();
    const bool image_ok = fast_load_image(smem, fa.image, fa.image_bytes, bar_img, fa.flags);
    pdl_wait();                                        // also when the image did not arrive: the dependents of this launch rely on it
    if (!image_ok) {
        if (kShard) shard_arrive(*ga.shard);           // the peers must not wait for this rank
        return;
    }
    const FastSmem T = fast_view(smem, fa.L);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, team = (int)threadIdx.x / kGemmTeamThreads;
    const uint32_t tid = threadIdx.x % kGemmTeamThreads, twarp = tid >> 5;
    for (uint32_t i = threadIdx.x; i < kGemmTeams * 2 * oa.words; i += kGemmThreads) hists[i] = 0u;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) { mbar_init(bar_free + i, 1); mbar_init(bar_x + i, 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t idesc = instr_desc_bf16_m128((uint32_t)ga.npad);
    uint8_t* const a_mine = a_buf + (uint32_t)team * kASet;
    uint8_t* const x_mine = b_buf + (x_double ? (uint32_t)team * x_set : 0u);
    unsigned long long* const ent = reinterpret_cast<unsigned long long*>(a_mine);
    uint32_t* const ent2 = reinterpret_cast<uint32_t*>(ent + kOrderBlocks);
    const uint32_t nd = ga.sp.per_row, bpr = (uint32_t)ga.bpr;
    const uint32_t dom_begin = split_begin(ga.sp, blockIdx.x), dom_end = split_begin(ga.sp, blockIdx.x + 1u);
    uint32_t mine = 0, base[2] = {0, 0};               // domains this team has done; domains either team had done before this row tile
    bool timeout = false;

    for (uint32_t rt = split_row(ga.sp, dom_begin); rt * nd < dom_end; ++rt) {
        const uint32_t tile0 = rt * nd, tile1 = tile0 + nd;
        const uint32_t d_begin = max(dom_begin, tile0) - tile0, d_end = min(dom_end, tile1) - tile0;
        // CTAs that share this row tile
        const uint32_t parts = dom_begin <= tile0 && tile1 <= dom_end ? 1u : split_owner(ga.sp, tile1 - 1u) - split_owner(ga.sp, tile0) + 1u;
        const uint16_t* gain_tile = gain + (int64_t)rt * kGemmRows * ga.bpr;
        bool fresh = true;
        for (uint32_t d = d_begin + (uint32_t)team; d < d_end; d += kGemmTeams, ++mine) {
            // ---- order
            OrderSpot<uint64_t> o;
            o.b0 = 0;
            o.row = rt * kGemmRows + (tid >> 3);
            o.b = (uint64_t)o.row * bpr + (d * kDomBlocks + (tid & 7u));
            o.pos = tid;
            o.there = d * kDomBlocks + (tid & 7u) < bpr;
            order_piece<kBig, kSg, kGemmTeamThreads>(fa, T, sg, oa, stream, hists + ((uint32_t)team * 2u + (mine & 1u)) * oa.words,
                                               hists + ((uint32_t)team * 2u + ((mine & 1u) ^ 1u)) * oa.words, ent, ent2, team, tid, o, (uint32_t)ga.n_out,
                                               (uint64_t)bpr * 64u, 64u, (uint32_t)kGemmTeamThreads, [&] {
                // the entries go over what the previous MMAs read
                if (mine > 0 && !mbar_wait(bar_free + team, (mine - 1u) & 1u)) timeout = true;
                if (x_double && tid == 0) request_x(smem_u32(x_mine), &xmap, (int)d, ga.npad, bar_x + team);
            });
            // ---- A: two chunks per warp, one from the expensive and one from the cheap end
            const unsigned long long e[2] = {ent[twarp * 32u + lane], ent[(31u - twarp) * 32u + lane]};
            uint32_t e2[2] = {0u, 0u};
            uint4 rec0, rec1;
            if (kBig) {
                e2[0] = ent2[twarp * 32u + lane]; e2[1] = ent2[(31u - twarp) * 32u + lane];
                big_load_record(fa.dc, (int)(e2[0] & 0x1ffffu), !(e2[0] >> 31), rec0, rec1);
            }
            team_barrier(team, kGemmTeamThreads);                         // all entries are in registers: A may overwrite them
            // one X buffer: it may be asked for once the MMAs of the tile's domain before this one (the other team's) are through with it;
            // looked at between the two chunks, waited for only when this domain's own MMAs are due
            const uint32_t i_tile = d - d_begin, before = team == 0 ? base[1] + (i_tile >> 1) - 1u : base[0] + (i_tile >> 1);
            bool asked = x_double != 0;
#pragma unroll 1
            for (int q = 0; q < 2; ++q) {
                if (q == 1 && !asked && tid == 0 && (i_tile == 0u || mbar_test(bar_free + (team ^ 1), before & 1u))) {
                    request_x(smem_u32(x_mine), &xmap, (int)d, ga.npad, bar_x + team);
                    asked = true;
                }
                OrderedBlock b{};
                if (!kBig) b = ordered_block<kSg>(fa, sg, oa, q == 0 ? e[0] : e[1]);
                else { const uint32_t y = q == 0 ? e2[0] : e2[1]; b.valid = !(y >> 31); b.pos = (y >> 17) & 1023u; }
                const uint32_t r = b.pos >> 3, c = b.pos & 7u;
                uint16_t gbits = 0;
                if (!kSg && b.valid) gbits = ldg_u16_here(kBig ? gain_at(ga, gain_tile, r, d * kDomBlocks + c) : gain_tile + (r * bpr + d * kDomBlocks + c));
                float gn = 0.f;                                           // the gain is converted once the block is unranked
                uint32_t w[12];
                if constexpr (kBig) {
                    DecodedBig dec{};
                    big_decode_record(T, rec0, rec1, b.valid ? (q == 0 ? e[0] : e[1]) : 0ull, b.valid, kFullMask, dec);
                    if (q == 0) big_load_record(fa.dc, (int)(e2[1] & 0x1ffffu), !(e2[1] >> 31), rec0, rec1);
                    gn = gain_to_float(gbits);
                    expand_bf16(dec.d, gn, w);
                    patch_id8_bf16(dec, gn, w);
                } else {
                    Decoded dec;
                    decode_known_class(T, b.valid ? b.cls : 0u, b.local, b.valid, dec);
                    if (!kSg) gn = gain_to_float(gbits);
                    if (kSg && b.valid) {
                        const float scale = sg.row_scale ? __ldg(sg.row_scale + (int64_t)rt * kGemmRows + r) : 1.f;
                        gn = __fmul_rn(__fmul_rn(scale, __ldg(sg.codebook + b.gain_index)), __uint_as_float(T.desc[b.cls * kFastDescStride + kFastDescRnorm]));
                    }
                    expand_bf16(dec, gn, w);
                }
                uint8_t* a_dst = a_mine + (c >> 2) * (kASet / 2) + (r >> 3) * 128u + (r & 7u) * 16u + 3u * (c & 3u) * 2048u;
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    *reinterpret_cast<uint4*>(a_dst + j * 2048) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            }
            fence_async_smem();
            team_barrier(team, kGemmTeamThreads);
            // ---- MMAs
            if (tid == 0) {
                if (!asked) {
                    if (i_tile > 0u && !mbar_wait(bar_free + (team ^ 1), before & 1u)) timeout = true;
                    request_x(smem_u32(x_mine), &xmap, (int)d, ga.npad, bar_x + team);
                }
                if (!mbar_wait_copies(bar_x + team, mine & 1u)) timeout = true;
                tc_fence_after();
                domain_mmas(tmem + 64u * (uint32_t)team, smem_u32(a_mine), smem_u32(x_mine), ga.npad, idesc, fresh);
                umma_commit(bar_free + team);
            }
            fresh = false;
        }
        const uint32_t n0 = (d_end - d_begin + 1u) / 2u, n1 = (d_end - d_begin) / 2u;
        // ---- epilogue: accumulators -> scratch (split-K) or Y
        __syncthreads();                                                  // both teams' MMAs of this tile are issued
        if (n0 > 0 && (warp >> 2) * 16 < ga.npad) {
            if (!mbar_wait(bar_free, (base[0] + n0 - 1u) & 1u)) timeout = true;
            if (n1 > 0 && !mbar_wait(bar_free + 1, (base[1] + n1 - 1u) & 1u)) timeout = true;
            tc_fence_after();
            carry_out<kShard>(ga, tmem, n1 > 0, parts > 1u, rt, warp, lane);
            tc_fence_before();
        }
        base[0] += n0; base[1] += n1;
        if (parts > 1u) {
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) *last_flag = (atomicAdd(ga.counters + rt, 1u) == parts - 1u);
            __syncthreads();
            if (*last_flag) {
                __threadfence();
                convert_tile<kShard>(ga, (uint32_t)rt);
                if (threadIdx.x == 0) ga.counters[rt] = 0u;
            }
        }
        __syncthreads();
    }
    if (timeout) atomicOr(fa.flags, 1u);
    if (kShard) {
        __threadfence_system();                           // this thread's stores to the peers' copies, before the CTA counts itself in
        shard_arrive(*ga.shard);
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}
