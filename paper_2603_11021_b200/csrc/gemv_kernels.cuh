// The fused dequant + GEMV kernels: the direct kernel (tensor-core reduction), the sorted layout (sort kernel and
// consumer) and the kernel that bins a segment's blocks by class itself.  Included by gemv.cu and gemm.cu inside their
// unnamed namespaces, after kernels_common.cuh.
#pragma once

// Fused dequant + GEMV.  The work is cut into units of 8 rows x 4 column blocks, numbered row group major, and
// every CTA takes an equal contiguous range of units.  In a unit lane (g, t) = (lane / 4, lane % 4) decodes the
// block (row g, column block 4q + t); its 12 packed bf16 pairs are the A fragments (rows 0..7; rows 8..15 are
// zero) of six m16n8k16 tensor-core MMAs whose B fragment carries the matching 4 x 24 activations (the same in
// all 8 columns), accumulating in binary32.  Row sums are collected in shared memory; a row group that is
// split between CTAs is finished through a zero-kept global scratch and an arrival counter.

__device__ __forceinline__ void mma_bf16_16816(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

template <bool kOutBf16, bool kShard>
__device__ __forceinline__ void store_y(const YOut& yo, int64_t row, float v)
{
    if (kOutBf16) {
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        reinterpret_cast<__nv_bfloat16*>(yo.y)[row] = h;
        if (kShard) {                                     // the single-GPU instantiations carry none of this
#pragma unroll
            for (int p = 0; p < kMaxShardPeers; ++p)      // static indices: the struct stays in the parameter bank
                if (p < yo.n_peer) reinterpret_cast<__nv_bfloat16*>(yo.peer[p])[row] = h;
        }
    } else {
        reinterpret_cast<float*>(yo.y)[row] = v;
        if (kShard) {
#pragma unroll
            for (int p = 0; p < kMaxShardPeers; ++p)
                if (p < yo.n_peer) reinterpret_cast<float*>(yo.peer[p])[row] = v;
        }
    }
}

// Stages x for a GEMV CTA: xs[cb * 12 + j] = the bf16 pair (x[24 cb + 2j], x[24 cb + 2j + 1]), zero beyond k_in; `words`
// = 12 x the number of column blocks staged.  16-byte loads where x allows them.
__device__ __forceinline__ void stage_x(uint32_t* xs, const uint16_t* __restrict__ x, int64_t k_in, uint32_t words, uint32_t tid, uint32_t nthreads)
{
    if ((reinterpret_cast<uintptr_t>(x) & 15) == 0) {
        const uint32_t full = (uint32_t)(k_in / 8);                          // whole groups of 8 elements
        for (uint32_t v = tid; v < words / 4; v += nthreads) {
            uint4 q = make_uint4(0u, 0u, 0u, 0u);
            if (v < full) q = __ldg(reinterpret_cast<const uint4*>(x) + v);
            else {
                uint32_t t[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t e = 8 * v + 2 * j;
                    const uint32_t lo = e < k_in ? __ldg(x + e) : 0u, hi = e + 1 < k_in ? __ldg(x + e + 1) : 0u;
                    t[j] = lo | hi << 16;
                }
                q = make_uint4(t[0], t[1], t[2], t[3]);
            }
            reinterpret_cast<uint4*>(xs)[v] = q;
        }
        return;
    }
    for (uint32_t i = tid; i < words; i += nthreads) {
        const uint32_t e = 2 * i;
        const uint32_t lo = e < k_in ? __ldg(x + e) : 0u, hi = e + 1 < k_in ? __ldg(x + e + 1) : 0u;
        xs[i] = lo | hi << 16;
    }
}

// End of a pass of a GEMV CTA over row groups rg0..rg1 (8 rows each; the CTA owns units [u_begin, u_end) of sp):
// row_sums(i), called by a whole warp, gives lanes 0..7 the CTA's sums for rows i..i + 7 of the pass.  One warp per row group, lanes
// 0..7 its rows, no CTA-wide barrier inside.  A group the CTA covers completely is final.  A group it shares with
// neighbouring CTAs goes through the scratch row in global memory: add, make the add visible, count the arrival;
// whoever arrives last reads the total, writes y and leaves scratch and counter zero for the next launch (groups shared
// by exactly two CTAs take a shorter way, below).
// The caller puts a __syncthreads() before (sums complete) and after (sums may be cleared) the call.
// slot0 (a multiple of 8) = first scratch row / pair slot of this matrix when one launch works on several matrices.
// kTrees = the trees of slots are part of the kernel, for launches some of whose groups are shared by three CTAs or more: where none is, their code
// alone cost the kernels on stored streams 0.1 to 0.2 us (72-bit code, 1400 x 1000 9.38 us without, 9.59 with it; shells 3, 2048 x 1024 5.00 and
// 5.09) and gemv_sorted_overlap_kernel nine registers.  gemv_sorted_kernel always has it: it comes out faster with it (1400 x 1000 6.53 us, 6.64 without;
// shape-gain 4096 x 11008 38.5 and 39.2).
template <bool kOutBf16, bool kShard, bool kTrees, typename RowSums>
__device__ __forceinline__ void finish_pass(const YOut& yo, const Split& sp, uint32_t rg0, uint32_t rg1, uint32_t u_begin, uint32_t u_end,
                                            int64_t n_out, float* __restrict__ scratch, uint32_t* __restrict__ counters, RowSums row_sums,
                                            int64_t slot0 = 0, int warp_of = -1, int nwarps_of = 0)
{
    // by default the warps of the CTA share the row groups; warp_of / nwarps_of let a subset of the warps (one warp) do it
    const uint32_t warp = warp_of >= 0 ? (uint32_t)warp_of : threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t nwarps = warp_of >= 0 ? (uint32_t)nwarps_of : blockDim.x >> 5;
    for (uint32_t rg = rg0 + warp; rg <= rg1; rg += nwarps) {
        const uint32_t first = rg * sp.per_row, next = first + sp.per_row;
        const bool whole = u_begin <= first && next <= u_end;
        const int64_t row = (int64_t)rg * kGemvGroupRows + lane;
        const bool mine = lane < kGemvGroupRows && row < n_out;
        const float part = row_sums((rg - rg0) * kGemvGroupRows);
        if (whole) {
            if (mine) {
                store_y<kOutBf16, kShard>(yo, row, part);
            }
            continue;
        }
        const uint32_t parts = split_owner(sp, next - 1u) - split_owner(sp, first) + 1u;
        if (parts == 2u) {
            // two CTAs share the group (the usual case): one compare-and-swap on a 64-bit slot carries both the sum
            // and the arrival.  Whoever finds the slot empty leaves (its sum, 1) there; the other gets that back from
            // its failed swap, adds its own sum, stores y and empties the slot.  One round trip each, no fence.
            if (mine) {
                unsigned long long* slot = reinterpret_cast<unsigned long long*>(scratch + kPairSlotOffset) + slot0 + row;
                const unsigned long long seen = atomicCAS(slot, 0ull, (unsigned long long)__float_as_uint(part) | 1ull << 32);
                if (seen != 0ull) {
                    store_y<kOutBf16, kShard>(yo, row, __fadd_rn(__uint_as_float((uint32_t)seen), part));
                    __stcg(slot, 0ull);
                }
            }
            continue;
        }
        if (kTrees && parts <= 8u && sp.trees) {
            // three to eight CTAs (short rows of small matrices): a tree of such slots, seven per row, over the CTAs in order.  Who finds a
            // slot empty is done; the other goes on to the next one with both sums.  Up to three round trips for the last to arrive, where
            // the way below takes a fence on either side of the counter and a read behind it (sorted 512 x 1024:
            // 8.0 -> 7.1 us, 1024 x 4096 10.6 -> 9.6)
            if (mine) {
                unsigned long long* const tree = reinterpret_cast<unsigned long long*>(scratch + kPairSlotOffset) + (kPairSlots - 8 * (slot0 + row + 1));
                float sum = part;
                uint32_t at = blockIdx.x - split_owner(sp, first), width = parts, node = 0;
                bool last = true;
                while (width > 1u) {
                    if ((at ^ 1u) < width) {
                        unsigned long long* const slot = tree + node + (at >> 1);
                        const unsigned long long seen = atomicCAS(slot, 0ull, (unsigned long long)__float_as_uint(sum) | 1ull << 32);
                        if (seen == 0ull) { last = false; break; }
                        __stcg(slot, 0ull);
                        sum = at & 1u ? __fadd_rn(__uint_as_float((uint32_t)seen), sum) : __fadd_rn(sum, __uint_as_float((uint32_t)seen));
                    }
                    at >>= 1; width = (width + 1u) >> 1; node += node ? 2u : 4u;
                }
                if (last) store_y<kOutBf16, kShard>(yo, row, sum);
            }
            continue;
        }
        if (mine) atomicAdd(scratch + slot0 + row, part);
        __threadfence();                               // every lane's add is performed before ...
        __syncwarp();
        uint32_t is_last = 0u;
        if (lane == 0) {
            __threadfence();                           // ... lane 0 counts the arrival
            is_last = atomicAdd(counters + slot0 / kGemvGroupRows + rg, 1u) == parts - 1u;
        }
        is_last = __shfl_sync(kFullMask, is_last, 0);
        if (is_last) {
            __threadfence();
            if (mine) {
                store_y<kOutBf16, kShard>(yo, row, __ldcg(scratch + slot0 + row));
                __stcg(scratch + slot0 + row, 0.f);
            }
            if (lane == 0) counters[slot0 / kGemvGroupRows + rg] = 0u;
        }
    }
}

// Last step of a row-sharded GEMV CTA (all threads call it, after their last store to y): counts the CTA in; the CTA
// that completes the grid raises the epoch in every peer's flag word.  The remote stores of y are plain stores; the block
// barrier below orders them before the system-scope fence of the thread that counts the CTA in, which makes them visible,
// cumulatively, before the flag (the usual barrier + fence + flag pattern: no fence per storing lane).
__device__ __forceinline__ void shard_arrive(const YOut& yo)
{
    if (yo.n_flag == 0) return;
    __syncthreads();
    if (threadIdx.x != 0) return;
    __threadfence_system();
    if (atomicAdd(yo.done, 1u) != gridDim.x - 1u) return;
    atomicExch(yo.done, 0u);
    // one system-scope fence releases everything before it for all the flag words: the stores themselves are relaxed (a
    // release store per word would pay the fence once per peer: measured 2 us each)
    __threadfence_system();
#pragma unroll
    for (int p = 0; p < kMaxShardPeers; ++p)
        if (p < yo.n_flag) asm volatile("st.relaxed.sys.global.u32 [%0], %1;" ::"l"(yo.flag[p]), "r"(yo.epoch) : "memory");
}

// sum_j w_j x_j over 12 packed bf16 pairs with binary32 accumulation: fma.rn.f32.bf16 takes the bf16 halves as they are
// (products of two bf16 values are exact in binary32, so this is the chain of 24 binary32 FMAs without the unpacking).
__device__ __forceinline__ float dot24_bf16(const uint32_t w[12], const uint32_t x[12])
{
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int j = 0; j < 12; ++j) {
        asm("{\n .reg .b16 wl, wh, xl, xh;\n mov.b32 {wl, wh}, %2;\n mov.b32 {xl, xh}, %3;\n"
            " fma.rn.f32.bf16 %0, wl, xl, %0;\n fma.rn.f32.bf16 %1, wh, xh, %1;\n}"
            : "+f"(s0), "+f"(s1) : "r"(w[j]), "r"(x[j]));
    }
    return s0 + s1;
}

// Row sums of a pass in shared memory: acc[row << shift | lane & mask], as many copies of every row (a power of two, up to one per
// lane) as kSortAccFloats floats hold.  An addition of floats in shared memory is a compare-and-swap loop that goes round once for
// every lane of the warp that meets the same address: 32 blocks of a warp fall into some 80 rows, and with one copy per warp
// parity instead of per lane that took 18 instructions and 15 passes over the banks per addition (stored 11008 x 4096: 56.4 -> 53.7 us).
constexpr uint32_t kSortAccFloats = 4 * kGemvGroupsPerPass * kGemvGroupRows;

__device__ __forceinline__ uint32_t acc_shift(uint32_t rows, uint32_t floats)
{
    uint32_t c = 5;
    while (c > 0 && (rows << c) > floats) --c;
    return c;
}

// Sums over the copies of rows first..first + 7, in lanes 0..7; the whole warp calls this.
__device__ __forceinline__ float acc_row_sums(const float* acc, uint32_t first, uint32_t shift)
{
    const uint32_t lane = threadIdx.x & 31u;
    float v = 0.f;
    for (uint32_t c = lane & 3u; c < (1u << shift); c += 4) v += acc[(first + (lane >> 2)) << shift | c];      // four lanes per row
    v += __shfl_xor_sync(kFullMask, v, 1);
    v += __shfl_xor_sync(kFullMask, v, 2);
    return __shfl_sync(kFullMask, v, (lane & 7u) * 4u);
}

// kFma: each lane forms its own dot product with binary32 FMAs instead (what small matrices of codes with many classes take, whose larger ones go to
// gemv_bin_kernel: the tensor core's sums are 1.3 to 1.6 times as far from exact ones, 1.0e-7 against 6.4e-8 of the 2-norm at 1000 x 1000).
template <bool kBig, bool kOutBf16, bool kSg, bool kShard, bool kFma, bool kTrees>
__global__ void __launch_bounds__(kGemvThreads, 1)
gemv_fast_kernel(FastArgs fa, const uint32_t* __restrict__ stream, const uint16_t* __restrict__ gain, SgArgs sg, Split sp, uint32_t groups_per_pass,
                 int64_t n_out, int64_t k_in, int64_t bpr, const uint16_t* __restrict__ x, YOut yo,
                 float* __restrict__ scratch, uint32_t* __restrict__ counters)
{
    FAST_PROLOGUE(if (kShard) shard_arrive(yo));
    const uint32_t nq = sp.per_row;                                 // units along K
    uint32_t* xs = reinterpret_cast<uint32_t*>(staging);            // [nq * 4][12] packed bf16 pairs of x
    float* acc = reinterpret_cast<float*>(xs + nq * 48);            // [groups_per_pass][8]
    stage_x(xs, x, k_in, nq * 48, threadIdx.x, blockDim.x);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const uint32_t kWarps = blockDim.x >> 5;
    const uint32_t u_begin = split_begin(sp, blockIdx.x), u_end = split_begin(sp, blockIdx.x + 1u);      // at least one unit
    const uint32_t rg_first = split_row(sp, u_begin), rg_last = split_row(sp, u_end - 1u);
    for (uint32_t rg0 = rg_first; rg0 <= rg_last; rg0 += groups_per_pass) {
        const uint32_t rg1 = min(rg0 + groups_per_pass - 1u, rg_last);
        const uint32_t shift = kFma ? acc_shift((rg1 - rg0 + 1u) * kGemvGroupRows, kSortAccFloats) : 0u;      // copies of the row sums
        for (uint32_t i = threadIdx.x; i < (kFma ? (rg1 - rg0 + 1u) * kGemvGroupRows << shift : groups_per_pass * kGemvGroupRows); i += blockDim.x) acc[i] = 0.f;
        __syncthreads();
        const uint32_t p_begin = max(u_begin, rg0 * nq), p_end = min(u_end, (rg1 + 1u) * nq);
        uint32_t kq, rg = split_row(sp, p_begin + (uint32_t)warp, kq);      // walked along with u: no division per unit
        // a block's words are requested while the one before it is unranked
        const int wbits = fa.dc.W + (kSg ? sg.bits : 0);
        int64_t cb = 0, row = 0;
        bool in = false;
        auto request = [&](uint32_t u) {
            while (kq >= nq) { kq -= nq; ++rg; }
            cb = kq * 4 + t; row = (int64_t)rg * kGemvGroupRows + g;
            in = u < p_end && row < n_out && cb < bpr;
            return request_block<kBig>(stream, kSg ? nullptr : gain, wbits, (uint64_t)(row * bpr + cb), in);
        };
        uint32_t u = p_begin + (uint32_t)warp;
        RawBlock<kBig> raw_next = request(u);
        while (u < p_end) {
            RawBlock<kBig> raw = raw_next;
            use_field_from_here(raw.field);
            const bool in_now = in;
            const uint32_t cb_now = (uint32_t)cb, rg_now = rg;
            u += kWarps; kq += kWarps;
            raw_next = request(u);
            uint32_t w[12];
            [[maybe_unused]] bool valid;
            if constexpr (kSg) valid = block_pairs_sg(fa, T, raw.field, sg, (int64_t)rg_now * kGemvGroupRows + g, in_now, w);
            else valid = block_pairs<kBig>(fa, T, raw, in_now, w);
            const uint4* xb = reinterpret_cast<const uint4*>(xs + cb_now * 12u);
            const uint4 x0 = xb[0], x1 = xb[1], x2 = xb[2];
            const uint32_t xv[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            if constexpr (kFma) {
                // a block whose index is out of range adds nothing, whatever its gain and its slice of x are (as in gemv_bin_kernel)
                atomicAdd(&acc[((rg_now - rg0) * kGemvGroupRows + g) << shift | ((uint32_t)(warp * 4 + t) & ((1u << shift) - 1u))], valid ? dot24_bf16(w, xv) : 0.f);
            } else {
#pragma unroll
                for (int q = 0; q < 6; ++q)
                    mma_bf16_16816(c, w[2 * q], 0u, w[2 * q + 1], 0u, xv[2 * q], xv[2 * q + 1]);
            }
            if (!kFma && t == 0) atomicAdd(&acc[(rg_now - rg0) * kGemvGroupRows + g], c[0]);
        }
        __syncthreads();
        // row groups this CTA covers completely are final; the (at most two) split ones go through the scratch
        finish_pass<kOutBf16, kShard, kTrees>(yo, sp, rg0, rg1, u_begin, u_end, n_out, scratch, counters, [&](uint32_t r) {
            if constexpr (kFma) return acc_row_sums(acc, r, shift);
            return lane < kGemvGroupRows ? acc[r + lane] : 0.f;
        });
        __syncthreads();                                   // the sums are read above: the next pass may clear them only now
    }
    if (kShard) shard_arrive(yo);
}

constexpr uint32_t kKindEven = 0u, kKindOdd = 1u, kKindOther = 2u, kKindNull = 3u;   // decoder form a class needs

// ===========================================================================
// Sorted layout for the fused GEMV (llvq_sort_blocks / llvq_gemv_sorted).
// The work is cut exactly as in gemv_fast_kernel: units of 8 rows x 4 column blocks, row group major, an equal
// contiguous range of units per CTA (for the CTA count of this device).  Inside a CTA's range the units are taken
// in segments of up to kSortSegUnits units, and the blocks of a segment are stored sorted by the decoder form
// their class needs (odd / even with Golay weight 8, 12, 16 / other) and its number of unranking steps (most
// expensive first), so that the 32 lanes of a warp run the same form with the same trip count.  Each block is a
// 64-bit entry: the stored index I unchanged in the low 48 bits, its position in the segment (unit * 32 + lane)
// in the high 16 bits; entries that do not exist (ragged edges) or are out of range carry I = 2^48 - 1.
// All of App. A runs in the GEMV kernel.  A warp takes 32 consecutive entries, each lane unranks its block and
// multiplies it with its own slice of x (binary32 FMAs), and adds the partial row sum to the CTA's row sums.
// ===========================================================================
constexpr int kSortSegUnits = 2048;                  // 65536 blocks
constexpr int kSortThreads = 1024;
constexpr unsigned long long kSortIndexMask = (1ull << 48) - 1ull;

// Calls f(tu0, tu1, rg0, rg1, first, last) for every segment [tu0, tu1) of CTA `cta` in order; rg0..rg1 = row
// groups of the pass the segment belongs to (a pass covers at most kGemvGroupsPerPass row groups); first / last =
// the segment opens / closes its pass.
template <typename F>
__device__ __forceinline__ void for_each_sorted_segment(const Split& sp, uint32_t cta, F f, uint32_t seg_units = kSortSegUnits)
{
    const uint32_t nq = sp.per_row, u_begin = split_begin(sp, cta), u_end = split_begin(sp, cta + 1u);
    if (u_begin >= u_end) return;
    const uint32_t rg_first = split_row(sp, u_begin), rg_last = split_row(sp, u_end - 1u);
    for (uint32_t rg0 = rg_first; rg0 <= rg_last; rg0 += kGemvGroupsPerPass) {
        const uint32_t rg1 = min(rg0 + kGemvGroupsPerPass - 1u, rg_last);
        const uint32_t p_begin = max(u_begin, rg0 * nq), p_end = min(u_end, (rg1 + 1u) * nq);
        for (uint32_t tu0 = p_begin; tu0 < p_end; tu0 += seg_units)
            f(tu0, min(tu0 + seg_units, p_end), rg0, rg1, tu0 == p_begin, tu0 + seg_units >= p_end);
    }
}

__global__ void __launch_bounds__(kSortThreads, 1)
sort_blocks_kernel(FastArgs fa, const uint32_t* __restrict__ stream, const uint16_t* __restrict__ sort_rank, int gain_bits, Split sp, int64_t n_out,
                   int64_t bpr, unsigned long long* __restrict__ out)
{
    FAST_PROLOGUE();
    __shared__ uint32_t hist[1024], cursor[1024];                  // one bin per class, in sort order; bin 1023 = no block
    const uint32_t nq = sp.per_row;
    for_each_sorted_segment(sp, blockIdx.x, [&](uint32_t tu0, uint32_t tu1, uint32_t, uint32_t, bool, bool) {
        const int entries = (int)(tu1 - tu0) * 32;
        hist[threadIdx.x] = 0; cursor[threadIdx.x] = 0;
        __syncthreads();
        // key and field of entry i of the segment; count = the first pass (out-of-range fields are counted once)
        auto entry_of = [&](int i, bool count, unsigned long long& field) {
            const int lane = i & 31;
            uint32_t kq;
            const uint32_t rg = split_row(sp, tu0 + (uint32_t)(i >> 5), kq);
            const int64_t row = (int64_t)rg * kGemvGroupRows + (lane >> 2), cb = kq * 4 + (lane & 3);
            field = kSortIndexMask;
            if (row >= n_out || cb >= bpr) return 1023u;
            const uint64_t f = load_field(stream, (uint64_t)(row * bpr + cb), (int)fa.L.W + gain_bits);   // shape index | gain index << W
            const uint64_t I = f & ((1ull << fa.L.W) - 1ull);
            if (I >= fa.n_points) { if (count) atomicAdd(fa.bad_index, 1ull); return 1023u; }
            uint64_t local;
            field = f;
            return (uint32_t)__ldg(sort_rank + fast_find_class(T, I, local));
        };
        for (int i = threadIdx.x; i < entries; i += kSortThreads) {
            unsigned long long field;
            atomicAdd(&hist[entry_of(i, true, field)], 1u);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t run = 0;
            for (int k = 0; k < 1024; ++k) { const uint32_t c = hist[k]; hist[k] = run; run += c; }
        }
        __syncthreads();
        // the entries are visited column block by column block (all rows of one, then the next): the blocks of a bin then come out
        // roughly ordered by column block, and the eight lanes that read x together read few different slices of it
        const uint32_t rg_a = split_row(sp, tu0), nrg = split_row(sp, tu1 - 1u) - rg_a + 1u;
        for (uint32_t e = threadIdx.x; e < nq * nrg * 32u; e += kSortThreads) {
            const uint32_t cb = e / (nrg * 8u), row = e - cb * (nrg * 8u);
            const uint32_t u = (rg_a + (row >> 3)) * nq + (cb >> 2);
            if (u < tu0 || u >= tu1) continue;
            const int i = (int)(u - tu0) * 32 + (int)((row & 7u) * 4u + (cb & 3u));
            unsigned long long field;
            const uint32_t key = entry_of(i, false, field);
            const uint32_t slot = hist[key] + atomicAdd(&cursor[key], 1u);
            out[(uint64_t)tu0 * 32 + slot] = field | (unsigned long long)i << 48;
        }
        __syncthreads();
    });
}

// App. A steps 2-4 for one entry of a sorted layout: class lookup, then the unranker form the class needs.  The
// lanes of a warp call this together; after sorting they almost always share the form (and the class).
__device__ __forceinline__ void decode_known_class(const FastSmem& T, uint32_t cls, uint64_t local, bool valid, Decoded& r)
{
    const uint32_t kind = !valid ? kKindNull : (T.desc[cls * kFastDescStride] >> 22) & 3u;     // the form is part of the descriptor's flags
    r.p0 = r.p1 = r.p2 = r.neg = r.vals_lo = r.vals_hi = 0u;
    // every form writes r only for its own lanes
    if (__any_sync(kFullMask, kind == kKindOdd)) {
        const bool mine = kind == kKindOdd;
        fast_decode_local<1>(T, mine ? cls : 0u, mine ? local : 0ull, mine, kFullMask, r);
    }
    if (__any_sync(kFullMask, kind == kKindEven)) {
        const bool mine = kind == kKindEven;
        fast_decode_local<0>(T, mine ? cls : 0u, mine ? local : 0ull, mine, kFullMask, r);
    }
    if (__any_sync(kFullMask, kind == kKindOther)) {
        const bool mine = kind == kKindOther;
        fast_decode_local<-1>(T, mine ? cls : 0u, mine ? local : 0ull, mine, kFullMask, r);
    }
}

__device__ __forceinline__ uint32_t decode_sorted_entry(const FastArgs& fa, const FastSmem& T, uint64_t I, bool valid, Decoded& r)
{
    uint64_t local = 0;
    const uint32_t cls = valid ? fast_find_class(T, I, local) : 0u;
    decode_known_class(T, cls, local, valid, r);
    return cls;
}

// One matrix of a launch that works through several matrices one after another (llvq_gemv_multi, llvq_gemv_sorted_multi):
// every CTA takes its share of each matrix in turn, so the table image, the launch and the ramp-up are paid once.
constexpr int kMaxMultiMats = 8;
struct GemvMat {
    const void* weights;        // stored stream or sorted entries
    const uint16_t* gain;
    const uint16_t* x;
    void* y;
    int64_t n_out, k_in;
    int64_t slot0;              // first scratch row / pair slot of this matrix (a multiple of 8)
    Split sp;
    int32_t bpr;                // column blocks per row
};
struct GemvMulti {
    GemvMat m[kMaxMultiMats];
    int n;
};

// Ask for the first chunk of every warp of this CTA in L2 (one request per 128-byte line).
__device__ __forceinline__ void prefetch_first_chunks(const unsigned long long* sorted, const Split& sp)
{
    const uint32_t ub = split_begin(sp, blockIdx.x), ue = split_begin(sp, blockIdx.x + 1u);
    if ((threadIdx.x & 15u) == 0u && ub + (threadIdx.x >> 5) < ue)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(sorted + (uint64_t)ub * 32 + threadIdx.x));
}

// The sorted-layout GEMV of one matrix by this CTA (all threads call it; shared memory behind `staging` is reused by the
// next call, which the caller separates with a block barrier).
template <bool kOutBf16, bool kSg, bool kShard>
__device__ __forceinline__ void gemv_sorted_body(const FastArgs& fa, const FastSmem& T, uint8_t* staging,
                                                 const unsigned long long* __restrict__ sorted, const uint16_t* __restrict__ gain, const SgArgs& sg,
                                                 const Split& sp, int64_t n_out, int64_t k_in, uint32_t bpr, const uint16_t* __restrict__ x,
                                                 const YOut& yo, float* __restrict__ scratch, uint32_t* __restrict__ counters, int64_t slot0,
                                                 uint32_t acc_floats)
{
    const uint32_t nq = sp.per_row;
    uint32_t* xs = reinterpret_cast<uint32_t*>(staging);            // [nq * 4][12] packed bf16 pairs of x
    float* acc = reinterpret_cast<float*>(xs + nq * 48);            // [acc_floats]
    uint32_t* next_chunk = reinterpret_cast<uint32_t*>(acc + acc_floats);
    stage_x(xs, x, k_in, nq * 48, threadIdx.x, blockDim.x);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t kWarps = blockDim.x >> 5;

    for_each_sorted_segment(sp, blockIdx.x, [&](uint32_t tu0, uint32_t tu1, uint32_t rg0, uint32_t rg1, bool first, bool last) {
        const uint32_t shift = acc_shift((rg1 - rg0 + 1u) * kGemvGroupRows, acc_floats);
        if (first)
            for (uint32_t i = threadIdx.x; i < (rg1 - rg0 + 1u) * kGemvGroupRows << shift; i += blockDim.x) acc[i] = 0.f;
        if (threadIdx.x == 0) *next_chunk = kWarps;
        __syncthreads();
        uint32_t kq_a;
        const uint32_t rg_off = split_row(sp, tu0, kq_a) - rg0;
        const uint32_t nchunks = tu1 - tu0;
        const unsigned long long* seg = sorted + (uint64_t)tu0 * 32 + lane;
        const uint16_t* gain_pass = gain + (int64_t)rg0 * kGemvGroupRows * bpr;
        uint32_t ch = (uint32_t)warp;
        unsigned long long e = ch < nchunks ? __ldg(seg + (uint64_t)ch * 32) : 0ull;
        while (ch < nchunks) {
            // chunks are handed out dynamically (their cost depends on the form); the next entry is fetched ahead
            uint32_t nxt = 0;
            if (lane == 0) nxt = atomicAdd(next_chunk, 1u);
            nxt = __shfl_sync(kFullMask, nxt, 0);
            const unsigned long long e_next = nxt < nchunks ? __ldg(seg + (uint64_t)nxt * 32) : 0ull;
            const uint64_t field = e & kSortIndexMask;
            const uint64_t I = kSg ? field & ((1ull << fa.L.W) - 1ull) : field;     // shape-gain form: gain index above the shape index
            const uint32_t pos = (uint32_t)(e >> 48);
            const bool valid = field != kSortIndexMask && I < fa.n_points;
            // where the block sits: unit = pos / 32 of the segment, (row, column block) = lane of the unit
            uint32_t kq;
            const uint32_t q = split_row(sp, kq_a + (pos >> 5), kq);
            const uint32_t rloc = (rg_off + q) * kGemvGroupRows + ((pos >> 2) & 7u);      // row inside the pass
            const uint32_t cb = kq * 4u + (pos & 3u);
            float gn = 0.f;
            uint16_t gbits = 0;
            if (!kSg && valid) gbits = ldg_u16_here(gain_pass + (rloc * bpr + cb));
            Decoded r;
            const uint32_t cls = decode_sorted_entry(fa, T, I, valid, r);
            if (!kSg) gn = gain_to_float(gbits);
            if (kSg && valid) {
                const float scale = sg.row_scale ? __ldg(sg.row_scale + (int64_t)rg0 * kGemvGroupRows + rloc) : 1.f;
                gn = __fmul_rn(__fmul_rn(scale, __ldg(sg.codebook + (uint32_t)(field >> fa.L.W))),
                               __uint_as_float(T.desc[cls * kFastDescStride + kFastDescRnorm]));
            }
            uint32_t w[12];
            expand_bf16(r, gn, w);
            const uint4* xb = reinterpret_cast<const uint4*>(xs + cb * 12u);
            const uint4 x0 = xb[0], x1 = xb[1], x2 = xb[2];
            const uint32_t xv[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
            const float dot = dot24_bf16(w, xv);
            if (valid) atomicAdd(&acc[rloc << shift | ((uint32_t)lane & ((1u << shift) - 1u))], dot);
            ch = nxt; e = e_next;
            use_from_here(e);
        }
        __syncthreads();
        if (!last) return;
        // end of the pass: row groups this CTA covers completely are final; the split ones go through the scratch
        auto row_sums = [&](uint32_t r) { return acc_row_sums(acc, r, shift); };
        const uint32_t ub = split_begin(sp, blockIdx.x), ue = split_begin(sp, blockIdx.x + 1u);     // recomputed here: not kept across the main loop
        finish_pass<kOutBf16, kShard, true>(yo, sp, rg0, rg1, ub, ue, n_out, scratch, counters, row_sums, slot0);
        __syncthreads();                                   // the sums are read above: the next pass may clear them only now
    });
}

template <bool kOutBf16, bool kSg, bool kShard>
__global__ void __launch_bounds__(kSortThreads, 1)
gemv_sorted_kernel(FastArgs fa, const unsigned long long* __restrict__ sorted, const uint16_t* __restrict__ gain, SgArgs sg,
                   Split sp, int64_t n_out, int64_t k_in, int64_t bpr, uint32_t acc_floats, const uint16_t* __restrict__ x, YOut yo,
                   float* __restrict__ scratch, uint32_t* __restrict__ counters)
{
    prefetch_first_chunks(sorted, sp);                  // while the table image is on its way
    FAST_PROLOGUE(if (kShard) shard_arrive(yo));
    gemv_sorted_body<kOutBf16, kSg, kShard>(fa, T, staging, sorted, gain, sg, sp, n_out, k_in, (uint32_t)bpr, x, yo, scratch, counters, 0, acc_floats);
    if (kShard) shard_arrive(yo);
}

// Several independent matrices in one launch (no output of one may be an input of another).
template <bool kOutBf16>
__global__ void __launch_bounds__(kSortThreads, 1)
gemv_sorted_multi_kernel(FastArgs fa, const __grid_constant__ GemvMulti mm, uint32_t acc_floats, float* __restrict__ scratch, uint32_t* __restrict__ counters)
{
    prefetch_first_chunks(static_cast<const unsigned long long*>(mm.m[0].weights), mm.m[0].sp);
    FAST_PROLOGUE();
    for (int i = 0; i < mm.n; ++i) {
        const GemvMat& M = mm.m[i];
        if (i + 1 < mm.n)
            prefetch_first_chunks(static_cast<const unsigned long long*>(mm.m[i + 1].weights), mm.m[i + 1].sp);
        YOut yo{};
        yo.y = M.y;
        gemv_sorted_body<kOutBf16, false, false>(fa, T, staging, static_cast<const unsigned long long*>(M.weights), M.gain, SgArgs{}, M.sp, M.n_out, M.k_in,
                                                 (uint32_t)M.bpr, M.x, yo, scratch, counters, M.slot0, acc_floats);
        __syncthreads();                                   // the next matrix restages x and clears the row sums
    }
}

// The same, without a block barrier between the matrices: a warp that finds no chunk of matrix i left goes on to matrix
// i + 1 while the others finish theirs, so the partly filled last round of chunks, the end of the pass and the staging of
// x of one matrix run under the next matrix's work.  Three sets of (x, row sums, chunk counter) rotate: the warp that
// completes matrix i (the last to run out of its chunks) ends the pass alone and then prepares set i % 3 for matrix
// i + 3.  Taken when every CTA's share of every matrix is one segment and one pass (checked on the host).
constexpr int kOverlapSets = 3;
constexpr uint32_t kOverlapSpins = 1u << 22;         // polls of a shared-memory flag before a warp gives up (never in a correct run)

struct OverlapSet {
    uint32_t next_chunk;
    uint32_t arrived;                                // warps that have run out of chunks of the set's matrix
    uint32_t ready;                                  // index + 1 of the matrix the set is prepared for
    uint32_t pad;
};

template <bool kOutBf16, bool kTrees>
__global__ void __launch_bounds__(kSortThreads, 1)
gemv_sorted_overlap_kernel(FastArgs fa, const __grid_constant__ GemvMulti mm, int xs_words, int acc_rows, uint32_t shift, float* __restrict__ scratch,
                           uint32_t* __restrict__ counters)
{
    prefetch_first_chunks(static_cast<const unsigned long long*>(mm.m[0].weights), mm.m[0].sp);
    FAST_PROLOGUE();
    // [kOverlapSets] x { x as packed pairs [xs_words] | row sums [acc_rows << shift] } | control words
    const int set_words = xs_words + (acc_rows << shift);
    uint32_t* sets = reinterpret_cast<uint32_t*>(staging);
    volatile OverlapSet* ctl = reinterpret_cast<volatile OverlapSet*>(sets + kOverlapSets * set_words);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t kWarps = blockDim.x >> 5;

    // prepare set i % kOverlapSets for matrix i with the calling threads (`nthreads` of them, numbered `tid`)
    auto prepare = [&](int i, int tid, int nthreads) {
        const GemvMat& M = mm.m[i];
        uint32_t* xs = sets + (i % kOverlapSets) * set_words;
        float* acc = reinterpret_cast<float*>(xs + xs_words);
        stage_x(xs, M.x, M.k_in, M.sp.per_row * 48u, (uint32_t)tid, (uint32_t)nthreads);
        for (int r = tid; r < acc_rows << shift >> 2; r += nthreads) reinterpret_cast<float4*>(acc)[r] = make_float4(0.f, 0.f, 0.f, 0.f);
    };

    if (threadIdx.x < kOverlapSets) { ctl[threadIdx.x].next_chunk = 0u; ctl[threadIdx.x].arrived = 0u; ctl[threadIdx.x].ready = 0u; }
    for (int i = 0; i < kOverlapSets && i < mm.n; ++i) prepare(i, (int)threadIdx.x, (int)blockDim.x);
    __syncthreads();
    if (threadIdx.x < kOverlapSets && (int)threadIdx.x < mm.n) ctl[threadIdx.x].ready = threadIdx.x + 1u;
    __syncthreads();

    for (int i = 0; i < mm.n; ++i) {
        const GemvMat& M = mm.m[i];
        const int set = i % kOverlapSets;
        const Split& sp = M.sp;
        const uint32_t ub = split_begin(sp, blockIdx.x), ue = split_begin(sp, blockIdx.x + 1u), bpr = (uint32_t)M.bpr;      // at least one unit
        uint32_t kq_a;
        const uint32_t rg0 = split_row(sp, ub, kq_a);
        // the set is prepared for this matrix long before a warp gets here; a bounded wait all the same
        {
            uint32_t spins = 0;
            while (ctl[set].ready != (uint32_t)i + 1u && ++spins < kOverlapSpins) {}
            if (ctl[set].ready != (uint32_t)i + 1u) { if (lane == 0) atomicOr(fa.flags, 1u); return; }
            __threadfence_block();
        }
        const uint32_t* xs = sets + set * set_words;
        float* acc = reinterpret_cast<float*>(sets + set * set_words + xs_words);
        const uint32_t nchunks = ue - ub;
        const unsigned long long* seg = static_cast<const unsigned long long*>(M.weights) + (uint64_t)ub * 32 + lane;
        const uint16_t* gain_pass = M.gain + (int64_t)rg0 * kGemvGroupRows * bpr;
        if (i + 1 < mm.n && warp == 0) {                    // ask for the next matrix's first chunks in L2
            const uint32_t ub2 = split_begin(mm.m[i + 1].sp, blockIdx.x), ue2 = split_begin(mm.m[i + 1].sp, blockIdx.x + 1u);
            const unsigned long long* nxt = static_cast<const unsigned long long*>(mm.m[i + 1].weights) + (uint64_t)ub2 * 32;
            for (int c = lane; c < 64 && ub2 + c / 2 < ue2; c += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(nxt + c * 16));
        }
        uint32_t ch = 0;
        if (lane == 0) ch = atomicAdd(const_cast<uint32_t*>(&ctl[set].next_chunk), 1u);
        ch = __shfl_sync(kFullMask, ch, 0);
        unsigned long long e = ch < nchunks ? __ldg(seg + (uint64_t)ch * 32) : 0ull;
        while (ch < nchunks) {
            uint32_t nxt = 0;
            if (lane == 0) nxt = atomicAdd(const_cast<uint32_t*>(&ctl[set].next_chunk), 1u);
            nxt = __shfl_sync(kFullMask, nxt, 0);
            const unsigned long long e_next = nxt < nchunks ? __ldg(seg + (uint64_t)nxt * 32) : 0ull;
            const uint64_t I = e & kSortIndexMask;
            const uint32_t pos = (uint32_t)(e >> 48);
            const bool valid = I != kSortIndexMask && I < fa.n_points;
            uint32_t kq;
            const uint32_t q = split_row(sp, kq_a + (pos >> 5), kq);
            const uint32_t rloc = q * kGemvGroupRows + ((pos >> 2) & 7u);                 // row inside the CTA's share
            const uint32_t cb = kq * 4u + (pos & 3u);
            float gn = 0.f;
            uint16_t gbits = 0;
            if (valid) gbits = ldg_u16_here(gain_pass + (rloc * bpr + cb));
            Decoded r;
            decode_sorted_entry(fa, T, I, valid, r);
            gn = gain_to_float(gbits);
            uint32_t w[12];
            expand_bf16(r, gn, w);
            const uint4* xb = reinterpret_cast<const uint4*>(xs + cb * 12u);
            const uint4 x0 = xb[0], x1 = xb[1], x2 = xb[2];
            const uint32_t xv[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
            const float dot = dot24_bf16(w, xv);
            if (valid) atomicAdd(&acc[rloc << shift | ((uint32_t)lane & ((1u << shift) - 1u))], dot);
            ch = nxt; e = e_next;
            use_from_here(e);
        }
        // out of chunks: count this warp in; the last one ends the pass and hands the set on
        __threadfence_block();
        uint32_t last = 0;
        if (lane == 0) last = atomicAdd(const_cast<uint32_t*>(&ctl[set].arrived), 1u) == kWarps - 1u;
        last = __shfl_sync(kFullMask, last, 0);
        if (last) {
            __threadfence_block();
            YOut yo{};
            yo.y = M.y;
            auto row_sums = [&](uint32_t r) { return acc_row_sums(acc, r, shift); };
            finish_pass<kOutBf16, false, kTrees>(yo, sp, rg0, split_row(sp, ue - 1u), ub, ue, M.n_out, scratch, counters, row_sums, M.slot0, 0, 1);
            __syncwarp();
            if (i + kOverlapSets < mm.n) {
                if (lane == 0) { ctl[set].next_chunk = 0u; ctl[set].arrived = 0u; }
                prepare(i + kOverlapSets, lane, 32);
                __threadfence_block();
                __syncwarp();
                if (lane == 0) ctl[set].ready = (uint32_t)(i + kOverlapSets) + 1u;
            }
        }
    }
}

// ===========================================================================
// Fused GEMV on the stored stream with the blocks ordered inside the kernel (order.cuh): the work split of gemv_fast_kernel.  A
// CTA's range of a pass is cut into an equal contiguous share per team of 8 warps, a share into pieces of 32 units (1024 blocks); a
// team orders a piece, its warps take 32 consecutive entries at a time, run the one unranker form they need, and each lane
// forms its own dot product, as in gemv_sorted_kernel.  A share's pieces are of equal size (the teams drift apart by
// themselves: first pieces of 8, 16, 24 and 32 units made shares of two pieces slower and long ones no faster).  28672 x 8192:
// 278 -> 235 us, 8192 x 8192: 82 -> 72 us, 11008 x 4096: 54.5 -> 53.7 us against gemv_bin_kernel, which orders up to 8192 blocks at a
// time as a phase of the whole block and is the faster one while that is the CTA's whole range (4096 x 4096: 23.7 against 26.9 us).
// ===========================================================================
constexpr int kOrderTeams = 4;
constexpr int kTeamThreads = kSortThreads / kOrderTeams;

// Bytes of the teams' areas in shared memory: chunk counters, two histograms per team, the entries of a piece per team.
__host__ __device__ inline size_t gemv_order_bytes(const OrderArgs& oa) { return 16 + (size_t)kOrderTeams * (2 * 4 * oa.words + kOrderBlocks * 8); }

// The span of the index stream and of the gains that this CTA's row groups cover is contiguous: request it from DRAM ahead
// of time; the ordering then reads it from L2.
template <bool kSg>
__device__ __forceinline__ void prefetch_stored_span(const FastArgs& fa, const uint32_t* stream, const uint16_t* gain, const SgArgs& sg,
                                                     const Split& sp, int64_t n_out, int64_t bpr)
{
    const uint32_t ub = split_begin(sp, blockIdx.x), ue = split_begin(sp, blockIdx.x + 1u);
    if (ub < ue) {
        const uint64_t b_first = (uint64_t)split_row(sp, ub) * kGemvGroupRows * (uint64_t)bpr;
        const uint64_t b_last = (uint64_t)min((int64_t)(split_row(sp, ue - 1u) + 1u) * kGemvGroupRows, n_out) * (uint64_t)bpr;
        const uint64_t wf = (uint64_t)fa.dc.W + (kSg ? (uint64_t)sg.bits : 0ull);
        prefetch_span_l2(stream, b_first * wf / 8, (b_last * wf + 7) / 8, threadIdx.x, blockDim.x);
        if (!kSg) prefetch_span_l2(gain, b_first * 2, b_last * 2, threadIdx.x, blockDim.x);
    }
}

// One matrix; `piece` = pieces this team has been through.
template <bool kOutBf16, bool kSg, bool kShard, bool kTrees>
__device__ __forceinline__ void gemv_order_body(const FastArgs& fa, const FastSmem& T, const OrderArgs& oa, uint32_t* xs, uint8_t* areas,
                                                const uint32_t* __restrict__ stream, const uint16_t* __restrict__ gain, const SgArgs& sg, const Split& sp,
                                                int64_t n_out, int64_t k_in, uint32_t bpr, const uint16_t* __restrict__ x, const YOut& yo,
                                                float* __restrict__ scratch, uint32_t* __restrict__ counters, int64_t slot0, uint32_t& piece)
{
    constexpr uint32_t kTeamWarps = kTeamThreads / 32;
    float* acc = reinterpret_cast<float*>(xs + sp.per_row * 48u);   // [kSortAccFloats]
    const uint32_t lane = threadIdx.x & 31, tid = threadIdx.x & (kTeamThreads - 1);
    const int team = (int)(threadIdx.x / kTeamThreads);
    uint32_t* next_chunk = reinterpret_cast<uint32_t*>(areas) + team;
    uint32_t* hist = reinterpret_cast<uint32_t*>(areas + 16) + (uint32_t)team * 2u * oa.words;
    unsigned long long* ent = reinterpret_cast<unsigned long long*>(areas + 16 + kOrderTeams * 2 * 4 * oa.words) + team * kOrderBlocks;
    stage_x(xs, x, k_in, sp.per_row * 48u, threadIdx.x, blockDim.x);
    for_each_sorted_segment(sp, blockIdx.x, [&](uint32_t p_begin, uint32_t p_end, uint32_t rg0, uint32_t rg1, bool, bool) {
        const uint32_t shift = acc_shift((rg1 - rg0 + 1u) * kGemvGroupRows, kSortAccFloats);
        for (uint32_t i = threadIdx.x; i < (rg1 - rg0 + 1u) * kGemvGroupRows << shift; i += blockDim.x) acc[i] = 0.f;
        __syncthreads();
        const uint32_t units = p_end - p_begin;
        const uint32_t t_begin = p_begin + (uint32_t)team * units / kOrderTeams, t_end = p_begin + ((uint32_t)team + 1u) * units / kOrderTeams;
        const uint16_t* gain_pass = gain + (int64_t)rg0 * kGemvGroupRows * bpr;
        const uint32_t npieces = (t_end - t_begin + 31u) / 32u, size = npieces ? (t_end - t_begin + npieces - 1u) / npieces : 1u;
        for (uint32_t u0 = t_begin; u0 < t_end; u0 += size, ++piece) {
            const uint32_t nchunks = min(size, t_end - u0);
            // a thread has one column block of the piece (of up to 128, 64 or 32) and every second, fourth or single row of it: a warp
            // reads 32 neighbouring fields, and a small piece is spread over all threads
            const uint32_t narrow = nchunks <= 8u ? 2u : nchunks <= 16u ? 1u : 0u, c = tid & (127u >> narrow), r = tid >> (7u - narrow);
            uint32_t kq;
            const uint32_t rg = split_row(sp, u0 + (c >> 2), kq);
            OrderSpot<uint32_t> o;
            o.row = rg * kGemvGroupRows + r;
            o.b0 = (uint64_t)rg0 * kGemvGroupRows * bpr;
            o.b = (o.row - rg0 * kGemvGroupRows) * bpr + kq * 4u + (c & 3u);
            o.pos = (c >> 2) * 32u + r * 4u + (c & 3u);
            o.there = (c >> 2) < nchunks && kq * 4u + (c & 3u) < bpr;
            order_piece<false, kSg, kTeamThreads>(fa, T, sg, oa, stream, hist + (piece & 1u) * oa.words, hist + ((piece & 1u) ^ 1u) * oa.words, ent, nullptr, team, tid,
                                                 o, min((uint32_t)n_out, (rg + 1u) * kGemvGroupRows), bpr << (1u + narrow), 2u << narrow, 8u << narrow, [&] { if (tid == 0) *next_chunk = kTeamWarps; });
            uint32_t kq_a;
            const uint32_t rg_off = split_row(sp, u0, kq_a) - rg0;
            uint32_t ch = tid >> 5;
            while (ch < nchunks) {
                uint32_t nxt = 0;
                if (lane == 0) nxt = atomicAdd(next_chunk, 1u);
                nxt = __shfl_sync(kFullMask, nxt, 0);
                const OrderedBlock b = ordered_block<kSg>(fa, sg, oa, ent[ch * 32u + lane]);
                uint32_t kqb;
                const uint32_t q = split_row(sp, kq_a + (b.pos >> 5), kqb);
                const uint32_t rloc = (rg_off + q) * kGemvGroupRows + ((b.pos >> 2) & 7u);    // row inside the pass
                const uint32_t cb = kqb * 4u + (b.pos & 3u);
                float gn = 0.f;
                uint16_t gbits = 0;
                if (!kSg && b.valid) gbits = ldg_u16_here(gain_pass + (rloc * bpr + cb));
                uint32_t w[12];
                if (kSg && b.valid) {
                    const float scale = sg.row_scale ? __ldg(sg.row_scale + (int64_t)rg0 * kGemvGroupRows + rloc) : 1.f;
                    gn = __fmul_rn(__fmul_rn(scale, __ldg(sg.codebook + b.gain_index)), __uint_as_float(T.desc[b.cls * kFastDescStride + kFastDescRnorm]));
                }
                Decoded d;
                decode_known_class(T, b.valid ? b.cls : 0u, b.local, b.valid, d);
                if (!kSg) gn = gain_to_float(gbits);
                expand_bf16(d, gn, w);
                const uint4* xb = reinterpret_cast<const uint4*>(xs + cb * 12u);
                const uint4 x0 = xb[0], x1 = xb[1], x2 = xb[2];
                const uint32_t xv[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
                const float dot = dot24_bf16(w, xv);
                if (b.valid) atomicAdd(&acc[rloc << shift | (lane & ((1u << shift) - 1u))], dot);
                ch = nxt;
            }
        }
        __syncthreads();
        const uint32_t ub = split_begin(sp, blockIdx.x), ue = split_begin(sp, blockIdx.x + 1u);     // recomputed here: not kept across the main loop
        finish_pass<kOutBf16, kShard, kTrees>(yo, sp, rg0, rg1, ub, ue, n_out, scratch, counters, [&](uint32_t i) { return acc_row_sums(acc, i, shift); }, slot0);
        __syncthreads();                                   // the sums are read above: the next pass may clear them only now
    }, 1u << 30);
}

// Where the areas lie for rows of up to nq units per row group; the histograms start at zero.
#define ORDER_PROLOGUE(nq)                                                                                         \
    uint32_t* xs = reinterpret_cast<uint32_t*>(staging);            /* [nq * 4][12] packed bf16 pairs of x */       \
    uint8_t* areas = reinterpret_cast<uint8_t*>(xs + (nq) * 48u) + kSortAccFloats * 4;                               \
    for (uint32_t i = threadIdx.x; i < kOrderTeams * 2 * oa.words; i += blockDim.x) reinterpret_cast<uint32_t*>(areas + 16)[i] = 0u; \
    uint32_t piece = 0;

template <bool kOutBf16, bool kSg, bool kShard, bool kTrees>
__global__ void __launch_bounds__(kSortThreads, 1)
gemv_order_kernel(FastArgs fa, const uint32_t* __restrict__ stream, OrderArgs oa, const uint16_t* __restrict__ gain, SgArgs sg,
                  Split sp, int64_t n_out, int64_t k_in, int64_t bpr, const uint16_t* __restrict__ x, YOut yo,
                  float* __restrict__ scratch, uint32_t* __restrict__ counters)
{
    prefetch_stored_span<kSg>(fa, stream, gain, sg, sp, n_out, bpr);       // while the table image is on its way
    FAST_PROLOGUE(if (kShard) shard_arrive(yo));
    ORDER_PROLOGUE(sp.per_row);
    gemv_order_body<kOutBf16, kSg, kShard, kTrees>(fa, T, oa, xs, areas, stream, gain, sg, sp, n_out, k_in, (uint32_t)bpr, x, yo, scratch, counters, 0, piece);
    if (kShard) shard_arrive(yo);
}

// Several independent matrices on their stored streams in one launch; max_nq = the largest number of units per row group.
template <bool kOutBf16, bool kTrees>
__global__ void __launch_bounds__(kSortThreads, 1)
gemv_order_multi_kernel(FastArgs fa, OrderArgs oa, const __grid_constant__ GemvMulti mm, uint32_t max_nq, float* __restrict__ scratch,
                        uint32_t* __restrict__ counters)
{
    prefetch_stored_span<false>(fa, static_cast<const uint32_t*>(mm.m[0].weights), mm.m[0].gain, SgArgs{}, mm.m[0].sp, mm.m[0].n_out, mm.m[0].bpr);
    FAST_PROLOGUE();
    ORDER_PROLOGUE(max_nq);
    for (int i = 0; i < mm.n; ++i) {
        const GemvMat& M = mm.m[i];
        if (i + 1 < mm.n)
            prefetch_stored_span<false>(fa, static_cast<const uint32_t*>(mm.m[i + 1].weights), mm.m[i + 1].gain, SgArgs{}, mm.m[i + 1].sp,
                                        mm.m[i + 1].n_out, mm.m[i + 1].bpr);
        YOut yo{};
        yo.y = M.y;
        gemv_order_body<kOutBf16, false, false, kTrees>(fa, T, oa, xs, areas, static_cast<const uint32_t*>(M.weights), M.gain, SgArgs{}, M.sp, M.n_out, M.k_in,
                                                       (uint32_t)M.bpr, M.x, yo, scratch, counters, M.slot0, piece);
    }
}

// ===========================================================================
// Fused GEMV on the stored stream with the blocks binned inside the kernel: the work split of gemv_fast_kernel, but a
// CTA first looks up the class of every block of a segment of up to kBinSegUnits units (S1-S2), orders the
// (class-local index, class, position) triples by the sorted layout's key with a counting sort in shared memory,
// and then proceeds like gemv_sorted_kernel on those entries (S3-S8): a warp takes 32 consecutive entries, runs
// the one unranker form they need and each lane forms its own dot product.
// ===========================================================================
constexpr int kBinSegUnits = 256;                    // at most 8192 blocks per segment
constexpr int kBinPerThread = kBinSegUnits * 32 / kSortThreads;   // 8

template <bool kOutBf16, bool kSg, bool kShard, bool kTrees>
__device__ __forceinline__ void gemv_bin_body(const FastArgs& fa, const FastSmem& T, uint8_t* staging, const uint32_t* __restrict__ stream,
                                              const uint16_t* __restrict__ sort_rank, const uint16_t* __restrict__ gain, const SgArgs& sg,
                                              const Split& sp, int64_t n_out, int64_t k_in, uint32_t bpr, uint32_t acc_floats,
                                              const uint16_t* __restrict__ x, const YOut& yo, float* __restrict__ scratch,
                                              uint32_t* __restrict__ counters, int64_t slot0)
{
    const uint32_t nq = sp.per_row;
    uint32_t* xs = reinterpret_cast<uint32_t*>(staging);            // [nq * 4][12] packed bf16 pairs of x
    float* acc = reinterpret_cast<float*>(xs + nq * 48);            // [acc_floats]
    uint32_t* last_flag = reinterpret_cast<uint32_t*>(acc + acc_floats);
    uint32_t* next_chunk = last_flag + 1;
    uint32_t* hist = last_flag + 4;                                  // [1024] bins in sort order; later their first slots
    uint32_t* cursor = hist + 1024;                                  // [1024]
    unsigned long long* ent = reinterpret_cast<unsigned long long*>(cursor + 1024);   // [kBinSegUnits * 32] class-local index | position << 48
    uint16_t* ent_cls = reinterpret_cast<uint16_t*>(ent + kBinSegUnits * 32);         // [kBinSegUnits * 32] class (| gain index << 10), 0xffff = no block
    stage_x(xs, x, k_in, nq * 48, threadIdx.x, blockDim.x);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t kWarps = blockDim.x >> 5;
    for_each_sorted_segment(sp, blockIdx.x, [&](uint32_t tu0, uint32_t tu1, uint32_t rg0, uint32_t rg1, bool first, bool last) {
        const uint32_t shift = acc_shift((rg1 - rg0 + 1u) * kGemvGroupRows, acc_floats);
        if (first)
            for (uint32_t i = threadIdx.x; i < (rg1 - rg0 + 1u) * kGemvGroupRows << shift; i += blockDim.x) acc[i] = 0.f;
        hist[threadIdx.x] = 0; cursor[threadIdx.x] = 0;
        if (threadIdx.x == 0) *next_chunk = kWarps;
        __syncthreads();
        uint32_t kq_a;
        const uint32_t rg_a = split_row(sp, tu0, kq_a), rg_off = rg_a - rg0;
        const int entries = (int)(tu1 - tu0) * 32;
        // ---- S1-S2 for the whole segment and the histogram of the sort keys
        unsigned long long mine_ent[kBinPerThread];
        uint32_t mine_key[kBinPerThread];
#pragma unroll
        for (int q = 0; q < kBinPerThread; ++q) {
            const int i = (int)threadIdx.x + q * kSortThreads;
            mine_key[q] = 0xffffffffu; mine_ent[q] = 0ull;
            if (i < entries) {
                const uint32_t pos = (uint32_t)i;
                uint32_t kq;
                const uint32_t qd = split_row(sp, kq_a + (pos >> 5), kq);
                const int64_t row = (int64_t)(rg_a + qd) * kGemvGroupRows + ((pos >> 2) & 7u), cb = (int64_t)kq * 4 + (pos & 3u);
                uint32_t key = 1023u, cls = 0xffffu;
                uint64_t local = 0;
                if (row < n_out && cb < bpr) {
                    const uint64_t f = load_field(stream, (uint64_t)(row * bpr + cb), (int)fa.L.W + (kSg ? sg.bits : 0));
                    const uint64_t I = kSg ? f & ((1ull << fa.L.W) - 1ull) : f;
                    if (I < fa.n_points) {
                        cls = fast_find_class(T, I, local);
                        key = __ldg(sort_rank + cls);
                        if (kSg) cls |= (uint32_t)(f >> fa.L.W) << 10;           // the gain index rides with the class
                    } else atomicAdd(fa.bad_index, 1ull);
                }
                mine_key[q] = key | cls << 16;
                mine_ent[q] = local | (unsigned long long)pos << 48;
                atomicAdd(&hist[key], 1u);
            }
        }
        __syncthreads();
        // exclusive prefix sum of the 1024 bins: one bin per thread
        {
            const uint32_t c = hist[threadIdx.x];
            uint32_t incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(kFullMask, incl, o); if (lane >= o) incl += t; }
            if (lane == 31) cursor[warp] = incl;                       // warp totals, parked in the cursor array for a moment
            __syncthreads();
            uint32_t before = 0;
            for (int w2 = 0; w2 < warp; ++w2) before += cursor[w2];
            __syncthreads();
            hist[threadIdx.x] = before + incl - c;
            cursor[threadIdx.x] = 0;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kBinPerThread; ++q) {
            if (mine_key[q] != 0xffffffffu) {
                const uint32_t key = mine_key[q] & 0xffffu;
                const uint32_t slot = hist[key] + atomicAdd(&cursor[key], 1u);
                ent[slot] = mine_ent[q];
                ent_cls[slot] = (uint16_t)(mine_key[q] >> 16);
            }
        }
        __syncthreads();
        // ---- S3-S8 on the ordered entries
        const uint32_t nchunks = tu1 - tu0;
        const uint16_t* gain_pass = gain + (int64_t)rg0 * kGemvGroupRows * bpr;
        for (uint32_t ch = (uint32_t)warp; ch < nchunks;) {
            uint32_t nxt = 0;
            if (lane == 0) nxt = atomicAdd(next_chunk, 1u);
            nxt = __shfl_sync(kFullMask, nxt, 0);
            const unsigned long long e = ent[ch * 32 + lane];
            const uint32_t cls16 = ent_cls[ch * 32 + lane];
            const bool valid = cls16 != 0xffffu;
            const uint32_t pos = (uint32_t)(e >> 48);
            uint32_t kq;
            const uint32_t q = split_row(sp, kq_a + (pos >> 5), kq);
            const uint32_t rloc = (rg_off + q) * kGemvGroupRows + ((pos >> 2) & 7u);
            const uint32_t cb = kq * 4u + (pos & 3u);
            const uint32_t cls = valid ? (kSg ? cls16 & 1023u : cls16) : 0u;
            float gn = 0.f;
            uint16_t gbits = 0;
            if (valid) {
                if (kSg) {
                    const float scale = sg.row_scale ? __ldg(sg.row_scale + (int64_t)rg0 * kGemvGroupRows + rloc) : 1.f;
                    gn = __fmul_rn(__fmul_rn(scale, __ldg(sg.codebook + (cls16 >> 10))), __uint_as_float(T.desc[cls * kFastDescStride + kFastDescRnorm]));
                } else {
                    gbits = ldg_u16_here(gain_pass + (rloc * bpr + cb));
                }
            }
            Decoded r;
            decode_known_class(T, cls, e & ((1ull << 48) - 1ull), valid, r);
            if (!kSg) gn = gain_to_float(gbits);
            uint32_t w[12];
            expand_bf16(r, gn, w);
            const uint4* xb = reinterpret_cast<const uint4*>(xs + cb * 12u);
            const uint4 x0 = xb[0], x1 = xb[1], x2 = xb[2];
            const uint32_t xv[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
            const float dot = dot24_bf16(w, xv);
            if (valid) atomicAdd(&acc[rloc << shift | ((uint32_t)lane & ((1u << shift) - 1u))], dot);
            ch = nxt;
        }
        __syncthreads();
        if (!last) return;
        auto row_sums = [&](uint32_t r) { return acc_row_sums(acc, r, shift); };
        const uint32_t ub = split_begin(sp, blockIdx.x), ue = split_begin(sp, blockIdx.x + 1u);     // recomputed here: not kept across the main loop
        finish_pass<kOutBf16, kShard, kTrees>(yo, sp, rg0, rg1, ub, ue, n_out, scratch, counters, row_sums, slot0);
        __syncthreads();
    }, (uint32_t)kBinSegUnits);
}

template <bool kOutBf16, bool kSg, bool kShard, bool kTrees>
__global__ void __launch_bounds__(kSortThreads, 1)
gemv_bin_kernel(FastArgs fa, const uint32_t* __restrict__ stream, const uint16_t* __restrict__ sort_rank, const uint16_t* __restrict__ gain, SgArgs sg,
                Split sp, int64_t n_out, int64_t k_in, int64_t bpr, uint32_t acc_floats, const uint16_t* __restrict__ x, YOut yo,
                float* __restrict__ scratch, uint32_t* __restrict__ counters)
{
    prefetch_stored_span<kSg>(fa, stream, gain, sg, sp, n_out, bpr);       // while the table image is on its way
    FAST_PROLOGUE(if (kShard) shard_arrive(yo));
    gemv_bin_body<kOutBf16, kSg, kShard, kTrees>(fa, T, staging, stream, sort_rank, gain, sg, sp, n_out, k_in, (uint32_t)bpr, acc_floats, x, yo, scratch, counters, 0);
    if (kShard) shard_arrive(yo);
}

// Several independent matrices on their stored streams in one launch.
template <bool kOutBf16, bool kTrees>
__global__ void __launch_bounds__(kSortThreads, 1)
gemv_bin_multi_kernel(FastArgs fa, const uint16_t* __restrict__ sort_rank, const __grid_constant__ GemvMulti mm, uint32_t acc_floats, float* __restrict__ scratch,
                      uint32_t* __restrict__ counters)
{
    prefetch_stored_span<false>(fa, static_cast<const uint32_t*>(mm.m[0].weights), mm.m[0].gain, SgArgs{}, mm.m[0].sp, mm.m[0].n_out, mm.m[0].bpr);
    FAST_PROLOGUE();
    for (int i = 0; i < mm.n; ++i) {
        const GemvMat& M = mm.m[i];
        if (i + 1 < mm.n)
            prefetch_stored_span<false>(fa, static_cast<const uint32_t*>(mm.m[i + 1].weights), mm.m[i + 1].gain, SgArgs{}, mm.m[i + 1].sp,
                                     mm.m[i + 1].n_out, mm.m[i + 1].bpr);
        YOut yo{};
        yo.y = M.y;
        gemv_bin_body<kOutBf16, false, false, kTrees>(fa, T, staging, static_cast<const uint32_t*>(M.weights), sort_rank, M.gain, SgArgs{}, M.sp, M.n_out, M.k_in,
                                              (uint32_t)M.bpr, acc_floats, M.x, yo, scratch, counters, M.slot0);
        __syncthreads();
    }
}
