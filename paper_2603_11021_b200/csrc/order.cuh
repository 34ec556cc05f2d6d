// Ordering of a stored stream inside the product kernels, in pieces of up to 1024 blocks: a team of warps looks up the classes of
// a piece's blocks (S1-S2) and puts them, in shared memory, into the order of the sorted layouts (decoder form, unranking
// steps, class); the team then unranks them (S3-S8) like entries of those layouts.  Included by gemv.cu and gemm.cu inside
// their unnamed namespaces, after kernels_common.cuh.
//
// The ordering is short of instructions but long in latency (stream words from L2, dependent table look-ups, a prefix sum).  As a
// phase of the whole thread block between block barriers it took 40 % of the time of the stored-stream GEMV at half the
// issue rate; several teams that drift apart, each with a named barrier of its own, fill one another's gaps.
#pragma once

constexpr int kOrderBlocks = 1024;                          // blocks of a piece
constexpr uint32_t kOrderPosShift = 22;                     // position in the top 10 bits of an entry's high word (class tables in shared memory)

struct OrderArgs {
    const uint16_t* sort_rank;      // sort key of every class (class tables in shared memory), else null
    uint32_t words;                 // bins of a histogram (32 times an odd number); the last bin is "no block"
    uint32_t cls_shift, gain_shift; // high word of an entry: class-local index >> 32 | class << cls_shift | gain index << gain_shift | position << 22
};

// Where the blocks of a thread lie in a piece: numbers b0 + b, b0 + b + b_step, .. in the stream, rows row, row + row_step, .. (there
// are n_out), position codes pos, pos + pos_step, ..; none of them where the column or the unit does not exist (!there).
// Count: what the bits of b and the steps are counted in.  Nothing limits the length of a row of the batched products: 64 bits, with
// b0 = 0.  A row of the GEMV has its slice of x in shared memory (192 bytes per 4 blocks of 227 KB), and the at most 1024 + 32
// rows of a pass then hold less than 2^23 blocks: 32 bits behind b0, their first block (11008 x 4096: 53.3 us, with 64 bits 53.4).
template <typename Count>
struct OrderSpot {
    uint64_t b0;
    Count b;
    uint32_t row, pos;
    bool there;
};

__device__ __forceinline__ void team_barrier(int team, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(threads) : "memory"); }

// Orders one piece; the kThreads threads of team `team` call this together, numbered tid.  hist / hist_next: this piece's
// histogram (zero on entry) and the next one's (zeroed here).  The entries go to ent (with kBig the class-local index) and, with
// kBig, ent2 (class | position << 17, bit 31 = no block); on return the piece is complete.
// before_write(): what has to be awaited before ent may be written.
template <bool kBig, bool kSg, int kThreads, typename Count, typename Before>
__device__ __forceinline__ void order_piece(const FastArgs& fa, const FastSmem& T, const SgArgs& sg, const OrderArgs& oa, const uint32_t* __restrict__ stream,
                                            uint32_t* hist, uint32_t* hist_next, unsigned long long* ent, uint32_t* ent2, int team, uint32_t tid,
                                            const OrderSpot<Count>& o, uint32_t n_out, Count b_step, uint32_t row_step, uint32_t pos_step, Before before_write)
{
    constexpr int kEach = kOrderBlocks / kThreads;
    const uint32_t lane = tid & 31u;
    const int wbits = fa.dc.W + (kSg ? sg.bits : 0);
    const uint32_t none = oa.words - 1u;
    uint64_t local[kEach];
    uint32_t hi[kEach], key[kEach], rank[kEach];             // hi: what the entry keeps beside the class-local index and the position
    {
        RawField<kBig> raw[kEach];
        const uint64_t bits0 = o.b0 * (uint64_t)wbits;
        const uint32_t* base = stream + (bits0 >> 5);
        const Count bits = o.b * (Count)wbits + ((uint32_t)bits0 & 31u), step = b_step * (Count)wbits;
        uint32_t in = 0;
#pragma unroll
        for (int q = 0; q < kEach; ++q) {
            const bool there = o.there && o.row + (uint32_t)q * row_step < n_out;
            const Count at = bits + (uint32_t)q * step;
            raw[q] = request_field_at<kBig>(base + (at >> 5), (uint32_t)at & 31u, wbits, there);
            in |= (uint32_t)there << q;
        }
        if constexpr (kBig) {
            // the searches of the thread's blocks go side by side: each is a chain of reads from L2 (bucket, offsets, offset, record)
            uint64_t lo[kEach];
            uint32_t high[kEach], a[kEach], z[kEach], h[kEach], valid = 0;
#pragma unroll
            for (int q = 0; q < kEach; ++q) {
                uint64_t h64;
                field_value(raw[q], wbits, lo[q], h64);
                high[q] = (uint32_t)h64;
                const bool v = ((in >> q) & 1u) && (h64 < fa.dc.n_hi || (h64 == fa.dc.n_hi && lo[q] < fa.dc.n_lo));
                if (((in >> q) & 1u) && !v) atomicAdd(fa.bad_index, 1ull);
                valid |= (uint32_t)v << q;
                a[q] = z[q] = 0u;
                if (v) {
                    const uint32_t bucket = big_bucket(fa.dc, lo[q], h64);
                    a[q] = __ldg(fa.dc.lut + bucket); z[q] = __ldg(fa.dc.lut + bucket + 1);
                }
            }
            while (true) {
                bool more = false;
#pragma unroll
                for (int q = 0; q < kEach; ++q) more = more || a[q] < z[q];
                if (!more) break;
                uint64_t ol[kEach];
                uint32_t oh[kEach];
#pragma unroll
                for (int q = 0; q < kEach; ++q) {
                    const uint32_t mid = (a[q] + z[q] + 1u) >> 1;
                    ol[q] = 0; oh[q] = 0;
                    if (a[q] < z[q]) { ol[q] = __ldg(fa.dc.off_lo + mid); oh[q] = __ldg(fa.dc.off_hi + mid); }
                }
#pragma unroll
                for (int q = 0; q < kEach; ++q) {
                    const uint32_t mid = (a[q] + z[q] + 1u) >> 1;
                    if (a[q] < z[q]) { if (oh[q] < high[q] || (oh[q] == high[q] && ol[q] <= lo[q])) a[q] = mid; else z[q] = mid - 1u; }
                }
            }
#pragma unroll
            for (int q = 0; q < kEach; ++q) {
                local[q] = 0; h[q] = 0;
                if ((valid >> q) & 1u) { local[q] = lo[q] - __ldg(fa.dc.off_lo + a[q]); h[q] = __ldg(reinterpret_cast<const uint32_t*>(fa.dc.big + a[q])); }
            }
#pragma unroll
            for (int q = 0; q < kEach; ++q) {
                const bool v = (valid >> q) & 1u;
                const uint32_t nlev = h[q] >> 28, nlev1 = (h[q] >> 24) & 7u, parity = (h[q] >> 16) & 1u;
                // coarse shape of the unranking; two bins per shape (by lane): the few common shapes would queue at one word each
                key[q] = v ? ((1u - parity) << 6 | (7u - min(nlev, 7u)) << 3 | nlev1) * 2u + (lane & 1u) : none;
                hi[q] = v ? a[q] : 1u << 31;
            }
        } else {
#pragma unroll
            for (int q = 0; q < kEach; ++q) {
                uint64_t lo, high;
                field_value(raw[q], wbits, lo, high);
                const bool there = (in >> q) & 1u;
                const uint64_t I = kSg ? lo & ((1ull << fa.L.W) - 1ull) : lo;
                const bool valid = there && I < fa.n_points;
                if (there && !valid) atomicAdd(fa.bad_index, 1ull);
                uint32_t cls = fa.L.ncls;                                 // no block
                key[q] = none; local[q] = 0;
                if (valid) {
                    cls = fast_find_class(T, I, local[q]);
                    key[q] = __ldg(oa.sort_rank + cls);
                }
                hi[q] = cls << oa.cls_shift;
                if (kSg) hi[q] |= (uint32_t)(lo >> fa.L.W) << oa.gain_shift;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < kEach; ++q) rank[q] = atomicAdd(hist + key[q], 1u);      // its place among the blocks of the same bin
    team_barrier(team, kThreads);
    if (tid < 32u) {                                          // counts -> first slots: one warp, words / 32 bins per lane
        const uint32_t each = oa.words / 32u;
        uint32_t sum = 0;
#pragma unroll 4
        for (uint32_t i = 0; i < each; ++i) sum += hist[lane * each + i];
        uint32_t incl = sum;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) { const uint32_t t = __shfl_up_sync(kFullMask, incl, s); if ((int)lane >= s) incl += t; }
        uint32_t run = incl - sum;
#pragma unroll 4
        for (uint32_t i = 0; i < each; ++i) { const uint32_t v = hist[lane * each + i]; hist[lane * each + i] = run; run += v; }
    } else {
        for (uint32_t i = tid - 32u; i < oa.words; i += kThreads - 32) hist_next[i] = 0u;
    }
    before_write();
    team_barrier(team, kThreads);
#pragma unroll
    for (int q = 0; q < kEach; ++q) {
        const uint32_t pos = o.pos + (uint32_t)q * pos_step, slot = hist[key[q]] + rank[q];
        if (kBig) {
            ent[slot] = local[q];
            ent2[slot] = hi[q] | pos << 17;
        } else {
            ent[slot] = local[q] | (unsigned long long)(hi[q] | pos << kOrderPosShift) << 32;
        }
    }
    team_barrier(team, kThreads);
}

// The fields of an entry.
struct OrderedBlock {
    uint64_t local;
    uint32_t cls, pos, gain_index;
    bool valid;
};

template <bool kSg>
__device__ __forceinline__ OrderedBlock ordered_block(const FastArgs& fa, const SgArgs& sg, const OrderArgs& oa, uint64_t x)
{
    OrderedBlock o;
    const uint32_t hi = (uint32_t)(x >> 32);
    o.local = (uint64_t)(hi & ((1u << oa.cls_shift) - 1u)) << 32 | (uint32_t)x;
    o.cls = (hi >> oa.cls_shift) & ((1u << (oa.gain_shift - oa.cls_shift)) - 1u);
    o.valid = o.cls < fa.L.ncls;
    o.gain_index = kSg ? (hi >> oa.gain_shift) & ((1u << sg.bits) - 1u) : 0u;
    o.pos = hi >> kOrderPosShift;
    return o;
}

// How a code's stored stream is ordered (host).  False where it is not: few classes (a warp of unrelated blocks costs little there),
// or entries that do not fit.
bool order_args(const llvq_ctx* ctx, int gain_bits, OrderArgs* oa)
{
    *oa = OrderArgs{};
    const size_t ncls = ctx->host.desc.size();
    if (!ctx->fast) {
        oa->words = 288;                                     // 128 shapes x 2 and "no block"
        return gain_bits == 0 && ncls <= (1u << 17);
    }
    if (!ctx->d_sort_rank || ncls < 64 || ncls > 1023 || ctx->host.W + gain_bits > 64) return false;
    auto bits = [](uint64_t v) { uint32_t b = 0; while (v >> b) ++b; return b; };
    const uint32_t local_high = std::max(bits(ctx->largest_class - 1), 32u) - 32u;
    oa->sort_rank = ctx->d_sort_rank;
    oa->words = (uint32_t)(ncls + 1 + 31) / 32 * 32;
    if ((oa->words / 32) % 2 == 0) oa->words += 32;          // an odd number of bins per lane of the prefix sum: no bank conflicts
    oa->cls_shift = local_high;
    oa->gain_shift = local_high + bits(ncls);
    return oa->gain_shift + (uint32_t)gain_bits <= kOrderPosShift;
}
