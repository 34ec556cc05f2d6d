// Fast dequantizer for codes whose tables fit in shared memory (few classes,
// indices up to 64 bits): App. A steps 1-4 with every table lookup served from
// shared memory, one thread per block of 24 weights.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "tables.h"

namespace llvq {

constexpr uint32_t kFullMask = 0xffffffffu;
constexpr int kPascalToBase14 = 2512;     // byte distance from pascal[t] to base14[t] in the table image

// Pointers into the CTA's copy of the table image.
struct FastSmem {
    const uint32_t* golay;
    const uint16_t* lut;
    const uint32_t* pascal;
    const uint32_t* base14;
    const uint16_t* r14;
    const uint8_t* pd6;
    const uint64_t* off;
    const uint32_t* desc;
    const uint64_t* recip64;  // images without class tables: reciprocals of the Pascal entries
    const uint32_t* recip32;
    uint32_t sub3, sub2;      // shared-window byte addresses of the tables of small subsets, 0 when the kernel did not load them
    uint32_t lut_shift;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// with_small_subsets: the kernel loaded L.total_ext bytes of the image, not only L.total
__device__ __forceinline__ FastSmem fast_view(const uint8_t* smem, const FastLayout& L, bool with_small_subsets = false)
{
    FastSmem T;
    T.golay = reinterpret_cast<const uint32_t*>(smem + L.golay);
    T.lut = reinterpret_cast<const uint16_t*>(smem + L.lut);
    T.pascal = reinterpret_cast<const uint32_t*>(smem + L.pascal);
    T.base14 = reinterpret_cast<const uint32_t*>(smem + L.base14);
    T.r14 = reinterpret_cast<const uint16_t*>(smem + L.r14);
    T.pd6 = smem + L.pd6;
    T.off = reinterpret_cast<const uint64_t*>(smem + L.off);
    T.desc = reinterpret_cast<const uint32_t*>(smem + L.desc);
    T.recip64 = reinterpret_cast<const uint64_t*>(smem + L.recip64);
    T.recip32 = reinterpret_cast<const uint32_t*>(smem + L.recip32);
    T.sub3 = with_small_subsets ? smem_addr(smem + L.sub3) : 0u;
    T.sub2 = with_small_subsets ? smem_addr(smem + L.sub2) : 0u;
    T.lut_shift = L.lut_shift;
    return T;
}

// Copy the table image into shared memory with bulk asynchronous copies (TMA,
// no multicast) tracked by one mbarrier.  Every thread of the CTA must call this.
// Returns false (for the whole CTA) if the copy did not complete within the
// wait limit; the error flag is then set and the caller must return.
__device__ __forceinline__ bool fast_load_image(uint8_t* dst, const uint8_t* __restrict__ src, uint32_t bytes,
                                                uint64_t* bar, uint32_t* err_flags)
{
    const uint32_t bar_a = smem_addr(bar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a), "r"(bytes) : "memory");
        constexpr uint32_t kChunk = 32768;
        for (uint32_t o = 0; o < bytes; o += kChunk) {
            uint32_t n = bytes - o < kChunk ? bytes - o : kChunk;
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_addr(dst + o)), "l"(src + o), "r"(n), "r"(bar_a) : "memory");
        }
    }
    uint32_t done = 0;
    for (uint32_t it = 0; it < (1u << 20) && !done; ++it) {
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(bar_a), "r"(0u) : "memory");
    }
    if (!done) {
        atomicOr(err_flags, 1u);
        // the copy may still be writing this CTA's shared memory: give it the same limit once more before the caller returns
        for (uint32_t it = 0; it < (1u << 20) && !done; ++it) {
            asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                         : "=r"(done) : "r"(bar_a), "r"(0u) : "memory");
        }
        done = 0;
    }
    return __syncthreads_and((int)done) != 0;
}

// r = a * b + c on the multiply-add pipe (the logic pipe is the busy one: sums of disjoint bit fields go here)
__device__ __forceinline__ uint32_t mad_u32(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

// Deposit the low bits of src into the coordinates of mask (layout of coords_of), lowest coordinate first, six per lookup.  The
// entry for mask byte f and source bits s is at f * 64 + (s ^ f): a plain table row per f would put every lane whose source bits
// are used up (s = 0: most lanes, where few slots are taken) into the same two banks whatever f is.  Counted over the classes
// of the 48-bit code, the 32 lanes of a warp need 30 instead of 55 passes over the banks for the deposits of a block.
__device__ __forceinline__ uint32_t deposit24(const uint8_t* pd6, uint32_t src, uint32_t mask)
{
    // how many source bits the lower groups consume: known from the mask alone, so the four lookups are independent
    const uint32_t c1 = __popc(mask & 0xffu), c2 = __popc(mask & 0xffffu), c3 = __popc(mask & 0xffffffu);
    const uint32_t f1 = __byte_perm(mask, 0u, 0x4441), f2 = __byte_perm(mask, 0u, 0x4442);
    const uint32_t r0 = pd6[mad_u32(mask & 0xffu, 64u, (src ^ mask) & 63u)];
    const uint32_t r1 = pd6[mad_u32(f1, 64u, ((src >> c1) ^ f1) & 63u)];
    const uint32_t r2 = pd6[mad_u32(f2, 64u, ((src >> c2) ^ f2) & 63u)];
    const uint32_t r3 = pd6[mad_u32(mask >> 24, 64u, ((src >> c3) ^ (mask >> 24)) & 63u)];
    return mad_u32(r3, 1u << 24, mad_u32(r2, 1u << 16, mad_u32(r1, 256u, r0)));
}

// The same with every coordinate in the mask: bit i of src -> coordinate i.
__device__ __forceinline__ uint32_t spread24(const uint8_t* pd6, uint32_t src)
{
    const uint8_t* row = pd6 + 0x77 * 64;
    const uint32_t r0 = row[(src & 63u) ^ 0x37u], r1 = row[((src >> 6) & 63u) ^ 0x37u], r2 = row[((src >> 12) & 63u) ^ 0x37u], r3 = row[(src >> 18) ^ 0x37u];
    return mad_u32(r3, 1u << 24, mad_u32(r2, 1u << 16, mad_u32(r1, 256u, r0)));
}

// Quotient of n (below 2^52) by d with inv = 1 / d rounded down, remainder in rem.  On the binary64 pipe, which nothing else uses:
// n and 2^52 + n / d, truncated, are formed in place in the mantissa; the quotient is at most one too small.
__device__ __forceinline__ uint64_t divide52(uint64_t n, uint32_t d, double inv, uint32_t& rem)
{
    const double nd = __hiloint2double((int)(0x43300000u | (uint32_t)(n >> 32)), (int)(uint32_t)n) - 4503599627370496.0;
    const double qd = __fma_rz(nd, inv, 4503599627370496.0);
    uint64_t q = (uint64_t)((uint32_t)__double2hiint(qd) & 0xfffffu) << 32 | (uint32_t)__double2loint(qd);
    rem = (uint32_t)n - (uint32_t)q * d;
    if (rem >= d) { rem -= d; ++q; }
    return q;
}

// Byte permute with a selector made at run time (__byte_perm clears bit 3 of every nibble first: here it is zero, or welcome).
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

template <int kOff>
__device__ __forceinline__ uint32_t lds_at(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(kOff));
    return v;
}

// One slot decision: take slot kPos iff at least C(kPos, t) subsets come before (t = elements still to place).
template <int kPos>
__device__ __forceinline__ void subset_step(uint32_t& col, uint32_t& rho, uint32_t& m, int top)
{
    if (kPos < top) {                                   // warp-uniform
        const uint32_t cnt = lds_at<kPos * 100>(col);   // C(kPos, t); column 0 is stored as 0xffffffff: never taken
        if (rho >= cnt) { rho -= cnt; m |= 1u << kPos; col -= 4u; }
    }
}

__device__ __forceinline__ uint32_t nth_subset(const FastSmem& T, uint32_t k, uint32_t rho, int top)
{
    static_assert(kLowBits == 14, "the slot decisions below cover slots 23..14");
    uint32_t m = 0;
    // byte address (shared window) of C(0, t); it walks down one column each time an element is taken
    uint32_t col = smem_addr(T.pascal) + k * 4u;
    subset_step<23>(col, rho, m, top); subset_step<22>(col, rho, m, top); subset_step<21>(col, rho, m, top);
    subset_step<20>(col, rho, m, top); subset_step<19>(col, rho, m, top); subset_step<18>(col, rho, m, top);
    subset_step<17>(col, rho, m, top); subset_step<16>(col, rho, m, top); subset_step<15>(col, rho, m, top);
    subset_step<14>(col, rho, m, top);
    const uint32_t first = lds_at<kPascalToBase14>(col);   // base14[t] sits right after the 625-entry Pascal table
    return m | (uint32_t)T.r14[first + rho];
}

// The rho-th k-subset of up to 24 slots for k <= 3: one lookup behind a four-word directory (T.sub3 != 0).
// From T.sub2 (k <= 2) it comes in the layout of coords_of.
__device__ __forceinline__ uint32_t small_subset(uint32_t table, uint32_t k, uint32_t rho)
{
    uint32_t first, m;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(first) : "r"(table + k * 4u));
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(m) : "r"(table + (first + rho) * 4u));
    return m;
}

// Result of the index -> point map in a form the consumers expand cheaply:
// three bit planes giving each position a value id (0..7), the table of
// absolute values per id, and the mask of negative positions (masks in the layout of coords_of; bit 31 of neg may be set).
struct Decoded {
    uint32_t p0, p1, p2;
    uint32_t neg;
    uint32_t vals_lo, vals_hi;     // absolute value of id 0..3 / 4..7, one byte each
};

// S2: class of index I (< N) and its class-local index.
__device__ __forceinline__ uint32_t fast_find_class(const FastSmem& T, uint64_t I, uint64_t& local)
{
    uint32_t cls = T.lut[(uint32_t)(I >> T.lut_shift)];
    while (I >= T.off[cls + 1]) ++cls;
    local = I - T.off[cls];
    return cls;
}

// S3-S6.  `mask` = the lanes of the warp that call this together.  kPar = -1: any class.  kPar = 1: all calling lanes
// hold odd classes.  kPar = 0: all calling lanes hold even classes of Golay weight 8, 12 or 16 (both slot groups have
// at most 16 slots).  The specialised forms drop the work the other parity needs (slot decisions above 16, sign deposits).
// Writes d only where `valid`: the caller presets it (zeros for "no block").
template <int kPar>
__device__ __forceinline__ void fast_decode_local(const FastSmem& T, uint32_t cls, uint64_t local, bool valid, uint32_t mask, Decoded& d)
{
    const uint4* D = reinterpret_cast<const uint4*>(T.desc + cls * kFastDescStride);
    const uint4 h = D[0], v = D[1], lw = D[2], mg = D[3];
    const uint32_t B = (h.x >> 8) & 0xff, flags = (h.x >> 16) & 0xff;
    const uint32_t nlev1 = kPar == 1 ? 0u : (h.x >> 24) & 0xf, nlev = valid ? h.x >> 28 : 0u;
    const uint32_t goff = h.y & 0xffff, A = h.y >> 16;
    const bool odd = kPar == 1 || (kPar == -1 && (flags & 1u));
    // the arrangement rank of every calling lane fits 32 bits (all but the largest class of the 48-bit code): no 64-bit division
    const bool rank32 = kPar != -1 && __all_sync(mask, !valid || (flags & kFastFlagRank32));

    // S3: r fastest, then the sign word s, then the arrangement rank p
    uint64_t q;
    uint32_t r;
    if (kPar == 1) { r = (uint32_t)local & 4095u; q = local >> 12; }
    else q = divide52(local, A, __hiloint2double((int)h.w, (int)h.z), r);
    const uint32_t s = kPar == 1 ? 0u : (uint32_t)q & ((1u << B) - 1u);
    const uint64_t p = kPar == 1 ? q : q >> B;

    // S4: Golay codeword
    const uint32_t word_c = T.golay[goff + r], c = word_c & kAllCoords;

    // S5: arrangement.  Group 1 lives on F1(c), group 0 on F0(c); an odd class is one group 0 on all positions.
    const uint32_t F1 = odd ? 0u : c;
    const uint32_t F0 = ~F1 & kAllCoords;
    uint32_t freem = kPar == 1 ? kAllCoords : F1;
    bool in_group0 = kPar == 1;
    uint32_t p0 = 0, p1 = 0, p2 = 0, bit1 = 0, nz0 = 0;
    uint32_t p32 = (uint32_t)p;
    const uint32_t lwords[4] = {lw.x, lw.y, lw.z, lw.w};
    const uint32_t magics[4] = {0u, mg.x, mg.y, mg.z};
    const int maxlev = __reduce_max_sync(mask, nlev);
#pragma unroll
    for (int l = 0; l < kFastMaxLevels; ++l) {
        if (l < maxlev) {
            if (kPar != 1 && !in_group0 && (uint32_t)l >= nlev1) {     // group 1 done: its filler gets id 1
                p0 |= freem;
                if (kPar == -1 && (flags & 8u)) bit1 |= freem;
                freem = F0; in_group0 = true;
            }
            // a lane whose class has fewer steps finds radix 1, k = 0 and all-ones reciprocals in its descriptor: the
            // division returns remainder 0 and the rank unchanged, the empty subset is placed (lanes without a block run
            // the steps of class 0, their result is dropped)
            const uint32_t word = lwords[l];
            const uint32_t radix = word & 0x3fffffu;
            const uint32_t k = (word >> 22) & 31u;
            const uint32_t nfree = (mg.w >> (8 * l)) & 0xffu;            // slots free before this step (0: no step)
            uint32_t rho;
            if (l + 1 == maxlev) {
                // the last step of the warp: what is left of the rank is the step's own digit (lanes whose class has fewer steps
                // hold 0 here and place the empty subset), no division
                rho = p32;
            } else if (l == 0 && !rank32) {
                p32 = (uint32_t)divide52(p, radix, __hiloint2double((int)v.w, (int)v.z), rho);
            } else {
                uint32_t qq = __umulhi(p32, l == 0 ? T.desc[cls * kFastDescStride + kFastDescMagic0] : magics[l]);
                uint32_t rem = p32 - qq * radix;
                if (rem >= radix) { rem -= radix; ++qq; }
                p32 = qq; rho = rem;
            }
            uint32_t a;
            if (kPar == 1 && l == 0 && T.sub2 != 0u && __all_sync(mask, k <= (uint32_t)kSub2MaxK)) {
                a = small_subset(T.sub2, k, rho);                       // odd, first step: every position is free
            } else {
                uint32_t rel;
                if (T.sub3 != 0u && __all_sync(mask, k <= (uint32_t)kSmallSubsetMaxK)) {
                    rel = small_subset(T.sub3, k, rho);                 // few elements: one lookup whatever the number of slots
                } else {
                    int top;
                    if (kPar == 0) top = 16;
                    else if (kPar == 1 && l == 0) top = 24;
                    else top = __reduce_max_sync(mask, nfree);
                    rel = nth_subset(T, k, rho, top);
                }
                a = kPar == 1 && l == 0 ? spread24(T.pd6, rel) : deposit24(T.pd6, rel, freem);
            }
            freem ^= a;
            constexpr int kId0 = kPar == 1 ? 1 : 2;                     // the value id of level l is 2 + l (odd classes alone: 1 + l)
            if ((l + kId0) & 1) p0 |= a;
            if ((l + kId0) & 2) p1 |= a;
            if ((l + kId0) & 4) p2 |= a;
            if (kPar != 0 && (word & (1u << 30))) bit1 |= a;
            if (kPar != 1 && in_group0 && (word >> 31)) nz0 |= a;
        }
    }
    if (kPar != 1 && !in_group0) {
        p0 |= freem;
        if (kPar == -1 && (flags & 8u)) bit1 |= freem;
        freem = F0;
    }
    if (kPar != 0 && (flags & 16u)) bit1 |= freem;              // filler of group 0 keeps id 0
    if (kPar != 1 && (flags & 4u)) nz0 |= freem;

    // S6: signs
    uint32_t neg;
    if (kPar == 1) {
        neg = c ^ bit1;                                         // 1 mod 4 on F0, 3 mod 4 on F1
    } else {
        // the bits of s go to the positions that carry a sign (F1 and the nonzero ones of F0) in ascending order, except the
        // last F1 position: its sign makes the sum 0 mod 8
        const uint32_t last_f1 = 1u << (((word_c & kLastPosBits) * kLastPosGather) >> 27);      // bit 31 for the zero word
        uint32_t neg_even = deposit24(T.pd6, s, (F1 | (odd ? 0u : nz0)) & ~last_f1);
        if ((__popc(neg_even & F1) + (flags >> 1)) & 1u) neg_even |= last_f1;
        neg = odd ? (c ^ bit1) : neg_even;
    }
    if (valid) {
        d.p0 = p0; d.p1 = p1; d.p2 = p2; d.neg = neg;
        if (kPar == 1) {
            const uint2 vo = *reinterpret_cast<const uint2*>(T.desc + cls * kFastDescStride + kFastDescValsOdd);
            d.vals_lo = vo.x; d.vals_hi = vo.y;
        } else {
            d.vals_lo = v.x; d.vals_hi = v.y;
        }
    }
}

__device__ __forceinline__ void fast_decode(const FastSmem& T, uint64_t I, bool valid, Decoded& d)
{
    d.p0 = d.p1 = d.p2 = d.neg = d.vals_lo = d.vals_hi = 0u;
    uint64_t local = 0;
    const uint32_t cls = valid ? fast_find_class(T, I, local) : 0u;
    fast_decode_local<-1>(T, cls, local, valid, kFullMask, d);
}

// ---- expansion helpers -------------------------------------------------------
constexpr uint32_t kPairs = 0x11111111u;     // bit r of every nibble: the coordinates 6 g + 2 r, 6 g + 2 r + 1 of the four groups

// Nibble n + 2 g of the result = bits (x, y, z) of coordinate 6 g + 2 r + n.
template <int r>
__device__ __forceinline__ uint32_t selectors(uint32_t x, uint32_t y, uint32_t z)
{
    return ((x >> r) & kPairs) | ((r == 0 ? y << 1 : y >> (r - (r > 0))) & (kPairs << 1)) | ((z << (2 - r)) & (kPairs << 2));
}

// Byte i of the result = 0xff where bit 4 i of x is set, else 0 (i = 0..3).  The other bits of x may be anything: as part of the
// selector they choose an equal byte or ask for its sign, which is the byte again.
__device__ __forceinline__ uint32_t ones_where(uint32_t x) { return prmt(0xff00ff00u, 0xff00ff00u, x); }

// The 24 coordinates as signed bytes, coordinate i in byte (i & 3) of word (i >> 2).
__device__ __forceinline__ void expand_bytes(const Decoded& d, uint32_t out[6])
{
    uint32_t t[6];                            // t[r + 3 q]: coordinates 2 r, 2 r + 1 of groups 2 q and 2 q + 1
    const uint32_t sel[3] = {selectors<0>(d.p0, d.p1, d.p2), selectors<1>(d.p0, d.p1, d.p2), selectors<2>(d.p0, d.p1, d.p2)};
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const uint32_t neg = ones_where(d.neg >> (j % 3 + (j < 3 ? 0 : 16)));
        const uint32_t a = prmt(d.vals_lo, d.vals_hi, sel[j % 3] >> (j < 3 ? 0 : 16));
        t[j] = (a ^ neg) + (neg & 0x01010101u);                                   // negated bytes are never zero
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        out[3 * q] = __byte_perm(t[3 * q], t[3 * q + 1], 0x5410);
        out[3 * q + 1] = __byte_perm(t[3 * q + 2], t[3 * q], 0x7610);
        out[3 * q + 2] = __byte_perm(t[3 * q + 1], t[3 * q + 2], 0x7632);
    }
}

// The 24 dequantized weights bf16_rn(gain * x_i) as 12 packed pairs (weight 2j in the low half of w[j]).
// All lanes of the warp must call this together: when no lane uses a value id above 3 (codes with few distinct
// values per class) the upper half of the value table is not formed and the sign takes its place in the selectors: ids 4..7 are
// the negated values then.
// The bit planes become selectors by masks and shifts alone because of where the coordinates lie in them (coords_of): 62 instructions
// with the products; with bit i = coordinate i the planes were spread arithmetically, 122 instructions (three-layer step 93.8 -> 87.7 us).
__device__ __forceinline__ void expand_bf16(const Decoded& d, float gain, uint32_t w[12])
{
    // bf16(gain * a) for the value ids; float(a) by the 2^23 trick (a <= 28)
    auto products = [&](uint32_t src, int i) {
        const float a0 = __uint_as_float(__byte_perm(src, 0x4b000000u, i ? 0x7442 : 0x7440)) - 8388608.f;
        const float a1 = __uint_as_float(__byte_perm(src, 0x4b000000u, i ? 0x7443 : 0x7441)) - 8388608.f;
        const __nv_bfloat162 b = __floats2bfloat162_rn(gain * a0, gain * a1);
        return *reinterpret_cast<const uint32_t*>(&b);
    };
    const uint32_t v01 = products(d.vals_lo, 0), v23 = products(d.vals_lo, 1);
    const uint32_t lo03 = __byte_perm(v01, v23, 0x6420), hi03 = __byte_perm(v01, v23, 0x7531);
    if (__any_sync(kFullMask, d.p2 != 0u)) {
        const uint32_t v45 = products(d.vals_hi, 0), v67 = products(d.vals_hi, 1);
        const uint32_t lo47 = __byte_perm(v45, v67, 0x6420), hi47 = __byte_perm(v45, v67, 0x7531);
        const uint32_t sel[3] = {selectors<0>(d.p0, d.p1, d.p2), selectors<1>(d.p0, d.p1, d.p2), selectors<2>(d.p0, d.p1, d.p2)};
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int r = j % 3, q = j / 3;
            const uint32_t s16 = q ? sel[r] >> 16 : sel[r];
            const uint32_t lob = prmt(lo03, lo47, s16);
            const uint32_t hib = prmt(hi03, hi47, s16) ^ (ones_where(d.neg >> (r + 16 * q)) & 0x80808080u);
            w[6 * q + r] = __byte_perm(lob, hib, 0x5140);
            w[6 * q + 3 + r] = __byte_perm(lob, hib, 0x7362);
        }
    } else {
        const uint32_t neg03 = hi03 ^ 0x80808080u;
        const uint32_t sel[3] = {selectors<0>(d.p0, d.p1, d.neg), selectors<1>(d.p0, d.p1, d.neg), selectors<2>(d.p0, d.p1, d.neg)};
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int r = j % 3, q = j / 3;
            const uint32_t s16 = q ? sel[r] >> 16 : sel[r];
            const uint32_t lob = prmt(lo03, lo03, s16), hib = prmt(hi03, neg03, s16);
            w[6 * q + r] = __byte_perm(lob, hib, 0x5140);
            w[6 * q + 3 + r] = __byte_perm(lob, hib, 0x7362);
        }
    }
}

}  // namespace llvq
