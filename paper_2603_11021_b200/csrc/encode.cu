// Encoder side of the library: nearest point of the code to a real vector (Sec. 3.1, Euclidean and angular
// scoring), point -> index (Sec. 3.2, the inverse of the dequantizer's steps) and packing of the stored fields.
// The paper defers the search itself to the literature; the search here is coset decoding of the whole lattice
// (exact for the unbounded lattice) plus a policy that keeps the result inside the shells of the code.
#include "llvq.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "ctx.h"
#include "tables.h"

using namespace llvq;

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr uint32_t kFlagSearchGaveUp = 4u; // LLVQ_FLAG_SEARCH_GAVE_UP

constexpr int kMaxShell = 53;              // llvq_create's limit
constexpr int kMaxCand = 64;               // cosets re-scored in binary64 per search; more (massive ties) means all 8192 are

// ---- the careful search: one vector per warp ----

// Units of its first stage: costs and moves are whole numbers of 1 / kCostScale.  The largest rounding error
// of a coordinate costs 1/4, i.e. 2046: sixteen of them stay below 2^15.
constexpr float kCostScale = 8184.f;
// Two cosets whose first-stage costs differ by more than this are in the same order in exact arithmetic: a cost carries at
// most 25 roundings of half a unit (24 coordinates and one move) and 0.1 from the binary32 errors, twice 12.6 is 25.2.
constexpr uint32_t kCostMargin = 26u;
constexpr uint32_t kParityBit = 0x8000u;   // where a cost carries the parity of its sum of z (adding costs adds the parities mod 2)
constexpr uint32_t kParityCode = 0x7676u;  // a byte-permute selector XOR this trades places with the one of the other parity
constexpr uint32_t kSelEven = 0x3244u;     // {high half of the first operand} stays high, low half zero; ^ kParityCode: moved low

// Per-warp scratch of the careful search.
struct __align__(128) WarpTables {
    uint2 nib[2][6][16];    // [parity][4 coordinates][bit pattern n]: {cost | move << 16, parity code | move of pattern ~n << 16}; rows of 128 bytes
    uint4 pk[24][2];        // [coordinate, octad by octad][parity] w(b), w(b + 2), w(b + 2), w(b) for offset b = parity:
                            //  w = cost | parity of z << 15 | cost of the other neighbour << 16
    uint32_t cand[kMaxCand - 1];
    uint32_t ncand;
};
static_assert((kMaxCand - 1) * 24 <= sizeof(WarpTables::nib) && 24 * sizeof(double) <= sizeof(WarpTables::pk), "the candidates' points and the input take the tables' place");

// Nibbles of the octad patterns [octad][a = 1..3] (x = 0), times 8 (the row bytes of WarpTables::nib they select): patterns are
// linear in (x, a), so the address of a pattern is that of (x, a & 4) XOR one of these.
struct PatternSteps {
    uint32_t lo[3][4], hi[3][4];
};

// sum of the values of lanes 0..23, added in lane order, one binary64 rounding per addition (every lane gets the sum)
__device__ __forceinline__ double seq_sum24(double v)
{
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < 24; ++i) acc = __dadd_rn(acc, __shfl_sync(kFull, v, i));
    return acc;
}

__device__ __forceinline__ uint2 lds64(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}

// kParityCode where the parity carried by a cost is odd, else 0 (one multiply-high beside the mask)
__device__ __forceinline__ uint32_t parity_code(uint32_t cost) { return __umulhi(cost & kParityBit, kParityCode << 17); }

// The point of coset (pi, codeword c) nearest to u (one coordinate per lane) in binary64, one rounding per operation: the
// rounded z, with the first coordinate of largest error moved to its other neighbour if the sum rule fails.  alone = no
// other point of the coset comes within 2e-6 of its rounding errors.
__device__ __forceinline__ int coset_point(double u, uint32_t c, int pi, int lane, bool& alone)
{
    const bool mine = lane < 24;
    const int b = pi + 2 * (int)((c >> lane) & 1u);
    const double tt = __dmul_rn(__dsub_rn(u, (double)b), 0.25);
    const double z = rint(tt);
    const double err = __dsub_rn(tt, z), mag = fabs(err);
    int x = mine ? b + 4 * (int)z : 0;
    const int sum = __reduce_add_sync(kFull, x);
    if ((sum & 7) != (pi ? 4 : 0)) {
        // the first coordinate with the largest |error| moves by 4 (binary64 magnitudes compare like their bit patterns)
        const unsigned long long key = mine ? (unsigned long long)__double_as_longlong(mag) : 0ull;
        const uint32_t top = __reduce_max_sync(kFull, (uint32_t)(key >> 32));
        const bool in_top = mine && (uint32_t)(key >> 32) == top;
        const uint32_t low = __reduce_max_sync(kFull, in_top ? (uint32_t)key : 0u);
        const int who = __ffs(__ballot_sync(kFull, in_top && (uint32_t)key == low)) - 1;
        const double largest = __longlong_as_double((long long)((unsigned long long)top << 32 | low));
        alone = __popc(__ballot_sync(kFull, mine && mag > largest - 1.0e-6)) == 1;
        if (lane == who) x += err > 0.0 ? 4 : (err < 0.0 ? -4 : 4);
    } else {
        alone = __all_sync(kFull, !mine || mag < 0.5 - 1.0e-6);
    }
    return x;
}

// Nearest point of the unbounded lattice to u (one coordinate per lane, lanes 0..23), as nearest_pairs below finds it, for the
// inputs to which two cosets are so close that whole-number costs do not tell them apart (about one in sixty).
// First stage: per parity and octad pattern {w, ~w} the best cost for an even and for an odd sum of z (a move included where the
// rounded z has the other parity), the minimum over the 512 triples of patterns that are codewords (GolayTrio); a lane holds (parity, x,
// half of the a).  Every coset within kCostMargin of the smallest cost is then listed and evaluated in binary64, coordinate by
// coordinate in lane order, one rounding per operation: its point, and, if there are several, the squared distance as the sum over
// the coordinates in order.  The smallest distance wins, the lowest (parity, codeword position) among equal ones; inside a coset the
// first coordinate with the largest error moves.  The result does not depend on the first stage's rounding.  Returns the coordinate of
// this lane (0 for lanes >= 24) and the squared norm of the point; unique = every other lattice point is farther from u by a margin
// far above any binary64 rounding.
// kTogether: the squared distances of several candidates are formed a lane each.  With 16 warps there is little to hide a chain of 24 additions per candidate
// behind (two lanes per vector, 174 763 integer vectors EUCLIDEAN 915 -> 710 us, Gaussian ones 215 -> 213); with 24 the code costs searches that need none of
// it more than it gains (52 000 Gaussian vectors 109.5 -> 111.5 us, 30 000 on half integers 97 -> 100).
template <bool kTogether>
__device__ __forceinline__ int nearest_careful_from(WarpTables& W, const GolayTrio& S, const PatternSteps& steps, const uint32_t (&row)[6],
                                                    const uint32_t* __restrict__ golay, const uint16_t* __restrict__ pos_by_low12, double u, int lane, int& norm2, bool& unique)
{
    const float uq = __shfl_sync(kFull, (float)u, lane < 24 ? S.coord[lane] : lane);   // octad order
    if (lane < 24) {
        uint32_t w[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            // rounding by adding 1.5 * 2^23 (the parity of z is then the last bit), whole numbers from adding 2^23: no conversions
            const float t = (uq - (float)b) * 0.25f, tr = t + 12582912.f;
            const float err = t - (tr - 12582912.f);
            const float cost = fmaf(err * err, kCostScale, 8388608.f), move = fmaf(fabsf(err), -2.f * kCostScale, 8388608.f + kCostScale);
            w[b] = __byte_perm(__float_as_uint(cost), __float_as_uint(move), 0x5410) | (__float_as_uint(tr) << 15 & kParityBit);
        }
        W.pk[lane][0] = make_uint4(w[0], w[2], w[2], w[0]);
        W.pk[lane][1] = make_uint4(w[1], w[3], w[3], w[1]);
    }
    if (lane == 0) W.ncand = 0u;
    __syncwarp();
    const int pi = lane >> 4;
    uint32_t octad_sum[3];                                      // low half: cost of a pattern + that of its complement | parity between them << 15
    // tables per nibble of an octad: lane = (parity, bit pattern), one group of 4 coordinates after the other
    {
        const int n = lane & 15;
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(&W.pk[0][pi]);
        uint32_t at[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) at[k] = base + 32u * (uint32_t)k + 8u * (uint32_t)((n >> k) & 1);
#pragma unroll
        for (int g = 0; g < 6; ++g) {
            uint2 v[4];                                         // this pattern's and the complement's choice at each coordinate
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = lds64(at[k] + 128u * g);
            const uint32_t sum = (v[0].x + v[1].x) + (v[2].x + v[3].x), sum_c = (v[0].y + v[1].y) + (v[2].y + v[3].y);
            const uint32_t move = __vminu2(__vimin3_u16x2(v[0].x, v[1].x, v[2].x), v[3].x);
            const uint32_t move_c = __vminu2(__vimin3_u16x2(v[0].y, v[1].y, v[2].y), v[3].y);
            W.nib[pi][g][n] = make_uint2((sum & 0x7fffu) | (move & 0xffff0000u), parity_code(sum) | (move_c & 0xffff0000u));
            octad_sum[g >> 1] = (g & 1 ? octad_sum[g >> 1] : 0u) + sum + sum_c;
        }
    }
    __syncwarp();
    // best costs of octad patterns: lane = (parity, h, x) scores those with a, b, c = 4 h .. 4 h + 3.  The 16 lanes of a parity
    // read one row of 128 bytes at a time: no bank conflicts
    uint32_t e[3][4];
#pragma unroll
    for (int o = 0; o < 3; ++o) {
        const uint32_t kd = __byte_perm(octad_sum[o] & 0x7fffu, 0u, 0x1010);
        const uint32_t sel0 = o == 2 && pi ? kSelEven ^ kParityCode : kSelEven;      // octad 2 of parity 1 is kept odd half first
        const uint32_t selc = parity_code(octad_sum[o]) ^ sel0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint2 lo = lds64(row[2 * o] ^ steps.lo[o][j]), hi = lds64(row[2 * o + 1] ^ steps.hi[o][j]);
            const uint32_t cost = __byte_perm(lo.x + hi.x, 0u, 0x1010);
            const uint32_t w = cost + __byte_perm(__vminu2(lo.x, hi.x), 0u, lo.y ^ hi.y ^ sel0);
            const uint32_t wc = kd - cost + __byte_perm(__vminu2(lo.y, hi.y), 0u, lo.y ^ hi.y ^ selc);
            e[o][j] = __vminu2(w, wc);
        }
    }
    uint32_t best_a[4];
    {
        // pairs (a, b) = (4 h + i, (4 h) ^ j): c = i ^ j.  The other half's b and c come from the lane that holds them
        uint32_t b[8], c[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            b[j] = e[1][j];
            b[4 + j] = __shfl_xor_sync(kFull, e[1][j], 8);
            c[j] = __shfl_sync(kFull, e[2][j], lane & ~8);
            c[4 + j] = __shfl_sync(kFull, e[2][j], lane | 8);
        }
        uint32_t bs[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) bs[j] = __byte_perm(b[j], 0u, 0x1032);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            best_a[i] = 0xffffffffu;
            const uint32_t ev = __byte_perm(e[0][i], 0u, 0x1010), od = __byte_perm(e[0][i], 0u, 0x3232);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t two = __viaddmin_u16x2(od, bs[j], ev + b[j]);         // {even, odd} sum of two octads
                best_a[i] = __viaddmin_u16x2(two, c[i ^ j], best_a[i]);
            }
            best_a[i] = min(best_a[i] & 0xffffu, best_a[i] >> 16);
        }
    }
    const uint32_t best = __reduce_min_sync(kFull, min(min(best_a[0], best_a[1]), min(best_a[2], best_a[3])));
    const uint32_t thr = best + kCostMargin;
    // list the cosets within the margin: for every (parity, x, a) that holds one, the 64 codewords behind it, two per lane
    for (int i = 0; i < 4; ++i) {
        for (uint32_t holders = __ballot_sync(kFull, best_a[i] <= thr); holders; holders &= holders - 1u) {
            const int owner = __ffs(holders) - 1;
            const int po = owner >> 4, x = owner & 7, a = 4 * ((owner >> 3) & 1) + i, b = lane & 7;
            const uint32_t nib = (uint32_t)__cvta_generic_to_shared(&W.nib[po][0][0]);
            const uint32_t p0 = S.pat[0][x * 8 + a] ^ (lane & 8 ? 255u : 0u), p1 = S.pat[1][x * 8 + b] ^ (lane & 16 ? 255u : 0u);
            uint32_t cost = 0, code = 0, move = 0xffffffffu;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const uint32_t p = g < 2 ? p0 : p1;
                const uint2 v = lds64(nib + 128u * g + 8u * ((p >> (4 * (g & 1))) & 15u));
                cost += v.x; code ^= v.y; move = __vminu2(move, v.x);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint32_t p2 = S.pat[2][x * 8 + (a ^ b)] ^ (e ? 255u : 0u);
                const uint2 v4 = lds64(nib + 512u + 8u * (p2 & 15u)), v5 = lds64(nib + 640u + 8u * (p2 >> 4));
                const uint32_t mv = __vminu2(move, __vminu2(v4.x, v5.x)) >> 16;
                const bool odd = ((code ^ v4.y ^ v5.y) & 0xffffu) != 0u;
                const uint32_t total = ((cost + v4.x + v5.x) & 0xffffu) + (odd != (po != 0) ? mv : 0u);
                if (total <= thr) {
                    const uint32_t slot = atomicAdd(&W.ncand, 1u);
                    const uint32_t c = (S.word[0][x * 8 + a] ^ (lane & 8 ? S.ones[0] : 0u)) |
                                       (S.word[1][x * 8 + b] ^ (lane & 16 ? S.ones[1] : 0u)) |
                                       (S.word[2][x * 8 + (a ^ b)] ^ (e ? S.ones[2] : 0u));
                    if (slot < (uint32_t)(kMaxCand - 1)) W.cand[slot] = (uint32_t)po << 24 | c;
                }
            }
        }
    }
    __syncwarp();
    const uint32_t listed = W.ncand;
    int best_x;
    if (listed == 1u) {
        const uint32_t k = W.cand[0];
        best_x = coset_point(u, k & 0xffffffu, (int)(k >> 24), lane, unique);
    } else if (kTogether && listed <= (uint32_t)(kMaxCand - 1)) {
        // the candidates' points one after the other, their squared distances a lane each: 24 dependent additions for all of them together
        unique = false;
        int8_t* const points = reinterpret_cast<int8_t*>(W.nib);                    // the costs are done with
        double* const us = reinterpret_cast<double*>(W.pk);
        if (lane < 24) us[lane] = u;
        for (uint32_t t = 0; t < listed; ++t) {
            const uint32_t k = W.cand[t];
            bool alone;
            const int x = coset_point(u, k & 0xffffffu, (int)(k >> 24), lane, alone);
            if (lane < 24) points[24 * t + (uint32_t)lane] = (int8_t)x;
        }
        __syncwarp();
        unsigned long long best_d2 = ~0ull;                                         // the bits of numbers that are not negative are in their order
        uint32_t best_id = 0xffffffffu, best_t = 0;
        for (uint32_t t = (uint32_t)lane; t < listed; t += 32u) {
            const uint32_t k = W.cand[t], id = k >> 24 << 12 | __ldg(pos_by_low12 + (k & 0xfffu));
            double acc = 0.0;
#pragma unroll
            for (int j = 0; j < 6; ++j) {
                const uint32_t four = reinterpret_cast<const uint32_t*>(points)[6u * t + (uint32_t)j];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double dd = __dsub_rn(us[4 * j + i], (double)(int8_t)(four >> (8 * i)));
                    acc = __dadd_rn(acc, __dmul_rn(dd, dd));
                }
            }
            const unsigned long long d2 = (unsigned long long)__double_as_longlong(acc);
            if (d2 < best_d2 || (d2 == best_d2 && id < best_id)) { best_d2 = d2; best_id = id; best_t = t; }
        }
        const uint32_t hi = __reduce_min_sync(kFull, (uint32_t)(best_d2 >> 32));
        const bool in_hi = (uint32_t)(best_d2 >> 32) == hi;
        const uint32_t lo = __reduce_min_sync(kFull, in_hi ? (uint32_t)best_d2 : 0xffffffffu);
        const bool nearest = in_hi && (uint32_t)best_d2 == lo;
        const uint32_t first = __reduce_min_sync(kFull, nearest ? best_id : 0xffffffffu);
        best_t = __shfl_sync(kFull, best_t, __ffs(__ballot_sync(kFull, nearest && best_id == first)) - 1);
        best_x = lane < 24 ? (int)points[24u * best_t + (uint32_t)lane] : 0;
    } else {
        unique = false;
        const uint32_t n = listed > (uint32_t)(kMaxCand - 1) ? 8192u : listed;      // too many near-ties to list: every coset
        double best_d2 = 1.0e300;
        uint32_t best_id = 0xffffffffu;
        best_x = 0;
        for (uint32_t t = 0; t < n; ++t) {
            uint32_t id = t, c;
            if (listed > (uint32_t)(kMaxCand - 1)) c = __ldg(golay + (t & 4095u));
            else { c = W.cand[t] & 0xffffffu; id = W.cand[t] >> 24 << 12 | __ldg(pos_by_low12 + (c & 0xfffu)); }
            bool alone;
            const int x = coset_point(u, c, (int)(id >> 12), lane, alone);
            const double dd = __dsub_rn(u, (double)x);
            const double d2 = seq_sum24(lane < 24 ? __dmul_rn(dd, dd) : 0.0);
            if (d2 < best_d2 || (d2 == best_d2 && id < best_id)) { best_d2 = d2; best_id = id; best_x = x; }
        }
    }
    norm2 = __reduce_add_sync(kFull, best_x * best_x);
    __syncwarp();
    return best_x;
}

// Where the nibbles of pattern (x, 4 h) of every octad are in W.
__device__ __forceinline__ void pattern_rows(WarpTables& W, const GolayTrio& S, int lane, uint32_t (&row)[6])
{
#pragma unroll
    for (int o = 0; o < 3; ++o) {
        const uint32_t p = S.pat[o][(lane & 7) * 8 + ((lane >> 1) & 4)], t = (uint32_t)__cvta_generic_to_shared(&W.nib[lane >> 4][2 * o][0]);
        row[2 * o] = t ^ (p & 15u) * 8u;
        row[2 * o + 1] = (t + 128u) ^ (p >> 4) * 8u;
    }
}

__device__ __noinline__ int nearest_careful(WarpTables& W, const GolayTrio& S, const PatternSteps& steps, const uint32_t* __restrict__ golay,
                                            const uint16_t* __restrict__ pos_by_low12, double u, int lane, int& norm2, bool& unique)
{
    uint32_t row[6];
    pattern_rows(W, S, lane, row);
    return nearest_careful_from<true>(W, S, steps, row, golay, pos_by_low12, u, lane, norm2, unique);
}

// ---- the search: two lanes per vector ----

// Units of the costs below: whole numbers of 1 / kPairScale.  Three octads cost at most 6 of the squares of the half spacing
// that a coordinate's offset is measured in (an octad with a move at most 2, two of them together at most 4 before the better
// combination is taken), 65400: 16 bits.
constexpr float kPairRoot = 104.403065f;   // sqrt(kPairScale)
constexpr float kPairScale = 10900.f;
// As kCostMargin: a sum of 24 costs carries 24 roundings of half a unit and 0.6 from binary32 errors (|u| up to 30).
constexpr uint32_t kPairMargin = 26u;
// The costs of the eight codewords of one triple of patterns are formed again from binary32 sums, 2.1 units off at most: what lies
// more than this above the smallest whole-number cost (12.6 off at most) is farther than the coset that has it.
constexpr uint32_t kWordMargin = 15u;

// Two forms of the kernel: kPairs = two lanes per vector, 16 warps of 16 vectors, all warps of the CTA in step (below); else one warp
// per vector, 24 warps, nearest_careful alone.
template <bool kPairs> constexpr int kEncWarps = kPairs ? 16 : 24;
template <bool kPairs> constexpr int kEncVecs = kPairs ? 16 : 1;          // vectors of a warp
// Shared memory of a warp: costs of the patterns of the six nibbles, [nibble][pattern][vector] (or the scratch of nearest_careful), and the
// inputs, [coordinate][vector].
constexpr uint32_t kNibRow = 16 * sizeof(uint2), kNibTable = 16 * kNibRow, kNibBytes = 6 * kNibTable;
static_assert(sizeof(WarpTables) + 24 <= kNibBytes, "nearest_careful works where the costs were");
template <bool kPairs> constexpr uint32_t kEncWarpBytes = kPairs ? kNibBytes : (uint32_t)sizeof(WarpTables) + 128u;
template <bool kPairs> constexpr size_t kEncSmem = kEncWarps<kPairs> * (kEncWarpBytes<kPairs> + 24 * kEncVecs<kPairs> * sizeof(float)) + sizeof(GolayTrio) + (kPairs ? kNibTable : 128);

// The patterns of a codeword on the three octads are x ^ a, x ^ b, x ^ a ^ b with x and a, b from two [8, 4] codes whose sums are
// the even words (Turyn's construction; GolayTrio has the order of coordinates in which these are the same two for every octad).
__device__ constexpr uint32_t turyn_a(uint32_t a)
{
    constexpr uint32_t a0 = kTurynA[0], a1 = kTurynA[1], a2 = kTurynA[2];
    return (a & 1 ? a0 : 0u) ^ (a & 2 ? a1 : 0u) ^ (a & 4 ? a2 : 0u);
}
__device__ constexpr uint32_t turyn_x(uint32_t x)
{
    constexpr uint32_t x0 = kTurynX[0], x1 = kTurynX[1], x2 = kTurynX[2];
    return (x & 1 ? x0 : 0u) ^ (x & 2 ? x1 : 0u) ^ (x & 4 ? x2 : 0u);
}

__device__ __forceinline__ void sts64(uint32_t a, uint32_t x, uint32_t y)
{
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

__device__ __forceinline__ uint32_t half_of(uint32_t v, int pi) { return pi ? v >> 16 : v & 0xffffu; }

// Costs of a part of the coordinates for an even and for an odd sum of its z, parity 0 of the lattice in the low halves, parity 1 in the high ones.
struct Cost {
    uint32_t even, odd;
};
__device__ __forceinline__ Cost operator+(const Cost& a, const Cost& b)
{
    return {__viaddmin_u16x2(a.odd, b.odd, a.even + b.even), __viaddmin_u16x2(a.odd, b.even, a.even + b.odd)};
}

// Cost of octad pattern `p` (of the a-code; the tables' addresses carry the x) or its complement, whichever is cheaper; lo, hi:
// where the costs of the octad's nibbles 0 are, with the x in the row bits.
__device__ __forceinline__ Cost pattern_cost(uint32_t lo, uint32_t hi, uint32_t p, uint32_t octad)
{
    const uint2 l = lds64((lo ^ (p & 15u) * kNibRow) + octad * 2u * kNibTable), h = lds64((hi ^ (p >> 4) * kNibRow) + octad * 2u * kNibTable);
    const uint2 lc = lds64((lo ^ (~p & 15u) * kNibRow) + octad * 2u * kNibTable), hc = lds64((hi ^ (~p >> 4 & 15u) * kNibRow) + octad * 2u * kNibTable);
    Cost c;
    c.even = __viaddmin_u16x2(lc.y, hc.y, __viaddmin_u16x2(lc.x, hc.x, __viaddmin_u16x2(l.y, h.y, l.x + h.x)));
    c.odd = __viaddmin_u16x2(lc.y, hc.x, __viaddmin_u16x2(lc.x, hc.y, __viaddmin_u16x2(l.y, h.x, l.x + h.y)));
    return c;
}

// What a search returns; both lanes of a vector hold the same, but for x: half of the point each.
struct Nearest {
    uint32_t x[3];          // coordinates 12 q .. 12 q + 11 as signed bytes (q = 0, 1: the lane of the pair; the halves of the warp)
    int norm2;              // squared norm of the point
    double dot;             // its inner product with u
    bool unique;            // every other lattice point is farther from u by a margin far above any binary64 rounding
};

// <u, x>, a coordinate per lane.
__device__ __forceinline__ double dot_of_warp(double u, int xi)
{
    double dot = u * (double)xi;
#pragma unroll
    for (int o = 16; o; o >>= 1) dot += __shfl_xor_sync(kFull, dot, o);
    return dot;
}

// More vectors per SM than this: two lanes take a vector, else a warp does.  Two lanes per vector use the chip best, but a CTA works on 256 vectors at a time
// for some 15 us.  Gaussian inputs, us for a warp per vector / two lanes by vectors per SM (of 148):
//   EUCLIDEAN shells 2..13  260 87 / 100  330 104 / 112  384 114 / 114  450 128 / 126;  both are equal at 265 (2..3), 365 (2..5), 385 (2..8), 430 (2..20), 460 (2..24)
//   ANGULAR   shells 2..13  100 143 / 181  136 184 / 190  150 200 / 193  200 255 / 200;  both are equal at 115 (2..3), 130 (2..5), 136 (2..8), 148 (2..20), 145 (2..24)
// EUCLIDEAN inputs on a coarse grid, many of which have several nearest cosets, would be better off with a warp per vector (us, a warp, before there were two forms / two lanes: 60 000
// vectors of integers 222 / 300, halves 158 / 203, quarters 140 / 162; 174 763 vectors 532 / 670, 376 / 407, 332 / 313), which the host cannot know; a block
// that changes over when it meets them costs all inputs 2.5 % and gains those 4 %.
constexpr uint64_t kPairsFromEuclidean = 384, kPairsFromAngular = 136;
// No more vectors than this left in a CTA: all of them go to nearest_careful.  The two metrics' largest cases, us: never (0) 817 / 869, 16 690 / 745, 40 670 / 721,
// 80 656 / 712.
constexpr int kFew = 40;
// The longest list: as many as shared memory has room for.  174 763 integer vectors 710 us with 48, 670 with 96; Gaussian ones 213 with either.
constexpr uint32_t kPendingMost = 96, kPendingEnough = 14;
// A vector of a CTA that waits for nearest_careful, and the answer.
struct Pending {
    double rn, radius, dot;
    const float* v;
    int norm2;
    bool unique;
    alignas(4) int8_t x[24];
};
struct PendingList {
    Pending list[kPendingMost];
    uint32_t count;
};

// Nearest point of the unbounded lattice to u = (v rn) radius, every operation rounded once to binary64 (v[16 i] holds coordinate i; v s1 s2
// is u in binary32; all in units of the integer coordinates).  Every lattice point is b + 4 z with b_i = parity + 2 c_i, c a
// Golay codeword, and sum z = parity (mod 2) (the sum rules of Sec. 2.4: all Golay weights are multiples of 4).  For each of the
// 2 x 4096 cosets the best z is the rounded one, with the coordinate of largest rounding error moved to its other neighbour when
// the sum rule fails.
// Two stages.  The first finds the coset of smallest cost in whole numbers.  Every part of the coordinates has
// two costs, for an even and for an odd sum of its z, 16 bits each for either parity of the lattice in one word; two parts combine by
// two additions and two add-and-minimum.  Coordinates combine to pairs and nibbles (tables in shared memory), these to the 64 patterns
// {w, ~w} of an octad, and the Golay code is the 512 triples (x, a, b) of such patterns (Turyn's construction).  Choosing a
// neighbour per part moves more than one coordinate only where that costs no less than one move, so this is the minimum over the
// cosets.  A lane makes three of the six tables and takes four of the eight x.  If the best (x, parity) leads all others by more than the
// rounding of the costs, its 64 triples are looked at again, then the best triple's eight codewords, and the coset that is left is
// evaluated as the oracle does: coordinate by coordinate, one binary64 rounding per operation, the first coordinate with the
// largest error moving where the sum rule asks for it.  Wherever a second candidate lies within the margin (one vector in
// sixty) the vector goes to nearest_careful, one per warp.  So the result does not depend on the first stage's rounding.
// Bound: the logic pipe (62 % busy, issue 57 %) and what a block barrier costs.  Against nearest_careful for every vector, 24 warps: 818 -> 400 warp
// instructions per search; 699 050 vectors EUCLIDEAN 1063 -> 669 us, 174 763 ANGULAR on shells 2..12 2035 -> 722 us (of it 2035 -> 1430 by the
// radii left out).
// All threads of the CTA call this together; `wanted` = this lane's vector is to be searched, `waiting` = it is on the list for
// nearest_careful at `spot`, `few` = so few of the CTA's are left that nearest_careful takes them all.  Returns whether r is the answer
// for this lane's vector.  (The list is worked off when almost every warp gets one of it, not after every search: 709 -> 695 us EUCLIDEAN.)
// The block barriers keep the warps in step: the code is long (some 1500 instructions once through, half of them four times), and warps that are
// each somewhere else in it fetch more instructions than the SM delivers (2 warps per scheduler: 3.0 of 5.8 stall cycles per
// instruction were fetches; 0.1 of 3.9 with the barriers, 1329 -> 942 us for the 174 763 vectors of the ANGULAR case).  One per search:
// with one per x the warps read their tables all at the same time and then computed (737 and 796 us, 709 and 762 with one per search).
__device__ __forceinline__ bool nearest_pairs(uint32_t nib, const float* v, const GolayTrio& S, const PatternSteps& steps, const uint32_t* __restrict__ golay,
                                              const uint16_t* __restrict__ pos_by_low12, WarpTables& careful, PendingList& pending, float s1, float s2, double rn,
                                              double radius, bool wanted, bool& waiting, uint32_t& spot, bool few, int warp, int lane, Nearest& r)
{
    const int q = lane >> 4;
    bool settled = false;
    if (!few) {
        const uint32_t tab = nib + 8u * (uint32_t)(lane & 15);
        const uint32_t* const coords = reinterpret_cast<const uint32_t*>(S.coord);
#pragma unroll 1
        for (uint32_t g = 3u * (uint32_t)q; g < 3u * (uint32_t)q + 3u; ++g) {
            const uint32_t four = coords[g];
            Cost n[4][2];                                            // by bit of the codeword
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float t0 = v[16u * ((four >> (8 * k)) & 31u)] * s1 * s2 * 0.25f;
                uint32_t w[2][2];
#pragma unroll
                for (int pi = 0; pi < 2; ++pi) {
                    // rounding by adding 1.5 * 2^23 (the parity of z is then the last bit), whole numbers from adding 2^23: no conversions
                    const float t = pi ? t0 - 0.25f : t0, tr = t + 12582912.f, err = t - (tr - 12582912.f);
                    const float a = fabsf(err) * kPairRoot, b = kPairRoot - a, c = 0.5f * kPairRoot - a, d = 0.5f * kPairRoot + a;
                    uint32_t sel = (__float_as_uint(tr) & 1u) * 0x4444u ^ 0x5410u;
                    if (pi == 1 && k == 0) sel ^= g == 4u ? 0x4444u : 0u;    // octad 2 of parity 1 is kept odd sum first: totals then have the parity that the cosets ask for
                    w[pi][0] = __byte_perm(__float_as_uint(fmaf(a, a, 8388608.f)), __float_as_uint(fmaf(b, b, 8388608.f)), sel);
                    // an offset larger by 2 moves t by a half: the error becomes 1/2 - |err|, and z one less where err was negative
                    sel ^= (uint32_t)((int)__float_as_uint(err) >> 31) & 0x4444u;
                    w[pi][1] = __byte_perm(__float_as_uint(fmaf(c, c, 8388608.f)), __float_as_uint(fmaf(d, d, 8388608.f)), sel);
                }
#pragma unroll
                for (int b = 0; b < 2; ++b) n[k][b] = {__byte_perm(w[0][b], w[1][b], 0x5410), __byte_perm(w[0][b], w[1][b], 0x7632)};
            }
            Cost pair[2][4];
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int b = 0; b < 4; ++b) pair[p][b] = n[2 * p][b & 1] + n[2 * p + 1][b >> 1];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const Cost c = pair[0][i & 3] + pair[1][i >> 2];
                sts64(tab + g * kNibTable + (uint32_t)i * kNibRow, c.even, c.odd);
            }
        }
        __syncwarp();                                                // either lane of a vector reads the tables that the other one made
        uint32_t best = 0xffffu, second = 0xffffu, group = 0;        // group: 2 x + parity
        uint32_t kept[8];                                            // the smallest costs of that x, by a
#pragma unroll
        for (int i = 0; i < 8; ++i) kept[i] = 0u;
#pragma unroll 1
        for (uint32_t x = 4u * (uint32_t)q; x < 4u * (uint32_t)q + 4u; ++x) {
            const uint32_t px = turyn_x(x);
            const uint32_t lo = tab ^ (px & 15u) * kNibRow, hi = (tab + kNibTable) ^ (px >> 4) * kNibRow;
            Cost b[8], c[8];
            uint32_t least[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) { b[j] = pattern_cost(lo, hi, turyn_a(j), 1u); c[j] = pattern_cost(lo, hi, turyn_a(j), 2u); }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                // the other two octads together for an even and for an odd sum of this one's z: four instructions for each b (six with the
                // first two octads combined first: 695 -> 669 us EUCLIDEAN, 749 -> 722 us ANGULAR)
                uint32_t even = 0xffffffffu, odd = 0xffffffffu;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    even = __viaddmin_u16x2(b[j].even, c[i ^ j].even, even);
                    odd = __viaddmin_u16x2(b[j].odd, c[i ^ j].even, odd);
                    even = __viaddmin_u16x2(b[j].odd, c[i ^ j].odd, even);
                    odd = __viaddmin_u16x2(b[j].even, c[i ^ j].odd, odd);
                }
                const Cost a = pattern_cost(lo, hi, turyn_a(i), 0u);
                least[i] = __viaddmin_u16x2(a.odd, odd, a.even + even);
            }
            const uint32_t m = __vminu2(__vimin3_u16x2(least[0], least[1], least[2]), __vminu2(__vimin3_u16x2(least[3], least[4], least[5]), __vminu2(least[6], least[7])));
            const uint32_t before = best;
#pragma unroll
            for (uint32_t pi = 0; pi < 2; ++pi) {
                const uint32_t mine = half_of(m, (int)pi);
                second = min(second, max(best, mine));
                group = mine < best ? 2u * x + pi : group;
                best = min(best, mine);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) kept[i] = best < before ? least[i] : kept[i];
        }
        __syncthreads();
        // the better lane of the two; its a within the margin
        uint32_t a_of = 0, b_of = 0, hits = 0;
        {
            const uint32_t best_o = __shfl_xor_sync(kFull, best, 16), second_o = __shfl_xor_sync(kFull, second, 16), group_o = __shfl_xor_sync(kFull, group, 16);
            const bool mine = best < best_o || (best == best_o && q == 0);
            second = min(max(best, best_o), mine ? second : second_o);
            best = min(best, best_o);
            settled = second > best + kPairMargin;
#pragma unroll
            for (uint32_t i = 0; i < 8; ++i)
                if (half_of(kept[i], (int)(group & 1u)) <= best + kPairMargin) { a_of = i; ++hits; }
            a_of |= hits << 8;
            const uint32_t a_of_o = __shfl_xor_sync(kFull, a_of, 16);
            a_of = mine ? a_of : a_of_o;
            group = mine ? group : group_o;
            settled &= a_of >> 8 == 1u;
            a_of &= 7u;
        }
        const int pi = (int)(group & 1u);
        const uint32_t px = turyn_x(group >> 1), pa = turyn_a(a_of);
        {
            // the b within the margin: four for either lane
            constexpr uint32_t upper = turyn_a(4);
            const uint32_t lo = tab ^ (px & 15u) * kNibRow, hi = (tab + kNibTable) ^ (px >> 4) * kNibRow;
            const uint32_t lo_a = lo ^ (pa & 15u) * kNibRow, hi_a = hi ^ (pa >> 4) * kNibRow;
            const uint32_t lo_q = q ? (upper & 15u) * kNibRow : 0u, hi_q = q ? (upper >> 4) * kNibRow : 0u;
            const Cost a = pattern_cost(lo_a, hi_a, 0u, 0u);
            hits = 0;
#pragma unroll
            for (uint32_t j = 0; j < 4; ++j) {
                const Cost two = a + pattern_cost(lo ^ lo_q, hi ^ hi_q, turyn_a(j), 1u), c = pattern_cost(lo_a ^ lo_q, hi_a ^ hi_q, turyn_a(j), 2u);
                if (half_of(__vminu2(two.even + c.even, two.odd + c.odd), pi) <= best + kPairMargin) { b_of = 4u * (uint32_t)q + j; ++hits; }
            }
            const uint32_t other = __shfl_xor_sync(kFull, hits << 8 | b_of, 16);
            settled &= hits + (other >> 8) == 1u;
            b_of = hits ? b_of : other & 7u;
        }
        // the triple's patterns and their complements: {cost with an even sum of z, with an odd one} from the coordinates, a nibble of
        // every octad for either lane
        const uint32_t pb = turyn_a(b_of);
        uint32_t patterns = (px ^ pa) | (px ^ pb) << 8 | (px ^ pa ^ pb) << 16, part[3], part_c[3];
        patterns >>= 4 * q;
        const float shift = pi ? 0.25f : 0.f;
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            const uint32_t four = coords[2 * o + q];
            float sum = 0.f, squares = 0.f, most = 0.f, fewest = 1.f;
            uint32_t parity = 0u;                                    // bit 0: of the sum of z; bit 1: of the number of negative errors
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float t = v[16u * ((four >> (8 * k)) & 31u)] * s1 * s2 * 0.25f - shift, tr = t + 12582912.f, err = t - (tr - 12582912.f);
                const uint32_t bit = (patterns >> (8 * o + k)) & 1u, negative = __float_as_uint(err) >> 31;
                const float mag = fabsf(fabsf(err) - __uint_as_float(bit * 0x3f000000u));
                squares = fmaf(mag, mag, squares);
                sum += mag;
                most = fmaxf(most, mag);
                fewest = fminf(fewest, mag);
                parity ^= ((__float_as_uint(tr) & 1u) ^ (bit & negative)) | negative << 1;
            }
            squares += __shfl_xor_sync(kFull, squares, 16);
            sum += __shfl_xor_sync(kFull, sum, 16);
            most = fmaxf(most, __shfl_xor_sync(kFull, most, 16));
            fewest = fminf(fewest, __shfl_xor_sync(kFull, fewest, 16));
            parity ^= __shfl_xor_sync(kFull, parity, 16);
            if (o == 2) parity ^= (uint32_t)pi;
            const float other = squares - sum + 2.f;                 // the complement's errors are 1/2 - mag
            const uint32_t stay = __float_as_uint(fmaf(squares, kPairScale, 8388608.f)), move = __float_as_uint(fmaf(squares + (1.f - 2.f * most), kPairScale, 8388608.f));
            const uint32_t stay_c = __float_as_uint(fmaf(other, kPairScale, 8388608.f)), move_c = __float_as_uint(fmaf(fmaf(2.f, fewest, other), kPairScale, 8388608.f));
            part[o] = __byte_perm(stay, move, parity & 1u ? 0x1054 : 0x5410);
            part_c[o] = __byte_perm(stay_c, move_c, (parity ^ parity >> 1) & 1u ? 0x1054 : 0x5410);
        }
        uint32_t word = 0;
        {
            hits = 0;
#pragma unroll
            for (int t = 0; t < 8; ++t) {                            // bit o: the complement on octad o
                const uint32_t a = t & 1 ? part_c[0] : part[0], b = t & 2 ? part_c[1] : part[1], c = t & 4 ? part_c[2] : part[2];
                const uint32_t all = __viaddmin_u16x2(__byte_perm(a, 0u, 0x3232), __byte_perm(b, 0u, 0x1032), __byte_perm(a, 0u, 0x1010) + b) + c;
                if (min(all & 0xffffu, all >> 16) <= best + kWordMargin) { word = (uint32_t)t; ++hits; }
            }
            settled &= hits == 1u;
            const uint32_t x8 = (group >> 1) * 8u;
            word = S.word[0][x8 + a_of] ^ (word & 1u ? S.ones[0] : 0u) ^ S.word[1][x8 + b_of] ^ (word & 2u ? S.ones[1] : 0u) ^
                   S.word[2][x8 + (a_of ^ b_of)] ^ (word & 4u ? S.ones[2] : 0u);
        }
        // the point of coset (pi, word), twelve coordinates for either lane
        {
            constexpr double kRint = 6755399441055744.0;             // 1.5 * 2^52: adding it rounds to a whole number, which is in the low word
            double most = -1.0, next = -1.0, u_most = 0.0, dot = 0.0;
            int sum = 0, who = 0, move = 4;
            const float* const mine = v + 16 * 12 * q;
            word >>= 12 * q;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                r.x[j] = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int k = 4 * j + i;
                    const double u = __dmul_rn(__dmul_rn((double)mine[16 * k], rn), radius);
                    const int b = pi + 2 * (int)((word >> k) & 1u);
                    const double bd = b & 2 ? (pi ? 3.0 : 2.0) : (pi ? 1.0 : 0.0);
                    const double tt = __dmul_rn(__dsub_rn(u, bd), 0.25), big = __dadd_rn(tt, kRint), z = __dsub_rn(big, kRint);
                    const double err = __dsub_rn(tt, z), mag = fabs(err);
                    const int xi = b + 4 * __double2loint(big);
                    r.x[j] |= (uint32_t)(xi & 0xff) << (8 * i);
                    sum += xi;
                    dot = fma(u, fma(z, 4.0, bd), dot);
                    next = mag > most ? most : fmax(next, mag);
                    if (mag > most) { most = mag; who = k; u_most = u; move = err < 0.0 ? -4 : 4; }
                }
            }
            sum += __shfl_xor_sync(kFull, sum, 16);
            const double most_o = __shfl_xor_sync(kFull, most, 16), next_o = __shfl_xor_sync(kFull, next, 16);
            const bool moved = (sum & 7) != (pi ? 4 : 0);
            next = fmax(fmin(most, most_o), fmax(next, next_o));
            if (moved && (q == 0 ? most >= most_o : most > most_o)) {    // the first coordinate with the largest error is here
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    if (who >> 2 == j) {
                        const uint32_t old = (r.x[j] >> (8 * (who & 3))) & 0xffu;
                        r.x[j] ^= (old ^ ((old + (uint32_t)move) & 0xffu)) << (8 * (who & 3));
                    }
                dot = fma((double)move, u_most, dot);
            }
            most = fmax(most, most_o);
            r.unique = moved ? next <= most - 1.0e-6 : most < 0.5 - 1.0e-6;
            r.dot = dot + __shfl_xor_sync(kFull, dot, 16);
            int n2 = 0;
#pragma unroll
            for (int j = 0; j < 3; ++j) n2 = __dp4a((int)r.x[j], (int)r.x[j], n2);
            r.norm2 = n2 + __shfl_xor_sync(kFull, n2, 16);
        }
    }
    // vectors with several candidates wait until there is one for almost every warp, or nothing else to do
    bool found = wanted && settled;
    waiting |= wanted && !settled;
    while (true) {
        __syncthreads();                                         // the costs of all warps are done with: nearest_careful works there
        const bool listing = waiting && spot >= kPendingMost;
        uint32_t mine = 0;
        if (listing && q == 0) {
            mine = atomicAdd(&pending.count, 1u);
            if (mine < kPendingMost) { Pending& p = pending.list[mine]; p.v = v; p.rn = rn; p.radius = radius; }
        }
        mine = __shfl_sync(kFull, mine, lane & 15);              // all lanes: those that list their vector need not have stayed together
        if (listing) spot = mine;
        __syncthreads();
        const uint32_t n = pending.count;
        if (n < (few ? 1u : kPendingEnough)) break;
        __syncthreads();
        if (threadIdx.x == 0) pending.count = 0u;
        for (uint32_t i = (uint32_t)warp; i < min(n, kPendingMost); i += (uint32_t)kEncWarps<true>) {
            Pending& p = pending.list[i];
            int norm2;
            bool unique;
            const double u = lane < 24 ? __dmul_rn(__dmul_rn((double)p.v[16 * lane], p.rn), p.radius) : 0.0;
            const int xi = nearest_careful(careful, S, steps, golay, pos_by_low12, u, lane, norm2, unique);
            const double dot = dot_of_warp(u, xi);
            if (lane < 24) p.x[lane] = (int8_t)xi;
            if (lane == 0) { p.norm2 = norm2; p.unique = unique; p.dot = dot; }
        }
        __syncthreads();
        if (waiting && spot < kPendingMost) {
            const Pending& p = pending.list[spot];
#pragma unroll
            for (int j = 0; j < 3; ++j) r.x[j] = reinterpret_cast<const uint32_t*>(p.x)[3 * q + j];
            r.norm2 = p.norm2; r.unique = p.unique; r.dot = p.dot;
            waiting = false;
            found = true;
        }
        spot = kPendingMost;
        if (n <= kPendingMost) break;
    }
    return found;
}

// The oracle's score of a candidate (24 signed bytes), one binary64 rounding per operation, sums in the order of the coordinates.
__device__ __noinline__ double exact_score(int metric, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t w4, uint32_t w5, const float* v, int stride, double rn)
{
    const uint32_t w[6] = {w0, w1, w2, w3, w4, w5};
    double acc = 0.0;
    int n2 = 0;
#pragma unroll
    for (int i = 0; i < 24; ++i) {
        const int x = (int)(int8_t)(w[i >> 2] >> (8 * (i & 3)));
        const double vi = (double)v[stride * i];
        n2 += x * x;
        if (metric == LLVQ_EUCLIDEAN) {
            const double dd = __dsub_rn(vi, (double)x);
            acc = __dadd_rn(acc, __dmul_rn(dd, dd));
        } else {
            acc = __dadd_rn(acc, __dmul_rn(__dmul_rn(vi, rn), (double)x));
        }
    }
    return metric == LLVQ_EUCLIDEAN ? -acc : __ddiv_rn(acc, __dsqrt_rn((double)n2));
}

// Shells m_from .. m_to as a mask (bit m = shell m; none if m_from > m_to).
__device__ __forceinline__ uint64_t shells(int m_from, int m_to)
{
    return m_from > m_to ? 0ull : (~0ull >> (63 - (m_to - m_from))) << m_from;
}

// Two lanes per input vector, each pair with its own progress: a vector that is done is replaced at once.  (One warp per vector, kPairs false:
// all pairs of lanes do the same.)
// Inputs are binary32 values, the scoring that decides runs in binary64 with one rounding per operation and sums over the
// coordinates in order.  EUCLIDEAN: if the nearest lattice point of the input lies in the code it is the
// answer (it is then also the nearest point of the cut, App. E "Spherical shaping").  Otherwise, and for ANGULAR always,
// the input direction is decoded at every shell radius sqrt(16 m); of the candidates inside the code the one nearest to
// the input (EUCLIDEAN) or with the largest cosine (ANGULAR) wins, the first radius on ties.  A zero input gives the
// point of index 0, (4, 4, 0^22), the first point of the first class of Shell(2) (Sec. 2.3).  Needs m_lo == 2 and
// m_hi >= 3 (checked on the host).  Scores are compared as binary64 sums in any order; where they come within 1e-9, as the oracle forms them.
// EUCLIDEAN does not need all the radii.  At distance r along the direction d of the input (length R) the nearest point x
// minimises |x|^2 - 2 r <x, d>; two minimisers at radii r < r' therefore satisfy <x, d> <= <x', d>, and
// |x'|^2 - 2 R <x', d> <= |x|^2 - 2 R <x, d> for r < r' <= R (symmetrically for R <= r' < r): the radius next to R that yields a
// point of the code beats all radii beyond it, by the margin reported as `unique`.  So the radii are tried
// outwards from R, on each side until such a point is found (inputs so long that a squared distance no longer resolves the
// margin try them all).
// Neither does ANGULAR.  With g = max_x 2 t <x, d> - |x|^2 = 2 t <x_t, d> - |x_t|^2 known from the decode at radius t, every lattice
// point of norm r satisfies <x, d> <= (g + r^2) / (2 t): its cosine stays below the best one found, c, if r lies strictly between
// the roots of r^2 - 2 t c r + g.  That rules out whole shells (`out`).  And as a maximum of lines g is convex in t: the nearest
// point's norm does not fall as t grows, so between two decoded radii it stays between theirs.  A radius at which only ruled-out
// shells are possible cannot change the result and is not decoded.  The order: downwards from m_hi while the points found lie in
// shells that could still win, then a leap to the radius that should rule out most of what is left below.  On Gaussian
// inputs, shells 2..12, 6.0 of 11 radii are decoded.
template <bool kPairs>
__global__ void __launch_bounds__(kEncWarps<kPairs> * 32, 1)
encode_search_kernel(const uint32_t* __restrict__ golay, EncTables et, const __grid_constant__ PatternSteps steps, const float* __restrict__ v, uint64_t n, int metric, int m_lo, int m_hi,
                     int8_t* __restrict__ points, uint32_t* __restrict__ flags)
{
    extern __shared__ __align__(1024) uint8_t enc_smem[];
    constexpr int kVecs = kEncVecs<kPairs>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane >> 4;
    const uint32_t start = (uint32_t)__cvta_generic_to_shared(enc_smem), align = kPairs ? kNibTable : 128u, nib0 = (start + align - 1u) & ~(align - 1u);
    uint8_t* const mem = enc_smem + (nib0 - start);
    const uint32_t nib = nib0 + (uint32_t)warp * kEncWarpBytes<kPairs>;
    WarpTables& careful = *reinterpret_cast<WarpTables*>(mem + warp * kEncWarpBytes<kPairs>);
    float* const mine_v = reinterpret_cast<float*>(mem + kEncWarps<kPairs> * kEncWarpBytes<kPairs>) + warp * (24 * kVecs) + (kPairs ? lane & 15 : 0);
    GolayTrio& S = *reinterpret_cast<GolayTrio*>(mem + kEncWarps<kPairs> * (kEncWarpBytes<kPairs> + 24 * kVecs * sizeof(float)));
    __shared__ double radius[kMaxShell + 1], per_radius[kMaxShell + 1];     // sqrt(16 m) and its reciprocal
    __shared__ uint32_t next_vec;
    __shared__ PendingList pending;
    if (threadIdx.x == 0) { next_vec = 0u; pending.count = 0u; }
    for (int i = threadIdx.x; i <= m_hi; i += blockDim.x) {
        radius[i] = __dsqrt_rn(__dmul_rn(16.0, (double)i));
        per_radius[i] = 1.0 / radius[i];
    }
    for (int i = threadIdx.x; i < (int)sizeof(GolayTrio) / 4; i += blockDim.x)
        reinterpret_cast<uint32_t*>(&S)[i] = __ldg(reinterpret_cast<const uint32_t*>(et.trio) + i);
    __syncthreads();
    const bool words = (reinterpret_cast<uintptr_t>(points) & 3u) == 0, quads = (reinterpret_cast<uintptr_t>(v) & 15u) == 0;
    const float reach = sqrtf(16.f * (float)m_hi) + 4.01f, reach2 = reach * reach;
    // a CTA's share is contiguous; its warps draw the vectors as they have room (some take several decodes)
    const uint64_t first = n / gridDim.x * blockIdx.x + min((uint64_t)blockIdx.x, n % gridDim.x);
    const uint32_t count = (uint32_t)(n / gridDim.x + (blockIdx.x < n % gridDim.x));

    [[maybe_unused]] uint32_t row[6];
    if constexpr (!kPairs) pattern_rows(careful, S, lane, row);
    bool active = false, drained = false;       // this lane's vector is being searched; there are no more
    bool starting = false, direct = false;      // its radii are about to be started; the input itself is decoded (else: its direction at shell radius m)
    bool waiting = false;                       // it is on the list for nearest_careful, at `spot`
    uint32_t spot = kPendingMost;
    bool outwards = false, ok = false;
    uint32_t t = 0, bx[3] = {0u, 0u, 0u};       // its number in the share, the best point
    double rn = 1.0, length = 0.0, best = 0.0;
    float s1 = 1.f;                              // a power of two that brings the input near length 1
    int best_m = 0, m = 0, m_start = 0, step = 0;
    int upper = 0, upper_shell = 0, lower = 0, lower_shell = 0;  // ANGULAR: the radii from `upper` on are settled, `lower` (0: none) is decoded; shells of their points
    uint64_t out = 0;
    const auto store = [&](const uint32_t (&x)[3]) {
        int8_t* const at = points + (first + t) * 24 + 12 * q;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (words) reinterpret_cast<uint32_t*>(at)[j] = x[j];
            else for (int i = 0; i < 4; ++i) at[4 * j + i] = (int8_t)(x[j] >> (8 * i));
        }
    };
    const uint32_t origin[3] = {q ? 0u : 0x0404u, 0u, 0u};       // the point of index 0
    while (true) {
        const uint32_t vacant = __ballot_sync(kFull, !active && !drained);
        if (vacant) {
            __syncwarp();                                        // the inputs that are about to be replaced are no longer read (a vote orders no memory)
            uint32_t base = 0;
            if (lane == 0) base = atomicAdd(&next_vec, kPairs ? (uint32_t)__popc(vacant & 0xffffu) : 1u);
            base = __shfl_sync(kFull, base, 0);
            if (!active && !drained) {
                t = base + (kPairs ? (uint32_t)__popc(vacant & ((1u << (lane & 15)) - 1u)) : 0u);
                drained = t >= count;
            }
            const bool taking = !active && !drained;
            const uint32_t takers = __ballot_sync(kFull, taking);
            if (taking) {
                float n2f = 0.f;
                uint32_t some = 0, finite = 1;
                const float* const from = v + (first + t) * 24 + (kPairs ? 12 * q : 0);
                if constexpr (kPairs) {
                    const auto take = [&](int k, float f) {
                        some |= f != 0.f; finite &= isfinite(f) ? 1u : 0u;
                        n2f = fmaf(f, f, n2f);
                        mine_v[kVecs * (12 * q + k)] = f;
                    };
                    if (quads) {
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            const float4 f = __ldg(reinterpret_cast<const float4*>(from) + k);
                            take(4 * k, f.x); take(4 * k + 1, f.y); take(4 * k + 2, f.z); take(4 * k + 3, f.w);
                        }
                    } else {
#pragma unroll 4
                        for (int k = 0; k < 12; ++k) take(k, __ldg(from + k));
                    }
                    n2f += __shfl_xor_sync(takers, n2f, 16);
                    some |= __shfl_xor_sync(takers, some, 16);
                    finite &= __shfl_xor_sync(takers, finite, 16);
                } else {
                    const float f = lane < 24 ? __ldg(from + lane) : 0.f;
                    if (lane < 24) mine_v[lane] = f;
                    n2f = f * f;
#pragma unroll
                    for (int o = 16; o; o >>= 1) n2f += __shfl_xor_sync(kFull, n2f, o);
                    some = __any_sync(kFull, f != 0.f); finite = __all_sync(kFull, isfinite(f));
                }
                // (the vectors that will be taken when the CTA is through with those it has)
                if (t + kEncWarps<kPairs> * kVecs < count) asm volatile("prefetch.global.L2 [%0];" ::"l"(from + kEncWarps<kPairs> * kVecs * 24));
                // no lattice point is farther than 4 from any input (covering radius): beyond radius sqrt(16 m_hi) + 4 the nearest
                // point is certainly outside the code and the decode can be skipped
                direct = metric == LLVQ_EUCLIDEAN && n2f <= reach2;
                starting = !direct;
                active = some && finite;
                ok = false;
                rn = 1.0;
                s1 = 1.f;
                if (!active) {
                    store(origin);
                    if (!finite) atomicOr(flags, kFlagSearchGaveUp);
                }
            }
        }
        __syncwarp();
        int busy = 0;
        bool few = false, found = true;
        if constexpr (kPairs) {
            busy = __syncthreads_count(active && q == 0);
            if (busy == 0 && __syncthreads_and(drained)) break;
            // (also where all that are left wait)
            few = busy <= kFew || __syncthreads_count(active && !waiting) == 0;
        } else {
            if (drained) break;
            if (!active) continue;
        }
        if (active && starting) {
            double n2 = 0.0;
#pragma unroll
            for (int i = 0; i < 24; ++i) { const double vi = (double)mine_v[kVecs * i]; n2 = __dadd_rn(n2, __dmul_rn(vi, vi)); }
            length = __dsqrt_rn(n2);
            rn = __ddiv_rn(1.0, length);
            outwards = metric == LLVQ_EUCLIDEAN && n2 < 1.0e9;
            // tried outwards: first down from the largest radius not above R, then up from the next one
            m = m_start = outwards ? max(m_lo - 1, (int)fmin(n2 * 0.0625, (double)m_hi)) : m_hi;
            step = -1;
            if (m < m_lo) { m = m_start + 1; step = 1; }
            upper = m_hi + 1; lower = 0; out = 0;
            starting = false;
            s1 = __uint_as_float((uint32_t)min(max(1150 - ((__double2hiint(length) >> 20) & 0x7ff), 1), 254) << 23);
        }
        __syncwarp();
        const double rad = direct || !active ? 1.0 : radius[m];
        const float s2 = direct || !active ? 1.f : (float)(rad * (rn / (double)s1));
        Nearest r;
        if constexpr (kPairs) {
            found = nearest_pairs(nib, mine_v, S, steps, golay, et.pos_by_low12, careful, pending, s1, s2, rn, rad, active && !waiting, waiting, spot, few, warp, lane, r);
        } else {
            int8_t* const point = reinterpret_cast<int8_t*>(&careful + 1);
            const double u = lane < 24 ? __dmul_rn(__dmul_rn((double)mine_v[lane], rn), rad) : 0.0;
            const int xi = nearest_careful_from<false>(careful, S, steps, row, golay, et.pos_by_low12, u, lane, r.norm2, r.unique);
            r.dot = direct ? 0.0 : dot_of_warp(u, xi);           // (not looked at where the input itself was decoded)
            if (lane < 24) point[lane] = (int8_t)xi;
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 3; ++j) r.x[j] = reinterpret_cast<const uint32_t*>(point)[3 * q + j];
        }
        __syncwarp();
        const int shell = r.norm2 >> 4;                          // lattice points have norms 16 m
        const bool in_code = shell >= m_lo && shell <= m_hi;
        const uint32_t unlike = __ballot_sync(kFull, ((r.x[0] ^ bx[0]) | (r.x[1] ^ bx[1]) | (r.x[2] ^ bx[2])) != 0u) >> (lane & 15) & 0x10001u;
        bool done = false;
        if (!found || !active) {
        } else if (direct) {
            direct = false;
            starting = !in_code;
            if (in_code) {
                done = ok = true;
#pragma unroll
                for (int j = 0; j < 3; ++j) bx[j] = r.x[j];
            }
        } else {
            if (in_code) {
                // the candidate's score, up to rounding: the cosine; EUCLIDEAN: 2 <v, x> - |x|^2, which is |v|^2 minus the squared distance
                double score, tol = 1.0e-9;
                if (metric == LLVQ_EUCLIDEAN) {
                    score = 2.0 * r.dot * length * per_radius[m] - (double)r.norm2;
                    tol = 1.0e-9 * (1.0 + length) + 1.0e-14 * length * length;
                } else {
                    score = r.dot * per_radius[m] * per_radius[shell];
                }
                bool better = !ok || score > best + tol;
                if (!better && !(score < best - tol)) {
                    if (!unlike) {
                        best_m = min(best_m, m);                 // the same point again
                    } else {
                        const uint32_t pair = 0x10001u << (lane & 15);
                        uint32_t w[6], b[6];
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            const uint32_t xo = __shfl_xor_sync(pair, r.x[j], 16), bo = __shfl_xor_sync(pair, bx[j], 16);
                            w[j] = q ? xo : r.x[j]; w[3 + j] = q ? r.x[j] : xo;
                            b[j] = q ? bo : bx[j]; b[3 + j] = q ? bx[j] : bo;
                        }
                        const double now = exact_score(metric, w[0], w[1], w[2], w[3], w[4], w[5], mine_v, kVecs, rn);
                        const double before = exact_score(metric, b[0], b[1], b[2], b[3], b[4], b[5], mine_v, kVecs, rn);
                        better = now > before || (now == before && m < best_m);
                    }
                }
                if (better) {
                    best = score; best_m = m; ok = true;
#pragma unroll
                    for (int j = 0; j < 3; ++j) bx[j] = r.x[j];
                }
            }
            if (metric == LLVQ_EUCLIDEAN) {
                if (in_code && outwards && r.unique) {           // this side is done
                    done = step > 0;
                    m = m_lo - 1;
                } else {
                    m += step;
                }
                if (step < 0 && m < m_lo) { m = m_start + 1; step = 1; }
                done |= m > m_hi;
            } else {
                if (ok) {
                    const float disc = (float)((rad * best) * (rad * best) - 2.0 * r.dot + (double)r.norm2);
                    if (disc > 0.01f) {
                        // strictly between the roots, by a margin far above the rounding
                        const float mid = (float)(rad * best), half = sqrtf(disc) - 0.002f;
                        const float from = fmaxf(mid - half, 0.f), to = fmaxf(mid + half, 0.f);
                        out |= shells(max((int)(from * from * 0.0625f) + 1, 2), min((int)(to * to * 0.0625f), m_hi));
                    }
                }
                if (m == upper - 1) { upper = m; upper_shell = shell; }
                else { lower = m; lower_shell = shell; }
                while (true) {
                    const uint64_t open = shells(lower ? max(lower_shell, m_lo) : m_lo, min(upper_shell, m_hi)) & ~out;
                    if (upper == m_lo || (!open && !lower)) { done = true; break; }
                    if (!open || upper == lower + 1) { upper = lower; upper_shell = lower_shell; lower = 0; continue; }
                    m = upper - 1;
                    if (!lower && upper_shell <= m_hi && ((out >> upper_shell) & 1u)) {
                        const float reached = 4.f * sqrtf((float)(63 - __clzll((long long)open))) - 1.5f;
                        m = min(m, max((int)(reached * reached * 0.0625f), m_lo + 1));
                    }
                    break;
                }
            }
        }
        if (done) {
            if (!ok) atomicOr(flags, kFlagSearchGaveUp);
            if (ok) store(bx);
            else store(origin);
            active = false;
        }
    }
}

// Bits kBit of the 24 bytes of w as a mask, byte i -> bit i: the eight bits of a pair of words are moved together by one multiplication
// (bits 8 i and 8 i + 4 meet the factors 2^(32 - 7 j); those with i = j are wanted, no two products fall together, so nothing carries).
template <int kBit>
__device__ __forceinline__ uint32_t bit_plane(const uint32_t (&w)[6])
{
    uint32_t r[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const uint32_t lo = w[2 * j] >> kBit, hi = kBit < 4 ? w[2 * j + 1] << (4 - kBit) : w[2 * j + 1] >> (kBit - 4);
        const unsigned long long p = (unsigned long long)((lo & 0x01010101u) | (hi & 0x10101010u)) * 0x102040800ull;
        r[j] = (uint32_t)(p >> 32) & 0xffu;
    }
    return r[0] | r[1] << 8 | r[2] << 16;
}

constexpr int kRankThreads = 256;
constexpr int kRankValues = 32;            // larger than any absolute value of a point: its square is at most 16 * 53

// Point -> index (Sec. 3.2; inverse of App. A steps 1-4), one thread per block.  A point that is not in the code
// gets index 0 and is counted in the out-of-range counter.  The absolute values are taken as bit planes over the 24
// coordinates: which coordinates hold a value is a few operations on masks, and the place of an element among
// the free slots is a population count.
__global__ void __launch_bounds__(kRankThreads)
rank_kernel(DevCode dc, EncTables et, const uint32_t* __restrict__ golay, const uint32_t* __restrict__ pascal,
            const int8_t* __restrict__ points, uint64_t n, unsigned long long* __restrict__ index)
{
    __shared__ uint64_t sig_of[kRankValues];
    __shared__ uint32_t choose[25 * 25];
    for (int i = threadIdx.x; i < kRankValues; i += kRankThreads) sig_of[i] = __ldg(et.sig_of_value + i);
    for (int i = threadIdx.x; i < 25 * 25; i += kRankThreads) choose[i] = __ldg(pascal + i);
    __syncthreads();
    const uint64_t b = (uint64_t)blockIdx.x * kRankThreads + threadIdx.x;
    if (b >= n) return;
    uint32_t w[6];
    const int8_t* const from = points + b * 24;
    if ((reinterpret_cast<uintptr_t>(points) & 7u) == 0) {
#pragma unroll
        for (int j = 0; j < 3; ++j) { const uint2 t = __ldg(reinterpret_cast<const uint2*>(from) + j); w[2 * j] = t.x; w[2 * j + 1] = t.y; }
    } else {
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            w[j] = 0;
            for (int i = 0; i < 4; ++i) w[j] |= (uint32_t)(uint8_t)__ldg(from + 4 * j + i) << (8 * i);
        }
    }
    const uint32_t all = 0xffffffu;
    const uint32_t odd = bit_plane<0>(w), neg = bit_plane<7>(w);
    uint32_t beyond = 0;
    uint64_t sig = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {                                              // absolute values
        const uint32_t m = (w[j] >> 7) & 0x01010101u;
        w[j] = (w[j] ^ m * 255u) + m;
        beyond |= w[j];
#pragma unroll
        for (int i = 0; i < 4; ++i) sig += sig_of[(w[j] >> (8 * i)) & (kRankValues - 1)];
    }
    const uint32_t bit1 = bit_plane<1>(w), bit2 = bit_plane<2>(w), bit3 = bit_plane<3>(w), bit4 = bit_plane<4>(w);
    const bool parity = odd != 0u;
    bool good = (odd == 0u || odd == all) && (beyond & 0xe0e0e0e0u) == 0u;
    const uint32_t c = parity ? bit1 ^ neg : bit1;                              // bit 1 of x - parity
    // the coordinates whose absolute value is v (a value of the point's parity)
    const auto holding = [&](uint32_t v) {
        return ~((bit1 ^ (0u - (v >> 1 & 1u))) | (bit2 ^ (0u - (v >> 2 & 1u))) | (bit3 ^ (0u - (v >> 3 & 1u))) | (bit4 ^ (0u - (v >> 4 & 1u)))) & all;
    };
    // class of the multiset of absolute values
    uint32_t cls = 0;
    bool found = false;
    uint32_t slot = (uint32_t)(sig >> 20) & et.hash_mask;
    for (uint32_t probe = 0; probe <= et.hash_mask; ++probe) {
        const uint64_t key = __ldg(et.hash_key + slot);
        if (key == sig) { cls = __ldg(et.hash_cls + slot); found = true; break; }
        if (key == 0) break;
        slot = (slot + 1) & et.hash_mask;
    }
    good &= found;
    unsigned long long I = 0;
    if (good) {
        const uint4* const record = reinterpret_cast<const uint4*>(dc.cls + cls);     // ClassDesc: 16 bytes, then 8 per level
        const uint4 h = __ldg(record);
        const uint32_t weight = (h.x >> 8) & 0xffu, B = (h.x >> 16) & 0xffu, signpar = h.x >> 24;
        const int nlev1 = (int)(h.y & 0xffu), nlev = nlev1 + (int)((h.y >> 8) & 0xffu);
        const uint32_t fill1 = (h.y >> 16) & 0xffu, fill0 = h.y >> 24, goff = h.z & 0xffffu, A = h.z >> 16;
        const uint32_t pos = __ldg(et.pos_by_low12 + (c & 0xfffu));
        good &= __ldg(golay + pos) == c;                                   // c must be a codeword
        const uint32_t r = pos - goff;
        good &= r < A;                                                     // ... of the weight the class needs
        const uint32_t F1 = parity ? 0u : c, F0 = ~F1 & all;
        uint32_t freem = parity ? all : F1;
        bool in0 = parity;
        unsigned long long p = 0, mult = 1;
        for (int l = 0; l < nlev; ++l) {
            if (!in0 && l >= nlev1) {                                      // the rest of group 1 holds its filler
                good &= (freem & ~holding(fill1)) == 0u;
                freem = F0; in0 = true;
            }
            const uint2 lv = __ldg(reinterpret_cast<const uint2*>(record + 1) + l);     // radix, slots | value << 8 | ...
            const uint32_t mine = holding((lv.y >> 8) & 0xffu) & freem;
            good &= (uint32_t)__popc(mine) == (lv.y & 0xffu);
            uint32_t rho = 0, t = 1;
            for (uint32_t left = mine; left; left &= left - 1u, ++t)       // combinatorial number system: sum of C(e_t, t), e_t = place among the free slots
                rho += choose[__popc(freem & ((left & (0u - left)) - 1u)) * 25 + t];
            p += mult * rho;
            mult *= lv.x;
            freem ^= mine;
        }
        if (!in0) {
            good &= (freem & ~holding(fill1)) == 0u;
            freem = F0;
        }
        good &= (freem & ~holding(fill0)) == 0u;
        unsigned long long s = 0;
        if (parity) {
            good &= neg == (c ^ bit1);                                     // 1 mod 4 on F0, 3 mod 4 on F1
        } else {
            // s = the signs of the positions that carry one (F1 and the nonzero ones of F0), ascending, without the last F1
            // position, whose sign the others fix (sum = 0 mod 8)
            const uint32_t last_f1 = F1 ? 0x80000000u >> __clz(F1) : 0u;
            if (weight) good &= ((neg & last_f1) != 0u) == (((__popc(neg & F1 & ~last_f1) + signpar) & 1u) != 0u);
            const uint32_t signs = (F1 | (F0 & (bit1 | bit2 | bit3 | bit4))) & ~last_f1;
            uint32_t bits = 0;
            for (uint32_t left = neg & signs; left; left &= left - 1u) bits |= 1u << __popc(signs & ((left & (0u - left)) - 1u));
            s = bits;
        }
        I = dc.off_lo[cls] + r + (unsigned long long)A * (s + (p << B));
    }
    if (!good) { I = 0; atomicAdd(dc.bad_index, 1ull); }
    index[b] = I;
}

// One thread per 32-bit word of the stored stream: gathers the fields that overlap it.
__global__ void __launch_bounds__(256)
pack_kernel(const unsigned long long* __restrict__ index, const uint8_t* __restrict__ gain_index, int W, int gain_bits,
            uint64_t n, uint32_t* __restrict__ out, uint64_t nwords)
{
    const uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nwords) return;
    const uint64_t bit0 = w * 32, wt = (uint64_t)(W + gain_bits);
    const unsigned long long keep = wt < 64 ? (1ull << wt) - 1ull : ~0ull;
    uint32_t acc = 0;
    for (uint64_t f = bit0 / wt; f < n && f * wt < bit0 + 32; ++f) {
        unsigned long long field = index[f];
        if (gain_index) field |= (unsigned long long)gain_index[f] << W;
        field &= keep;
        const uint64_t start = f * wt;
        acc |= start >= bit0 ? (uint32_t)(field << (start - bit0)) : (uint32_t)(field >> (bit0 - start));
    }
    out[w] = acc;
}

int status_of_launch() { return cudaGetLastError() == cudaSuccess ? LLVQ_OK : LLVQ_ECUDA; }

int launch_rank(const llvq_ctx* ctx, const int8_t* d_points, uint64_t nblocks, uint64_t* d_index, cudaStream_t st)
{
    const unsigned grid = (unsigned)((nblocks + kRankThreads - 1) / kRankThreads);
    rank_kernel<<<grid, kRankThreads, 0, st>>>(ctx->dev, ctx->enc, ctx->d_golay, ctx->enc.pascal, d_points, nblocks,
                                      reinterpret_cast<unsigned long long*>(d_index));
    return status_of_launch();
}

int check_encoder(const llvq_ctx* ctx, uint64_t nblocks)
{
    if (!ctx || ctx->device < 0) return LLVQ_EINVAL;
    if (!ctx->can_encode || nblocks > (1ull << 31) * 256ull) return LLVQ_EUNSUPPORTED;
    return LLVQ_OK;
}

}  // namespace

extern "C" {

int llvq_encode_blocks(const llvq_ctx* ctx, const float* d_v_f32, uint64_t nblocks, int metric,
                       int8_t* d_points, uint64_t* d_index, void* stream)
{
    if (ctx && ctx->device >= 0 && nblocks == 0) return LLVQ_OK;
    if (int e = check_encoder(ctx, nblocks)) return e;
    if (!d_v_f32 || !d_points || !d_index || (metric != LLVQ_EUCLIDEAN && metric != LLVQ_ANGULAR)) return LLVQ_EINVAL;
    if (!aligned(d_v_f32, 4) || !aligned(d_index, 8)) return LLVQ_EALIGN;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return LLVQ_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    PatternSteps steps;
    for (int o = 0; o < 3; ++o)
        for (int j = 0; j < 4; ++j) { steps.lo[o][j] = (ctx->trio.pat[o][j] & 15u) * 8u; steps.hi[o][j] = (uint32_t)(ctx->trio.pat[o][j] >> 4) * 8u; }
    const unsigned grid = (unsigned)std::min<uint64_t>(nblocks, (uint64_t)ctx->sm_count);
    const bool pairs = nblocks > (uint64_t)ctx->sm_count * (metric == LLVQ_EUCLIDEAN ? kPairsFromEuclidean : kPairsFromAngular);
    const auto launch = [&](auto form) -> int {
        constexpr bool kPairs = decltype(form)::value;
        if (!allow_smem<encode_search_kernel<kPairs>>(ctx->smem_limits, ctx->smem_most, kEncSmem<kPairs>)) return LLVQ_ECUDA;
        encode_search_kernel<kPairs><<<grid, kEncWarps<kPairs> * 32, kEncSmem<kPairs>, st>>>(ctx->d_golay, ctx->enc, steps, d_v_f32, nblocks, metric, ctx->host.m_lo,
                                                                                           ctx->host.m_hi, d_points, ctx->dev.flags);
        return status_of_launch();
    };
    if (int e = pairs ? launch(std::true_type{}) : launch(std::false_type{})) return e;
    return launch_rank(ctx, d_points, nblocks, d_index, st);
}

int llvq_rank_blocks(const llvq_ctx* ctx, const int8_t* d_points, uint64_t nblocks, uint64_t* d_index, void* stream)
{
    if (ctx && ctx->device >= 0 && nblocks == 0) return LLVQ_OK;
    if (int e = check_encoder(ctx, nblocks)) return e;
    if (!d_points || !d_index) return LLVQ_EINVAL;
    if (!aligned(d_index, 8)) return LLVQ_EALIGN;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return LLVQ_ECUDA;
    return launch_rank(ctx, d_points, nblocks, d_index, (cudaStream_t)stream);
}

int llvq_pack_fields(const llvq_ctx* ctx, const uint64_t* d_index, const uint8_t* d_gain_index, int gain_bits,
                     uint64_t nblocks, void* d_fields, void* stream)
{
    if (!ctx || ctx->device < 0 || gain_bits < 0 || gain_bits > 8) return LLVQ_EINVAL;
    if (ctx->host.W + gain_bits > 64) return LLVQ_EUNSUPPORTED;
    if (nblocks == 0) return LLVQ_OK;
    if (!d_index || !d_fields || (gain_bits > 0 && !d_gain_index)) return LLVQ_EINVAL;
    if (!aligned(d_index, 8) || !aligned(d_fields, 16)) return LLVQ_EALIGN;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return LLVQ_ECUDA;
    const uint64_t nwords = llvq_field_bytes(ctx, nblocks, gain_bits) / 4;
    if (nwords > (1ull << 31) * 256ull) return LLVQ_EUNSUPPORTED;
    pack_kernel<<<(unsigned)((nwords + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const unsigned long long*>(d_index), gain_bits ? d_gain_index : nullptr, ctx->host.W, gain_bits, nblocks,
        static_cast<uint32_t*>(d_fields), nwords);
    return status_of_launch();
}

}  // extern "C"
