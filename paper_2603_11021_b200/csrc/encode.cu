// Encoder side of the library: nearest point of the code to a real vector (Sec. 3.1, Euclidean and angular
// scoring), point -> index (Sec. 3.2, the inverse of the dequantizer's steps) and packing of the stored fields.
// The paper defers the search itself to the literature; the search here is coset decoding of the whole lattice
// (exact for the unbounded lattice) plus a policy that keeps the result inside the shells of the code.
#include "llvq.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "ctx.h"
#include "tables.h"

using namespace llvq;

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr int kEncWarps = 24;              // vectors in flight per CTA (one CTA per SM), one warp each
constexpr uint32_t kFlagSearchGaveUp = 4u; // LLVQ_FLAG_SEARCH_GAVE_UP

constexpr int kMaxShell = 53;              // llvq_create's limit
constexpr int kMaxCand = 64;               // cosets re-scored in binary64 per search; more (massive ties) means all 8192 are

// Units of the first stage of the search: costs and moves are whole numbers of 1 / kCostScale.  The largest rounding error
// of a coordinate costs 1/4, i.e. 2046: sixteen of them stay below 2^15.
constexpr float kCostScale = 8184.f;
// Two cosets whose first-stage costs differ by more than this are in the same order in exact arithmetic: a cost carries at
// most 25 roundings of half a unit (24 coordinates and one move) and 0.1 from the binary32 errors, twice 12.6 is 25.2.
constexpr uint32_t kCostMargin = 26u;
constexpr uint32_t kParityBit = 0x8000u;   // where a cost carries the parity of its sum of z (adding costs adds the parities mod 2)
constexpr uint32_t kParityCode = 0x7676u;  // a byte-permute selector XOR this trades places with the one of the other parity
constexpr uint32_t kSelEven = 0x3244u;     // {high half of the first operand} stays high, low half zero; ^ kParityCode: moved low

// Per-warp scratch of the lattice search.
struct __align__(128) WarpTables {
    uint2 nib[2][6][16];    // [parity][4 coordinates][bit pattern n]: {cost | move << 16, parity code | move of pattern ~n << 16}; rows of 128 bytes
    uint4 pk[24][2];        // [coordinate, octad by octad][parity] w(b), w(b + 2), w(b + 2), w(b) for offset b = parity:
                            //  w = cost | parity of z << 15 | cost of the other neighbour << 16
    uint32_t cand[kMaxCand - 1];
    uint32_t ncand;
};

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

// Nearest point of the unbounded lattice to u (one coordinate per lane, lanes 0..23; all in units of the integer
// coordinates).  Every lattice point is b + 4 z with b_i = parity + 2 c_i, c a Golay codeword, and sum z = parity
// (mod 2) (the sum rules of Sec. 2.4: all Golay weights are multiples of 4).  For each of the 2 x 4096 cosets the
// best z is the rounded one, with the coordinate of largest rounding error moved to its other neighbour when the
// sum rule fails.
// Two stages.  The first finds the smallest cost over all cosets in whole numbers, along a trio of octads (GolayTrio): per
// parity and octad pattern {w, ~w} the best cost for an even and for an odd sum of z (a move included where the rounded z has
// the other parity), packed as two 16-bit halves; over the 512 triples those add up, the even and odd sums of three octads
// combining to the parity the coset needs.  A minimum over the parities of the three octads never moves more than one
// coordinate where one move is the better choice, so this is the minimum over the 8192 cosets.  A lane holds (parity, x,
// half of the a): 32 pairs (a, b), three instructions each with the packed add-and-minimum of this architecture.
// Every coset within kCostMargin of the smallest cost is then listed (usually one) and evaluated in binary64, coordinate by
// coordinate in lane order, one rounding per operation: its point, and, if there are several, the squared distance as the
// sum over the coordinates in order.  The smallest distance wins, the lowest (parity, codeword position) among equal ones;
// inside a coset the first coordinate with the largest error moves.  The result does not depend on the first stage's
// rounding.  Returns the coordinate of this lane (0 for lanes >= 24) and the squared norm of the point; unique = every other
// lattice point is farther from u by a margin far above any binary64 rounding.
// Bound: the integer / logic pipe (78 % busy, 818 instructions per decode; the shared-memory pipe is at 54 %).  Scoring the 8192
// cosets one by one took about 6000 instructions and was bound by bank conflicts: 38.9 -> 1.13 ms for the 699 050 vectors of a
// 4096 x 4096 matrix (EUCLIDEAN, indexing included), 32.0 -> 2.06 ms for the 174 763 of 1024 x 4096 (ANGULAR on shells 2..12, 11 decodes each).
// Steps on the way: rows of 128 bytes per (parity, nibble) read by the 16 lanes of one parity instead of rows shared by both
// parities (1.38 -> 1.31 ms), roundings by additions instead of conversions and 24 warps drawing their vectors from a shared
// counter instead of fixed strides (-> 1.13 ms).
__device__ __forceinline__ int lattice_nearest(WarpTables& W, const GolayTrio& S, const PatternSteps& steps,
                                               const uint32_t (&row)[6], const uint32_t* __restrict__ golay, const uint16_t* __restrict__ pos_by_low12, double u, int lane, int& norm2, bool& unique)
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

// One warp per input vector; inputs are binary32 values, all scoring runs in binary64 with one rounding per operation and
// sums over the coordinates in order.  EUCLIDEAN: if the nearest lattice point of the input lies in the code it is the
// answer (it is then also the nearest point of the cut, App. E "Spherical shaping").  Otherwise, and for ANGULAR always,
// the input direction is decoded at every shell radius sqrt(16 m); of the candidates inside the code the one nearest to
// the input (EUCLIDEAN) or with the largest cosine (ANGULAR) wins, the first radius on ties.  A zero input gives the
// point of index 0, (4, 4, 0^22), the first point of the first class of Shell(2) (Sec. 2.3).  Needs m_lo == 2 and
// m_hi >= 3 (checked on the host).
// EUCLIDEAN does not need all the radii.  At distance r along the direction d of the input (length R) the nearest point x
// minimises |x|^2 - 2 r <x, d>; two minimisers at radii r < r' therefore satisfy <x, d> <= <x', d>, and
// |x'|^2 - 2 R <x', d> <= |x|^2 - 2 R <x, d> for r < r' <= R (symmetrically for R <= r' < r): the radius next to R that yields a
// point of the code beats all radii beyond it, by the margin that lattice_nearest reports as `unique`.  So the radii are tried
// outwards from R, on each side until such a point is found (inputs so long that a squared distance no longer resolves the
// margin try them all).  ANGULAR needs every radius; the exact score is formed only where a binary32 one comes near the best.
__global__ void __launch_bounds__(kEncWarps * 32, 1)
encode_search_kernel(const uint32_t* __restrict__ golay, EncTables et, const __grid_constant__ PatternSteps steps, const float* __restrict__ v, uint64_t n, int metric, int m_lo, int m_hi,
                     int8_t* __restrict__ points, uint32_t* __restrict__ flags)
{
    extern __shared__ __align__(128) uint8_t enc_smem[];
    WarpTables* tabs = reinterpret_cast<WarpTables*>(enc_smem);
    GolayTrio& S = *reinterpret_cast<GolayTrio*>(enc_smem + kEncWarps * sizeof(WarpTables));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ double radius[kMaxShell + 1];                     // sqrt(16 m)
    __shared__ uint32_t next_vec;
    if (threadIdx.x == 0) next_vec = 0u;
    for (int i = threadIdx.x; i <= m_hi; i += blockDim.x) radius[i] = __dsqrt_rn(__dmul_rn(16.0, (double)i));
    for (int i = threadIdx.x; i < (int)sizeof(GolayTrio) / 4; i += blockDim.x)
        reinterpret_cast<uint32_t*>(&S)[i] = __ldg(reinterpret_cast<const uint32_t*>(et.trio) + i);
    __syncthreads();
    WarpTables& W = tabs[warp];
    uint32_t row[6];                                             // where the nibbles of pattern (x, 4 h) of every octad are
#pragma unroll
    for (int o = 0; o < 3; ++o) {
        const uint32_t p = S.pat[o][(lane & 7) * 8 + ((lane >> 1) & 4)], t = (uint32_t)__cvta_generic_to_shared(&W.nib[lane >> 4][2 * o][0]);
        row[2 * o] = t ^ (p & 15u) * 8u;
        row[2 * o + 1] = (t + 128u) ^ (p >> 4) * 8u;
    }
    const float reach = sqrtf(16.f * (float)m_hi) + 4.01f, reach2 = reach * reach;
    // a CTA's share is contiguous; its warps draw the vectors one by one (some take several decodes, and the schedulers favour some warps)
    const uint64_t first = n / gridDim.x * blockIdx.x + min((uint64_t)blockIdx.x, n % gridDim.x);
    const uint32_t count = (uint32_t)(n / gridDim.x + (blockIdx.x < n % gridDim.x));
    while (true) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(&next_vec, 1u);
        t = __shfl_sync(kFull, t, 0);
        if (t >= count) break;
        const uint64_t vec = first + t;
        const float vf = lane < 24 ? __ldg(v + vec * 24 + lane) : 0.f;
        const double vi = (double)vf;
        int bestx = lane == 0 || lane == 1 ? 4 : 0;              // the point of index 0
        const bool zero = __all_sync(kFull, vf == 0.f), finite = __all_sync(kFull, isfinite(vf));
        bool ok = zero;
        if (!zero && finite) {
            bool direct = false;                                 // the input itself is decoded (else: its direction at shell radius m)
            if (metric == LLVQ_EUCLIDEAN) {
                // no lattice point is farther than 4 from any input (covering radius): beyond radius sqrt(16 m_hi) + 4 the nearest
                // point is certainly outside the code and the decode can be skipped
                float n2f = vf * vf;
#pragma unroll
                for (int o = 16; o; o >>= 1) n2f += __shfl_xor_sync(kFull, n2f, o);
                direct = n2f <= reach2;
            }
            double rn = 0.0, best = -1.0e300;
            float best_f = -2.f;
            int best_m = 0, m = 0, m_start = 0, step = 0;        // step 0: the radii have not been started
            bool outwards = false;
            while (true) {                                       // (one copy of the search in the code: two would not fit the instruction cache)
                if (!direct) {
                    if (step == 0) {
                        const double n2 = seq_sum24(__dmul_rn(vi, vi));
                        rn = __ddiv_rn(1.0, __dsqrt_rn(n2));
                        outwards = metric == LLVQ_EUCLIDEAN && n2 < 1.0e9;
                        // tried outwards: first down from the largest radius not above R, then up from the next one
                        m = m_start = outwards ? max(m_lo - 1, (int)fmin(n2 * 0.0625, (double)m_hi)) : m_hi;
                        step = -1;
                    }
                    if (step < 0 && m < m_lo) { m = m_start + 1; step = 1; }
                    if (m > m_hi) break;
                }
                const double u = direct ? vi : __dmul_rn(__dmul_rn(vi, rn), radius[m]);
                int norm2;
                bool unique;
                const int x = lattice_nearest(W, S, steps, row, golay, et.pos_by_low12, u, lane, norm2, unique);
                const bool in_code = norm2 >= 16 * m_lo && norm2 < 16 * m_hi + 16;
                if (direct) {
                    if (in_code) { ok = true; bestx = x; break; }
                    direct = false;
                    continue;
                }
                const int m_now = m;
                m += step;
                if (!in_code) continue;
                double score;
                if (metric == LLVQ_EUCLIDEAN) {
                    const double dd = __dsub_rn(vi, (double)x);
                    score = -seq_sum24(lane < 24 ? __dmul_rn(dd, dd) : 0.0);
                } else {
                    float s = (float)__dmul_rn(vi, rn) * (float)x;
#pragma unroll
                    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
                    s *= rsqrtf((float)norm2);
                    if (s < best_f - 1.0e-5f) continue;          // binary32 errors stay below 3e-6
                    best_f = fmaxf(best_f, s);
                    const double dot = seq_sum24(lane < 24 ? __dmul_rn(__dmul_rn(vi, rn), (double)x) : 0.0);
                    score = __ddiv_rn(dot, __dsqrt_rn((double)norm2));
                }
                if (!ok || score > best || (score == best && m_now < best_m)) { best = score; bestx = x; best_m = m_now; ok = true; }
                if (outwards && unique) {                        // this side is done
                    if (step > 0) break;
                    m = m_lo - 1;
                }
            }
        }
        if (!ok) {
            bestx = lane == 0 || lane == 1 ? 4 : 0;
            if (lane == 0) atomicOr(flags, kFlagSearchGaveUp);
        }
        if (lane < 24) points[vec * 24 + lane] = (int8_t)bestx;
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
// Bound: instruction issue and dependent reads (class record, codeword).  With a loop over the 24 coordinates per value, and the free
// slots gathered bit by bit, encoding 699 050 Gaussian vectors (EUCLIDEAN) took 1126 us in all; 1063 us with masks.
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
    const size_t smem = kEncWarps * sizeof(WarpTables) + sizeof(GolayTrio);
    if (!allow_smem<encode_search_kernel>(ctx->smem_limits, ctx->smem_most, smem)) return LLVQ_ECUDA;
    PatternSteps steps;
    for (int o = 0; o < 3; ++o)
        for (int j = 0; j < 4; ++j) { steps.lo[o][j] = (ctx->trio.pat[o][j] & 15u) * 8u; steps.hi[o][j] = (uint32_t)(ctx->trio.pat[o][j] >> 4) * 8u; }
    const unsigned grid = (unsigned)std::min<uint64_t>(nblocks, (uint64_t)ctx->sm_count);
    encode_search_kernel<<<grid, kEncWarps * 32, smem, st>>>(ctx->d_golay, ctx->enc, steps, d_v_f32, nblocks, metric, ctx->host.m_lo, ctx->host.m_hi,
                                                            d_points, ctx->dev.flags);
    if (int e = status_of_launch()) return e;
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
