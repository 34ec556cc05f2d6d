// Host-side table generator of the LLVQ library: Golay codewords, class list
// with cardinalities and offsets, per-class unranking descriptors.
// Written independently of the test oracle; the two are compared in the tests.
#pragma once
#include <cstdint>
#include <vector>

namespace llvq {

typedef unsigned __int128 u128;

constexpr int kDim = 24;
constexpr int kMaxLevels = 8;

// One "choose k of the slots still free" step of the arrangement unranking (App. A step 4).
struct LevelDesc {
    uint32_t radix;   // C(n, k)
    uint8_t k;        // slots taken by this value
    uint8_t val;      // absolute value placed
    uint8_t n;        // slots free before this step
    uint8_t pad;
};
static_assert(sizeof(LevelDesc) == 8, "LevelDesc layout");

// Everything the kernels need to rebuild a point of one class from its
// class-local index (App. A steps 3-4).  Group 1 = positions F1(c) (values
// = 2 mod 4 of an even class); group 0 = positions F0(c) of an even class, or
// all 24 positions of an odd class.
struct ClassDesc {
    uint8_t parity;    // 0 even, 1 odd
    uint8_t w;         // even: Golay weight required (= #coordinates 2 mod 4)
    uint8_t B;         // free sign bits
    uint8_t signpar;   // even: (#values 4 mod 8 + #values 6 mod 8) & 1
    uint8_t nlev1;     // unranking steps in group 1
    uint8_t nlev0;     // unranking steps in group 0
    uint8_t fill1;     // value filling the rest of group 1 (unused if w == 0)
    uint8_t fill0;     // value filling the rest of group 0
    uint16_t goff;     // first admissible codeword in the sorted Golay table
    uint16_t A;        // number of admissible codewords
    uint32_t m;        // shell
    LevelDesc lev[kMaxLevels];   // group-1 steps first, then group-0 steps
};
static_assert(sizeof(ClassDesc) == 16 + 8 * kMaxLevels, "ClassDesc layout");

// Compact form of ClassDesc for the codes whose class tables stay in global memory (32 bytes, two 16-byte loads): the
// radix of a step is C(free slots, k) from the Pascal triangle in shared memory and its reciprocals come from two tables
// beside it, so only the multiplicities and the values are stored per class.  Value ids: 0 = filler of group 0,
// 1 = filler of group 1, 2 + l = level l.
struct BigDesc {
    uint8_t w, B;
    uint8_t flags;         // bit0 parity, bit1 signpar, bit2 fill0 is nonzero, bit3 fill1 has value bit 1, bit4 fill0 has value bit 1
    uint8_t nlev;          // nlev1 | (nlev1 + nlev0) << 4
    uint16_t goff, A;
    uint8_t val[8];        // absolute value of ids 0..7
    uint8_t k[8];          // slots taken by level 0..7 (bytes 7 unused: at most 7 levels)
    uint8_t val8;          // absolute value of id 8 (classes with 9 distinct values)
    uint8_t lvl_bit1;      // bit l: the value of level l has value bit 1 (= 2 or 3 mod 4)
    uint8_t lvl_nz;        // bit l: the value of level l is nonzero
    uint8_t small_k;       // bit l: level l takes at most kSmallSubsetMaxK slots (part of the sorted layouts' key)
    uint32_t pad;
};
static_assert(sizeof(BigDesc) == 32, "BigDesc layout");

struct ClassInfo {           // host-only description, for queries and tests
    int m, parity, w, B;
    uint64_t A;
    u128 card, offset;
    std::vector<int> values, mults;   // distinct absolute values descending
};

struct HostTables {
    int m_lo = 0, m_hi = 0, W = 0;
    u128 N = 0;
    std::vector<uint32_t> golay;          // 4096 words sorted by (weight, value)
    int woff[25] = {0}, wcnt[25] = {0};
    std::vector<ClassInfo> info;
    std::vector<ClassDesc> desc;
    std::vector<u128> offset;             // nclasses + 1 entries, offset[nclasses] = N
    uint32_t pascal[25 * 25] = {0};       // C(n, k) at [n * 25 + k]
    int max_levels = 0;
};

// Returns false if the code is outside what the kernels support.
bool build_tables(int m_lo, int m_hi, HostTables& out);

}  // namespace llvq

// ---------------------------------------------------------------------------
// Shared-memory table image for codes with few classes ("fast path"): one
// contiguous blob, copied into every CTA's shared memory by bulk copies.
// ---------------------------------------------------------------------------
namespace llvq {

constexpr int kBigBucketBits = 20;     // buckets of the class lookup of codes with class tables in global memory (4 MB, in L2): the bisection between a bucket's first
                                       // and last class takes 1.4 steps per warp of the 72-bit code (2^16 buckets: 4.4); some buckets hold thousands of classes
constexpr int kFastMaxLevels = 4;      // unranking steps per class on the fast path
constexpr int kFastDescValsOdd = 18;   // words 18, 19: absolute value of id 0..7 in the numbering of the odd-only decoder form
constexpr int kFastDescRnorm = 16;     // word holding 1 / sqrt(16 m) as binary32
constexpr int kFastDescMagic0 = 17;    // word holding floor(2^32 / radix) of level 0 (used when the arrangement rank fits 32 bits)
constexpr uint32_t kFastFlagRank32 = 32u;   // descriptor flag: the class has fewer than 2^32 arrangements
constexpr int kSmallSubsetMaxK = 3;    // the table of all k-subsets of 24 slots covers k = 0..3
constexpr int kSmallSubsetWords = 4 + 1 + 24 + 276 + 2024;   // [first entry of k = 0..3][the subsets, by k, each group in numeric order]
constexpr int kSub2MaxK = 2;
constexpr int kSub2Words = 4 + 1 + 24 + 276;
constexpr int kFastDescStride = 20;    // words between descriptors: 80 bytes spread consecutive classes over all bank groups
constexpr int kLowBits = 14;           // slots resolved by one table lookup in the subset unranking

// Where the decoders keep the 24 coordinates in a 32-bit mask: coordinate 6 g + 2 r + n is bit 8 g + 4 n + r (g = 0..3, r = 0..2,
// n = 0, 1).  Byte g holds a group of six coordinates, which is what a deposit into free positions works on (the order inside a
// byte does not matter there, its table returns the bits where they belong); and bit r of the eight nibbles belongs to the
// coordinate pairs (2 r, 2 r + 1) of the four groups, so that a mask and two shifts turn bit planes into byte-permute
// selectors (expand_bf16).  Bits 3 and 7 of a byte are free.
constexpr uint32_t kAllCoords = 0x77777777u;
inline uint32_t coord_bit(int i) { return 1u << (8 * (i / 6) + 4 * (i & 1) + (i % 6) / 2); }
inline uint32_t coords_of(uint32_t dense)      // bit i = coordinate i -> the layout above
{
    uint32_t m = 0;
    for (int i = 0; i < kDim; ++i) if ((dense >> i) & 1u) m |= coord_bit(i);
    return m;
}
// The free bits of a codeword in the image name its last coordinate: bits 3, 7, 11, 15, 19 = bits 4..0 of that coordinate's bit
// position, gathered by one multiplication (no sums collide).  The zero word names bit 31, which belongs to no coordinate.
constexpr uint32_t kLastPosBits = 0x00088888u, kLastPosGather = 0x10842100u;


// Byte offsets of the parts of the image (all 16-byte aligned) and scalars the kernels need.
struct FastLayout {
    uint32_t golay;       // u32[4096] in the layout of coords_of, the last coordinate named in the free bits
    uint32_t lut;         // u16[4096]  class of the first index of bucket (I >> lut_shift)
    uint32_t pascal;      // u32[25*25]; images with class tables hold the rows from 14 on only (the offset is still that of row 0)
    uint32_t base14;      // u32[16]: [k] = first entry of the k-subsets of 14 slots in r14
    uint32_t r14;         // u16[16384]: the k-subsets of 14 slots as bit masks, k = 0..14, each in numeric order
    uint32_t pd6;         // u8[0x78 * 64]: [f << 6 | (s ^ (f & 63))] = low bits of s deposited into the coordinates of a byte f, lowest first
    uint32_t off;         // u64[ncls + 1]
    uint32_t desc;        // u32[ncls][kFastDescStride]
    uint32_t total;       // bytes of the image proper, multiple of 16
    uint32_t recip64;     // binary64[25*25] 1 / C(n, k) rounded down and
    uint32_t recip32;     // u32[25*25] floor(2^32 / C(n, k)) (0xffffffff for C = 1): images without class tables only, else 0
    uint32_t sub3;        // u32[kSmallSubsetWords], behind the image proper: kernels with room for it load total_ext bytes
    uint32_t sub2;        // u32[kSub2Words], behind sub3: directory and subsets for k = 0..2 in the layout of coords_of
    uint32_t total_ext;   // bytes including sub3 and sub2, multiple of 16
    uint32_t lut_shift;
    uint32_t ncls;
    uint32_t W;
};

// Word layout of a fast descriptor:
//  0: w | B << 8 | flags << 16 | nlev1 << 24 | nlev << 28
//       flags: bit0 parity, bit1 signpar, bit2 fill0 is nonzero, bit3 fill1 has value bit 1, bit4 fill0 has value bit 1,
//              bit5 the arrangement rank of the class fits 32 bits, bits 6-7 decoder form (0 even with weight 8 / 12 / 16, 1 odd, 2 other)
//  1: goff | A << 16
//  2,3: 1 / A as binary64, rounded down
//  4,5: absolute value of id 0..7 (one byte each): id 0 = fill0, id 1 = fill1, ids 2.. = levels in order
//  6,7: 1 / radix of level 0 as binary64, rounded down
//  8..11: level l: radix | k << 22 | id << 27 | (value bit 1) << 30 | (value nonzero) << 31; steps the class does not have:
//         radix 1, k 0, reciprocals 1.0 / 0xffffffff (dividing by them leaves the rank unchanged and gives remainder 0)
//  12..14: floor(2^32 / radix) of levels 1..3
//  15: n (free slots before the step) of levels 0..3, one byte each
//  16: binary32 bits of 1 / |x| = 1 / sqrt(16 m) (formed in binary64, rounded once), for the shape-gain form
//  17: floor(2^32 / radix) of level 0
//  18,19: odd classes: absolute value of id 0..7 with id 0 = fill0 and ids 1.. = levels in order (the form that decodes odd
//         classes alone numbers the levels from 1: there is no group 1 whose filler would take id 1)
// with_classes = false builds only the class-independent tables (Golay, Pascal, subsets, deposit): codes whose class
// tables do not fit shared memory keep those in global memory.
bool build_fast_image(const HostTables& t, FastLayout& layout, std::vector<uint8_t>& image, bool with_classes = true);
void build_big_descs(const HostTables& t, std::vector<BigDesc>& out);
void build_bucket_table(const HostTables& t, std::vector<uint32_t>& lut);   // see tables.cpp

// Encoder side (point -> class).  Signature of a class: sum over its 24 absolute values of a fixed pseudo-random
// 64-bit number per value (the multiset fixes shell and parity).  build_class_hash() fills an open-addressing
// table (linear probing from (signature >> 20) & (size - 1), key 0 = empty) and returns false if two classes of the
// code share a signature.
uint64_t sig_of_value(int a);
bool build_class_hash(const HostTables& t, std::vector<uint64_t>& keys, std::vector<uint32_t>& cls);

// The Golay code cut along a trio of octads (three disjoint codewords of weight 8).  Restricted to one octad the codewords
// are the 128 words of even weight, complementing a codeword on one octad gives another codeword, and up to complements
// the code is { (s[x, a], s[x, b], s[x, a ^ b]) : x, a, b = 0..7 }: 512 triples, each standing for 8 codewords
// (Conway & Sloane, "Sphere Packings, Lattices and Groups", ch. 11: the Turyn construction).  s[x, a] is linear: the sum of a word
// of the [8, 4] code spanned by kTurynX and 0xff and one of that spanned by kTurynA and 0xff, which have only 0 and 0xff in common.
constexpr uint32_t kTurynA[3] = {0x1e, 0x66, 0xaa}, kTurynX[3] = {0x36, 0x5a, 0x8e};
struct GolayTrio {
    uint32_t word[3][64];   // [octad][x * 8 + a] the codeword's bits on the octad, as bits of the 24 coordinates
    uint32_t ones[3];       // the octads
    uint8_t pat[3][64];     // the same bits packed: bit p = coordinate coord[8 * octad + p]; the same for all three octads
    uint8_t coord[24];      // coordinates octad by octad, in the order that makes the patterns those of kTurynA and kTurynX
};
bool build_golay_trio(const HostTables& t, GolayTrio& out);

}  // namespace llvq
