// Pieces shared by all kernels: the device view of a code's tables, the stored-format bit unpacking (S1), the
// packed representation of a decoded point and the gain step (S7).
#pragma once
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "tables.h"

namespace llvq {

// Device view of one code's class tables in global memory (pointers owned by the context).  Codes whose class
// tables fit shared memory use the copies inside the table image instead.
struct DevCode {
    const ClassDesc* cls;           // [nclasses] (codes whose tables fit shared memory: read by the encoder's indexing kernel)
    const BigDesc* big;             // [nclasses] compact records (codes whose class tables stay in global memory)
    const uint64_t* off_lo;         // [nclasses + 1] low 64 bits of the class offsets
    const uint32_t* off_hi;         // [nclasses + 1] bits 64.. of the class offsets
    const uint32_t* lut;            // [2^kBigBucketBits + 1] class of the first index of bucket (I >> (W - kBigBucketBits)), then the last class; codes with class tables in global memory
    unsigned long long* bad_index;  // device counter of fields with I >= N
    uint32_t* flags;                // device error flags
    uint64_t n_lo, n_hi;            // N
    int nclasses;
    int W;
};

// ---- S1: bit unpack --------------------------------------------------------
// Field b occupies stream bits [b*W, (b+1)*W).  Reads only the 32-bit words the field touches.
__device__ __forceinline__ void load_index(const uint32_t* __restrict__ s, uint64_t b, int W, uint64_t& lo, uint64_t& hi)
{
    uint64_t bp = b * (uint64_t)W;
    uint64_t wi = bp >> 5;
    int sh = (int)(bp & 31);
    int nw = (sh + W + 31) >> 5;                        // 1..4 words
    uint32_t w0 = __ldg(s + wi);
    uint32_t w1 = nw > 1 ? __ldg(s + wi + 1) : 0u;
    uint32_t w2 = nw > 2 ? __ldg(s + wi + 2) : 0u;
    uint32_t w3 = nw > 3 ? __ldg(s + wi + 3) : 0u;
    uint64_t a = ((uint64_t)w1 << 32) | w0, c = ((uint64_t)w3 << 32) | w2;
    if (sh) { lo = (a >> sh) | (c << (64 - sh)); hi = c >> sh; }
    else    { lo = a; hi = c; }
    if (W < 64) { lo &= (1ull << W) - 1; hi = 0; }
    else if (W == 64) hi = 0;
    else hi &= (1ull << (W - 64)) - 1;
}

// Field b of a stream of W-bit fields, W <= 64: at most three 32-bit words, the third only when the field reaches it.
__device__ __forceinline__ uint64_t load_field(const uint32_t* __restrict__ stream, uint64_t b, int W)
{
    const uint64_t bp = b * (uint64_t)W;
    const uint32_t* p = stream + (bp >> 5);
    const int sh = (int)(bp & 31);
    const int last = sh + W;                                     // bits of the field counted from the first word
    const uint32_t w0 = __ldg(p);
    const uint32_t w1 = last > 32 ? __ldg(p + 1) : 0u;
    const uint32_t w2 = last > 64 ? __ldg(p + 2) : 0u;
    uint64_t v = (((uint64_t)w1 << 32) | w0) >> sh;
    if (sh) v |= (uint64_t)w2 << (64 - sh);
    return W < 64 ? v & ((1ull << W) - 1) : v;
}

// The 32-bit words that hold a field, as they are in the stream: requested with the loads of one block while another is being
// unranked, put together when the block's turn comes.  kBig: indices above 64 bits (four words), else at most 64 bits (three).
template <bool kBig>
struct RawField {
    uint32_t w0, w1, w2, w3, shift;
};

// The field that starts `bits` bits behind the word p0.
template <bool kBig>
__device__ __forceinline__ RawField<kBig> request_field_at(const uint32_t* __restrict__ p0, uint32_t bits, int W, bool in)
{
    RawField<kBig> f;
    const uint32_t* p = p0 + (bits >> 5);
    f.shift = bits & 31u;
    const uint32_t last = in ? f.shift + (uint32_t)W : 0u;       // bits counted from the first word (0: nothing is read)
    f.w0 = f.w1 = f.w2 = f.w3 = 0u;
    if (last > 0u) asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(f.w0) : "l"(p));
    if (last > 32u) asm volatile("ld.global.nc.u32 %0, [%1+4];" : "=r"(f.w1) : "l"(p));
    if (last > 64u) asm volatile("ld.global.nc.u32 %0, [%1+8];" : "=r"(f.w2) : "l"(p));
    if (kBig && last > 96u) asm volatile("ld.global.nc.u32 %0, [%1+12];" : "=r"(f.w3) : "l"(p));
    return f;
}

template <bool kBig>
__device__ __forceinline__ RawField<kBig> request_field(const uint32_t* __restrict__ stream, uint64_t b, int W, bool in)
{
    const uint64_t bp = b * (uint64_t)W;
    return request_field_at<kBig>(stream + (bp >> 5), (uint32_t)bp & 31u, W, in);
}

// Keeps whatever is formed from the words behind this point.
template <bool kBig>
__device__ __forceinline__ void use_field_from_here(RawField<kBig>& f)
{
    asm volatile("" : "+r"(f.w0), "+r"(f.w1), "+r"(f.w2), "+r"(f.w3));
}

template <bool kBig>
__device__ __forceinline__ void field_value(const RawField<kBig>& f, int W, uint64_t& lo, uint64_t& hi)
{
    const uint32_t v0 = __funnelshift_r(f.w0, f.w1, f.shift), v1 = __funnelshift_r(f.w1, f.w2, f.shift);
    lo = (uint64_t)v1 << 32 | v0;
    hi = 0u;
    if (kBig) {
        const uint32_t v2 = __funnelshift_r(f.w2, f.w3, f.shift);
        if (W > 64) hi = v2 & ((1u << (W - 64)) - 1u);           // W <= 72
        else if (W < 64) lo &= (1ull << W) - 1ull;
    } else if (W < 64) {
        lo &= (1ull << W) - 1ull;
    }
}

// ---- S7: gain ---------------------------------------------------------------
// A 16-bit read-only load that stays where it is written among the other volatile statements (the decoders' table
// reads): issued before a block is unranked, its result is first used when the weights are formed.
__device__ __forceinline__ uint16_t ldg_u16_here(const uint16_t* p)
{
    uint16_t v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ float gain_to_float(uint16_t bits)
{
    asm volatile("" : "+h"(bits));          // the conversion stays behind the volatile statements before it (the load may still be in flight there)
    return __half2float(__ushort_as_half(bits));
}

}  // namespace llvq
