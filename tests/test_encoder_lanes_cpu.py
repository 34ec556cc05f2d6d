"""The encoder's search with a thread block of lanes that do not run in step (no GPU).  CUDA promises that lanes of a warp meet only where a barrier, a
shuffle or a vote says so.  Here the kernel's own text runs on the CPU, every lane on a stack of its own, and whoever runs goes on to the next
such meeting before anyone else moves.  Errors are a shuffle from a lane that is not among those named, a meeting that some lane never comes
to, and a table entry read or overwritten with no barrier between the lanes that share it."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_11021_b200", "csrc")

LANES = r"""
#include <ucontext.h>
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <vector>
#include "llvq.h"
#include "tables.h"

#define __device__
#define __global__
#define __grid_constant__
#define __noinline__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __align__(n) __attribute__((aligned(n)))
using std::isfinite; using std::max; using std::min;
struct uint2 { uint32_t x, y; };
struct alignas(16) uint4 { uint32_t x, y, z, w; };
struct alignas(16) float4 { float x, y, z, w; };
struct Dim { unsigned x; };
static uint2 make_uint2(uint32_t x, uint32_t y) { return {x, y}; }
static uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return {x, y, z, w}; }
struct EncTables { const uint16_t* pos_by_low12; const llvq::GolayTrio* trio; };

// ---- lanes ----
struct Lane {
    ucontext_t at;
    std::vector<char> stack = std::vector<char>(256 * 1024);
    enum { kRuns, kAtWarp, kAtBlock, kDone } state = kRuns;
    uint32_t mask = 0, orders = 1;       // orders: barriers of the warp or the block this lane has passed
    uint64_t value = 0, seen[32];        // what this lane brought; what everyone brought (block: the total)
};
static std::vector<Lane> lanes;
static ucontext_t scheduler;
static Dim threadIdx, blockIdx{0}, blockDim, gridDim{1};
[[noreturn]] static void fail(const char* what) { std::fprintf(stderr, "lane %u of warp %u: %s\n", threadIdx.x & 31, threadIdx.x >> 5, what); std::_Exit(2); }

static void leave(Lane& me)
{
    const unsigned who = threadIdx.x;
    if (swapcontext(&me.at, &scheduler)) std::abort();
    threadIdx.x = who;
}

// All lanes of the mask meet; the last one to come goes on at once.
static Lane& meet(uint32_t mask, uint64_t value)
{
    const unsigned warp0 = threadIdx.x & ~31u;
    Lane& me = lanes[threadIdx.x];
    if (!(mask >> (threadIdx.x & 31) & 1)) fail("not one of the lanes it names");
    me.state = Lane::kAtWarp; me.mask = mask; me.value = value;
    for (unsigned i = 0; i < 32; ++i)
        if ((mask >> i & 1) && (lanes[warp0 + i].state != Lane::kAtWarp || lanes[warp0 + i].mask != mask)) { leave(me); return me; }
    for (unsigned i = 0; i < 32; ++i)
        if (mask >> i & 1) {
            for (unsigned j = 0; j < 32; ++j) lanes[warp0 + i].seen[j] = lanes[warp0 + j].value;
            lanes[warp0 + i].state = Lane::kRuns;
        }
    return me;
}

static uint64_t meet_block(uint64_t value)
{
    Lane& me = lanes[threadIdx.x];
    me.state = Lane::kAtBlock; me.value = value;
    uint64_t total = 0;
    for (Lane& l : lanes) {
        if (l.state != Lane::kAtBlock) { leave(me); return me.seen[0]; }
        total += l.value;
    }
    for (Lane& l : lanes) { l.state = Lane::kRuns; l.seen[0] = total; ++l.orders; }
    return total;
}

template <typename F> static void run_block(unsigned threads, bool descending, F kernel)
{
    static F* entry;
    entry = &kernel;
    blockDim.x = threads;
    lanes = std::vector<Lane>(threads);
    for (Lane& l : lanes) {
        getcontext(&l.at);
        l.at.uc_stack.ss_sp = l.stack.data(); l.at.uc_stack.ss_size = l.stack.size(); l.at.uc_link = &scheduler;
        makecontext(&l.at, +[] { (*entry)(); lanes[threadIdx.x].state = Lane::kDone; }, 0);
    }
    for (bool moved = true; moved;) {
        moved = false;
        for (unsigned i = 0; i < threads; ++i) {
            const unsigned t = descending ? threads - 1 - i : i;
            if (lanes[t].state != Lane::kRuns) continue;
            threadIdx.x = t;
            moved = true;
            if (swapcontext(&scheduler, &lanes[t].at)) std::abort();
        }
    }
    for (unsigned t = 0; t < threads; ++t)
        if (lanes[t].state != Lane::kDone) { threadIdx.x = t; fail("waits for lanes that do not come"); }
}

// ---- what the kernel calls ----
template <typename T> static uint64_t bits_of(T v) { uint64_t b = 0; std::memcpy(&b, &v, sizeof v); return b; }
template <typename T, typename S> static T as(S b) { T v; std::memcpy(&v, &b, sizeof v); return v; }
template <typename T> static T __shfl_sync(uint32_t mask, T v, int from)
{
    if (!(mask >> (from & 31) & 1)) fail("shuffle from a lane that is not among those it names");
    return as<T>(meet(mask, bits_of(v)).seen[from & 31]);
}
template <typename T> static T __shfl_xor_sync(uint32_t mask, T v, int other) { return __shfl_sync(mask, v, (int)(threadIdx.x & 31) ^ other); }
static void __syncwarp() { ++meet(~0u, 0).orders; }
static uint32_t __ballot_sync(uint32_t mask, bool p)
{
    Lane& me = meet(mask, p);
    uint32_t r = 0;
    for (int i = 0; i < 32; ++i) r |= (uint32_t)((mask >> i & 1) && me.seen[i]) << i;
    return r;
}
static bool __any_sync(uint32_t mask, bool p) { return __ballot_sync(mask, p) != 0; }
static bool __all_sync(uint32_t mask, bool p) { return __ballot_sync(mask, p) == mask; }
template <typename T, typename F> static T reduce(uint32_t mask, T v, F f)
{
    Lane& me = meet(mask, bits_of(v));
    for (int i = 0; i < 32; ++i) if ((mask >> i & 1) && i != (int)(threadIdx.x & 31)) v = f(v, as<T>(me.seen[i]));
    return v;
}
static int __reduce_add_sync(uint32_t m, int v) { return reduce(m, v, [](int a, int b) { return a + b; }); }
static uint32_t __reduce_max_sync(uint32_t m, uint32_t v) { return reduce(m, v, [](uint32_t a, uint32_t b) { return max(a, b); }); }
static uint32_t __reduce_min_sync(uint32_t m, uint32_t v) { return reduce(m, v, [](uint32_t a, uint32_t b) { return min(a, b); }); }
static uint32_t __activemask() { return 1u << (threadIdx.x & 31); }      // no one else need be here
static void __syncthreads() { meet_block(0); }
static int __syncthreads_count(bool p) { return (int)meet_block(p); }
static bool __syncthreads_and(bool p) { return meet_block(p) == lanes.size(); }
static uint32_t atomicAdd(uint32_t* p, uint32_t v) { const uint32_t old = *p; *p += v; return old; }
static void atomicOr(uint32_t* p, uint32_t v) { *p |= v; }
template <typename T> static T __ldg(const T* p) { return *p; }
static int __popc(uint32_t v) { return __builtin_popcount(v); }
static int __ffs(uint32_t v) { return __builtin_ffs((int)v); }
static int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }
static uint32_t __byte_perm(uint32_t x, uint32_t y, uint32_t s)
{
    const uint64_t all = (uint64_t)y << 32 | x;
    uint32_t r = 0;
    for (int i = 0; i < 4; ++i) r |= (uint32_t)(all >> 8 * (s >> 4 * i & 7) & 0xff) << 8 * i;
    return r;
}
static uint32_t __vminu2(uint32_t a, uint32_t b) { return min(a >> 16, b >> 16) << 16 | min(a & 0xffffu, b & 0xffffu); }
static uint32_t __vimin3_u16x2(uint32_t a, uint32_t b, uint32_t c) { return __vminu2(__vminu2(a, b), c); }
static uint32_t __viaddmin_u16x2(uint32_t a, uint32_t b, uint32_t c) { return __vminu2(((a >> 16) + (b >> 16)) << 16 | ((a + b) & 0xffffu), c); }
static int __dp4a(int a, int b, int c) { for (int i = 0; i < 32; i += 8) c += (int)(int8_t)(a >> i) * (int8_t)(b >> i); return c; }
static double __dadd_rn(double a, double b) { return a + b; }
static double __dsub_rn(double a, double b) { return a - b; }
static double __dmul_rn(double a, double b) { return a * b; }
static double __ddiv_rn(double a, double b) { return a / b; }
static double __dsqrt_rn(double a) { return std::sqrt(a); }
static uint32_t __float_as_uint(float v) { return as<uint32_t>(v); }
static float __uint_as_float(uint32_t v) { return as<float>(v); }
static long long __double_as_longlong(double v) { return as<long long>(v); }
static double __longlong_as_double(long long v) { return as<double>(v); }
static int __double2loint(double v) { return (int)(uint32_t)as<uint64_t>(v); }
static int __double2hiint(double v) { return (int)(as<uint64_t>(v) >> 32); }
alignas(1024) static uint8_t enc_smem[232448];
static size_t __cvta_generic_to_shared(const void* p) { return (size_t)(static_cast<const uint8_t*>(p) - enc_smem); }
// Shared memory, 8 bytes at a time: lanes of a warp see each other's only across a barrier (shuffles and votes order no memory).
static struct { uint32_t writer, written, read[32]; } uses[sizeof enc_smem / 8];
static uint2 read_shared(uint32_t a)
{
    if (a % 8 || a + 8 > sizeof enc_smem) fail("read outside shared memory");
    auto& u = uses[a / 8];
    const uint32_t now = lanes[threadIdx.x].orders;
    if (u.writer != threadIdx.x && u.written >= now) fail("read of what another lane wrote, with no barrier between them");
    u.read[threadIdx.x & 31] = now;
    uint2 v;
    std::memcpy(&v, enc_smem + a, 8);
    return v;
}
static void write_shared(uint32_t a, uint32_t x, uint32_t y)
{
    if (a % 8 || a + 8 > sizeof enc_smem) fail("write outside shared memory");
    auto& u = uses[a / 8];
    const uint32_t now = lanes[threadIdx.x].orders;
    for (uint32_t i = 0; i < 32; ++i)
        if (i != (threadIdx.x & 31) && u.read[i] >= now) fail("write over what another lane has read, with no barrier between them");
    u.writer = threadIdx.x; u.written = now;
    const uint2 v{x, y};
    std::memcpy(enc_smem + a, &v, 8);
}
"""

MAIN = r"""
int main(int, char** argv)
{
    const int metric = std::atoi(argv[1]), m_hi = std::atoi(argv[2]), n = std::atoi(argv[3]);
    const bool descending = std::atoi(argv[4]) != 0;
    HostTables h;
    GolayTrio trio;
    if (!build_tables(2, m_hi, h) || !build_golay_trio(h, trio)) return 3;
    std::vector<uint16_t> pos(4096);
    for (int i = 0; i < 4096; ++i) pos[h.golay[i] & 0xfffu] = (uint16_t)i;
    PatternSteps steps;
    for (int o = 0; o < 3; ++o)
        for (int j = 0; j < 4; ++j) { steps.lo[o][j] = (trio.pat[o][j] & 15u) * 8u; steps.hi[o][j] = (uint32_t)(trio.pat[o][j] >> 4) * 8u; }
    std::vector<float> v((size_t)n * 24 + 4);
    std::vector<int8_t> points((size_t)n * 24);
    if (std::fread(v.data(), 4, (size_t)n * 24, stdin) != (size_t)n * 24) return 4;
    std::memset(enc_smem, 0xa5, sizeof enc_smem);
    uint32_t flags = 0;
    run_block(kEncWarps<kForm> * 32, descending, [&] {
        encode_search_kernel<kForm>(h.golay.data(), EncTables{pos.data(), &trio}, steps, v.data(), (uint64_t)n, metric, 2, m_hi, points.data(), &flags);
    });
    std::fwrite(points.data(), 1, points.size(), stdout);
    return 0;
}
"""


@pytest.fixture(scope="module", params=["two lanes per vector", "a warp per vector"])
def search(request, tmp_path_factory):
    """The kernel in one of its forms as a program: input vectors -> points."""
    text = open(os.path.join(CSRC, "encode.cu")).read()
    text = text[text.index("using namespace llvq;"):text.index("template <int kBit>")] + "\n}  // namespace\n"
    for pattern, to in [(r'asm volatile\("ld\.shared\.v2[^;]*;[^;]*;', "v = read_shared(a);"), (r'asm volatile\("st\.shared\.v2[^;]*;[^;]*;', "write_shared(a, x, y);"),
                        (r'asm volatile\("prefetch[^;]*;[^;]*;', ";"), (r"extern __shared__ [^;]*;", "")]:
        text, found = re.subn(pattern, to, text)
        assert found == 1, pattern
    text = text.replace("__shared__ ", "static ")
    assert "asm" not in text
    d = tmp_path_factory.mktemp("lanes")
    (d / "t.cpp").write_text(LANES + text + MAIN.replace("kForm", str(request.param == "two lanes per vector").lower()))
    subprocess.check_call([shutil.which("g++") or "c++", "-O1", "-std=c++17", "-w", "-ffp-contract=off", "-fno-strict-aliasing", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                           str(d / "t.cpp"), os.path.join(CSRC, "tables.cpp"), "-o", str(d / "t")])

    def run(v, metric, m_hi, descending):
        r = subprocess.run([str(d / "t"), str(metric), str(m_hi), str(len(v)), str(int(descending))], input=v.astype(np.float32).tobytes(), capture_output=True, timeout=300)
        assert r.returncode == 0, r.stderr.decode()
        return np.frombuffer(r.stdout, dtype=np.int8).reshape(len(v), 24)
    return run


def _check(oracle_mod, search, v, metric, m_hi, descending):
    want, _ = oracle_mod.Code(2, m_hi).encode(v.astype(np.float64), getattr(oracle_mod, metric), threads=4)
    assert np.array_equal(search(v, getattr(oracle_mod, metric), m_hi, descending), want)


@pytest.mark.parametrize("descending", [False, True])
@pytest.mark.parametrize("metric,m_hi", [("EUCLIDEAN", 13), ("ANGULAR", 5)])
def test_list_of_waiting_vectors(oracle_mod, search, metric, m_hi, descending):
    # so few vectors that all of them go through a block's list
    v = (np.random.default_rng(22).standard_normal((40, 24)) * 2.5).astype(np.float32)
    v[::4] = np.round(v[::4] * 2) / 2
    _check(oracle_mod, search, v, metric, m_hi, descending)


@pytest.mark.parametrize("descending", [False, True])
def test_tables_are_read_after_all_their_lanes_have_written(oracle_mod, search, descending):
    # near points of the code: one candidate each, all of them found in the tables; more vectors than a block has at a time, so that some are replaced
    rng, o = np.random.default_rng(23), oracle_mod.Code(2, 13)
    v = o.unrank([o.N // 330 * j + 5 for j in range(330)]) + 0.3 * rng.standard_normal((330, 24))
    _check(oracle_mod, search, v.astype(np.float32), "EUCLIDEAN", 13, descending)
