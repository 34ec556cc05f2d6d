"""What the host settles with the CUDA runtime ahead of a launch, against a runtime made of a few fakes (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def _run(tmp_path, source):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    subprocess.check_call([shutil.which("g++") or "c++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_2603_11021_b200", "csrc"),
                           "-I", os.path.join(CUDA, "include"), str(src), "-o", str(exe)])
    return subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)


# two contexts on two threads launch one kernel with different sizes; the first thread's call into the runtime takes effect last
SMEM = r"""
#include "launch_host.h"
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>

static std::mutex m;
static std::condition_variable cv;
static int calls, done, attribute;

cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { *a = {}; a->sharedSizeBytes = 1024; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int value)
{
    std::unique_lock<std::mutex> l(m);
    const int me = calls++;
    cv.notify_all();
    if (me == 0) cv.wait_for(l, std::chrono::seconds(5), [] { return done > 0; });      // set only behind the other thread's
    if (value > 232448 - 1024) return cudaErrorInvalidValue;
    attribute = value;
    ++done;
    cv.notify_all();
    return cudaSuccess;
}

void kernel(int) {}

int main()
{
    static llvq::SmemLimits a, b;
    bool ok[2] = {};
    std::thread first([&] { ok[0] = llvq::allow_smem<kernel>(a, 232448, SIZE_A); });
    { std::unique_lock<std::mutex> l(m); cv.wait_for(l, std::chrono::seconds(5), [] { return calls > 0; }); }
    std::thread second([&] { ok[1] = llvq::allow_smem<kernel>(b, 232448, SIZE_B); });
    first.join(); second.join();
    for (auto* c : {&a, &b})                               // whatever was promised to either, later launches can have
        for (int size : {SIZE_A, SIZE_B}) ok[0] = ok[0] && llvq::allow_smem<kernel>(*c, 232448, size) && attribute >= size;
    const bool refuses = !llvq::allow_smem<kernel>(a, 232448, 232448 - 1023);
    std::printf("%d %d %d\n", ok[0], ok[1], refuses);
    return ok[0] && ok[1] && refuses ? 0 : 1;
}
"""


@pytest.mark.parametrize("a,b", [(200 * 1024, 210 * 1024), (100 * 1024, 200 * 1024)])
def test_two_threads_that_need_different_sizes(tmp_path, a, b):
    r = _run(tmp_path, SMEM.replace("SIZE_A", str(a)).replace("SIZE_B", str(b)))
    assert r.returncode == 0, r.stdout + r.stderr


# a look-up of the driver's function that fails is made again by the next call; a thread without a context gets one
X_MAP = r"""
#include "launch_host.h"
#include <cstdio>

static int lookups, encodes;
static bool bound;

static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box,
                       const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill)
{
    ++encodes;
    return bound && dims[0] == 48 && dims[1] == 3 && strides[0] == 96 && box[1] == 16 ? CUDA_SUCCESS : CUDA_ERROR_INVALID_CONTEXT;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* r)
{
    *fn = lookups ? reinterpret_cast<void*>(encode) : nullptr;
    *r = lookups++ ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int device) { bound = device == 5; return cudaSuccess; }

int main()
{
    CUtensorMap map;
    bool ok[3];
    for (bool& o : ok) o = llvq::make_x_map(5, nullptr, 48, 3, 16, &map);
    std::printf("%d %d %d, %d look-ups, %d calls\n", ok[0], ok[1], ok[2], lookups, encodes);
    return !ok[0] && ok[1] && ok[2] && lookups == 2 && encodes == 3 ? 0 : 1;
}
"""


def test_tensor_map_of_x_after_a_failed_look_up_and_without_a_context(tmp_path):
    r = _run(tmp_path, X_MAP)
    assert r.returncode == 0, r.stdout + r.stderr
