"""Device allocations under memory pressure, on the CPU: the allocation helpers compiled against a fake
CUDA runtime whose cudaMalloc fails when told to. A failed allocation first gives back the memory kept
of destroyed states and is tried once more; a buffer that could not grow is empty and is
allocated anew by the next, smaller request instead of handing out a null pointer."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1507_08157_gb300", "csrc")

RUNTIME = """
#pragma once
#include <cstdlib>
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
inline int fail = 0, live = 0;                     // calls that fail from now on, blocks held
inline cudaError_t cudaMalloc(void **p, size_t n) {
    if (fail > 0) { --fail; return cudaErrorMemoryAllocation; }
    *p = std::malloc(n); ++live; return cudaSuccess;
}
inline cudaError_t cudaFree(void *p) { if (p) { std::free(p); --live; } return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
"""

MAIN = """
#include "device_memory.h"
#include <cstdio>
static bool spare = false;
bool tddft::release_spare_slabs() { const bool had = spare; spare = false; return had; }
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\\n", __LINE__, #x); return 1; }
template <typename F> bool no_memory(F f) { try { f(); } catch (const std::bad_alloc &) { return true; } return false; }
int main() {
    using namespace tddft;
    Scratch s;
    float *p = s.get(100);
    CHECK(p && s.get(50) == p && live == 1);
    fail = 1;                                      // nothing to give back
    CHECK(no_memory([&] { s.get(1000); }) && live == 0);
    CHECK(s.get(50) != nullptr && live == 1);      // not the freed block of 100
    fail = 1, spare = true;                        // a kept state makes room
    CHECK(s.get(2000) != nullptr && !spare && live == 1);
    Mem m;
    fail = 1, spare = true;
    CHECK(m.alloc<double>(0) != nullptr && !spare && live == 2);
    fail = 2, spare = true;
    CHECK(no_memory([&] { m.alloc<int>(7); }) && m.ptrs.size() == 1 && live == 2);
    m.release();
    CHECK(live == 1 && m.ptrs.empty());
    return 0;
}
"""


def test_failed_allocations_leave_nothing_dangling(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([gxx, "-std=c++17", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout


def test_sources_allocate_through_the_helper():
    # the one word that reports expired waits is made once per process, before anything else
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        calls = text.count("cudaMalloc(")
        assert calls == (2 if f == "device_memory.h" else 1 if f == "tc_gemm.cu" else 0), f


BUILD = """
#include "tddft_internal.h"
#include <cstdio>
namespace tddft {
bool fp64_grid_build(cudaStream_t st, Mem &mem, const TileSet<double> &chi, const TileSet<double> &phi,
                     const std::vector<int> &coff, const std::vector<int> &poff, bool quads, Fp64Grid &G);
}
extern "C" {                       // for Mem's inline parts here; the library has its own runtime
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaMalloc(void **, size_t) { return cudaErrorMemoryAllocation; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
}
int main() {
    using namespace tddft;
    TileSet<double> chi{}, phi{};
    chi.ntiles = phi.ntiles = 1;
    Mem mem;
    Fp64Grid G;
    const bool made = fp64_grid_build(nullptr, mem, chi, phi, {0, 8}, {0, 4}, true, G);
    return made || !mem.ptrs.empty() || G.fm || G.pm;
}
"""


def test_float64_digit_tables_that_do_not_fit_leave_the_other_kernels(tmp_path):
    # without a device every allocation fails: no tables, and no error that would refuse the context
    gxx, inc = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.isdir(inc):
        pytest.skip("no g++ or CUDA headers")
    from paper_1507_08157_gb300 import build
    lib = build.build()
    (tmp_path / "build.cpp").write_text(BUILD)
    exe = str(tmp_path / "build")
    subprocess.run([gxx, "-std=c++17", "-I", inc, "-I", CSRC, str(tmp_path / "build.cpp"), lib, "-o", exe], check=True)
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="", LD_LIBRARY_PATH=os.path.dirname(lib))
    res = subprocess.run([exe], capture_output=True, text=True, env=env)
    assert res.returncode == 0, (res.returncode, res.stderr)
