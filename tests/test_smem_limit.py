"""Host-only: a kernel's limit of dynamic shared memory while threads with launches of different sizes make their first calls (the runtime's
calls replaced by ones that play the order)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """#include "fdc_internal.h"
#include <cstdio>
#include <functional>
static int allowed = 48 * 1024;                      // of the kernel, as the runtime holds it
static std::function<void()> before, after;          // what another thread does around the first call that sets it
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 227 * 1024; return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { *a = {}; a->sharedSizeBytes = 64; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v)
{
    if (v > 227 * 1024 - 64) return cudaErrorInvalidValue;
    auto f = before, g = after;
    before = after = nullptr;
    if (f) f();
    allowed = v;
    if (g) g();
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = 74; return cudaSuccess; }
}
namespace fdc { int set_cuda_error(cudaError_t) { return FDC_ERR_CUDA; } }
static fdc::SmemLimit limit;
static fdc::PairsPlaceable placeable;
static bool launch(bool ask, size_t bytes)           // as the launchers do it: false if the runtime would refuse the launch
{
    if (ask && placeable.all(nullptr, 384, bytes, 148, limit) != FDC_OK) return false;
    return fdc::raise_dynamic_smem(nullptr, bytes, limit) == FDC_OK && bytes <= (size_t)allowed;
}
int main(int, char** v)
{
    const bool ask = v[1][0] == '1';
    const size_t small = 190 * 1024, large = 226 * 1024;
    bool ok = true;
    before = after = [&] { ok = launch(ask, large) && ok; };         // the other thread's first two launches
    ok = launch(ask, small) && ok;
    ok = launch(ask, large) && launch(ask, small) && ok;
    ok = !launch(false, 228 * 1024) && ok;           // more than there is: still refused
    puts(ok ? "ok" : "refused");
}
"""


@pytest.mark.parametrize("ask", ["0", "1"], ids=["launcher", "placement_asked_first"])
def test_first_calls_of_two_threads(tmp_path, ask):
    (tmp_path / "s.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2602_02864_b200", "csrc"),
                           "-I", "/usr/local/cuda/include", str(tmp_path / "s.cpp"), "-o", str(tmp_path / "s")])
    assert subprocess.run([str(tmp_path / "s"), ask], capture_output=True, text=True).stdout.strip() == "ok"
