"""Host-only: what the cluster kernels use instead of divisions, against the division."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """#include "fdc_internal.h"
#include <cstdio>
int main() {
    for (uint32_t n = 1; n < 256; ++n) {
        const uint32_t inv = fdc::div_inverse((int)n), top = n <= 16 ? 1u << 28 : 1u << 24;
        auto by = [&](uint32_t x) { return fdc::div_by(x, inv); };
        for (uint32_t k = 0; k < 20000; ++k)
            for (uint32_t x : {k, k * n, k * n + n - 1, top - 1 - k, (top - 1) / n * n - k % 2})
                if (x < top && by(x) != x / n) { printf("%u / %u\\n", x, n); return 1; }
        if (n <= 16)
            for (int parts = 0; parts < 3000; ++parts)
                for (int r = 0; r <= (int)n; ++r)
                    if (fdc::run_begin(r, (int)n, parts, by) != (int)((long long)r * parts / n)) { printf("run %d %u %d\\n", r, n, parts); return 1; }
    }
    puts("ok");
}
"""


def test_inverse_and_runs(tmp_path):
    (tmp_path / "d.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2602_02864_b200", "csrc"),
                           "-I", "/usr/local/cuda/include", str(tmp_path / "d.cpp"), "-o", str(tmp_path / "d")])
    assert subprocess.run([str(tmp_path / "d")], capture_output=True, text=True).stdout.strip() == "ok"
