"""Host-only checks of the C-ABI library: it loads, exports every symbol the header
declares, and rejects bad arguments before touching a device."""
import ctypes
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2602_02864_b200 import build
    build.build()
    from paper_2602_02864_b200 import fdc
    return fdc


def test_exports_match_header(lib):
    hdr = open(os.path.join(ROOT, "include", "fdc.h")).read()
    hdr = re.sub(r"/\*.*?\*/", "", hdr, flags=re.S)
    names = set(re.findall(r"\b(fdc_[a-z_0-9]+)\s*\(", hdr))
    assert {"fdc_plan_graph", "fdc_frontier", "fdc_build_masks", "fdc_kv_append", "fdc_decode_attn"} <= names
    dll = ctypes.CDLL(lib.LIB_PATH)
    for n in sorted(names):
        assert hasattr(dll, n), f"{n} declared in fdc.h but not exported"


def test_struct_layouts(lib, tmp_path):
    """The ctypes mirrors have the layout a C compiler gives the header's structs."""
    import subprocess
    src = tmp_path / "sz.c"
    src.write_text('#include <stdio.h>\n#include <stddef.h>\n#include "fdc.h"\nint main(void){printf("%zu %zu %zu %zu %zu\\n",'
                   'sizeof(fdc_graph_desc),sizeof(fdc_kv_desc),sizeof(fdc_sizes),'
                   'offsetof(fdc_kv_desc,stride_scene),offsetof(fdc_sizes,state_bytes));return 0;}\n')
    exe = tmp_path / "sz"
    subprocess.check_call(["gcc", "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)])
    got = [int(x) for x in subprocess.check_output([str(exe)]).split()]
    assert got == [ctypes.sizeof(lib.fdc_graph_desc), ctypes.sizeof(lib.fdc_kv_desc), ctypes.sizeof(lib.fdc_sizes),
                   lib.fdc_kv_desc.stride_scene.offset, lib.fdc_sizes.state_bytes.offset]


def test_plan_rejects_bad_templates_on_host(lib):
    def code(*a):
        with pytest.raises(lib.FdcError) as e:
            lib.fdc_plan_graph(*a)
        return e.value.code
    assert code(3, [(0, 1), (1, 2), (2, 0)], [4, 4, 4], None, 8, 2) == lib.FDC_ERR_CYCLE
    assert code(2, [(1, 1)], [4, 4], None, 8, 2) == lib.FDC_ERR_CYCLE
    assert code(2, [(0, 5)], [4, 4], None, 8, 2) == lib.FDC_ERR_RANGE
    assert code(0, [], [], None, 8, 2) == lib.FDC_ERR_RANGE
    assert code(65, [], [1] * 65, None, 8, 2) == lib.FDC_ERR_RANGE
    assert code(2, [], [4, 0], None, 8, 2) == lib.FDC_ERR_RANGE
    assert code(2, [], [4, 4], [0, 4], 8, 2) == lib.FDC_ERR_RANGE
    assert code(2, [], [4, 4], None, -1, 2) == lib.FDC_ERR_RANGE
    assert code(2, [], [4, 4], None, 8, 0) == lib.FDC_ERR_RANGE
    assert "cycle" in lib.fdc_strerror(lib.FDC_ERR_CYCLE)
    assert lib.fdc_kernel_name(1) == "ref_cuda_core"
    assert lib.fdc_launch_count() >= 0


def test_cluster_size_that_a_device_cannot_place(tmp_path):
    """The cut of a launch is made for a whole B200; a device that cannot place clusters of that size gets the next
    smaller one it can, down to single blocks."""
    import subprocess
    src = tmp_path / "fit.cpp"
    src.write_text('#include "fdc_internal.h"\n#include <cstdio>\n#include <cstdlib>\n'
                   'int main(int, char** v) { const unsigned long fits = strtoul(v[2], nullptr, 0); int asked = 0;\n'
                   'const int n = fdc::largest_placeable(atoi(v[1]), [&](int k) { ++asked; return ((fits >> k) & 1) != 0; });\n'
                   'printf("%d %d\\n", n, asked); return 0; }\n')
    exe = tmp_path / "fit"
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2602_02864_b200", "csrc"),
                           "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)])

    def largest(nblk, sizes):
        return [int(x) for x in subprocess.check_output([str(exe), str(nblk), str(sum(1 << k for k in sizes))]).split()]
    assert largest(16, range(1, 17)) == [16, 1]               # a whole B200: what was asked for, one look
    assert largest(16, range(1, 13))[0] == 12
    assert largest(16, [1, 2, 4, 8])[0] == 8
    assert largest(6, [1, 2, 4, 8])[0] == 4
    assert largest(8, [])[0] == 1                             # (single blocks are not asked about)
    assert largest(1, [])[0] == 1


def test_runs_of_a_cluster_are_equal(tmp_path):
    """The blocks of a cluster share a pair's tile parts out evenly, whatever the parts hold, and leave none out."""
    import subprocess
    src = tmp_path / "runs.cpp"
    src.write_text('#include "fdc_internal.h"\n#include <cstdio>\n'
                   'int main() { for (int n = 1; n <= 16; ++n) for (int parts = 0; parts <= 2200; ++parts) {\n'
                   'const uint32_t inv = fdc::div_inverse(n); auto begin = [&](int r) { return fdc::run_begin(r, n, parts, [&](uint32_t x) { return fdc::div_by(x, inv); }); };\n'
                   'if (begin(0) != 0 || begin(n) != parts) { printf("ends %d %d\\n", n, parts); return 1; }\n'
                   'for (int r = 0; r < n; ++r) { const int k = begin(r + 1) - begin(r);\n'
                   'if (k < parts / n || k > (parts + n - 1) / n) { printf("run %d of %d: %d of %d\\n", r, n, k, parts); return 1; } } }\n'
                   'return 0; }\n')
    exe = tmp_path / "runs"
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2602_02864_b200", "csrc"),
                           "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
