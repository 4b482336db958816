"""Host-only checks of the choice of kernel and cut, at shapes where the other choice was timed and lost."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """#include "fdc_internal.h"
#include <cstdio>
int main() {
    fdc::ClusterProblem c; long long pairs; fdc::ClusterShape h;
    while (scanf("%lld %d %d %d %d", &pairs, &c.mmax, &c.head_dim, &c.P, &c.T) == 5) {
        c.pairs = pairs; c.sm_count = 148;
        const int k = fdc::route_problem(c, &h);
        const int groups = ((c.mmax + 15) / 16 + h.qsplit - 1) / h.qsplit;
        printf("%d %d %d %d %d\\n", k, h.nblk, h.qsplit, h.per_sm, fdc::cluster_ring(c.head_dim, groups * 16, h.nblk, h.per_sm));
    }
}
"""


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    """shapes (pairs, query rows, head_dim, prefix, template rows) -> (cluster kernel, blocks, clusters a pair, blocks per SM, ring)"""
    from paper_2602_02864_b200 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("routes")
    (d / "routes.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2602_02864_b200", "csrc"),
                           "-I", "/usr/local/cuda/include", str(d / "routes.cpp"), "-o", str(d / "routes"), lib, "-Wl,-rpath," + os.path.dirname(lib)])

    def ask(shapes):
        out = subprocess.run([str(d / "routes")], input="\n".join(" ".join(str(x) for x in s) for s in shapes), capture_output=True, text=True, check=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return ask


# us a layer: the choice / the other
@pytest.mark.parametrize("shape,cluster", [
    ((4, 7, 128, 1024, 512), True),           # 6.1 / 13.8
    ((4, 42, 128, 2048, 512), True),          # 9.8 / 17.7
    ((8, 7, 128, 5409, 810), True),           # 13.9 / 19.9
    ((192, 36, 128, 2168, 630), False),       # 67 / 102
    ((200, 48, 128, 1644, 360), False),       # 59 / 80
    ((64, 128, 128, 1024, 2048), False)])     # 34 / 57
def test_kernel(route, shape, cluster):
    assert bool(route([shape])[0][0]) == cluster


@pytest.mark.parametrize("shape,cut", [
    ((4, 7, 128, 1024, 512), (16, 1, 2)),     # 6.1 us a layer; (16, 1, 1) 7.2
    ((96, 35, 64, 1892, 168), (1, 3, 2)),     # 19.7; (1, 2, 2) 28.2
    ((94, 35, 64, 14115, 539), (2, 1, 2)),    # 58.5; (1, 2, 2) 78.5
    ((32, 42, 64, 4096, 768), (2, 3, 2))])    # 18.3; (6, 1, 2) 21.4
def test_cut(route, shape, cut):
    assert route([shape])[0][1:4] == cut


def test_long_runs_have_the_deeper_ring(route):
    assert route([(56, 12, 128, 4737, 108)])[0][3] == 1          # (3, 1, 1) 25.0 us a layer, (3, 1, 2) 33.3


def test_every_cut_has_room_for_the_partials(route):
    """No cut is taken whose blocks find no room for what the others send them beside their own partials (the launch would fall back to
    the CUDA-core kernel): clusters with more than 48 rows and two blocks per SM, head_dim 128."""
    shapes = [(pairs, rows, d, p, 512) for d in (64, 128) for pairs in (1, 2, 4, 12, 24, 32, 48, 64, 96, 128, 140, 152, 200, 300)
              for rows in (1, 16, 17, 32, 48, 49, 64, 72, 80, 96, 105, 112, 128) for p in (0, 256, 1024, 2048, 4096, 6166, 16384, 32768)]
    got = route(shapes)
    assert len(got) == len(shapes)
    assert all(g[4] > 0 for g in got)
    assert any(g[1] > 1 and g[3] == 2 for g in got) and any(g[1] > 1 and g[3] == 1 for g in got)


TWO_PARTS = """#include "fdc_internal.h"
#include <cstdio>
int main() {
    long long pairs; int mmax, P, nt;
    while (scanf("%lld %d %d %d", &pairs, &mmax, &P, &nt) == 4) printf("%d\\n", fdc::pairs_in_two_parts(pairs, mmax, P, nt, 148));
}
"""


@pytest.fixture(scope="module")
def two_parts(tmp_path_factory):
    """shapes (pairs, query rows, prefix, tiles a pair at most) -> the launch goes to the builds for pairs in two parts (148 CTAs)"""
    from paper_2602_02864_b200 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("two")
    (d / "two.cpp").write_text(TWO_PARTS)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2602_02864_b200", "csrc"),
                           "-I", "/usr/local/cuda/include", str(d / "two.cpp"), "-o", str(d / "two"), lib, "-Wl,-rpath," + os.path.dirname(lib)])

    def ask(shapes):
        out = subprocess.run([str(d / "two")], input="\n".join(" ".join(str(x) for x in s) for s in shapes), capture_output=True, text=True, check=True).stdout
        return [x == "1" for x in out.split()]
    return ask


def split_of_whole_lists(scenes, hkv, mmax, P, nt, n_cta=148):
    """Parts of a pair when every scene lists `nt` tiles, as the tcgen05 kernels cut them (0: equal shares)."""
    prefix = min(P // 64, nt)
    length = 4 * prefix + 6 * (nt - prefix)
    part = next(t for t in range(min(length, 32), length + 1) if scenes * -(-length // t) <= n_cta // hkv)
    avg = scenes * hkv * (length + 32) // n_cta
    return 0 if avg * (2 if mmax > 64 else 1) >= 800 and part * 100 > avg * 108 else -(-length // part)


# us a layer, plain build / build for pairs in two parts
@pytest.mark.parametrize("shape,two", [
    ((64, 128, 1024, 48), True),              # 38.6 / 34.0
    ((72, 128, 5632, 120), True),             # 69.3 / 65.0: 128 rows
    ((74, 128, 24576, 416), False),           # 100 tiles per CTA and more: the whole template 1.00 to 1.01
    ((64, 64, 1024, 32), True),               # 32.6 / 27.1
    ((64, 36, 2048, 41), False),              # 25.6 / 26.7
    ((68, 63, 2048, 41), False),              # 9 fields x 7 heads, fan, the whole template 0.957
    ((64, 64, 8192, 142), False),             # 16 fields x 4 heads, wide, 55.1 / 55.9 in its later passes, the whole template 0.999
    ((72, 91, 2048, 47), False),              # 13 fields x 7 heads, wide, the whole template 0.974
    ((64, 128, 176 * 64, 208), False),        # 93.4 / 95.9: equal shares
    ((64, 128, 80 * 64, 176), False),         # 99.2 / 103.5: equal shares
    ((64, 128, 135 * 64, 231), False)])       # 117.3 / 128.1: equal shares
def test_pairs_in_two_parts(two_parts, shape, two):
    assert two_parts([shape])[0] == two


def test_pairs_in_two_parts_are_cut_in_two(two_parts):
    shapes = [(scenes, hkv, mmax, P, P // 64 + beyond) for hkv in (1, 2, 4, 5, 8) for scenes in range(-(-50 // hkv), 74 // hkv + 1) for mmax in (36, 64, 72, 128)
              for P in (0, 500, 1024, 2048, 5120, 8192, 13312, 20480, 28672) for beyond in (3, 16, 32, 48, 96)]
    got = two_parts([(s * h, m, P, nt) for s, h, m, P, nt in shapes])
    assert any(got) and not all(got)
    assert all(split_of_whole_lists(*x) == 2 for x, g in zip(shapes, got) if g)
