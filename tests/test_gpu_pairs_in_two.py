"""Launches whose pairs come in two parts each (50 to 74 (scene, KV head) pairs, more than 32 query rows, 32 tiles a pair and more): parts
that are spread over the pair's tile list and hand each other half of their results.  Against the CPU checker at the edges: the fewest and the most pairs, an odd
number of KV heads (pairs that do not begin at an even block merge as ever), few and many tiles beyond the prefix, scenes that end before the others (pairs in more
parts), both kernels, both ways of appending."""
import pytest

from harness import run_and_compare
from paper_2602_02864_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [False, True], ids=["append_kernel", "append_inside_attention"])
@pytest.mark.parametrize("hq,hkv,fields,batch,prefix,cap_lo,cap_hi", [
    (32, 8, 9, 8, 2048, 3, 30),          # 64 pairs, 36 rows, hardly a tile beyond the prefix
    (32, 8, 16, 7, 1500, 40, 70),        # 56 pairs, 64 rows, a prefix that is no whole number of tiles
    (32, 8, 32, 8, 1024, 20, 70),        # 64 pairs, 128 rows, spread parts
    (28, 4, 18, 18, 1337, 30, 60),       # 72 pairs, 126 rows
    (15, 5, 24, 13, 1100, 30, 70),       # 65 pairs, 72 rows; an odd number of KV heads
    (4, 2, 64, 37, 2050, 2, 12)])        # 74 pairs, 128 rows
def test_two_parts(hq, hkv, fields, batch, prefix, cap_lo, cap_hi, fused):
    w = wl.random_template(7700 + fields + batch, n_nodes=fields, edge_prob=0.03, cap_lo=cap_lo, cap_hi=cap_hi, batch=batch, prefix_len=prefix, fixed_hi=2,
                           hq=hq, hkv=hkv, head_dim=128, dtype="bf16")
    w.max_active, w.layers = w.n_nodes, 2
    assert 32 < w.max_active * (hq // hkv) <= 128 and 50 <= batch * hkv <= 74
    r = run_and_compare(w, check_steps={0, 1, 14}, kernel=3, max_steps=15, fused_append=fused)
    assert r["checked"] > 0
