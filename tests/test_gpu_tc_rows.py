"""The row form of the tcgen05 kernel (more than 64 query rows per (scene, KV head) pair) against the CPU checker:
widths around its row quadrants, segments of one and of a few tiles, prefixes that are and are not whole tiles (and
none), more pairs than thread blocks, both ways of appending."""
import pytest

from harness import run_and_compare
from paper_2602_02864_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [False, True], ids=["append_kernel", "append_inside_attention"])
@pytest.mark.parametrize("hq,hkv,fields,batch,prefix", [
    (5, 1, 13, 1, 0), (5, 1, 13, 2, 63), (28, 4, 10, 3, 1500), (28, 4, 18, 2, 64), (32, 8, 17, 2, 700), (32, 8, 24, 20, 1024), (4, 2, 64, 2, 129),
    (16, 1, 8, 160, 200), (32, 8, 32, 1, 4100)])
def test_row_form_shapes(hq, hkv, fields, batch, prefix, fused):
    w = wl.random_template(9100 + fields + batch, n_nodes=fields, edge_prob=0.06, cap_lo=2, cap_hi=70, batch=batch, prefix_len=prefix, fixed_hi=2,
                           hq=hq, hkv=hkv, head_dim=128, dtype="bf16")
    w.max_active = w.n_nodes
    assert 64 < w.max_active * (hq // hkv) <= 128
    r = run_and_compare(w, check_steps={0, 1, 9, 33}, kernel=3, max_steps=34, fused_append=fused)
    assert r["checked"] > 0
