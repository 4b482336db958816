"""Launches whose pairs come in two parts each (50 to 74 (scene, KV head) pairs, more than 32 query rows, 32 tiles a pair and more, of which
those beyond the prefix weigh at least half, or 120 query rows and more): parts that are spread over the pair's tile list and hand each other half of
their results.  Against the CPU checker at the edges: the fewest and the most pairs, 65 to 128 and up to 64 query rows at work, whole and
broken row quadrants, prefixes that are and are not whole tiles, pairs cut in one or three parts because the scenes' lengths have parted, pairs that do not
begin at an even block (an odd number of KV heads behind one), parts too short to be spread, scenes that have ended, both ways of appending."""
import pytest
import torch

from harness import make_oracle, run_and_compare
from paper_2602_02864_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def workload(hq, hkv, fields, batch, prefix, cap_lo, cap_hi):
    """Independent fields: all of them are at work in the first pass."""
    w = wl.random_template(7700 + fields + batch, n_nodes=fields, edge_prob=0.0, cap_lo=cap_lo, cap_hi=cap_hi, batch=batch, prefix_len=prefix, fixed_hi=2,
                           hq=hq, hkv=hkv, head_dim=128, dtype="bf16")
    w.max_active, w.layers = w.n_nodes, 2
    assert 32 < w.max_active * (hq // hkv) <= 128 and 50 <= batch * hkv <= 74
    return w


def parts_of_scenes(w, oracle, step, n_cta):
    """Parts of a pair in every scene, as the tcgen05 kernels cut them with one part per block, and the tiles that it lists."""
    tiles = [len(oracle.tables(s, step)["tiles"]) if oracle.active(s, step) else 0 for s in range(w.batch)]
    length = [4 * min(w.prefix_len // 64, t) + 6 * max(0, t - w.prefix_len // 64) for t in tiles]
    part = next(t for t in range(min(max(length), 32), max(length) + 1) if sum(-(-x // t) for x in length) <= n_cta // w.hkv)
    return [-(-x // part) for x in length], tiles


# what the checked passes hold: the most query rows at work, and which of the cases of `seen` below
@pytest.mark.parametrize("fused", [False, True], ids=["append_kernel", "append_inside_attention"])
@pytest.mark.parametrize("hq,hkv,fields,batch,prefix,cap_lo,cap_hi,steps,rows,holds", [
    (32, 8, 32, 8, 1024, 64, 64, (0, 1, 14), 128, {"two", "three"}),                                  # 64 pairs
    (28, 4, 18, 18, 1337, 40, 70, (0, 5, 20), 126, {"two"}),                                         # 72 pairs, a broken tile and quadrant
    (28, 7, 30, 8, 900, 20, 80, (0, 5, 20), 120, {"two", "three", "odd"}),                            # 56 pairs
    (4, 2, 64, 37, 500, 20, 40, (0, 5, 30, 35), 128, {"two", "one", "three", "ended"}),               # 74 pairs; bitmaps too long for shared memory
    (15, 5, 24, 13, 1100, 30, 70, (0, 14, 50), 72, {"two", "three", "odd", "ended"}),                 # 65 pairs
    (32, 8, 16, 7, 1030, 64, 80, (0, 1, 14), 64, {"two", "three"}),                                   # up to 64 rows
    (64, 4, 4, 13, 128, 500, 520, (1, 5, 14), 64, {"two", "one", "short"})])                          # 52 pairs, few tiles yet
def test_two_parts(hq, hkv, fields, batch, prefix, cap_lo, cap_hi, steps, rows, holds, fused):
    w = workload(hq, hkv, fields, batch, prefix, cap_lo, cap_hi)
    n_cta, oracle, seen, widest = torch.cuda.get_device_properties(0).multi_processor_count, make_oracle(w), set(), 0
    for step in steps:
        parts, tiles = parts_of_scenes(w, oracle, step, n_cta)
        first = 0                                          # block that a pair begins at
        for s, k in enumerate(parts):
            seen.add({0: "ended", 1: "one", 2: "two", 3: "three"}.get(k, "more"))
            if k == 2 and (hkv * first) % 2:
                seen.add("odd")
            if k == 2 and tiles[s] - prefix // 64 < 8:
                seen.add("short")
            first += k
            widest = max(widest, len(oracle.active(s, step)) * (hq // hkv))
    assert widest == rows and seen - {"more"} >= holds, (widest, seen)
    r = run_and_compare(w, check_steps=set(steps), kernel=3, max_steps=max(steps) + 1, fused_append=fused)
    assert r["checked"] > 0


# The scratch tells the builds apart: a block that hands over half of its part writes half of its slot, one whose partial is merged by the block that
# comes last writes all of it.  The choice of kernel is the library's.
@pytest.mark.parametrize("hq,hkv,fields,batch,prefix,slot,two", [
    (32, 8, 32, 8, 1024, 64, True), (28, 4, 18, 18, 1337, 64, True), (4, 2, 64, 37, 500, 30, True), (32, 8, 32, 8, 4096, 64, True), (32, 8, 16, 7, 1024, 72, True),
    (32, 8, 16, 8, 8192, 48, False), (28, 4, 13, 18, 2048, 64, False), (32, 8, 9, 8, 2048, 64, False)])
def test_the_build_that_runs(hq, hkv, fields, batch, prefix, slot, two):
    from paper_2602_02864_b200 import fdc
    D, rows, pairs = 128, fields * (hq // hkv), batch * hkv
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sess = fdc.DecodeSession(fields, [], [slot] * fields, None, prefix, fields, batch)
    k, v = (torch.zeros(batch, 1, hkv, prefix + slot * fields, D, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    q = torch.ones(batch, fields, hq, D, dtype=torch.bfloat16, device="cuda")
    out = torch.zeros_like(q)
    sess.bind_cache(k, v, hq)
    sess.init(None)
    sess.frontier()
    sess.build_masks()
    sess.workspace.view(torch.float32).fill_(float("nan"))
    sess.decode_attn(0, q, out, D ** -0.5)
    assert sess.status() == 0
    slots = 2 * sms + pairs
    written = (~sess.workspace.view(torch.float32)[:slots * rows * D].view(slots, rows * D).isnan()).sum(dim=1)
    written = written[written > 0]
    sess.close()
    assert len(written) == 2 * pairs
    # (up to 64 rows the halves are of 32 rows each, with fewer rows not quite halves)
    assert bool((written < rows * D).all()) == two and bool((written == rows * D).all()) != two
    assert not two or int(written.sum()) == pairs * rows * D
