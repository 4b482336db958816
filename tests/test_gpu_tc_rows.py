"""The row form of the tcgen05 kernel (more than 64 query rows per (scene, KV head) pair) against the CPU checker:
widths around its row quadrants, segments of one and of a few tiles, prefixes that are and are not whole tiles (and
none), more pairs than thread blocks, both ways of appending."""
import pytest
import torch

from harness import check_close, f32, run_and_compare
from oracle import attention as oatt
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


@pytest.mark.parametrize("tiles_per_block,equal_shares", [(70, False), (112, True)])
def test_row_form_split_of_long_prefixes(tiles_per_block, equal_shares):
    """64 pairs on 148 blocks: one part per block leaves 20 blocks idle; from 100 prefix tiles per block every block gets an
    equal share (seen in the scratch: block c's partial of pair i lies in slot c + i).  A sampled scene's and KV head's
    output against the CPU checker."""
    from paper_2602_02864_b200 import fdc
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pairs, fields, batch, hkv, D = 64, 32, 8, 8, 128
    prefix = tiles_per_block * sms // pairs * 64
    sess = fdc.DecodeSession(fields, [], [64] * fields, None, prefix, fields, batch)
    fdc.fdc_set_attn_kernel(sess.plan, 3)
    g = torch.Generator(device="cuda").manual_seed(3)
    k, v = (torch.empty(batch, 1, hkv, prefix + 64 * fields, D, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.5, generator=g) for _ in range(2))
    q = torch.empty(batch, fields, 4 * hkv, D, dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    out = torch.zeros_like(q)
    sess.bind_cache(k, v, 4 * hkv)
    sess.init(None)
    sess.frontier()
    sess.build_masks()
    sess.workspace.view(torch.float32).fill_(float("nan"))
    sess.decode_attn(0, q, out, D ** -0.5)
    assert sess.status() == 0
    slots = 2 * sms + pairs
    partials = sess.workspace.view(torch.float32)[:slots * 128 * D].view(slots, 128 * D)
    written = int((~partials.isnan()).any(dim=1).nonzero().max())
    last = sms // pairs * pairs - 1 + pairs - 1            # last block of the one-part split, last pair
    assert written > last if equal_shares else written <= last
    sess.close()
    s, h = 5, 3
    vis = torch.zeros(fields, prefix + 64 * fields, dtype=torch.bool)
    vis[:, :prefix] = True
    vis[torch.arange(fields), prefix + 64 * torch.arange(fields)] = True
    ref = oatt.attention(f32(q[s, :, 4 * h:4 * h + 4]), f32(k[s, 0, h:h + 1]), f32(v[s, 0, h:h + 1]), vis.numpy(), D ** -0.5)
    check_close(f32(out[s, :, 4 * h:4 * h + 4]), ref, "bf16")


@pytest.mark.parametrize("hq,hkv,fields,batch,prefix", [(28, 4, 10, 3, 500), (32, 8, 20, 20, 129), (4, 2, 50, 1, 64)])
def test_row_form_whole_schedules(hq, hkv, fields, batch, prefix):
    """Several layers a pass (launches after the first read ahead of the dependency wait) with the append inside; the
    cache is compared bit for bit at the end."""
    w = wl.random_template(9400 + fields + batch, n_nodes=fields, edge_prob=0.02, cap_lo=2, cap_hi=30, batch=batch, prefix_len=prefix, fixed_hi=2,
                           hq=hq, hkv=hkv, head_dim=128, dtype="bf16")
    w.max_active, w.layers = w.n_nodes, 3
    assert 64 < w.max_active * (hq // hkv) <= 128
    r = run_and_compare(w, check_steps={0, 1, 2, 11, 23}, kernel=3, fused_append=True)
    assert r["checked"] > 0
