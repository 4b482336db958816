"""The cluster kernels (bf16: fdc_set_attn_kernel 2, the automatic choice for head_dim 64 and for small passes;
fp32: the automatic choice) against the CPU checker at the sizes where its splits, rings and groups can go wrong."""
import pytest
import torch

from harness import run_and_compare
from paper_2602_02864_b200 import workloads as wl

pytestmark = pytest.mark.gpu


# query rows per pair (hq / hkv x fields) around the group sizes 16 / 32 / 64 / 128; blocks per pair 16, 8, a
# few, one; prefixes that are and are not whole tiles, empty, shorter than one stage; runs much longer
# than the ring (few blocks per pair and a long prefix: every stage is reused many times)
@pytest.mark.parametrize("head_dim,hq,hkv,fields,batch,prefix", [
    (64, 14, 2, 1, 1, 31), (64, 14, 2, 5, 1, 1531), (64, 4, 2, 8, 3, 640), (64, 14, 2, 9, 24, 2100), (64, 4, 2, 32, 40, 1000),
    (64, 16, 1, 8, 200, 1024), (64, 2, 2, 17, 2, 0),
    (128, 4, 4, 1, 1, 64), (128, 28, 4, 3, 1, 4095), (128, 32, 8, 4, 6, 3000), (128, 32, 8, 9, 19, 2048), (128, 8, 2, 32, 5, 1025),
    (128, 16, 8, 8, 20, 4000), (128, 8, 8, 20, 2, 97)])
def test_cluster_kernel_shapes(head_dim, hq, hkv, fields, batch, prefix):
    w = wl.random_template(7100 + fields + batch, n_nodes=fields, edge_prob=0.15, cap_lo=2, cap_hi=70, batch=batch, prefix_len=prefix, fixed_hi=2,
                           hq=hq, hkv=hkv, head_dim=head_dim, dtype="bf16")
    w.max_active = w.n_nodes
    steps = {0, 1, 9, 33}
    r = run_and_compare(w, check_steps=steps, kernel=2, max_steps=34)
    assert r["checked"] > 0


# fp32: query rows per pair around what a lane's tile holds (8 / 16 / 24 / 32 rows) and wider pairs, which are cut
# over several clusters; one block per pair (many pairs) up to eight
@pytest.mark.parametrize("head_dim,hq,hkv,fields,batch,prefix", [
    (64, 4, 2, 1, 1, 33), (64, 14, 2, 2, 3, 200), (64, 4, 2, 9, 30, 1000), (64, 16, 8, 16, 2, 700), (64, 2, 2, 33, 1, 0),
    (128, 32, 8, 2, 1, 2048), (128, 28, 4, 3, 2, 1531), (128, 32, 8, 6, 12, 600), (128, 32, 8, 9, 2, 129), (128, 8, 2, 32, 3, 500)])
def test_fp32_cluster_kernel_shapes(head_dim, hq, hkv, fields, batch, prefix):
    w = wl.random_template(8100 + fields + batch, n_nodes=fields, edge_prob=0.15, cap_lo=2, cap_hi=70, batch=batch, prefix_len=prefix, fixed_hi=2,
                           hq=hq, hkv=hkv, head_dim=head_dim, dtype="f32")
    w.max_active = w.n_nodes
    r = run_and_compare(w, check_steps={0, 1, 9, 33}, max_steps=34)
    assert r["checked"] > 0


# fp32: what a field's rows hold is nobody's business but the fields' that see them.  Infinities and NaN in one field's K and V
# rows (new ones and earlier ones, a tile shared with its neighbours among them) leave the other fields' results as they are, bit
# for bit.  Query rows per pair for all tile heights of the kernel (8 / 16 / 24 / 32 rows, more than one cluster).
@pytest.mark.parametrize("head_dim,hq,hkv,fields,batch,prefix", [
    (64, 4, 2, 3, 2, 70), (64, 16, 2, 3, 1, 600), (128, 16, 4, 4, 1, 33), (128, 28, 4, 3, 2, 200), (128, 32, 8, 8, 9, 129), (64, 8, 2, 16, 1, 0)])
def test_fp32_siblings_are_independent(head_dim, hq, hkv, fields, batch, prefix):
    from paper_2602_02864_b200 import fdc
    passes, bad = 5, 1
    cap = [9 + 5 * (v % 4) for v in range(fields)]
    sess = fdc.DecodeSession(fields, [], cap, None, prefix, fields, batch)
    g = torch.Generator(device="cuda").manual_seed(11)
    shape = (batch, 1, hkv, prefix + sum(cap), head_dim)
    k, v = (torch.randn(shape, generator=g, device="cuda") for _ in range(2))
    q = torch.randn(batch, fields, hq, head_dim, generator=g, device="cuda")
    sess.bind_cache(k, v, hq)
    sess.init(None)
    for _ in range(passes):
        sess.frontier()
    sess.build_masks()
    r0 = prefix + sum(cap[:bad])

    def attend(rows):
        k[:, :, :, r0:r0 + passes], v[:, :, :, r0:r0 + passes] = rows
        out = torch.zeros_like(q)
        sess.decode_attn(0, q, out, head_dim ** -0.5)
        return out

    clean = attend((k[:, :, :, r0:r0 + passes].clone(), v[:, :, :, r0:r0 + passes].clone()))
    assert torch.isfinite(clean).all()
    others = [b for b in range(fields) if b != bad]
    for kx, vx in ((0.5, float("inf")), (float("nan"), float("nan")), (float("inf"), -float("inf")), (float("nan"), 1.0)):
        out = attend((torch.full((), kx, device="cuda"), torch.full((), vx, device="cuda")))
        assert not torch.isfinite(out[:, bad]).all()
        assert torch.equal(out[:, others], clean[:, others])
    assert sess.status() == 0
    sess.close()


# The same kernel with several layers a pass (launches after the first read ahead of the dependency wait), whole schedules (the
# cache is compared bit for bit at the end) and both ways of appending: few fields and query rows cut over several clusters;
# more than 32 fields (two stages of new rows), cut and uncut; more parts beyond the prefix in one block than have their
# visibility in shared memory (32 fields: 32 parts; 50: 20); a field's rows past the table that new rows are taken out of.
@pytest.mark.parametrize("fused", [False, True], ids=["append_kernel", "append_inside_attention"])
@pytest.mark.parametrize("head_dim,hq,hkv,fields,cap_hi,batch,prefix", [
    (64, 14, 2, 6, 40, 2, 700), (64, 2, 2, 40, 12, 1, 200), (64, 8, 8, 32, 60, 20, 100), (128, 28, 4, 6, 40, 1, 2048), (128, 4, 2, 50, 24, 2, 300),
    (128, 8, 8, 50, 40, 12, 20)])
def test_cluster_kernel_whole_schedules(head_dim, hq, hkv, fields, cap_hi, batch, prefix, fused):
    w = wl.random_template(7300 + fields + batch, n_nodes=fields, edge_prob=0.01, cap_lo=2, cap_hi=cap_hi, batch=batch, prefix_len=prefix, fixed_hi=2,
                           hq=hq, hkv=hkv, head_dim=head_dim, dtype="bf16")
    w.max_active, w.layers = w.n_nodes, 2
    r = run_and_compare(w, check_steps={0, 1, 2, 11, 23, 38}, kernel=2, fused_append=fused)
    assert r["checked"] > 0


# fp32 with several layers a pass, whole schedules
@pytest.mark.parametrize("head_dim,hq,hkv,fields,batch,prefix", [(64, 14, 2, 3, 2, 300), (128, 32, 8, 8, 2, 129), (128, 8, 2, 20, 1, 1000)])
def test_fp32_cluster_kernel_whole_schedules(head_dim, hq, hkv, fields, batch, prefix):
    w = wl.random_template(8300 + fields + batch, n_nodes=fields, edge_prob=0.1, cap_lo=2, cap_hi=30, batch=batch, prefix_len=prefix, fixed_hi=2,
                           hq=hq, hkv=hkv, head_dim=head_dim, dtype="f32")
    w.max_active, w.layers = w.n_nodes, 3
    r = run_and_compare(w, check_steps={0, 1, 2, 11, 23, 38})
    assert r["checked"] > 0


# fp32, one query row a field, fields that end one after the other while the prefix is long enough for stages without a mask: every number of
# rows at work from the widest down to one, half tiles and whole ones (24 rows: up to 12 / more), one group of warps and two
# (32 rows: up to 16 / more), and clusters of a pair that run out of rows (48, 56: several clusters of 24, 32)
@pytest.mark.parametrize("head_dim,fields,batch,hkv,prefix", [
    (64, 24, 1, 2, 700), (64, 24, 30, 4, 130), (64, 32, 2, 2, 400), (64, 48, 1, 2, 520), (64, 56, 2, 1, 300), (128, 24, 1, 2, 700), (128, 24, 24, 4, 130),
    (128, 20, 3, 1, 1500), (128, 32, 2, 2, 400), (128, 48, 1, 2, 520), (128, 64, 1, 1, 260)])
def test_fp32_every_number_of_rows(head_dim, fields, batch, hkv, prefix):
    w = wl.random_template(8500 + fields + batch, n_nodes=fields, edge_prob=0.0, cap_lo=fields + 1, cap_hi=fields + 1, batch=batch, prefix_len=prefix, fixed_hi=0,
                           hq=hkv, hkv=hkv, head_dim=head_dim, dtype="f32")
    w.max_active, w.lens = fields, w.lens.copy()
    w.lens[:] = [1 + (v * 7) % fields if fields % 7 else 1 + (v * 5) % fields for v in range(fields)]
    r = run_and_compare(w)
    assert r["steps"] == fields and r["checked"] > 0


# Sequential decoding of one or two query rows a pair over a long prefix: clusters of 16 blocks, of which 8 or 12 own no part of the result (4 or 8
# chunks of 16 columns); several layers a pass, append apart and inside
@pytest.mark.parametrize("fused", [False, True], ids=["append_kernel", "append_inside_attention"])
@pytest.mark.parametrize("head_dim,hq,hkv,prefix", [(64, 2, 2, 2000), (64, 4, 2, 2000), (128, 4, 4, 2000)])
def test_blocks_that_own_no_part_of_the_result(head_dim, hq, hkv, prefix, fused):
    w = wl.random_template(9100 + hq, n_nodes=3, edge_prob=1.0, cap_lo=4, cap_hi=8, batch=1, prefix_len=prefix, fixed_hi=1, hq=hq, hkv=hkv, head_dim=head_dim, dtype="bf16")
    w.max_active, w.layers = 1, 3
    r = run_and_compare(w, kernel=2, fused_append=fused)
    assert r["checked"] > 0


# head_dim 64 and fp32 serve a tile list in any order (head_dim 128 in bf16 reports one that does not begin with the prefix): a prefix tile and one beyond
# the prefix change places, and first and last.  Several layers, so that the later ones read the list ahead of the dependency wait.
@pytest.mark.parametrize("dtype,head_dim,hq,hkv,prefix", [("bf16", 64, 14, 2, 1000), ("f32", 64, 4, 2, 1000), ("f32", 128, 8, 2, 1000)])
def test_lists_in_any_order(dtype, head_dim, hq, hkv, prefix):
    from paper_2602_02864_b200 import fdc
    fields, batch, layers, passes, slot = 3, 2, 3, 30, 40
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    sess = fdc.DecodeSession(fields, [], [slot] * fields, None, prefix, fields, batch)
    g = torch.Generator(device="cuda").manual_seed(12)
    k, v = (torch.randn(batch, layers, hkv, prefix + slot * fields, head_dim, generator=g, device="cuda").to(dt) for _ in range(2))
    q = torch.randn(layers, batch, fields, hq, head_dim, generator=g, device="cuda").to(dt)
    sess.bind_cache(k, v, hq)
    sess.init(None)
    for _ in range(passes):
        sess.frontier()
    npre = prefix // 64
    outs = []
    for swap in ([], [(3, npre)], [(0, npre + 1), (npre - 1, npre)]):
        sess.build_masks()
        assert int(sess.ntiles.min()) >= npre + 2
        for i, j in swap:
            sess.tiles[:, [i, j]] = sess.tiles[:, [j, i]]
        out = torch.zeros_like(q)
        for l in range(layers):
            sess.decode_attn(l, q[l], out[l], head_dim ** -0.5)
        outs.append(out.double())
    assert sess.status() == 0
    # (another order of the same sums: fp32 rounding, and weights and outputs rounded to bf16, 2^-9 each, against other maxima)
    tol = 2e-6 if dtype == "f32" else 2 ** -7
    for o in outs[1:]:
        assert (o - outs[0]).norm() <= tol * outs[0].norm()
    sess.close()


# Every cut that the library takes can be launched: one kernel a call (a call that fell back would launch two).  Clusters with 80 and
# 112 query rows and two blocks per SM find no room for the partials (that none is taken at any shape: test_routes.py); the output of the first and
# the last scene against the checker.
@pytest.mark.parametrize("hq,hkv,fields,batch,prefix", [(20, 4, 16, 32, 1024), (28, 4, 16, 24, 2048), (128, 8, 8, 3, 512), (28, 4, 15, 35, 6166), (32, 8, 18, 38, 3980)])
def test_the_cut_leaves_room_for_the_partials(hq, hkv, fields, batch, prefix):
    from harness import check_close, f32
    from oracle import attention
    from paper_2602_02864_b200 import fdc
    sess = fdc.DecodeSession(fields, [], [16] * fields, None, prefix, fields, batch)
    k, v = (torch.randn(batch, 1, hkv, prefix + 16 * fields, 128, device="cuda").mul_(0.5).to(torch.bfloat16) for _ in range(2))
    q = torch.randn(batch, fields, hq, 128, device="cuda", dtype=torch.bfloat16)
    sess.bind_cache(k, v, hq)
    fdc.fdc_set_attn_kernel(sess.plan, 2)
    sess.init(None)
    sess.frontier()
    sess.build_masks()
    before, out = fdc.fdc_launch_count(), torch.empty_like(q)
    sess.decode_attn(0, q, out, 128 ** -0.5)
    assert fdc.fdc_launch_count() == before + 1 and sess.status() == 0
    for s in (0, batch - 1):
        vis = torch.ones(fields, prefix + 16 * fields, dtype=torch.bool)
        vis[:, prefix:] = torch.eye(fields, dtype=torch.bool).repeat_interleave(16, 1) & (torch.arange(16 * fields) % 16 == 0)      # its own first row
        check_close(f32(out[s]), attention.attention(f32(q[s]), f32(k[s, 0]), f32(v[s, 0]), vis.numpy(), 128 ** -0.5), "bf16", f"scene {s}")
    sess.close()
