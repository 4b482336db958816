"""Caches expanded over scenes or KV heads (a stride of 0): no tensor map describes them, so every choice of kernel has
to end at the one that follows the strides itself.  And that kernel (CUDA cores) in fp32, which is otherwise reached by
nothing else."""
import pytest
import torch

from harness import check_close, f32, run_and_compare
from oracle import attention as oatt
from oracle import schedule as sch
from paper_2602_02864_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [0, 1, 2, 3])
@pytest.mark.parametrize("over", ["scenes", "heads", "both"])
@pytest.mark.parametrize("dtype,head_dim,hq,hkv", [("f32", 64, 4, 2), ("f32", 128, 8, 4), ("bf16", 64, 4, 2), ("bf16", 128, 8, 4), ("bf16", 128, 80, 4)])
def test_expanded_cache(dtype, head_dim, hq, hkv, over, kernel):
    from paper_2602_02864_b200 import fdc
    w = wl.random_template(9300 + hkv, n_nodes=5, edge_prob=0.0, cap_lo=3, cap_hi=20, batch=3, prefix_len=150, hq=hq, hkv=hkv, head_dim=head_dim, dtype=dtype)
    sess = fdc.DecodeSession(w.n_nodes, w.edges, w.slot_cap, w.n_fixed, w.prefix_len, w.max_active, w.batch)
    fdc.fdc_set_attn_kernel(sess.plan, kernel)
    shape = (w.batch if over == "heads" else 1, 1, hkv if over == "scenes" else 1, w.rows, head_dim)
    g = torch.Generator(device="cuda").manual_seed(5)
    k, v = (torch.randn(shape, generator=g, device="cuda").to(w.torch_dtype).expand(w.batch, 1, hkv, w.rows, head_dim) for _ in range(2))
    q = torch.randn(w.batch, w.max_active, hq, head_dim, generator=g, device="cuda").to(w.torch_dtype)
    out = torch.full_like(q, 7.0)
    sess.bind_cache(k, v, hq)
    assert sess.kv.stride_scene == 0 or sess.kv.stride_head == 0
    sess.init(torch.from_numpy(w.lens).cuda())
    sess.frontier()
    sess.build_masks()
    sess.decode_attn(0, q, out, w.softmax_scale)
    assert sess.status() == 0
    sess.close()
    for s in range(w.batch):
        lens = w.lens[s].tolist()
        first = sch.simulate(w.n_nodes, w.edges, lens, w.n_fixed)[0]
        tab = sch.pass_tables(w.n_nodes, w.edges, w.slot_cap, lens, w.n_fixed, w.prefix_len, first)
        A = len(first)
        ref = oatt.attention(f32(q[s, :A]), f32(k[s, 0]), f32(v[s, 0]), tab["vis"], w.softmax_scale)
        check_close(f32(out[s, :A]), ref, dtype, f"scene {s}")


@pytest.mark.parametrize("head_dim", [64, 128])
def test_fp32_on_cuda_cores(head_dim):
    w = wl.cfg0_tiny()
    w.head_dim = head_dim
    r = run_and_compare(w, kernel=1)
    assert r["steps"] == 48 and r["checked"] == 96 * 4
