"""The work that programs have this library do, as cases that can be timed and compared.

A case is one forward pass of parallel chain-of-thought decoding through the public binding:
Algorithm 1's step (frontier), Eq. 1's bitmaps (build_masks), then per layer the KV append and the
masked attention of all ready fields of every scene.  The pass is somewhere inside the template's
schedule: `pass_no` earlier passes have been played, and every call resumes from that point (the
scheduler state is plain caller-owned memory and is copied back first).  With submit = "loop" the
case is the whole template instead: pre-filled field-name rows, then every pass until no field is
ready, as one CUDA graph launch.

    listed()         the listed cases
    draw(rng)        one more case of the same ranges
    prepare(case, s) the program's state before the call (cache, inputs, session, graph)
    run(state)       one call; returns everything it computed
    work(case)       bytes and operations the call cannot do without
    tolerance(case)  how far two correct implementations may differ
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2602_02864_b200 import fdc
from paper_2602_02864_b200.device_loop import DeviceLoop

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(name, template, fields, slot, len_lo, fixed, prefix, scenes, layers, hq, hkv, head_dim, dtype, submit, fused,
          pass_no, kv_scale=0.5, q_scale=1.0):
    """template  fan: `fields` independent fields -> summary -> final; wide: `fields` leaves -> two summaries of a
                 random half each -> final; diamond: a root -> `fields` children -> summary; free: `fields`
                 independent fields; chain: the same one after the other (ordinary autoregressive decoding)
    slot, len_lo rows reserved per field; a field is len_lo..slot rows long (len_lo 0: no lengths given, it runs to its slot)
    fixed        up to this many pre-filled field-name rows at the head of a slot
    submit       eager: every call issued by the host; graph: the pass replayed as one CUDA graph; loop: the whole template
    fused        the append is carried out by the attention kernel (an option, off by default)"""
    return {"name": name, "template": template, "fields": fields, "slot": slot, "len_lo": len_lo, "fixed": fixed, "prefix": prefix,
            "scenes": scenes, "layers": layers, "hq": hq, "hkv": hkv, "head_dim": head_dim, "dtype": dtype, "submit": submit,
            "fused": fused, "pass_no": pass_no, "kv_scale": kv_scale, "q_scale": q_scale}


def listed():
    return [
        # The smallest problem: one fp32 layer, root -> 4 fields -> summary, called directly; the 4 fields are being decoded.
        _case("tiny_f32", "diamond", 4, 16, 16, 0, 256, 1, 1, 4, 2, 64, "f32", "eager", False, 24, 1.0),
        # fp32 caches at the size of an ordinary model: a full-precision run of a batch of scenes.
        _case("f32_8scenes", "fan", 6, 64, 32, 0, 2048, 8, 4, 32, 8, 128, "f32", "graph", False, 20),
        # Half-billion-class heads (head_dim 64, 14 query heads on 2 KV heads), one scene, every call issued by
        # the host and the append a kernel of its own: the library as it is used without any option.
        _case("d64_1scene_eager", "fan", 6, 64, 32, 0, 1531, 1, 24, 14, 2, 64, "bf16", "eager", False, 20),
        # The same heads, a batch of scenes with multi-camera prefixes.
        _case("d64_16scenes", "fan", 6, 96, 16, 0, 4096, 16, 24, 14, 2, 64, "bf16", "graph", True, 40),
        # One scene of a 7B-class model decoding a single field: ordinary sequential decoding, latency-bound.
        _case("7b_1scene_chain", "chain", 8, 64, 32, 0, 1024, 1, 28, 28, 4, 128, "bf16", "graph", True, 200),
        # The same model with the six perception fields in flight.
        _case("7b_1scene", "fan", 6, 64, 32, 0, 2048, 1, 28, 28, 4, 128, "bf16", "graph", True, 30),
        # The headline workload: 16 scenes, multi-camera prefix, lengths drawn per scene, replayed pass.
        _case("batched_16scenes", "fan", 6, 96, 16, 0, 4096, 16, 32, 32, 8, 128, "bf16", "graph", True, 40),
        # Wide graph: 16 leaves of every scene decode at once (64 query rows per KV head).
        _case("wide_8scenes", "wide", 16, 48, 48, 0, 8192, 8, 32, 32, 8, 128, "bf16", "graph", True, 24, 1.0),
        # 32 fields at once (128 query rows per KV head) over a short prefix.
        _case("32fields_short", "free", 32, 64, 64, 0, 1024, 8, 32, 32, 8, 128, "bf16", "graph", True, 32),
        # 32 fields at once over the longest prefix, scores with a real model's spread.
        _case("32fields_long", "free", 32, 64, 64, 0, 32768, 8, 4, 32, 8, 128, "bf16", "graph", True, 32, 0.5, 3.0),
        # The largest batch: 64 scenes of 4 fields over a long prefix.
        _case("64scenes_long", "free", 4, 64, 64, 0, 16384, 64, 3, 32, 8, 128, "bf16", "graph", True, 32),
        # A whole template in one graph launch: field-name rows written first, no lengths given (fields run to
        # their slot), odd prefix and slots, three scenes, the append a kernel of its own.
        _case("loop_3scenes", "fan", 5, 23, 0, 6, 1000, 3, 8, 28, 4, 128, "bf16", "loop", False, 0),
    ]


# (query heads, KV heads, head_dim) in use
HEADS = [(28, 4, 128), (32, 8, 128), (32, 8, 128), (14, 2, 64), (4, 2, 64)]
MOST = {"bf16": (10e9, 500e9), "f32": (0.55e9, 6e9)}     # bytes and operations of one drawn pass (the listed ones have more)


def draw(rng):
    """One more case: sizes over the listed ones' ranges (over their logarithm where those are wide)."""
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))
    while True:
        hq, hkv, d = rng.choice(HEADS)
        dtype = "f32" if rng.random() < 0.15 else "bf16"
        template = rng.choice(["fan", "fan", "wide", "diamond", "free", "free", "chain"])
        widest = 128 // (hq // hkv)
        lo = {"wide": 2, "fan": 2, "diamond": 2}.get(template, 1)
        fields = log_int(lo, min(32, widest))
        slot = rng.randint(16, 96)
        len_lo = rng.choice([0, max(8, slot // 6), slot // 2, slot])
        c = _case("", template, fields, slot, len_lo, rng.choice([0, 0, 3, 6]), log_int(256, 32768), log_int(1, 64), 1, hq, hkv, d, dtype,
                  rng.choice(["graph", "graph", "graph", "eager"]), rng.random() < 0.7, 0, 0.5, rng.choice([1.0, 1.0, 3.0]))
        del c["name"]
        c["pass_no"] = rng.randrange(max(s[2] for s in _schedule(c)))
        one = work(c)
        # as many layers as a model has, while the pass stays below the largest listed one
        room = min(MOST[dtype][0] / one["bytes"], MOST[dtype][1] / one["flops"])
        if room < 1.0:
            continue
        c["layers"] = min(rng.choice([8, 24, 28, 32]), int(room))
        return c


# ------------------------------------------------------------------------------------------------
# templates and their schedules
# ------------------------------------------------------------------------------------------------

def _template(c):
    """(nodes, edges, slot rows, field-name rows, widest frontier)"""
    k, t = c["fields"], c["template"]
    if t == "fan":
        n, edges, wide = k + 2, [(i, k) for i in range(k)] + [(k, k + 1)], k
    elif t == "wide":
        rng = np.random.default_rng(k)
        n, wide = k + 3, k
        edges = [(int(leaf), agg) for agg in (k, k + 1) for leaf in sorted(rng.choice(k, size=(k + 1) // 2, replace=False))]
        edges += [(k, k + 2), (k + 1, k + 2)]
    elif t == "diamond":
        n, edges, wide = k + 2, [(0, i) for i in range(1, k + 1)] + [(i, k + 1) for i in range(1, k + 1)], k
    elif t == "free":
        n, edges, wide = k, [], k
    else:
        n, edges, wide = k, [(i, i + 1) for i in range(k - 1)], 1
    fixed = [(3 + v * 2) % (c["fixed"] + 1) for v in range(n)]
    return n, edges, [c["slot"]] * n, fixed, max(1, wide)


def _lengths(c):
    """int32 [scenes][nodes]: rows of every field, field-name rows included."""
    n, _, cap, fixed, _ = _template(c)
    if not c["len_lo"]:
        return np.tile(np.array(cap, np.int32), (c["scenes"], 1))
    rng = np.random.default_rng(260202864 + c["slot"] * 131 + c["fields"])
    lens = rng.integers(c["len_lo"], c["slot"] + 1, size=(c["scenes"], n)).astype(np.int32)
    return np.maximum(lens, np.array(fixed, np.int32) + 1)


def _schedule(c):
    """Per scene: first pass and one past the last pass of every field, and the scene's number of passes."""
    n, edges, _, fixed, _ = _template(c)
    lens = _lengths(c)
    out = []
    for s in range(c["scenes"]):
        start, end = [0] * n, [0] * n
        for v in range(n):                                   # (edges go from lower to higher ids)
            start[v] = max([end[u] for u, w in edges if w == v], default=0)
            end[v] = start[v] + int(lens[s, v]) - fixed[v]
        out.append((start, end, max(end)))
    return out


def _pass_work(c, sched, pass_no):
    """Active fields, rows some field sees (each once), (field, row) pairs that are seen; over all scenes."""
    n, edges, _, fixed, _ = _template(c)
    anc = [set() for _ in range(n)]
    for v in range(n):
        for u, w in edges:
            if w == v:
                anc[v] |= anc[u] | {u}
    active = rows = pairs = 0
    for start, end, _ in sched:
        now = [v for v in range(n) if start[v] <= pass_no < end[v]]
        have = [fixed[v] + min(max(pass_no + 1 - start[v], 0), end[v] - start[v]) for v in range(n)]
        seen = [0] * n
        for v in now:
            for u in range(n):
                r = have[u] if u == v or u in anc[v] else (fixed[u] if u < v else 0)
                seen[u] = max(seen[u], r)
                pairs += r
        active += len(now)
        pairs += len(now) * c["prefix"]
        rows += sum(seen) + (c["prefix"] if now else 0)
    return active, rows, pairs


def work(c):
    """Every visible K/V row read once for all fields and heads that share it; queries and new K/V rows read
    once; outputs, new cache rows and the pass's bitmaps written once."""
    es = 4 if c["dtype"] == "f32" else 2
    row = 2 * c["hkv"] * c["head_dim"] * es
    n, _, cap, fixed, wide = _template(c)
    words = -(-sum(cap) // 64)
    sched = _schedule(c)
    passes = range(max(s[2] for s in sched)) if c["submit"] == "loop" else [c["pass_no"]]
    b = f = 0.0
    for i in passes:
        active, rows, pairs = _pass_work(c, sched, i)
        b += c["layers"] * (rows * row + active * (2 * c["hq"] * c["head_dim"] * es + 2 * row)) + active * words * 8
        f += c["layers"] * pairs * c["hq"] * c["head_dim"] * 4.0
    if c["submit"] == "loop":
        b += 2.0 * c["layers"] * c["scenes"] * sum(fixed) * row
    return {"bytes": float(b), "flops": float(f)}


def tolerance(c):
    """bf16: the weights of the attention are rounded to bf16 (2^-9 each) before they meet V, and so is the
    output.  Measured over the listed cases: 2.2e-3 to 2.4e-3 against a 64-bit computation, 3.0e-3 to 3.2e-3
    between two kernels that round against different references, single values up to 0.04 of the root mean
    square.  fp32: 4e-7 to 6e-7 against 64 bits, single values 6e-6; sums in another order a few times that."""
    return {"rel": 1e-2, "max": 0.15} if c["dtype"] == "bf16" else {"rel": 5e-6, "max": 1e-4}


# ------------------------------------------------------------------------------------------------
# the program
# ------------------------------------------------------------------------------------------------

class State:
    pass


def prepare(c, seed):
    dev = "cuda"
    n, edges, cap, fixed, wide = _template(c)
    dt, L, B = DTYPES[c["dtype"]], c["layers"], c["scenes"]
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    st = State()
    st.case, st.scale = c, 1.0 / c["head_dim"] ** 0.5
    st.sess = fdc.DecodeSession(n, edges, cap, fixed if c["fixed"] else None, c["prefix"], wide, B, dev)
    st.sess.set_fused_append(c["fused"])
    shape = (B, L, c["hkv"], c["prefix"] + sum(cap), c["head_dim"])

    def normal(*shape, scale):
        return torch.empty(shape, dtype=dt, device=dev).normal_(0.0, scale, generator=gen)
    # the cache as prefill and the earlier passes left it
    st.k, st.v = normal(*shape, scale=c["kv_scale"]), normal(*shape, scale=c["kv_scale"])
    st.q = normal(L, B, wide, c["hq"], c["head_dim"], scale=c["q_scale"])
    st.k_new, st.v_new = (normal(L, B, wide, c["hkv"], c["head_dim"], scale=c["kv_scale"]) for _ in range(2))
    st.out = torch.zeros_like(st.q)
    st.sess.bind_cache(st.k, st.v, c["hq"])
    # the scenes' lengths come in an order of the seed's own
    lens = torch.from_numpy(_lengths(c)).to(dev)[torch.randperm(B, generator=gen, device=dev)]
    st.lens = lens.contiguous() if c["len_lo"] else None
    if c["submit"] == "loop":
        nf = sum(fixed)
        st.k_fixed, st.v_fixed = (normal(L, B, c["hkv"], max(nf, 1), c["head_dim"], scale=c["kv_scale"]) for _ in range(2))
        st.log = torch.zeros((sum(cap),) + tuple(st.out.shape), dtype=dt, device=dev)
        st.at = torch.zeros(1, dtype=torch.int64, device=dev)
        st.sess.init(st.lens)
        st.sess.frontier()
        st.sess.build_masks()
        _layers(st)                                          # a first pass outside the capture
        torch.cuda.synchronize()
        st.loop = DeviceLoop(st.sess, lambda stream: _loop_body(st, stream), sum(cap))
        return st
    st.sess.init(st.lens)
    for _ in range(c["pass_no"]):
        st.sess.frontier()
    st.resume = st.sess.state.clone()
    if c["submit"] == "graph":
        _one_pass(st)                                        # a first pass outside the capture
        st.out.zero_()
        torch.cuda.synchronize()
        st.graph = torch.cuda.CUDAGraph()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(st.graph, stream=side, capture_error_mode="thread_local"):
            _one_pass(st)
        torch.cuda.current_stream().wait_stream(side)
    else:
        st.sess.use_stream(torch.cuda.current_stream())
    return st


def _layers(st, stream=None):
    for l in range(st.case["layers"]):
        st.sess.kv_append(l, st.k_new[l], st.v_new[l], stream)
        st.sess.decode_attn(l, st.q[l], st.out[l], st.scale, stream)


def _one_pass(st):
    st.sess.state.copy_(st.resume)
    st.sess.frontier()
    st.sess.build_masks()
    _layers(st)


def _loop_body(st, stream):
    """One pass of the loop: the model's layers, its outputs kept, the next pass's tables."""
    _layers(st, stream)
    st.log.index_copy_(0, st.at, st.out[None])
    st.at.add_(1)
    st.sess.frontier(None, stream)
    st.sess.build_masks(stream)


def run(st):
    s, c = st.sess, st.case
    P = c["prefix"]
    got = {"n_active": s.n_active, "node": s.node, "tok_idx": s.tok_idx, "kv_row": s.kv_row, "pos_id": s.pos_id, "all_done": s.all_done,
           "mask": s.mask, "umask": s.umask, "ntiles": s.ntiles,
           "k_rows": st.k[:, :, :, P:], "v_rows": st.v[:, :, :, P:]}     # all rows of the cache that decoding may write
    if c["submit"] == "loop":
        st.at.zero_()
        s.init(st.lens)
        for l in range(c["layers"]):
            s.write_fixed(l, st.k_fixed[l], st.v_fixed[l])
        s.frontier()
        s.build_masks()
        st.loop.launch()
        return dict(got, out=st.log, passes=st.loop.passes)
    if c["submit"] == "graph":
        st.graph.replay()
    else:
        _one_pass(st)
    return dict(got, out=st.out)
