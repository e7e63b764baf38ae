"""The work that a user of this library has it do, as cases that can be timed.

A case is one of three kinds:
  step   one denoising step at the merge layer through ``MergeLayerStep``: attention + importance map, select, merge,
         then the post-merge layers (projection + attention on the shortened sequence); host-launched, or replayed as
         the CUDA graph a program records once per problem
  block  a whole post-merge block on the shortened sequence (projection, attention, output projection, feed-forward
         network) through ``MergeLayerStep.post_block``
  kv     select + merge of a cached K/V prefix through ``Context``
Inputs follow ``workload.py``: visual tokens in clusters (centre N(0,1), noise 0.1), prompt and response rows N(0,1),
weights N(0, 0.02), a tenth of the visual keys and the decider queries moved by a shared direction of norm 4 per head.
"""
import math

import numpy as np
import torch

from paper_2511_12280_b200 import binding as B_
from paper_2511_12280_b200.pipeline import MergeLayerStep

CLUSTERS = 128
SIGMA_W = 0.02


def _requests(case):
    """Per request (visual, prompt, response, deciders, keep ratio).  A batch spreads its lengths over [visual_min, visual]
    and [prompt_min, prompt] and its deciders and keep ratios likewise: ragged, and the same for every seed."""
    B = case["batch"]
    if B == 1:
        return [(case["visual"], case["prompt"], case["response"], case["deciders"], case["keep"])]
    out = []
    for b in range(B):
        f = ((b * 5 + 2) % B) / (B - 1)
        v = case["visual_min"] + int(f * (case["visual"] - case["visual_min"]))
        p = case["prompt_min"] + int((1 - f) * (case["prompt"] - case["prompt_min"]))
        d = max(1, min(case["response"], case["deciders"] - 3 * (b % 4)))
        out.append((v, p, case["response"], d, min(1.0, case["keep"] * (0.4, 1.0, 2.0)[b % 3])))
    return out


def _step_case(name, dtype, heads, head_dim, visual, prompt, response, deciders, keep, post, batch=1, visual_min=0,
               prompt_min=0, graph=False):
    c = dict(kind="step", dtype=dtype, heads=heads, head_dim=head_dim, batch=batch, visual=visual, visual_min=visual_min,
             prompt=prompt, prompt_min=prompt_min, response=response, deciders=deciders, keep=keep, post=post, graph=graph)
    return dict(c, name=name) if name else c


def _block_case(name, heads, head_dim, ffn, batch, visual, visual_min, prompt, prompt_min, response, keep):
    c = dict(kind="block", dtype="bf16", heads=heads, head_dim=head_dim, ffn=ffn, batch=batch, visual=visual,
             visual_min=visual_min, prompt=prompt, prompt_min=prompt_min, response=response, deciders=8, keep=keep)
    return dict(c, name=name) if name else c


def _kv_case(name, dtype, heads, head_dim, batch, visual, visual_min, prompt, prompt_min, keep, mean):
    c = dict(kind="kv", dtype=dtype, heads=heads, head_dim=head_dim, batch=batch, visual=visual, visual_min=visual_min,
             prompt=prompt, prompt_min=prompt_min, response=0, deciders=0, keep=keep, mean=mean)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one small fp32 merge layer, where latency and launches are everything
        _step_case("tiny_fp32", "fp32", 4, 64, 256, 16, 16, 8, 0.25, 0),
        # fp32 storage at a middle size, with two post-merge layers
        _step_case("image_fp32", "fp32", 8, 64, 1024, 64, 64, 32, 0.25, 2),
        # a narrow model with 64-wide heads; odd lengths throughout
        _step_case("narrow_odd", "bf16", 16, 64, 577, 45, 101, 17, 0.3, 2),
        # one image in a wide model, strong pruning, the merge layer alone
        _step_case("image", "bf16", 32, 128, 1024, 64, 64, 32, 0.10, 0),
        # a multi-crop image with three post-merge layers
        _step_case("crops", "bf16", 32, 128, 4096, 128, 64, 32, 0.25, 3),
        # a step in the middle of a schedule, replayed as the graph recorded for it
        _step_case("schedule_graph", "bf16", 32, 128, 2048, 64, 64, 32, 0.25, 3, graph=True),
        # the first step of a schedule: no decider yet, so nothing is merged and the layers run at full length
        _step_case("first_step", "bf16", 32, 128, 2048, 64, 64, 0, 1.0, 3),
        # serving: eight ragged requests in one packed batch
        _step_case("batch", "bf16", 32, 128, 4096, 256, 64, 48, 0.25, 3, batch=8, visual_min=1024, prompt_min=32),
        # several images in one request: the longest sequence, the merge layer alone, an odd number of tokens
        _step_case("many_images", "bf16", 32, 128, 12287, 128, 64, 32, 0.10, 0),
        # a whole block after the merge, one request
        _block_case("block", 32, 128, 12288, 1, 4096, 0, 128, 0, 64, 0.25),
        # the same for a ragged batch of shortened sequences
        _block_case("block_batch", 32, 128, 12288, 4, 4096, 1024, 256, 32, 64, 0.25),
        # merging a cached K/V prefix (MEAN aggregation of keys and values)
        _kv_case("kv_prefix", "bf16", 32, 128, 1, 4096, 0, 128, 0, 0.25, True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: visual tokens 256 .. 12287 (fp32 up to 1024), 1 .. 8 requests, widths 256 .. 4096."""
    limit = max(work(c)["flops"] for c in listed())
    while True:
        what = rng.choice(["step", "step", "step", "fp32", "block", "kv"])
        heads, head_dim = rng.choice([(32, 128), (32, 128), (16, 128), (16, 64), (8, 64)])
        batch = rng.choice([1, 1, 1, rng.randint(2, 8)])
        keep = rng.choice([0.1, 0.25, 0.5, round(rng.uniform(0.05, 0.75), 3)])
        prompt, response = _log(rng, 16, 256), rng.choice([16, 64, 64, rng.randint(16, 128)])
        deciders = rng.randint(1, min(response, 48))
        pmin = rng.randint(8, prompt)
        if what == "fp32":
            v = _log(rng, 256, 1024)
            h, d = rng.choice([(4, 64), (8, 64), (8, 32), (4, 128)])
            c = _step_case(None, "fp32", h, d, v, prompt, response, deciders, keep, rng.randint(0, 2), rng.choice([1, 1, 2]),
                           max(128, v // 2), pmin, rng.random() < 0.3)
        elif what == "block":
            v = _log(rng, 512, 4096)
            c = _block_case(None, heads, head_dim, heads * head_dim * 3, batch, v, v // 4, prompt, pmin, response, keep)
        elif what == "kv":
            v = _log(rng, 512, 8192)
            c = _kv_case(None, rng.choice(["bf16", "bf16", "bf16", "fp32"]) if v <= 1024 else "bf16", heads, head_dim, batch, v,
                         v // 4, prompt, pmin, keep, rng.random() < 0.5)
        else:
            v = _log(rng, 256, 12287)
            c = _step_case(None, "bf16", heads, head_dim, v, prompt, response, deciders, keep, rng.choice([0, 2, 3]), batch,
                           max(128, v // 4), pmin, rng.random() < 0.3)
        if work(c)["flops"] <= limit:
            return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _normal(g, *shape, sigma=1.0):
    return torch.randn(*shape, generator=g, device="cuda") * sigma


def _weights(g, rows, cols, dt):
    return _normal(g, rows, cols, sigma=SIGMA_W).to(dt)


def _sizes(case, reqs):
    n_vis = [r[0] for r in reqs]
    keep = [B_.d3tom_keep_count(v, r) if (case["kind"] != "step" or d) else v for v, _, _, d, r in reqs]
    return n_vis, [r[1] for r in reqs], [r[2] for r in reqs], keep


def _qkv(case, g, reqs):
    """Q, K, V of the packed batch, the decider positions of every request (ascending)."""
    H, dh, dt = case["heads"], case["head_dim"], _dtype(case)
    D = H * dh
    w = [_normal(g, D, D, sigma=SIGMA_W) for _ in range(3)]
    parts, dec = ([], [], []), []
    for v, p, o, nd, _ in reqs:
        centres = _normal(g, CLUSTERS, D)
        ids = torch.randint(0, CLUSTERS, (v,), generator=g, device="cuda")
        x = torch.cat([centres[ids] + _normal(g, v, D, sigma=0.1), _normal(g, p + o, D)]).to(dt).float()
        u = _normal(g, H, dh)
        u = 4.0 * (u / u.norm(dim=1, keepdim=True)).reshape(1, D)
        salient = torch.randperm(v, generator=g, device="cuda")[: max(1, round(0.1 * v))]
        pos = torch.randperm(o, generator=g, device="cuda")[:nd].sort().values + (v + p) if o else torch.zeros(0, dtype=torch.int64, device="cuda")
        q, k, val = (x @ m.T for m in w)
        k[salient] += u
        q[pos] += u
        for part, t in zip(parts, (q, k, val)):
            part.append(t.to(dt))
        dec.append(pos.cpu().numpy().astype(np.int32))
    return [torch.cat(p).contiguous() for p in parts] + [dec]


def _make_step(case, reqs, dec, n_post):
    n_vis, n_prompt, n_resp, keep = _sizes(case, reqs)
    total = sum(n_vis) + sum(n_prompt) + sum(n_resp)
    step = MergeLayerStep(case["heads"], case["head_dim"], _dtype(case), total, len(reqs), sum(len(d) for d in dec),
                          max(n_vis), n_post=n_post)
    step.set_problem(n_vis, n_prompt, n_resp, dec, keep)
    return step


def prepare(case, seed):
    g, reqs, dt = _gen(seed), _requests(case), _dtype(case)
    D = case["heads"] * case["head_dim"]
    if case["kind"] == "step":
        q, k, v, dec = _qkv(case, g, reqs)
        step = _make_step(case, reqs, dec, case["post"])
        w = [_weights(g, 3 * D, D, dt) for _ in range(case["post"])]
        s = dict(kind="step", step=step, q=q, k=k, v=v, w=w, graph=None)
        s["out"] = dict(attn_out=step.attn_out[: step.total], importance=step.importance[: step.total_vis],
                        keep_mask=step.keep_mask[: step.total_vis], assign=step.assign[: step.total_vis],
                        member_count=step.member_count[: step.total_kept], src_of_dst=step.src_of_dst[: step.total_out],
                        hidden_out=step.hidden_out[: step.total_out],
                        layers=[step.layer_out[l][: step.total_out] for l in range(case["post"])])
        if case["graph"]:
            s["graph"] = step.capture(q, k, v, w)
        return s
    if case["kind"] == "block":
        step = _make_step(case, reqs, [np.zeros(0, np.int32)] * len(reqs), 1)
        m, n = case["ffn"], step.total_out
        s = dict(kind="block", step=step, x=_normal(g, n, D).to(dt), w_qkv=_weights(g, 3 * D, D, dt), w_o=_weights(g, D, D, dt),
                 w_gate_up=_weights(g, 2 * m, D, dt), w_down=_weights(g, D, m, dt))
        s["out"] = step.layer_out[0][:n]
        return s
    _, k, v, dec = _qkv(case, g, reqs)
    n_vis, n_prompt, n_resp, keep = _sizes(case, reqs)
    step = _make_step(case, reqs, dec, 0)              # (its index arrays and output buffers; the calls below are the context's)
    s = dict(kind="kv", step=step, k=k, v=v, mode=B_.AGG_MEAN if case["mean"] else B_.AGG_SUM,
             importance=torch.rand(step.total_vis, generator=g, device="cuda").square_() * 8.0 + 0.01,
             v_out=torch.empty_like(step.hidden_out))
    s["out"] = dict(k_out=step.hidden_out[: step.total_out], v_out=s["v_out"][: step.total_out],
                    keep_mask=step.keep_mask[: step.total_vis], assign=step.assign[: step.total_vis],
                    member_count=step.member_count[: step.total_kept], src_of_dst=step.src_of_dst[: step.total_out])
    return s


def run(s):
    st = s["step"]
    if s["kind"] == "step":
        if s["graph"] is not None:
            s["graph"].replay()
        else:
            st.run(s["q"], s["k"], s["v"], s["w"])
    elif s["kind"] == "block":
        st.post_block(0, s["x"], s["w_qkv"], s["w_o"], s["w_gate_up"], s["w_down"])
    else:
        st.ctx.d3tom_select(s["importance"], st.cu_vis, st.keep_d, st.cu_kept, st.nB, st.max_visual, st.kept_idx, st.keep_mask)
        st.ctx.d3tom_merge_kv(s["mode"], s["k"], s["v"], st.cu_seqlens, st.n_visual_d, st.cu_vis, st.kept_idx, st.cu_kept, st.nB,
                              st.D, st.total, st.total_out, st.max_visual, st.max_kept, st.hidden_out, s["v_out"], st.cu_out,
                              st.assign, st.member_count, st.src_of_dst)
    return s["out"]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    reqs = _requests(case)
    es = 2 if case["dtype"] == "bf16" else 4
    D = case["heads"] * case["head_dim"]
    flops = nbytes = 0.0
    n_in = n_out = 0
    for v, p, o, d, r in reqs:
        k = max(1, min(v, math.floor(r * v + 1e-9))) if (case["kind"] != "step" or d) else v
        n, nm = v + p + o, p + o + k
        n_in, n_out = n_in + n, n_out + nm
        if case["kind"] == "step":
            flops += 4.0 * n * n * D + 2.0 * (v - k) * k * D + case["post"] * 4.0 * nm * nm * D
            nbytes += v * (4 + 1 + 4) + k * 4
        elif case["kind"] == "kv":
            flops += 2.0 * (v - k) * k * D
            nbytes += v * (4 + 1 + 4) + k * 4
        else:
            flops += 4.0 * nm * nm * D
    if case["kind"] == "step":
        flops += case["post"] * 6.0 * n_out * D * D
        nbytes += 4.0 * n_in * D * es + n_out * (D * es + 4) + case["post"] * (3.0 * D * D + n_out * D) * es
    elif case["kind"] == "kv":
        nbytes += 2.0 * (n_in + n_out) * D * es + n_out * 4
    else:
        m = case["ffn"]
        flops += n_out * (8.0 * D * D + 6.0 * D * m)
        nbytes += (4.0 * D * D + 3.0 * D * m + 2.0 * n_out * D) * es
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # A pruned token whose two best cosines agree to rounding may go to either (its slot is one of the whole values that
    # may differ; the rows of the two kept tokens then change by a little), which is what "max" and "differ" leave room for.
    if case["dtype"] == "fp32":
        return {"rel": 2e-3, "max": 0.3, "differ": 0.005}
    return {"rel": 1e-2, "max": 0.5, "differ": 0.005}


# ------------------------------------------------------------------ the same in 64 bits
def _attention64(q, k, v, heads, dh, decider, n_vis):
    """softmax(q k^T / sqrt(dh)) v of one request, one head at a time, and the decider rows' mass on the visual keys."""
    n = q.shape[0]
    out = torch.empty(n, heads * dh, dtype=torch.float64, device=q.device)
    imp = torch.zeros(n_vis, dtype=torch.float64, device=q.device)
    for h in range(heads):
        c = slice(h * dh, (h + 1) * dh)
        kh, vh = k[:, c].double(), v[:, c].double()
        for r0 in range(0, n, 4096):
            a = torch.softmax(q[r0:r0 + 4096, c].double() @ kh.T / math.sqrt(dh), dim=1)
            out[r0:r0 + 4096, c] = a @ vh
        if len(decider):
            rows = torch.as_tensor(decider, dtype=torch.int64, device=q.device)
            imp += torch.softmax(q[rows, c].double() @ kh.T / math.sqrt(dh), dim=1)[:, :n_vis].sum(0)
    return out, imp


def exact(case, seed):
    """Attention states and importance of a step (the merged rows follow a ranking and have no value of their own in
    64 bits: a near-tie falls either way), a block's output, the merged caches of a prefix."""
    H, dh = case["heads"], case["head_dim"]
    D = H * dh
    reqs = _requests(case)
    s = prepare(dict(case, graph=False), seed)
    st = s["step"]
    if s["kind"] == "step":
        dec_h, cu = st.dec_pos.cpu().numpy(), st.cu_dec_h
        outs = [_attention64(*(t[st.cu_seqlens_h[b]:st.cu_seqlens_h[b + 1]] for t in (s["q"], s["k"], s["v"])), H, dh,
                             dec_h[cu[b]:cu[b + 1]], st.n_visual_h[b]) for b in range(len(reqs))]
        return dict(attn_out=torch.cat([o for o, _ in outs]), importance=torch.cat([i for _, i in outs]), keep_mask=None,
                    assign=None, member_count=None, src_of_dst=None, hidden_out=None, layers=[None] * case["post"])
    if s["kind"] == "block":
        x, m = s["x"].double(), case["ffn"]
        qkv = x @ s["w_qkv"].double().T
        at = torch.cat([_attention64(*(qkv[st.cu_out_h[b]:st.cu_out_h[b + 1], i * D:(i + 1) * D] for i in range(3)), H, dh, [], 0)[0]
                        for b in range(len(reqs))])
        x1 = x + at @ s["w_o"].double().T
        gate = x1 @ s["w_gate_up"][:m].double().T
        act = torch.nn.functional.silu(gate) * (x1 @ s["w_gate_up"][m:].double().T)
        return x1 + act @ s["w_down"].double().T
    ks, vs = [], []
    for b, (v, p, o, _, _) in enumerate(reqs):
        lo, kc = int(st.cu_seqlens_h[b]), st.keep_h[b]
        imp = s["importance"][int(st.cu_vis_h[b]):int(st.cu_vis_h[b]) + v]
        kept = torch.sort(torch.sort(imp, descending=True, stable=True).indices[:kc]).values
        pruned = torch.ones(v, dtype=torch.bool, device="cuda")
        pruned[kept] = False
        K, V = s["k"][lo:lo + v + p].double(), s["v"][lo:lo + v + p].double()
        Kn = K[:v] / K[:v].norm(dim=1, keepdim=True).clamp_min(1e-300)
        to = (Kn[pruned] @ Kn[kept].T).argmax(dim=1)
        n = torch.ones(kc, dtype=torch.float64, device="cuda").index_add_(0, to, torch.ones(len(to), dtype=torch.float64, device="cuda"))
        for dst, t in ((ks, K), (vs, V)):
            merged = t[:v][kept].index_add(0, to, t[:v][pruned])
            dst.append(torch.cat([merged / n[:, None] if case["mean"] else merged, t[v:]]))
    return dict(k_out=torch.cat(ks), v_out=torch.cat(vs), keep_mask=None, assign=None, member_count=None, src_of_dst=None)
