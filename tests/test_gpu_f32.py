"""fp32 storage: the CUDA-core attention and matrix kernels at the edges of their tiles, against float64."""
import math

import numpy as np
import pytest
import torch

from paper_2511_12280_b200 import binding as B_

pytestmark = pytest.mark.gpu


def _unaligned(t):
    """The same values 4 bytes off a 16-byte boundary (the scalar-copy path)."""
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)[1:]
    return flat.copy_(t.reshape(-1)).reshape(t.shape)


def _close(got, want):
    # fp32 sums of up to a few thousand terms: rounding grows like sqrt(terms) * 2^-24, far inside 1e-5 + 1e-4 |want|
    want = want.cpu().numpy()
    err = np.abs(got.double().cpu().numpy() - want)
    assert np.isfinite(err).all() and (err <= 1e-5 + 1e-4 * np.abs(want)).all(), err.max()


def _launches(call):
    """(grid, dynamic shared memory) of each kernel of `call`, read from a recorded graph."""
    from cuda.bindings import driver
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = driver.CUgraph(graph.raw_cuda_graph())
    _, _, n = driver.cuGraphGetNodes(raw)
    err, nodes, n = driver.cuGraphGetNodes(raw, n)
    assert err == driver.CUresult.CUDA_SUCCESS
    out = []
    for node in nodes[:n]:
        if driver.cuGraphNodeGetType(node)[1] == driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            p = driver.cuGraphKernelNodeGetParams(node)[1]
            out.append(((p.gridDimX, p.gridDimY, p.gridDimZ), p.sharedMemBytes))
    return out


# rows and heads that take 4, 8 and (up to 32 channels, from ceil(rows / 8) x heads x requests > 16 x SMs on: 700 x 32 x 4 and
# 2400 x 8 x 32) 16 rows per warp; head sizes below, at and above the padded widths 32 / 64 / 128
@pytest.mark.parametrize("lens,H,dh", [([1], 2, 64), ([15, 16, 17], 4, 64), ([31, 33], 2, 32), ([255, 257], 1, 36),
                                       ([130], 3, 128), ([65, 1, 200], 2, 100), ([1152], 8, 64), ([700], 32, 4), ([288], 4, 64),
                                       ([600], 4, 128), ([2400], 8, 32), ([1400, 1400], 8, 64), ([620], 32, 100), ([620], 32, 128)])
@pytest.mark.parametrize("aligned", [True, False])
def test_attention_and_importance_fp32(lens, H, dh, aligned):
    g = torch.Generator().manual_seed(sum(lens) + dh)
    n, D, B = sum(lens), H * dh, len(lens)
    q, k, v = (torch.randn(n, D, generator=g).cuda() for _ in range(3))
    if not aligned:
        q, k, v = _unaligned(q), _unaligned(k), _unaligned(v)
    out = torch.full((n, D), float("nan"), device="cuda")
    if not aligned:
        out = _unaligned(out)
    vis = [max(1, m // 2) for m in lens]
    dec = [np.arange(m - max(1, m // 8), m, dtype=np.int32) for m in lens]      # the last rows of every request
    cs = lambda a: torch.tensor(np.concatenate([[0], np.cumsum(a)]), dtype=torch.int32, device="cuda")
    ctx = B_.Context(n, B, H, dh, sum(len(d) for d in dec), max(vis))
    imp = torch.full((sum(vis),), float("nan"), device="cuda")
    ctx.d3tom_attn_importance(q, k, v, cs(lens), torch.tensor(vis, dtype=torch.int32, device="cuda"),
                              torch.tensor(np.concatenate(dec), device="cuda"), cs([len(d) for d in dec]), B, n, max(lens), max(vis),
                              sum(len(d) for d in dec), 1 / math.sqrt(dh), out, imp, cs(vis))
    lo = v0 = 0
    for m, nv, d in zip(lens, vis, dec):
        qb, kb, vb = (t[lo:lo + m].double().reshape(m, H, dh).transpose(0, 1) for t in (q, k, v))
        a = torch.softmax(qb @ kb.transpose(1, 2) / math.sqrt(dh), dim=2)
        _close(out[lo:lo + m], (a @ vb).transpose(0, 1).reshape(m, D))
        _close(imp[v0:v0 + nv], a[:, torch.tensor(d.astype(np.int64), device="cuda"), :nv].sum((0, 1)))
        lo, v0 = lo + m, v0 + nv
    assert ctx.device_status() == 0


# products in 32 x 32, 64 x 64 and 32 x 64 tiles (linear and gate-up; the down product of a feed-forward network has its own),
# K with and without a remainder of the k-blocks and of the vectors
SHAPES = [(1, 4, 4), (33, 130, 65), (70, 31, 40), (200, 256, 512), (640, 512, 1536), (65, 1000, 33), (384, 96, 3000), (384, 100, 768),
          (384, 768, 768), (512, 130, 1536), (256, 33, 1024)]


def tile_that_runs(rows, n_cols, call):
    """The tile shape of a dense layer's launch, from its grid."""
    (grid, _), = _launches(call)
    ran = [(bm, bn) for bm, bn in ((32, 32), (32, 64), (64, 64)) if grid == (-(-n_cols // bn), -(-rows // bm), 1)]
    assert ran, grid
    return ran[0]


def test_the_dense_shapes_cover_every_tile():
    def linear(rows, K, N):
        x, w, y = torch.zeros(rows, K, device="cuda"), torch.zeros(N, K, device="cuda"), torch.empty(rows, N, device="cuda")
        return tile_that_runs(rows, N, lambda: ctx.d3tom_linear(x, w, None, rows, K, N, y))

    def proj(rows, D):
        x, w = torch.zeros(rows, D, device="cuda"), torch.zeros(3 * D, D, device="cuda")
        out = [torch.empty(rows, D, device="cuda") for _ in range(3)]
        return tile_that_runs(rows, 3 * D, lambda: ctx.d3tom_proj_qkv(x, w, rows, D, *out))

    ctx = B_.Context(2000, 1, 1, 4, 1, 1)
    assert {linear(*s) for s in SHAPES} == {(32, 32), (32, 64), (64, 64)}
    assert linear(384, 768, 768) == proj(512, 512) == proj(384, 130) == (32, 64)
    assert proj(1500, 100) == (64, 64) and proj(33, 100) == (32, 32)


@pytest.mark.parametrize("rows,K,N", SHAPES)
@pytest.mark.parametrize("aligned", [True, False])
def test_linear_and_gate_up_fp32(rows, K, N, aligned):
    g = torch.Generator().manual_seed(rows + K)
    x, w, wd = (torch.randn(*s, generator=g).cuda() * c for s, c in (((rows, K), 1.0), ((2 * N, K), 0.05), ((K, N), 0.05)))
    r = torch.randn(rows, N, generator=g).cuda()
    if not aligned:
        x, w = _unaligned(x), _unaligned(w)
    ctx = B_.Context(rows, 1, 1, 4, 1, 1)
    y = torch.full((rows, N), float("nan"), device="cuda")
    ctx.d3tom_linear(x, w[:N], r, rows, K, N, y)
    _close(y, r.double() + x.double() @ w[:N].double().T)
    act, out = torch.full((rows, N), float("nan"), device="cuda"), torch.full((rows, K), float("nan"), device="cuda")
    ctx.d3tom_ffn(x, w, wd, None, rows, K, N, act, out)
    h = torch.nn.functional.silu(x.double() @ w[:N].double().T) * (x.double() @ w[N:].double().T)
    _close(act, h)
    _close(out, act.double() @ wd.double().T)


# 32 x 64 tiles (with and without remainders), 64 x 64 and 32 x 32
@pytest.mark.parametrize("rows,H,dh", [(512, 8, 64), (384, 13, 10), (1500, 5, 20), (33, 5, 20)])
@pytest.mark.parametrize("aligned", [True, False])
def test_projection_fp32(rows, H, dh, aligned):
    g = torch.Generator().manual_seed(rows)
    D = H * dh
    x, w = torch.randn(rows, D, generator=g).cuda(), torch.randn(3 * D, D, generator=g).cuda() * 0.05
    if not aligned:
        x, w = _unaligned(x), _unaligned(w)
    ctx = B_.Context(rows, 1, H, 4, 1, 1)
    out = [torch.full((rows, D), float("nan"), device="cuda") for _ in range(3)]
    ctx.d3tom_proj_qkv(x, w, rows, D, *out)
    for i, t in enumerate(out):
        _close(t, x.double() @ w[i * D:(i + 1) * D].double().T)


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,K,N", [(33, 130, 65), (70, 36, 40), (200, 256, 96)])
def test_unaligned_buffers_give_the_same_bits(dt, n, K, N):
    # fp32: asynchronous copies or scalar loads; bf16 on the CUDA-core kernels: loads of four elements or scalar ones
    g = torch.Generator().manual_seed(n)
    x, w, r = (torch.randn(*s, generator=g).cuda().to(dt) for s in ((n, K), (N, K), (n, N)))
    qkv = [torch.randn(n, 72, generator=g).cuda().to(dt) for _ in range(3)]
    cu = torch.tensor([0, n], dtype=torch.int32, device="cuda")
    ctx = B_.Context(n, 1, 2, 36, 1, n)
    ctx.set_reference_kernels(True)
    outs = []
    for move in (lambda t: t, _unaligned):
        y, o = move(torch.empty(n, N, dtype=dt, device="cuda")), move(torch.empty(n, 72, dtype=dt, device="cuda"))
        ctx.d3tom_linear(move(x), move(w), move(r), n, K, N, y)
        ctx.d3tom_attn_varlen(*(move(t) for t in qkv), cu, 1, n, n, 36 ** -0.5, o)
        torch.cuda.synchronize()
        outs.append((y.clone(), o.clone()))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    # (fp32 sums of at most 256 terms of unit variance; bf16 rounds the result once more)
    want = r.double() + x.double() @ w.double().T
    assert ((outs[0][0].double() - want).abs() <= (1e-4 if dt == torch.float32 else 2.0 ** -8) * (1 + want.abs())).all()


def test_small_calls_fill_an_sm_with_shared_memory_only_under_launch_overlap():
    n, H, dh = 64, 2, 64
    q, k, v = (torch.randn(n, H * dh, device="cuda") for _ in range(3))
    out, y, w = torch.empty_like(q), torch.empty_like(q), torch.randn(H * dh, H * dh, device="cuda")
    cu = torch.tensor([0, n], dtype=torch.int32, device="cuda")
    ctx = B_.Context(n, 1, H, dh, 1, n)

    def call():
        ctx.d3tom_attn_varlen(q, k, v, cu, 1, n, n, 0.125, out)
        ctx.d3tom_linear(q, w, None, n, H * dh, H * dh, y)

    with_overlap = [b for _, b in _launches(call)]
    got = out.clone(), y.clone()
    B_.d3tom_set_launch_overlap(False)
    try:
        without = [b for _, b in _launches(call)]
        assert torch.equal(got[0], out) and torch.equal(got[1], y)
    finally:
        B_.d3tom_set_launch_overlap(True)
    assert len(with_overlap) == len(without) == 2
    # one CTA per SM of 227 KB while kernels overlap; otherwise what the kernels use: at most 150 KB
    assert all(b > 220 * 1024 for b in with_overlap) and all(b < 150 * 1024 for b in without), (with_overlap, without)


def _heads_tails(n):
    """Row ranges to run by themselves: short, middle and long, so that other tiles serve them than the whole batch."""
    return [(0, 1), (n // 3, n // 3 + 33), (0, n // 2), (n - 200, n)]


@pytest.mark.parametrize("n,K,N", [(1500, 512, 768), (640, 130, 200), (2000, 96, 512), (700, 1000, 96), (3000, 33, 64)])
def test_dense_layers_give_a_row_the_same_bits_alone_and_in_a_batch(n, K, N):
    g = torch.Generator().manual_seed(n + K)
    x, w, wd = (torch.randn(*s, generator=g).cuda() * c for s, c in (((n, K), 1.0), ((2 * N, K), 0.05), ((K, N), 0.05)))
    wq = torch.randn(3 * K, K, generator=g).cuda() * 0.05
    ctx = B_.Context(n, 1, 1, 4, 1, 1)

    def run(a, b):
        m = b - a
        xs = x[a:b].contiguous()
        y, act, out = torch.empty(m, N, device="cuda"), torch.empty(m, N, device="cuda"), torch.empty(m, K, device="cuda")
        q, k, v = (torch.empty(m, K, device="cuda") for _ in range(3))
        ctx.d3tom_linear(xs, w[:N], None, m, K, N, y)
        ctx.d3tom_ffn(xs, w, wd, xs, m, K, N, act, out)
        ctx.d3tom_proj_qkv(xs, wq, m, K, q, k, v)
        return y, act, out, q, k, v

    whole = run(0, n)
    for a, b in _heads_tails(n):
        for got, want in zip(run(a, b), whole):
            assert torch.equal(got, want[a:b]), (a, b)


# one request among others, with lengths at which 4, 8 and (32 channels) 16 rows per warp serve the launch
@pytest.mark.parametrize("lens,H,dh", [([288, 40], 4, 64), ([290, 1200, 1300], 8, 32), ([288, 900, 100], 4, 64), ([288, 1400, 1400], 8, 64), ([150, 700], 32, 128),
                                       ([75, 31], 2, 36)])
def test_attention_importance_and_merge_give_a_request_the_same_bits_alone_and_in_a_batch(lens, H, dh):
    g = torch.Generator().manual_seed(sum(lens))
    D = H * dh
    q, k, v = (torch.randn(sum(lens), D, generator=g).cuda() for _ in range(3))
    vis, keep = [m // 2 for m in lens], [m // 5 for m in lens]
    cs = lambda a: torch.tensor(np.concatenate([[0], np.cumsum(a)]), dtype=torch.int32, device="cuda")
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    kept = [torch.randperm(nv, generator=g)[:kc].sort().values.to(torch.int32).cuda() for nv, kc in zip(vis, keep)]

    def run(which):
        m, B, lo = [lens[i] for i in which], len(which), [sum(lens[:i]) for i in which]
        n, nv, kc = sum(m), [vis[i] for i in which], [keep[i] for i in which]
        rows = torch.cat([torch.arange(a, a + b) for a, b in zip(lo, m)]).cuda()
        qq, kk, vv = (t[rows].contiguous() for t in (q, k, v))
        dec = i32(np.concatenate([np.arange(b - b // 8, b) for b in m]))
        cu_dec = [b // 8 for b in m]
        ctx = B_.Context(n, B, H, dh, int(sum(cu_dec)), max(nv))
        out, imp = torch.empty(n, D, device="cuda"), torch.empty(sum(nv), device="cuda")
        ctx.d3tom_attn_importance(qq, kk, vv, cs(m), i32(nv), dec, cs(cu_dec), B, n, max(m), max(nv), int(sum(cu_dec)), dh ** -0.5,
                                  out, imp, cs(nv))
        lo_out = [b - c + e for b, c, e in zip(m, nv, kc)]
        total_out = sum(lo_out)
        h_out, assign = torch.empty(total_out, D, device="cuda"), torch.empty(sum(nv), dtype=torch.int32, device="cuda")
        count, src = torch.empty(sum(kc), dtype=torch.int32, device="cuda"), torch.empty(total_out, dtype=torch.int32, device="cuda")
        ctx.d3tom_merge(B_.AGG_SUM, out, cs(m), i32(nv), cs(nv), torch.cat([kept[i] for i in which]), cs(kc), B, D, n, total_out,
                        max(nv), max(kc), h_out, cs(lo_out), assign, count, src)
        torch.cuda.synchronize()
        assert ctx.device_status() == 0
        ctx.close()
        return out[:m[0]], imp[:nv[0]], assign[:nv[0]], count[:kc[0]], h_out[:lo_out[0]]

    alone, together = run([0]), run(list(range(len(lens))))
    for a, b in zip(alone, together):
        assert torch.equal(a, b)


# kept counts and lengths on either side of the line between one block per row and tiles of 16 x 32: same bits
@pytest.mark.parametrize("V,k,D", [(9, 3, 4096), (512, 24, 64), (500, 5, 72), (1024, 8, 1000), (33, 32, 256), (4096, 8, 512), (4800, 8, 4096)])
def test_similarity_fp32_gives_the_same_bits_by_rows_and_by_tiles(V, k, D):
    g = torch.Generator().manual_seed(V)
    n, P, pad, pad_keep = V + 4, 4, 5000, 40
    x = torch.randn(n + pad, D, generator=g).cuda()
    kept = torch.randperm(V, generator=g)[:k].sort().values.to(torch.int32)
    more = torch.randperm(pad, generator=g)[:pad_keep].sort().values.to(torch.int32)
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    got = []
    for B in (1, 2):                      # alone, and with a request beside it that is long enough for the tiles
        vis, keep, lens = [V, pad][:B], [k, pad_keep][:B], [n, pad][:B]
        cs = lambda a: i32([0] + list(np.cumsum(a)))
        out_lens = [k + P, pad_keep][:B]
        ctx = B_.Context(sum(lens), B, D // 8, 8, 1, max(vis))
        out = torch.empty(sum(out_lens), D, device="cuda")
        assign, sim = torch.empty(sum(vis), dtype=torch.int32, device="cuda"), torch.full((sum(vis), max(keep)), 7.0, device="cuda")
        count, src = (torch.empty(m, dtype=torch.int32, device="cuda") for m in (sum(keep), sum(out_lens)))
        ctx.d3tom_merge(B_.AGG_SUM, x[:sum(lens)], cs(lens), i32(vis), cs(vis), torch.cat([kept, more][:B]).cuda(), cs(keep), B, D,
                        sum(lens), sum(out_lens), max(vis), max(keep), out, cs(out_lens), assign, count, src, sim)
        torch.cuda.synchronize()
        assert ctx.device_status() == 0
        got.append((assign[:V], sim[:V, :k], out[:k + P], count[:k]))
        ctx.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)
    unit = torch.nn.functional.normalize(x[:V].double(), dim=1)
    cos = unit @ unit[kept.long().cuda()].T
    pruned = torch.ones(V, dtype=torch.bool, device="cuda")
    pruned[kept.long().cuda()] = False
    # (32 chains of at most D / 32 products of unit rows, added pairwise: far inside 1e-5)
    assert (got[0][1][pruned].double() - cos[pruned]).abs().max() <= 1e-5
    assert torch.equal(got[0][0][pruned].long(), got[0][1][pruned].argmax(dim=1))


# one block per 32 keys with a warp per head (up to eight heads and sixteen deciders), and the kernel with partial sums beyond:
# deciders below, at and above either limit, ragged numbers of keys
@pytest.mark.parametrize("H", [1, 4, 5, 8, 9])
@pytest.mark.parametrize("V,n_dec", [(1, 1), (31, 4), (33, 4), (300, 3), (95, 5), (64, 8), (33, 9), (31, 16), (32, 17), (33, 32), (300, 33), (95, 70)])
def test_importance_of_few_heads(H, V, n_dec):
    dev, dh = torch.device("cuda", 0), 32
    g = torch.Generator().manual_seed(V + H)
    n_vis, n_resp = [V, 2 * V + 3], [n_dec + 2, n_dec]
    lens = [a + b for a, b in zip(n_vis, n_resp)]
    N, cu = sum(lens), np.concatenate([[0], np.cumsum(lens)])
    q, k, v = (torch.randn(N, H * dh, generator=g).to(dev) for _ in range(3))
    dec = [np.arange(a, a + n_dec, dtype=np.int32) for a in n_vis]
    i32 = lambda a: torch.as_tensor(np.asarray(a, np.int32), device=dev)
    ctx = B_.Context(N, 2, H, dh, 2 * n_dec, max(n_vis))
    out, imp = torch.empty_like(q), torch.full((sum(n_vis) + 1,), -7.0, device=dev)
    ctx.d3tom_attn_importance(q, k, v, i32(cu), i32(n_vis), i32(np.concatenate(dec)), i32([0, n_dec, 2 * n_dec]), 2, N, max(lens),
                              max(n_vis), 2 * n_dec, dh ** -0.5, out, imp, i32([0, n_vis[0], sum(n_vis)]))
    torch.cuda.synchronize()
    want = []
    for b in range(2):
        rows = slice(int(cu[b]), int(cu[b + 1]))
        qh, kh = (t[rows].double().reshape(lens[b], H, dh).transpose(0, 1) for t in (q, k))
        a = torch.softmax(qh[:, torch.as_tensor(dec[b], dtype=torch.int64, device=dev)] @ kh.transpose(1, 2) * dh ** -0.5, dim=2)
        want.append(a[:, :, : n_vis[b]].sum((0, 1)))
    want = torch.cat(want)
    # every term is a probability with an fp32 relative error of about 1e-5 (scores of magnitude 10 in the exponent)
    assert imp[-1].item() == -7.0 and ((imp[:-1].double() - want).abs() <= 1e-4 * want + 1e-7 * n_dec * H).all()
    ctx.close()


def test_importance_of_a_replay_with_more_deciders_than_were_captured():
    # the host's count is that of the capture; what is summed is the device's list, whichever kernel sums it
    dev, H, dh, V, n = torch.device("cuda", 0), 2, 32, 70, 90
    g = torch.Generator().manual_seed(5)
    q, k, v = (torch.randn(n, H * dh, generator=g).to(dev) for _ in range(3))
    i32 = lambda *a: torch.tensor(a, dtype=torch.int32, device=dev)
    pos, cu_dec, imp, out = torch.arange(V, V + 17, dtype=torch.int32, device=dev), i32(0, 8), torch.zeros(V, device=dev), torch.empty_like(q)
    ctx = B_.Context(n, 1, H, dh, 17, V)
    cu, nv, cu_vis = i32(0, n), i32(V), i32(0, V)
    call = lambda n_dec: ctx.d3tom_attn_importance(q, k, v, cu, nv, pos, cu_dec, 1, n, n, V, n_dec, dh ** -0.5, out, imp, cu_vis)
    call(8)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(8)
    for n_dec in (8, 9, 17):
        cu_dec.copy_(i32(0, n_dec))
        graph.replay()
        torch.cuda.synchronize()
        got = imp.clone()
        call(17)                                   # the kernel for longer lists
        torch.cuda.synchronize()
        assert (got - imp).abs().max() <= 1e-6 * n_dec * H     # probabilities, summed in another order
    ctx.close()
