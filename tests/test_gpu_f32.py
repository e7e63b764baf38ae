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


# rows and heads that take 16, 8 and 4 rows per warp; head sizes below, at and above the padded widths 32 / 64 / 128
@pytest.mark.parametrize("lens,H,dh", [([1], 2, 64), ([15, 16, 17], 4, 64), ([31, 33], 2, 32), ([255, 257], 1, 36),
                                       ([130], 3, 128), ([65, 1, 200], 2, 100), ([1152], 8, 64), ([700], 32, 4), ([288], 4, 64),
                                       ([600], 4, 128), ([2400], 8, 32)])
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


# products that take 64 x 64, 32 x 64 and 32 x 32 tiles, K with and without a remainder of the k-blocks and of the vectors
@pytest.mark.parametrize("rows,K,N", [(1, 4, 4), (33, 130, 65), (70, 31, 40), (200, 256, 512), (640, 512, 1536), (65, 1000, 33),
                                      (384, 96, 3000)])
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


def _shared_memory_of_kernels(call):
    """Dynamic shared memory that each kernel of `call` asks for, read from a recorded graph."""
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
            out.append(driver.cuGraphKernelNodeGetParams(node)[1].sharedMemBytes)
    return out


def test_small_calls_fill_an_sm_with_shared_memory_only_under_launch_overlap():
    n, H, dh = 64, 2, 64
    q, k, v = (torch.randn(n, H * dh, device="cuda") for _ in range(3))
    out, y, w = torch.empty_like(q), torch.empty_like(q), torch.randn(H * dh, H * dh, device="cuda")
    cu = torch.tensor([0, n], dtype=torch.int32, device="cuda")
    ctx = B_.Context(n, 1, H, dh, 1, n)

    def call():
        ctx.d3tom_attn_varlen(q, k, v, cu, 1, n, n, 0.125, out)
        ctx.d3tom_linear(q, w, None, n, H * dh, H * dh, y)

    with_overlap = _shared_memory_of_kernels(call)
    got = out.clone(), y.clone()
    B_.d3tom_set_launch_overlap(False)
    try:
        without = _shared_memory_of_kernels(call)
        assert torch.equal(got[0], out) and torch.equal(got[1], y)
    finally:
        B_.d3tom_set_launch_overlap(True)
    assert len(with_overlap) == len(without) == 2
    # one CTA per SM of 227 KB while kernels overlap; otherwise what the kernels use: at most 150 KB
    assert all(b > 220 * 1024 for b in with_overlap) and all(b < 150 * 1024 for b in without), (with_overlap, without)
