"""d3tom_merge_kv (the merge applied to a cached K/V prefix, Sec. 4.4) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import d3tom_oracle as orc
from paper_2511_12280_b200 import binding as B_
from paper_2511_12280_b200 import workload as wl

import parity_util as pu

pytestmark = pytest.mark.gpu


def run_case(w, mode, keep_ratio=0.25, seed=0):
    """The caches are the workload's K and V rows of each request's [visual | prompt] prefix;
    the kept set is a seeded random subset (the routing does not depend on how it was chosen)."""
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(seed)
    D, dt = w.D, w.dtype
    cu_full = w.cu_seqlens
    rows = np.concatenate([np.arange(cu_full[b], cu_full[b] + w.n_visual[b] + w.n_prompt[b]) for b in range(w.B)])
    k_h = w.k.reshape(-1, D)[rows].contiguous()
    v_h = w.v.reshape(-1, D)[rows].contiguous()
    lens = [v + p for v, p in zip(w.n_visual, w.n_prompt)]
    keep = [max(1, int(keep_ratio * v)) for v in w.n_visual]
    kept = [np.sort(rng.choice(v, k, replace=False)).astype(np.int32) for v, k in zip(w.n_visual, keep)]
    cs = lambda a: np.concatenate([[0], np.cumsum(a)]).astype(np.int32)
    cu, cu_vis, cu_kept = cs(lens), cs(w.n_visual), cs(keep)
    out_lens = [n - v + k for n, v, k in zip(lens, w.n_visual, keep)]
    cu_out = cs(out_lens)
    total, total_out = int(cu[-1]), int(cu_out[-1])
    t = lambda a: torch.as_tensor(np.asarray(a, np.int32), device=dev)
    ctx = B_.Context(total, w.B, w.H, w.dh, 1, max(w.n_visual))
    k_d, v_d = k_h.to(dev), v_h.to(dev)
    k_out = torch.full((total_out, D), float("nan"), dtype=k_d.dtype, device=dev)
    v_out = torch.full((total_out, D), float("nan"), dtype=k_d.dtype, device=dev)
    assign = torch.full((int(cu_vis[-1]),), -9, dtype=torch.int32, device=dev)
    member_count = torch.full((int(cu_kept[-1]),), -9, dtype=torch.int32, device=dev)
    src = torch.full((total_out,), -9, dtype=torch.int32, device=dev)
    sim = torch.full((int(cu_vis[-1]), max(keep)), float("nan"), dtype=torch.float32, device=dev)
    ctx.d3tom_merge_kv(mode, k_d, v_d, t(cu), t(w.n_visual), t(cu_vis), t(np.concatenate(kept)), t(cu_kept), w.B, D, total,
                       total_out, max(w.n_visual), max(keep), k_out, v_out, t(cu_out), assign, member_count, src, sim)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    # routing: the oracle's arg-max on the GPU's own similarity values, bit-exact; values against fp64 cosines
    kn, vn = pu.f64(k_h), pu.f64(v_h)
    a_gpu, sim_gpu = assign.cpu().numpy(), sim.cpu().numpy()
    assign_list = []
    for b in range(w.B):
        Vb, kb = w.n_visual[b], keep[b]
        Kb = kn[cu[b]:cu[b] + Vb]
        pruned = np.setdiff1d(np.arange(Vb), kept[b])
        s = sim_gpu[cu_vis[b] + pruned][:, :kb]
        assert np.isfinite(s).all()
        want = orc.assign(Kb, kept[b], sim=s)
        assert np.array_equal(a_gpu[cu_vis[b]:cu_vis[b + 1]], want)
        cos, _ = orc.cosine_matrix(Kb, kept[b])
        assert np.abs(s - cos).max() <= 5e-5
        assign_list.append(want)
    res = orc.merge_kv(kn, vn, cu, w.n_visual, kept, orc.MEAN if mode == B_.AGG_MEAN else orc.SUM, dt, assignment_list=assign_list)
    assert np.array_equal(res["cu_seqlens_out"], cu_out)
    assert np.array_equal(member_count.cpu().numpy(), res["member_count"])
    assert np.array_equal(src.cpu().numpy(), res["src_of_dst"])
    ek = pu.assert_close(pu.f64(k_out), res["k_out"], dt, "merged key cache")
    ev = pu.assert_close(pu.f64(v_out), res["v_out"], dt, "merged value cache")
    ctx.close()
    return dict(err=(ek, ev), total_out=total_out, members=member_count.cpu().numpy(), pruned=total - total_out)


@pytest.mark.parametrize("mode", [B_.AGG_SUM, B_.AGG_MEAN])
def test_merge_kv_small_ragged(mode):
    reqs = [dict(V=300, P=17, O=4, n_dec=1, r=0.3), dict(V=129, P=1, O=4, n_dec=1, r=0.1), dict(V=517, P=40, O=4, n_dec=1, r=0.5)]
    run_case(wl.make_workload("kv", "bf16", 2, 128, 41, 16, reqs), mode)


def test_merge_kv_fp32_path():
    reqs = [dict(V=200, P=9, O=4, n_dec=1, r=0.3), dict(V=77, P=3, O=4, n_dec=1, r=0.1)]
    run_case(wl.make_workload("kv32", "fp32", 2, 32, 42, 8, reqs), B_.AGG_SUM)


def test_merge_kv_llada_shape():
    # the prefix cache of the LLaDA-8B-shaped config: 1024 visual + 64 prompt rows of width 4096, keep 10 %
    run_case(wl.config("C1"), B_.AGG_MEAN, keep_ratio=0.10)


def takes_lists(dt, payloads, B, D, total, total_out, max_visual, max_kept):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return B_.d3tom_merge_member_lists(sms, dt, payloads, B, D, total, total_out, max_visual, max_kept)


HEAVY = 32            # a kept token with this many members or more is aggregated by whole blocks
STREAM_ROWS = 4096    # from this many output rows on the streaming pipeline aggregates


@pytest.mark.parametrize("mode", [B_.AGG_SUM, B_.AGG_MEAN])
def test_merge_kv_both_caches_in_one_launch_of_the_streaming_pipeline(mode):
    res = run_case(wl.make_workload("kvl", "bf16", 2, 64, 43, 64, [dict(V=4700, P=9, O=4, n_dec=1, r=0.92)]), mode, keep_ratio=0.92)
    assert res["total_out"] >= STREAM_ROWS


# long member lists: on either side of what the list kernel keeps in registers (8192 visual tokens), and rows of 16 chunks
# with more than eight heavy (row, chunk) items per SM possible, so that more blocks than SMs walk over them
@pytest.mark.parametrize("mode", [B_.AGG_SUM, B_.AGG_MEAN])
@pytest.mark.parametrize("V,r,H,dh", [(8000, 0.01, 2, 64), (9000, 0.01, 2, 64), (17000, 0.02, 2, 64), (3000, 0.02, 32, 128)])
def test_merge_kv_both_caches_in_one_launch_with_long_member_lists(V, r, H, dh, mode):
    res = run_case(wl.make_workload("kvh", "bf16", H, dh, 43, 64, [dict(V=V, P=9, O=4, n_dec=1, r=r)]), mode, keep_ratio=r)
    assert takes_lists(torch.bfloat16, 2, 1, H * dh, V + 9, res["total_out"], V, max(1, int(r * V)))
    heavy, chunks = int((res["members"] >= HEAVY).sum()), max(1, H * dh // 256)
    assert res["total_out"] < STREAM_ROWS and heavy >= 30
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if chunks > 1:
        blocks = res["pruned"] // HEAVY * chunks // 8
        assert blocks > sms and heavy * chunks > 2 * blocks       # several items per block


def test_merge_kv_value_cache_written_over_the_key_cache():
    dev, D, V, P, k = torch.device("cuda", 0), 256, 300, 5, 40
    g = torch.Generator().manual_seed(3)
    kc, vc = (torch.randn(V + P, D, generator=g).to(torch.bfloat16).to(dev) for _ in range(2))
    i32 = lambda *a: torch.tensor(a, dtype=torch.int32, device=dev)
    kept = torch.arange(0, V, V // k, dtype=torch.int32, device=dev)[:k].contiguous()
    ctx = B_.Context(V + P, 1, 2, 128, 1, V)
    idx = [torch.empty(V + P, dtype=torch.int32, device=dev) for _ in range(3)]
    n = k + P
    outs = []
    for over in (False, True):
        a, b = kc.clone(), vc.clone()
        k_out, v_out = torch.empty(n, D, dtype=torch.bfloat16, device=dev), a[:n] if over else torch.empty(n, D, dtype=torch.bfloat16, device=dev)
        ctx.d3tom_merge_kv(B_.AGG_SUM, a, b, i32(0, V + P), i32(V), i32(0, V), kept, i32(0, k), 1, D, V + P, n, V, k, k_out, v_out,
                           i32(0, n), *idx)
        torch.cuda.synchronize()
        outs.append((k_out.clone(), v_out.clone()))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    ctx.close()


@pytest.mark.parametrize("v_over_k", [False, True])
@pytest.mark.parametrize("V,k", [(300, 40), (8000, 300), (5000, 4200)])    # aggregation without lists, with lists, and streaming
def test_merge_kv_key_cache_written_over_the_value_cache(V, k, v_over_k):
    dev, D, P = torch.device("cuda", 0), 256, 5
    assert takes_lists(torch.bfloat16, 2, 1, D, V + P, k + P, V, k) == (V != 300)
    g = torch.Generator().manual_seed(V)
    kc, vc = (torch.randn(V + P, D, generator=g).to(torch.bfloat16).to(dev) for _ in range(2))
    i32 = lambda *a: torch.tensor(a, dtype=torch.int32, device=dev)
    kept = torch.randperm(V, generator=g)[:k].sort().values.to(torch.int32).to(dev)
    ctx = B_.Context(V + P, 1, 2, 128, 1, V)
    idx = [torch.empty(V + P, dtype=torch.int32, device=dev) for _ in range(3)]
    n = k + P
    outs = []
    for over in (False, True):
        a, b = kc.clone(), vc.clone()
        # (five rows into the other cache: the overlap need not start where the cache does)
        k_out = b[5:5 + n] if over else torch.empty(n, D, dtype=torch.bfloat16, device=dev)
        v_out = a[:n] if over and v_over_k else torch.empty(n, D, dtype=torch.bfloat16, device=dev)
        ctx.d3tom_merge_kv(B_.AGG_MEAN, a, b, i32(0, V + P), i32(V), i32(0, V), kept, i32(0, k), 1, D, V + P, n, V, k, k_out, v_out,
                           i32(0, n), *idx)
        torch.cuda.synchronize()
        outs.append((k_out.clone(), v_out.clone()))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    ctx.close()


# Member lists of both aggregations (a batch builds lists, the last set, one request, does not): lists at both sides of what one
# warp adds (31, 32, 33 members, several parts of eight and of thirty-two), kept tokens without members, requests of a row or two,
# one and two payloads, nothing pruned.  Every visual token is a multiple of its kept token's unit vector, so the assignment and
# the sums over K are exact in either type; the sums over V are compared with float64.
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("H,counts", [(4, [[0, 1, 31, 32, 33, 0, 2], [64, 65], [255, 0, 0, 257, 3]]), (9, [[7] * 60, [0] * 9]),
                                      (4, [[1500, 2, 0, 40, 41, 33, 32, 31, 100]]), (5, [[0], [1], [0, 0, 0], [5, 0, 90]])])
def test_members_of_a_batch_and_of_one_request(H, counts, dtype):
    dev, dh = torch.device("cuda", 0), 64
    D, dt = H * dh, torch.float32 if dtype == "fp32" else torch.bfloat16
    rng = np.random.default_rng(len(counts) + H)
    K, owner, kept, n_vis, n_prompt = [], [], [], [], [3, 0, 9, 1][: len(counts)]
    for c in counts:
        ids = rng.permutation(np.repeat(np.arange(len(c)), np.asarray(c) + 1))
        first = np.array([np.flatnonzero(ids == i)[0] for i in range(len(c))])          # a kept token: its group's first
        order = np.argsort(first)                                                      # slots follow positions
        slot_of = np.empty(len(c), np.int64)
        slot_of[order] = np.arange(len(c))
        x = np.zeros((len(ids), D))
        x[np.arange(len(ids)), ids] = rng.integers(1, 3, len(ids))
        K.append(x)
        owner.append(slot_of[ids])
        kept.append(np.sort(first))
        n_vis.append(len(ids))
    B = len(counts)
    lens, keep = [v + p for v, p in zip(n_vis, n_prompt)], [len(k) for k in kept]
    cs = lambda a: np.concatenate([[0], np.cumsum(a)]).astype(np.int32)
    cu, cu_vis, cu_kept, cu_out = cs(lens), cs(n_vis), cs(keep), cs([n - v + k for n, v, k in zip(lens, n_vis, keep)])
    k_h = np.concatenate([np.concatenate([x, rng.integers(-3, 4, (p, D))]) for x, p in zip(K, n_prompt)])
    k_d = torch.as_tensor(k_h, device=dev).to(dt)
    v_d = torch.as_tensor(rng.standard_normal(k_h.shape), device=dev).to(dt)
    t = lambda a: torch.as_tensor(np.asarray(a, np.int32), device=dev)
    total, total_out = int(cu[-1]), int(cu_out[-1])
    ctx = B_.Context(total, B, H, dh, 1, max(n_vis))
    for second in (True, False):
        outs = [torch.full((total_out + 1, D), float("nan"), dtype=dt, device=dev) for _ in range(2)]
        ints = [torch.full((n + 1,), -9, dtype=torch.int32, device=dev) for n in (cu_vis[-1], cu_kept[-1], total_out)]
        tail = (t(cu), t(n_vis), t(cu_vis), t(np.concatenate(kept)), t(cu_kept), B, D, total, total_out, max(n_vis), max(keep))
        if second:
            ctx.d3tom_merge_kv(B_.AGG_SUM, k_d, v_d, *tail, outs[0], outs[1], t(cu_out), *ints)
        else:
            ctx.d3tom_merge(B_.AGG_SUM, k_d, *tail, outs[0], t(cu_out), *ints)
        torch.cuda.synchronize()
        assign, count, src = (x.cpu().numpy() for x in ints)
        assert assign[-1] == count[-1] == src[-1] == -9
        for b in range(B):
            s, o, lo = slice(cu_vis[b], cu_vis[b + 1]), cu_out[b], cu[b]
            assert np.array_equal(assign[s], owner[b])
            assert np.array_equal(count[cu_kept[b]:cu_kept[b + 1]], np.bincount(owner[b], minlength=keep[b]) - 1)
            assert np.array_equal(src[o:cu_out[b + 1]] - lo, np.concatenate([kept[b], np.arange(n_vis[b], lens[b])]))
            for got, x in zip(outs[: 2 if second else 1], (k_d, v_d)):
                rows = x[lo:cu[b + 1]].double().cpu().numpy()
                want = np.zeros((keep[b], D))
                np.add.at(want, owner[b], rows[: n_vis[b]])
                scale = np.zeros((keep[b], D))
                np.add.at(scale, owner[b], np.abs(rows[: n_vis[b]]))
                want, scale = np.concatenate([want, rows[n_vis[b]:]]), np.concatenate([scale, np.abs(rows[n_vis[b]:])])
                err = np.abs(got[o:cu_out[b + 1]].double().cpu().numpy() - want)
                # fp32 sums of up to 1500 terms (each rounding 2^-24 of the running sum), one rounding to the storage type
                eps = 2.0 ** -24 * 64 * scale + (2.0 ** -8 * np.abs(want) if dtype == "bf16" else 0)
                assert (err <= eps + 1e-30).all()
        assert torch.isnan(outs[0][-1]).all()
    ctx.close()


# The aggregation that finds the members itself against the one with member lists, which the same request takes beside a second
# one: the same bits.  One, two, four and eight rows per block, one to sixteen column parts (D of 37 heads: ragged chunks), lists on
# either side of what a lane holds (31, 32) and of what the whole block adds (47, 48, 127, 128, 129), several long lists in a block, one
# list with every token, nothing pruned, one token.
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("H,counts", [(37, [31, 32, 33, 0, 2, 47, 48, 127, 128, 129, 256, 300]), (37, [64, 40, 0, 5] + [4, 0] * 33),
                                      (64, [300, 60, 130] + [5] * 99), (20, [130, 40, 128, 33, 0] + [1] * 294),
                                      (16, [129, 127, 40, 33] + [0] * 828), (4, [129, 127, 40, 30, 33, 128, 32, 31] + [0, 1] * 100),
                                      (4, [1500]), (37, [2000, 0]), (4, [200, 90]), (37, [0] * 100), (4, [0])])
def test_members_found_by_scanning_give_the_bits_of_the_lists(H, counts, dtype):
    dev, D = torch.device("cuda", 0), 64 * H
    rng = np.random.default_rng(H + len(counts))
    k, P = len(counts), 5
    ids = rng.permutation(np.repeat(np.arange(k), np.asarray(counts) + 1))
    V = len(ids)
    kept = np.sort([np.flatnonzero(ids == i)[0] for i in range(k)])
    x = np.zeros((V + P, D))
    x[np.arange(V), ids] = rng.integers(1, 3, V)                   # multiples of a unit vector per kept token
    x[V:] = rng.standard_normal((P, D))
    extra = np.eye(4, D)                                           # a second request: two visual tokens, one kept, two other rows
    t = lambda a: torch.as_tensor(np.asarray(a, np.int32), device=dev)
    k_d = torch.as_tensor(np.concatenate([x, extra]), device=dev).to(dtype)
    v_d = torch.as_tensor(rng.standard_normal((V + P + 4, D)), device=dev).to(dtype)
    ctx = B_.Context(V + P + 4, 2, H, 64, 1, max(V, 2))
    for payloads in (1, 2):
        got = []
        single_lists = takes_lists(dtype, payloads, 1, D, V + P, k + P, V, k)
        assert not single_lists or payloads == 2 or dtype == torch.float32
        for B in (1, 2):
            n, m, n_vis, n_kept = V + P + (4 if B == 2 else 0), k + P + (3 if B == 2 else 0), [V, 2][:B], [k, 1][:B]
            cs = lambda a: t(np.concatenate([[0], np.cumsum(a)]))
            cu, cu_out = cs([V + P, 4][:B]), cs([k + P, 3][:B])
            assert takes_lists(dtype, payloads, B, D, n, m, max(n_vis), max(n_kept)) == (B == 2 or single_lists)
            outs = [torch.full((m + 1, D), float("nan"), dtype=dtype, device=dev) for _ in range(2)]
            ints = [torch.full((c + 1,), -9, dtype=torch.int32, device=dev) for c in (sum(n_vis), sum(n_kept), m)]
            tail = (cu, t(n_vis), cs(n_vis), t(np.concatenate([kept, [0]])[: sum(n_kept)]), cs(n_kept), B, D, n, m, max(n_vis), max(n_kept))
            if payloads == 2:
                ctx.d3tom_merge_kv(B_.AGG_MEAN, k_d[:n], v_d[:n], *tail, *outs, cu_out, *ints)
            else:
                ctx.d3tom_merge(B_.AGG_SUM, k_d[:n], *tail, outs[0], cu_out, *ints)
            torch.cuda.synchronize()
            assert all(i[-1].item() == -9 for i in ints) and all(torch.isnan(o[-1]).all() for o in outs)
            got.append([o[: k + P] for o in outs[:payloads]] + [i[:c] for i, c in zip(ints, (V, k, k + P))])
        assert all(torch.equal(a, b) for a, b in zip(*got))
        order = np.argsort([np.flatnonzero(ids == i)[0] for i in range(k)])
        assert np.array_equal(got[0][-2].cpu().numpy(), np.asarray(counts)[order])
    ctx.close()
