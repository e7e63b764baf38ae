"""d3tom_linear and d3tom_ffn (Algorithm 1, FFN_l: the rest of a post-merge block) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import d3tom_oracle as orc
from paper_2511_12280_b200 import binding as B_
from paper_2511_12280_b200 import workload as wl

import parity_util as pu

pytestmark = pytest.mark.gpu


def make_ctx(rows, dtype):
    # the dense layers use no scratch of the context; head geometry only has to be valid
    return B_.Context(max(rows, 1), 1, 2, 64 if dtype == "bf16" else 8, 1, 1)


def run_linear(rows, K, N, dtype, residual, in_place=False, seed=0):
    dev = torch.device("cuda", 0)
    t = wl.block_inputs(seed, rows, max(K, N), 8, dtype)
    x = t["x"][:, :K].contiguous()
    w = t["w_o"][:N, :K].contiguous() * 4           # keeps outputs O(1) at small K
    res = t["residual"][:, :N].contiguous() if residual else None
    ctx = make_ctx(rows, dtype)
    xd, wd = x.to(dev), w.to(dev)
    if in_place:
        out = res.to(dev); resd = out
    else:
        out = torch.full((rows, N), float("nan"), dtype=x.dtype, device=dev)
        resd = res.to(dev) if residual else None
    ctx.d3tom_linear(xd, wd, resd, rows, K, N, out)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    want = orc.linear(pu.f64(x), pu.f64(w), pu.f64(res) if residual else None, dtype)
    pu.assert_close(pu.f64(out), want, dtype, "linear %dx%dx%d" % (rows, K, N))
    ctx.close()


@pytest.mark.parametrize("N", [128, 384, 512, 768])      # tile widths 128, 192 / 128, 256, 256 / 192
def test_linear_bf16_every_tile_width_ragged_rows(N):
    run_linear(300, 256, N, "bf16", residual=True)


def test_linear_bf16_without_residual_and_in_place():
    run_linear(300, 192, 256, "bf16", residual=False)
    run_linear(129, 320, 256, "bf16", residual=True, in_place=True)
    run_linear(1, 64, 128, "bf16", residual=True)


def test_linear_and_ffn_bf16_long_k_few_tiles_cut_into_k_slices():
    # six tiles for 148 SMs and 64 k-blocks: the tiles of the (only, incomplete) round are cut into K slices whose
    # partial sums meet in the workspace; the same for the gate/up pass of the feed-forward network
    run_linear(300, 4096, 512, "bf16", residual=True, seed=3)
    run_ffn(300, 4096, 256, "bf16", seed=4)


def test_linear_and_ffn_bf16_many_single_cta_tiles_at_a_short_k():
    # 1500 rows x 12288 columns: four rounds of 128-row tiles over the SMs, for the linear layer and for the gate/up pass; the
    # last row tile has 92 of 128 rows.  1216 rows: 9.5 row tiles
    for rows, K in ((1500, 64), (1500, 128), (1216, 64), (1216, 128)):
        assert pair_width(rows, 12288, K) == 0
        run_linear(rows, K, 12288, "bf16", residual=K == 64, seed=rows + K)
    assert pair_width(1500, 12288, 128, gate_up=True) == 0
    run_ffn(1500, 128, 6144, "bf16", seed=7)


def run_proj(rows, H, dh, seed=0):
    dev = torch.device("cuda", 0)
    D = H * dh
    t = wl.block_inputs(seed, rows, D, 8, "bf16")
    x = t["x"][:, :D].contiguous()
    g = torch.Generator().manual_seed(seed + 1)
    w = (torch.randn(3 * D, D, generator=g) * (4.0 / D ** 0.5)).to(torch.bfloat16)
    ctx = B_.Context(max(rows, 1), 1, H, dh, 1, 1)
    q, k, v = (torch.full((rows, D), float("nan"), dtype=torch.bfloat16, device=dev) for _ in range(3))
    ctx.d3tom_proj_qkv(x.to(dev), w.to(dev), rows, D, q, k, v)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    want = orc.proj_qkv(pu.f64(x), pu.f64(w), H, "bf16")
    for got, ref, name in zip((q, k, v), want, "qkv"):
        pu.assert_close(pu.f64(got), ref.reshape(rows, D), "bf16", "%s of the projection, %d rows, D = %d" % (name, rows, D))
    ctx.close()


def test_dense_layers_on_cta_pairs():
    # 256 x 256 tiles computed by two CTAs (each holds its 128 rows of x and half of the weight tile): a ragged last
    # row tile whose second CTA has no rows at all, whole tiles, more tiles than pairs (several rounds); the output
    # projection with and without residual and the gated feed-forward network (gate rows in one CTA, up rows in the other)
    B_.d3tom_set_pair_tiles(256)
    try:
        run_proj(64, 4, 128)
        run_proj(300, 4, 128, seed=1)
        run_proj(1216, 8, 128, seed=2)
        run_proj(5000, 2, 128, seed=3)
        run_linear(300, 256, 512, "bf16", residual=True)
        run_linear(129, 320, 256, "bf16", residual=True, in_place=True)
        run_linear(2500, 192, 768, "bf16", residual=False)
        run_ffn(300, 256, 512, "bf16", seed=5)
        run_ffn(2300, 128, 384, "bf16", seed=6)
    finally:
        B_.d3tom_set_pair_tiles(-1)


def test_long_dense_layers_take_cta_pairs_by_default():
    # from about two thousand rows on the library picks the pair tiles itself
    run_proj(2304, 4, 128, seed=7)
    run_linear(2100, 256, 512, "bf16", residual=True, seed=8)
    run_ffn(2100, 256, 256, "bf16", seed=9)


def pair_width(rows, n_cols, K, gate_up=False):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return B_.d3tom_pair_tile_width(sms, sms // 2, rows, n_cols, K, gate_up)


# nine 256-row tiles on 74 pairs: eight column tiles fill one round, so the width follows the number of columns: 128, 160,
# 160 with an overhang, 192, 192 with an overhang, 224, 224 with an overhang, 256; K of one, three, four and seventeen
# 64-deep blocks (the narrower tiles take two blocks per ring stage)
@pytest.mark.parametrize("N,K,width", [(1024, 192, 128), (1280, 64, 160), (1152, 1088, 160), (1536, 256, 192), (1408, 192, 192),
                                       (1792, 192, 224), (1664, 256, 224), (2048, 192, 256)])
def test_pair_tiles_of_every_width(N, K, width):
    assert pair_width(2100, N, K) == width
    run_linear(2100, K, N, "bf16", residual=True, seed=N)


# rows, H (heads of 128), width: 192 straddles q | k and k | v; 256 and 128 columns of 1152, which 256 does not divide; a
# layer below 2048 rows
@pytest.mark.parametrize("rows,H,width", [(2100, 4, 192), (3333, 3, 256), (4000, 3, 128), (400, 13, 160)])
def test_pair_tiles_projection(rows, H, width):
    assert pair_width(rows, 3 * H * 128, H * 128) == width
    run_proj(rows, H, 128, seed=20 + H)


# halves of 80 gate and 80 up rows; of 112; 160 in two rounds, the last tile hanging over the edge of both matrices; a layer
# below 2048 rows
@pytest.mark.parametrize("rows,D,m,width", [(2100, 128, 640, 160), (2100, 256, 896, 224), (2100, 128, 1152, 160), (400, 2048, 1920, 128)])
def test_pair_tiles_gate_up(rows, D, m, width):
    assert pair_width(rows, 2 * m, D, gate_up=True) == width
    run_ffn(rows, D, m, "bf16", seed=23)


def test_pair_tiles_below_2048_rows_with_an_overhang():
    assert pair_width(1930, 4736, 512) == 192          # 4736 = 24 tiles of 192 and one of 128
    run_linear(1930, 512, 4736, "bf16", residual=True, seed=26)


# single-CTA tiles from 2048 rows on: one round of K slices, and a width that 256 does not divide at a short K
@pytest.mark.parametrize("rows,K,N", [(2100, 16384, 128), (2048, 8192, 384), (2100, 128, 640), (2600, 512, 384)])
def test_long_layers_that_keep_single_cta_tiles(rows, K, N):
    assert pair_width(rows, N, K) == 0
    run_linear(rows, K, N, "bf16", residual=True, seed=K)


# between 513 and 2047 rows, and single-CTA tiles from 2048 rows on, by the fitted costs: each width of either kind, ragged rows
@pytest.mark.parametrize("rows,K,N,width", [(513, 1024, 384, 0), (769, 1024, 2816, 160), (700, 1024, 3968, 192), (513, 2048, 4736, 224),
                                            (2047, 1024, 768, 0), (2049, 1024, 384, 0), (2600, 1024, 1024, 192)])
def test_tile_shapes_by_cost(rows, K, N, width):
    assert pair_width(rows, N, K) == width
    run_linear(rows, K, N, "bf16", residual=True, seed=rows)


# calls of up to 127 rows store row by row, longer ones 64 bytes of eight rows at a time
@pytest.mark.parametrize("rows", [1, 31, 127, 128, 129])
def test_dense_layers_at_the_ends_of_the_short_calls(rows):
    run_proj(rows, 2, 128, seed=rows)
    run_linear(rows, 128, 256, "bf16", residual=False, seed=rows)
    run_linear(rows, 128, 256, "bf16", residual=True, in_place=True, seed=rows)
    run_ffn(rows, 128, 256, "bf16", seed=rows)


def test_linear_fp32_odd_sizes():
    run_linear(70, 50, 45, "fp32", residual=True)
    run_linear(33, 7, 3, "fp32", residual=False)


def run_ffn(rows, D, m, dtype, residual=True, seed=1, sample_rows=None):
    dev = torch.device("cuda", 0)
    t = wl.block_inputs(seed, rows, D, m, dtype)
    scale = 4.0 if D < 1024 else 1.0                  # keeps gate pre-activations O(1) at small D
    x, wgu, wdn = t["x"], t["w_gate_up"] * scale, t["w_down"] * scale
    res = t["residual"] if residual else None
    ctx = make_ctx(rows, dtype)
    act = torch.full((rows, m), float("nan"), dtype=x.dtype, device=dev)
    out = torch.full((rows, D), float("nan"), dtype=x.dtype, device=dev)
    ctx.d3tom_ffn(x.to(dev), wgu.to(dev), wdn.to(dev), res.to(dev) if residual else None, rows, D, m, act, out)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    sel = np.arange(rows) if sample_rows is None else np.asarray(sample_rows)
    xs, rs = pu.f64(x)[sel], (pu.f64(res)[sel] if residual else None)
    want_out, want_act = orc.ffn(xs, pu.f64(wgu), pu.f64(wdn), rs, dtype)
    act_g, out_g = pu.f64(act)[sel], pu.f64(out)[sel]
    pu.assert_close(act_g, want_act, dtype, "ffn activation")
    # second product fed the GPU's own activation (a bf16 rounding flip in act cannot cascade), then free-running
    pu.assert_close(out_g, orc.linear(act_g, pu.f64(wdn), rs, dtype), dtype, "ffn output, teacher-forced")
    pu.assert_close(out_g, want_out, dtype, "ffn output")
    if sample_rows is not None:
        assert torch.isfinite(out.float()).all() and torch.isfinite(act.float()).all()
    ctx.close()


def test_ffn_bf16_ragged_rows_several_tiles():
    run_ffn(300, 256, 384, "bf16")
    run_ffn(127, 128, 128, "bf16", residual=False)


def test_ffn_fp32_odd_sizes():
    run_ffn(37, 24, 20, "fp32")


def test_ffn_bf16_llada_shape_sampled_rows():
    # rows of the shortened sequence of the 4096-visual-token configuration, d = 4096, m = 12288;
    # the oracle computes a sample of rows (the layers act row by row)
    run_ffn(1216, 4096, 12288, "bf16", sample_rows=[0, 1, 127, 128, 640, 1151, 1152, 1215])


def test_linear_bf16_llada_shape_sampled_rows():
    dev = torch.device("cuda", 0)
    rows, D = 1216, 4096
    t = wl.block_inputs(2, rows, D, 8, "bf16")
    ctx = make_ctx(rows, "bf16")
    out = torch.full((rows, D), float("nan"), dtype=torch.bfloat16, device=dev)
    ctx.d3tom_linear(t["x"].to(dev), t["w_o"].to(dev), t["residual"].to(dev), rows, D, D, out)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0 and torch.isfinite(out.float()).all()
    sel = np.array([0, 127, 128, 1000, 1215])
    want = orc.linear(pu.f64(t["x"])[sel], pu.f64(t["w_o"]), pu.f64(t["residual"])[sel], "bf16")
    pu.assert_close(pu.f64(out)[sel], want, "bf16", "output projection")
    ctx.close()


def test_unsupported_shapes_and_bad_arguments_are_refused_on_the_host():
    dev = torch.device("cuda", 0)
    ctx = make_ctx(64, "bf16")
    z = lambda *s: torch.zeros(*s, dtype=torch.bfloat16, device=dev)
    lib = B_.load()
    with pytest.raises(RuntimeError, match="UNSUPPORTED|unsupported"):
        ctx.d3tom_linear(z(64, 64), z(100, 64), None, 64, 64, 100, z(64, 100))       # N not a multiple of 128
    with pytest.raises(RuntimeError, match="UNSUPPORTED|unsupported"):
        ctx.d3tom_linear(z(64, 40), z(128, 40), None, 64, 40, 128, z(64, 128))        # K not a multiple of 64
    with pytest.raises(RuntimeError, match="UNSUPPORTED|unsupported"):
        ctx.d3tom_ffn(z(64, 128), z(200, 128), z(128, 100), None, 64, 128, 100, z(64, 100), z(64, 128))
    x = z(64, 128)
    with pytest.raises(RuntimeError, match="INVALID|invalid"):
        ctx.d3tom_linear(x, z(128, 128), None, 64, 128, 128, x)                       # out must not be x
    ctx.d3tom_linear(x, z(128, 128), None, 0, 128, 128, z(64, 128))                  # no rows: nothing to do
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    ctx.close()


def test_whole_post_merge_block_after_a_merge_step():
    # merge-layer step, then one LLaDA-shaped block (attention, output projection, gated FFN, two residuals) on the
    # shortened ragged batch; every stage is checked against the oracle fed with the GPU's previous stage
    w = wl.make_workload("blk", "bf16", 2, 128, 41, 16, [dict(V=300, P=17, O=24, n_dec=5, r=0.3),
                                                          dict(V=200, P=9, O=8, n_dec=2, r=0.5)], post_layers=1)
    step = pu.make_step(w, sim_debug=False)
    dev = step.dev
    D, m = step.D, 384
    t = wl.block_inputs(7, 8, D, m, "bf16")
    w_o, w_gu, w_dn = t["w_o"] * 2, t["w_gate_up"] * 4, t["w_down"] * 4
    q, k, v = w.q_for().to(dev), w.k.to(dev), w.v.to(dev)
    step.attn_importance(q, k, v); step.select(); step.merge()
    x = step.hidden_out
    y = step.post_block(0, x, w.w_post[0].to(dev), w_o.to(dev), w_gu.to(dev), w_dn.to(dev))
    torch.cuda.synchronize()
    assert step.ctx.device_status() == 0
    n = step.total_out
    xg = pu.f64(x)[:n]
    attn = orc.post_layer(xg, pu.f64(w.w_post[0]), step.cu_out_h, w.H, "bf16").reshape(n, D)
    x1 = orc.linear(attn, pu.f64(w_o), xg, "bf16")
    pu.assert_close(pu.f64(step.block_x1)[:n], x1, "bf16", "x + attn W_o")
    x1g = pu.f64(step.block_x1)[:n]
    want, _ = orc.ffn(x1g, pu.f64(w_gu), pu.f64(w_dn), x1g, "bf16")
    pu.assert_close(pu.f64(y)[:n], want, "bf16", "block output")
    step.ctx.close()
