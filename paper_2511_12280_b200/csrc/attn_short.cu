// The attention kernel of attn_tc.cu for calls so short that single 128-row query tiles do not fill the SMs (Sec. 3.2.1, A =
// softmax(QK^T * scale); the layers after l* on a short sequence), bf16, head_dim 64 or 128.
//
// One CTA = (request, head, 128 query rows).  With one query tile there is no second one to work while S, P and O of the first
// wait for each other, so the chain of a key tile (softmax, PV, the next QK^T, two barrier hops, about 3000 cycles) is all there
// is.  Tensor memory has the other tile's S columns to spare: key tile j uses S buffer j & 1, QK^T runs two key tiles ahead, and
// the chain is the softmax alone (about 1600 cycles).  The arithmetic is that of attn_tc.cu (speculative exponentials, lazy
// rescaling, P in two halves, one row per thread): the same bits.
// Measured, attn_tc.cu / here (us): 64 rows x 32 heads x 128 6.2 / 5.2, 512 x 32 x 128 10.5 / 8.6, 1100 x 16 x 128 21.2 / 14.1,
// 319 x 16 x 64 8.2 / 6.6, 723 x 16 x 64 12.1 / 9.8, 1000 x 8 x 64 14.5 / 11.7, eight requests of 200 x 8 x 64 8.7 / 5.8; with
// the importance map 723 x 16 x 64 21.0 / 19.0, 360 x 32 x 128 17.1 / 15.4.
//
//   warps 0-3  softmax and epilogue (one row per thread = one TMEM lane)
//   warp  4    TMA producer: Q, rings of three K and three V tiles
//   warp  5    one thread issues every tcgen05.mma: PV_j, then QK^T_(j+2) into the buffer PV_j has just read
// S_j complete says that QK^T_j has read its K tile and, issued before it, PV_(j-2) its V tile and P: the loader waits for that and
// requests K_(j+3) and V_(j+1).  Every wait is bounded.
#include "common.cuh"
#include "ptx.cuh"

namespace {

constexpr int kTile = 128;
constexpr int kThreads = 192;
constexpr int kRing = 3;
constexpr float kRescaleThreshold = 8.0f;

template <int DH> struct ShortSmem {
  static constexpr int kTileBytes = kTile * DH * 2;
  static constexpr int kBytes = (1 + 2 * kRing) * kTileBytes + 1024 + 256;
};

using ptx::max3;
using ptx::pack_bf16x2;
using ptx::tmem_st16;

// kImp: the launch also feeds the importance map; kShort: requests of at most 48 rows (how the output is stored)
template <int DH, bool kImp, bool kShort>
__global__ void __launch_bounds__(kThreads, 1)
attn_short_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                  const __grid_constant__ CUtensorMap tmap_v, AttnArgs a) {
  constexpr int kTileBytes = ShortSmem<DH>::kTileBytes;
  constexpr int kHalfBytes = kTile * 128;               // one 64-column sub-tile: 128 rows x 128 bytes
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* q_s = smem;
  uint8_t* k_s = q_s + kTileBytes;
  uint8_t* v_s = k_s + kRing * kTileBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(v_s + kRing * kTileBytes);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;                          // [3]
  uint64_t* v_full = bars + 4;                          // [3]
  uint64_t* s_full = bars + 7;                          // [4] (index j & 3: QK^T_(j+4) needs K_(j+4), which the loader requests
                                                        //     after it has seen S_(j+1), so no one who waits for S_j can miss it)
  uint64_t* p_lo = bars + 11;                           // [2]  P columns of keys 0..63 written (and O consistent)
  uint64_t* p_hi = bars + 13;                           // [2]  P columns of keys 64..127 written
  uint64_t* pv_last = bars + 15;                        // the last PV but one
  uint64_t* o_final = bars + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 17);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = ptx::uniform_warp(), lane = threadIdx.x & 31;
  // barriers and tensor memory first (on-chip only), then wait for the kernels before this one
  if (threadIdx.x == 0) {
    ptx::mbar_init(q_full, 1); ptx::mbar_init(pv_last, 1); ptx::mbar_init(o_final, 1);
    for (int i = 0; i < kRing; ++i) { ptx::mbar_init(&k_full[i], 1); ptx::mbar_init(&v_full[i], 1); }
    for (int i = 0; i < 4; ++i) ptx::mbar_init(&s_full[i], 1);
    for (int i = 0; i < 2; ++i) { ptx::mbar_init(&p_lo[i], 4); ptx::mbar_init(&p_hi[i], 4); }
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) { ptx::tmem_alloc(tmem_slot, 512); ptx::tmem_relinquish(); }
  ptx::tc_fence_before_sync();
  __syncthreads();                                      // (the next kernel's blocks may come once tensor memory is ours)
  ptx::tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  grid_dependency_enter();
  // heads fastest, the last query tiles (the response rows; decider rows do extra work) first
  const int per_req = a.H * a.nqb;                      // (nqb: 128-row tiles of the longest request)
  const int b = (int)blockIdx.x / per_req, lin = (int)blockIdx.x - b * per_req;
  const int h = lin % a.H, q0 = (a.nqb - 1 - lin / a.H) * kTile;
  const int lo = a.cu_seqlens[b], n = a.cu_seqlens[b + 1] - lo;
  const int n_kv = q0 < n ? (n + kTile - 1) / kTile : 0;    // 0: the request does not reach this tile
  constexpr uint32_t kColO = 256;

  if (n_kv == 0) {
    // nothing to do but to give tensor memory back
  } else if (warp == 4) {
    // ------------------------------------------------------------ TMA producer
    if (ptx::elect_one()) {
      ptx::prefetch_tensormap(&tmap_q); ptx::prefetch_tensormap(&tmap_k); ptx::prefetch_tensormap(&tmap_v);
      auto load_tile = [&](uint8_t* dst, const CUtensorMap* tm, uint64_t* bar, int row) {
        ptx::mbar_arrive_expect_tx(bar, kTileBytes);
        for (int hf = 0; hf < DH / 64; ++hf) ptx::tma_load_2d(dst + hf * kHalfBytes, tm, bar, h * DH + hf * 64, row);
      };
      auto load_k = [&](int t) { load_tile(k_s + t % kRing * kTileBytes, &tmap_k, &k_full[t % kRing], lo + t * kTile); };
      auto load_v = [&](int t) { load_tile(v_s + t % kRing * kTileBytes, &tmap_v, &v_full[t % kRing], lo + t * kTile); };
      load_tile(q_s, &tmap_q, q_full, lo + q0);
      for (int t = 0; t < kRing && t < n_kv; ++t) { load_k(t); load_v(t); }
      for (int j = 0; j + 1 < n_kv; ++j) {
        if (!ptx::mbar_wait(&s_full[j & 3], (j >> 2) & 1, abort_flag, a.dev_status)) break;
        if (j + 1 >= kRing) load_v(j + 1);              // (V_(j-2), the slot's last tile, has been read)
        if (j + kRing < n_kv) load_k(j + kRing);
      }
    }
  } else if (warp == 5) {
    // ------------------------------------------------------------ MMA issuer
    if (ptx::elect_one()) {
      constexpr uint32_t idesc_qk = ptx::idesc_bf16_f32(kTile, kTile, 0, 0);   // S = Q K^T, both K-major
      constexpr uint32_t idesc_pv = ptx::idesc_bf16_f32(kTile, DH, 0, 1);      // O += P V, V is MN-major
      const ptx::SmemDesc q_desc = ptx::smem_desc_kmajor_sw128(ptx::smem_u32(q_s));
      const ptx::SmemDesc k_desc0 = ptx::smem_desc_kmajor_sw128(ptx::smem_u32(k_s));
      const ptx::SmemDesc v_desc0 = ptx::smem_desc_mnmajor_sw128(ptx::smem_u32(v_s), kHalfBytes);
      auto issue_qk = [&](int t) {
        const ptx::SmemDesc kd = ptx::smem_desc_advance(k_desc0, t % kRing * kTileBytes);
#pragma unroll
        for (int kk = 0; kk < DH / 16; ++kk) {
          const uint32_t off = (kk / 4) * kHalfBytes + (kk % 4) * 32;
          ptx::mma_ss(tmem + (uint32_t)(t & 1) * 128u, ptx::smem_desc_advance(q_desc, off), ptx::smem_desc_advance(kd, off), idesc_qk,
                      kk > 0 ? 1u : 0u);
        }
        ptx::mma_commit(&s_full[t & 3]);
      };
      auto issue_pv_half = [&](int t, int half, bool accumulate) {
        const ptx::SmemDesc vd = ptx::smem_desc_advance(v_desc0, t % kRing * kTileBytes + half * 4 * 2048);
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4)                           // 16 keys per instruction
          ptx::mma_ts(tmem + kColO, tmem + (uint32_t)(t & 1) * 128u + (half * 4 + k4) * 8, ptx::smem_desc_advance(vd, k4 * 2048),
                      idesc_pv, (accumulate || half > 0 || k4 > 0) ? 1u : 0u);
      };
      bool ok = ptx::mbar_wait(q_full, 0, abort_flag, a.dev_status);
      for (int t = 0; t < 2 && t < n_kv && ok; ++t) {
        ok = ptx::mbar_wait(&k_full[t], 0, abort_flag, a.dev_status);
        if (!ok) break;
        ptx::tc_fence_after_sync();
        issue_qk(t);
      }
      for (int j = 0; j < n_kv && ok; ++j) {                     // (the softmax warps have seen V_j and K_(j+2) land)
        ok = ptx::mbar_wait(&p_lo[j & 1], (j >> 1) & 1, abort_flag, a.dev_status);
        if (!ok) break;
        ptx::tc_fence_after_sync();
        issue_pv_half(j, 0, j > 0);
        ok = ptx::mbar_wait(&p_hi[j & 1], (j >> 1) & 1, abort_flag, a.dev_status);
        if (!ok) break;
        ptx::tc_fence_after_sync();
        issue_pv_half(j, 1, true);
        if (j + 2 < n_kv) issue_qk(j + 2);
        else ptx::mma_commit(j + 1 < n_kv ? pv_last : o_final);
      }
    }
  } else {
    // ------------------------------------------------------------ softmax + epilogue
    const int row = warp * 32 + lane;              // row in the tile == TMEM lane
    const int q_row = q0 + row;                    // row in the request
    const bool valid_row = q_row < n;
    const uint32_t lane_addr = (uint32_t)(warp * 32) << 16;
    const uint32_t t_o = tmem + lane_addr + kColO;
    // is this row a decider of the request?  (deciders are response rows: a row below the visual count skips the look-up)
    int dec_slot = -1, n_vis = 0;
    if (kImp) n_vis = a.n_visual[b];
    if (kImp && valid_row && q_row >= n_vis) {
      int l = a.cu_deciders[b], r = a.cu_deciders[b + 1];
      while (l < r) {
        const int mid = (l + r) >> 1, pos = a.decider_pos[mid];
        if (pos == q_row) { dec_slot = mid; break; }
        if (pos < q_row) l = mid + 1; else r = mid;
      }
    }
    float* score_row = dec_slot >= 0 ? a.score_scratch + ((size_t)h * a.max_deciders + dec_slot) * a.vis_stride : nullptr;

    float m_used = -INFINITY;
    float2 l2 = make_float2(0.f, 0.f);             // the row sum, kept as two partial sums
    const float c = a.scale_log2;
    const float2 c2 = make_float2(c, c);
    bool ok = true;
    for (int j = 0; j < n_kv; ++j) {
      const uint32_t t_s = tmem + lane_addr + (uint32_t)(j & 1) * 128u;
      ok = __all_sync(0xffffffffu, ptx::mbar_wait(&s_full[j & 3], (j >> 2) & 1, abort_flag, a.dev_status));
      if (!ok) break;
      ptx::tc_fence_after_sync();
      // ---- the whole score row of this tile: 128 fp32 values, one TMEM lane
      uint32_t sr[kTile];
      ptx::tmem_ld32(t_s, sr);
      ptx::tmem_ld32(t_s + 32, sr + 32);
      ptx::tmem_ld32(t_s + 64, sr + 64);
      ptx::tmem_ld32(t_s + 96, sr + 96);
      ptx::tmem_wait_ld();
      const int n_valid = n - j * kTile;                  // keys of this tile that belong to the request
      if (n_valid < kTile) {                              // ragged last tile: keys past the end score -inf
#pragma unroll
        for (int e = 0; e < kTile; ++e) if (e >= n_valid) sr[e] = 0xff800000u;
      }
      // ---- p = exp2(s*c - m) in four chunks of 32 keys.  The first two chunks are computed
      //      against the maximum known BEFORE this tile, while the tile's own maximum is still being
      //      reduced: any reference within 2^8 of the true maximum is exact after the final division,
      //      so the result stands unless the maximum grew by more than that (then it is redone).
      uint32_t pk[2][16];
      float2 l_tile = make_float2(0.f, 0.f);
      auto exp_chunk = [&](int ch, float m_ref, uint32_t (&out)[16], float2& lsum) {
        const float2 nm2 = make_float2(-m_ref, -m_ref);
        float2 t2[16];
#pragma unroll
        for (int e = 0; e < 16; ++e)
          t2[e] = __ffma2_rn(make_float2(__uint_as_float(sr[ch * 32 + 2 * e]), __uint_as_float(sr[ch * 32 + 2 * e + 1])),
                             c2, nm2);
#pragma unroll
        for (int e = 0; e < 16; ++e) { t2[e].x = ptx::ex2(t2[e].x); t2[e].y = ptx::ex2(t2[e].y); }
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          out[e] = pack_bf16x2(t2[e].x, t2[e].y);
          lsum = __fadd2_rn(lsum, t2[e]);
        }
      };
      exp_chunk(0, m_used, pk[0], l_tile);                // (first tile: against -inf, always redone below)
      exp_chunk(1, m_used, pk[1], l_tile);
      // ---- row maximum: 8 independent chains of three-input maxima
      float mx[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) mx[t] = fmaxf(__uint_as_float(sr[2 * t]), __uint_as_float(sr[2 * t + 1]));
#pragma unroll
      for (int e = 16; e < kTile; e += 16)
#pragma unroll
        for (int t = 0; t < 8; ++t)
          mx[t] = max3(mx[t], __uint_as_float(sr[e + 2 * t]), __uint_as_float(sr[e + 2 * t + 1]));
      const float mxa = max3(max3(mx[0], mx[1], mx[2]), max3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7]));
      const float m_new = fmaxf(m_used, mxa * c);
      const bool need = (m_new - m_used) > kRescaleThreshold;   // first tile: inf > threshold
      if (__any_sync(0xffffffffu, need)) {
        const float alpha = need ? exp2f(m_used - m_new) : 1.f;
        if (j > 0) {
          // S_j being there says that PV_(j-2) has completed: O is touched once PV_(j-1) has, which the commit behind
          // QK^T_(j+1) says, or the one behind the last PV but one
          ok = __all_sync(0xffffffffu, j + 1 < n_kv ? ptx::mbar_wait(&s_full[(j + 1) & 3], ((j + 1) >> 2) & 1, abort_flag, a.dev_status)
                                                    : ptx::mbar_wait(pv_last, 0, abort_flag, a.dev_status));
          if (!ok) break;
          ptx::tc_fence_after_sync();
#pragma unroll 1
          for (int c0 = 0; c0 < DH; c0 += 32) {
            uint32_t r[32];
            ptx::tmem_ld32(t_o + c0, r);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
            ptx::tmem_st32(t_o + c0, r);
          }
          ptx::tmem_wait_st();
        }
        l2.x *= alpha; l2.y *= alpha;
        if (need) m_used = m_new;
        l_tile = make_float2(0.f, 0.f);                   // the speculative half is redone against the new maximum
        exp_chunk(0, m_used, pk[0], l_tile);
        exp_chunk(1, m_used, pk[1], l_tile);
      }
      // ---- the bf16 P tile goes into the first 64 columns of the S buffer; the tensor pipe is told after each half
      tmem_st16(t_s, pk[0]);                             // keys 32*ch .. +31 -> P columns 16*ch .. +15
      tmem_st16(t_s + 16, pk[1]);
      exp_chunk(2, m_used, pk[0], l_tile);
      ptx::tmem_wait_st();
      ptx::tc_fence_before_sync();
      // V_j and K_(j+2) must have landed before the tensor pipe is sent on (it does not check)
      ok = __all_sync(0xffffffffu, ptx::mbar_wait(&v_full[j % kRing], (j / kRing) & 1, abort_flag, a.dev_status));
      if (ok && j + 2 < n_kv)
        ok = __all_sync(0xffffffffu, ptx::mbar_wait(&k_full[(j + 2) % kRing], ((j + 2) / kRing) & 1, abort_flag, a.dev_status));
      if (!ok) break;
      if (lane == 0) ptx::mbar_arrive(&p_lo[j & 1]);
      tmem_st16(t_s + 32, pk[0]);
      exp_chunk(3, m_used, pk[1], l_tile);
      tmem_st16(t_s + 48, pk[1]);
      l2 = __fadd2_rn(l2, l_tile);
      ptx::tmem_wait_st();
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&p_hi[j & 1]);
      // Decider rows: the raw scores over the visual keys go out AFTER P has been announced: the stores (one row per
      // lane, 512 bytes each, uncoalesced) then run while the tensor pipe works on this tile instead of delaying it
      // (the score registers stay live until the next key tile's load).
      if (kImp && score_row != nullptr && j * kTile < n_vis) {
        const int key0 = j * kTile;
#pragma unroll
        for (int e = 0; e < kTile; e += 4) {
          if (key0 + e + 3 < n_vis) {
            *reinterpret_cast<float4*>(score_row + key0 + e) =
                make_float4(__uint_as_float(sr[e]), __uint_as_float(sr[e + 1]), __uint_as_float(sr[e + 2]),
                            __uint_as_float(sr[e + 3]));
          } else {
#pragma unroll
            for (int t = 0; t < 4; ++t) if (key0 + e + t < n_vis) score_row[key0 + e + t] = __uint_as_float(sr[e + t]);
          }
        }
      }
    }
    // ---- epilogue: O / l -> bf16 -> global
    if (ok) ok = __all_sync(0xffffffffu, ptx::mbar_wait(o_final, 0, abort_flag, a.dev_status));
    ptx::tc_fence_after_sync();
    if (ok) {
      const float l_sum = l2.x + l2.y;
      const float inv_l = 1.f / l_sum;
      const int warp_row = q_row - lane;           // this warp's 32 rows
      __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(a.out) + ((size_t)(lo + warp_row) * a.H + h) * DH;
#pragma unroll 1
      for (int c0 = 0; c0 < DH; c0 += 32) {
        uint32_t r[32], w[16];
        ptx::tmem_ld32(t_o + c0, r);
        ptx::tmem_wait_ld();
#pragma unroll
        for (int t = 0; t < 16; ++t)
          w[t] = pack_bf16x2(__uint_as_float(r[2 * t]) * inv_l, __uint_as_float(r[2 * t + 1]) * inv_l);
        ptx::store_rows_64b<kShort>(dst + c0, (size_t)a.H * DH * 2, n - warp_row, w);
      }
      if (kImp && dec_slot >= 0) a.lse_scratch[(size_t)h * a.max_deciders + dec_slot] = make_float2(m_used, l_sum);
    }
    ptx::tc_fence_before_sync();
  }
  __syncthreads();
  if (warp == 0) ptx::tmem_dealloc(tmem, 512);
}

template <int DH>
int launch(d3tom_ctx* ctx, const AttnArgs& a, cudaStream_t s) {
  CUtensorMap tq, tk, tv;
  const uint64_t rows = (uint64_t)a.total_tokens, cols = (uint64_t)a.H * DH;
  int r = make_tmap_bf16_2d(&tq, a.q, rows, cols, cols, kTile);
  if (r == 0) r = make_tmap_bf16_2d(&tk, a.k, rows, cols, cols, kTile);
  if (r == 0) r = make_tmap_bf16_2d(&tv, a.v, rows, cols, cols, kTile);
  if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
  const bool short_call = a.max_seqlen <= 48;
  auto kernel = a.decider_pos != nullptr ? (short_call ? attn_short_kernel<DH, true, true> : attn_short_kernel<DH, true, false>)
                                         : (short_call ? attn_short_kernel<DH, false, true> : attn_short_kernel<DH, false, false>);
  D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ShortSmem<DH>::kBytes));
  AttnArgs k = a;
  k.nqb = ceil_div(a.max_seqlen, kTile);
  D3TOM_CUDA_TRY(ctx, launch_serialized(kernel, a.B * a.H * k.nqb, kThreads, ShortSmem<DH>::kBytes, s, tq, tk, tv, k));
  D3TOM_LAUNCH_CHECK(ctx);
  return D3TOM_OK;
}

}  // namespace

// Calls whose 128-row query tiles (of the longest request, for every request) all have an SM of their own; D3TOM_ERR_UNSUPPORTED
// otherwise.
int launch_attn_short(d3tom_ctx* ctx, const AttnArgs& a, cudaStream_t s) {
  if ((long long)a.B * a.H * ceil_div(a.max_seqlen, kTile) > ctx->sm_count) return D3TOM_ERR_UNSUPPORTED;
  if (a.dh == 128) return launch<128>(ctx, a, s);
  if (a.dh == 64) return launch<64>(ctx, a, s);
  return D3TOM_ERR_UNSUPPORTED;
}
