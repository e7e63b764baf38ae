// bf16 x bf16 -> fp32 "NT" GEMM on tcgen05 tensor cores, C[m, n] = sum_k A[m, k] B[n, k],
// with four fused epilogues:
//
//   kEpiProj  the Q,K,V projection of a post-merge layer (Sec. 3.2.1, Q = H W_Q,
//             K = H W_K): rounds to bf16 and writes the tile into q, k or v.
//   kEpiSim   the similarity step of the merge (Sec. 3.2.2, arg max of the cosine
//             over the kept set): scales the dot products by the two inverse norms
//             and folds every pruned row's candidates into its packed 64-bit
//             running maximum, so the (V x k) similarity matrix never reaches HBM.
//   kEpiLinear  y = residual + x W^T rounded to bf16: the attention output projection and the
//             down projection of the feed-forward network (Algorithm 1, FFN_l; the fourth
//             d x d matrix of the 4nd^2 term and the third d x m matrix of the 3ndm term).
//   kEpiGateUp  the first two d x m matrices of the feed-forward network in one pass: a 256-wide
//             tile is 128 gate rows and the 128 up rows of the same features, and the epilogue
//             writes act = silu(gate) * up, so neither product reaches HBM.
//
// Persistent CTAs (one per SM) walk over the 128 x BN output tiles, M fastest so that the
// BN x K operand stays hot in L2 while the M tiles that share it are computed.  Warps 0
// and 6 stream 128x64 / BNx64 operand tiles with TMA into a ring of 128-byte-swizzled
// stages and keep streaming across tile boundaries; one thread of warp 1 issues tcgen05.mma
// (M = 128, N = BN, K = 16) into one of TWO TMEM accumulators; warps 2..5 read the other
// accumulator back with tcgen05.ld (one row per thread) and run the epilogue meanwhile.
#include <math.h>

#include "common.cuh"
#include "ptx.cuh"

namespace {

constexpr int kBM = 128, kBK = 64;
constexpr int kGemmThreads = 224;      // warps: 0 A loads, 1 MMA, 2..5 epilogue, 6 B loads

enum { kEpiProj = 0, kEpiSim = 1, kEpiLinear = 2, kEpiGateUp = 3 };
constexpr int kShortRows = 127;       // calls of at most this many rows (less than a row tile) store row by row
constexpr int kMaxKSplits = 4;        // K slices per tile at most when the last slice to arrive adds them all
constexpr int kCoopSlices = 16;       // K slices per similarity tile at most (every slice adds its own share of the columns)
constexpr uint64_t kSliceWaitNs = 200000ull;   // after this long a slice leaves its share of a tile to the last one

struct GemmParams {
  int num_k_blocks;           // K / 64
  int m_tiles, n_tiles, batch;   // tile grid (per request for the similarity); tiles outside a request are skipped
  int k_splits;               // tiles from `full_tiles` on have their K range cut into this many work units
  int full_tiles;             // the first tiles of the walk are whole work units (0: every tile is cut)
  float* split_ws;            // [(tiles - full_tiles) * k_splits][BN][128] fp32 partial tiles (column-major: coalesced per warp)
  int* split_counters;        // [tiles] parts done; zero between launches
  // projection
  __nv_bfloat16* out[3];      // q, k, v
  int out_rows;               // total tokens
  int out_cols;               // D
  // linear / gate-up: rows are out_rows
  __nv_bfloat16* lin_out;     // [out_rows, ld_out]
  const __nv_bfloat16* residual;   // [out_rows, ld_out] or null (linear only; may be lin_out itself)
  int ld_out;                 // N of the linear layer; m for the gate-up pass
  int up_row_offset;          // gate-up: row of the weight matrix where the up matrix starts (m)
  // similarity
  const int32_t* cu_seqlens; const int32_t* cu_vis; const int32_t* cu_kept; const int32_t* assign;
  const float* inv_norm; const float* inv_norm_kept;
  unsigned long long* best; float* sim_debug; int max_kept;
  int bn, stages;             // CTA pairs: columns of a tile (a multiple of 32, at most 256) and ring stages
  int* dev_status;
};

// Work unit u of the walk: tile t, K slice sp of nsp.  Whole tiles come first, so the cut tiles are the last
// (incomplete) round over the SMs: its few tiles are spread over all SMs instead of occupying a full tile time.
struct Unit {
  int t, sp, nsp, kb0, kb1;
  __device__ __forceinline__ void set(const GemmParams& p, int u) {
    if (u < p.full_tiles) { t = u; sp = 0; nsp = 1; }
    else { const int r = u - p.full_tiles; t = p.full_tiles + r / p.k_splits; sp = r - (t - p.full_tiles) * p.k_splits; nsp = p.k_splits; }
    kb0 = sp * p.num_k_blocks / nsp; kb1 = (sp + 1) * p.num_k_blocks / nsp;
  }
};

// A CTA tile is 128 x BN with two accumulators (the epilogue of a tile overlaps the main loop of the next).
template <int BN> struct GemmSmem {
  static constexpr int kABytes = kBM * kBK * 2, kBBytes = BN * kBK * 2;
  static constexpr int kStages = BN == 256 ? 4 : (BN == 192 ? 5 : 6);   // as many as fit in 227 KB
  static constexpr int kAccStride = BN <= 128 ? 128 : 256;              // TMEM columns between the two accumulators
  static constexpr int kBytes = kStages * (kABytes + kBBytes) + 1024 /*alignment slack*/ + 256 /*barriers*/ + BN * 4;
};

template <int N> struct Const { static constexpr int value = N; };

// Where tile `t` of the walk lies: rows of A, rows of B, and for the similarity the request
// it belongs to.  Returns false for a tile of the bounding grid that a request does not reach.
template <int BN, int EPI>
struct TileCoord {
  int m0, n0, a_row, b_row, b, Vb, kb, v0, k0;
  const int* prefix;      // similarity with a ragged batch: tiles before request b (shared memory), or null
  __device__ __forceinline__ bool set(const GemmParams& p, int t) {
    int mi, ni;
    if (EPI == kEpiSim && prefix != nullptr) {
      // only the tiles that exist are numbered: request b owns [prefix[b], prefix[b + 1]), M fastest
      b = 0;
      while (prefix[b + 1] <= t) ++b;
      const int local = t - prefix[b];
      v0 = p.cu_vis[b]; Vb = p.cu_vis[b + 1] - v0;
      k0 = p.cu_kept[b]; kb = p.cu_kept[b + 1] - k0;
      const int mt = (Vb + kBM - 1) / kBM;
      mi = local % mt; ni = local / mt;
      m0 = mi * kBM; n0 = ni * BN;
      a_row = p.cu_seqlens[b] + m0;
      b_row = k0 + n0;
      return true;
    }
    mi = t % p.m_tiles;
    const int rest = t / p.m_tiles;
    ni = rest % p.n_tiles;
    b = rest / p.n_tiles;
    // (a gate-up tile covers BN / 2 output features: its B rows are 128 gate rows and 128 up rows)
    m0 = mi * kBM; n0 = ni * (EPI == kEpiGateUp ? BN / 2 : BN); a_row = m0; b_row = n0;
    Vb = kb = v0 = k0 = 0;
    if (EPI == kEpiSim) {
      v0 = p.cu_vis[b]; Vb = p.cu_vis[b + 1] - v0;
      k0 = p.cu_kept[b]; kb = p.cu_kept[b + 1] - k0;
      if (m0 >= Vb || n0 >= kb || kb >= Vb) return false;   // nothing pruned in this request, or outside it
      a_row = p.cu_seqlens[b] + m0;
      b_row = k0 + n0;
    }
    return true;
  }
};

constexpr int kMaxPrefixBatch = 64;     // ragged batches up to this many requests number only the tiles that exist

// kShort: dense layers without a residual of at most kShortRows rows (how the results are stored, see store_rows_64b)
template <int BN, int EPI, bool kShort = false>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b, GemmParams p) {
  using S = GemmSmem<BN>;
  constexpr int kStages = S::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* a_s = smem;
  uint8_t* b_s = smem + kStages * S::kABytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * (S::kABytes + S::kBBytes));
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;       // [2]
  uint64_t* acc_empty = acc_full + 2;         // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* ink_s = reinterpret_cast<float*>(smem + kStages * (S::kABytes + S::kBBytes) + 256);

  const int warp = ptx::uniform_warp(), lane = threadIdx.x & 31;
  // barriers and tensor memory first (on-chip only), then wait for the kernels before this one
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { ptx::mbar_init(&full[s], 2); ptx::mbar_init(&empty[s], 1); }   // A and B loaders
    for (int i = 0; i < 2; ++i) { ptx::mbar_init(&acc_full[i], 1); ptx::mbar_init(&acc_empty[i], 4); }   // one arrival per epilogue warp
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 2) { ptx::tmem_alloc(tmem_slot, 2 * S::kAccStride); ptx::tmem_relinquish(); }
  grid_dependency_wait();
  grid_dependency_release();
  int total_units = p.full_tiles + (p.m_tiles * p.n_tiles * p.batch - p.full_tiles) * p.k_splits;   // a unit = one tile, or one K slice of a tile
  // A batch of requests of different sizes: the bounding grid (batch x largest request) is mostly holes, and
  // walking it leaves the SMs unevenly loaded.  Every CTA numbers the tiles that exist (a prefix over requests).
  __shared__ int tile_prefix[kMaxPrefixBatch + 1];
  const bool use_prefix = EPI == kEpiSim && p.batch > 1 && p.batch <= kMaxPrefixBatch;
  if (use_prefix) {
    if (threadIdx.x == 0) {
      int run = 0;
      for (int b = 0; b < p.batch; ++b) {
        tile_prefix[b] = run;
        const int Vb = p.cu_vis[b + 1] - p.cu_vis[b], kb = p.cu_kept[b + 1] - p.cu_kept[b];
        if (kb < Vb) run += ((Vb + kBM - 1) / kBM) * ((kb + BN - 1) / BN);
      }
      tile_prefix[p.batch] = run;
    }
  }

  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  if (use_prefix) total_units = tile_prefix[p.batch] * p.k_splits;      // (the similarity cuts every tile or none)
  const uint32_t tmem_base = *tmem_slot;
  TileCoord<BN, EPI> tc;
  tc.prefix = use_prefix ? tile_prefix : nullptr;

  if (warp == 0 || warp == 6) {
    // ------------------------------------------------------------ TMA producers: warp 0 streams A, warp 6 streams B
    // (issuing a load and its barrier traffic costs the issuing thread a few hundred cycles per
    // k-block; two threads keep ahead of 128 x 192 tiles, one does not)
    if (ptx::elect_one()) {
      const bool is_a = warp == 0;
      const CUtensorMap* tm = is_a ? &tmap_a : &tmap_b;
      uint8_t* ring = is_a ? a_s : b_s;
      const int stage_bytes = is_a ? S::kABytes : S::kBBytes;
      ptx::prefetch_tensormap(tm);
      int it = 0;                                   // k-blocks loaded so far, over all tiles
      bool ok = true;
      Unit un;
      for (int u = blockIdx.x; u < total_units && ok; u += gridDim.x) {
        un.set(p, u);
        if (!tc.set(p, un.t)) continue;
        const int row0 = is_a ? tc.a_row : tc.b_row;
        for (int kbk = un.kb0; kbk < un.kb1; ++kbk, ++it) {
          const int s = it % kStages;
          ok = ptx::mbar_wait(&empty[s], ((it / kStages) & 1) ^ 1, abort_flag, p.dev_status);
          if (!ok) break;
          ptx::mbar_arrive_expect_tx(&full[s], stage_bytes);
          if (EPI == kEpiGateUp && !is_a) {        // two boxes of BN / 2 rows: gate rows, then the up rows of the same features
            ptx::tma_load_2d(ring + s * stage_bytes, tm, &full[s], kbk * kBK, row0);
            ptx::tma_load_2d(ring + s * stage_bytes + stage_bytes / 2, tm, &full[s], kbk * kBK, p.up_row_offset + row0);
          } else {
            ptx::tma_load_2d(ring + s * stage_bytes, tm, &full[s], kbk * kBK, row0);
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (ptx::elect_one()) {
      constexpr uint32_t idesc = ptx::idesc_bf16_f32(kBM, BN, 0, 0);
      const ptx::SmemDesc a_desc0 = ptx::smem_desc_kmajor_sw128(ptx::smem_u32(a_s));
      const ptx::SmemDesc b_desc0 = ptx::smem_desc_kmajor_sw128(ptx::smem_u32(b_s));
      int it = 0, lt = 0;                           // k-blocks and tiles consumed so far
      bool ok = true;
      Unit un;
      for (int u = blockIdx.x; u < total_units && ok; u += gridDim.x) {
        un.set(p, u);
        if (!tc.set(p, un.t)) continue;
        const int kb0 = un.kb0, kb1 = un.kb1;
        const int buf = lt & 1;
        const uint32_t acc_use = (uint32_t)(lt >> 1);               // how often this buffer has been used
        ok = ptx::mbar_wait(&acc_empty[buf], (acc_use & 1) ^ 1, abort_flag, p.dev_status);   // epilogue done with it
        if (!ok) break;
        ptx::tc_fence_after_sync();
        const uint32_t tmem_acc = tmem_base + (uint32_t)buf * S::kAccStride;
        for (int kbk = kb0; kbk < kb1; ++kbk, ++it) {
          const int s = it % kStages;
          ok = ptx::mbar_wait(&full[s], (it / kStages) & 1, abort_flag, p.dev_status);
          if (!ok) break;
          ptx::tc_fence_after_sync();
          const ptx::SmemDesc ad = ptx::smem_desc_advance(a_desc0, s * S::kABytes), bd = ptx::smem_desc_advance(b_desc0, s * S::kBBytes);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)
            ptx::mma_ss(tmem_acc, ptx::smem_desc_advance(ad, kk * 32), ptx::smem_desc_advance(bd, kk * 32), idesc,
                        (kbk > kb0 || kk > 0) ? 1u : 0u);
          ptx::mma_commit(&empty[s]);     // frees the stage once these MMAs have read it
        }
        if (ok) ptx::mma_commit(&acc_full[buf]);
        ++lt;
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue: warp w may touch TMEM lanes 32*(w%4) .. +31
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;           // row of the tile owned by this thread
    const int et = threadIdx.x - 64;               // 0..127 among the epilogue threads
    int lt = 0;
    __shared__ int s_prev;
    Unit un;
    for (int u = blockIdx.x; u < total_units; u += gridDim.x) {
      un.set(p, u);
      const int t = un.t, sp = un.sp;
      if (!tc.set(p, t)) continue;
      const int buf = lt & 1;
      const uint32_t acc_use = (uint32_t)(lt >> 1);
      if (EPI == kEpiSim) {
        // inverse norms of this tile's kept rows; the four epilogue warps share them (named barrier 1)
        asm volatile("bar.sync 1, 128;" ::: "memory");          // everyone is done with the previous tile's values
        for (int j = et; j < BN; j += 128) ink_s[j] = (tc.n0 + j < tc.kb) ? p.inv_norm_kept[tc.k0 + tc.n0 + j] : 0.f;
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
      const bool ok = __all_sync(0xffffffffu, ptx::mbar_wait(&acc_full[buf], acc_use & 1, abort_flag, p.dev_status));
      if (!ok) break;
      ptx::tc_fence_after_sync();
      const uint32_t t_row = tmem_base + (uint32_t)buf * S::kAccStride + ((uint32_t)(quarter * 32) << 16);
      // A tile whose K range is cut into slices on different SMs: every unit writes its partial sums out (column-major, so
      // a warp's 32 rows are one 128-byte line) and counts itself in.  Dense layers: the unit that completes the tile
      // adds the parts in the order of the K slices and runs the epilogue on the sums (the counter is left at zero
      // again).  Similarity: every slice adds up its share of the columns (below).  Same values whichever unit comes last.
      const bool split = un.nsp > 1;
      constexpr bool coop = EPI == kEpiSim;                     // every slice adds up a share of the columns, or the last one adds all
      const int ws_tile = t - p.full_tiles;                     // cut tiles are numbered from zero in the workspace
      bool last = true;
      if (split) {
        float* part = p.split_ws + (size_t)(ws_tile * un.nsp + sp) * BN * kBM;
        const int live_cols = EPI == kEpiSim ? min(BN, tc.kb - tc.n0) : BN;      // (columns past the kept set are never read)
#pragma unroll 1
        for (int c = 0; c < live_cols; c += 32) {
          uint32_t r[32];
          ptx::tmem_ld32(t_row + c, r);
          ptx::tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) part[(size_t)(c + i) * kBM + row] = __uint_as_float(r[i]);
        }
        ptx::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&acc_empty[buf]);          // the accumulator is free again
        __threadfence();
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (!coop) {
          if (et == 0) s_prev = atomicAdd(p.split_counters + ws_tile, 1);
          asm volatile("bar.sync 1, 128;" ::: "memory");
          last = s_prev == un.nsp - 1;
          if (last) {
            if (et == 0) p.split_counters[ws_tile] = 0;
            __threadfence();
          }
        } else {
          // The slices of a tile are neighbouring CTAs and normally all resident: wait until all have written, then each
          // adds up its own share of the columns.  Nothing depends on that, though: a slice that has waited kSliceWaitNs
          // (the SMs may be held by another stream) leaves its share to the slice that arrives last.
          // Counter word: bits 0..7 slices arrived, 8..15 shares done, 16..31 shares left behind.
          if (et == 0) {
            int* ctr = p.split_counters + ws_tile;
            const int before = atomicAdd(ctr, 1);
            s_prev = 1 << sp;                                                    // shares this CTA adds up
            if ((before & 0xff) == un.nsp - 1) {
              s_prev |= (int)((uint32_t)before >> 16);
            } else {
              const uint64_t t0 = ptx::globaltimer_ns();
              uint32_t polls = 0;
              while ((*static_cast<const volatile int*>(ctr) & 0xff) < un.nsp) {
                if ((++polls & 0x3fu) == 0u && ptx::globaltimer_ns() - t0 > kSliceWaitNs) {
                  // (had the last slice arrived before this word was set, it did not see it: the share is still ours)
                  if ((atomicOr(ctr, (int)(1u << (16 + sp))) & 0xff) < un.nsp) s_prev = 0;
                  break;
                }
              }
            }
          }
          asm volatile("bar.sync 1, 128;" ::: "memory");
          __threadfence();
        }
      }
      // 32 accumulator columns of this thread's row: from tensor memory, or the sum of the slices
      auto load32 = [&](int c, float (&acc)[32]) {
        if (EPI == kEpiSim || !split) {          // (the similarity's slices never come here: they add up their columns above)
          uint32_t r[32];
          ptx::tmem_ld32(t_row + c, r);
          ptx::tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] = __uint_as_float(r[i]);
        } else {
          // all slices of the 32 columns are requested before any is added (one round trip, not one per slice)
          float part[kMaxKSplits][32];
#pragma unroll
          for (int q = 0; q < kMaxKSplits; ++q) {
            const float* src = p.split_ws + ((size_t)(ws_tile * un.nsp + q) * BN + c) * kBM + row;
            if (q < un.nsp) {
#pragma unroll
              for (int i = 0; i < 32; ++i) part[q][i] = __ldcg(src + (size_t)i * kBM);
            }
          }
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] = 0.f;
#pragma unroll
          for (int q = 0; q < kMaxKSplits; ++q)
            if (q < un.nsp) {
#pragma unroll
              for (int i = 0; i < 32; ++i) acc[i] += part[q][i];
            }
        }
      };
      if (!last) { ++lt; continue; }
      if (coop && split) {
        // shares of the tile's live columns in groups of eight, this slice's own and any left behind: the sums over all
        // slices (ascending slice order), then the arg-max over those columns; the 64-bit maximum over slices and tiles
        // is order-independent
        const int nsp = un.nsp;                                  // 2 .. 16
        const int groups = (min(BN, tc.kb - tc.n0) + 7) >> 3;
        const int shares = s_prev;
        const int m = tc.m0 + row;
        const int g = tc.v0 + m;
        const bool active = m < tc.Vb && p.assign[g] < 0;
        const float inm = active ? p.inv_norm[g] : 0.f;
        float best_sim = -INFINITY;
        int best_slot = 0;
        int cb, ce;                                              // columns of the share in hand
        float* dbg = (p.sim_debug != nullptr && active) ? p.sim_debug + (size_t)g * p.max_kept + tc.n0 : nullptr;
        const float* tile_ws = p.split_ws + (size_t)ws_tile * nsp * BN * kBM + row;
        // kQ slices x kC columns of loads in flight (64 words a thread)
        auto add_up = [&](auto q_tag, auto c_tag) {
          constexpr int kQ = decltype(q_tag)::value, kC = decltype(c_tag)::value;
#pragma unroll 1
          for (int c = cb; c < ce; c += kC) {
            float dot[kC];
#pragma unroll
            for (int i = 0; i < kC; ++i) dot[i] = 0.f;
#pragma unroll 1
            for (int q0 = 0; q0 < nsp; q0 += kQ) {
              float part[kQ][kC];
#pragma unroll
              for (int q = 0; q < kQ; ++q)
                if (q0 + q < nsp) {
                  const float* src = tile_ws + ((size_t)(q0 + q) * BN + c) * kBM;
#pragma unroll
                  for (int i = 0; i < kC; ++i)
                    if (c + (i & ~7) < ce) part[q][i] = __ldcg(src + (size_t)i * kBM);
                }
#pragma unroll
              for (int q = 0; q < kQ; ++q)
                if (q0 + q < nsp) {
#pragma unroll
                  for (int i = 0; i < kC; ++i)
                    if (c + (i & ~7) < ce) dot[i] += part[q][i];
                }
            }
#pragma unroll
            for (int i = 0; i < kC; ++i) {
              const int sidx = tc.n0 + c + i;
              if (active && c + i < ce && sidx < tc.kb) {
                const float sim = (dot[i] * inm) * ink_s[c + i] + 0.0f;
                if (sim > best_sim) { best_sim = sim; best_slot = sidx; }
                if (dbg != nullptr) dbg[c + i] = sim;
              }
            }
          }
        };
        bool any = false;
#pragma unroll 1
        for (int left = shares; left != 0; left &= left - 1) {   // (ascending columns: the lowest slot wins a tie)
          const int share = __ffs(left) - 1;
          cb = share * groups / nsp * 8; ce = (share + 1) * groups / nsp * 8;
          any |= cb < ce;
          if (nsp > 4) add_up(Const<8>{}, Const<8>{});
          else add_up(Const<4>{}, Const<16>{});
        }
        if (active && any) {
          const unsigned long long mine =
              ((unsigned long long)ordered_key(best_sim) << 32) | (0xffffffffu - (unsigned)best_slot);
          atomicMax(p.best + g, mine);
        }
        // whoever finishes the last share leaves the counter at zero (a slice that left its share behind is not coming back)
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (et == 0 && shares != 0) {
          const int n = __popc(shares), before = atomicAdd(p.split_counters + ws_tile, n << 8);
          if (((before >> 8) & 0xff) + n == nsp) p.split_counters[ws_tile] = 0;
        }
        ++lt;
        continue;
      }
      const int warp_row = tc.m0 + quarter * 32, n_valid = p.out_rows - warp_row;      // dense layers: this warp's 32 rows
      if (EPI == kEpiProj) {
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          float r[32];
          load32(c, r);
          // 32 divides D, so a 32-column piece lies in one of q, k, v even when the tile straddles two of them
          const int gcol = tc.n0 + c, which = gcol / p.out_cols;
          if (which < 3) {                           // (a tile width that does not divide 3 D: the last tile hangs over)
            uint32_t w[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              __nv_bfloat162 h2 = __floats2bfloat162_rn(r[2 * j], r[2 * j + 1]);
              w[j] = *reinterpret_cast<uint32_t*>(&h2);
            }
            ptx::store_rows_64b<kShort>(p.out[which] + (size_t)warp_row * p.out_cols + (gcol - which * p.out_cols),
                                (size_t)p.out_cols * 2, n_valid, w);
          }
        }
      } else if (EPI == kEpiLinear) {
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          float r[32];
          load32(c, r);
          if (tc.n0 + c < p.ld_out) {
            uint32_t w[16];
            if (!kShort && p.residual != nullptr) {
              ptx::load_rows_64b(p.residual + (size_t)warp_row * p.ld_out + tc.n0 + c, (size_t)p.ld_out * 2, n_valid, w);
            } else {
#pragma unroll
              for (int i = 0; i < 16; ++i) w[i] = 0u;
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              __nv_bfloat162 h2 = __floats2bfloat162_rn(r[2 * j] + __uint_as_float(w[j] << 16),
                                                        r[2 * j + 1] + __uint_as_float(w[j] & 0xffff0000u));
              w[j] = *reinterpret_cast<uint32_t*>(&h2);
            }
            // (out may be the residual buffer: the piece of a row is read and written by the same lane)
            ptx::store_rows_64b<kShort>(p.lin_out + (size_t)warp_row * p.ld_out + tc.n0 + c, (size_t)p.ld_out * 2, n_valid, w);
          }
        }
      } else if (EPI == kEpiGateUp) {
#pragma unroll 1
        for (int c = 0; c < BN / 2; c += 32) {
          float g[32], up[32];
          load32(c, g);
          load32(BN / 2 + c, up);
          uint32_t w[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float g0 = g[2 * j], g1 = g[2 * j + 1];
            // silu(g) = g / (1 + exp(-g)); for very negative g the divisor is inf and the quotient 0
            __nv_bfloat162 h2 = __floats2bfloat162_rn(__fdividef(g0, 1.f + __expf(-g0)) * up[2 * j],
                                                      __fdividef(g1, 1.f + __expf(-g1)) * up[2 * j + 1]);
            w[j] = *reinterpret_cast<uint32_t*>(&h2);
          }
          ptx::store_rows_64b<kShort>(p.lin_out + (size_t)warp_row * p.ld_out + tc.n0 + c, (size_t)p.ld_out * 2, n_valid, w);
        }
      } else {
        const int m = tc.m0 + row;
        const int g = tc.v0 + m;
        const bool active = m < tc.Vb && p.assign[g] < 0;     // a pruned token of this request
        const float inm = active ? p.inv_norm[g] : 0.f;
        float best_sim = -INFINITY;                        // strict > below: the lowest slot wins a tie
        int best_slot = 0;
        float* dbg = (p.sim_debug != nullptr && active) ? p.sim_debug + (size_t)g * p.max_kept + tc.n0 : nullptr;
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          float dot[32];
          load32(c, dot);
          if (active) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              const int sidx = tc.n0 + c + i;
              if (sidx < tc.kb) {
                // the value the arg-max compares; + 0 turns a negative zero into the positive one
                const float sim = (dot[i] * inm) * ink_s[c + i] + 0.0f;
                if (sim > best_sim) { best_sim = sim; best_slot = sidx; }
                if (dbg != nullptr) dbg[c + i] = sim;
              }
            }
          }
        }
        if (active) {
          const unsigned long long mine =
              ((unsigned long long)ordered_key(best_sim) << 32) | (0xffffffffu - (unsigned)best_slot);
          atomicMax(p.best + g, mine);
        }
      }
      if (split) { ++lt; continue; }                      // (its accumulator was released when the partial went out)
      // the accumulator may be overwritten once all four warps have read it
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&acc_empty[buf]);
      ++lt;
    }
    ptx::tc_fence_before_sync();
  }
  __syncthreads();
  if (warp == 2) ptx::tmem_dealloc(tmem_base, 2 * S::kAccStride);
}

// ---------------------------------------------------------------- CTA pairs
// Two CTAs of a cluster (ranks 0 and 1, neighbouring SMs) compute one 256 x bn tile with `cta_group::2` MMAs: each CTA
// holds its own 128 rows of A and HALF of the B tile (bn / 2 rows) in shared memory, the tensor cores of both read both
// halves, and each CTA's 128 x bn accumulator lands in its own tensor memory.  Per k-block a CTA pulls 16 + bn / 16 KB out
// of L2: 32 KB for 512 tensor cycles at bn = 256, where the single-CTA 128 x 256 tile needs 48 KB
// and is bound by what an SM can pull out of L2 (about 56 B per cycle).
// The width is chosen at run time (any multiple of 32 up to 256: the instruction descriptor, the tensor map's box and the
// ring's strides are data), because what separates the widths is how the tiles fill the rounds over the pairs.
//   * both CTAs run the same warp roles; each loader thread waits on its OWN `empty` barrier and loads its own boxes, whose
//     bytes are counted on rank 0's `full` barrier (rank 0's loader threads expect the bytes of both CTAs);
//   * one thread of rank 0 issues every MMA and commits to the `empty` / `acc_full` barriers of BOTH CTAs;
//   * the epilogue warps of both CTAs arrive on rank 0's `acc_empty` barrier (8 arrivals);
//   * before a CTA leaves, its loaders have seen every commit aimed at it, rank 0 has seen every epilogue arrival, and
//     the two CTAs meet in a cluster barrier; tensor memory is allocated and freed by warp 2 of both CTAs together.
// Whole tiles only (no K split); every mbarrier wait is bounded as elsewhere.
// 64-deep boxes of each operand per stage.  Two for the narrower tiles: a barrier check and a commit then serve eight MMAs
// instead of four, whose overhead shows where an MMA is short (128 columns: 0.33 -> 0.29 us per 64 of K, 192: 0.35 -> 0.31);
// one for the wider ones, whose ring would be left with three stages (256 columns: 0.32 against 0.33 us).
__host__ __device__ constexpr int pair_sub(int bn) { return bn <= 192 ? 2 : 1; }
constexpr int kPairMaxStages = 8;
constexpr int kPairSmemLimit = 227 * 1024;
__host__ __device__ constexpr int pair_stage_bytes(int bn) { return pair_sub(bn) * (kBM * kBK * 2 + (bn / 2) * kBK * 2); }
constexpr int pair_stages(int bn) {
  const int fit = (kPairSmemLimit - 1024 - 256) / pair_stage_bytes(bn);
  return fit < kPairMaxStages ? fit : kPairMaxStages;
}
constexpr int pair_smem_bytes(int bn) { return pair_stages(bn) * pair_stage_bytes(bn) + 1024 /*alignment slack*/ + 256 /*barriers*/; }

// stage index and phase of a ring of p.stages buffers
struct RingPos {
  int s = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void next(int stages) { if (++s == stages) { s = 0; phase ^= 1u; } }
};

template <int EPI, int kSub>           // kSub == pair_sub(p.bn)
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b, GemmParams p) {
  static_assert(EPI != kEpiSim, "the dense layers only");
  constexpr int kABytes = kBM * kBK * 2;                   // one box of A; of B: bn / 2 rows of 128 bytes (whole 8-row swizzle groups)
  const int bn = p.bn, stages = p.stages, b_bytes = (bn / 2) * kBK * 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* a_s = smem;
  uint8_t* b_s = smem + stages * kSub * kABytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + stages * kSub * (kABytes + b_bytes));
  uint64_t* empty = full + kPairMaxStages;
  uint64_t* acc_full = empty + kPairMaxStages;   // [2]
  uint64_t* acc_empty = acc_full + 2;            // [2] (rank 0's are the ones in use)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = ptx::uniform_warp(), lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  const bool leader = rank == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { ptx::mbar_init(&full[s], 2); ptx::mbar_init(&empty[s], 1); }   // A and B loaders of rank 0; one commit
    for (int i = 0; i < 2; ++i) { ptx::mbar_init(&acc_full[i], 1); ptx::mbar_init(&acc_empty[i], 8); }   // four epilogue warps in each CTA
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 2) { ptx::tmem_alloc_pair(tmem_slot, 512); ptx::tmem_relinquish_pair(); }
  grid_dependency_wait();
  grid_dependency_release();
  ptx::tc_fence_before_sync();
  ptx::cluster_sync();                     // the peer's barriers exist before anything arrives on them
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  const int tiles = p.m_tiles * p.n_tiles;
  const int n_pairs = gridDim.x >> 1, pair = blockIdx.x >> 1;
  // tile t: M fastest, so that the pairs of a round share their B tiles in L2
  auto tile_m0 = [&](int t) { return (t % p.m_tiles) * (2 * kBM); };
  auto tile_n0 = [&](int t) { return (t / p.m_tiles) * (EPI == kEpiGateUp ? bn / 2 : bn); };

  if (warp == 0 || warp == 6) {
    // ------------------------------------------------------------ TMA producers: warp 0 streams A, warp 6 streams B
    if (ptx::elect_one()) {
      const bool is_a = warp == 0;
      const CUtensorMap* tm = is_a ? &tmap_a : &tmap_b;
      uint8_t* ring = is_a ? a_s : b_s;
      const int box_bytes = is_a ? kABytes : b_bytes;
      ptx::prefetch_tensormap(tm);
      int it = 0;
      RingPos r;
      bool ok = true;
      for (int t = pair; t < tiles && ok; t += n_pairs) {
        const int n0 = tile_n0(t);
        // this CTA's rows: its half of the 256 rows of A; its half of the B tile (gate rows for rank 0, up rows for rank 1)
        const int row0 = is_a ? tile_m0(t) + (int)rank * kBM
                              : (EPI == kEpiGateUp ? (leader ? n0 : p.up_row_offset + n0) : n0 + (int)rank * (bn / 2));
        for (int kbk = 0; kbk < p.num_k_blocks; kbk += kSub, ++it, r.next(stages)) {
          const int sub = min(kSub, p.num_k_blocks - kbk);
          ok = ptx::mbar_wait(&empty[r.s], r.phase ^ 1u, abort_flag, p.dev_status);
          if (!ok) break;
          if (leader) ptx::mbar_arrive_expect_tx(&full[r.s], 2 * sub * box_bytes);     // this operand's boxes of both CTAs
#pragma unroll
          for (int b = 0; b < kSub; ++b)
            if (b < sub) ptx::tma_load_2d_pair(ring + (r.s * kSub + b) * box_bytes, tm, &full[r.s], (kbk + b) * kBK, row0);
        }
      }
      // every commit aimed at this CTA's `empty` barriers has landed before the CTA may leave
      for (int j = it > stages ? it - stages : 0; j < it && ok; ++j)
        ok = ptx::mbar_wait(&empty[j % stages], (j / stages) & 1, abort_flag, p.dev_status);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (rank 0 only)
    if (leader && ptx::elect_one()) {
      const uint32_t idesc = ptx::idesc_bf16_f32(2 * kBM, bn, 0, 0);
      const ptx::SmemDesc a_desc0 = ptx::smem_desc_kmajor_sw128(ptx::smem_u32(a_s));
      const ptx::SmemDesc b_desc0 = ptx::smem_desc_kmajor_sw128(ptx::smem_u32(b_s));
      int lt = 0;
      RingPos r;
      bool ok = true;
      for (int t = pair; t < tiles && ok; t += n_pairs, ++lt) {
        const int buf = lt & 1;
        ok = ptx::mbar_wait(&acc_empty[buf], ((lt >> 1) & 1) ^ 1, abort_flag, p.dev_status);   // both epilogues done with it
        if (!ok) break;
        ptx::tc_fence_after_sync();
        const uint32_t tmem_acc = tmem_base + (uint32_t)buf * 256u;
        for (int kbk = 0; kbk < p.num_k_blocks; kbk += kSub, r.next(stages)) {
          ok = ptx::mbar_wait(&full[r.s], r.phase, abort_flag, p.dev_status);
          if (!ok) break;
          ptx::tc_fence_after_sync();
          const ptx::SmemDesc ad = ptx::smem_desc_advance(a_desc0, r.s * kSub * kABytes);
          const ptx::SmemDesc bd = ptx::smem_desc_advance(b_desc0, r.s * kSub * b_bytes);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)
            ptx::mma_ss_pair(tmem_acc, ptx::smem_desc_advance(ad, kk * 32), ptx::smem_desc_advance(bd, kk * 32), idesc,
                             (kbk > 0 || kk > 0) ? 1u : 0u);
          if (kSub > 1 && kbk + 1 < p.num_k_blocks) {
            const ptx::SmemDesc ad1 = ptx::smem_desc_advance(ad, kABytes), bd1 = ptx::smem_desc_advance(bd, b_bytes);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              ptx::mma_ss_pair(tmem_acc, ptx::smem_desc_advance(ad1, kk * 32), ptx::smem_desc_advance(bd1, kk * 32), idesc, 1u);
          }
          ptx::mma_commit_pair(&empty[r.s], 3);      // frees the stage in both CTAs once these MMAs have read it
        }
        if (ok) ptx::mma_commit_pair(&acc_full[buf], 3);
      }
      // the peer's epilogue arrivals for the last tiles have landed before this CTA may leave
      for (int j = lt > 2 ? lt - 2 : 0; j < lt && ok; ++j)
        ok = ptx::mbar_wait(&acc_empty[j & 1], (j >> 1) & 1, abort_flag, p.dev_status);
    }
  } else {
    // ------------------------------------------------------------ epilogue: warp w may touch TMEM lanes 32*(w%4) .. +31
    // 32 columns at a time
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    int lt = 0;
    for (int t = pair; t < tiles; t += n_pairs, ++lt) {
      const int buf = lt & 1;
      const bool ok = __all_sync(0xffffffffu, ptx::mbar_wait(&acc_full[buf], (lt >> 1) & 1, abort_flag, p.dev_status));
      if (!ok) break;
      ptx::tc_fence_after_sync();
      const uint32_t t_row = tmem_base + (uint32_t)buf * 256u + ((uint32_t)(quarter * 32) << 16);
      const int grow = tile_m0(t) + (int)rank * kBM + row;
      const int n0 = tile_n0(t);
      // columns of the tile that exist
      const int width = EPI == kEpiGateUp ? min(bn / 2, p.ld_out - n0) : min(bn, (EPI == kEpiProj ? 3 * p.out_cols : p.ld_out) - n0);
      const bool live = grow < p.out_rows;
#pragma unroll 1
      for (int c = 0; c < width; c += 32) {
        uint32_t r[32];
        ptx::tmem_ld32(t_row + c, r);
        if (EPI == kEpiGateUp) {
          uint32_t up[32];
          ptx::tmem_ld32(t_row + bn / 2 + c, up);
          ptx::tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float g = __uint_as_float(r[i]);
            // silu(g) = g / (1 + exp(-g)); for very negative g the divisor is inf and the quotient 0
            r[i] = __float_as_uint(__fdividef(g, 1.f + __expf(-g)) * __uint_as_float(up[i]));
          }
        } else {
          ptx::tmem_wait_ld();
        }
        // the piece's destination: one row of one output; only a gate-up half of 80 or 112 columns ends in half a piece
        __nv_bfloat16* base;
        size_t ld;
        if (EPI == kEpiProj) {
          const int gcol = n0 + c, which = gcol / p.out_cols;      // (32 divides D: a piece lies in one of q, k, v)
          base = p.out[which] + (gcol - which * p.out_cols);
          ld = (size_t)p.out_cols;
        } else {
          base = p.lin_out + n0 + c;
          ld = (size_t)p.ld_out;
        }
        uint32_t w[16];
        if (EPI == kEpiLinear && p.residual != nullptr) {
          ptx::load_rows_64b(p.residual + (size_t)(grow - lane) * ld + n0 + c, ld * 2, p.out_rows - (grow - lane), w);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) w[i] = 0u;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float lo = __uint_as_float(r[2 * j]), hi = __uint_as_float(r[2 * j + 1]);
          if (EPI == kEpiLinear) { lo += __uint_as_float(w[j] << 16); hi += __uint_as_float(w[j] & 0xffff0000u); }
          __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
          w[j] = *reinterpret_cast<uint32_t*>(&h2);
        }
        if (EPI != kEpiGateUp || c + 32 <= width) {
          ptx::store_rows_64b(base + (size_t)(grow - lane) * ld, ld * 2, p.out_rows - (grow - lane), w);
        } else if (live) {
#pragma unroll
          for (int i = 0; i < 2; ++i)
            *reinterpret_cast<uint4*>(base + (size_t)grow * ld + i * 8) = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
        }
      }
      // the accumulator may be overwritten once the four warps of both CTAs have read it: tell rank 0
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if (leader) ptx::mbar_arrive(&acc_empty[buf]);
        else ptx::mbar_arrive_cluster(&acc_empty[buf], 0);
      }
    }
  }
  __syncwarp();                            // (the lanes that ran a role's loop rejoin their warp before the aligned barrier)
  ptx::tc_fence_before_sync();
  ptx::cluster_sync();                     // neither CTA frees tensor memory or leaves while the other may still reach it
  if (warp == 2) ptx::tmem_dealloc_pair(tmem_base, 512);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// The dense layers walk whole tiles; when the last round over the SMs is incomplete, its tiles are cut into K
// slices so that the round costs a fraction of a tile time plus the exchange of partial sums.  Costs in units of
// one k-block of main loop (about 0.35 us): a cut round costs about 30 + 5 per slice on top of its k-blocks (measured:
// 15 - 18 us; reading the slices back through bulk copies instead of register loads did not change it, so it is the
// cold start of the short main loops and the fence / counter round trips rather than the read-back), so cutting
// pays for long K only: the down projection of the feed-forward network, not the 64-k-block projections.
// Returns the number of slices (1: the tiles stay whole).
int tail_slices(int sms, int tiles, int num_k_blocks) {
  const int rem = tiles % sms;
  int best = num_k_blocks, best_s = 1;
  for (int sp = 2; sp <= kMaxKSplits && rem > 0; ++sp) {
    if (num_k_blocks / sp < 8 || rem * sp > 2 * sms) break;      // slices too short / more parts than the workspace holds
    const int rounds = (rem * sp + sms - 1) / sms;
    const int cost = rounds * ((num_k_blocks + sp - 1) / sp) + 30 + 5 * sp;
    if (cost < best) { best = cost; best_s = sp; }
  }
  return best_s;
}
void plan_tail_split(const d3tom_ctx* ctx, GemmParams& p) {
  const int tiles = p.m_tiles * p.n_tiles * p.batch;
  p.k_splits = tail_slices(ctx->sm_count, tiles, p.num_k_blocks);
  p.full_tiles = p.k_splits > 1 ? tiles - tiles % ctx->sm_count : tiles;
}

// What a dense layer costs in tiles of one shape (us): `start` once, per 64 of K `round` for each full round of tiles over the
// SMs (or the pairs) and `part` + `part_r` x (its share of the SMs) for an incomplete last one, which leaves more of L2 to
// each, and `more` for every round after the first (an epilogue that nothing hides).  Fitted to 250 layers (64 .. 8000 rows,
// K 512 .. 12288, 1024 .. 12288 columns) timed in every shape, each after a pause, with the operands in L2; over them the cheapest
// shape by these figures is 0.4 % slower than the fastest one.  pair_tile_width asks them for the shape between 513 and 2047 rows
// only; below and above its older rules stand, which were fitted back to back under the board's power limit.
struct TileCost { int width; double start, round, part, part_r, more; };
constexpr TileCost kOneCost[] = {{256, 7.13, 0.401, 0.283, 0.093, 1.80}, {192, 6.13, 0.284, 0.214, 0.084, 1.78},
                                 {128, 4.96, 0.222, 0.144, 0.067, 0.72}};
constexpr TileCost kPairCost[] = {{256, 7.89, 0.345, 0.267, 0.088, 2.12}, {224, 7.42, 0.299, 0.225, 0.089, 1.41},
                                  {192, 7.09, 0.255, 0.191, 0.087, 1.55}, {160, 6.55, 0.221, 0.162, 0.068, 1.15},
                                  {128, 6.04, 0.192, 0.122, 0.078, 1.18}};
double tile_time(const TileCost& c, long long tiles, int units, int num_k_blocks) {
  const double full = (double)(tiles / units), rest = (double)(tiles % units) / units;
  const double rounds = full + (rest > 0 ? 1.0 : 0.0);
  return c.start + num_k_blocks * (c.round * full + (rest > 0 ? c.part + c.part_r * rest : 0.0)) + c.more * (rounds - 1.0);
}

// Width of single-CTA tiles (one that divides the columns; 128 always does).  By rounds alone, weighed 667 / 633 / 600 for 256 /
// 192 / 128 columns, it took 256 too often at a long K (2600 rows x 6144 x 2048: 1.20 x the time of 128); a K below 1024 is
// start and epilogue, where fewer rounds are right (130 x 256 x 12288: 192 columns 8.2 us, 128 9.3).
int one_m_tile_width(int sms, int rows, int ncols, int num_k_blocks) {
  int bn = 128;
  double best = 1e30;
  for (const TileCost& c : kOneCost) {
    if (ncols % c.width != 0) continue;
    const long long tiles = (long long)ceil_div(rows, kBM) * (ncols / c.width);
    const double t = num_k_blocks >= 16 ? tile_time(c, tiles, sms, num_k_blocks)
                                        : (double)((tiles + sms - 1) / sms) * (c.width == 256 ? 667.0 : c.width == 192 ? 633.0 : 600.0);
    if (t < best) { best = t; bn = c.width; }
  }
  return bn;
}

template <int BN, int EPI>
int launch_gemm(d3tom_ctx* ctx, const CUtensorMap& ta, const CUtensorMap& tb, GemmParams p, cudaStream_t s) {
  if (EPI != kEpiSim) {
    p.split_ws = ctx->gemm_split_ws; p.split_counters = ctx->gemm_split_counters;
    plan_tail_split(ctx, p);
  }
  const long long tiles = (long long)p.m_tiles * p.n_tiles * p.batch;
  const long long units = p.full_tiles + (tiles - p.full_tiles) * p.k_splits;
  if (units <= 0) return D3TOM_OK;
  const int grid = (int)(units < ctx->sm_count ? units : ctx->sm_count);          // persistent: one CTA per SM
  auto kernel = gemm_tc_kernel<BN, EPI>;
  if constexpr (EPI != kEpiSim) {
    if (p.out_rows <= kShortRows && p.residual == nullptr) kernel = gemm_tc_kernel<BN, EPI, true>;
  }
  D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmSmem<BN>::kBytes));
  D3TOM_CUDA_TRY(ctx, launch_serialized(kernel, grid, kGemmThreads, GemmSmem<BN>::kBytes, s, ta, tb, p));
  return D3TOM_OK;
}

// How many CTA pairs of this kernel the device holds at once (asked once per device; 0 = clusters of two cannot be
// launched here, and the caller keeps single-CTA tiles).
template <int EPI>
int resident_pairs(d3tom_ctx* ctx) {
  static int cached[64] = {};
  int& pairs = cached[ctx->device & 63];
  if (pairs == 0) {
    auto kernel = gemm_pair_kernel<EPI, 1>;      // (both forms: one CTA per SM, the same shared memory)
    pairs = -1;
    if (ctx->sm_count >= 2 &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmemLimit) == cudaSuccess) {
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(ctx->sm_count & ~1)); cfg.blockDim = dim3(kGemmThreads);
      cfg.dynamicSmemBytes = kPairSmemLimit; cfg.attrs = attr; cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0)
        pairs = n < ctx->sm_count / 2 ? n : ctx->sm_count / 2;
    }
    if (pairs < 0) (void)cudaGetLastError();     // (the refusal is not an error of the call in hand)
  }
  return pairs > 0 ? pairs : 0;
}

template <int EPI>
int launch_gemm_pair(d3tom_ctx* ctx, const CUtensorMap& ta, const CUtensorMap& tb, GemmParams p, cudaStream_t s) {
  const long long tiles = (long long)p.m_tiles * p.n_tiles;
  if (tiles <= 0) return D3TOM_OK;
  const int pairs = resident_pairs<EPI>(ctx);
  if (pairs <= 0) return D3TOM_ERR_UNSUPPORTED;
  p.stages = pair_stages(p.bn);
  const int smem = pair_smem_bytes(p.bn);
  auto kernel = pair_sub(p.bn) == 2 ? gemm_pair_kernel<EPI, 2> : gemm_pair_kernel<EPI, 1>;
  // (the attribute belongs to the current device: set on every call, a process may drive several GPUs)
  D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmemLimit));
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = g_d3tom_launch_overlap ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * (tiles < pairs ? tiles : pairs))); cfg.blockDim = dim3(kGemmThreads);
  cfg.dynamicSmemBytes = smem; cfg.stream = s; cfg.attrs = attr; cfg.numAttrs = 2;
  D3TOM_CUDA_TRY(ctx, cudaLaunchKernelEx(&cfg, kernel, ta, tb, p));
  return D3TOM_OK;
}

// Width of the CTA-pair tiles for a dense layer of `rows` x `ncols` outputs (for the gate-up pass the columns of both
// matrices), or 0 for single-CTA tiles.
//   - 513 .. 2047 rows, K of 1024 and more: the shape that is cheapest by the costs above.  A rule by rounds that weighed 256-row
//     single-CTA tiles against pairs took neither the best width nor the better kind (us, rule / now): linear 1216 x 4096 x 4096
//     48.9 / 33.1, 1408 x 4096 x 4096 53.4 / 40.1, 1216 x 12288 x 4096 119 / 97, 1216 x 4096 x 12288 107 / 92,
//     1408 x 1024 x 6144 23.2 / 19.2; the 256-row tiles, never the fastest of the 250 layers, are gone.  (With pairs switched off, or
//     where none fits, 128-row tiles serve these layers too: of 200 random ones of 300 .. 3000 rows 185 are as fast as with 256-row
//     tiles or faster, the others up to 15 % slower, 1133 x 12288 x 6400 141 / 163 us.)
//   - other layers below 2048 rows: rounds, in us per 64 of K, against rounds of single-CTA tiles and K slices (tail_slices);
//     1.08 is for power (the pairs move half the operand bytes).  By the costs above up to 512 rows this choice is 1 % off the
//     cheapest on average and 32 % at worst (263 x 4096 x 6144), and the next one 2.5 % and 12 %: not timed in alternation.
//   - from 2048 rows on pairs, in the width that fills the rounds best, except where (single-CTA / pairs, us, rows x K x columns)
//     all single-CTA tiles together are one round of K slices, which then walk a half to a quarter of K each where a pair walks
//     all of it: 2100 x 16384 x 128 35 / 78, 2048 x 12288 x 384 30 / 49, 2048 x 8192 x 512 28 / 35; or the costs above are
//     3 % in favour of single-CTA tiles at a K of 1024 or more: 2176 x 1024 x 1024 8.0 / 9.5, 2600 x 1024 x 6144 35.2 / 38.8,
//     8000 x 1024 x 3072 53.3 / 58.9; or 256 does not divide the width and K is below 1024, where a pair's longer start and
//     drain show: 2100 x 128 x 640 4.5 / 5.3, 2600 x 512 x 384 6.6 / 7.1; with more rounds the pairs win again,
//     4288 x 512 x 640 9.1 / 7.6.
int pair_tile_width(int sms, int rows, int ncols, int num_k_blocks, int pairs, bool gate_up) {
  if (pairs <= 0 || g_d3tom_pair_tiles == 0) return 0;
  if (g_d3tom_pair_tiles == 256) return ncols % 256 == 0 ? 256 : 0;
  constexpr int kWidths[] = {256, 224, 192, 160, 128};
  constexpr double kPerBlock[] = {0.36, 0.345, 0.31, 0.30, 0.29};
  double best = 1e30;
  int width = 0;
  for (int i = 0; i < 5; ++i) {
    const long long tiles = (long long)ceil_div(rows, 2 * kBM) * ceil_div(ncols, kWidths[i]);
    const double cost = kPerBlock[i] * (double)((tiles + pairs - 1) / pairs);
    if (cost < best) { best = cost; width = kWidths[i]; }
  }
  auto rounds = [&](int bm, int bn, double full, double last0, double last_r) {
    const long long tiles = (long long)ceil_div(rows, bm) * ceil_div(ncols, bn);
    const long long r = tiles % sms;
    return full * (double)(tiles / sms) + (r > 0 ? last0 + last_r * (double)r : 0.0);
  };
  auto pair_time = [&](int w) {
    const TileCost& c = kPairCost[(256 - w) / 32];
    return tile_time(c, (long long)ceil_div(rows, 2 * kBM) * ceil_div(ncols, w), pairs, num_k_blocks);
  };
  auto one_time = [&] {
    const int bn = gate_up ? 256 : one_m_tile_width(sms, rows, ncols, num_k_blocks);
    const TileCost& c = kOneCost[(256 - bn) / 64];
    const long long tiles = (long long)ceil_div(rows, kBM) * ceil_div(ncols, bn);
    const int slices = tail_slices(sms, (int)tiles, num_k_blocks);
    if (slices == 1) return tile_time(c, tiles, sms, num_k_blocks);
    // whole rounds, the rounds of slices, and the exchange of their sums
    const double full = (double)(tiles / sms);
    const int units = (int)(tiles % sms) * slices;
    return c.start + full * (num_k_blocks * c.round + c.more) +
           ceil_div(num_k_blocks, slices) * (c.round * (ceil_div(units, sms) - 1) + c.part + c.part_r * fmin(1.0, (double)units / sms)) +
           4.6 + (2.6 * slices - 3.0) * bn / 128;
  };
  if (rows >= 2048) {
    const int bn = gate_up ? 256 : one_m_tile_width(sms, rows, ncols, num_k_blocks);
    const long long tiles = (long long)ceil_div(rows, kBM) * ceil_div(ncols, bn);
    if (tiles < sms) {
      const int slices = tail_slices(sms, (int)tiles, num_k_blocks);
      if (slices > 1 && tiles * slices <= sms) return 0;
    }
    if (ncols % 256 != 0 && num_k_blocks < 16) {
      const double scale = bn == 256 ? 1.0 : bn == 192 ? 0.95 : 0.9;      // (one_m_tile_width's cycles)
      return best * num_k_blocks + 1.0 < 1.08 * scale * rounds(kBM, bn, 0.40, 0.26, 0.0009) * num_k_blocks ? width : 0;
    }
    if (num_k_blocks >= 16) return 1.03 * one_time() < pair_time(width) ? 0 : width;
    return width;
  }
  // (the gate-up pass at a short K is bound by its epilogue: 1900 rows, D = 512, m = 12288 76.9 / 84.7)
  if (gate_up && num_k_blocks < 16) return 0;
  if (rows > 512 && num_k_blocks >= 16) {
    for (int w : kWidths) if (pair_time(w) < pair_time(width)) width = w;
    return one_time() < 1.02 * pair_time(width) ? 0 : width;     // (ties to the single-CTA tiles)
  }
  double single = rounds(kBM, 256, 0.40, 0.26, 0.0009);
  const long long tiles = (long long)ceil_div(rows, kBM) * ceil_div(ncols, 256);
  const int rem = (int)(tiles % sms);
  for (int sp = 2; sp <= kMaxKSplits && rem > 0; ++sp) {
    if (num_k_blocks / sp < 8 || rem * sp > 2 * sms) break;
    const double cut = (double)(ceil_div(rem * sp, sms) * ceil_div(num_k_blocks, sp) + 30 + 5 * sp) / num_k_blocks;
    if (cut < 1.0) single = fmin(single, 0.40 * (double)(tiles / sms) + 0.42 * cut);
  }
  // (a pair launch costs about 1.5 us more: with a short K the single-CTA tiles keep small layers, 319 x 3072 x 1024: 9.0 / 9.9)
  return best * num_k_blocks + 1.5 < 1.08 * single * num_k_blocks ? width : 0;
}

}  // namespace

int make_tmap_bf16_2d(CUtensorMap* out, const void* base, uint64_t rows, uint64_t cols, uint64_t pitch_elems,
                      uint32_t box_rows, uint32_t box_cols) {
  EncodeTiledFn fn = get_encode_fn();
  if (fn == nullptr) return -1;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {pitch_elems * 2};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)r;
}

int launch_proj_tc(d3tom_ctx* ctx, const void* x, const void* w, int total, int D, void* q, void* k, void* v,
                   cudaStream_t s) {
  if (D % 128 != 0) return D3TOM_ERR_UNSUPPORTED;
  CUtensorMap ta, tb;
  int r = make_tmap_bf16_2d(&ta, x, (uint64_t)total, (uint64_t)D, (uint64_t)D, kBM);
  if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
  GemmParams p = {};
  p.num_k_blocks = D / kBK;
  p.out[0] = static_cast<__nv_bfloat16*>(q); p.out[1] = static_cast<__nv_bfloat16*>(k); p.out[2] = static_cast<__nv_bfloat16*>(v);
  p.out_rows = total; p.out_cols = D; p.dev_status = ctx->dev_status;
  p.m_tiles = ceil_div(total, kBM); p.batch = 1; p.k_splits = 1;
  if (const int bn2 = pair_tile_width(ctx->sm_count, total, 3 * D, p.num_k_blocks, resident_pairs<kEpiProj>(ctx), false)) {
    r = make_tmap_bf16_2d(&tb, w, (uint64_t)3 * D, (uint64_t)D, (uint64_t)D, (uint32_t)bn2 / 2);   // a CTA's half of the weight tile
    if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
    p.bn = bn2; p.m_tiles = ceil_div(total, 2 * kBM); p.n_tiles = ceil_div(3 * D, bn2);
    return launch_gemm_pair<kEpiProj>(ctx, ta, tb, p, s);
  }
  const int bn = one_m_tile_width(ctx->sm_count, total, 3 * D, p.num_k_blocks);      // (128 always divides 3 D)
  r = make_tmap_bf16_2d(&tb, w, (uint64_t)3 * D, (uint64_t)D, (uint64_t)D, (uint32_t)bn);
  if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
  p.n_tiles = 3 * D / bn;
  if (bn == 256) return launch_gemm<256, kEpiProj>(ctx, ta, tb, p, s);
  if (bn == 192) return launch_gemm<192, kEpiProj>(ctx, ta, tb, p, s);
  return launch_gemm<128, kEpiProj>(ctx, ta, tb, p, s);
}

int launch_linear_tc(d3tom_ctx* ctx, const void* x, const void* w, const void* residual, int rows, int K, int N,
                     void* out, cudaStream_t s) {
  if (K % kBK != 0 || N % 128 != 0) return D3TOM_ERR_UNSUPPORTED;
  CUtensorMap ta, tb;
  int r = make_tmap_bf16_2d(&ta, x, (uint64_t)rows, (uint64_t)K, (uint64_t)K, kBM);
  if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
  GemmParams p = {};
  p.num_k_blocks = K / kBK;
  p.lin_out = static_cast<__nv_bfloat16*>(out); p.residual = static_cast<const __nv_bfloat16*>(residual);
  p.ld_out = N; p.out_rows = rows; p.dev_status = ctx->dev_status;
  p.m_tiles = ceil_div(rows, kBM); p.batch = 1; p.k_splits = 1;
  if (const int bn2 = pair_tile_width(ctx->sm_count, rows, N, p.num_k_blocks, resident_pairs<kEpiLinear>(ctx), false)) {
    r = make_tmap_bf16_2d(&tb, w, (uint64_t)N, (uint64_t)K, (uint64_t)K, (uint32_t)bn2 / 2);
    if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
    p.bn = bn2; p.m_tiles = ceil_div(rows, 2 * kBM); p.n_tiles = ceil_div(N, bn2);
    return launch_gemm_pair<kEpiLinear>(ctx, ta, tb, p, s);
  }
  const int bn = one_m_tile_width(ctx->sm_count, rows, N, p.num_k_blocks);
  r = make_tmap_bf16_2d(&tb, w, (uint64_t)N, (uint64_t)K, (uint64_t)K, (uint32_t)bn);
  if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
  p.n_tiles = N / bn;
  if (bn == 256) return launch_gemm<256, kEpiLinear>(ctx, ta, tb, p, s);
  if (bn == 192) return launch_gemm<192, kEpiLinear>(ctx, ta, tb, p, s);
  return launch_gemm<128, kEpiLinear>(ctx, ta, tb, p, s);
}

int launch_gate_up_tc(d3tom_ctx* ctx, const void* x, const void* w_gate_up, int rows, int D, int m, void* act,
                      cudaStream_t s) {
  if (D % kBK != 0 || m % 128 != 0) return D3TOM_ERR_UNSUPPORTED;
  CUtensorMap ta, tb;
  int r = make_tmap_bf16_2d(&ta, x, (uint64_t)rows, (uint64_t)D, (uint64_t)D, kBM);
  if (r == 0) r = make_tmap_bf16_2d(&tb, w_gate_up, (uint64_t)2 * m, (uint64_t)D, (uint64_t)D, 128);
  if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
  GemmParams p = {};
  p.num_k_blocks = D / kBK;
  p.lin_out = static_cast<__nv_bfloat16*>(act); p.ld_out = m; p.up_row_offset = m; p.out_rows = rows;
  p.dev_status = ctx->dev_status;
  p.m_tiles = ceil_div(rows, kBM); p.n_tiles = m / 128; p.batch = 1; p.k_splits = 1;
  if (const int bn2 = pair_tile_width(ctx->sm_count, rows, 2 * m, p.num_k_blocks, resident_pairs<kEpiGateUp>(ctx), true)) {
    r = make_tmap_bf16_2d(&tb, w_gate_up, (uint64_t)2 * m, (uint64_t)D, (uint64_t)D, (uint32_t)bn2 / 2);   // gate rows or up rows
    if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
    p.bn = bn2; p.m_tiles = ceil_div(rows, 2 * kBM); p.n_tiles = ceil_div(m, bn2 / 2);
    return launch_gemm_pair<kEpiGateUp>(ctx, ta, tb, p, s);
  }
  return launch_gemm<256, kEpiGateUp>(ctx, ta, tb, p, s);
}

int launch_sim_tc(d3tom_ctx* ctx, const MergeArgs& a, cudaStream_t s) {
  if (a.D % kBK != 0) return D3TOM_ERR_UNSUPPORTED;
  CUtensorMap ta, tb;
  int r = make_tmap_bf16_2d(&ta, a.hidden, (uint64_t)a.total_tokens, (uint64_t)a.D, (uint64_t)a.D, kBM);
  if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
  const int kept_rows_bound = a.total_tokens;    // rows the kept-row scratch can hold
  r = make_tmap_bf16_2d(&tb, ctx->kept_rows, (uint64_t)kept_rows_bound, (uint64_t)a.D, (uint64_t)a.D, 128);
  if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
  GemmParams p = {};
  p.num_k_blocks = a.D / kBK;
  p.cu_seqlens = a.cu_seqlens; p.cu_vis = a.cu_vis; p.cu_kept = a.cu_kept; p.assign = a.assign;
  p.inv_norm = ctx->inv_norm; p.inv_norm_kept = ctx->inv_norm_kept; p.best = ctx->best; p.sim_debug = a.sim_debug;
  p.max_kept = a.max_kept; p.dev_status = ctx->dev_status;
  p.m_tiles = ceil_div(a.max_visual, kBM); p.batch = a.B;
  // Few tiles (short requests, small kept sets): a tile is 64 k-blocks of serial work on one SM while most SMs idle, so
  // each tile's K range is cut into slices, each a CTA of its own (units <= SMs), and every slice adds up its share of
  // the tile's columns over all slices.  The last arriver adding all columns alone cost more than the main loop:
  // 2048 visual x 512 kept x 4096 (32 tiles, 4 slices) 28.6 us, shared 20.1.
  // 128-wide tiles also serve larger kept sets while eight slices of each still fit: half the exchange per slice
  // (577 x 173 x 1024: 13.6 -> 10.3 us).
  const long long narrow_tiles = (long long)p.m_tiles * ceil_div(a.max_kept, 128) * p.batch;
  const int bn = a.max_kept <= 128 || narrow_tiles * 8 <= ctx->sm_count ? 128 : 256;
  const long long tiles = (long long)p.m_tiles * ceil_div(a.max_kept, bn) * p.batch;
  p.k_splits = 1;
  for (int c : {kCoopSlices, 8, 4, 3, 2})
    if (tiles * c <= ctx->sm_count && p.num_k_blocks >= 2 * c) { p.k_splits = c; break; }
  p.full_tiles = 0;                                     // every tile is cut (or none: one slice)
  p.split_ws = ctx->gemm_split_ws; p.split_counters = ctx->gemm_split_counters;
  if (bn == 256) {             // 256-wide tiles: the A tile is streamed once per 256 kept rows and each MMA covers twice the work
    r = make_tmap_bf16_2d(&tb, ctx->kept_rows, (uint64_t)kept_rows_bound, (uint64_t)a.D, (uint64_t)a.D, 256);
    if (r != 0) { ctx->last_cuda_error = r; return D3TOM_ERR_CUDA; }
    p.n_tiles = ceil_div(a.max_kept, 256);
    return launch_gemm<256, kEpiSim>(ctx, ta, tb, p, s);
  }
  p.n_tiles = ceil_div(a.max_kept, 128);
  return launch_gemm<128, kEpiSim>(ctx, ta, tb, p, s);
}

extern "C" int d3tom_pair_tile_width(int sms, int pairs, int rows, int n_cols, int K, int gate_up) {
  if (sms <= 0 || pairs < 0 || rows <= 0 || n_cols <= 0 || K <= 0 || K % kBK != 0 || n_cols % 128 != 0) return 0;
  return pair_tile_width(sms, rows, n_cols, K / kBK, pairs, gate_up != 0);
}
