// Bidirectional attention on CUDA cores (fp32 arithmetic) and the importance
// finishing kernel shared with the tensor-core attention.
//
// A warp owns RW (16, 8 or 4) query rows of one (request, head) and visits the keys 32 at a time with an online softmax
// (log2 domain); the NW warps of a CTA share the K and V tiles, which come by asynchronous copies into two stages.  Scores
// and P V run as register tiles out of shared memory (lane layout of f32_tile.cuh); P passes from lane to lane through
// shared memory of the warp.  Every score is one chain of multiply-adds over head_dim, every output one chain over the
// keys, and the row sums are added in the order of a butterfly over 32 keys: the arithmetic does not depend on how rows
// are spread over warps.
// Decider rows additionally write their raw q.k scores over the visual keys to
// the score scratch and their final (M, l) pair to the lse scratch; the
// finishing kernel turns those into S_j = sum_h sum_{i in D} A_ij.
//
// Bound: issue slots and shared memory at one to three warps per scheduler (1152 rows x 8 heads x 64: fp32 pipe 49 % busy,
// issue 58 %, shared-memory wavefronts 66 %).  One warp per query row, every lane walking a key of its own through global
// memory, took 1139 us at 1152 rows x 8 heads x 64 where this takes 83, and 111 us at 288 x 4 x 64 where this takes 11.4.
#include "common.cuh"
#include "f32_tile.cuh"

namespace {

constexpr int kKeyTile = 32;
constexpr int kPStride = kKeyTile + 4;         // floats per row of a warp's P tile (see f32_tile.cuh)

// DHP: head_dim rounded up to 32, 64 or 128 (padding columns are zero)
template <int DHP, int RW, int NW> struct SimtSmem {
  static constexpr int kBM = RW * NW, kLd = DHP + 4;
  static constexpr int kQ = kBM * kLd, kKv = kKeyTile * kLd, kP = NW * RW * kPStride;
  static constexpr int kBytes = (kQ + 4 * kKv + kP) * 4 + kBM * 4;
};

template <int N> struct Rows { static constexpr int value = N; };

template <typename T, int DHP, int RW, int NW>
__global__ void __launch_bounds__(NW * 32)
attn_simt_kernel(AttnArgs a, bool vec) {
  using S = SimtSmem<DHP, RW, NW>;
  constexpr int kLd = S::kLd, kCols = DHP / 32, kR = RW / 4;      // 4-column groups of the output and rows per lane
  extern __shared__ float4 smem_f4[];
  float* q_s = reinterpret_cast<float*>(smem_f4);
  float* kv_s = q_s + S::kQ;                              // stage st: K tile, V tile
  float* p_all = kv_s + 4 * S::kKv;
  int* dec_s = reinterpret_cast<int*>(p_all + S::kP);
  grid_dependency_enter();
  const int b = blockIdx.z, h = blockIdx.y, tid = threadIdx.x;
  const int lo = a.cu_seqlens[b], n = a.cu_seqlens[b + 1] - lo;
  const int q0 = blockIdx.x * S::kBM;
  if (q0 >= n) return;
  const int dh = a.dh;
  const size_t ld = (size_t)a.H * dh;
  const T* qg = static_cast<const T*>(a.q) + (size_t)(lo + q0) * ld + (size_t)h * dh;
  const T* kg = static_cast<const T*>(a.k) + (size_t)lo * ld + (size_t)h * dh;
  const T* vg = static_cast<const T*>(a.v) + (size_t)lo * ld + (size_t)h * dh;
  // `rows` rows from row `r0` of a head's matrix; rows past the request and columns past head_dim become zeros
  constexpr int kVecs = DHP / 4, kStep = NW * 32 / kVecs > 0 ? NW * 32 / kVecs : 1;        // vectors per row, rows per pass of the CTA
  static_assert(NW * 32 >= kVecs, "a pass covers whole rows");
  const int lrow = tid / kVecs, lcol = (tid % kVecs) * 4;
  auto load_rows = [&](auto rows, float* dst, const T* src, int r0, int n_rows) {
    static_assert(decltype(rows)::value % kStep == 0, "every thread loads the same number of vectors");
    src += (size_t)(r0 + lrow) * ld;
    f32::load_vecs<T, decltype(rows)::value / kStep>(dst + lrow * kLd + lcol, kStep * kLd, [&](int u) {
      return f32::RowRef<T>{src + (size_t)u * kStep * ld, r0 + lrow + u * kStep < n_rows};
    }, lcol, dh, vec);
  };
  auto load_tile = [&](int t) {                           // K and V of key tile t, one copy group (empty past the end)
    if (t * kKeyTile < n) {
      float* st = kv_s + (t & 1) * 2 * S::kKv;
      load_rows(Rows<kKeyTile>{}, st, kg, t * kKeyTile, n);
      load_rows(Rows<kKeyTile>{}, st + S::kKv, vg, t * kKeyTile, n);
    }
    f32::cp_async_commit();
  };
  load_rows(Rows<S::kBM>{}, q_s, qg, 0, n - q0);
  load_tile(0);
  load_tile(1);
  // which of the rows are deciders?  (strictly ascending list: binary search)
  int n_vis = 0;
  if (a.decider_pos != nullptr) n_vis = a.n_visual[b];
  for (int row = tid; row < S::kBM; row += NW * 32) {
    int slot = -1;
    if (a.decider_pos != nullptr) {
      int l = a.cu_deciders[b], r = a.cu_deciders[b + 1];
      while (l < r) {
        const int mid = (l + r) >> 1, p = a.decider_pos[mid];
        if (p == q0 + row) { slot = mid; break; }
        if (p < q0 + row) l = mid + 1; else r = mid;
      }
    }
    dec_s[row] = slot;
  }

  const int warp = tid >> 5, lane = tid & 31, ty = f32::lane_ty(lane), tx = f32::lane_tx(lane);
  const float* qw = q_s + warp * RW * kLd + ty * kLd;
  float* pw = p_all + warp * RW * kPStride;
  float m[kR], l[kR];
  float2 o[kR][kCols][2];
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < kCols; ++c) o[r][c][0] = o[r][c][1] = make_float2(0.f, 0.f);
  }
  const int n_tiles = (n + kKeyTile - 1) / kKeyTile;
  for (int t = 0; t < n_tiles; ++t) {
    f32::cp_async_wait<1>();                              // this tile has landed (the next may be on its way)
    __syncthreads();
    const int j0 = t * kKeyTile;
    const float* kw = kv_s + (t & 1) * 2 * S::kKv + tx * kLd;
    const float* vw = kv_s + (t & 1) * 2 * S::kKv + S::kKv + tx * 4;
    float s[kR][4];
#pragma unroll
    for (int r = 0; r < kR; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) s[r][j] = 0.f;
    {
      float4 av[2][kR], bv[2][4];
      auto fetch = [&](int buf, int k) {
#pragma unroll
        for (int r = 0; r < kR; ++r) av[buf][r] = *reinterpret_cast<const float4*>(qw + r * 4 * kLd + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) bv[buf][j] = *reinterpret_cast<const float4*>(kw + j * 8 * kLd + k);
      };
      fetch(0, 0);
#pragma unroll
      for (int k = 0; k < DHP; k += 4) {                  // the next step's operands are read while this step multiplies
        const int bf = (k >> 2) & 1;
        if (k + 4 < DHP) fetch(bf ^ 1, k + 4);
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int r = 0; r < kR; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 x = av[bf][r], y = bv[bf][j];
              s[r][j] = e == 0 ? fmaf(x.x, y.x, s[r][j]) : e == 1 ? fmaf(x.y, y.y, s[r][j]) : e == 2 ? fmaf(x.z, y.z, s[r][j])
                                                                                          : fmaf(x.w, y.w, s[r][j]);
            }
      }
    }
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const int row = ty + 4 * r;
      const int slot = dec_s[warp * RW + row];
      float mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int key = j0 + tx + 8 * j;
        if (slot >= 0 && key < n_vis) a.score_scratch[((size_t)h * a.max_deciders + slot) * a.vis_stride + key] = s[r][j];
        s[r][j] = key < n ? __fmul_rn(s[r][j], a.scale_log2) : -INFINITY;
        mx = fmaxf(mx, s[r][j]);
      }
      const float m_new = fmaxf(m[r], f32::max_over_tx(mx));
      const float corr = exp2f(m[r] - m_new);             // first tile: exp2(-inf) = 0
      float p[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        p[j] = j0 + tx + 8 * j < n ? exp2f(__fsub_rn(s[r][j], m_new)) : 0.f;
        pw[row * kPStride + tx + 8 * j] = p[j];
      }
      l[r] = fmaf(l[r], corr, f32::sum_over_tx((p[0] + p[2]) + (p[1] + p[3])));
      m[r] = m_new;
#pragma unroll
      for (int c = 0; c < kCols; ++c)
#pragma unroll
        for (int e = 0; e < 2; ++e) { o[r][c][e].x *= corr; o[r][c][e].y *= corr; }
    }
    __syncwarp();
    float4 p4[2][kR], v4[2][kCols];
    auto fetch_p = [&](int buf, int k) {
#pragma unroll
      for (int r = 0; r < kR; ++r) p4[buf][r] = *reinterpret_cast<const float4*>(pw + (ty + 4 * r) * kPStride + k);
    };
    auto fetch_v = [&](int buf, int k) {
#pragma unroll
      for (int c = 0; c < kCols; ++c) v4[buf][c] = *reinterpret_cast<const float4*>(vw + k * kLd + c * 32);
    };
    fetch_p(0, 0);
    fetch_v(0, 0);
#pragma unroll
    for (int k = 0; k < kKeyTile; ++k) {                  // the next step's operands are read while this step multiplies
      const int pb = (k >> 2) & 1, vb = k & 1;
      if ((k & 3) == 0 && k + 4 < kKeyTile) fetch_p(pb ^ 1, k + 4);
      if (k + 1 < kKeyTile) fetch_v(vb ^ 1, k + 1);
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        const float4 p = p4[pb][r];
        const float pk = (k & 3) == 0 ? p.x : (k & 3) == 1 ? p.y : (k & 3) == 2 ? p.z : p.w;
        const float2 pp = make_float2(pk, pk);
#pragma unroll
        for (int c = 0; c < kCols; ++c) {
          o[r][c][0] = __ffma2_rn(pp, make_float2(v4[vb][c].x, v4[vb][c].y), o[r][c][0]);
          o[r][c][1] = __ffma2_rn(pp, make_float2(v4[vb][c].z, v4[vb][c].w), o[r][c][1]);
        }
      }
    }
    __syncthreads();                                      // everyone is done with this stage
    load_tile(t + 2);
  }
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    const int row = warp * RW + ty + 4 * r;
    if (q0 + row >= n) continue;
    const float inv_l = 1.f / l[r];
    T* dst = static_cast<T*>(a.out) + (size_t)(lo + q0 + row) * ld + (size_t)h * dh;
#pragma unroll
    for (int c = 0; c < kCols; ++c) {
      const int col = c * 32 + tx * 4;
      if (col >= dh) continue;
      const float y[4] = {o[r][c][0].x * inv_l, o[r][c][0].y * inv_l, o[r][c][1].x * inv_l, o[r][c][1].y * inv_l};
      if (sizeof(T) == 4 && vec) {
        *reinterpret_cast<float4*>(dst + col) = make_float4(y[0], y[1], y[2], y[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) dst[col + e] = Storage<T>::from_float(y[e]);
      }
    }
    if (tx == 0 && dec_s[row] >= 0) a.lse_scratch[(size_t)h * a.max_deciders + dec_s[row]] = make_float2(m[r], l[r]);
  }
}

// One block = (256 visual keys, head, request).
//   partial[h][cu_vis[b] + j] = sum over the request's deciders (ascending) of exp2(score * c - M) / l
// The last of the H blocks of a key range to finish (a counter per range, left at zero again
// afterwards) adds the H partials in ascending head order:
//   importance[g] = sum over heads of partial[h][g]
// so the result does not depend on which block that is: no float atomics, reproducible.
constexpr int kImpThreads = 256;
constexpr int kImpDecChunk = 128;
// Up to this many heads and deciders one block per 32 keys (below).  One request, attention + importance, partial sums / one pass
// (us), by deciders at 1024 keys x 4 heads x 64 fp32: 4 64.3 / 61.0, 8 65.0 / 61.4, 16 64.4 / 62.5, 32 64.9 / 64.4, 64 67.6 / 68.9;
// 256 keys x 4: 8 19.5 / 15.8, 16 18.7 / 16.9, 64 19.7 / 22.0; 12000 keys x 4 bf16: 8 232 / 227, 16 232 / 229, 64 284 / 285;
// 256 keys x 8: 8 26.8 / 22.5, 16 25.0 / 23.7, 64 27.2 / 29.0.  With many heads (1024 keys x 32, 32 deciders 47.2 / 53.1) a block's
// 128-byte pieces of many rows are the longer way to the same bytes.
constexpr int kImpBlockDeciders = 16;
constexpr int kImpBlockHeads = 8;
constexpr int kImpBlockLoads = 8;      // scores in flight per lane

__global__ void __launch_bounds__(kImpThreads)
importance_finish_kernel(const float* __restrict__ score, const float2* __restrict__ lse,
                         const int32_t* __restrict__ n_visual, const int32_t* __restrict__ cu_deciders,
                         const int32_t* __restrict__ cu_vis, int max_deciders, int vis_stride, float scale_log2,
                         float* __restrict__ partial, int partial_stride, int H, int* __restrict__ counters,
                         float* __restrict__ importance) {
  grid_dependency_enter();
  const int b = blockIdx.z, h = blockIdx.y;
  const int Vb = n_visual[b];
  if ((int)blockIdx.x * kImpThreads >= Vb) return;              // uniform: no key of this request in the range
  const int j = blockIdx.x * kImpThreads + threadIdx.x;
  const int d0 = cu_deciders[b], d1 = cu_deciders[b + 1];
  __shared__ float neg_m[kImpDecChunk], inv_l[kImpDecChunk];
  __shared__ int is_last;
  const int jj = j < Vb ? j : Vb - 1;                           // threads past the end read a valid column, write nothing
  float acc = 0.f;
  for (int dc = d0; dc < d1; dc += kImpDecChunk) {
    const int nd = min(kImpDecChunk, d1 - dc);
    __syncthreads();
    if (threadIdx.x < nd) {
      const float2 ml = lse[(size_t)h * max_deciders + dc + threadIdx.x];
      neg_m[threadIdx.x] = -ml.x;
      inv_l[threadIdx.x] = 1.0f / ml.y;
    }
    __syncthreads();
    const float* col = score + ((size_t)h * max_deciders + dc) * vis_stride + jj;
    // (the loads of 16 deciders are in flight together; the sum still runs in ascending decider order)
#pragma unroll 16
    for (int d = 0; d < nd; ++d)
      acc = fmaf(exp2f(fmaf(col[(size_t)d * vis_stride], scale_log2, neg_m[d])), inv_l[d], acc);
  }
  const int g0 = cu_vis[b];
  if (j < Vb) partial[(size_t)h * partial_stride + g0 + j] = acc;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    int* ctr = counters + (size_t)b * gridDim.x + blockIdx.x;
    const int prev = atomicAdd(ctr, 1);
    is_last = prev == H - 1;
    if (is_last) *ctr = 0;                                      // ready for the next call
  }
  __syncthreads();
  if (is_last && j < Vb) {
    __threadfence();
    float tot = 0.f;
#pragma unroll 8
    for (int hh = 0; hh < H; ++hh) tot += __ldcg(partial + (size_t)hh * partial_stride + g0 + j);
    importance[g0 + j] = tot;
  }
}

// The same sums in one pass: one block = 32 visual keys of a request, one warp per head; the heads meet in shared memory.  Two
// dependent rounds of loads instead of five (no partials through global memory, no counter): what a small call costs is that
// chain.
__global__ void __launch_bounds__(32 * kImpBlockHeads)
importance_finish_block_kernel(const float* __restrict__ score, const float2* __restrict__ lse,
                        const int32_t* __restrict__ n_visual, const int32_t* __restrict__ cu_deciders,
                        const int32_t* __restrict__ cu_vis, int max_deciders, int vis_stride, float scale_log2, int H,
                        float* __restrict__ importance) {
  __shared__ float part[kImpBlockHeads][32];
  grid_dependency_wait();
  // (a batch keeps the next kernel back until it ends: blocks of an fp32 attention launch that came in beside this kernel's many
  // small ones piled up on some SMs, eight requests x 1 head x 64 called back to back 150 -> 257 us, 160 so)
  if (gridDim.y == 1) grid_dependency_release();
  const int b = blockIdx.y, h = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Vb = n_visual[b], j = blockIdx.x * 32 + lane;
  const int d0 = cu_deciders[b], d1 = cu_deciders[b + 1], g0 = cu_vis[b];
  if ((int)blockIdx.x * 32 >= Vb) return;                       // uniform: no key of this request in the range
  const int jj = j < Vb ? j : Vb - 1;                           // lanes past the end read a valid column, write nothing
  float acc = 0.f;
  // (the host's count chose this kernel, the device's list is what is summed: a captured call may be replayed with a longer one)
  for (int d = d0; d < d1; d += kImpBlockLoads) {
    const int nd = min(kImpBlockLoads, d1 - d);
    const float2 ml = lane < nd ? lse[(size_t)h * max_deciders + d + lane] : make_float2(0.f, 1.f);
    const float neg_m = -ml.x, inv_l = 1.0f / ml.y;
    const float* col = score + ((size_t)h * max_deciders + d) * vis_stride + jj;
    float x[kImpBlockLoads];                                    // (all loads in flight; the sum runs in ascending order)
#pragma unroll
    for (int u = 0; u < kImpBlockLoads; ++u) if (u < nd) x[u] = col[(size_t)u * vis_stride];
#pragma unroll
    for (int u = 0; u < kImpBlockLoads; ++u)
      if (u < nd)
        acc = fmaf(exp2f(fmaf(x[u], scale_log2, __shfl_sync(0xffffffffu, neg_m, u))), __shfl_sync(0xffffffffu, inv_l, u), acc);
  }
  part[h][lane] = acc;
  __syncthreads();
  if (h == 0 && j < Vb) {
    float tot = 0.f;
    for (int hh = 0; hh < H; ++hh) tot += part[hh][lane];
    importance[g0 + j] = tot;
  }
}

}  // namespace

namespace {

template <typename T, int DHP, int RW, int NW>
int launch_simt(d3tom_ctx* ctx, const AttnArgs& a, cudaStream_t s) {
  using S = SimtSmem<DHP, RW, NW>;
  // copies and stores of four elements where the caller's buffers allow them (head_dim is a multiple of 4)
  const uintptr_t bits = (uintptr_t)a.q | (uintptr_t)a.k | (uintptr_t)a.v | (uintptr_t)a.out;
  const bool vec = bits % (4 * sizeof(T)) == 0;
  dim3 grid(ceil_div(a.max_seqlen, S::kBM), a.H, a.B);
  const int smem = spread_smem(ctx, grid, S::kBytes, 4);
  // (the attribute belongs to the current device: set on every call, a process may drive several GPUs; always to the same
  // value, since another thread may be launching with another size)
  D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(attn_simt_kernel<T, DHP, RW, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  D3TOM_CUDA_TRY(ctx, launch_serialized(attn_simt_kernel<T, DHP, RW, NW>, grid, NW * 32, smem, s, a, vec));
  return D3TOM_OK;
}

// Rows per warp: 8, or 4 where there are so few warps that most schedulers would idle (up to two eight-row warps per SM),
// or 16 for rows of up to 32 channels once the SMs are full of warps (from 16 eight-row warps per SM on): there a score's
// shared-memory reads weigh most and sixteen rows share them.  Measured, 4 / 8 / 16 rows (us): 288 rows x 4 heads x 64
// 11.4 / 16.7 / 29.2; 500 x 4 x 64 19.3 / 28.1 / 51.8; 600 x 4 x 64 35.6 / 32.9 / 63.3; 1152 x 8 x 64 111 / 82.6 / 132;
// with 16 eight-row warps per SM and more, 8 / 16: 2400 x 8 x 64 396 / 438, 1152 x 32 x 128 614 / 665, 2400 x 8 x 128
// 785 / 929, 2400 x 8 x 32 290 / 252.
template <typename T, int DHP>
int launch_simt_dh(d3tom_ctx* ctx, const AttnArgs& a, cudaStream_t s) {
  const long long sms = ctx->sm_count > 0 ? ctx->sm_count : 148;
  const long long warps8 = (long long)ceil_div(a.max_seqlen, 8) * a.H * a.B;
  if (warps8 <= 2 * sms) return launch_simt<T, DHP, 4, 4>(ctx, a, s);
  if constexpr (DHP == 32) {
    if (warps8 > 16 * sms) return launch_simt<T, DHP, 16, 4>(ctx, a, s);
  }
  return launch_simt<T, DHP, 8, 4>(ctx, a, s);
}

template <typename T>
int launch_simt_t(d3tom_ctx* ctx, const AttnArgs& a, cudaStream_t s) {
  if (a.dh > 64) return launch_simt_dh<T, 128>(ctx, a, s);
  return a.dh > 32 ? launch_simt_dh<T, 64>(ctx, a, s) : launch_simt_dh<T, 32>(ctx, a, s);
}

}  // namespace

int launch_attn_simt(d3tom_ctx* ctx, d3tom_dtype dt, const AttnArgs& a, cudaStream_t s) {
  if (dt == D3TOM_FP32) return launch_simt_t<float>(ctx, a, s);
  return launch_simt_t<__nv_bfloat16>(ctx, a, s);
}

int launch_importance_finish(d3tom_ctx* ctx, const AttnArgs& a, int n_deciders, int max_visual, float* importance,
                             const int32_t* cu_vis, cudaStream_t s) {
  if (max_visual <= 0) return D3TOM_OK;
  if (a.H <= kImpBlockHeads && n_deciders <= kImpBlockDeciders) {
    D3TOM_CUDA_TRY(ctx, launch_serialized(importance_finish_block_kernel, dim3(ceil_div(max_visual, 32), a.B), a.H * 32, 0, s,
                                          a.score_scratch, a.lse_scratch, a.n_visual, a.cu_deciders, cu_vis, a.max_deciders,
                                          a.vis_stride, a.scale_log2, a.H, importance));
    return D3TOM_OK;
  }
  dim3 grid(ceil_div(max_visual, kImpThreads), a.H, a.B);
  D3TOM_CUDA_TRY(ctx, launch_serialized(importance_finish_kernel, grid, kImpThreads, 0, s, a.score_scratch, a.lse_scratch,
                                        a.n_visual, a.cu_deciders, cu_vis, a.max_deciders, a.vis_stride, a.scale_log2,
                                        ctx->imp_partial, ctx->lim.max_total_tokens, a.H, ctx->imp_counters, importance));
  return D3TOM_OK;
}
