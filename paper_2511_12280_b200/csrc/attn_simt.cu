// Bidirectional attention on CUDA cores (fp32 arithmetic) and the importance
// finishing kernel shared with the tensor-core attention.
//
// One CTA owns BM = 128 / KG query rows of one (request, head) and visits the keys 32 KG at a time.  Its 8 warps are
// 8 / KG row groups of 16 rows times KG key groups of 32 keys: a warp runs the online softmax (log2 domain) of its
// own 16 rows over its own keys, and the KG partial results (m, l, O) of a row are combined once at the end, in key
// group order.  Scores and P V both run as 16 x 32 register tiles out of shared memory (f32_tile.cuh); P passes from
// lane to lane through 2 KB of shared memory per warp.  K and V have one buffer each: the next K tile is copied while
// the softmax and P V of this one run, the next V tile under the next scores.
//
// Bound: the fp32 pipe and the latency of one or two warps per scheduler (FMA pipe about half busy).  One warp per
// query row, every lane walking a key of its own through global memory, took 1139 us at 1152 rows x 8 heads x 64 where
// this takes 82, and 111 us at 288 x 4 x 64 where this takes 14.
//
// Decider rows additionally write their raw q.k scores over the visual keys to
// the score scratch and their final (M, l) pair to the lse scratch; the
// finishing kernel turns those into S_j = sum_h sum_{i in D} A_ij.
#include "common.cuh"
#include "f32_tile.cuh"

namespace {

constexpr int kSimtWarps = 8;
constexpr int kPStride = 36;         // floats per row of a warp's P tile (32 + 4: see f32_tile.cuh)

// DHP: head_dim rounded up to 32, 64 or 128 (padding columns are zero); KG: key groups
template <int DHP, int KG> struct SimtSmem {
  static constexpr int kBM = 128 / KG, kKeys = 32 * KG, kLd = DHP + 4;
  static constexpr int kQ = kBM * kLd, kK = kKeys * kLd, kP = kSimtWarps * 16 * kPStride;
  static constexpr int kBytes = (kQ + 2 * kK + kP) * 4 + kBM * 4;
  static_assert(2 * kK >= 128 * DHP, "the partial outputs of all key groups are combined in the K and V buffers");
};

template <typename T, int DHP, int KG>
__global__ void __launch_bounds__(kSimtWarps * 32, 1)
attn_simt_kernel(AttnArgs a, bool vec) {
  using S = SimtSmem<DHP, KG>;
  constexpr int kLd = S::kLd, kCols = DHP / 32;         // 4-column groups of the output per lane
  extern __shared__ float4 smem_f4[];
  float* q_s = reinterpret_cast<float*>(smem_f4);
  float* k_s = q_s + S::kQ;
  float* v_s = k_s + S::kK;
  float* p_all = v_s + S::kK;
  int* dec_s = reinterpret_cast<int*>(p_all + S::kP);
  grid_dependency_enter();
  const int b = blockIdx.z, h = blockIdx.y, tid = threadIdx.x;
  const int lo = a.cu_seqlens[b], n = a.cu_seqlens[b + 1] - lo;
  const int q0 = blockIdx.x * S::kBM;
  if (q0 >= n) return;
  const int H = a.H, dh = a.dh;
  const size_t ld = (size_t)H * dh;
  const T* qg = static_cast<const T*>(a.q) + (size_t)(lo + q0) * ld + (size_t)h * dh;
  const T* kg = static_cast<const T*>(a.k) + (size_t)lo * ld + (size_t)h * dh;
  const T* vg = static_cast<const T*>(a.v) + (size_t)lo * ld + (size_t)h * dh;
  // `rows` rows from row `r0` of a head's matrix; rows past the request and columns past head_dim become zeros
  constexpr int kVecs = DHP / 4, kStep = kSimtWarps * 32 / kVecs;        // vectors per row, rows per pass of the block
  const int lrow = tid / kVecs, lcol = (tid % kVecs) * 4;
  auto load_rows = [&](float* dst, const T* src, int r0, int rows, int n_rows) {
    dst += lrow * kLd + lcol;
    src += (size_t)(r0 + lrow) * ld;
    for (int r = lrow; r < rows; r += kStep, dst += kStep * kLd, src += kStep * ld)
      f32::load4<T>(dst, src, lcol, dh, r0 + r < n_rows, vec);
  };
  load_rows(q_s, qg, 0, S::kBM, n - q0);
  load_rows(k_s, kg, 0, S::kKeys, n);
  f32::cp_async_commit();
  load_rows(v_s, vg, 0, S::kKeys, n);
  f32::cp_async_commit();
  // which of the rows are deciders?  (strictly ascending list: binary search)
  int n_vis = 0;
  if (a.decider_pos != nullptr) n_vis = a.n_visual[b];
  if (tid < S::kBM) {
    int slot = -1;
    if (a.decider_pos != nullptr) {
      int l = a.cu_deciders[b], r = a.cu_deciders[b + 1];
      while (l < r) {
        const int mid = (l + r) >> 1, p = a.decider_pos[mid];
        if (p == q0 + tid) { slot = mid; break; }
        if (p < q0 + tid) l = mid + 1; else r = mid;
      }
    }
    dec_s[tid] = slot;
  }

  const int warp = tid >> 5, lane = tid & 31, ty = f32::lane_ty(lane), tx = f32::lane_tx(lane);
  const int rg = warp / KG, key_g = warp - rg * KG;     // row group, key group
  const float* qw = q_s + rg * 16 * kLd;
  const float* kw = k_s + key_g * 32 * kLd;
  const float* vw = v_s + key_g * 32 * kLd;
  float* pw = p_all + warp * 16 * kPStride;
  float m[4], l[4];
  float2 o[4][kCols][2];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < kCols; ++c) o[r][c][0] = o[r][c][1] = make_float2(0.f, 0.f);
  }
  for (int j0 = 0; j0 < n; j0 += S::kKeys) {
    const int key0 = j0 + key_g * 32;
    const bool live = key0 < n;                         // (whole warp)
    f32::cp_async_wait<1>();                            // K has landed (V may be on its way)
    __syncthreads();
    float2 s2[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) s2[r][j] = make_float2(0.f, 0.f);
    if (live) f32::dot_16x32<kLd, kLd, DHP / 4>(s2, qw, kw, ty, tx);
    __syncthreads();                                    // everyone is done with this K tile
    if (j0 + S::kKeys < n) load_rows(k_s, kg, j0 + S::kKeys, S::kKeys, n);
    f32::cp_async_commit();
    if (live) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int row = ty + 4 * r;
        const int slot = dec_s[rg * 16 + row];
        float s[4];
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int key = key0 + tx + 8 * j;
          const float raw = s2[r][j].x + s2[r][j].y;
          if (slot >= 0 && key < n_vis) a.score_scratch[((size_t)h * a.max_deciders + slot) * a.vis_stride + key] = raw;
          s[j] = key < n ? raw * a.scale_log2 : -INFINITY;
          mx = fmaxf(mx, s[j]);
        }
        const float m_new = fmaxf(m[r], f32::max_over_tx(mx));
        const float corr = exp2f(m[r] - m_new);         // first tile: exp2(-inf) = 0
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float p = key0 + tx + 8 * j < n ? exp2f(s[j] - m_new) : 0.f;
          pw[row * kPStride + tx + 8 * j] = p;
          sum += p;
        }
        l[r] = fmaf(l[r], corr, sum);                   // this lane's keys only; the lanes are added up at the end
        m[r] = m_new;
#pragma unroll
        for (int c = 0; c < kCols; ++c)
#pragma unroll
          for (int e = 0; e < 2; ++e) { o[r][c][e].x *= corr; o[r][c][e].y *= corr; }
      }
    }
    f32::cp_async_wait<1>();                            // V has landed (the next K may be on its way)
    __syncthreads();
    if (live) {
      float4 p4[2][4], v4[2][kCols];
      auto fetch_p = [&](int buf, int k) {
#pragma unroll
        for (int r = 0; r < 4; ++r) p4[buf][r] = *reinterpret_cast<const float4*>(pw + (ty + 4 * r) * kPStride + k);
      };
      auto fetch_v = [&](int buf, int k) {
#pragma unroll
        for (int c = 0; c < kCols; ++c) v4[buf][c] = *reinterpret_cast<const float4*>(vw + k * kLd + c * 32 + tx * 4);
      };
      fetch_p(0, 0);
      fetch_v(0, 0);
#pragma unroll
      for (int k = 0; k < 32; ++k) {                    // the next step's operands are read while this step multiplies
        const int pb = (k >> 2) & 1, vb = k & 1;
        if ((k & 3) == 0 && k + 4 < 32) fetch_p(pb ^ 1, k + 4);
        if (k + 1 < 32) fetch_v(vb ^ 1, k + 1);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
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
    }
    __syncthreads();                                    // everyone is done with this V tile (and this P)
    if (j0 + S::kKeys < n) load_rows(v_s, vg, j0 + S::kKeys, S::kKeys, n);
    f32::cp_async_commit();
  }
  // ---- the KG partial results of every row, in key group order: [KG][BM][DHP] outputs and (m, l) pairs
  float* o_s = k_s;
  float2* ml_s = reinterpret_cast<float2*>(p_all);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int slot = key_g * S::kBM + rg * 16 + ty + 4 * r;
    const float sum = f32::sum_over_tx(l[r]);
    if (tx == 0) ml_s[slot] = make_float2(m[r], sum);
#pragma unroll
    for (int c = 0; c < kCols; ++c)
      *reinterpret_cast<float4*>(o_s + (size_t)slot * DHP + c * 32 + tx * 4) =
          make_float4(o[r][c][0].x, o[r][c][0].y, o[r][c][1].x, o[r][c][1].y);
  }
  __syncthreads();
  T* out = static_cast<T*>(a.out) + (size_t)(lo + q0) * ld + (size_t)h * dh;
  for (int i = tid; i < S::kBM * (DHP / 4); i += kSimtWarps * 32) {
    const int r = i / (DHP / 4), c = (i - r * (DHP / 4)) * 4;
    if (q0 + r >= n || c >= dh) continue;
    float mm = ml_s[r].x;
#pragma unroll
    for (int g = 1; g < KG; ++g) mm = fmaxf(mm, ml_s[g * S::kBM + r].x);
    float lsum = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int g = 0; g < KG; ++g) {
      const float2 ml = ml_s[g * S::kBM + r];
      const float w = exp2f(ml.x - mm);                 // a key group without keys: exp2(-inf) = 0
      const float4 x = *reinterpret_cast<const float4*>(o_s + (size_t)(g * S::kBM + r) * DHP + c);
      lsum = fmaf(ml.y, w, lsum);
      acc.x = fmaf(x.x, w, acc.x); acc.y = fmaf(x.y, w, acc.y); acc.z = fmaf(x.z, w, acc.z); acc.w = fmaf(x.w, w, acc.w);
    }
    const float inv_l = 1.f / lsum;
    const float y[4] = {acc.x * inv_l, acc.y * inv_l, acc.z * inv_l, acc.w * inv_l};
    T* dst = out + (size_t)r * ld + c;
    if (sizeof(T) == 4 && vec) {
      *reinterpret_cast<float4*>(dst) = make_float4(y[0], y[1], y[2], y[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) dst[e] = Storage<T>::from_float(y[e]);
    }
    if (c == 0 && dec_s[r] >= 0) a.lse_scratch[(size_t)h * a.max_deciders + dec_s[r]] = make_float2(mm, lsum);
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

}  // namespace

namespace {

template <typename T, int DHP, int KG>
int launch_simt(d3tom_ctx* ctx, const AttnArgs& a, cudaStream_t s) {
  using S = SimtSmem<DHP, KG>;
  // 16-byte copies and stores where the caller's buffers allow them (head_dim is a multiple of 4)
  const uintptr_t bits = (uintptr_t)a.q | (uintptr_t)a.k | (uintptr_t)a.v | (uintptr_t)a.out;
  const bool vec = sizeof(T) == 4 && bits % 16 == 0;
  dim3 grid(ceil_div(a.max_seqlen, S::kBM), a.H, a.B);
  // (the attribute belongs to the current device: set on every call, a process may drive several GPUs)
  D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(attn_simt_kernel<T, DHP, KG>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kBytes));
  D3TOM_CUDA_TRY(ctx, launch_serialized(attn_simt_kernel<T, DHP, KG>, grid, kSimtWarps * 32, S::kBytes, s, a, vec));
  return D3TOM_OK;
}

// Rows per CTA (128 / KG): the fewest rounds of CTAs over the SMs times key blocks per CTA.  Few CTAs leave SMs idle, so
// short calls cut the rows finer and let more warps share a row's keys.  Measured, KG = 2 / 4 / 8 (us): 288 rows x 4
// heads x 64: 25.1 / 17.1 / 13.5; 600 x 8 x 64: 48.2 / 51.5 / 48.7; 1152 x 8 x 64: 82 / 89 / 108; 700 x 4 x 128: 88 / 55;
// 1152 x 32 x 128: 558 / 611; a batch of two of 700 x 8 x 64: 102 / 90 / 88.
template <typename T>
int launch_simt_t(d3tom_ctx* ctx, const AttnArgs& a, cudaStream_t s) {
  const int sms = ctx->sm_count > 0 ? ctx->sm_count : 148;
  int kg = 2;
  long long best = 0;
  for (int c = 2; c <= 8; c *= 2) {
    const long long ctas = (long long)ceil_div(a.max_seqlen, 128 / c) * a.H * a.B;
    const long long cost = ((ctas + sms - 1) / sms) * ceil_div(a.max_seqlen, 32 * c);
    if (c == 2 || cost < best) { best = cost; kg = c; }
  }
  if (a.dh > 64) return kg == 2 ? launch_simt<T, 128, 2>(ctx, a, s) : launch_simt<T, 128, 4>(ctx, a, s);
  if (a.dh > 32)
    return kg == 2 ? launch_simt<T, 64, 2>(ctx, a, s) : kg == 4 ? launch_simt<T, 64, 4>(ctx, a, s) : launch_simt<T, 64, 8>(ctx, a, s);
  return kg == 2 ? launch_simt<T, 32, 2>(ctx, a, s) : kg == 4 ? launch_simt<T, 32, 4>(ctx, a, s) : launch_simt<T, 32, 8>(ctx, a, s);
}

}  // namespace

int launch_attn_simt(d3tom_ctx* ctx, d3tom_dtype dt, const AttnArgs& a, cudaStream_t s) {
  if (dt == D3TOM_FP32) return launch_simt_t<float>(ctx, a, s);
  return launch_simt_t<__nv_bfloat16>(ctx, a, s);
}

int launch_importance_finish(d3tom_ctx* ctx, const AttnArgs& a, int max_visual, float* importance,
                             const int32_t* cu_vis, cudaStream_t s) {
  if (max_visual <= 0) return D3TOM_OK;
  dim3 grid(ceil_div(max_visual, kImpThreads), a.H, a.B);
  D3TOM_CUDA_TRY(ctx, launch_serialized(importance_finish_kernel, grid, kImpThreads, 0, s, a.score_scratch, a.lse_scratch,
                                        a.n_visual, a.cu_deciders, cu_vis, a.max_deciders, a.vis_stride, a.scale_log2,
                                        ctx->imp_partial, ctx->lim.max_total_tokens, a.H, ctx->imp_counters, importance));
  return D3TOM_OK;
}
