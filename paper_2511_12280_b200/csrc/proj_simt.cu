// "NT" matrix products on CUDA cores, C[m, n] = sum_k A[m, k] B[n, k] with fp32 arithmetic: the fp32 storage path (and,
// for bf16, a debugging aid) of the dense layers (Sec. 3.2.1, Q = H W_Q, K = H W_K; Algorithm 1, FFN_l) and of the
// similarity with its arg-max (Sec. 3.2.2).
//
// Dense layers: a CTA of 8 warps computes a (16 WM) x (32 WN) tile; WK warps share a 16 x 32 register tile (f32_tile.cuh) and cut
// every k-block of 32 WK between them, so that small products, which have few tiles, keep short chains.  k-blocks come
// through a ring of kStages buffers by 16-byte asynchronous copies.
// One order of sums for every tile shape: an output is four chains of multiply-adds (even and odd k apart), chain c over
// the 32-deep pieces c, c + 4, c + 8, ... of K, and the four are added in this order.  A warp that owns more than one
// chain walks its k-blocks chain by chain (the sums so far wait in shared memory: in registers they would cost the second
// CTA per SM).  So a row has the same bits alone and in any batch, whichever tile serves it.
// Bound: the fp32 pipe and shared memory (a lane reads 8 vectors per 64 multiply-adds): 42 TFLOP/s at 1152 x 12288 x 4096
// (pipe 60 % busy, shared-memory wavefronts 59 %), 31 at 384 x 1536 x 512 (19 us; one output per thread and two
// shared-memory reads per multiply-add took 83).
#include "common.cuh"
#include "f32_tile.cuh"

namespace {

constexpr int kStages = 3;
enum { kSimtProj = 0, kSimtLinear = 1, kSimtGateUp = 2 };

template <typename T> struct SimtGemm {
  const T* a; const T* b;          // A rows of the products, B rows (for the gate-up pass: gate rows, then the up rows from row n_cols on)
  int rows, n_cols, K;
  bool vec;                        // vectors of four elements are aligned
  T* out[3];                       // projection: q, k, v; otherwise out[0]
  const T* residual;
  int D;                           // projection: columns of one output
};

template <int EPI, int WM, int WN, int WK> struct SimtGemmSmem {
  static constexpr int kBM = 16 * WM, kBN = 32 * WN, kBK = 32 * WK, kLd = kBK + 4;
  static constexpr int kB = kBN * (EPI == kSimtGateUp ? 2 : 1);
  static constexpr int kStage = (kBM + kB) * kLd;        // floats
  static constexpr int kMats = EPI == kSimtGateUp ? 2 : 1;
  static constexpr int kSums = WK == 4 ? 0 : 8 * kMats * 16 * 32;       // floats: sums of each warp's finished chains
  static constexpr int kBytes = (kStages * kStage + kSums) * 4;
  static_assert(WM * WN * WK == 8, "eight warps");
  static_assert(kStages * kStage >= (WK - 1) * kBM * kB, "the slices' sums are exchanged in the ring");
};

template <typename T, int EPI, int WM, int WN, int WK>
__global__ void __launch_bounds__(256, EPI != kSimtGateUp && WK < 4 ? 2 : 1)
gemm_simt_kernel(SimtGemm<T> p) {
  using S = SimtGemmSmem<EPI, WM, WN, WK>;
  constexpr int kLd = S::kLd, kMats = EPI == kSimtGateUp ? 2 : 1;
  extern __shared__ float4 smem_f4[];
  float* ring = reinterpret_cast<float*>(smem_f4);
  grid_dependency_enter();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ty = f32::lane_ty(lane), tx = f32::lane_tx(lane);
  const int wk = warp % WK, wn = (warp / WK) % WN, wm = warp / (WK * WN);
  const int m0 = blockIdx.y * S::kBM, n0 = blockIdx.x * S::kBN;
  const int rows = p.rows, cols = p.n_cols;
  const T* a = p.a;
  const T* b = p.b;
  const int nkb = (p.K + S::kBK - 1) / S::kBK;
  // this thread's vectors of every k-block: the same column of rows lrow, lrow + kStep, ... of the A and B tiles
  constexpr int kV = S::kBK / 4, kStep = 256 / kV, kLoads = (S::kBM + S::kB) / kStep;
  static_assert((S::kBM + S::kB) % kStep == 0, "every thread loads the same number of vectors");
  const int lrow = tid / kV, lcol = (tid % kV) * 4;
  const T* src[kLoads];
  unsigned src_ok = 0u;
#pragma unroll
  for (int u = 0; u < kLoads; ++u) {
    const int r = lrow + u * kStep;
    bool ok;
    if (r < S::kBM) {
      ok = m0 + r < rows;
      src[u] = a + (size_t)(ok ? m0 + r : 0) * p.K;
    } else {
      const int rb = r - S::kBM, mat = rb / S::kBN, col = n0 + rb - mat * S::kBN;
      ok = col < cols;
      src[u] = b + (size_t)(ok ? mat * cols + col : 0) * p.K;
    }
    src_ok |= (ok ? 1u : 0u) << u;
  }
  // The walk over the k-blocks: those of residue 0 of the block number modulo kTurns, then residue 1, ... (one chain per
  // warp each); kb_load is the next one to load, nkb when there is none.
  constexpr int kTurns = 4 / WK;
  int kb_load = 0, turn_load = 0;
  auto load_next = [&](float* stage) {
    if (kb_load < nkb) {
      float* dst = stage + lrow * kLd + lcol;
      const int c = kb_load * S::kBK + lcol;
      f32::load_vecs<T, kLoads>(dst, kStep * kLd, [&](int u) { return f32::RowRef<T>{src[u], ((src_ok >> u) & 1u) != 0u}; }, c, p.K, p.vec);
      kb_load += kTurns;
      if (kTurns > 1 && kb_load >= nkb) kb_load = ++turn_load < kTurns ? turn_load : nkb;
    }
    f32::cp_async_commit();
  };
  float2 acc[kMats][4][4];
  auto clear_acc = [&] {
#pragma unroll
    for (int t = 0; t < kMats; ++t)
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[t][r][j] = make_float2(0.f, 0.f);
  };
  constexpr int kTile = kMats * 16 * 32;
  float4* sums = reinterpret_cast<float4*>(ring + kStages * S::kStage + warp * kTile) + lane;      // of this lane's outputs
  auto end_chain = [&](bool first) {
#pragma unroll
    for (int t = 0; t < kMats; ++t)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float4* sum = sums + (t * 4 + r) * 32;
        float4 v = make_float4(acc[t][r][0].x + acc[t][r][0].y, acc[t][r][1].x + acc[t][r][1].y,
                               acc[t][r][2].x + acc[t][r][2].y, acc[t][r][3].x + acc[t][r][3].y);
        if (!first) { const float4 o = *sum; v = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w); }
        *sum = v;
      }
    clear_acc();
  };
  clear_acc();
#pragma unroll
  for (int i = 0; i < kStages - 1; ++i) load_next(ring + i * S::kStage);
  float* st = ring;                                       // this k-block's stage, and the one read before it
  float* st_before = ring + (kStages - 1) * S::kStage;
  for (int turn = 0; turn < kTurns && turn < nkb; ++turn) {
    for (int kb = turn; kb < nkb; kb += kTurns) {
      f32::cp_async_wait<kStages - 2>();
      __syncthreads();                     // this block is there for everyone, and everyone is done with the one before
      load_next(st_before);
      const float* aw = st + wm * 16 * kLd + wk * 32;
      const float* bw = st + (S::kBM + wn * 32) * kLd + wk * 32;
#pragma unroll
      for (int t = 0; t < kMats; ++t) f32::dot_16x32<kLd, kLd, 8>(acc[t], aw, bw + t * S::kBN * kLd, ty, tx);
      st_before = st;
      st = st == ring + (kStages - 1) * S::kStage ? ring : st + S::kStage;
    }
    if (turn < kTurns - 1) end_chain(turn == 0);          // (the last chain stays in the accumulators; zeros where K has no piece for it)
  }
  float c[kMats][4][4];
#pragma unroll
  for (int t = 0; t < kMats; ++t)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
      for (int j = 0; j < 4; ++j) c[t][r][j] = acc[t][r][j].x + acc[t][r][j].y;
      if (WK == 1) {
        const float4 o = sums[(t * 4 + r) * 32];
        c[t][r][0] = o.x + c[t][r][0]; c[t][r][1] = o.y + c[t][r][1]; c[t][r][2] = o.z + c[t][r][2]; c[t][r][3] = o.w + c[t][r][3];
      }
    }
  if (WK > 1) {
    // the chains of a register tile meet in shared memory and are added by the first warp
    f32::cp_async_wait<0>();
    __syncthreads();
    float* mine = ring + ((wm * WN + wn) * (WK - 1) + (wk - 1)) * kTile;
    if (wk > 0) {
#pragma unroll
      for (int t = 0; t < kMats; ++t)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) mine[((t * 4 + r) * 4 + j) * 32 + lane] = c[t][r][j];
    }
    __syncthreads();
    if (wk > 0) return;
    const float* others = ring + (wm * WN + wn) * (WK - 1) * kTile + lane;
#pragma unroll
    for (int t = 0; t < kMats; ++t)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float* o = others + (t * 4 + r) * 4 * 32;
        if (WK == 2) {                     // chain 0 waits here, chain 1 with the other warp
          const float4 s0 = sums[(t * 4 + r) * 32], s1 = sums[(t * 4 + r) * 32 + kTile / 4];
          const float s01[4] = {s0.x + s1.x, s0.y + s1.y, s0.z + s1.z, s0.w + s1.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) c[t][r][j] = (s01[j] + c[t][r][j]) + o[j * 32];
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) c[t][r][j] = ((c[t][r][j] + o[j * 32]) + o[j * 32 + kTile]) + o[j * 32 + 2 * kTile];
        }
      }
  }
  const int row0 = m0 + wm * 16 + ty, col0 = n0 + wn * 32 + tx;
  if (EPI == kSimtLinear && p.residual != nullptr) {
    // all of the lane's residuals are requested before the first result is stored (out may be the residual buffer, so a
    // store would hold the next load back)
    T res[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (row0 + 4 * r < rows && col0 + 8 * j < cols) res[r][j] = p.residual[(size_t)(row0 + 4 * r) * cols + col0 + 8 * j];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (row0 + 4 * r < rows && col0 + 8 * j < cols) c[0][r][j] += Storage<T>::to_float(res[r][j]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int col = col0 + 8 * j;
    if (col >= cols) continue;
    const int which = EPI == kSimtProj ? col / p.D : 0, ld = EPI == kSimtProj ? p.D : cols;
    T* out = (which == 0 ? p.out[0] : which == 1 ? p.out[1] : p.out[2]) + (col - which * ld);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (row0 + 4 * r >= rows) continue;
      float y = c[0][r][j];
      if (EPI == kSimtGateUp) y = y / (1.f + expf(-y)) * c[kMats - 1][r][j];
      out[(size_t)(row0 + 4 * r) * ld] = Storage<T>::from_float(y);
    }
  }
}

template <typename T, int EPI, int WM, int WN, int WK>
int launch_shape(d3tom_ctx* ctx, const SimtGemm<T>& p, cudaStream_t s) {
  using S = SimtGemmSmem<EPI, WM, WN, WK>;
  dim3 grid(ceil_div(p.n_cols, S::kBN), ceil_div(p.rows, S::kBM));
  const int smem = spread_smem(ctx, grid, S::kBytes, 3);      // (a step with two layers of 384 rows x 512: 264 -> 238 us)
  // (the attribute belongs to the current device: set on every call, a process may drive several GPUs; always to the same
  // value, since another thread may be launching with another size)
  D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(gemm_simt_kernel<T, EPI, WM, WN, WK>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  D3TOM_CUDA_TRY(ctx, launch_serialized(gemm_simt_kernel<T, EPI, WM, WN, WK>, grid, 256, smem, s, p));
  return D3TOM_OK;
}

// Tile shape: the fewest rounds over the SMs weighted by the tile's area and by what a finer tile costs per element (its
// operands are read more often: measured 1.5 for 32 x 32 at 640 x 1536 x 512), so that only a product with few 64 x 64
// tiles is cut finer, its k-blocks shared by two or four warps.
template <typename T, int EPI>
int launch_simt_gemm(d3tom_ctx* ctx, SimtGemm<T> p, cudaStream_t s) {
  const uintptr_t bits = (uintptr_t)p.a | (uintptr_t)p.b;
  p.vec = p.K % 4 == 0 && bits % (4 * sizeof(T)) == 0;
  const long long sms = ctx->sm_count > 0 ? ctx->sm_count : 148;
  auto cost = [&](int bm, int bn, double scale) {
    const long long tiles = (long long)ceil_div(p.rows, bm) * ceil_div(p.n_cols, bn);
    return scale * (double)((tiles + sms - 1) / sms) * bm * bn;
  };
  const double large = cost(64, 64, 1.0), middle = cost(32, 64, 1.2), small = cost(32, 32, 1.5);
  if (large <= middle && large <= small) return launch_shape<T, EPI, 4, 2, 1>(ctx, p, s);
  if (middle <= small) return launch_shape<T, EPI, 2, 2, 2>(ctx, p, s);
  return launch_shape<T, EPI, 2, 1, 4>(ctx, p, s);
}

template <typename T>
int proj_t(d3tom_ctx* ctx, const void* x, const void* w, int total, int D, void* q, void* k, void* v, cudaStream_t s) {
  SimtGemm<T> p = {};
  p.a = static_cast<const T*>(x); p.b = static_cast<const T*>(w);
  p.rows = total; p.n_cols = 3 * D; p.K = D; p.D = D;
  p.out[0] = static_cast<T*>(q); p.out[1] = static_cast<T*>(k); p.out[2] = static_cast<T*>(v);
  return launch_simt_gemm<T, kSimtProj>(ctx, p, s);
}

template <typename T, int EPI>
int linear_t(d3tom_ctx* ctx, const void* x, const void* w, const void* residual, int rows, int K, int N, void* out,
             cudaStream_t s) {
  SimtGemm<T> p = {};
  p.a = static_cast<const T*>(x); p.b = static_cast<const T*>(w);
  p.rows = rows; p.n_cols = N; p.K = K;
  p.residual = static_cast<const T*>(residual); p.out[0] = static_cast<T*>(out);
  return launch_simt_gemm<T, EPI>(ctx, p, s);
}

// ---------------------------------------------------------------- similarity
// One CTA = 16 visual rows x 32 kept rows of one request.  The dot product of a pair is 32 chains of multiply-adds, chain
// l over the 16-byte vectors l, l + 32, ... of the rows, added up as a butterfly (distances 16, 8, 4, 2, 1): a fixed order
// that does not depend on the tile, so near-ties of the arg-max fall the same way whatever the launch looks like.  Warp w
// runs the chains w, w + 8, w + 16, w + 24 of the whole tile on vectors from shared memory (a lane 4 x 4 pairs) and adds
// those four; the eight sums meet in shared memory.  Bound: the fp32 pipe; one warp per pair reading both rows from L2
// took 46 us at 1024 visual x 256 kept x 512 where this takes 21.
constexpr int kSimRows = 16, kSimCols = 32;

template <typename T> struct SimSmem {
  static constexpr int kVec = Storage<T>::kVec, kChunk = 32 * kVec, kLd = kChunk + 4;
  static constexpr int kStage = (kSimRows + kSimCols) * kLd;
  static constexpr int kBytes = kStages * kStage * 4;
  static_assert(kStages * kStage >= 8 * kSimRows * kSimCols, "the warps' sums are exchanged in the ring");
};

template <typename T>
__global__ void __launch_bounds__(256)
sim_simt_kernel(const T* __restrict__ hidden, const T* __restrict__ kept_rows, const int32_t* __restrict__ cu_seqlens,
                const int32_t* __restrict__ cu_vis, const int32_t* __restrict__ cu_kept, const int32_t* __restrict__ assign,
                const float* __restrict__ inv_norm, const float* __restrict__ inv_norm_kept, int D, int max_kept,
                unsigned long long* __restrict__ best, float* __restrict__ sim_debug) {
  using S = SimSmem<T>;
  constexpr int kVec = S::kVec, kChunk = S::kChunk, kLd = S::kLd;
  extern __shared__ float4 smem_f4[];
  float* ring = reinterpret_cast<float*>(smem_f4);
  grid_dependency_enter();
  const int rq = blockIdx.z, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ty = f32::lane_ty(lane), tx = f32::lane_tx(lane);
  const int v0 = cu_vis[rq], Vb = cu_vis[rq + 1] - v0, k0 = cu_kept[rq], kb = cu_kept[rq + 1] - k0;
  const int m0 = blockIdx.y * kSimRows, s0 = blockIdx.x * kSimCols;
  if (m0 >= Vb || s0 >= kb || kb >= Vb) return;
  // a tile of kept rows only has nothing to do
  if (!__syncthreads_or(tid < kSimRows && m0 + tid < Vb && assign[v0 + m0 + tid] < 0)) return;
  const T* a = hidden + (size_t)(cu_seqlens[rq] + m0) * D;
  const T* b = kept_rows + (size_t)(k0 + s0) * D;
  const int n_chunks = (D + kChunk - 1) / kChunk;
  // this thread's vectors of every chunk: the same column of rows lrow, lrow + kStep, ...
  constexpr int kV = kChunk / 4, kStep = 256 / kV, kLoads = (kSimRows + kSimCols) / kStep;
  const int lrow = tid / kV, lcol = (tid % kV) * 4;
  const T* src[kLoads];
  unsigned src_ok = 0u;
#pragma unroll
  for (int u = 0; u < kLoads; ++u) {
    const int r = lrow + u * kStep;
    const bool is_a = r < kSimRows, ok = is_a ? m0 + r < Vb : s0 + r - kSimRows < kb;
    src[u] = is_a ? a + (size_t)(ok ? r : 0) * D : b + (size_t)(ok ? r - kSimRows : 0) * D;
    src_ok |= (ok ? 1u : 0u) << u;
  }
  auto load_chunk = [&](int t) {
    if (t < n_chunks) {
      float* dst = ring + (t % kStages) * S::kStage + lrow * kLd + lcol;
      f32::load_vecs<T, kLoads>(dst, kStep * kLd, [&](int u) { return f32::RowRef<T>{src[u], ((src_ok >> u) & 1u) != 0u}; },
                                t * kChunk + lcol, D, true);         // (rows are 16-byte aligned: the preparation reads them so)
    }
    f32::cp_async_commit();
  };
  float acc[4][4][4];                      // [chain of this warp][r][j]
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[q][r][j] = 0.f;
  for (int t = 0; t < kStages - 1; ++t) load_chunk(t);
  for (int t = 0; t < n_chunks; ++t) {
    f32::cp_async_wait<kStages - 2>();
    __syncthreads();
    load_chunk(t + kStages - 1);
    const float* st = ring + (t % kStages) * S::kStage;
    const float* ar = st + ty * kLd;
    const float* br = st + (kSimRows + tx) * kLd;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
      for (int e = 0; e < kVec; e += 4) {
        const int c = (warp + 8 * q) * kVec + e;
        float4 av[4], bv[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) av[r] = *reinterpret_cast<const float4*>(ar + r * 4 * kLd + c);
#pragma unroll
        for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const float4*>(br + j * 8 * kLd + c);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[q][r][j] = fmaf(av[r].x, bv[j].x, acc[q][r][j]);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[q][r][j] = fmaf(av[r].y, bv[j].y, acc[q][r][j]);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[q][r][j] = fmaf(av[r].z, bv[j].z, acc[q][r][j]);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[q][r][j] = fmaf(av[r].w, bv[j].w, acc[q][r][j]);
      }
    }
  }
  f32::cp_async_wait<0>();
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j)            // distances 16 and 8
      ring[(warp * kSimRows + ty + 4 * r) * kSimCols + tx + 8 * j] =
          (acc[0][r][j] + acc[2][r][j]) + (acc[1][r][j] + acc[3][r][j]);
  __syncthreads();
#pragma unroll
  for (int rr = 0; rr < kSimRows / 8; ++rr) {
    const int row = warp * (kSimRows / 8) + rr, m = m0 + row, g = v0 + m, s = s0 + lane;
    float v[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) v[w] = ring[(w * kSimRows + row) * kSimCols + lane];
    const float dot = ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));      // distances 4, 2, 1
    unsigned long long mine = 0ull;
    if (m < Vb && s < kb && assign[g] < 0) {                      // a pruned token and one of the kept ones
      const float sim = (dot * inv_norm[g]) * inv_norm_kept[k0 + s] + 0.0f;      // the value the arg-max compares (never -0)
      mine = ((unsigned long long)ordered_key(sim) << 32) | (0xffffffffu - (unsigned)s);
      if (sim_debug != nullptr) sim_debug[(size_t)g * max_kept + s] = sim;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, mine, d);
      mine = o > mine ? o : mine;
    }
    if (lane == 0 && mine != 0ull) atomicMax(best + g, mine);
  }
}

// The same with one block per visual row: warp w scores slots w, w + 8, ..., lane l running chain l.  Same bits.
template <typename T>
__global__ void __launch_bounds__(256)
sim_rows_kernel(const T* __restrict__ hidden, const T* __restrict__ kept_rows, const int32_t* __restrict__ cu_seqlens,
                const int32_t* __restrict__ cu_vis, const int32_t* __restrict__ cu_kept, const int32_t* __restrict__ assign,
                const float* __restrict__ inv_norm, const float* __restrict__ inv_norm_kept, int D, int max_kept,
                unsigned long long* __restrict__ best, float* __restrict__ sim_debug) {
  constexpr int kVec = Storage<T>::kVec;
  grid_dependency_enter();
  const int rq = blockIdx.y, m = blockIdx.x, v0 = cu_vis[rq];
  if (m >= cu_vis[rq + 1] - v0) return;
  const int g = v0 + m;
  if (assign[g] >= 0) return;                                     // a kept token
  const int k0 = cu_kept[rq], kb = cu_kept[rq + 1] - k0;
  const T* hm = hidden + (size_t)(cu_seqlens[rq] + m) * D;
  const float inm = inv_norm[g];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long mine = 0ull;
  for (int s = warp; s < kb; s += 8) {
    const T* hk = kept_rows + (size_t)(k0 + s) * D;
    float dot = 0.f;
    for (int c = lane * kVec; c < D; c += 32 * kVec) {
      float x[kVec], y[kVec];
      Storage<T>::load(hm + c, x);
      Storage<T>::load(hk + c, y);
#pragma unroll
      for (int i = 0; i < kVec; ++i) dot = fmaf(x[i], y[i], dot);
    }
    dot = warp_sum(dot);
    const float sim = (dot * inm) * inv_norm_kept[k0 + s] + 0.0f;
    if (lane == 0) {
      const unsigned long long packed = ((unsigned long long)ordered_key(sim) << 32) | (0xffffffffu - (unsigned)s);
      mine = packed > mine ? packed : mine;
      if (sim_debug != nullptr) sim_debug[(size_t)g * max_kept + s] = sim;
    }
  }
  __shared__ unsigned long long red[8];
  if (lane == 0) red[warp] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long r = red[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) r = red[w] > r ? red[w] : r;
    best[g] = r;
  }
}

template <typename T>
int sim_t(d3tom_ctx* ctx, const MergeArgs& a, cudaStream_t s) {
  if (a.max_kept <= 0) return D3TOM_OK;
  const T* hidden = static_cast<const T*>(a.hidden);
  const T* kept_rows = static_cast<const T*>(ctx->kept_rows);
  const dim3 grid(ceil_div(a.max_kept, kSimCols), ceil_div(a.max_visual, kSimRows), a.B);
  // One block per row where there are few dot products: a tile is one serial pass over D on one SM, and with few kept
  // tokens most of its columns are empty.  Whole merges, rows / tiles (us; visual, kept, D): 9, 3, 4096 20.5 / 34.4;
  // 512, 24, 512 18.9 / 20.6, with 32 kept equal; 1024, 8, 1024 20 / 23, with 16 kept 25.9 / 24.9.  Eight kept tokens or
  // fewer until the rows no longer come out of L2: 10000, 4, 1024 90 / 108; 4096, 8, 4096 and 6000, 4, 4096 equal; 8000, 8,
  // 4096 251 / 191.
  const long long rows = (long long)a.max_visual * a.B;
  if ((a.max_kept <= 24 && rows <= 512) || (a.max_kept <= 8 && rows * a.D <= (24ll << 20))) {
    D3TOM_CUDA_TRY(ctx, launch_serialized(sim_rows_kernel<T>, dim3(a.max_visual, a.B), 256, 0, s, hidden, kept_rows, a.cu_seqlens,
                                          a.cu_vis, a.cu_kept, a.assign, ctx->inv_norm, ctx->inv_norm_kept, a.D, a.max_kept,
                                          ctx->best, a.sim_debug));
    return D3TOM_OK;
  }
  D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(sim_simt_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, SimSmem<T>::kBytes));
  D3TOM_CUDA_TRY(ctx, launch_serialized(sim_simt_kernel<T>, grid, 256, SimSmem<T>::kBytes, s, hidden, kept_rows, a.cu_seqlens,
                                        a.cu_vis, a.cu_kept, a.assign, ctx->inv_norm, ctx->inv_norm_kept, a.D, a.max_kept,
                                        ctx->best, a.sim_debug));
  return D3TOM_OK;
}

}  // namespace

int launch_linear_simt(d3tom_ctx* ctx, d3tom_dtype dt, const void* x, const void* w, const void* residual, int rows,
                       int K, int N, void* out, cudaStream_t s) {
  if (dt == D3TOM_FP32) return linear_t<float, kSimtLinear>(ctx, x, w, residual, rows, K, N, out, s);
  return linear_t<__nv_bfloat16, kSimtLinear>(ctx, x, w, residual, rows, K, N, out, s);
}

int launch_gate_up_simt(d3tom_ctx* ctx, d3tom_dtype dt, const void* x, const void* w_gate_up, int rows, int D, int m,
                        void* act, cudaStream_t s) {
  if (dt == D3TOM_FP32) return linear_t<float, kSimtGateUp>(ctx, x, w_gate_up, nullptr, rows, D, m, act, s);
  return linear_t<__nv_bfloat16, kSimtGateUp>(ctx, x, w_gate_up, nullptr, rows, D, m, act, s);
}

int launch_proj_simt(d3tom_ctx* ctx, d3tom_dtype dt, const void* x, const void* w, int total, int D, void* q, void* k,
                     void* v, cudaStream_t s) {
  if (dt == D3TOM_FP32) return proj_t<float>(ctx, x, w, total, D, q, k, v, s);
  return proj_t<__nv_bfloat16>(ctx, x, w, total, D, q, k, v, s);
}

int launch_sim_simt(d3tom_ctx* ctx, const MergeArgs& a, cudaStream_t s) {
  if (a.dt == D3TOM_FP32) return sim_t<float>(ctx, a, s);
  return sim_t<__nv_bfloat16>(ctx, a, s);
}
