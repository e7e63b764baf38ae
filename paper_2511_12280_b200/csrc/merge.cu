// Similarity-based merging (Sec. 3.2.2; Algorithm 1, the loop over V_merge and
// the removal of the merged positions), everything except the similarity itself
// (gemm_tc.cu; proj_simt.cu for fp32 storage):
//
//   prepare   slot of every visual token in the kept list (-1 = pruned), 1/|h| of
//             every visual row, and a packed copy of the kept rows (the second
//             operand of the similarity)
//   finish    destination slots, per-slot member lists, aggregation in a fixed
//             order and compaction into the shortened sequence
//
// The arg-max is a 64-bit maximum over (order-preserving similarity bits << 32
// | ~slot): the largest similarity wins and, among equals, the lowest slot, no
// matter in which order candidates arrive.
#include <type_traits>

#include "common.cuh"

namespace {

// ---------------------------------------------------------------- prepare
// sum of squares of the 16 bytes of storage in `raw`
template <typename T> __device__ __forceinline__ float sq_raw(uint4 raw);
template <> __device__ __forceinline__ float sq_raw<float>(uint4 raw) {
  const float a = __uint_as_float(raw.x), b = __uint_as_float(raw.y), c = __uint_as_float(raw.z), d = __uint_as_float(raw.w);
  return fmaf(a, a, fmaf(b, b, fmaf(c, c, d * d)));
}
template <> __device__ __forceinline__ float sq_raw<__nv_bfloat16>(uint4 raw) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xffff0000u);
    s = fmaf(lo, lo, fmaf(hi, hi, s));
  }
  return s;
}

// One WARP per visual row (no block-wide synchronisation, so many rows are in flight per
// SM): its slot in the kept list (-1 for a pruned row), a cleared arg-max word, the
// inverse norm and, for kept rows, a copy into the packed second operand of the similarity.
constexpr int kPrepWarps = 8;
constexpr int kPrepInFlight = 8;       // 16-byte loads in flight per lane

template <typename T>
__global__ void __launch_bounds__(kPrepWarps * 32)
prepare_rows_kernel(const T* __restrict__ hidden, const int32_t* __restrict__ cu_seqlens,
                    const int32_t* __restrict__ cu_vis, const int32_t* __restrict__ kept_idx,
                    const int32_t* __restrict__ cu_kept, int D, int32_t* __restrict__ assign,
                    unsigned long long* __restrict__ best, float* __restrict__ inv_norm,
                    float* __restrict__ inv_norm_kept, T* __restrict__ kept_rows, int* __restrict__ n_heavy) {
  constexpr int kVec = Storage<T>::kVec;
  grid_dependency_enter();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *n_heavy = 0;   // counted by the members kernel, two launches on
  const int b = blockIdx.y, lane = threadIdx.x & 31;
  const int m = blockIdx.x * kPrepWarps + (threadIdx.x >> 5);
  const int v0 = cu_vis[b];
  if (m >= cu_vis[b + 1] - v0) return;                       // whole warp
  const int g = v0 + m;
  const int k0 = cu_kept[b], kb = cu_kept[b + 1] - k0;
  const uint4* src = reinterpret_cast<const uint4*>(hidden + (size_t)(cu_seqlens[b] + m) * D);
  const int n_vec = D / kVec;                                 // 16-byte vectors of the row
  // the first batch of row loads goes out before the slot search so that the two latencies overlap
  uint4 raw[kPrepInFlight];
#pragma unroll
  for (int u = 0; u < kPrepInFlight; ++u) {
    const int vi = lane + u * 32;
    if (vi < n_vec) raw[u] = src[vi];
  }
  // slot of position m in the ascending kept list: a 32-way search (each step narrows the range
  // 32-fold with one load per lane and a ballot)
  int lo = 0, len = kb;
  while (len > 32) {
    const int stride = (len + 31) >> 5;
    const int idx = lo + lane * stride;
    const bool le = idx < lo + len && kept_idx[k0 + idx] <= m;
    const int n_le = __popc(__ballot_sync(0xffffffffu, le));   // lanes are ascending: the `le` lanes form a prefix
    if (n_le == 0) { len = 0; break; }                          // every kept position is larger than m
    const int new_lo = lo + (n_le - 1) * stride;
    len = min(stride, lo + len - new_lo);
    lo = new_lo;
  }
  const bool eq = lane < len && kept_idx[k0 + lo + lane] == m;
  const unsigned eqb = __ballot_sync(0xffffffffu, eq);
  const int slot = eqb ? lo + __ffs(eqb) - 1 : -1;
  uint4* dst = slot >= 0 ? reinterpret_cast<uint4*>(kept_rows + (size_t)(k0 + slot) * D) : nullptr;
  float ss = 0.f;
  for (int base = 0; base < n_vec; base += kPrepInFlight * 32) {
    if (base > 0) {
#pragma unroll
      for (int u = 0; u < kPrepInFlight; ++u) {
        const int vi = base + lane + u * 32;
        if (vi < n_vec) raw[u] = src[vi];
      }
    }
#pragma unroll
    for (int u = 0; u < kPrepInFlight; ++u) {
      const int vi = base + lane + u * 32;
      if (vi < n_vec) {
        ss += sq_raw<T>(raw[u]);
        if (dst != nullptr) dst[vi] = raw[u];
      }
    }
  }
  ss = warp_sum(ss);
  if (lane == 0) {
    const float inv = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
    inv_norm[g] = inv;
    assign[g] = slot;
    best[g] = 0ull;
    if (slot >= 0) inv_norm_kept[k0 + slot] = inv;
  }
}

// ---------------------------------------------------------------- finish
constexpr int kMemberThreads = 1024;
constexpr int kMemberSmemSlots = 12 * 1024;        // kept counts up to this keep their counters in shared memory
constexpr int kBitmapBytes = 64 * 1024;            // shared memory for the per-warp position bitmaps
constexpr int kHeavy = 32;                         // a kept token with this many members or more is "heavy"

// One block per request: destination slots, member counts, list offsets and the member
// lists.  Lists of fewer than kHeavy members are left in arrival order (the aggregation
// kernel orders them inside a warp).  Heavy lists are rewritten in ascending position
// here, by marking the members in a bitmap over the request's positions and reading the
// bits back in order, and their slots are appended to `heavy_slots`.
// Dynamic shared memory: [counters (kb ints, when kb <= kMemberSmemSlots)] [bitmaps].
__global__ void __launch_bounds__(kMemberThreads)
members_kernel(const int32_t* __restrict__ cu_vis, const int32_t* __restrict__ cu_kept,
               const unsigned long long* __restrict__ best, int32_t* __restrict__ assign,
               int32_t* __restrict__ member_count, int32_t* __restrict__ member_off,
               int32_t* __restrict__ cursor, int32_t* __restrict__ member_list,
               int32_t* __restrict__ heavy_slots, int* __restrict__ n_heavy, int ctr_ints, int bitmap_warps,
               const int32_t* __restrict__ cu_seqlens, const int32_t* __restrict__ cu_seqlens_out,
               const int32_t* __restrict__ kept_idx, int4* __restrict__ row_desc) {
  extern __shared__ int dyn_s[];
  grid_dependency_enter();
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int v0 = cu_vis[b], V = cu_vis[b + 1] - v0;
  const int k0 = cu_kept[b], kb = cu_kept[b + 1] - k0;
  const int pruned_base = v0 - k0;                 // pruned tokens of earlier requests
  const int lo = cu_seqlens[b], out0 = cu_seqlens_out[b], n_out = cu_seqlens_out[b + 1] - out0;
  // prompt / response rows are copied: member count -1 marks them
  for (int r = kb + tid; r < n_out; r += kMemberThreads) row_desc[out0 + r] = make_int4(lo + V + (r - kb), -1, 0, lo);
  int* ctr = kb <= ctr_ints ? dyn_s : cursor + k0;
  unsigned* bitmaps = reinterpret_cast<unsigned*>(dyn_s + ctr_ints);
  __shared__ int warp_tot[32];
  __shared__ int carry;
  // the request's heavy kept tokens, so that the sorting warps below need not walk over all kept tokens
  constexpr int kHeavyLocal = 2048;
  __shared__ int heavy_local[kHeavyLocal];
  __shared__ int n_heavy_local;
  if (tid == 0) n_heavy_local = 0;
  for (int s = tid; s < kb; s += kMemberThreads) ctr[s] = 0;
  __syncthreads();
  // requests of up to kSlotRegs x 1024 visual tokens keep every token's slot in a register between the counting
  // pass and the filling pass (one round trip to global memory less); -1: a kept token
  constexpr int kSlotRegs = 8;
  const bool in_regs = V <= kSlotRegs * kMemberThreads;
  int my_slot[kSlotRegs];
#pragma unroll
  for (int i = 0; i < kSlotRegs; ++i) {
    my_slot[i] = -1;
    const int m = tid + i * kMemberThreads;
    if (in_regs && m < V) {
      const unsigned long long w = best[v0 + m];
      if (w != 0ull) my_slot[i] = (int)(0xffffffffu - (unsigned)(w & 0xffffffffull));   // a pruned token (kept tokens keep best == 0)
    }
  }
#pragma unroll
  for (int i = 0; i < kSlotRegs; ++i)
    if (my_slot[i] >= 0) {
      assign[v0 + tid + i * kMemberThreads] = my_slot[i];
      atomicAdd(&ctr[my_slot[i]], 1);
    }
  for (int m = tid; m < V && !in_regs; m += kMemberThreads) {
    const int g = v0 + m;
    const unsigned long long w = best[g];
    if (w != 0ull) {
      const int slot = (int)(0xffffffffu - (unsigned)(w & 0xffffffffull));
      assign[g] = slot;
      atomicAdd(&ctr[slot], 1);
    }
  }
  if (tid == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < kb; base += kMemberThreads) {
    const int s = base + tid;
    const int c = s < kb ? ctr[s] : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    int chunk_total = 0;
    if (warp == 0) {
      const int w = warp_tot[lane];
      int winc = w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, winc, o);
        if (lane >= o) winc += t;
      }
      warp_tot[lane] = winc - w;
      chunk_total = __shfl_sync(0xffffffffu, winc, 31);
    }
    __syncthreads();
    const int excl = carry + warp_tot[warp] + incl - c;
    if (s < kb) {
      member_count[k0 + s] = c;
      member_off[k0 + s] = pruned_base + excl;
      ctr[s] = pruned_base + excl;
      if (c >= kHeavy) {
        heavy_slots[atomicAdd(n_heavy, 1)] = k0 + s;
        const int li = atomicAdd(&n_heavy_local, 1);
        if (li < kHeavyLocal) heavy_local[li] = s;
      }
      // what the aggregation needs to know about this output row, in one 16-byte record
      row_desc[out0 + s] = make_int4(lo + kept_idx[k0 + s], c, pruned_base + excl, lo);
    }
    __syncthreads();
    if (tid == 0) carry += chunk_total;
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < kSlotRegs; ++i)
    if (my_slot[i] >= 0) member_list[atomicAdd(&ctr[my_slot[i]], 1)] = tid + i * kMemberThreads;
  for (int m = tid; m < V && !in_regs; m += kMemberThreads) {
    const int g = v0 + m;
    if (best[g] != 0ull) member_list[atomicAdd(&ctr[assign[g]], 1)] = m;
  }
  __syncthreads();
  // ---- heavy lists into ascending order (one warp per list, bitmap_warps warps take part)
  if (warp < bitmap_warps) {
    const int words = (V + 31) >> 5;
    unsigned* bm = bitmaps + (size_t)warp * words;
    const int nh = n_heavy_local;
    const bool listed = nh <= kHeavyLocal;         // else (more heavy tokens than the list holds): walk over all kept tokens
    for (int h = warp; h < (listed ? nh : kb); h += bitmap_warps) {
      const int s = listed ? heavy_local[h] : h;
      const int cnt = member_count[k0 + s];
      if (cnt < kHeavy) continue;                  // uniform over the warp
      const int off = member_off[k0 + s];
      for (int w = lane; w < words; w += 32) bm[w] = 0u;
      __syncwarp();
      for (int i = lane; i < cnt; i += 32) {
        const int m = member_list[off + i];
        atomicOr(&bm[m >> 5], 1u << (m & 31));
      }
      __syncwarp();
      int written = 0;
      for (int w0 = 0; w0 < words; w0 += 32) {     // 32 words = 1024 positions per pass, in order
        const int w = w0 + lane;
        unsigned bits = w < words ? bm[w] : 0u;
        const int n = __popc(bits);
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          int t = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += t;
        }
        int dst = off + written + incl - n;
        while (bits) {
          member_list[dst++] = (w << 5) + __ffs(bits) - 1;
          bits &= bits - 1;
        }
        written += __shfl_sync(0xffffffffu, incl, 31);
      }
      __syncwarp();
    }
  }
}

// acc += the 16 bytes of storage in `raw`, element by element
template <typename T> __device__ __forceinline__ void add_raw(float (&acc)[Storage<T>::kVec], uint4 raw);
template <> __device__ __forceinline__ void add_raw<float>(float (&acc)[4], uint4 raw) {
  acc[0] += __uint_as_float(raw.x); acc[1] += __uint_as_float(raw.y);
  acc[2] += __uint_as_float(raw.z); acc[3] += __uint_as_float(raw.w);
}
template <> __device__ __forceinline__ void add_raw<__nv_bfloat16>(float (&acc)[8], uint4 raw) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    acc[2 * i] += __uint_as_float(w[i] << 16);
    acc[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);
  }
}

constexpr int kAggWarps = 8;
constexpr int kAggUnroll = 4;            // rows in flight per lane
constexpr int kAggCpw = 4;               // 512-byte chunks of a row handled by one warp of a light row

// acc += rows[0..n) of `req` (row indices held one per lane in `rows`), in that order,
// kAggUnroll loads in flight
template <typename T>
__device__ __forceinline__ void add_rows(float (&acc)[Storage<T>::kVec], const T* req, int D, int rows, int n) {
  for (int i = 0; i < n; i += kAggUnroll) {
    uint4 raw[kAggUnroll];
#pragma unroll
    for (int u = 0; u < kAggUnroll; ++u) {
      const int rr = __shfl_sync(0xffffffffu, rows, (i + u) & 31);
      if (i + u < n) raw[u] = *reinterpret_cast<const uint4*>(req + (size_t)rr * D);
    }
#pragma unroll
    for (int u = 0; u < kAggUnroll; ++u)
      if (i + u < n) add_raw<T>(acc, raw[u]);
  }
}

// Aggregation and compaction.  Blocks [heavy_blocks, ...): one WARP per (output row, group of
// kAggCpw 512-byte chunks of the row), one 16-byte vector per lane and chunk, so that one chain
// of index loads is followed by up to kAggUnroll x kAggCpw row loads in flight.  Rows [0, k_b) of a request are the
// merged kept visual tokens, the rest are the prompt and response rows, copied.  The kept
// row comes first, then its members in ascending position, fp32 accumulation, one rounding;
// the (short) member list is ordered with shuffles inside the warp.
// Blocks [0, heavy_blocks): one BLOCK per (heavy kept token, chunk); beyond the actual number they leave at once.  Its list is already
// ascending; warp w adds the kept row (w = 0) and the 32-member segments w, w + 8, ...,
// and the eight partial sums are added in warp order.  Every order is a fixed function of
// the sorted list, so results do not depend on scheduling.
// blockIdx.y = 1: the same for a second payload (the V cache beside the K cache), in the same launch: the two share
// nothing but the lists, and either alone leaves the SMs waiting on latency (4096 + 128 rows of 8 KB: 2 x 12.1 us one
// after the other).
template <typename T>
__global__ void __launch_bounds__(kAggWarps * 32)
aggregate_compact_kernel(const T* __restrict__ hidden_1, const T* __restrict__ hidden_2, const int32_t* __restrict__ cu_seqlens,
                         const int32_t* __restrict__ n_visual, const int32_t* __restrict__ kept_idx,
                         const int32_t* __restrict__ cu_kept, const int32_t* __restrict__ cu_seqlens_out, int B, int D,
                         int chunks, int total_out, int heavy_blocks, int mean,
                         const int32_t* __restrict__ member_count, const int32_t* __restrict__ member_off,
                         const int32_t* __restrict__ member_list, const int32_t* __restrict__ heavy_slots,
                         const int* __restrict__ n_heavy, const int4* __restrict__ row_desc, T* __restrict__ out_1,
                         T* __restrict__ out_2, int32_t* __restrict__ src_of_dst) {
  constexpr int kVec = Storage<T>::kVec;
  grid_dependency_enter();
  const T* __restrict__ hidden = blockIdx.y == 0 ? hidden_1 : hidden_2;      // (the second payload: same lists, same rows)
  T* __restrict__ hidden_out = blockIdx.y == 0 ? out_1 : out_2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float acc[kVec];
#pragma unroll
  for (int e = 0; e < kVec; ++e) acc[e] = 0.f;

  if ((int)blockIdx.x < heavy_blocks) {
    // ------------------------------------------------------------ a heavy kept token (these blocks take the longest: first in the grid)
    // (the host cannot know how many kept tokens are heavy: a fixed number of blocks walks over them)
    const int n_items = *n_heavy * chunks;
    for (int item = (int)blockIdx.x; item < n_items; item += heavy_blocks) {
    const int hi = item / chunks, ch = item - hi * chunks;
#pragma unroll
    for (int e = 0; e < kVec; ++e) acc[e] = 0.f;
    const int ks = heavy_slots[hi];                              // slot in the packed kept list
    const int b = find_segment(cu_kept, B, ks);
    const int r = ks - cu_kept[b];
    const int lo = cu_seqlens[b];
    const int row = cu_seqlens_out[b] + r;
    const int c = (ch * 32 + lane) * kVec;
    const bool live = c < D;
    const T* req = hidden + (size_t)lo * D + (live ? c : 0);
    const int pos = kept_idx[ks], cnt = member_count[ks], off = member_off[ks];
    if (warp == 0) add_raw<T>(acc, *reinterpret_cast<const uint4*>(req + (size_t)pos * D));
    for (int seg = warp; seg * 32 < cnt; seg += kAggWarps) {
      const int n = min(32, cnt - seg * 32);
      const int mine = lane < n ? member_list[off + seg * 32 + lane] : 0;
      add_rows<T>(acc, req, D, mine, n);
    }
    __shared__ float part[kAggWarps][32][Storage<T>::kVec + 1];
#pragma unroll
    for (int e = 0; e < kVec; ++e) part[warp][lane][e] = acc[e];
    __syncthreads();
    if (warp == 0 && live) {
      for (int w = 1; w < kAggWarps; ++w)
#pragma unroll
        for (int e = 0; e < kVec; ++e) acc[e] += part[w][lane][e];
      const float inv_denom = mean ? 1.0f / (float)(1 + cnt) : 1.f;
#pragma unroll
      for (int e = 0; e < kVec; ++e) acc[e] *= inv_denom;
      Storage<T>::store(hidden_out + (size_t)row * D + c, acc);
    }
    if (ch == 0 && blockIdx.y == 0 && threadIdx.x == 0) src_of_dst[row] = lo + pos;
    __syncthreads();                                            // `part` is reused by the next item
    }
    return;
  }

  // ------------------------------------------------------------ light rows: one warp per (row, group of kAggCpw chunks)
  const int groups = (chunks + kAggCpw - 1) / kAggCpw;
  const int gw = ((int)blockIdx.x - heavy_blocks) * kAggWarps + warp;
  const int row = gw / groups, cg = gw - row * groups;
  if (row >= total_out) return;                                 // whole warp
  const int4 desc = row_desc[row];                             // {source row, members (-1: copy), list offset, request's first row}
  const int cnt = desc.y, off = desc.z, lo = desc.w;
  const int pos = desc.x - lo;                                  // position in the request
  int col[kAggCpw];
  bool live[kAggCpw];
#pragma unroll
  for (int j = 0; j < kAggCpw; ++j) {
    col[j] = ((cg * kAggCpw + j) * 32 + lane) * kVec;
    live[j] = col[j] < D;
    if (!live[j]) col[j] = 0;                                   // lanes past the row end read column 0, write nothing
  }
  const T* req = hidden + (size_t)lo * D;
  T* dst = hidden_out + (size_t)row * D;
  if (cg == 0 && blockIdx.y == 0 && lane == 0) src_of_dst[row] = desc.x;

  if (cnt < 0) {                                                // prompt / response row: copy
    uint4 raw[kAggCpw];
#pragma unroll
    for (int j = 0; j < kAggCpw; ++j) raw[j] = *reinterpret_cast<const uint4*>(req + (size_t)pos * D + col[j]);
#pragma unroll
    for (int j = 0; j < kAggCpw; ++j) if (live[j]) *reinterpret_cast<uint4*>(dst + col[j]) = raw[j];
    return;
  }
  if (cnt >= kHeavy) return;                                    // a heavy block does this row
  // lane t ends up holding the t-th row to add: the kept row, then the members by ascending
  // position (distinct values, ranked by counting the smaller ones)
  const int mine = lane < cnt ? member_list[off + lane] : 0x7fffffff;
  int rank = 0;
  for (int j = 0; j < cnt; ++j) rank += __shfl_sync(0xffffffffu, mine, j) < mine ? 1 : 0;
  int ordered = pos;
  for (int j = 0; j < cnt; ++j) {
    const int v = __shfl_sync(0xffffffffu, mine, j), rj = __shfl_sync(0xffffffffu, rank, j);
    if (lane == rj + 1) ordered = v;
  }
  float accs[kAggCpw][kVec];
#pragma unroll
  for (int j = 0; j < kAggCpw; ++j)
#pragma unroll
    for (int e = 0; e < kVec; ++e) accs[j][e] = 0.f;
  const int n = cnt + 1;
  for (int i = 0; i < n; i += kAggUnroll) {                     // kAggUnroll rows x kAggCpw chunks in flight
    uint4 raw[kAggUnroll][kAggCpw];
#pragma unroll
    for (int u = 0; u < kAggUnroll; ++u) {
      const int rr = __shfl_sync(0xffffffffu, ordered, (i + u) & 31);
      if (i + u < n) {
#pragma unroll
        for (int j = 0; j < kAggCpw; ++j) raw[u][j] = *reinterpret_cast<const uint4*>(req + (size_t)rr * D + col[j]);
      }
    }
#pragma unroll
    for (int u = 0; u < kAggUnroll; ++u)
      if (i + u < n) {
#pragma unroll
        for (int j = 0; j < kAggCpw; ++j) add_raw<T>(accs[j], raw[u][j]);
      }
  }
  const float inv_denom = mean ? 1.0f / (float)(1 + cnt) : 1.f;
#pragma unroll
  for (int j = 0; j < kAggCpw; ++j)
    if (live[j]) {
#pragma unroll
      for (int e = 0; e < kVec; ++e) accs[j][e] *= inv_denom;
      Storage<T>::store(dst + col[j], accs[j]);
    }
}

// Aggregation and compaction of ONE request of up to kScanVisual visual tokens without member lists.  A block takes `rows` (1, 2,
// 4, 8) consecutive kept tokens and one of `col_blocks` parts of their columns (blockIdx.y: payload); its eight warps share out
// rows and columns.  It finds the members itself: it reads the request's packed arg-max words once and builds a bitmap per row,
// out of which the positions come in ascending order.  That takes the place of a launch of one block that counted, listed and
// sorted (4 - 9 us in which the other SMs waited) and of the lists' round trip; it costs V x 8 bytes out of L2 per block.  The
// blocks after them copy the prompt and response rows.  Bound: three dependent rounds of loads, then HBM / L2.
// The sums run in the order of aggregate_compact_kernel: the kept row, then its members by position, fp32, one rounding; rows
// with kHeavy members or more: eight partial sums, 32-member segment s in sum s % 8, added in order.  A long list is a chain of
// loads on the one SM that has it, so it is spread: a warp per (row, chunk), or from kBlockList members on (kBlockListFew where
// the block has so few (row, chunk) pairs that most of its warps would idle) a warp per partial sum, two chunks at a time (one at a
// time: 2048 -> 205 x 4096 with six tenths in one cluster 60 us, 53 so).  Words are turned into
// bitmaps by ballot: with shared atomics a cluster that most tokens fall into (its tokens share a word) was serialised, 2045 -> 204
// x 2048, six tenths in one of 32 clusters, 117 us with eight rows per block and atomics, 42 by ballot, 49 with lists.
constexpr int kScanVisual = 8 * 1024;    // 8 bitmaps and a list of 16-bit positions: 24 KB beside 18 KB of partial sums
constexpr int kBlockList = 128, kBlockListFew = 48;
constexpr int kLongUnroll = 8;           // rows of a long list in flight per lane

template <typename T>
__global__ void __launch_bounds__(kAggWarps * 32, 2)
aggregate_scan_kernel(const T* __restrict__ hidden_1, const T* __restrict__ hidden_2, const int32_t* __restrict__ cu_seqlens,
                      const int32_t* __restrict__ cu_vis, const int32_t* __restrict__ kept_idx,
                      const int32_t* __restrict__ cu_kept, const unsigned long long* __restrict__ best, int D, int chunks,
                      int total_out, int rows_log2, int col_blocks, int words, int mean, int32_t* __restrict__ assign,
                      int32_t* __restrict__ member_count, T* __restrict__ out_1, T* __restrict__ out_2,
                      int32_t* __restrict__ src_of_dst) {
  constexpr int kVec = Storage<T>::kVec;
  extern __shared__ unsigned scan_s[];                           // [rows][words] bitmaps, then the long lists
  __shared__ int light_s[kAggWarps][32];
  __shared__ int long_s[kAggWarps];                              // members of a row with a long list, 0: short
  __shared__ int4 long_at[kAggWarps];                            // those rows: {row, start of the list, position, members}
  __shared__ int next_task;
  __shared__ float part_s[2][kAggWarps][kVec][32];
  const int rows = 1 << rows_log2;
  unsigned short* list_s = reinterpret_cast<unsigned short*>(scan_s + rows * words);
  grid_dependency_enter();
  const T* __restrict__ hidden = (blockIdx.y == 0 ? hidden_1 : hidden_2) + (size_t)cu_seqlens[0] * D;
  T* __restrict__ hidden_out = blockIdx.y == 0 ? out_1 : out_2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int V = cu_vis[1] - cu_vis[0], kb = cu_kept[1] - cu_kept[0];
  const int kept_blocks = ((kb + rows - 1) >> rows_log2) * col_blocks;
  if ((int)blockIdx.x >= kept_blocks) {
    // ---- prompt and response rows: one warp per (row, kAggCpw chunks)
    const int groups = (chunks + kAggCpw - 1) / kAggCpw, step = ((int)gridDim.x - kept_blocks) * kAggWarps;
    for (int t = ((int)blockIdx.x - kept_blocks) * kAggWarps + warp; t < (total_out - kb) * groups; t += step) {
      const int row = kb + t / groups, cg = t % groups, from = V + row - kb;
      uint4 raw[kAggCpw];
#pragma unroll
      for (int j = 0; j < kAggCpw; ++j) {
        const int c = ((cg * kAggCpw + j) * 32 + lane) * kVec;
        if (c < D) raw[j] = *reinterpret_cast<const uint4*>(hidden + (size_t)from * D + c);
      }
#pragma unroll
      for (int j = 0; j < kAggCpw; ++j) {
        const int c = ((cg * kAggCpw + j) * 32 + lane) * kVec;
        if (c < D) *reinterpret_cast<uint4*>(hidden_out + (size_t)row * D + c) = raw[j];
      }
      if (cg == 0 && blockIdx.y == 0 && lane == 0) src_of_dst[row] = cu_seqlens[0] + from;
    }
    return;
  }
  const int rg = (int)blockIdx.x / col_blocks, cb = (int)blockIdx.x - rg * col_blocks;
  const int wrow = warp & (rows - 1), sub = warp >> rows_log2, subs = kAggWarps >> rows_log2;   // `subs` warps share a row
  const int r0 = rg * rows, r1 = min(r0 + rows, kb), row = r0 + wrow;
  const bool reports = cb == 0 && blockIdx.y == 0;               // one block per row group writes what it found
  const int c0 = cb * chunks / col_blocks, c1 = (cb + 1) * chunks / col_blocks;      // this block's chunks
  const int pos = row < r1 ? kept_idx[cu_kept[0] + row] : 0;     // source row in the request

  // ---- the members of this block's rows: a warp looks at 32 consecutive tokens, which are one word of each row's bitmap
  const int n_words = kb < V ? (V + 31) >> 5 : 0;                // (0: nothing was pruned)
  if (tid == 0) next_task = 0;
  constexpr int kInFlight = 8;
  const unsigned long long* words_in = best + cu_vis[0];
  for (int base = warp; base < n_words; base += kInFlight * kAggWarps) {
    unsigned rel[kInFlight];                                     // first ~slot of a pruned token, 0 of a kept one
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) {
      const int m = (base + u * kAggWarps) * 32 + lane;
      rel[u] = m < V ? (unsigned)(words_in[m] & 0xffffffffull) : 0u;
    }
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) {
      const int wi = base + u * kAggWarps;
      if (wi >= n_words) break;                                  // uniform
      rel[u] = 0xffffffffu - rel[u] - (unsigned)r0;              // row in the block
      const bool in = rel[u] < (unsigned)(r1 - r0);
      if (reports && in) assign[cu_vis[0] + wi * 32 + lane] = r0 + (int)rel[u];
      // lane r: the tokens whose row has the three bits of r
      const unsigned b_in = __ballot_sync(0xffffffffu, in), b0 = __ballot_sync(0xffffffffu, rel[u] & 1u),
                     b1 = __ballot_sync(0xffffffffu, rel[u] & 2u), b2 = __ballot_sync(0xffffffffu, rel[u] & 4u);
      const unsigned mine = b_in & (lane & 1 ? b0 : ~b0) & (lane & 2 ? b1 : ~b1) & (lane & 4 ? b2 : ~b2);
      if (lane < rows) scan_s[lane * words + wi] = mine;
    }
  }
  __syncthreads();

  // ---- they are counted and, where they are many, listed for all warps
  const unsigned* bm = scan_s + wrow * words;                    // (a row past the end: an empty one)
  int cnt = 0;
  for (int w = lane; w < n_words; w += 32) cnt += __popc(bm[w]);
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (row < r1 && reports && sub == 0 && lane == 0) {
    member_count[cu_kept[0] + row] = cnt;
    src_of_dst[row] = cu_seqlens[0] + pos;
  }
  // the positions marked in the row's bitmap, in order, to dst
  auto list_positions = [&](auto* dst) {
    int written = 0;
    for (int w0 = 0; w0 < n_words; w0 += 32) {
      unsigned v = w0 + lane < n_words ? bm[w0 + lane] : 0u;
      const int n = __popc(v);
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      int at = written + incl - n;
      while (v) {
        dst[at++] = ((w0 + lane) << 5) + __ffs(v) - 1;
        v &= v - 1;
      }
      written += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
  };
  const bool heavy = cnt >= kHeavy;
  if (sub == 0 && lane == 0) long_s[wrow] = heavy ? cnt : 0;
  __syncthreads();
  const int block_list = rows * (c1 - c0) <= 4 ? kBlockListFew : kBlockList;
  int n_long = 0, n_block = 0, n_list = 0;                       // (no token is in two lists: together at most V positions)
  for (int pass = 0; pass < 2; ++pass) {                         // first the rows for the whole block (n_block of them)
    for (int r = 0; r < rows; ++r) {
      const int hc = long_s[r];
      if (hc == 0 || (hc >= block_list) != (pass == 0)) continue;
      if (sub == 0 && wrow == r) {
        list_positions(list_s + n_list);
        if (lane == 0) long_at[n_long] = make_int4(r0 + r, n_list, pos, hc);
      }
      n_list += hc;
      ++n_long;
    }
    if (pass == 0) n_block = n_long;
  }
  if (n_long > 0) __syncthreads();                               // uniform

  if (row < r1 && !heavy) {
    T* dst = hidden_out + (size_t)row * D;
    int ordered = pos;                                           // lane t: the t-th row to add
    if (cnt > 0) {
      list_positions(light_s[warp]);
      if (lane > 0 && lane <= cnt) ordered = light_s[warp][lane - 1];
    }
    const int n = cnt + 1;
    const float inv_denom = mean ? 1.0f / (float)(1 + cnt) : 1.f;
    // kCpw chunks of the row from chunk cg on, kUnroll rows in flight
    auto add_light = [&](int cg, auto chunks_at_once, auto rows_at_once) {
      constexpr int kCpw = decltype(chunks_at_once)::value, kUnroll = decltype(rows_at_once)::value;
      int col[kCpw];
      bool live[kCpw];
#pragma unroll
      for (int j = 0; j < kCpw; ++j) {
        col[j] = ((cg + j) * 32 + lane) * kVec;
        live[j] = cg + j < c1 && col[j] < D;
        if (!live[j]) col[j] = cg * 32 * kVec;                   // lanes past the end read a column in hand, write nothing
      }
      float accs[kCpw][kVec];
#pragma unroll
      for (int j = 0; j < kCpw; ++j)
#pragma unroll
        for (int e = 0; e < kVec; ++e) accs[j][e] = 0.f;
      for (int i = 0; i < n; i += kUnroll) {
        uint4 raw[kUnroll][kCpw];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
          const int rr = __shfl_sync(0xffffffffu, ordered, (i + u) & 31);
          if (i + u < n) {
#pragma unroll
            for (int j = 0; j < kCpw; ++j) raw[u][j] = *reinterpret_cast<const uint4*>(hidden + (size_t)rr * D + col[j]);
          }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
          if (i + u < n) {
#pragma unroll
            for (int j = 0; j < kCpw; ++j) add_raw<T>(accs[j], raw[u][j]);
          }
      }
#pragma unroll
      for (int j = 0; j < kCpw; ++j)
        if (live[j]) {
#pragma unroll
          for (int e = 0; e < kVec; ++e) accs[j][e] *= inv_denom;
          Storage<T>::store(dst + col[j], accs[j]);
        }
    };
    // (a chunk for every warp of the row: more rows at a time instead; 1024 -> 102 x 4096 24.6 / 23.0, 256 -> 64 x 256 fp32 10.8 / 9.8)
    if (c1 - c0 <= subs) {
      if (sub < c1 - c0) add_light(c0 + sub, std::integral_constant<int, 1>(), std::integral_constant<int, 12>());
    } else {
      for (int cg = c0 + sub * kAggCpw; cg < c1; cg += subs * kAggCpw)
        add_light(cg, std::integral_constant<int, kAggCpw>(), std::integral_constant<int, kAggUnroll>());
    }
  }
  if (n_long == 0) return;                                       // uniform

  // acc += rows [i0, i1) of a long list, kLongUnroll loads in flight
  auto add_list = [&](float (&acc)[kVec], const T* src, const unsigned short* list, int i0, int i1) {
    for (int i = i0; i < i1; i += kLongUnroll) {
      uint4 raw[kLongUnroll];
#pragma unroll
      for (int u = 0; u < kLongUnroll; ++u)
        if (i + u < i1) raw[u] = *reinterpret_cast<const uint4*>(src + (size_t)list[i + u] * D);
#pragma unroll
      for (int u = 0; u < kLongUnroll; ++u)
        if (i + u < i1) add_raw<T>(acc, raw[u]);
    }
  };
  auto clear = [](float (&acc)[kVec]) {
#pragma unroll
    for (int e = 0; e < kVec; ++e) acc[e] = 0.f;
  };
  const int n_chunks = c1 - c0;
  // ---- the longest lists: (row, two chunks) by the whole block, one warp per partial sum
  const int n_pairs = (n_chunks + 1) >> 1;
  for (int t = 0; t < n_block * n_pairs; ++t) {
    const int4 at = long_at[t / n_pairs];
    const int hc = at.w, cc = c0 + 2 * (t % n_pairs);
    const bool two = cc + 1 < c1;                                // uniform
    int c[2];
    bool live[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      c[j] = ((cc + j) * 32 + lane) * kVec;
      live[j] = (j == 0 || two) && c[j] < D;
      if (!live[j]) c[j] = cc * 32 * kVec;
    }
    float acc[2][kVec];
    clear(acc[0]);
    clear(acc[1]);
    if (warp == 0) {
#pragma unroll
      for (int j = 0; j < 2; ++j) add_raw<T>(acc[j], *reinterpret_cast<const uint4*>(hidden + (size_t)at.z * D + c[j]));
    }
    const unsigned short* list = list_s + at.y;
    for (int seg = warp; seg * 32 < hc; seg += kAggWarps) {
      const int i1 = min(hc, seg * 32 + 32);
      for (int i = seg * 32; i < i1; i += kLongUnroll) {
        uint4 raw[kLongUnroll][2];
#pragma unroll
        for (int u = 0; u < kLongUnroll; ++u)
          if (i + u < i1) {
            const T* src = hidden + (size_t)list[i + u] * D;
            raw[u][0] = *reinterpret_cast<const uint4*>(src + c[0]);
            if (two) raw[u][1] = *reinterpret_cast<const uint4*>(src + c[1]);
          }
#pragma unroll
        for (int u = 0; u < kLongUnroll; ++u)
          if (i + u < i1) {
            add_raw<T>(acc[0], raw[u][0]);
            if (two) add_raw<T>(acc[1], raw[u][1]);
          }
      }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < kVec; ++e) part_s[j][warp][e][lane] = acc[j][e];
    __syncthreads();
    if (warp < 2 && (warp == 0 ? live[0] : live[1])) {
      const float inv_denom = mean ? 1.0f / (float)(1 + hc) : 1.f;
      float sum[kVec];
#pragma unroll
      for (int e = 0; e < kVec; ++e) {
        sum[e] = part_s[warp][0][e][lane];
#pragma unroll
        for (int w = 1; w < kAggWarps; ++w) sum[e] += part_s[warp][w][e][lane];
        sum[e] *= inv_denom;
      }
      Storage<T>::store(hidden_out + (size_t)at.x * D + (warp == 0 ? c[0] : c[1]), sum);
    }
    __syncthreads();
  }
  // ---- the other long lists: (row, chunk) by whichever warp is free
  const int n_tasks = (n_long - n_block) * n_chunks;
  while (n_tasks > 0) {
    int t = 0;
    if (lane == 0) t = atomicAdd(&next_task, 1);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= n_tasks) break;
    const int4 at = long_at[n_block + t / n_chunks];
    const int hc = at.w, c = ((c0 + t % n_chunks) * 32 + lane) * kVec;
    const T* src = hidden + (c < D ? c : 0);
    float total[kVec];
    for (int w = 0; w < min(kAggWarps, (hc + 31) >> 5); ++w) {   // partial sum w: the segments w, w + 8, ...
      float acc[kVec];
      clear(acc);
      if (w == 0) add_raw<T>(acc, *reinterpret_cast<const uint4*>(src + (size_t)at.z * D));
      for (int seg = w; seg * 32 < hc; seg += kAggWarps) add_list(acc, src, list_s + at.y, seg * 32, min(hc, seg * 32 + 32));
#pragma unroll
      for (int e = 0; e < kVec; ++e) total[e] = w == 0 ? acc[e] : total[e] + acc[e];
    }
    const float inv_denom = mean ? 1.0f / (float)(1 + hc) : 1.f;
#pragma unroll
    for (int e = 0; e < kVec; ++e) total[e] *= inv_denom;
    if (c < D) Storage<T>::store(hidden_out + (size_t)at.x * D + c, total);
  }
}

}  // namespace

int launch_merge_prepare(d3tom_ctx* ctx, const MergeArgs& a, cudaStream_t s) {
  dim3 grid(ceil_div(a.max_visual, kPrepWarps), a.B);
  if (a.dt == D3TOM_FP32)
    D3TOM_CUDA_TRY(ctx, launch_serialized(prepare_rows_kernel<float>, grid, kPrepWarps * 32, 0, s,
                                          static_cast<const float*>(a.hidden), a.cu_seqlens, a.cu_vis, a.kept_idx,
                                          a.cu_kept, a.D, a.assign, ctx->best, ctx->inv_norm, ctx->inv_norm_kept,
                                          static_cast<float*>(ctx->kept_rows), ctx->n_heavy));
  else
    D3TOM_CUDA_TRY(ctx, launch_serialized(prepare_rows_kernel<__nv_bfloat16>, grid, kPrepWarps * 32, 0, s,
                                          static_cast<const __nv_bfloat16*>(a.hidden), a.cu_seqlens, a.cu_vis,
                                          a.kept_idx, a.cu_kept, a.D, a.assign, ctx->best, ctx->inv_norm,
                                          ctx->inv_norm_kept, static_cast<__nv_bfloat16*>(ctx->kept_rows), ctx->n_heavy));
  return D3TOM_OK;
}

// Chunks of 512 bytes per row.
static int row_chunks(d3tom_dtype dt, int D) { return ceil_div(D, 32 * (dt == D3TOM_FP32 ? 4 : 8)); }
// One request: as many kept tokens as the host's sizes allow (their number, where max_visual or max_kept is exact).
static int kept_bound(int total_tokens, int total_out, int max_visual, int max_kept) {
  const int kept = max_visual - (total_tokens - total_out);
  return kept < 0 ? 0 : (kept < max_kept ? kept : max_kept);
}

// How a call aggregates without lists (aggregate_scan_kernel): rows per block and parts of the columns; col_blocks 0: with lists.
// Fitted to merges of one request (64 .. 8192 visual tokens, one to half of them kept, rows of 256 .. 4736, both types, one and
// two payloads, clusters even or up to 95 % of the tokens in one), each timed with lists and in every shape; over 260 of them this
// rule takes 0.93 of the lists' time, and more than 1.03 of it four times, 1.12 at worst.
//   - blocks: columns down to two chunks, then fewer rows, then single chunks, until the kept rows have seven blocks for five SMs: a
//     list that most tokens are on is then added by as many SMs as there are.  (Always eight rows and four parts: up to four times
//     the lists' time, 3399 -> 2 x 4736 70 / 279 us, 619 -> 61 x 3072, 8 clusters, 27 / 50.)  1024 -> 102 x 4096 26.0 / 23.0, with half
//     of the tokens in one cluster 34.8 / 35.6; fewer and larger blocks were up to 1.5 us faster with even clusters and up to 70 slower.
//   - not where all blocks together read more than kScanTokens words: 2048 -> 512 x 4096 36.8 / 35.7, with 60 % in one cluster 56 /
//     81; 5187 -> 1296 x 2048 114 / 207;
//   - nor long rows with a quarter kept and more: the one long list that such a call may have keeps a few SMs busy after the others,
//     1367 -> 341 x 4096 51 / 72, 734 -> 367 x 3072, K and V, 27 / 41.
//   - nothing pruned: whole rows, eight per block as soon as that gives two blocks for five SMs: 0.5 .. 0.8 of the time with lists.
constexpr long long kScanTokens = 300 * 1000;
struct ScanPlan { int rows_log2, col_blocks; };
static ScanPlan scan_plan(int sms, int B, int chunks, int payloads, int total_tokens, int total_out, int max_visual, int max_kept) {
  ScanPlan p = {3, 0};
  if (B != 1 || max_visual > kScanVisual || total_out >= kStreamMinRows || total_out <= 0) return p;
  const int pruned = total_tokens - total_out, kept = kept_bound(total_tokens, total_out, max_visual, max_kept);
  int cols = 1;
  auto blocks = [&] { return (long long)((kept + (1 << p.rows_log2) - 1) >> p.rows_log2) * cols; };      // per payload
  if (pruned == 0) {
    while (p.rows_log2 > 0 && blocks() * payloads < 2 * sms / 5) --p.rows_log2;
  } else {
    if (chunks > 8 && pruned <= 3 * kept) return p;
    const int target = 7 * sms / 5, most = chunks < 16 ? chunks : 16;
    while (cols * 4 <= chunks && cols * 2 <= most && blocks() < target) cols *= 2;
    while (p.rows_log2 > 0 && blocks() < target) --p.rows_log2;
    while (cols * 2 <= most && blocks() < target) cols *= 2;
    if (max_visual * blocks() * payloads > kScanTokens) return p;
  }
  p.col_blocks = cols;
  return p;
}

extern "C" int d3tom_merge_member_lists(int sms, d3tom_dtype dt, int payloads, int B, int D, int total_tokens, int total_out,
                                        int max_visual, int max_kept) {
  if (sms <= 0 || D <= 0 || total_out < 0 || total_tokens < total_out || max_visual < 0 || max_kept < 0) return 1;
  return scan_plan(sms, B, row_chunks(dt, D), payloads, total_tokens, total_out, max_visual, max_kept).col_blocks == 0 ? 1 : 0;
}

int launch_merge_finish(d3tom_ctx* ctx, const MergeArgs& args, cudaStream_t s) {
  MergeArgs a = args;
  // (decided once: payloads launched one by one follow it too)
  const ScanPlan plan = scan_plan(ctx->sm_count, a.B, row_chunks(a.dt, a.D), a.second != nullptr ? 2 : 1, a.total_tokens, a.total_out,
                                  a.max_visual, a.max_kept);
  a.scan_rows_log2 = plan.rows_log2; a.scan_col_blocks = plan.col_blocks;
  if (a.scan_col_blocks > 0) return launch_merge_aggregate(ctx, a, s);
  // (the attribute belongs to the current device: set on every call, a process may drive several GPUs)
  D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(members_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           kMemberSmemSlots * (int)sizeof(int) + kBitmapBytes));
  // shared memory of the members kernel: counters when they fit, then one position bitmap per sorting warp
  const int ctr_ints = a.max_kept <= kMemberSmemSlots ? a.max_kept : 0;
  const int words = ceil_div(a.max_visual > 0 ? a.max_visual : 1, 32);
  int bitmap_warps = kBitmapBytes / (words * 4);
  if (bitmap_warps > kMemberThreads / 32) bitmap_warps = kMemberThreads / 32;
  if (bitmap_warps < 1) return D3TOM_ERR_UNSUPPORTED;              // more than 512 Ki visual tokens in one request
  const size_t smem = (size_t)ctr_ints * sizeof(int) + (size_t)bitmap_warps * words * 4;
  // the count of heavy kept tokens is zeroed by the prepare kernel, which runs whenever there are visual tokens
  if (a.max_visual <= 0) D3TOM_CUDA_TRY(ctx, cudaMemsetAsync(ctx->n_heavy, 0, sizeof(int), s));
  D3TOM_CUDA_TRY(ctx, launch_serialized(members_kernel, a.B, kMemberThreads, smem, s, a.cu_vis, a.cu_kept, ctx->best, a.assign,
                                        a.member_count, ctx->member_off, ctx->member_cursor, ctx->member_list,
                                        ctx->heavy_slots, ctx->n_heavy, ctr_ints, bitmap_warps, a.cu_seqlens,
                                        a.cu_seqlens_out, a.kept_idx, ctx->row_desc));
  return launch_merge_aggregate(ctx, a, s);
}

// aggregation + compaction of a.hidden into a.hidden_out (and of a.second into a.second_out) with the member lists the
// context holds
int launch_merge_aggregate(d3tom_ctx* ctx, const MergeArgs& a, cudaStream_t s) {
  const int mean = a.mode == D3TOM_AGG_MEAN ? 1 : 0;
  if (a.total_out <= 0) return D3TOM_OK;
  if (a.second != nullptr) {
    // One payload's output may lie where the other's input is: then they run one after the other, the payload whose input
    // is about to be overwritten first.  Where each output lies over the other's input no order works, and the second
    // payload's rows wait in the scratch of the gathered kept rows (free once the similarity has run).
    const size_t esize = a.dt == D3TOM_FP32 ? 4 : 2, in = (size_t)a.total_tokens * a.D * esize, out = (size_t)a.total_out * a.D * esize;
    auto overlap = [&](const void* x, const void* y) {
      return (uintptr_t)x < (uintptr_t)y + in && (uintptr_t)y < (uintptr_t)x + out;
    };
    const bool over_first = overlap(a.second_out, a.hidden), over_second = overlap(a.hidden_out, a.second);
    if (over_first || over_second) {
      MergeArgs first = a, second = a;
      first.second = second.second = nullptr;
      first.second_out = second.second_out = nullptr;
      second.hidden = a.second;
      second.hidden_out = over_first && over_second ? ctx->kept_rows : a.second_out;
      int st = launch_merge_aggregate(ctx, over_second ? second : first, s);
      if (st == D3TOM_OK) st = launch_merge_aggregate(ctx, over_second ? first : second, s);
      if (st == D3TOM_OK && over_first && over_second)
        D3TOM_CUDA_TRY(ctx, cudaMemcpyAsync(a.second_out, ctx->kept_rows, out, cudaMemcpyDeviceToDevice, s));
      return st;
    }
  }
  {   // the streaming pipeline takes every row size it supports; the kernel below is the general one
    const int st = launch_merge_aggregate_stream(ctx, a, s);
    if (st != D3TOM_ERR_UNSUPPORTED) return st;
  }
  const int chunks = row_chunks(a.dt, a.D);
  if (a.scan_col_blocks > 0) {
    const int words = ceil_div(a.max_visual, 32), kept = kept_bound(a.total_tokens, a.total_out, a.max_visual, a.max_kept);
    const size_t smem = (size_t)words * ((4 << a.scan_rows_log2) + 64);
    // (the kernel reads the exact number of kept tokens; blocks beyond theirs copy, at least one in case the bound is not tight)
    const int copies = ceil_div((a.total_out - kept) * ceil_div(chunks, kAggCpw), kAggWarps);
    const dim3 grid(ceil_div(kept, 1 << a.scan_rows_log2) * a.scan_col_blocks + (copies > 0 ? copies : 1), a.second != nullptr ? 2 : 1);
    auto launch = [&](auto* tag) -> cudaError_t {
      using T = typename std::remove_pointer<decltype(tag)>::type;
      return launch_serialized(aggregate_scan_kernel<T>, grid, kAggWarps * 32, smem, s, static_cast<const T*>(a.hidden),
                               static_cast<const T*>(a.second), a.cu_seqlens, a.cu_vis, a.kept_idx, a.cu_kept, ctx->best, a.D, chunks,
                               a.total_out, a.scan_rows_log2, a.scan_col_blocks, words, mean, a.assign, a.member_count,
                               static_cast<T*>(a.hidden_out), static_cast<T*>(a.second_out), a.src_of_dst);
    };
    D3TOM_CUDA_TRY(ctx, a.dt == D3TOM_FP32 ? launch(static_cast<float*>(nullptr)) : launch(static_cast<__nv_bfloat16*>(nullptr)));
    return D3TOM_OK;
  }
  const long long warps = (long long)a.total_out * ceil_div(chunks, kAggCpw);
  const int light_blocks = (int)((warps + kAggWarps - 1) / kAggWarps);
  // at most (pruned tokens) / kHeavy kept tokens can be heavy; the blocks beyond the actual number leave at once
  const int max_heavy = (a.total_tokens - a.total_out) / kHeavy;
  // (one block per SM, and more once so many are possible that one per SM would walk over dozens of (row, chunk) items:
  // 12287 visual tokens, 10 % kept, 55 -> 42 us; four per SM for everyone delays the light rows of short requests, 9.4 -> 10.8)
  const int heavy_items = max_heavy * chunks, sms = ctx->sm_count;
  const int heavy_blocks = min(heavy_items, max(sms, min(4 * sms, heavy_items / 8)));
  const dim3 blocks(light_blocks + heavy_blocks, a.second != nullptr ? 2 : 1);
  if (a.dt == D3TOM_FP32)
    D3TOM_CUDA_TRY(ctx, launch_serialized(aggregate_compact_kernel<float>, blocks, kAggWarps * 32, 0, s,
        static_cast<const float*>(a.hidden), static_cast<const float*>(a.second), a.cu_seqlens, a.n_visual, a.kept_idx, a.cu_kept, a.cu_seqlens_out, a.B, a.D,
        chunks, a.total_out, heavy_blocks, mean, a.member_count, ctx->member_off, ctx->member_list, ctx->heavy_slots,
        ctx->n_heavy, ctx->row_desc, static_cast<float*>(a.hidden_out), static_cast<float*>(a.second_out), a.src_of_dst));
  else
    D3TOM_CUDA_TRY(ctx, launch_serialized(aggregate_compact_kernel<__nv_bfloat16>, blocks, kAggWarps * 32, 0, s,
        static_cast<const __nv_bfloat16*>(a.hidden), static_cast<const __nv_bfloat16*>(a.second), a.cu_seqlens, a.n_visual, a.kept_idx, a.cu_kept, a.cu_seqlens_out,
        a.B, a.D, chunks, a.total_out, heavy_blocks, mean, a.member_count, ctx->member_off, ctx->member_list,
        ctx->heavy_slots, ctx->n_heavy, ctx->row_desc, static_cast<__nv_bfloat16*>(a.hidden_out),
        static_cast<__nv_bfloat16*>(a.second_out), a.src_of_dst));
  return D3TOM_OK;
}
