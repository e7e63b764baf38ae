// Keep / merge partition (Sec. 3.2.1; Algorithm 1, TopK): per request the k
// visual tokens of highest importance under the total order (score descending,
// index ascending), emitted ascending by position.
//
// One CTA per request.  Requests of up to 16384 visual tokens keep their keys in
// registers (select_reg_kernel, below); longer ones use select_kernel: the scores
// are mapped to order-preserving 32-bit keys and staged in shared memory.  A most-significant-digit radix select (4 passes
// of 8 bits, warp-aggregated histogram updates) finds the key T of rank k and
// how many keys equal to T still belong to the kept set; the equal keys of
// lowest index are taken.  A final ordered pass writes the mask and the
// ascending index list with a block-wide prefix sum, so the result does not
// depend on thread scheduling: it is bit-exact and reproducible.
#include "common.cuh"

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;

struct SelectShared {
  unsigned hist[256];
  unsigned warp_tot[kWarps];
  unsigned prefix, remaining, carry;
};

template <bool kKeysInSmem>
__global__ void __launch_bounds__(kThreads)
select_kernel(const float* __restrict__ importance, const int32_t* __restrict__ cu_vis,
              const int32_t* __restrict__ keep_count, const int32_t* __restrict__ cu_kept,
              int32_t* __restrict__ kept_idx, uint8_t* __restrict__ keep_mask) {
  extern __shared__ uint32_t keys_s[];
  __shared__ SelectShared sh;
  grid_dependency_enter();
  const int b = blockIdx.x;
  const int v0 = cu_vis[b], V = cu_vis[b + 1] - v0;
  const float* sc = importance + v0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (V <= 0) return;
  int k = keep_count[b];
  k = k < 0 ? 0 : (k > V ? V : k);          // as select_reg_kernel: a count outside [0, V] cannot leave the segment

  if (kKeysInSmem) {
    for (int j = tid; j < V; j += kThreads) keys_s[j] = ordered_key(sc[j]);
  }
  auto key_at = [&](int j) -> uint32_t { return kKeysInSmem ? keys_s[j] : ordered_key(sc[j]); };
  if (tid == 0) { sh.prefix = 0u; sh.remaining = (unsigned)k; }
  __syncthreads();

  // ---- radix select of the k-th largest key ----
  uint32_t mask = 0u;
  const int v_round = ((V + 31) / 32) * 32;
  for (int pass = 0; pass < (k > 0 ? 4 : 0); ++pass) {   // k = 0: nothing is kept, there is no key of rank k
    const int shift = 24 - 8 * pass;
    for (int d = tid; d < 256; d += kThreads) sh.hist[d] = 0u;
    __syncthreads();
    const uint32_t prefix = sh.prefix;
    for (int j = tid; j < v_round; j += kThreads) {   // whole warps iterate together
      uint32_t digit = 0xffffffffu;
      if (j < V) {
        const uint32_t key = key_at(j);
        if ((key & mask) == prefix) digit = (key >> shift) & 255u;
      }
      const unsigned peers = __match_any_sync(0xffffffffu, digit);
      if (digit != 0xffffffffu && lane == __ffs(peers) - 1) atomicAdd(&sh.hist[digit], __popc(peers));
    }
    __syncthreads();
    if (warp == 0) {
      // lane owns digits 255-8*lane .. 248-8*lane (descending); find where the
      // running count from the top reaches `remaining`
      unsigned cnt[8], mine = 0u;
#pragma unroll
      for (int i = 0; i < 8; ++i) { cnt[i] = sh.hist[255 - (lane * 8 + i)]; mine += cnt[i]; }
      unsigned incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      const unsigned excl = incl - mine;
      const unsigned rem = sh.remaining;
      __syncwarp();
      if (excl < rem && rem <= incl) {          // exactly one lane
        unsigned run = excl;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (run < rem && rem <= run + cnt[i]) {
            sh.prefix = prefix | ((uint32_t)(255 - (lane * 8 + i)) << shift);
            sh.remaining = rem - run;
          }
          run += cnt[i];
        }
      }
    }
    mask |= 255u << shift;
    __syncthreads();
  }
  const uint32_t T = sh.prefix;          // key of rank k
  const unsigned need_eq = k > 0 ? sh.remaining : 0u; // how many keys == T are kept (lowest indices first)

  // ---- ordered output pass ----
  if (tid == 0) sh.carry = 0u;           // packed running totals: (greater << 16 | equal) per chunk, 32-bit each below
  __shared__ unsigned run_gt, run_eq;
  if (tid == 0) { run_gt = 0u; run_eq = 0u; }
  __syncthreads();
  int32_t* out = kept_idx + cu_kept[b];
  uint8_t* mk = keep_mask + v0;
  for (int base = 0; base < V; base += kThreads) {
    const int j = base + tid;
    uint32_t key = 0u;
    bool gt = false, eq = false;
    if (j < V && k > 0) { key = key_at(j); gt = key > T; eq = key == T; }
    // packed per-thread counts: high 16 bits greater, low 16 bits equal (chunk <= 1024)
    unsigned val = (gt ? 0x10000u : 0u) | (eq ? 1u : 0u);
    unsigned incl = val;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) sh.warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      unsigned w = sh.warp_tot[lane];
      unsigned winc = w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        unsigned t = __shfl_up_sync(0xffffffffu, winc, o);
        if (lane >= o) winc += t;
      }
      sh.warp_tot[lane] = winc - w;       // exclusive over warps
      if (lane == 31) sh.carry = winc;    // chunk total
    }
    __syncthreads();
    const unsigned excl = sh.warp_tot[warp] + incl - val;
    const unsigned gt_before = run_gt + (excl >> 16);
    const unsigned eq_before = run_eq + (excl & 0xffffu);
    if (j < V) {
      const bool keep = gt || (eq && eq_before < need_eq);
      mk[j] = keep ? 1 : 0;
      if (keep) out[gt_before + min(eq_before, need_eq)] = j;
    }
    __syncthreads();
    if (tid == 0) { run_gt += sh.carry >> 16; run_eq += sh.carry & 0xffffu; }
    __syncthreads();
  }
}

// Requests of up to 1024 x IPT visual tokens (IPT 1 .. 16; 12287 tokens: 14.4 us, 20.5 with
// the staged kernel above): every thread keeps IPT CONSECUTIVE keys in registers, so the ordered
// output needs a single block-wide prefix sum and the keys are read once.  The radix select takes digits of 12 bits
// from the highest bit of (key - smallest key) on (the first digit then spreads them over many bins, where the sign and
// the exponent they share would crowd a few) and stops as soon as every key that shares the digits so far is kept: mostly after
// the second digit.  A thread owns the same four bins in every pass and clears them as it reads them, which saves the barrier
// of a separate clearing phase.  Bound: latency of one block, three barriers a pass.
constexpr int kRegBinsMax = 4096;

template <int IPT>
__global__ void __launch_bounds__(kThreads)
select_reg_kernel(const float* __restrict__ importance, const int32_t* __restrict__ cu_vis,
                  const int32_t* __restrict__ keep_count, const int32_t* __restrict__ cu_kept,
                  int32_t* __restrict__ kept_idx, uint8_t* __restrict__ keep_mask) {
  __shared__ uint4 hist4[kRegBinsMax / 4];
  __shared__ unsigned warp_tot[kWarps], warp_lo[kWarps], warp_hi[kWarps];
  __shared__ unsigned sh_prefix, sh_remaining, sh_whole;
  unsigned* hist = reinterpret_cast<unsigned*>(hist4);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int d = tid; d < kRegBinsMax; d += kThreads) hist[d] = 0u;      // on-chip only: before the dependency wait
  grid_dependency_enter();
  const int b = blockIdx.x;
  const int v0 = cu_vis[b], V = cu_vis[b + 1] - v0;
  if (V <= 0) return;
  int k = keep_count[b];
  k = k < 0 ? 0 : (k > V ? V : k);
  const float* sc = importance + v0;
  const int j0 = tid * IPT;
  uint32_t key[IPT];
#pragma unroll
  for (int i = 0; i < IPT; ++i) key[i] = (j0 + i < V) ? ordered_key(sc[j0 + i]) : 0u;

  // inclusive prefix sum of `val` over the block in thread order; every warp scans the 32 warp totals itself
  auto block_scan = [&](unsigned val, unsigned& total) -> unsigned {
    unsigned incl = val;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    unsigned w = warp_tot[lane], winc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += t;
    }
    total = __shfl_sync(0xffffffffu, winc, 31);
    const unsigned before = __shfl_sync(0xffffffffu, winc - w, warp);
    return incl + before;
  };

  // The keys are taken relative to the smallest one, so that the radix select starts at the highest bit of their range; it
  // stops as soon as all keys that share the digits so far are kept.
  uint32_t lo_key = 0xffffffffu, hi_key = 0u;
#pragma unroll
  for (int i = 0; i < IPT; ++i)
    if (j0 + i < V) { lo_key = min(lo_key, key[i]); hi_key = max(hi_key, key[i]); }
  lo_key = __reduce_min_sync(0xffffffffu, lo_key);
  hi_key = __reduce_max_sync(0xffffffffu, hi_key);
  if (lane == 0) { warp_lo[warp] = lo_key; warp_hi[warp] = hi_key; }
  __syncthreads();                          // (the cleared histogram as well)
  lo_key = __reduce_min_sync(0xffffffffu, warp_lo[lane]);
  hi_key = __reduce_max_sync(0xffffffffu, warp_hi[lane]);
#pragma unroll
  for (int i = 0; i < IPT; ++i) key[i] -= lo_key;                // (those past the end are never looked at)
  int top = 32 - __clz((int)(hi_key - lo_key));                  // no key has a bit from `top` on
  uint32_t prefix = 0u;
  unsigned rem = (unsigned)k;
  bool whole = k == V;                      // every key with this prefix is kept
  if (k <= 0) { top = 0; prefix = 0xffffffffu; }                 // (nothing is kept: no key above, none of the equal ones)
  while (top > 0 && !whole) {
    const int shift = top > 12 ? top - 12 : 0;
    const uint32_t mask = top < 32 ? 0xffffffffu << top : 0u, digits = (1u << (top - shift)) - 1u;
#pragma unroll
    for (int i = 0; i < IPT; ++i)
      if (j0 + i < V && (key[i] & mask) == prefix) atomicAdd(&hist[(key[i] >> shift) & digits], 1u);
    __syncthreads();
    // thread t owns four bins, 4095 - 4 t downwards (the running count goes from the top digit), and leaves them clear
    uint4* mine4 = hist4 + (kThreads - 1 - tid);
    const uint4 c4 = *mine4;
    *mine4 = make_uint4(0u, 0u, 0u, 0u);
    const unsigned cnt[4] = {c4.w, c4.z, c4.y, c4.x};
    const unsigned mine = (c4.x + c4.y) + (c4.z + c4.w);
    unsigned total;
    const unsigned incl = block_scan(mine, total);
    const unsigned excl = incl - mine;
    if (excl < rem && rem <= incl) {                      // exactly one thread: the digit of the key of rank k
      unsigned run = excl;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (run < rem && rem <= run + cnt[i]) {
          sh_prefix = prefix | ((uint32_t)(4 * (kThreads - 1 - tid) + 3 - i) << shift);
          sh_remaining = rem - run;
          sh_whole = rem - run == cnt[i] ? 1u : 0u;
        }
        run += cnt[i];
      }
    }
    __syncthreads();
    prefix = sh_prefix;
    rem = sh_remaining;
    whole = sh_whole != 0u;
    top = shift;
  }
  // kept: the keys above T, and of the keys equal to T the `need_eq` at the lowest positions
  uint32_t T = prefix;                      // the key of rank k; or, if its lower digits were not looked at, ...
  unsigned need_eq = rem;
  if (whole && T > 0u) { T -= 1u; need_eq = 0u; }       // ... the largest value below every key with its upper digits

  // ---- ordered output: one prefix sum over the per-thread counts (greater << 16 | equal)
  unsigned val = 0u;
#pragma unroll
  for (int i = 0; i < IPT; ++i)
    if (j0 + i < V) val += (key[i] > T ? 0x10000u : 0u) + (key[i] == T ? 1u : 0u);
  __syncthreads();                          // warp_tot is reused
  unsigned total;
  const unsigned incl = block_scan(val, total);
  unsigned gt_before = (incl - val) >> 16, eq_before = (incl - val) & 0xffffu;
  int32_t* out = kept_idx + cu_kept[b];
  uint8_t* mk = keep_mask + v0;
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    const int j = j0 + i;
    if (j < V) {
      const bool gt = key[i] > T, eq = key[i] == T;
      const bool keep = gt || (eq && eq_before < need_eq);
      mk[j] = keep ? 1 : 0;
      if (keep) out[gt_before + min(eq_before, need_eq)] = j;
      gt_before += gt ? 1u : 0u;
      eq_before += eq ? 1u : 0u;
    }
  }
}

}  // namespace

int launch_select(d3tom_ctx* ctx, const float* importance, const int32_t* cu_vis, const int32_t* keep_count,
                  const int32_t* cu_kept, int B, int max_visual, int32_t* kept_idx, uint8_t* keep_mask,
                  cudaStream_t s) {
  const size_t smem = (size_t)max_visual * sizeof(uint32_t);
  if (max_visual <= 16 * kThreads) {          // keys in registers
    if (max_visual <= kThreads) D3TOM_CUDA_TRY(ctx, launch_serialized(select_reg_kernel<1>, B, kThreads, 0, s, importance, cu_vis, keep_count, cu_kept, kept_idx, keep_mask));
    else if (max_visual <= 2 * kThreads) D3TOM_CUDA_TRY(ctx, launch_serialized(select_reg_kernel<2>, B, kThreads, 0, s, importance, cu_vis, keep_count, cu_kept, kept_idx, keep_mask));
    else if (max_visual <= 4 * kThreads) D3TOM_CUDA_TRY(ctx, launch_serialized(select_reg_kernel<4>, B, kThreads, 0, s, importance, cu_vis, keep_count, cu_kept, kept_idx, keep_mask));
    else if (max_visual <= 8 * kThreads) D3TOM_CUDA_TRY(ctx, launch_serialized(select_reg_kernel<8>, B, kThreads, 0, s, importance, cu_vis, keep_count, cu_kept, kept_idx, keep_mask));
    else D3TOM_CUDA_TRY(ctx, launch_serialized(select_reg_kernel<16>, B, kThreads, 0, s, importance, cu_vis, keep_count, cu_kept, kept_idx, keep_mask));
  } else if (smem <= 160 * 1024) {
    // (the attribute belongs to the current device: set on every call, a process may drive several GPUs)
    D3TOM_CUDA_TRY(ctx, cudaFuncSetAttribute(select_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
    D3TOM_CUDA_TRY(ctx, launch_serialized(select_kernel<true>, B, kThreads, smem, s, importance, cu_vis, keep_count, cu_kept, kept_idx, keep_mask));
  } else {
    D3TOM_CUDA_TRY(ctx, launch_serialized(select_kernel<false>, B, kThreads, 0, s, importance, cu_vis, keep_count, cu_kept, kept_idx, keep_mask));
  }
  D3TOM_LAUNCH_CHECK(ctx);
  return D3TOM_OK;
}
