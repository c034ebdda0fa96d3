// Device-side plumbing shared by the kernel translation units (sm_103a):
// warp reductions, wavevectors, and the item loop of single- and multi-cell
// launches.
#pragma once

#include "mp_common.cuh"

namespace mp {

// ------------------------------------------------------------------ helpers
__device__ __forceinline__ float shfl_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ double shfl_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <class T>
__device__ __forceinline__ T shfl_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <class R>
__device__ __forceinline__ R signed_freq_scale(int k, int n, R two_pi_over_L) {
  const int s = (k <= n / 2) ? k : k - n;
  return two_pi_over_L * (R)s;
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// col / kx of a column index (< 2^18, kx <= 2^8): exact by the multiplier
// ceil(2^32 / kx), whose excess kx_magic kx - 2^32 < kx keeps col times it
// below 2^32.
template <class R>
__device__ __forceinline__ int div_kx(const CellDev<R>& c, int col) {
  return c.kx_magic ? (int)__umulhi((unsigned)col, c.kx_magic) : col;
}

// ------------------------------------------------------------------ multi-cell plumbing
// Entry owning global item g: the last e with pre[e] <= g (binary search).
__device__ __forceinline__ int find_entry(const long long* pre, int n, long long g) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= g) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Cooperative copy of a cell descriptor into shared memory (callers fence with
// barriers on both sides).
template <class R>
__device__ __forceinline__ void load_cell(CellDev<R>& dst, const CellDev<R>* src) {
  static_assert(sizeof(CellDev<R>) % 4 == 0, "descriptor size");
  const int* s4 = reinterpret_cast<const int*>(src);
  int* d4 = reinterpret_cast<int*>(&dst);
  for (int i = threadIdx.x; i < (int)(sizeof(CellDev<R>) / 4); i += blockDim.x) d4[i] = s4[i];
}

// Runs `body(cell, local_item, fresh)` over a launch's items: the single cell `c0`
// (items 0..n0-1), or, for MULTI, every entry of `w` with its cell staged in
// shared memory `cs` (reloaded when a block moves to the next cell).  A cell
// whose round control says stop (a later round of a batched window after
// its loop ended) has its items skipped; the flag only changes between
// launches, so every thread of the block reads the same value.  `fresh` tells
// the body that this is the block's first item of the cell.
template <class R, bool MULTI, class Body>
__device__ __forceinline__ void for_items(const CellDev<R>& c0, long long n0, const Work<R>& w,
                                          CellDev<R>& cs, Body body) {
  if constexpr (!MULTI) {
    for (long long g = blockIdx.x; g < n0; g += gridDim.x) body(c0, g, g == (long long)blockIdx.x);
  } else {
    // contiguous ranges: a block's consecutive items mostly share a cell
    const long long total = w.pre[w.n_act];
    const long long per = (total + gridDim.x - 1) / gridDim.x;
    const long long g0 = (long long)blockIdx.x * per;
    const long long g1 = (g0 + per < total) ? g0 + per : total;
    if (g0 >= g1) return;
    int e = find_entry(w.pre, w.n_act, g0);
    int cur = -1;
    bool halted = false, fresh = false;
    for (long long g = g0; g < g1; ++g) {
      while (g >= w.pre[e + 1]) ++e;
      const int slot = w.act[e];
      if (slot != cur) {
        __syncthreads();
        load_cell(cs, w.cells + slot);
        __syncthreads();
        cur = slot;
        fresh = true;
        halted = cs.rctl != nullptr && __ldcg(&cs.rctl->stop) != 0;
      }
      if (!halted) body(cs, g - w.pre[e], fresh);
      fresh = false;
    }
  }
}

}  // namespace mp
