// Kernels of one fixed-point iteration of the micropolar FFT scheme (sm_103a)
// and their launchers.  Spectral buffer layout: complex spec[(kz N2 + ky) KX
// + kx][18], 18 = (tau or e^: 9 comps, mu or gamma^: 9 comps), KX = N1 / 2
// (the Nyquist column kx = N1 / 2 is never stored: the Green operator zeroes
// it) or 1 when N1 == 1.
//
// One iteration (Algorithm 2 while-loop) runs
//   y-forward  ->  z-forward + Green + z-inverse  ->  y-inverse  ->  pass A
// where pass A does, row by row along x: inverse x transform, + (E, Gamma),
// Algorithm 1, error partials against the previous iterate, polarizations
// tau = t - A0 e, mu = m - B0 gamma, forward x transform.
#include "mp_kernels.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "mp_constitutive.cuh"
#include "mp_device.cuh"
#include "mp_fft.cuh"
#include "mp_limits.cuh"
#include "mp_lines.cuh"
#include "mp_plan.cuh"
#include "mp_tma.cuh"

namespace mp {

// The line passes' own translation units compile them, except the z pass of
// flat cells (N2 = 1), at the end of this one.
#define MP_LINES_ELSEWHERE(R)                      \
  MP_INSTANTIATE_LINE(R, kYForward, extern)        \
  MP_INSTANTIATE_LINE(R, kYInverse, extern)        \
  MP_INSTANTIATE_LINE(R, kZReduced, extern)        \
  MP_INSTANTIATE_LINE_MULTI(R, kYForward, extern)  \
  MP_INSTANTIATE_LINE_MULTI(R, kYInverse, extern)  \
  MP_INSTANTIATE_LINE_MULTI(R, kZReduced, extern)
MP_LINES_ELSEWHERE(float)
MP_LINES_ELSEWHERE(double)

// 8 warps per block.  Registers are split between the SM's four sub-partitions
// (16 K each), so with 2 blocks per SM (4 warps per sub-partition) a thread
// may use up to 128 registers; a 9-warp block would cap it at 96.
constexpr int kThreads = 256;
// Shared memory per block on sm_103a (opt-in maximum) and the part of it the
// dynamic tiles may use: the multi-cell kernels also hold a cell descriptor
// and a few reduction words in static shared memory.
constexpr size_t kSmemOptin = 227 * 1024;
constexpr size_t kSmemStaticReserve = 2048;
constexpr size_t kSmemBudget = kSmemOptin - kSmemStaticReserve;

// ------------------------------------------------------------------ x pass (pass A)
// Packed real transform of a row of N1 reals through a complex transform of
// length M = N1 / 2: z[n] = x[2n] + i x[2n+1].
//   forward:  X[k] = (Z[k] + conj Z[M-k]) / 2 - (i / 2) W_N1^k (Z[k] - conj Z[M-k])
//   inverse:  Z[k] = (X[k] + conj X[M-k]) + i W_N1^-k (X[k] - conj X[M-k]),  X[M] = 0
// (X[M] is the Nyquist bin, which the Green operator sets to zero; X[0] is
// real for a real row and its imaginary part is ignored).  Tiles are AoS:
// point k of line (rr, c) at [(rr M + k) 18 + c].

// s + i conj(w) d, the packed pre-step of a pair a, b (s = a + b, d = a - b,
// w = W_N1^k), and (s - i w d) / 2, the post-step.  The product enters the sum
// by fused multiply-adds: one rounding less than forming it first.
template <class R>
__device__ __forceinline__ cpx<R> packed_pre(cpx<R> a, cpx<R> b, cpx<R> w) {
  const cpx<R> s = cadd(a, b), d = csub(a, b);
  return cmake<R>(fma(w.y, d.x, fma(-w.x, d.y, s.x)), fma(w.y, d.y, fma(w.x, d.x, s.y)));
}
template <class R>
__device__ __forceinline__ cpx<R> packed_post(cpx<R> a, cpx<R> b, cpx<R> w) {
  const cpx<R> s = cadd(a, b), d = csub(a, b);
  return cmake<R>(R(0.5) * fma(w.y, d.x, fma(w.x, d.y, s.x)), R(0.5) * fma(w.y, d.y, fma(-w.x, d.x, s.y)));
}

__device__ __forceinline__ int div_m(int q, int M, int msh) { return msh >= 0 ? (q >> msh) : (q / M); }

template <class R>
__device__ __forceinline__ void x_inverse_pre(const cpx<R>* X, cpx<R>* Z, int rows, int M, int msh,
                                              const cpx<R>* tw) {
  const int total = rows * M * 18;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int c = idx % 18;
    const int q = idx / 18;          // rr * M + k
    const int rr = div_m(q, M, msh), k = q - rr * M;
    const cpx<R>* x = X + rr * M * 18 + c;
    cpx<R> a = x[k * 18];
    if (k == 0) a.y = R(0);
    const cpx<R> b = (k == 0) ? cmake<R>(R(0), R(0)) : cconj(x[(M - k) * 18]);
    Z[idx] = packed_pre(a, b, tw[k]);
  }
}

// The inverse pre-step fused into the first (Ns = 1) Stockham stage: each
// butterfly forms its RADIX inputs Z[j + r M / RADIX] from X (as
// x_inverse_pre does) instead of reading them from a separate pass, which
// saves one shared-memory pass and one barrier per item.
template <class R, int RADIX, int M>
__device__ __forceinline__ void stage_first_inv_packed(const cpx<R>* __restrict__ X, cpx<R>* __restrict__ out,
                                                       int rows, const cpx<R>* __restrict__ tw) {
  constexpr int nb = M / RADIX;
  constexpr int rs = M * 18;
  const int total = rows * nb * 18;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int c = idx % 18;
    const int q = idx / 18;
    const int rr = q / nb, j = q % nb;
    const cpx<R>* x = X + rr * rs + c;
    cpx<R> v[RADIX];
#pragma unroll
    for (int r = 0; r < RADIX; ++r) {
      const int k = j + r * nb;
      cpx<R> a = x[k * 18];
      if (k == 0) a.y = R(0);
      const cpx<R> b = (k == 0) ? cmake<R>(R(0), R(0)) : cconj(x[(M - k) * 18]);
      v[r] = packed_pre(a, b, tw[k]);
    }
    if constexpr (RADIX == 3) dft3<R, +1>(v);
    else if constexpr (RADIX == 4) dft4<R, +1>(v);
    else if constexpr (RADIX == 8) dft8<R, +1>(v);
    else dft16<R, +1>(v);
    cpx<R>* dst = out + rr * rs + c + (j * RADIX) * 18;
#pragma unroll
    for (int r = 0; r < RADIX; ++r) dst[r * 18] = v[r];
  }
}

// ---- x transforms of the lengths in x_plan: the radices are compile-time, the
// length is not (one body serves every length with that radix).  Rows hold M
// points; butterfly j of a stage takes points j + r M / RADIX.
template <class Body>
__device__ __forceinline__ void x_butterflies(int rows, int nb, Body body) {
  const unsigned magic = nb > 1 ? 0xffffffffu / (unsigned)nb + 1u : 0u;  // q / nb for q < 2^16
  for (int idx = threadIdx.x; idx < rows * nb * 18; idx += blockDim.x) {
    const int q = idx / 18, c = idx - q * 18;
    const int rr = nb > 1 ? (int)__umulhi((unsigned)q, magic) : q;
    body(c, rr, q - rr * nb);
  }
}

// First inverse stage with the packed pre-step (as stage_first_inv_packed).
template <class R, int RADIX>
__device__ __forceinline__ void x_inv_first(const cpx<R>* X, cpx<R>* out, int rows, int M, const cpx<R>* tw) {
  const int nb = M / RADIX;
  x_butterflies(rows, nb, [=](int c, int rr, int j) {
    const cpx<R>* x = X + rr * M * 18 + c;
    cpx<R> v[RADIX];
#pragma unroll
    for (int r = 0; r < RADIX; ++r) {
      const int k = j + r * nb;
      cpx<R> a = x[k * 18], b = cconj(x[(k == 0 ? 0 : M - k) * 18]);
      if (k == 0) {
        a.y = R(0);
        b = cmake<R>(R(0), R(0));
      }
      v[r] = packed_pre(a, b, tw[k]);
    }
    dft<R, +1, RADIX>(v);
    cpx<R>* dst = out + (rr * M + j * RADIX) * 18 + c;
#pragma unroll
    for (int r = 0; r < RADIX; ++r) dst[r * 18] = v[r];
  });
}
// Last inverse stage (Ns = M / RADIX).
template <class R, int RADIX>
__device__ __forceinline__ void x_inv_last(const cpx<R>* in, cpx<R>* out, int rows, int M, const cpx<R>* tw) {
  const int nb = M / RADIX;
  x_butterflies(rows, nb, [=](int c, int rr, int j) {
    const int o = (rr * M + j) * 18 + c;
    cpx<R> v[RADIX];
    v[0] = in[o];
#pragma unroll
    for (int r = 1; r < RADIX; ++r) v[r] = cmul(in[o + r * nb * 18], twiddle<R, +1>(tw, 2 * r * j));
    dft<R, +1, RADIX>(v);
#pragma unroll
    for (int r = 0; r < RADIX; ++r) out[o + r * nb * 18] = v[r];
  });
}
// First forward stage (Ns = 1).
template <class R, int RADIX>
__device__ __forceinline__ void x_fwd_first(const cpx<R>* in, cpx<R>* out, int rows, int M) {
  const int nb = M / RADIX;
  x_butterflies(rows, nb, [=](int c, int rr, int j) {
    const cpx<R>* src = in + (rr * M + j) * 18 + c;
    cpx<R> v[RADIX];
#pragma unroll
    for (int r = 0; r < RADIX; ++r) v[r] = src[r * nb * 18];
    dft<R, -1, RADIX>(v);
    cpx<R>* dst = out + (rr * M + j * RADIX) * 18 + c;
#pragma unroll
    for (int r = 0; r < RADIX; ++r) dst[r * 18] = v[r];
  });
}
// Last forward stage with the packed post-step: butterflies u and Ns - u of a
// line hold each other's partners (as x_forward_last_post; u = 0 and, for even
// Ns, u = Ns / 2 are their own).  Ns = 1 is a whole transform.
template <class R, int RADIX>
__device__ __forceinline__ void x_fwd_last(const cpx<R>* in, cpx<R>* X, int rows, int M, const cpx<R>* tw) {
  const int ns = M / RADIX, units = ns / 2 + 1;
  x_butterflies(rows, units, [=](int c, int rr, int u) {
    const cpx<R>* src = in + rr * M * 18 + c;
    cpx<R>* dst = X + rr * M * 18 + c;
    auto butterfly = [&](int j, cpx<R>(&v)[RADIX]) {
      v[0] = src[j * 18];
#pragma unroll
      for (int r = 1; r < RADIX; ++r) {
        v[r] = src[(j + r * ns) * 18];
        if (ns > 1) v[r] = cmul(v[r], twiddle<R, -1>(tw, 2 * r * j));
      }
      dft<R, -1, RADIX>(v);
    };
    auto post = [&](int k, cpx<R> a, cpx<R> zp) {
      dst[k * 18] = packed_post(a, cconj(zp), tw[k]);
    };
    cpx<R> v[RADIX];
    butterfly(u, v);
    if (u == 0) {
#pragma unroll
      for (int r = 0; r < RADIX; ++r) post(ns * r, v[r], v[(RADIX - r) % RADIX]);
    } else if (2 * u == ns) {
#pragma unroll
      for (int r = 0; r < RADIX; ++r) post(u + ns * r, v[r], v[RADIX - 1 - r]);
    } else {
      cpx<R> w[RADIX];
      butterfly(ns - u, w);
#pragma unroll
      for (int r = 0; r < RADIX; ++r) {
        post(u + ns * r, v[r], w[RADIX - 1 - r]);
        post(ns - u + ns * r, w[r], v[RADIX - 1 - r]);
      }
    }
  });
}

// Inverse of packed rows in b0 by plan P (count > 0); returns the result's
// buffer.  Ends with a barrier.
template <class R>
__device__ __forceinline__ cpx<R>* x_inv_planned(cpx<R>* b0, cpx<R>* b1, int rows, int M, const XPlan& P,
                                                 const cpx<R>* tw) {
  switch (P.r0) {
    case 2: x_inv_first<R, 2>(b0, b1, rows, M, tw); break;
    case 3: x_inv_first<R, 3>(b0, b1, rows, M, tw); break;
    case 4: x_inv_first<R, 4>(b0, b1, rows, M, tw); break;
    case 6: x_inv_first<R, 6>(b0, b1, rows, M, tw); break;
    case 8: x_inv_first<R, 8>(b0, b1, rows, M, tw); break;
    case 9: x_inv_first<R, 9>(b0, b1, rows, M, tw); break;
    default: x_inv_first<R, 12>(b0, b1, rows, M, tw); break;
  }
  __syncthreads();
  if (P.count == 1) return b1;
  switch (P.r1) {
    case 3: x_inv_last<R, 3>(b1, b0, rows, M, tw); break;
    case 6: x_inv_last<R, 6>(b1, b0, rows, M, tw); break;
    case 8: x_inv_last<R, 8>(b1, b0, rows, M, tw); break;
    default: x_inv_last<R, 9>(b1, b0, rows, M, tw); break;
  }
  __syncthreads();
  return b0;
}
// Forward of the packed rows in z, post-step included; the result replaces z.
template <class R>
__device__ __forceinline__ void x_fwd_planned(cpx<R>* z, cpx<R>* other, int rows, int M, const XPlan& P,
                                              const cpx<R>* tw) {
  const cpx<R>* in = z;  // one stage: each thread replaces the line it holds
  if (P.count == 2) {
    switch (P.r0) {
      case 6: x_fwd_first<R, 6>(z, other, rows, M); break;
      case 8: x_fwd_first<R, 8>(z, other, rows, M); break;
      case 9: x_fwd_first<R, 9>(z, other, rows, M); break;
      default: x_fwd_first<R, 12>(z, other, rows, M); break;
    }
    __syncthreads();
    in = other;
  }
  switch (P.count == 2 ? P.r1 : P.r0) {
    case 2: x_fwd_last<R, 2>(in, z, rows, M, tw); break;
    case 3: x_fwd_last<R, 3>(in, z, rows, M, tw); break;
    case 4: x_fwd_last<R, 4>(in, z, rows, M, tw); break;
    case 6: x_fwd_last<R, 6>(in, z, rows, M, tw); break;
    case 8: x_fwd_last<R, 8>(in, z, rows, M, tw); break;
    default: x_fwd_last<R, 9>(in, z, rows, M, tw); break;
  }
}

// Inverse x transform of packed rows: the spectral rows X in b0 -> the
// packed real rows (returned: b0 or b1).  Ends with a barrier.
template <class R>
__device__ cpx<R>* tile_fft_x_inv_packed(cpx<R>* b0, cpx<R>* b1, int rows, const RadixPlan& p, int msh,
                                         const cpx<R>* tw) {
  auto sync_swap = [&]() {
    __syncthreads();
    cpx<R>* t = b0;
    b0 = b1;
    b1 = t;
  };
  switch (p.m) {
    case 256:
      stage_first_inv_packed<R, 8, 256>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, +1, 8, 8, 256>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, +1, 4, 64, 256>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 128:  // as the forward transform: 16 x 8 in FP32, 8 x 4 x 4 in FP64
      if constexpr (sizeof(R) == 4) {
        stage_first_inv_packed<R, 16, 128>(b0, b1, rows, tw); sync_swap();
        stage_fixed<R, +1, 8, 16, 128>(b0, b1, rows, tw); sync_swap();
      } else {
        stage_first_inv_packed<R, 8, 128>(b0, b1, rows, tw); sync_swap();
        stage_fixed<R, +1, 4, 8, 128>(b0, b1, rows, tw); sync_swap();
        stage_fixed<R, +1, 4, 32, 128>(b0, b1, rows, tw); sync_swap();
      }
      return b0;
    case 64:
      stage_first_inv_packed<R, 8, 64>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, +1, 8, 8, 64>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 32:
      stage_first_inv_packed<R, 8, 32>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, +1, 4, 8, 32>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 16:
      stage_first_inv_packed<R, 4, 16>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, +1, 4, 4, 16>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 24:
      stage_first_inv_packed<R, 8, 24>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, +1, 3, 8, 24>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 12:
      stage_first_inv_packed<R, 4, 12>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, +1, 3, 4, 12>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 8:
      stage_first_inv_packed<R, 8, 8>(b0, b1, rows, tw); sync_swap();
      return b0;
    default:
      if (const XPlan P = x_plan(p.m); P.count > 0) return x_inv_planned<R>(b0, b1, rows, p.m, P, tw);
      x_inverse_pre<R>(b0, b1, rows, p.m, msh, tw);
      __syncthreads();
      return tile_fft<R, +1>(b1, b0, rows, p, tw);
  }
}

template <class R>
__device__ __forceinline__ void x_forward_post(const cpx<R>* Z, cpx<R>* X, int rows, int M, int msh,
                                               const cpx<R>* tw) {
  const int total = rows * M * 18;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int c = idx % 18;
    const int q = idx / 18;
    const int rr = div_m(q, M, msh), k = q - rr * M;
    const cpx<R>* z = Z + rr * M * 18 + c;
    cpx<R> a = z[k * 18];
    cpx<R> b = cconj(z[(k == 0 ? 0 : M - k) * 18]);
    X[idx] = packed_post(a, b, tw[k]);
  }
}

// The last forward Stockham stage of a length-M transform (radix RADIX,
// Ns = M / RADIX, twiddle stride 2) fused with the packed-real post-step.
// Output k = j + Ns r of butterfly j pairs with output M - k, which butterfly
// Ns - j produces at r' = RADIX - 1 - r (butterfly 0: r' = RADIX - r mod
// RADIX; butterfly Ns / 2 pairs with itself): one thread takes butterflies j
// and Ns - j of a line, so both partners are in its registers and X goes
// straight to shared memory, without a separate post pass.
template <class R, int M, int RADIX>
__device__ __forceinline__ void x_forward_last_post(const cpx<R>* __restrict__ in, cpx<R>* __restrict__ X,
                                                    int rows, const cpx<R>* __restrict__ tw) {
  constexpr int NS = M / RADIX, UNITS = NS / 2 + 1, LN = 18, RS = M * LN;
  const int total = rows * UNITS * LN;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int c = idx % LN;
    const int q = idx / LN;
    const int rr = q / UNITS, u = q - rr * UNITS;
    const cpx<R>* src = in + rr * RS + c;
    cpx<R>* dst = X + rr * RS + c;
    // butterfly j of the stage (as stage_fixed<R, -1, RADIX, NS, M>)
    auto butterfly = [&](int j, cpx<R>(&v)[RADIX]) {
      v[0] = src[j * LN];
#pragma unroll
      for (int r = 1; r < RADIX; ++r) v[r] = cmul(src[(j + r * NS) * LN], twiddle<R, -1>(tw, 2 * r * j));
      if constexpr (RADIX == 4) dft4<R, -1>(v);
      else dft8<R, -1>(v);
    };
    // X[k] = (s - i W_N1^k d) / 2, s = Z[k] + conj(Z[M - k]), d = Z[k] - conj(Z[M - k])
    auto post = [&](int k, cpx<R> a, cpx<R> zp) {
      dst[k * LN] = packed_post(a, cconj(zp), tw[k]);
    };
    cpx<R> v[RADIX];
    butterfly(u, v);
    if (u == 0) {
#pragma unroll
      for (int r = 0; r < RADIX; ++r) post(NS * r, v[r], v[(RADIX - r) % RADIX]);
    } else if (u == NS / 2) {
#pragma unroll
      for (int r = 0; r < RADIX; ++r) post(NS / 2 + NS * r, v[r], v[RADIX - 1 - r]);
    } else {
      cpx<R> w[RADIX];
      butterfly(NS - u, w);
#pragma unroll
      for (int r = 0; r < RADIX; ++r) {
        post(u + NS * r, v[r], w[RADIX - 1 - r]);
        post(NS - u + NS * r, w[r], v[RADIX - 1 - r]);
      }
    }
  }
}

enum PassMode { kIter = 0, kStart = 1, kXFwd = 2, kXInv = 3 };

// Shared-memory plan of pass A: a fixed header (barriers, reduction scratch,
// the block's error totals) then the buffers for `rows` rows of N1 voxels.
template <class R>
struct PassASmem {
  static constexpr size_t bar_off = 0;                                 // 2 mbarriers
  static constexpr size_t red_off = 64;                                // [16 warps][8] doubles
  static constexpr size_t acc_off = red_off + 16 * 8 * sizeof(double);  // [kErrPartials]
  static constexpr size_t head = ((acc_off + kErrPartials * sizeof(double)) + 127) / 128 * 128;
  size_t fft_bytes, b0_off, b1_off, prev_off, hist_off, pq_off, dc_off, tw_off, carry_off, total;
  __host__ __device__ PassASmem(int n1, int rows) {
    const int M = (n1 > 1) ? n1 / 2 : 1;
    const size_t nvi = (size_t)rows * n1;
    fft_bytes = (size_t)rows * M * 18 * sizeof(cpx<R>);  // multiple of 16
    b0_off = head;
    b1_off = b0_off + fft_bytes;
    prev_off = b1_off + fft_bytes;
    hist_off = prev_off + nvi * 20 * sizeof(R);
    pq_off = hist_off + nvi * 20 * sizeof(R);
    dc_off = pq_off + nvi * 2 * sizeof(double);
    tw_off = dc_off + ((18 * (size_t)rows * sizeof(R) + 15) / 16) * 16;  // x twiddles W_N1^k, k < N1
    carry_off = tw_off + ((n1 * sizeof(cpx<R>) + 15) / 16) * 16;
    // per-thread running error maxima [4][kThreads] (R), sums [4][kThreads] and
    // row sums [kThreads] (double), kept here rather than in registers
    total = carry_off + (size_t)kThreads * (4 * sizeof(R) + 5 * sizeof(double));
  }
};

// A voxel's 20-value record (previous iterate or history) between shared
// memory and registers in 16-byte pieces: records are 80 (FP32) / 160 (FP64)
// bytes apart, so per-value accesses by consecutive threads would hit the
// same banks four (two) ways; 16-byte accesses of 8 threads cover all 32 banks.
__device__ __forceinline__ void load_rec(const float* p, float* r) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const float4 a = q[k];
    r[4 * k] = a.x;
    r[4 * k + 1] = a.y;
    r[4 * k + 2] = a.z;
    r[4 * k + 3] = a.w;
  }
}
__device__ __forceinline__ void load_rec(const double* p, double* r) {
  const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
  for (int k = 0; k < 10; ++k) {
    const double2 a = q[k];
    r[2 * k] = a.x;
    r[2 * k + 1] = a.y;
  }
}
__device__ __forceinline__ void store_rec(float* p, const float* r) {
  float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
  for (int k = 0; k < 5; ++k) q[k] = make_float4(r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3]);
}
__device__ __forceinline__ void store_rec(double* p, const double* r) {
  double2* q = reinterpret_cast<double2*>(p);
#pragma unroll
  for (int k = 0; k < 10; ++k) q[k] = make_double2(r[2 * k], r[2 * k + 1]);
}

// 18-value records (the predictor base elast) are 72 / 144 bytes apart: 8- /
// 16-byte pieces.
__device__ __forceinline__ void load_rec18(const float* p, float* r) {
  const float2* q = reinterpret_cast<const float2*>(p);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const float2 a = q[k];
    r[2 * k] = a.x;
    r[2 * k + 1] = a.y;
  }
}
__device__ __forceinline__ void load_rec18(const double* p, double* r) {
  const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double2 a = q[k];
    r[2 * k] = a.x;
    r[2 * k + 1] = a.y;
  }
}
__device__ __forceinline__ void store_rec18(float* p, const float* r) {
  float2* q = reinterpret_cast<float2*>(p);
#pragma unroll
  for (int k = 0; k < 9; ++k) q[k] = make_float2(r[2 * k], r[2 * k + 1]);
}
__device__ __forceinline__ void store_rec18(double* p, const double* r) {
  double2* q = reinterpret_cast<double2*>(p);
#pragma unroll
  for (int k = 0; k < 9; ++k) q[k] = make_double2(r[2 * k], r[2 * k + 1]);
}

// Contiguous values between global and shared memory, in 16-byte pieces when
// the global side starts on a 16-byte boundary (smem always does), the rest
// value by value.  Loads are asynchronous (cp_async_wait_all and a barrier
// follow).
template <class R>
__device__ __forceinline__ void copy_values_in(R* dst, const R* src, int n) {
  constexpr int PV = 16 / (int)sizeof(R);
  const int nv = (reinterpret_cast<uintptr_t>(src) & 15) == 0 ? n / PV : 0;
  for (int i = threadIdx.x; i < nv; i += blockDim.x) cp_async16(dst + i * PV, src + i * PV);
  for (int i = nv * PV + threadIdx.x; i < n; i += blockDim.x) cp_async_value(dst + i, src + i);
}
template <class R>
__device__ __forceinline__ void copy_values_out(R* dst, const R* src, int n) {
  constexpr int PV = 16 / (int)sizeof(R);
  const int nv = (reinterpret_cast<uintptr_t>(dst) & 15) == 0 ? n / PV : 0;
  for (int i = threadIdx.x; i < nv; i += blockDim.x)
    reinterpret_cast<float4*>(dst)[i] = reinterpret_cast<const float4*>(src)[i];
  for (int i = nv * PV + threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// Record a timeout and leave: the caller has seen a bounded wait fail.
__device__ __forceinline__ void flag_timeout(int* status) {
  if (threadIdx.x == 0 && status) atomicOr(status, 1);
}

// One pass-A work item: `rows` consecutive rows (y, z) of a cell = a
// contiguous range of voxels and of spectral rows.  Rows, previous iterate,
// history and plastic strains move between global and shared memory by bulk
// asynchronous copies (TMA); the spectral rows are requested first so that the
// inverse transform runs while the per-voxel records are still in flight.
// Leaves the item's 8 error maxima / sums in red[0..7] (thread 0..7 views, see
// below) and its 36 row sums in `itm` (kIter only).  Returns false when a
// bounded wait expired (uniform across the block).
template <class R, int MODE, bool MULTI>
__device__ __forceinline__ bool pass_a_item(const CellDev<R>& c, long long item, unsigned char* smem_raw,
                                            uint32_t& parity, double* itm, R* tms, const R* fin_tau,
                                            const R* fin_mu, R* fout_e, R* fout_g, bool reload) {
  const int rows = c.rows_a;
  const int N1 = c.n1;
  const int M = c.kx;                 // complex entries per row (N1 / 2, or 1)
  const int msh = (M & (M - 1)) == 0 ? __ffs(M) - 1 : -1;
  const bool packed = (N1 > 1);
  const PassASmem<R> L(N1, rows);
  cpx<R>* b0 = reinterpret_cast<cpx<R>*>(smem_raw + L.b0_off);
  cpx<R>* b1 = reinterpret_cast<cpx<R>*>(smem_raw + L.b1_off);
  R* prev_s = reinterpret_cast<R*>(smem_raw + L.prev_off);
  R* hist_s = reinterpret_cast<R*>(smem_raw + L.hist_off);
  double2* pq_s = reinterpret_cast<double2*>(smem_raw + L.pq_off);
  double* red = reinterpret_cast<double*>(smem_raw + PassASmem<R>::red_off);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + PassASmem<R>::bar_off);
  R* dcin = reinterpret_cast<R*>(smem_raw + L.dc_off);
  cpx<R>* tws = reinterpret_cast<cpx<R>*>(smem_raw + L.tw_off);
  const long long nrows = (long long)c.n2 * c.n3;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool use_vox = (MODE == kIter || MODE == kStart);
  const bool use_spec_in = (MODE == kIter || MODE == kXInv);

  const long long row0 = item * rows;
  const int nr = (int)min((long long)rows, nrows - row0);
  const int nvi = nr * N1;
  const long long v0 = row0 * N1;
  // ---------------------------------------------------------- issue loads
  // the cell's constants and x twiddle table (read many times per item, from
  // shared memory): staged for the block's first item of each cell
  if (reload) {
    if (use_vox && threadIdx.x < 18) tms[threadIdx.x] = (R)c.tmean[threadIdx.x];
    for (int k = threadIdx.x; k < N1; k += blockDim.x) tws[k] = c.tw[0][k];
  }
  if (threadIdx.x == 0) {
    // the block's next item (single cell), fetched into L2 while this one runs
    if (!MULTI && item + gridDim.x < c.items_a) {
      const long long r1 = (item + gridDim.x) * rows;
      const int n1r = (int)min((long long)rows, nrows - r1);
      if (use_spec_in) bulk_prefetch_l2(c.spec + r1 * M * 18, (uint32_t)(n1r * M * 18 * sizeof(cpx<R>)));
      if (use_vox) {
        const uint32_t bp = (uint32_t)(n1r * N1 * 20 * sizeof(R));
        bulk_prefetch_l2(c.prev + r1 * N1 * 20, bp);
        bulk_prefetch_l2(c.hist + r1 * N1 * 20, bp);
        bulk_prefetch_l2(c.pq + r1 * N1 * 2, (uint32_t)(n1r * N1 * 2 * sizeof(double)));
      }
    }
    bulk_wait_read();     // the previous item's stores have read shared memory
    fence_proxy_async();  // and every thread's reads of it precede the new loads
    if (use_spec_in) {
      const uint32_t bytes = (uint32_t)(nr * M * 18 * sizeof(cpx<R>));
      mbar_arrive_expect_tx(&bars[0], bytes);
      bulk_load(b0, c.spec + row0 * M * 18, bytes, &bars[0]);
    }
    if (use_vox) {
      const uint32_t bp = (uint32_t)(nvi * 20 * sizeof(R));
      const uint32_t bq = (uint32_t)(nvi * 2 * sizeof(double));
      mbar_arrive_expect_tx(&bars[1], 2 * bp + bq);
      bulk_load(prev_s, c.prev + v0 * 20, bp, &bars[1]);
      bulk_load(hist_s, c.hist + v0 * 20, bp, &bars[1]);
      bulk_load(pq_s, c.pq + v0 * 2, bq, &bars[1]);
    }
  }
  cpx<R>* zbuf = b0;  // buffer holding the packed real rows
  // Without loads to wait for (forward-only mode), the barrier that orders
  // thread 0's wait for the previous item's bulk stores (which may still be
  // reading b0) before every thread's writes to b0 must be explicit.
  // The component call's fields (9 values a voxel) are staged in the unused
  // record buffers: voxel by voxel they are 36 (72) bytes apart (at 256^3 in
  // FP32 the forward pass took 755 us and the inverse one 1443).
  if (MODE == kXFwd) {
    copy_values_in(prev_s, fin_tau + v0 * 9, nvi * 9);
    copy_values_in(hist_s, fin_mu + v0 * 9, nvi * 9);
    cp_async_wait_all();
  }
  if (!use_spec_in && !use_vox) __syncthreads();
  // ---------------------------------------------------------- inverse x
  if (use_spec_in) {
    const bool ok = mbar_wait(&bars[0], parity);
    if (__syncthreads_or(!ok)) return false;
    if (MODE == kIter)
      for (int l = threadIdx.x; l < 18 * nr; l += blockDim.x) {
        const int rr = l / 18, cc = l - rr * 18;
        dcin[cc * rows + rr] = b0[rr * M * 18 + cc].x;
      }
    if (packed) {
      zbuf = tile_fft_x_inv_packed<R>(b0, b1, nr, c.px, msh, tws);
    }
  }
  if (use_vox) {
    const bool ok = mbar_wait(&bars[1], parity);
    if (__syncthreads_or(!ok)) return false;
  }
    // ---------------------------------------------------------- per voxel
    R dmax[4] = {R(0), R(0), R(0), R(0)};
    R dsum[4] = {R(0), R(0), R(0), R(0)};
    for (int lv = threadIdx.x; lv < nvi; lv += blockDim.x) {
      const int rr = lv / N1, x = lv - rr * N1;
      const int zb = (rr * M + (packed ? (x >> 1) : 0)) * 18;  // first comp of the voxel's complex
      const long long v = v0 + lv;
      // value q of the inverse-transformed row at this voxel (read where it is
      // used, so that only one level's values are in registers at a time)
      const R* zv = reinterpret_cast<const R*>(zbuf + zb) + ((packed && (x & 1)) ? 1 : 0);
      if (MODE == kXInv) {
#pragma unroll
        for (int q = 0; q < 9; ++q) {
          prev_s[lv * 9 + q] = zv[2 * q];
          hist_s[lv * 9 + q] = zv[2 * (9 + q)];
        }
        continue;
      }
      // value q of this voxel goes to the real (even x) or imaginary (odd x)
      // part of its packed complex entry
      R* zr = reinterpret_cast<R*>(zbuf + zb) + ((packed && (x & 1)) ? 1 : 0);
      if (!packed) {
#pragma unroll
        for (int q = 0; q < 18; ++q) zr[2 * q + 1] = R(0);
      }
      if (MODE == kXFwd) {
#pragma unroll
        for (int q = 0; q < 9; ++q) {
          zr[2 * q] = prev_s[lv * 9 + q];
          zr[2 * (9 + q)] = hist_s[lv * 9 + q];
        }
        continue;
      }
      // The voxel's two levels (Algorithm 1's macro level: e, t, f_t; micro
      // level: gamma, m, f_m) are independent: they run one after the other so
      // that only one level's tensors are held in registers at a time.  Records
      // (80 bytes apart) move in 16-byte pieces:
      //   previous iterate  {e0-3} {e4-7} {e8 g0 g1 g2} {g3-6} {g7 g8 f_t f_m}
      //   history           {ht0-3} {ht4-7} {ht8 hm0 hm1 hm2} {hm3-6} {hm7 hm8 phase 0}
      float4* pv4 = reinterpret_cast<float4*>(prev_s + lv * 20);
      const float4* hv4 = reinterpret_cast<const float4*>(hist_s + lv * 20);
      R* pv = prev_s + lv * 20;
      const R* hv = hist_s + lv * 20;
      const PhaseDev<R>& P = c.phases[(int)hv[18]];
      const double2 pq = pq_s[lv];
      const R fto = pv[18], fmo = pv[19];
      const R a0 = c.ref.mu + c.ref.kap, b0 = c.ref.mu - c.ref.kap;
      const bool din = MODE == kIter && c.delta_in != 0, dout = MODE == kIter && c.delta_out != 0;
      const R* sv = c.src ? c.src + v * 18 : nullptr;
      R ft, fm, e8;
      // ---- macro level
      {
        R e[9], eo[9], ht[9], t[9];
        if constexpr (sizeof(R) == 4) {
          const float4 q0 = pv4[0], q1 = pv4[1], q2 = pv4[2];
          const float4 h0 = hv4[0], h1 = hv4[1], h2 = hv4[2];
          eo[0] = q0.x; eo[1] = q0.y; eo[2] = q0.z; eo[3] = q0.w;
          eo[4] = q1.x; eo[5] = q1.y; eo[6] = q1.z; eo[7] = q1.w; eo[8] = q2.x;
          ht[0] = h0.x; ht[1] = h0.y; ht[2] = h0.z; ht[3] = h0.w;
          ht[4] = h1.x; ht[5] = h1.y; ht[6] = h1.z; ht[7] = h1.w; ht[8] = h2.x;
        } else {
#pragma unroll
          for (int q = 0; q < 9; ++q) {
            eo[q] = pv[q];
            ht[q] = hv[q];
          }
        }
        // de9: the strain change that enters the polarization, e - E (full
        // form) or e^i - e^{i-1} (increment form)
        R de9[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) de9[q] = (MODE == kIter) ? zv[2 * q] : R(0);
#pragma unroll
        for (int q = 0; q < 9; ++q) e[q] = (MODE == kIter) ? (din ? eo[q] : c.E[q]) + de9[q] : eo[q];
        double pn = pq.x;
        // the pass needs the scale factor only (p is formed at the commit)
        return_macro<R, sizeof(R) == 4 ? 1 : 2>(P, e, ht, pn, t, pn, ft);
        if (MODE == kIter) {
          if (dout) {
#pragma unroll
            for (int q = 0; q < 9; ++q) de9[q] = e[q] - eo[q];
          }
          const R trd = de9[0] + de9[4] + de9[8];
          // previous stresses rebuilt from the stored strains and scale factor
          // (t = tr/3 d + f_t dev(t_trial)), in the same operation order
          const R tre = (eo[0] + eo[4]) + eo[8];
          const R vol = vol_of(trial_t(P, ht[0], eo[0], eo[0], true, tre), trial_t(P, ht[4], eo[4], eo[4], true, tre),
                               trial_t(P, ht[8], eo[8], eo[8], true, tre));
          R de = R(0), dt = R(0);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int l = 0; l < 3; ++l) {
              const int i = 3 * k + l, j = 3 * l + k;
              const R to = scaled_t(trial_t(P, ht[i], eo[i], eo[j], k == l, tre), k == l, vol, fto);
              const R d1 = e[i] - eo[i], d2 = t[i] - to;
              de += d1 * d1;
              dt += d2 * d2;
              // full form: tau - tau_c = (t - <t>_prev) - A0 (e - E); the
              // constants tau_c = <t>_prev - A0 E only change the k = 0 term,
              // which the Green operator drops, and the transforms then round
              // relative to a field of fluctuations.  Increment form:
              // tau(e^i) - tau(e^{i-1}) = (t - t_prev) - A0 (e^i - e^{i-1}).
              R ae = a0 * de9[i] + b0 * de9[j];
              if (k == l) ae += c.ref.lam * trd;
              // manufactured source (eq. manufactured_polarization_stress); it
              // cancels in the increment form
              if (sv && !dout) ae += sv[i];
              zr[2 * i] = (t[i] - (dout ? to : tms[i])) - ae;
            }
          }
          de = sqrt(de);
          dt = sqrt(dt);
          dmax[0] = max(dmax[0], de); dmax[1] = max(dmax[1], dt);
          dsum[0] += de; dsum[1] += dt;
        } else {
#pragma unroll
          for (int q = 0; q < 9; ++q) de9[q] = e[q] - c.E[q];
          const R trd = de9[0] + de9[4] + de9[8];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int l = 0; l < 3; ++l) {
              const int i = 3 * k + l, j = 3 * l + k;
              R ae = a0 * de9[i] + b0 * de9[j];
              if (k == l) ae += c.ref.lam * trd;
              if (sv) ae += sv[i];
              zr[2 * i] = (t[i] - tms[i]) - ae;
            }
          }
        }
        if constexpr (sizeof(R) == 4) {
          pv4[0] = make_float4(e[0], e[1], e[2], e[3]);
          pv4[1] = make_float4(e[4], e[5], e[6], e[7]);
        } else {
#pragma unroll
          for (int q = 0; q < 8; ++q) pv[q] = e[q];
        }
        e8 = e[8];
      }
      // ---- micro level
      {
        R g[9], go[9], hm[9], m[9];
        if constexpr (sizeof(R) == 4) {
          const float4 q2 = pv4[2], q3 = pv4[3], q4 = pv4[4];
          const float4 h2 = hv4[2], h3 = hv4[3], h4 = hv4[4];
          go[0] = q2.y; go[1] = q2.z; go[2] = q2.w; go[3] = q3.x; go[4] = q3.y;
          go[5] = q3.z; go[6] = q3.w; go[7] = q4.x; go[8] = q4.y;
          hm[0] = h2.y; hm[1] = h2.z; hm[2] = h2.w; hm[3] = h3.x; hm[4] = h3.y;
          hm[5] = h3.z; hm[6] = h3.w; hm[7] = h4.x; hm[8] = h4.y;
        } else {
#pragma unroll
          for (int q = 0; q < 9; ++q) {
            go[q] = pv[9 + q];
            hm[q] = hv[9 + q];
          }
        }
        R dg9[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) dg9[q] = (MODE == kIter) ? zv[2 * (9 + q)] : R(0);
#pragma unroll
        for (int q = 0; q < 9; ++q) g[q] = (MODE == kIter) ? (din ? go[q] : c.G[q]) + dg9[q] : go[q];
        double qn = pq.y;
        return_micro<R, sizeof(R) == 4 ? 1 : 2>(P, g, hm, qn, m, qn, fm);
        if (MODE == kIter) {
          if (dout) {
#pragma unroll
            for (int q = 0; q < 9; ++q) dg9[q] = g[q] - go[q];
          }
          const R trd = dg9[0] + dg9[4] + dg9[8];
          const R trg = (go[0] + go[4]) + go[8];
          R dg = R(0), dm = R(0);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int l = 0; l < 3; ++l) {
              const int i = 3 * k + l, j = 3 * l + k;
              const R mo = trial_m(P, hm[i], go[i], go[j], k == l, trg) * fmo;
              const R d3 = g[i] - go[i], d4 = m[i] - mo;
              dg += d3 * d3;
              dm += d4 * d4;
              R bg = c.ref.beta * dg9[i] + c.ref.gamma * dg9[j];
              if (k == l) bg += c.ref.alpha * trd;
              if (sv && !dout) bg += sv[9 + i];
              zr[2 * (9 + i)] = (m[i] - (dout ? mo : tms[9 + i])) - bg;
            }
          }
          dg = sqrt(dg);
          dm = sqrt(dm);
          dmax[2] = max(dmax[2], dg); dmax[3] = max(dmax[3], dm);
          dsum[2] += dg; dsum[3] += dm;
        } else {
#pragma unroll
          for (int q = 0; q < 9; ++q) dg9[q] = g[q] - c.G[q];
          const R trd = dg9[0] + dg9[4] + dg9[8];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int l = 0; l < 3; ++l) {
              const int i = 3 * k + l, j = 3 * l + k;
              R bg = c.ref.beta * dg9[i] + c.ref.gamma * dg9[j];
              if (k == l) bg += c.ref.alpha * trd;
              if (sv) bg += sv[9 + i];
              zr[2 * (9 + i)] = (m[i] - tms[9 + i]) - bg;
            }
          }
        }
        if constexpr (sizeof(R) == 4) {
          pv4[2] = make_float4(e8, g[0], g[1], g[2]);
          pv4[3] = make_float4(g[3], g[4], g[5], g[6]);
          pv4[4] = make_float4(g[7], g[8], ft, fm);
        } else {
          pv[8] = e8;
#pragma unroll
          for (int q = 0; q < 9; ++q) pv[9 + q] = g[q];
          pv[18] = ft;
          pv[19] = fm;
        }
      }
    }
    if (MODE == kXInv) {
    __syncthreads();
    copy_values_out(fout_e + v0 * 9, prev_s, nvi * 9);
    copy_values_out(fout_g + v0 * 9, hist_s, nvi * 9);
    parity ^= 1u;
    return true;
  }
  // the new iterate goes back to global memory while the forward transform runs
  fence_proxy_async();
  __syncthreads();
  if (use_vox && threadIdx.x == 0) {
    bulk_store(c.prev + v0 * 20, prev_s, (uint32_t)(nvi * 20 * sizeof(R)));
    bulk_commit();
  }
  // ---------------------------------------------------------- forward x
  cpx<R>* X;
  if (sizeof(R) == 4 && packed && (M == 128 || M == 64 || M == 32)) {
    // FP32: the first stage of the compile-time plan, then its last stage
    // fused with the post-step (128: 16 x 8, 64: 8 x 8, 32: 8 x 4)
    cpx<R>* other = (zbuf == b0) ? b1 : b0;
    if (M == 128) stage_fixed<R, -1, 16, 1, 128>(zbuf, other, nr, tws);
    else if (M == 64) stage_fixed<R, -1, 8, 1, 64>(zbuf, other, nr, tws);
    else stage_fixed<R, -1, 8, 1, 32>(zbuf, other, nr, tws);
    __syncthreads();
    if (M == 128) x_forward_last_post<R, 128, 8>(other, zbuf, nr, tws);
    else if (M == 64) x_forward_last_post<R, 64, 8>(other, zbuf, nr, tws);
    else x_forward_last_post<R, 32, 4>(other, zbuf, nr, tws);
    X = zbuf;
  } else if (const XPlan P = x_plan(M); packed && P.count > 0) {
    // (the plan of a packed row; M = N1 / 2)
    x_fwd_planned<R>(zbuf, (zbuf == b0) ? b1 : b0, nr, M, P, tws);
    X = zbuf;
  } else if (packed) {
    cpx<R>* other = (zbuf == b0) ? b1 : b0;
    cpx<R>* Z = tile_fft_x_fwd<R>(zbuf, other, nr, c.px, tws);
    cpx<R>* dst = (Z == b0) ? b1 : b0;
    x_forward_post<R>(Z, dst, nr, M, msh, tws);
    X = dst;
  } else {
    X = zbuf;
  }
  fence_proxy_async();
  __syncthreads();
  if (threadIdx.x == 0) {
    bulk_store(c.spec + row0 * M * 18, X, (uint32_t)(nr * M * 18 * sizeof(cpx<R>)));
    bulk_commit();
  }
  // ---------------------------------------------------------- error partials of the item
  // Per-voxel norms of the FP32 (or FP64) field differences are formed in the
  // field type; their maxima are exact in any precision, and their sums (the
  // average measure) and the row sums behind the means are accumulated in FP64.
  if (MODE == kIter) {
    // the sums only enter the average measure (eq. err_average)
    const bool want_sum = c.err_kind != 0;
    if constexpr (MULTI) {
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const R mx = shfl_max(dmax[a]);
        const double sm = want_sum ? shfl_sum((double)dsum[a]) : 0.0;
        if (lane == 0) {
          red[warp * 8 + a] = (double)mx;
          red[warp * 8 + 4 + a] = sm;
        }
      }
    } else {
      R* cmx = reinterpret_cast<R*>(smem_raw + L.carry_off);
      double* csm = reinterpret_cast<double*>(cmx + 4 * kThreads);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        R& m = cmx[a * kThreads + threadIdx.x];
        m = max(m, dmax[a]);
        if (want_sum) csm[a * kThreads + threadIdx.x] += (double)dsum[a];
      }
    }
    // Row sums.  With the unnormalised inverse along x, sum_x e~ = N1 X_in[0],
    // so sum_x e = N1 (E + X_in[0]); the forward DC is sum_x tau.  Thread q + 36 k
    // sums value q over rows k, k + P, ... (P groups of 36 threads): the FP64
    // pipe takes a warp's instruction in 17 cycles however few lanes it has, and
    // 36 threads over all 16 rows of a 16^3 item kept it busy for 3200.
    double* csum = reinterpret_cast<double*>(smem_raw + L.carry_off + kThreads * (4 * sizeof(R) + 4 * sizeof(double)));
    const int P = (int)blockDim.x / 36, part = (int)threadIdx.x / 36, q = (int)threadIdx.x - 36 * part;
    double rsum = 0.0;
    if (part < P && part < nr) {
      if (q < 18) {
        const double mean = (double)((q < 9) ? c.E[q] : c.G[q - 9]);
        for (int rr = part; rr < nr; rr += P) rsum += (double)dcin[q * rows + rr];
        rsum = (double)N1 * ((double)((nr - part + P - 1) / P) * mean + rsum);
      } else {
        for (int rr = part; rr < nr; rr += P) rsum += (double)X[rr * M * 18 + (q - 18)].x;
      }
    }
    if constexpr (!MULTI) csum[threadIdx.x] += rsum;
    else csum[threadIdx.x] = rsum;
    if constexpr (MULTI) {
      __syncthreads();
      const int nwarp = blockDim.x >> 5;
      if (threadIdx.x < 36) {
        double v = csum[threadIdx.x];
        for (int k = 1; k < P && k < nr; ++k) v += csum[threadIdx.x + 36 * k];
        itm[8 + threadIdx.x] = v;
      } else if (threadIdx.x >= 64 && threadIdx.x < 72) {
        const int w0 = (int)threadIdx.x - 64;
        double v = red[w0];
        for (int w = 1; w < nwarp; ++w) {
          const double vv = red[w * 8 + w0];
          v = (w0 < 4) ? fmax(v, vv) : v + vv;
        }
        itm[w0] = v;
      }
    }
  }
  __syncthreads();
  parity ^= 1u;
  return true;
}

// ------------------------------------------------------------------ iteration error
// eq. err with eq. err_local (max) or eq. err_average (mean).  Denominators
// ||<a>|| are floored by their dimensional partner through the voxel size h
// (den_e >= h |<gamma>|, den_gamma >= |<e>| / h, den_t >= |<m>| / h,
// den_m >= h |<t>|), since ||<gamma>|| = 0 whenever the mean curvature is zero,
// each ||<a>|| taken as the larger of its value now and the largest of the
// converged increments so far (a cyclic load passes through zero means).
// out[0] = err, out[1..4] = err_e, err_t, err_gamma, err_m, out[5] = status.
// Run by warp 0 of the block, one lane per component, then one per field (the
// chip's FP64 pipe is narrow and its latency long: one thread took ~10 us);
// out[0..5] are written by lanes 0..3.
struct FinishScratch {
  double mean[18], dev[18], stress[18], norm[4], ratio[4];
};
template <class R>
__device__ __forceinline__ void finish_err(const CellDev<R>& c, const double* s, int err_kind, double* out,
                                           FinishScratch& w) {
  const int lane = threadIdx.x;
  const double iv = c.inv_nvox;
  const int lev = lane < 9 ? 0 : 1, i = lane - 9 * lev;  // lanes 0..17: component i of the macro / micro level
  if (lane < 18) {
    const double mean = s[8 + lane] * iv;
    w.mean[lane] = mean;
    w.dev[lane] = mean - (double)(lev == 0 ? c.E[i] : c.G[i]);
  }
  __syncwarp();
  // The transformed polarization was tau - tau_c = (t - T_c) - A0 (e - E) (T_c =
  // c.tmean as read by pass A), so <t> = <tau - tau_c> + T_c + A0 (<e> - E) and
  // likewise <m>; <t>, <m> then become the constants of the next iteration.
  // In the increment form it was (t - t_prev) - A0 (e - e_prev), so the same
  // formula holds with T_c = <t_prev> (the unrounded last mean) and
  // <e_prev> = E.
  if (lane < 18) {
    const int k = i / 3, l = i - 3 * k, j = 3 * l + k;
    const double* x = w.dev + 9 * lev;
    const double a = lev == 0 ? (double)c.ref.mu + (double)c.ref.kap : (double)c.ref.beta;
    const double b = lev == 0 ? (double)c.ref.mu - (double)c.ref.kap : (double)c.ref.gamma;
    const double d = lev == 0 ? (double)c.ref.lam : (double)c.ref.alpha;
    const double tr = x[0] + x[4] + x[8];
    const double tc = c.delta_out ? c.tmean[lane] : (double)(R)c.tmean[lane];
    const double m = s[26 + lane] * iv + tc + a * x[i] + b * x[j] + (k == l ? d * tr : 0.0);
    w.stress[lane] = m;
    c.tmean[lane] = m;
  }
  __syncwarp();
  // fields in the order e, t, gamma, m; magnitudes: the means now or, if
  // larger, the largest of the converged increments so far (a cyclic load
  // passing through a zero mean)
  if (lane < 4) {
    const double* v = ((lane & 1) ? w.stress : w.mean) + 9 * (lane >> 1);
    double n = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) n += v[q] * v[q];
    w.norm[lane] = fmax(sqrt(n), c.tmean[18 + lane]);
  }
  __syncwarp();
  if (lane < 4) {
    const double h = c.h;
    const double other = w.norm[lane ^ 2];  // the dimensional partner: e - gamma, t - m
    const double den = fmax(w.norm[lane], (lane == 0 || lane == 3) ? h * other : other / h);
    const double num = (err_kind == 0) ? s[lane] : s[4 + lane] * iv;
    const double ea = den == 0.0 ? (num == 0.0 ? 0.0 : INFINITY) : num / den;
    w.ratio[lane] = ea;
    out[1 + lane] = ea;
  }
  __syncwarp();
  if (lane == 0) {
    double err = 0.0;
    for (int a = 0; a < 4; ++a)
      if (!(w.ratio[a] <= err)) err = w.ratio[a];  // propagates NaN
    out[0] = err;
    out[5] = c.status ? (double)__ldcg(c.status) : 0.0;
  }
}

// Fixed-order FP64 fold of `nparts` records of NQ doubles (max for the first
// NMAX values, sums for the rest) by one block of kFoldThreads; the total
// lands in s[].  Thread (q, g) folds value q over the g-th contiguous range of
// records in record order (neighbouring q read neighbouring doubles), then
// thread q folds the ranges in order.  The loop is bound by the latency of its
// loads and FP64 additions, so the ranges are as many as the block holds.
constexpr int kFoldThreads = 512;
template <int NQ>
constexpr int kFoldGroups = kFoldThreads / NQ;
template <int NQ, int NMAX>
__device__ __forceinline__ void fold_records(const double* __restrict__ records, long long nparts, double* s,
                                             double (*part)[NQ]) {
  constexpr int NG = kFoldGroups<NQ>;
  const int t = threadIdx.x;
  if (t < NG * NQ) {
    const int q = t % NQ, g = t / NQ;
    const long long per = (nparts + NG - 1) / NG;
    const long long b0 = (long long)g * per;
    const long long b1 = (b0 + per < nparts) ? b0 + per : nparts;
    double v = 0.0;
#pragma unroll 8
    for (long long b = b0; b < b1; ++b) {
      const double x = records[b * NQ + q];
      v = (q < NMAX) ? fmax(v, x) : v + x;
    }
    part[g][q] = v;
  }
  __syncthreads();
  if (t < NQ) {
    double v = part[0][t];
#pragma unroll
    for (int g = 1; g < NG; ++g) v = (t < NMAX) ? fmax(v, part[g][t]) : v + part[g][t];
    s[t] = v;
  }
  __syncthreads();
}

// The error reduction of a single cell, by the blocks of pass A themselves: the
// last block of each group of kTailGroup to finish folds the group's records,
// the last group's block folds those and forms the error measure (a launch of
// its own took 15 us: one SM's FP64 pipe, two lanes wide, had all 304 records
// to add).  Records are folded in index order, so the result does not depend
// on which blocks come last.
// loop: decide the fixed-point loop on the device (Algorithm 2's while test)
// for a launch inside a conditional WHILE node: out[6] counts the iterations
// of the loop, which continues while no failure is recorded, err is finite,
// err <= div_limit, err > tol, fewer than max_iter iterations ran and
// (stag > 0) the stagnation watch (stall_step with window stag) has not
// tripped: out[7], out[8] hold the last low and its iteration, out[10] the
// longest gap between lows, out[9] = 1 records a stop by the watch.
// out[11]: nanoseconds from the end of the last block's items to here, the
// reduction's share of pass A.
constexpr int kTailGroup = 16;
template <class R>
__device__ void finish_blocks(const CellDev<R>& c, double* partials, const double* acc, const ErrTail& tail) {
  constexpr int NQ = kErrPartials, SPLIT = 2;
  __shared__ double part[SPLIT][NQ], s[NQ];
  __shared__ FinishScratch fin;
  __shared__ int last;
  const unsigned long long entered = globaltimer_ns();
  const int t = threadIdx.x, grid = (int)gridDim.x, group = (int)blockIdx.x / kTailGroup;
  const int groups = (grid + kTailGroup - 1) / kTailGroup;
  double* records = partials + (long long)kTailRecords * NQ;  // the blocks', after the groups'
  // true in every thread of the block that finished last of `of`
  auto arrive = [&](unsigned* counter, int of) {
    __threadfence();
    __syncthreads();
    if (t == 0) {
      last = atomicAdd(counter, 1u) == (unsigned)(of - 1);
      if (last) *counter = 0u;  // for the next launch
    }
    __syncthreads();
    if (last) __threadfence();
    return last != 0;
  };
  // folds n records at r into s (max for the first four values, sums else)
  auto fold = [&](const double* r, int n) {
    const int q = t % NQ, g = t / NQ, per = (n + SPLIT - 1) / SPLIT;
    if (g < SPLIT) {
      double v = 0.0;
#pragma unroll 8
      for (int b = g * per; b < min(n, (g + 1) * per); ++b) {
        const double x = __ldcg(r + (long long)b * NQ + q);
        v = (q < 4) ? fmax(v, x) : v + x;
      }
      part[g][q] = v;
    }
    __syncthreads();
    if (t < NQ) s[t] = (t < 4) ? fmax(part[0][t], part[1][t]) : part[0][t] + part[1][t];
    __syncthreads();
  };
  for (int i = t; i < NQ; i += blockDim.x) records[(long long)blockIdx.x * NQ + i] = acc[i];
  const int size = min(kTailGroup, grid - group * kTailGroup);
  if (!arrive(tail.counters + group, size)) return;
  fold(records + (long long)group * kTailGroup * NQ, size);
  if (t < NQ) partials[group * NQ + t] = s[t];
  if (!arrive(tail.counters + kTailRecords, groups)) return;
  fold(partials, groups);
  if (t < 32) finish_err<R>(c, s, tail.err_kind, tail.out, fin);
  if (t == 0) tail.out[11] = (double)(globaltimer_ns() - entered);
  if (t == 0 && tail.loop) {
    double* out = tail.out;
    const int it = (int)out[6] + 1;
    out[6] = (double)it;
    const double err = out[0];
    bool go = out[5] == 0.0 && isfinite(err) && err <= tail.div_limit && err > tail.tol && it < tail.max_iter;
    if (go && tail.stag > 0) {
      double ref_err = out[7];
      int it_ref = (int)out[8], gap = (int)out[10];
      if (stall_step(err, it, tail.stag, tail.adapt != 0, ref_err, it_ref, gap)) {
        go = false;
        out[9] = 1.0;
      }
      out[7] = ref_err;
      out[8] = (double)it_ref;
      out[10] = (double)gap;
    }
    cudaGraphSetConditional(tail.handle, go ? 1u : 0u);
  }
}

// Pass A over a cell (single: per-block error totals in `partials`) or over
// the entries of a multi-cell launch (per-item partials in each cell's ipart).
template <class R, int MODE, bool MULTI>
__global__ void __launch_bounds__(kThreads, (sizeof(R) == 4 ? 2 : 1))
    k_pass_a(CellDev<R> c0, Work<R> w, double* partials, const R* fin_tau, const R* fin_mu,
             R* fout_e, R* fout_g, ErrTail tail) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ CellDev<R> cs;
  __shared__ double itm[kErrPartials];
  __shared__ R tms[18];  // <t>, <m> of the cell's previous iteration (subtracted constants)
  double* acc = reinterpret_cast<double*>(smem_raw + PassASmem<R>::acc_off);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw + PassASmem<R>::bar_off);
  if (threadIdx.x == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    fence_barrier_init();
  }
  for (int i = threadIdx.x; i < kErrPartials; i += blockDim.x) acc[i] = 0.0;
  __syncthreads();
  uint32_t parity = 0;
  bool failed = false;
  int* status = c0.status;
  // the per-thread carries (error maxima and sums, row sums) start at zero; they
  // sit after the item buffers for the block's row count
  const PassASmem<R> SL(c0.n1 > 0 ? c0.n1 : 1, c0.rows_a > 0 ? c0.rows_a : 1);
  if constexpr (!MULTI) {
    R* cmx = reinterpret_cast<R*>(smem_raw + SL.carry_off);
    double* csm = reinterpret_cast<double*>(cmx + 4 * kThreads);
    for (int a = 0; a < 4; ++a) {
      cmx[a * kThreads + threadIdx.x] = R(0);
      csm[a * kThreads + threadIdx.x] = 0.0;
    }
    csm[4 * kThreads + threadIdx.x] = 0.0;
  }
  for_items<R, MULTI>(c0, c0.items_a, w, cs, [&](const CellDev<R>& c, long long item, bool fresh) {
    if (failed) {
      flag_timeout(c.status);  // every cell with a skipped item reports the failure
      return;
    }
    if (!pass_a_item<R, MODE, MULTI>(c, item, smem_raw, parity, itm, tms, fin_tau, fin_mu, fout_e, fout_g,
                                     fresh)) {
      failed = true;
      status = c.status;
      return;
    }
    if (MODE == kIter) {
      if constexpr (MULTI) {
        for (int i = threadIdx.x; i < kErrPartials; i += blockDim.x)
          c.ipart[item * kErrPartials + i] = itm[i];
        __syncthreads();
      }
    }
  });
  if (MODE == kIter && !MULTI && !failed) {
    // the block's error maxima and sums from the per-thread carries
    double* red = reinterpret_cast<double*>(smem_raw + PassASmem<R>::red_off);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const R* cmx = reinterpret_cast<const R*>(smem_raw + SL.carry_off);
      const double* csm = reinterpret_cast<const double*>(cmx + 4 * kThreads);
      const R mx = shfl_max(cmx[a * kThreads + threadIdx.x]);
      const double sm = shfl_sum(csm[a * kThreads + threadIdx.x]);
      if (lane == 0) {
        red[warp * 8 + a] = (double)mx;
        red[warp * 8 + 4 + a] = sm;
      }
    }
    __syncthreads();
    if (threadIdx.x < 8) {
      double a = red[threadIdx.x];
      for (int wi = 1; wi < (int)(blockDim.x >> 5); ++wi) {
        const double vv = red[wi * 8 + threadIdx.x];
        a = (threadIdx.x < 4) ? fmax(a, vv) : a + vv;
      }
      acc[threadIdx.x] = a;
    }
    if (threadIdx.x < 36) {
      const double* csum = reinterpret_cast<const double*>(smem_raw + SL.carry_off +
                                                           kThreads * (4 * sizeof(R) + 4 * sizeof(double)));
      double v = csum[threadIdx.x];
      for (int k = 1; k < (int)blockDim.x / 36; ++k) v += csum[threadIdx.x + 36 * k];
      acc[8 + threadIdx.x] = v;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) bulk_wait_all();
  if (failed) {
    // wait (bounded) for this block's loads still in flight, then report
    if (threadIdx.x == 0) {
      if (MODE == kIter || MODE == kXInv) mbar_wait(&bars[0], parity);
      if (MODE == kIter || MODE == kStart) mbar_wait(&bars[1], parity);
    }
    __syncthreads();
    flag_timeout(status);
  }
  // (a failed block still counts as finished: the last one reports the status)
  if constexpr (MODE == kIter && !MULTI) finish_blocks<R>(c0, partials, acc, tail);
}

// Algorithm 2's loop test for one batched cell after an iteration whose error
// row is e (err, four terms, status), with the batched engine's FP32
// stagnation watch; the same comparisons, in the same order and arithmetic,
// as the host's replay of the rows.
__device__ void round_decide(RoundCtl& rc, const double* e) {
  const double err = e[0];
  rc.it += 1;
  rc.rounds += 1;
  bool stop = false;
  if (e[5] != 0.0) {
    stop = true;  // a bounded wait expired
  } else if (!isfinite(err) || err > rc.div_limit) {
    stop = true;  // diverged
  } else {
    const bool more = rc.target >= 0 ? rc.it < rc.target : err > rc.tol;
    if (!more) {
      stop = true;  // converged, or the prescribed count reached
    } else if (rc.target < 0 && rc.it >= rc.max_iter) {
      stop = true;  // not converged
    } else if (rc.stag_iters > 0) {
      // the host switches the schedule where the watch trips
      if (stall_step(err, rc.it, rc.stag_iters, rc.adapt != 0, rc.ref_err, rc.it_ref, rc.gap)) stop = true;
    }
  }
  if (rc.rounds >= rc.max_rounds) stop = true;
  rc.stop = stop ? 1 : 0;
}

// One cluster of kFoldCluster blocks per entry: each folds a quarter of the
// cell's per-item records on its own SM's FP64 pipe (one block took 24 us for
// the 461 records of a 48^3 cell), the first takes the others' totals from
// their shared memory, in rank order.
constexpr int kFoldCluster = 4;
template <class R>
__global__ void __cluster_dims__(kFoldCluster, 1, 1) __launch_bounds__(kFoldThreads) k_reduce_err_multi(Work<R> w) {
  namespace cg = cooperative_groups;
  __shared__ double s[kErrPartials];
  __shared__ double part[kFoldGroups<kErrPartials>][kErrPartials];
  __shared__ FinishScratch fin;
  __shared__ CellDev<R> cs;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  load_cell(cs, w.cells + w.act[blockIdx.x / kFoldCluster]);
  __syncthreads();
  RoundCtl* rc = cs.rctl;
  // (uniform over the cluster: the flag only changes at the end of this kernel,
  // after the cluster's last barrier)
  if (rc != nullptr && __ldcg(&rc->stop) != 0) return;
  const long long per = (cs.items_a + kFoldCluster - 1) / kFoldCluster, b0 = rank * per;
  const long long n = cs.items_a - b0 < per ? cs.items_a - b0 : per;
  fold_records<kErrPartials, 4>(cs.ipart + b0 * kErrPartials, n > 0 ? n : 0, s, part);
  cluster.sync();
  if (rank == 0 && threadIdx.x < kErrPartials) {
    double v = s[threadIdx.x];
    for (int k = 1; k < kFoldCluster; ++k) {
      const double x = cluster.map_shared_rank(s, k)[threadIdx.x];
      v = (threadIdx.x < 4) ? fmax(v, x) : v + x;
    }
    s[threadIdx.x] = v;
  }
  cluster.sync();  // the others' shared memory lives until it has been read
  if (rank == 0 && threadIdx.x < 32) {
    double* out = rc != nullptr ? rc->rows + 8 * rc->rounds : cs.err_out;
    finish_err<R>(cs, s, cs.err_kind, out, fin);
    __syncwarp();
    if (threadIdx.x == 0 && rc != nullptr) round_decide(*rc, out);
  }
}

// ------------------------------------------------------------------ state set-up
// Zero initial state (Algorithm 2 initialisation) and the first predictor
// e = E, gamma = Gamma of the first load increment.  Items: 256-voxel chunks.
template <class R>
__device__ __forceinline__ void init_chunk(const CellDev<R>& c, long long chunk) {
  const long long v = chunk * 256 + threadIdx.x;
  if (threadIdx.x >= 256 || v >= c.nvox) return;
  R* pv = c.prev + v * 20;
  R* hv = c.hist + v * 20;
  R* el = c.elast + v * 18;
  // in 16- / 8-byte pieces (value by value a 256^3 FP32 cell took 4.9 ms)
  R rec[20];
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    rec[q] = c.E[q];
    rec[9 + q] = c.G[q];
  }
  rec[18] = rec[19] = R(1);
  store_rec(pv, rec);
#pragma unroll
  for (int q = 0; q < 20; ++q) rec[q] = R(0);
  store_rec18(el, rec);
  rec[18] = (R)c.phase[v];  // phase id travels with the history record
  store_rec(hv, rec);
  reinterpret_cast<double2*>(c.pq)[v] = make_double2(0.0, 0.0);
}

template <class R, bool MULTI>
__global__ void __launch_bounds__(256) k_init(CellDev<R> c0, Work<R> w) {
  __shared__ CellDev<R> cs;
  for_items<R, MULTI>(c0, (c0.nvox + 255) / 256, w, cs,
                      [&](const CellDev<R>& c, long long chunk, bool) { init_chunk<R>(c, chunk); });
}

// ------------------------------------------------------------------ commit
// Error-free sum of two single-precision values (Knuth's TwoSum): s + err =
// a + b exactly.  Accumulating x into (hi, lo) as hi, err = TwoSum(hi, x),
// lo += err is compensated summation: the pair carries the running sum to
// about 2^-48 of its magnitude, so per-thread sums of FP32 values lose
// nothing against an FP64 accumulator at the voxel counts of one thread, at
// six single-precision additions instead of one FP64 addition.
__device__ __forceinline__ void two_sum_acc(float2& acc, float x) {
  const float s = __fadd_rn(acc.x, x);
  const float bb = __fsub_rn(s, acc.x);
  const float err = __fadd_rn(__fsub_rn(acc.x, __fsub_rn(s, bb)), __fsub_rn(x, bb));
  acc.x = s;
  acc.y = __fadd_rn(acc.y, err);
}

// Algorithm 2, end of a load increment: the converged iterate becomes the
// history of Algorithm 1; homogenized sums; when c.predict, the linear-
// extrapolation predictor of the next increment, e' = e_n + ratio (e_n - e_{n-1}).
// Per 256-voxel chunk: sums of t (9), m (9), e (9), gamma (9), p, q, t_eq, m_eq
// in that order (p and q are FP64 values, the others field-type values).
// COLS: instead of reducing the chunk, add the thread's values to its own
// column of `cols` ([kAvgPartials][blockDim] 8-byte slots; single-cell
// commit): FP64 columns for FP64 fields and for p, q, compensated FP32
// (hi, lo) pairs for the field-type values of FP32 fields.
template <class R, bool COLS>
__device__ __forceinline__ void commit_chunk(const CellDev<R>& c, long long chunk, double* out40,
                                             double (*red)[kAvgPartials], double* cols) {
  R val[kAvgPartials];  // [36], [37] unused (p, q are FP64)
#pragma unroll
  for (int i = 0; i < kAvgPartials; ++i) val[i] = R(0);
  double p = 0.0, q = 0.0;
  const long long v = chunk * 256 + threadIdx.x;
  if (threadIdx.x < 256 && v < c.nvox) {
    // records move in 16- / 8-byte pieces (they are 80 / 72 bytes apart)
    R* pv = c.prev + v * 20;
    R* hv = c.hist + v * 20;
    R pr[20], hr[20];
    load_rec(pv, pr);
    load_rec(hv, hr);
    const R* e = pr;
    const R* g = pr + 9;
    const PhaseDev<R>& P = c.phases[(int)hr[18]];
    double2 pq = reinterpret_cast<const double2*>(c.pq)[v];
    R t[9], m[9];
    R ft, fm;
    radial_return<R>(P, e, g, hr, hr + 9, pq.x, pq.y, t, m, p, q, ft, fm);
    R ae[9], bg[9];
    apply_A<R>(P.lam, P.mu, P.kap, e, ae);
    apply_B<R>(P.alpha, P.beta, P.gamma, g, bg);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      val[i] = t[i];
      val[9 + i] = m[i];
      val[18 + i] = e[i];
      val[27 + i] = g[i];
      hr[i] = t[i] - ae[i];
      hr[9 + i] = m[i] - bg[i];
    }
    store_rec(hv, hr);
    reinterpret_cast<double2*>(c.pq)[v] = make_double2(p, q);
    equivalents<R>(P, t, m, val[38], val[39]);
    if (c.predict) {
      const R ratio = (R)c.ratio;
      R* el = c.elast + v * 18;
      R old[18];
      load_rec18(el, old);
      store_rec18(el, pr);  // e, gamma (the first 18 values of the iterate record)
#pragma unroll
      for (int i = 0; i < 18; ++i) pr[i] = pr[i] + ratio * (pr[i] - old[i]);
      store_rec(pv, pr);    // the predictor, with the last scale factors
    }
  }
  const int bd = (int)blockDim.x;
  if constexpr (COLS) {
    // thread-private columns: no cross-thread work per chunk
    double* dc = cols + threadIdx.x;
#pragma unroll
    for (int i = 0; i < kAvgPartials; ++i) {
      if (i == 36) {
        dc[i * bd] += p;
      } else if (i == 37) {
        dc[i * bd] += q;
      } else if constexpr (sizeof(R) == 4) {
        float2* fc = reinterpret_cast<float2*>(dc + i * bd);
        float2 a = *fc;
        two_sum_acc(a, (float)val[i]);
        *fc = a;
      } else {
        dc[i * bd] += (double)val[i];
      }
    }
    return;
  }
  // Records per chunk: the field-type values are transposed through shared
  // memory and summed in FP64 by (value, part) threads, p and q by warp
  // shuffles.  (Shuffling all 40 values cost 1600 warp additions a chunk on the
  // FP64 pipe, 17 cycles each: the commit of a 32-cell batch took 755 us.  The
  // 344 of this form cost a 512-cell batch nothing against FP32 pairs, which
  // keep fewer bits: 14.50 s with either.)
  constexpr int PITCH = 257, PARTS = 6, LEN = (256 + PARTS - 1) / PARTS;
  R* tile = reinterpret_cast<R*>(cols);  // [kAvgPartials][PITCH]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
#pragma unroll
  for (int i = 0; i < kAvgPartials; ++i)
    if (i != 36 && i != 37) tile[i * PITCH + t] = val[i];
  const double ps = shfl_sum(p), qs = shfl_sum(q);
  if (lane == 0) {
    red[warp][36] = ps;
    red[warp][37] = qs;
  }
  __syncthreads();
  if (t < PARTS * kAvgPartials) {
    const int i = t % kAvgPartials, part = t / kAvgPartials;
    if (i != 36 && i != 37) {
      const R* v = tile + i * PITCH;
      const int k1 = min(256, (part + 1) * LEN);
      double sm = 0.0;
#pragma unroll 4
      for (int k = part * LEN; k < k1; ++k) sm += (double)v[k];
      red[part][i] = sm;
    }
  }
  __syncthreads();
  if (t < kAvgPartials) {
    double sm = 0.0;
    const int n = (t == 36 || t == 37) ? (bd >> 5) : PARTS;
    for (int k = 0; k < n; ++k) sm += red[k][t];
    out40[t] = sm;
  }
  __syncthreads();
}

// Single: each thread accumulates its voxels' values in its own shared-memory
// column across the block's chunks (FP64, or compensated FP32 pairs for the
// values of FP32 fields); the block folds the columns once, in FP64, into
// partials[block][40] (a fixed grid gives a fixed order).  Multi:
// per-chunk records in each cell's apart.
template <class R, bool MULTI>
__global__ void __launch_bounds__(256) k_commit(CellDev<R> c0, Work<R> w, double* partials) {
  // single: [kAvgPartials][256] 8-byte slots; multi: the chunk's values, [kAvgPartials][257] of R
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ CellDev<R> cs;
  __shared__ double red[8][kAvgPartials];
  __shared__ double chunk_sum[kAvgPartials];
  double* cols = reinterpret_cast<double*>(smem_raw);
  if constexpr (!MULTI) {
    for (int i = threadIdx.x; i < kAvgPartials * (int)blockDim.x; i += blockDim.x) cols[i] = 0.0;
  }
  for_items<R, MULTI>(c0, (c0.nvox + 255) / 256, w, cs, [&](const CellDev<R>& c, long long chunk, bool) {
    commit_chunk<R, !MULTI>(c, chunk, chunk_sum, red, cols);
    if constexpr (MULTI) {
      if (threadIdx.x < kAvgPartials) c.apart[chunk * kAvgPartials + threadIdx.x] = chunk_sum[threadIdx.x];
      __syncthreads();
    }
  });
  if constexpr (!MULTI) {
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = warp; i < kAvgPartials; i += nw) {
      const bool pair = sizeof(R) == 4 && i != 36 && i != 37;  // compensated FP32 (hi, lo) column
      double sm = 0.0;
      for (int k = lane; k < (int)blockDim.x; k += 32) {
        if (pair) {
          const float2 a = reinterpret_cast<const float2*>(cols)[i * blockDim.x + k];
          sm += (double)a.x + (double)a.y;
        } else {
          sm += cols[i * blockDim.x + k];
        }
      }
      sm = shfl_sum(sm);
      if (lane == 0) partials[(long long)blockIdx.x * kAvgPartials + i] = sm;
    }
  }
}

// The loading-history magnitudes of the error measure (cell scalars 18..21)
// after a committed increment whose averages are row[0..35] (T, M, <e>, <gamma>):
// lanes 0..3 form ||<e>||, ||T||, ||<gamma>||, ||M||.
__device__ __forceinline__ void update_history(const double* row, double* scalars) {
  const int a = threadIdx.x;
  if (a < 4) {
    const double* v = row + ((a & 1) ? 0 : 18) + 9 * (a >> 1);
    double n = 0.0;
    for (int q = 0; q < 9; ++q) n += v[q] * v[q];
    scalars[18 + a] = fmax(scalars[18 + a], sqrt(n));
  }
}

// Sum of commit records (block partials of a single cell, chunk records of a
// batched one) in a fixed order, divided by the voxel count.  (The commit of a
// 64^3 cell with its averages took 67.5 us with one thread per value, 52 so.)
__device__ __forceinline__ void average_records(const double* records, long long n, double inv_nvox, double* out,
                                                double* scalars) {
  __shared__ double row[kAvgPartials];
  __shared__ double part[kFoldGroups<kAvgPartials>][kAvgPartials];
  fold_records<kAvgPartials, 0>(records, n, row, part);
  if (threadIdx.x < kAvgPartials) out[threadIdx.x] = row[threadIdx.x] = row[threadIdx.x] * inv_nvox;
  __syncthreads();
  update_history(row, scalars);
}

__global__ void __launch_bounds__(kFoldThreads) k_reduce_avg(const double* partials, int nparts, double inv_nvox,
                                                             double* out, double* scalars) {
  average_records(partials, nparts, inv_nvox, out, scalars);
}

// One block per entry: the cell's chunk records -> c.avg_out.
template <class R>
__global__ void __launch_bounds__(kFoldThreads) k_reduce_avg_multi(Work<R> w) {
  __shared__ CellDev<R> cs;
  load_cell(cs, w.cells + w.act[blockIdx.x]);
  __syncthreads();
  average_records(cs.apart, (cs.nvox + 255) / 256, cs.inv_nvox, cs.avg_out, cs.tmean);
}

// Final-state fields in FP64: e, gamma from `src` (prev or elast), t = h_t + A e,
// m = h_m + B gamma (the history form of the converged stresses), p, q.
template <class R>
__global__ void k_fields(CellDev<R> c, const R* src, int src_stride, double* fe, double* fg,
                         double* ft, double* fm, double* fp, double* fq) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < c.nvox;
       v += (long long)gridDim.x * blockDim.x) {
    const R* s = src + v * src_stride;
    const R* hv = c.hist + v * 20;
    R e[9], g[9], t[9], m[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      e[q] = s[q];
      g[q] = s[9 + q];
    }
    const PhaseDev<R> P = c.phases[c.phase[v]];
    apply_A<R>(P.lam, P.mu, P.kap, e, t);
    apply_B<R>(P.alpha, P.beta, P.gamma, g, m);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      if (fe) fe[v * 9 + q] = (double)e[q];
      if (fg) fg[v * 9 + q] = (double)g[q];
      if (ft) ft[v * 9 + q] = (double)(hv[q] + t[q]);
      if (fm) fm[v * 9 + q] = (double)(hv[9 + q] + m[q]);
    }
    if (fp) fp[v] = c.pq[2 * v];
    if (fq) fq[v] = c.pq[2 * v + 1];
  }
}

// ------------------------------------------------------------------ component: Algorithm 1
// Material points in chunks of one block's threads.  The six input tensors of
// a chunk (9 values a point) come in through shared memory: read from global
// memory value by value they are 36 (72) bytes apart, and every load of a warp
// touched nine times the sectors it used (2.1 M FP32 points took 212 us).  The
// copies are 16-byte pieces when every array starts on a 16-byte boundary
// (VEC), else single values; a point's 9 values are an odd stride, so reading
// them back is free of bank conflicts.  The stresses leave the same way.
template <class R>
struct PointArrays {
  const uint16_t* phase;
  const R* in[6];  // e, gamma, e_n, gamma_n, t_n, m_n
  const double *p_n, *q_n;
  R* out[2];  // t, m
  double *p, *q;
};
// Phase tables of up to this many rows travel as a kernel argument; larger
// ones lie in global memory.
constexpr int kTablePhases = 12;
template <class R>
struct PhaseTable {
  PhaseDev<R> row[kTablePhases];
};
constexpr int kPointThreads = 128;

template <class R, bool VEC>
__global__ void __launch_bounds__(kPointThreads)
    k_radial_return_points(const __grid_constant__ PhaseTable<R> table, const PhaseDev<R>* phases, int n_phases,
                           long long count, const __grid_constant__ PointArrays<R> P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int chunk = (int)blockDim.x, words = 9 * chunk;
  R* in = reinterpret_cast<R*>(smem_raw);  // [6][words]
  PhaseDev<R>* rows = reinterpret_cast<PhaseDev<R>*>(in + 6 * words);
  if (!phases) {
    const int* src = reinterpret_cast<const int*>(table.row);
    for (int i = threadIdx.x; i < n_phases * (int)(sizeof(PhaseDev<R>) / 4); i += blockDim.x)
      reinterpret_cast<int*>(rows)[i] = src[i];
  }
  constexpr int PV = 16 / (int)sizeof(R);  // values per 16-byte piece
  for (long long base = (long long)blockIdx.x * chunk; base < count; base += (long long)gridDim.x * chunk) {
    const int n = (int)(count - base < chunk ? count - base : chunk);
    const int nv = VEC ? 9 * n / PV : 0;  // pieces; the rest value by value
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      const R* src = P.in[a] + base * 9;
      R* dst = in + a * words;
      for (int i = threadIdx.x; i < nv; i += blockDim.x) cp_async16(dst + i * PV, src + i * PV);
      for (int i = nv * PV + threadIdx.x; i < 9 * n; i += blockDim.x) cp_async_value(dst + i, src + i);
    }
    const int i = threadIdx.x;
    int pid = 0;
    double pn = 0.0, qn = 0.0;
    if (i < n) {
      pid = min((int)P.phase[base + i], n_phases - 1);
      pn = P.p_n[base + i];
      qn = P.q_n[base + i];
    }
    cp_async_wait_all();
    __syncthreads();
    if (i < n) {
      const PhaseDev<R>& ph = phases ? phases[pid] : rows[pid];
      const R *pe = in + 9 * i, *pg = pe + words, *pen = pg + words, *pgn = pen + words, *ptn = pgn + words,
              *pmn = ptn + words;
      R ee[9], gg[9], en[9], gn[9], ht[9], hm[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        ee[k] = pe[k];
        gg[k] = pg[k];
        en[k] = pen[k];
        gn[k] = pgn[k];
      }
      // history form of eq. trial_stresses: h_t = t_n - A e_n, h_m = m_n - B gamma_n
      apply_A<R>(ph.lam, ph.mu, ph.kap, en, ht);
      apply_B<R>(ph.alpha, ph.beta, ph.gamma, gn, hm);
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        ht[k] = ptn[k] - ht[k];
        hm[k] = pmn[k] - hm[k];
      }
      R tt[9], mm[9];
      double pp, qq;
      R ft, fm;
      radial_return<R>(ph, ee, gg, ht, hm, pn, qn, tt, mm, pp, qq, ft, fm);
      // the point's stresses take the place of its strains
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        in[9 * i + k] = tt[k];
        in[words + 9 * i + k] = mm[k];
      }
      P.p[base + i] = pp;
      P.q[base + i] = qq;
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      R* dst = P.out[a] + base * 9;
      const R* src = in + a * words;
      for (int k = threadIdx.x; k < nv; k += blockDim.x)
        reinterpret_cast<float4*>(dst)[k] = reinterpret_cast<const float4*>(src)[k];
      for (int k = nv * PV + threadIdx.x; k < 9 * n; k += blockDim.x) dst[k] = src[k];
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ launchers

template <class R>
size_t smem_pass_a(int n1, int rows) { return PassASmem<R>(n1, rows).total; }

template <class R>
constexpr size_t kCommitTile = (size_t)kAvgPartials * 257 * sizeof(R);  // multi-cell commit, a chunk's values
constexpr size_t kCommitSmem = (size_t)kAvgPartials * 256 * sizeof(double);  // single-cell commit columns

namespace {
struct RuntimeApi {
  using Error = cudaError_t;
  static constexpr Error ok = cudaSuccess, invalid = cudaErrorInvalidValue;
  static Error device(int& dev) { return cudaGetDevice(&dev); }
  static Error static_smem(const void* fn, size_t& bytes) {
    cudaFuncAttributes fa;
    const Error e = cudaFuncGetAttributes(&fa, fn);
    bytes = e == cudaSuccess ? fa.sharedSizeBytes : 0;
    return e;
  }
  static Error raise(const void* fn, size_t bytes) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  }
  static Error occupancy(const void* fn, int threads, size_t smem, int& blocks) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, threads, smem);
  }
};

KernelLimits<RuntimeApi>& kernel_limits() {
  static KernelLimits<RuntimeApi> limits(kSmemOptin, kSmemStaticReserve);
  return limits;
}
}  // namespace

cudaError_t raise_smem(const void* fn, bool tiled) { return kernel_limits().raise(fn, tiled); }

int resident_blocks(const void* fn, int threads, size_t smem, bool tiled) {
  return std::max(1, kernel_limits().resident(fn, tiled, threads, smem));
}

template <class R>
int grid_for(const void* fn, int threads, size_t smem, long long work, int nsm, bool tiled = true) {
  const long long g = std::min<long long>(work, (long long)resident_blocks(fn, threads, smem, tiled) * nsm);
  return (int)std::max<long long>(g, 1);
}

template <class R>
cudaError_t launch_fft_y(const LaunchCfg& L, const CellDev<R>& c, int dir, cudaStream_t st) {
  if (c.n2 == 1) return cudaSuccess;
  return dir < 0 ? launch_line<R, kYForward>(c, L.grid_y, st) : launch_line<R, kYInverse>(c, L.grid_y, st);
}

template <class R>
cudaError_t launch_green_z(const LaunchCfg& L, const CellDev<R>& c, cudaStream_t st) {
  return c.n2 == 1 ? launch_line<R, kZFull>(c, L.grid_z, st) : launch_line<R, kZReduced>(c, L.grid_z, st);
}

template <class R>
cudaError_t launch_pass_a_iter(const LaunchCfg& L, const CellDev<R>& c, double* partials, const ErrTail& tail,
                               cudaStream_t st) {
  const cudaError_t e = raise_smem((const void*)k_pass_a<R, kIter, false>, true);
  if (e != cudaSuccess) return e;
  ErrTail t = tail;
  t.counters = reinterpret_cast<unsigned*>(partials + (size_t)(kTailRecords + L.grid_max) * kErrPartials);
  k_pass_a<R, kIter, false><<<L.grid_a, L.threads_a, smem_pass_a<R>(c.n1, c.rows_a), st>>>(
      c, Work<R>{}, partials, nullptr, nullptr, nullptr, nullptr, t);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_start(const LaunchCfg& L, const CellDev<R>& c, int first, cudaStream_t st) {
  const cudaError_t e = raise_smem((const void*)k_pass_a<R, kStart, false>, true);
  if (e != cudaSuccess) return e;
  if (first) k_init<R, false><<<L.grid_v, 256, 0, st>>>(c, Work<R>{});
  k_pass_a<R, kStart, false><<<L.grid_a, L.threads_a, smem_pass_a<R>(c.n1, c.rows_a), st>>>(
      c, Work<R>{}, nullptr, nullptr, nullptr, nullptr, nullptr, ErrTail{});
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_commit(const LaunchCfg& L, const CellDev<R>& c, double* partials, double* avg_out,
                          cudaStream_t st) {
  const cudaError_t e = raise_smem((const void*)k_commit<R, false>, false);
  if (e != cudaSuccess) return e;
  k_commit<R, false><<<L.grid_v, 256, kCommitSmem, st>>>(c, Work<R>{}, partials);
  k_reduce_avg<<<1, kFoldThreads, 0, st>>>(partials, L.grid_v, c.inv_nvox, avg_out, c.tmean);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ multi-cell launches
template <class R>
cudaError_t launch_multi_iteration(const MultiCfg<R>& m, cudaStream_t st) {
  cudaError_t e = raise_smem((const void*)k_pass_a<R, kIter, true>, true);
  if (e != cudaSuccess) return e;
  if (m.items_y > 0 && (e = launch_line_multi<R, kYForward>(m.wy, m.grid_y, m.smem_y, st)) != cudaSuccess) return e;
  if (m.items_z > 0 && (e = launch_line_multi<R, kZReduced>(m.wz, m.grid_z, m.smem_z, st)) != cudaSuccess) return e;
  if (m.items_y > 0 && (e = launch_line_multi<R, kYInverse>(m.wy, m.grid_y, m.smem_y, st)) != cudaSuccess) return e;
  if (m.items_a > 0)
    k_pass_a<R, kIter, true><<<m.grid_a, kThreads, m.smem_a, st>>>(CellDev<R>{}, m.wa, nullptr, nullptr,
                                                                    nullptr, nullptr, nullptr, ErrTail{});
  if (m.wa.n_act > 0) k_reduce_err_multi<R><<<m.wa.n_act * kFoldCluster, kFoldThreads, 0, st>>>(m.wa);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_multi_start(const MultiCfg<R>& m, cudaStream_t st) {
  const cudaError_t e = raise_smem((const void*)k_pass_a<R, kStart, true>, true);
  if (e != cudaSuccess) return e;
  if (m.items_v0 > 0) k_init<R, true><<<m.grid_v0, 256, 0, st>>>(CellDev<R>{}, m.wv0);
  if (m.items_s > 0)
    k_pass_a<R, kStart, true><<<m.grid_s, kThreads, m.smem_a, st>>>(CellDev<R>{}, m.ws, nullptr, nullptr,
                                                                     nullptr, nullptr, nullptr, ErrTail{});
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_multi_commit(const MultiCfg<R>& m, cudaStream_t st) {
  const cudaError_t e = raise_smem((const void*)k_commit<R, true>, false);
  if (e != cudaSuccess) return e;
  if (m.items_v > 0) k_commit<R, true><<<m.grid_v, 256, kCommitTile<R>, st>>>(CellDev<R>{}, m.wv, nullptr);
  if (m.wv.n_act > 0) k_reduce_avg_multi<R><<<m.wv.n_act, kFoldThreads, 0, st>>>(m.wv);
  return cudaGetLastError();
}

template <class R>
void multi_grids(MultiCfg<R>& m, int nsm) {
  m.grid_y = std::min(line_multi_grid<R, kYForward>(m.items_y, m.smem_y, nsm),
                      line_multi_grid<R, kYInverse>(m.items_y, m.smem_y, nsm));
  m.grid_z = line_multi_grid<R, kZReduced>(m.items_z, m.smem_z, nsm);
  m.grid_a = grid_for<R>((const void*)k_pass_a<R, kIter, true>, kThreads, m.smem_a, m.items_a, nsm);
  m.grid_s = grid_for<R>((const void*)k_pass_a<R, kStart, true>, kThreads, m.smem_a, m.items_s, nsm);
  long long g = m.items_v < 8ll * nsm ? m.items_v : 8ll * nsm;
  m.grid_v = (int)(g > 0 ? g : 1);
  g = m.items_v0 < 8ll * nsm ? m.items_v0 : 8ll * nsm;
  m.grid_v0 = (int)(g > 0 ? g : 1);
}

template <class R>
cudaError_t launch_fields(const LaunchCfg& L, const CellDev<R>& c, int from_elast, double* fe,
                          double* fg, double* ft, double* fm, double* fp, double* fq, cudaStream_t st) {
  const R* src = from_elast ? c.elast : c.prev;
  const int stride = from_elast ? 18 : 20;
  k_fields<R><<<L.grid_v, 256, 0, st>>>(c, src, stride, fe, fg, ft, fm, fp, fq);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_green_apply(const LaunchCfg& L, const CellDev<R>& c, const R* tau, const R* mu,
                               R* e_out, R* g_out, cudaStream_t st, int* ctl, int nsm) {
  cudaError_t e = raise_smem((const void*)k_pass_a<R, kXFwd, false>, true);
  if (e == cudaSuccess) e = raise_smem((const void*)k_pass_a<R, kXInv, false>, true);
  if (e != cudaSuccess) return e;
  const size_t sa = smem_pass_a<R>(c.n1, c.rows_a);
  k_pass_a<R, kXFwd, false><<<L.grid_a, L.threads_a, sa, st>>>(c, Work<R>{}, nullptr, tau, mu, nullptr, nullptr, ErrTail{});
  bool fused = false;
  if constexpr (sizeof(R) == 4) {
    if (ctl) {
      fused = true;
      if ((e = launch_spectral(c, ctl, nsm, st)) != cudaSuccess) return e;
    }
  }
  if (!fused) {
    if ((e = launch_fft_y<R>(L, c, -1, st)) != cudaSuccess) return e;
    if ((e = launch_green_z<R>(L, c, st)) != cudaSuccess) return e;
    if ((e = launch_fft_y<R>(L, c, +1, st)) != cudaSuccess) return e;
  }
  k_pass_a<R, kXInv, false><<<L.grid_a, L.threads_a, sa, st>>>(c, Work<R>{}, nullptr, nullptr, nullptr, e_out, g_out, ErrTail{});
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_radial_return(int nsm, long long count, const uint16_t* phase, int n_phases,
                                 const PhaseDev<R>* host_phases, const PhaseDev<R>* dev_phases, const R* e,
                                 const R* g, const R* e_n, const R* g_n, const R* t_n, const R* m_n,
                                 const double* p_n, const double* q_n, R* t, R* m, double* p, double* q,
                                 cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  PhaseTable<R> table{};
  if (!dev_phases) {
    if (n_phases > kTablePhases) return cudaErrorInvalidValue;
    for (int k = 0; k < n_phases; ++k) table.row[k] = host_phases[k];
  }
  PointArrays<R> P{phase, {e, g, e_n, g_n, t_n, m_n}, p_n, q_n, {t, m}, p, q};
  uintptr_t low = 0;
  for (const R* a : P.in) low |= reinterpret_cast<uintptr_t>(a);
  for (const R* a : P.out) low |= reinterpret_cast<uintptr_t>(a);
  const bool vec = low % 16 == 0;
  // a small call spreads its points over all SMs (5037 FP64 points in 20 blocks
  // of 256 took 21 us, on the FP64 pipes of 20 SMs)
  int threads = kPointThreads;
  while (threads > 32 && count < (long long)threads * 2 * nsm) threads /= 2;
  const size_t smem = 54 * (size_t)threads * sizeof(R) + (dev_phases ? 0 : n_phases * sizeof(PhaseDev<R>));
  const void* fn = vec ? (const void*)k_radial_return_points<R, true> : (const void*)k_radial_return_points<R, false>;
  const int grid = grid_for<R>(fn, threads, smem, (count + threads - 1) / threads, nsm, false);
  void* args[] = {&table, (void*)&dev_phases, &n_phases, &count, &P};
  return cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, smem, st);
}
int max_table_phases() { return kTablePhases; }

// Element-wise precision conversion of device state (cells moving between
// the FP32 and FP64 engines).
template <class S, class D>
__global__ void k_convert(const S* __restrict__ src, D* __restrict__ dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = (D)src[i];
}

template <class S, class D>
cudaError_t launch_convert(const S* src, D* dst, long long n, int nsm, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  long long blocks = (n + 255) / 256;
  if (blocks > 8ll * nsm) blocks = 8ll * nsm;
  k_convert<S, D><<<(int)blocks, 256, 0, st>>>(src, dst, n);
  return cudaGetLastError();
}
template cudaError_t launch_convert<float, double>(const float*, double*, long long, int, cudaStream_t);
template cudaError_t launch_convert<double, float>(const double*, float*, long long, int, cudaStream_t);

template <class R>
LaunchCfg make_launch_cfg(const CellDev<R>& c, int nsm, int rows_wanted, bool shared) {
  LaunchCfg L;
  // rows per pass-A item: about 256 voxels per block (FP64: 128, see below) or
  // as asked, within the shared-memory budget; a cell alone takes fewer rows
  // rather than leave SMs without an item, down to a warp of voxels
  const long long nrows = (long long)c.n2 * c.n3;
  int rows = rows_wanted;
  if (rows <= 0) {
    const int want = sizeof(R) == 8 && !shared ? 128 : 256;
    rows = c.n1 >= want ? 1 : want / c.n1;
    if (!shared) {
      const int least = (32 + c.n1 - 1) / c.n1;
      rows = std::max(std::min(rows, least), (int)std::min<long long>(rows, (nrows + nsm - 1) / nsm));
    }
  }
  while (rows > 1 && smem_pass_a<R>(c.n1, rows) > kSmemBudget) rows /= 2;
  if ((long long)rows > nrows) rows = (int)nrows;
  L.rows = rows;
  const long long items = (nrows + rows - 1) / rows;
  L.items_a = items;
  // Threads: an item of up to 128 voxels keeps 128 busy.  In FP64 (up to 255
  // registers a thread) that lets two blocks share an SM, so that one's
  // material update fills the FP64 pipe while the other loads or waits at a
  // barrier; an item too large for that keeps the SM's 256.
  const size_t smem_a = smem_pass_a<R>(c.n1, rows);
  L.threads_a = !shared && (long long)rows * c.n1 <= 128 && (sizeof(R) == 4 || 2 * smem_a <= kSmemOptin) ? 128 : kThreads;
  L.grid_a = std::min(grid_for<R>((const void*)k_pass_a<R, kIter, false>, L.threads_a, smem_a, items, nsm),
                      kPassABlocks * nsm);
  L.grid_max = kPassABlocks * nsm;
  CellDev<R> t = c;
  t.cols_y = L.cols_y = tile_columns(c.n2, (long long)c.n3 * c.kx, sizeof(R) == 8, shared, nsm);
  t.cols_z = L.cols_z = tile_columns(c.n3, (long long)c.n2 * c.kx, sizeof(R) == 8, shared, nsm);
  if (!shared) {
    if (c.n2 > 1) L.grid_y = std::min(line_grid<R, kYForward>(t, nsm), line_grid<R, kYInverse>(t, nsm));
    L.grid_z = c.n2 == 1 ? line_grid<R, kZFull>(t, nsm) : line_grid<R, kZReduced>(t, nsm);
  }
  long long vb = (c.nvox + 255) / 256;
  L.grid_v = (int)(vb < 4ll * nsm ? vb : 4ll * nsm);
  return L;
}

template <class R>
bool sizes_fit(int n1, int n2, int n3) {
  // a y / z tile holds at least one whole column of 18 lines (the longest in
  // FP64, 384, takes the whole budget)
  return smem_pass_a<R>(n1, 1) <= kSmemBudget && smem_line<R>(n2, 1, 18) <= kSmemBudget &&
         smem_line<R>(n3, 1, 18) <= kSmemBudget;
}

#define MP_INSTANTIATE(R)                                                                            \
  template cudaError_t launch_fft_y<R>(const LaunchCfg&, const CellDev<R>&, int, cudaStream_t);       \
  template cudaError_t launch_green_z<R>(const LaunchCfg&, const CellDev<R>&, cudaStream_t);          \
  template cudaError_t launch_pass_a_iter<R>(const LaunchCfg&, const CellDev<R>&, double*, const ErrTail&, cudaStream_t); \
  template cudaError_t launch_start<R>(const LaunchCfg&, const CellDev<R>&, int, cudaStream_t);       \
  template cudaError_t launch_commit<R>(const LaunchCfg&, const CellDev<R>&, double*, double*,        \
                                        cudaStream_t);                                               \
  template cudaError_t launch_multi_iteration<R>(const MultiCfg<R>&, cudaStream_t);                   \
  template cudaError_t launch_multi_start<R>(const MultiCfg<R>&, cudaStream_t);                       \
  template cudaError_t launch_multi_commit<R>(const MultiCfg<R>&, cudaStream_t);                      \
  template void multi_grids<R>(MultiCfg<R>&, int);                                                   \
  template size_t smem_pass_a<R>(int, int);                                                          \
  template cudaError_t launch_fields<R>(const LaunchCfg&, const CellDev<R>&, int, double*, double*,   \
                                        double*, double*, double*, double*, cudaStream_t);           \
  template cudaError_t launch_green_apply<R>(const LaunchCfg&, const CellDev<R>&, const R*, const R*,  \
                                             R*, R*, cudaStream_t, int*, int);                       \
  template cudaError_t launch_radial_return<R>(int, long long, const uint16_t*, int, const PhaseDev<R>*, \
                                               const PhaseDev<R>*, const R*, const R*, const R*,      \
                                               const R*, const R*, const R*, const double*,           \
                                               const double*, R*, R*, double*, double*, cudaStream_t); \
  template LaunchCfg make_launch_cfg<R>(const CellDev<R>&, int, int, bool);                                  \
  template bool sizes_fit<R>(int, int, int);

MP_INSTANTIATE(float)
MP_INSTANTIATE(double)

MP_INSTANTIATE_LINE(float, kZFull)
MP_INSTANTIATE_LINE(double, kZFull)

}  // namespace mp
