// Shared-memory Stockham FFT building blocks (sm_103a).  Transforms are
// unnormalised; the solver folds the 1 / (N1 N2 N3) of the inverse into the
// Green operator.
#pragma once

#include "mp_common.cuh"

namespace mp {

// DIR = -1: forward kernel exp(-2 pi i k n / M); DIR = +1: inverse.
template <class R, int DIR>
__device__ __forceinline__ cpx<R> twiddle(const cpx<R>* tw, int idx) {
  cpx<R> w = tw[idx];
  if (DIR > 0) w.y = -w.y;
  return w;
}

// multiply by DIR * i  (the quarter-turn W_4 = exp(DIR i pi / 2))
template <class R, int DIR>
__device__ __forceinline__ cpx<R> rot90(cpx<R> a) {
  return DIR < 0 ? cmake<R>(a.y, -a.x) : cmake<R>(-a.y, a.x);
}

template <class R, int DIR>
__device__ __forceinline__ void dft2(cpx<R>* v) {
  cpx<R> a = v[0], b = v[1];
  v[0] = cadd(a, b);
  v[1] = csub(a, b);
}

template <class R, int DIR>
__device__ __forceinline__ void dft3(cpx<R>* v) {
  // W_3 = -1/2 + DIR i sqrt(3)/2
  const R half = R(0.5);
  const R s3 = R(0.86602540378443864676372317075294);
  cpx<R> a = v[0], t = cadd(v[1], v[2]), u = csub(v[1], v[2]);
  cpx<R> base = cmake<R>(a.x - half * t.x, a.y - half * t.y);
  const cpx<R> r = rot90<R, DIR>(u);
  v[0] = cadd(a, t);
  v[1] = cfma(r, s3, base);
  v[2] = cfma(r, -s3, base);
}

template <class R, int DIR>
__device__ __forceinline__ void dft4(cpx<R>* v) {
  cpx<R> t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
  cpx<R> t2 = cadd(v[1], v[3]), t3 = csub(v[1], v[3]);
  v[0] = cadd(t0, t2);
  v[2] = csub(t0, t2);
  // t1 +- DIR i t3, component by component: no packing of the turned value
  if constexpr (DIR < 0) {
    v[1] = cmake<R>(t1.x + t3.y, t1.y - t3.x);
    v[3] = cmake<R>(t1.x - t3.y, t1.y + t3.x);
  } else {
    v[1] = cmake<R>(t1.x - t3.y, t1.y + t3.x);
    v[3] = cmake<R>(t1.x + t3.y, t1.y - t3.x);
  }
}

template <class R, int DIR>
__device__ __forceinline__ void dft8(cpx<R>* v) {
  // split into even / odd 4-point DFTs, combine with W_8^k = exp(DIR 2 pi i k / 8)
  cpx<R> e[4] = {v[0], v[2], v[4], v[6]};
  cpx<R> o[4] = {v[1], v[3], v[5], v[7]};
  dft4<R, DIR>(e);
  dft4<R, DIR>(o);
  const R h = R(0.70710678118654752440084436210485);
  // W_8^1 = h (1 + DIR i), W_8^2 = DIR i, W_8^3 = h (-1 + DIR i)
  cpx<R> o1 = cmake<R>(o[1].x - DIR * o[1].y, o[1].y + DIR * o[1].x);
  cpx<R> o2 = rot90<R, DIR>(o[2]);
  cpx<R> o3 = cmake<R>(-o[3].x - DIR * o[3].y, -o[3].y + DIR * o[3].x);
  v[0] = cadd(e[0], o[0]);
  v[4] = csub(e[0], o[0]);
  v[1] = cfma(o1, h, e[1]);
  v[5] = cfma(o1, -h, e[1]);
  v[2] = cadd(e[2], o2);
  v[6] = csub(e[2], o2);
  v[3] = cfma(o3, h, e[3]);
  v[7] = cfma(o3, -h, e[3]);
}

// 16-point DFT as 4 x 4: 4-point DFTs over n1 of x[4 n1 + n2], twiddles
// W_16^(n2 k1), 4-point DFTs over n2; output index k1 + 4 k2.
template <class R, int DIR>
__device__ __forceinline__ void dft16(cpx<R>* v) {
  cpx<R> a[4][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    cpx<R> t[4] = {v[n2], v[4 + n2], v[8 + n2], v[12 + n2]};
    dft4<R, DIR>(t);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) a[n2][k1] = t[k1];
  }
  // W_16^m = cos(2 pi m / 16) + DIR i sin(2 pi m / 16), m = n2 k1 in {1, 2, 3, 4, 6, 9}
  const R c1 = R(0.92387953251128675612818318939679);  // cos(pi/8)
  const R s1 = R(0.38268343236508977172845998403040);  // sin(pi/8)
  const R h = R(0.70710678118654752440084436210485);
  auto rot = [&](cpx<R> x, R cr, R si) {  // x * (cr + DIR i si)
    return cmake<R>(x.x * cr - DIR * x.y * si, x.y * cr + DIR * x.x * si);
  };
  a[1][1] = rot(a[1][1], c1, s1);
  a[1][2] = rot(a[1][2], h, h);
  a[1][3] = rot(a[1][3], s1, c1);
  a[2][1] = rot(a[2][1], h, h);
  a[2][2] = rot90<R, DIR>(a[2][2]);
  a[2][3] = rot(a[2][3], -h, h);
  a[3][1] = rot(a[3][1], s1, c1);
  a[3][2] = rot(a[3][2], -h, h);
  a[3][3] = rot(a[3][3], -c1, -s1);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    cpx<R> t[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
    dft4<R, DIR>(t);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = t[k2];
  }
}

// 9-point DFT as 3 x 3: 3-point DFTs over x[3 n1 + n2], twiddles W_9^(n2 k1),
// 3-point DFTs over n2; output index k1 + 3 k2.
template <class R, int DIR>
__device__ __forceinline__ void dft9(cpx<R>* v) {
  cpx<R> a[3][3];
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    cpx<R> t[3] = {v[n2], v[3 + n2], v[6 + n2]};
    dft3<R, DIR>(t);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) a[n2][k1] = t[k1];
  }
  auto rot = [&](cpx<R> x, R cr, R si) {  // x * (cr + DIR i si)
    return cmake<R>(x.x * cr - DIR * x.y * si, x.y * cr + DIR * x.x * si);
  };
  const R c1 = R(0.76604444311897803520239265055542), s1 = R(0.64278760968653932632264340990726);   // 2 pi / 9
  const R c2 = R(0.17364817766693034885171662676931), s2 = R(0.98480775301220805936674302458952);   // 4 pi / 9
  const R c4 = R(-0.93969262078590838405410927732473), s4 = R(0.34202014332566873304409961468226);  // 8 pi / 9
  a[1][1] = rot(a[1][1], c1, s1);
  a[1][2] = rot(a[1][2], c2, s2);
  a[2][1] = rot(a[2][1], c2, s2);
  a[2][2] = rot(a[2][2], c4, s4);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    cpx<R> t[3] = {a[0][k1], a[1][k1], a[2][k1]};
    dft3<R, DIR>(t);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = t[k2];
  }
}

template <class R, int DIR, int RADIX>
__device__ __forceinline__ void dft(cpx<R>* v);

// DFT of coprime factors A x B (the prime-factor map: no twiddles).  Input
// n = (B n1 + A n2) mod A B, output k = (k1 B (B^-1 mod A) + k2 A (A^-1 mod B))
// mod A B.
template <class R, int DIR, int A, int B>
__device__ __forceinline__ void dft_coprime(cpx<R>* v) {
  constexpr auto inv = [](int x, int m) {
    int r = 0;
    while ((x * r) % m != 1 % m) ++r;
    return r;
  };
  constexpr int N = A * B, CB = B * inv(B % A, A), CA = A * inv(A % B, B);
  cpx<R> a[B][A];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) {
    cpx<R> t[A];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) t[n1] = v[(B * n1 + A * n2) % N];
    dft<R, DIR, A>(t);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) a[n2][k1] = t[k1];
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    cpx<R> t[B];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) t[n2] = a[n2][k1];
    dft<R, DIR, B>(t);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[(k1 * CB + k2 * CA) % N] = t[k2];
  }
}

template <class R, int DIR, int RADIX>
__device__ __forceinline__ void dft(cpx<R>* v) {
  if constexpr (RADIX == 1) return;
  else if constexpr (RADIX == 2) dft2<R, DIR>(v);
  else if constexpr (RADIX == 3) dft3<R, DIR>(v);
  else if constexpr (RADIX == 4) dft4<R, DIR>(v);
  else if constexpr (RADIX == 6) dft_coprime<R, DIR, 2, 3>(v);
  else if constexpr (RADIX == 8) dft8<R, DIR>(v);
  else if constexpr (RADIX == 9) dft9<R, DIR>(v);
  else if constexpr (RADIX == 12) dft_coprime<R, DIR, 4, 3>(v);
  else if constexpr (RADIX == 16) dft16<R, DIR>(v);
  else {
    static_assert(RADIX == 18, "no DFT of this radix");
    dft_coprime<R, DIR, 2, 9>(v);
  }
}

// Stages of a y / z line of length n: two for every length up to 324, so that
// the line crosses shared memory once between them; lengths a thread holds
// whole take one.
struct LinePlan {
  int count, r0, r1, r2;
};
__host__ __device__ constexpr LinePlan line_plan(int n) {
  switch (n) {
    case 1: case 2: case 4: case 6: case 8: case 12: case 16: case 18: return {1, n, 1, 1};
    case 24: return {2, 6, 4, 1};
    case 32: return {2, 8, 4, 1};
    case 36: return {2, 6, 6, 1};
    case 48: return {2, 8, 6, 1};
    case 54: return {2, 9, 6, 1};
    case 64: return {2, 8, 8, 1};
    case 72: return {2, 9, 8, 1};
    case 96: return {2, 12, 8, 1};
    case 108: return {2, 12, 9, 1};
    case 128: return {2, 16, 8, 1};
    case 144: return {2, 12, 12, 1};
    case 162: return {2, 18, 9, 1};
    case 192: return {2, 16, 12, 1};
    case 216: return {2, 18, 12, 1};
    case 256: return {2, 16, 16, 1};
    case 288: return {2, 18, 16, 1};
    case 324: return {2, 18, 18, 1};
    case 384: return {3, 8, 8, 6};
    case 432: return {3, 9, 8, 6};
    case 486: return {3, 9, 9, 6};
    case 512: return {3, 8, 8, 8};
    default: return {0, 1, 1, 1};
  }
}
// Gap (complex values) after every r0 points of a two-stage column between its
// stages: r0 lines and the gap advance the shared-memory banks as one line
// does (a multiple of 16 complex values is a multiple of all banks, in FP32
// and FP64), so a warp writes neighbouring butterflies like neighbouring points.
__host__ __device__ constexpr int line_gap(int n, int lines) {
  return line_plan(n).count == 2 ? (lines * 32 - lines * (line_plan(n).r0 - 1)) % 16 : 0;
}
// Complex values of such a column; an even number, so that tiles stay aligned.
__host__ __device__ constexpr int line_pitch(int n, int lines) {
  return (n * lines + n / line_plan(n).r0 * line_gap(n, lines) + 1) / 2 * 2;
}
// Complex entries of the table region of a line tile: n twiddles and n
// frequencies, in whole 16-byte pieces.
__host__ __device__ constexpr int line_table(int n) { return (n + (n + 1) / 2 + 1) / 2 * 2; }

// Tiles are stored component-interleaved ("AoS"): element (row rr, point n,
// component c) of a tile with `rows` rows of M points lives at
// base[(rr M + n) 18 + c], exactly as the spectral buffer stores a row.  A
// transform line is (rr, c), with stride 18 between its points.  Threads take
// (c, j, rr) with c fastest, so a warp reads and writes consecutive complex
// values: the stages are free of shared-memory bank conflicts and need no
// transposition on load or store.
//
// One Stockham stage of radix R (2, 3, 4 or 8) with Ns = product of the radices already
// applied: butterfly j of a line reads points j + r M / R (r < R), multiplies
// point r by W_M^(r (j mod Ns) M / (Ns R)), takes the R-point DFT and writes
// output r to point (j / Ns) Ns R + (j mod Ns) + r Ns.  The last stage leaves
// natural order (no bit reversal).  The host orders radix-3 stages last, so
// only those divide by a non-power-of-two Ns.
// The packed x axis' table holds the 2 M roots: W_M^k = tw[2 k].
template <class R, int DIR>
__device__ void stage_aos(const cpx<R>* __restrict__ in, cpx<R>* __restrict__ out, int rows, int M,
                          int radix, int Ns, const cpx<R>* __restrict__ tw) {
  constexpr int MAXR = 8;
  const int nb = M / radix;
  const int total = rows * nb * 18;
  const int tstep = M / (Ns * radix);
  const bool ns_pow2 = (Ns & (Ns - 1)) == 0;
  const int ns_sh = __ffs(Ns) - 1;
  const bool nb_pow2 = (nb & (nb - 1)) == 0;
  const int nb_sh = __ffs(nb) - 1;
  const int rs = M * 18;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int c = idx % 18;
    const int q = idx / 18;
    int rr = 0, j = q;
    if (rows > 1) {
      rr = nb_pow2 ? (q >> nb_sh) : (q / nb);
      j = q - rr * nb;
    }
    const int kk = ns_pow2 ? (j & (Ns - 1)) : (j % Ns);
    const int jq = ns_pow2 ? (j >> ns_sh) : (j / Ns);
    const cpx<R>* src = in + rr * rs + c;
    cpx<R> v[MAXR];
    v[0] = src[j * 18];
#pragma unroll
    for (int r = 1; r < MAXR; ++r) {
      if (r < radix) {
        cpx<R> x = src[(j + r * nb) * 18];
        const int e = r * kk * tstep;  // < M
        v[r] = e == 0 ? x : cmul(x, twiddle<R, DIR>(tw, e * 2));
      }
    }
    switch (radix) {
      case 2: dft2<R, DIR>(v); break;
      case 3: dft3<R, DIR>(v); break;
      case 4: dft4<R, DIR>(v); break;
      default: dft8<R, DIR>(v); break;
    }
    cpx<R>* dst = out + rr * rs + c + (jq * Ns * radix + kk) * 18;
#pragma unroll
    for (int r = 0; r < MAXR; ++r) {
      if (r < radix) dst[r * Ns * 18] = v[r];
    }
  }
}

// The same stage with the radix, Ns and the line length M known at compile time
// (index arithmetic folds to shifts and constants, and only the one butterfly
// is instantiated).
template <class R, int DIR, int RADIX, int NS, int M>
__device__ __forceinline__ void stage_fixed(const cpx<R>* __restrict__ in, cpx<R>* __restrict__ out, int rows,
                                            const cpx<R>* __restrict__ tw) {
  constexpr int nb = M / RADIX;
  constexpr int tstep = M / (NS * RADIX);
  constexpr int rs = M * 18;
  const int total = rows * nb * 18;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int c = idx % 18;
    const int q = idx / 18;
    const int rr = q / nb, j = q % nb;
    const int kk = j % NS, jq = j / NS;
    const cpx<R>* src = in + rr * rs + c;
    cpx<R> v[RADIX];
    v[0] = src[j * 18];
#pragma unroll
    for (int r = 1; r < RADIX; ++r) {
      const cpx<R> x = src[(j + r * nb) * 18];
      v[r] = (NS == 1) ? x : cmul(x, twiddle<R, DIR>(tw, r * kk * tstep * 2));
    }
    dft<R, DIR, RADIX>(v);
    cpx<R>* dst = out + rr * rs + c + (jq * NS * RADIX + kk) * 18;
#pragma unroll
    for (int r = 0; r < RADIX; ++r) dst[r * NS * 18] = v[r];
  }
}

// Transform every line of an AoS tile by the run-time radix plan; data starts in
// b0, the result pointer (b0 or b1) is returned.  Ends with a barrier.
template <class R, int DIR>
__device__ cpx<R>* tile_fft(cpx<R>* b0, cpx<R>* b1, int rows, const RadixPlan& p, const cpx<R>* tw) {
  cpx<R>* in = b0;
  cpx<R>* out = b1;
  int Ns = 1;
  for (int s = 0; s < p.nstages; ++s) {
    stage_aos<R, DIR>(in, out, rows, p.m, p.radix[s], Ns, tw);
    Ns *= p.radix[s];
    __syncthreads();
    cpx<R>* t = in;
    in = out;
    out = t;
  }
  return in;
}

// Plan of a packed x transform of length m without compile-time stages of its
// own: one stage (a thread holds the line) or two.  count 0: the run-time
// radix plan.
struct XPlan {
  int count, r0, r1;
};
__host__ __device__ constexpr XPlan x_plan(int m) {
  switch (m) {
    case 2: case 3: case 4: case 6: case 9: return {1, m, 1};
    case 18: return {2, 6, 3};
    case 27: return {2, 9, 3};
    case 36: return {2, 6, 6};
    case 48: return {2, 8, 6};
    case 54: return {2, 9, 6};
    case 72: return {2, 9, 8};
    case 81: return {2, 9, 9};
    case 96: return {2, 12, 8};
    case 108: return {2, 12, 9};
    default: return {0, 1, 1};
  }
}

// The forward x transform inside pass A of the lengths whose post-step is a
// pass of its own: common lengths unrolled at compile time (radix <= 8, radix 3
// last; 128, 64 and 32 in FP64 only - FP32 fuses their last stage with the
// post-step), others by the run-time radix plan.
// (256 is met in FP32 only, but the registers of a 128^3 cell's pass A come out
// worse with the case outside the switch: 257 -> 265 us.)
template <class R>
__device__ cpx<R>* tile_fft_x_fwd(cpx<R>* b0, cpx<R>* b1, int rows, const RadixPlan& p, const cpx<R>* tw) {
  auto sync_swap = [&]() {
    __syncthreads();
    cpx<R>* t = b0;
    b0 = b1;
    b1 = t;
  };
  if constexpr (sizeof(R) == 8) {
    switch (p.m) {
      case 128:
        stage_fixed<R, -1, 8, 1, 128>(b0, b1, rows, tw); sync_swap();
        stage_fixed<R, -1, 4, 8, 128>(b0, b1, rows, tw); sync_swap();
        stage_fixed<R, -1, 4, 32, 128>(b0, b1, rows, tw); sync_swap();
        return b0;
      case 64:
        stage_fixed<R, -1, 8, 1, 64>(b0, b1, rows, tw); sync_swap();
        stage_fixed<R, -1, 8, 8, 64>(b0, b1, rows, tw); sync_swap();
        return b0;
      case 32:
        stage_fixed<R, -1, 8, 1, 32>(b0, b1, rows, tw); sync_swap();
        stage_fixed<R, -1, 4, 8, 32>(b0, b1, rows, tw); sync_swap();
        return b0;
      default: break;
    }
  }
  switch (p.m) {
    case 256:
      stage_fixed<R, -1, 8, 1, 256>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, -1, 8, 8, 256>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, -1, 4, 64, 256>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 24:
      stage_fixed<R, -1, 8, 1, 24>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, -1, 3, 8, 24>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 16:
      stage_fixed<R, -1, 4, 1, 16>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, -1, 4, 4, 16>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 12:
      stage_fixed<R, -1, 4, 1, 12>(b0, b1, rows, tw); sync_swap();
      stage_fixed<R, -1, 3, 4, 12>(b0, b1, rows, tw); sync_swap();
      return b0;
    case 8:
      stage_fixed<R, -1, 8, 1, 8>(b0, b1, rows, tw); sync_swap();
      return b0;
    default: return tile_fft<R, -1>(b0, b1, rows, p, tw);
  }
}

}  // namespace mp
