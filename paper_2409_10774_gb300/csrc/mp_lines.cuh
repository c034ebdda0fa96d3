// The y and z passes of one fixed-point iteration: transforms along the two
// outer axes and the Green operator between them (sm_103a).
//
// Fewer fields along z.  The Green operator needs the 18 components of
// (tau^, mu^) only through
//   f_l = i xi_k tau^_kl,   g_l = i xi_k mu^_kl + (eps : tau^)_l,
// and x1, x2 are known once the y transform is done.  So the y pass leaves,
// per point (kx, ky, z) and l = 0..2, the four values
//   A_l = i (x1 tau_1l + x2 tau_2l),                 T_l = tau_3l,
//   B_l = i (x1 mu_1l + x2 mu_2l) + (eps : tau)_l,   M_l = mu_3l,
// and the z pass, after its forward transform, forms f_l = A_l + i x3 T_l and
// g_l = B_l + i x3 M_l.  It hands back u_l, e_3l, phi_l, gamma_l3, from
// which the inverse y pass forms the 18 components of (e~, gamma~) while it
// reads them.  The z pass so transforms, reads and writes 12 values per point
// instead of 18, and the passes move 84 complex values per point instead of
// 108.  A_l, B_l are rounded before the z transform and i x1 u_l, i x2 u_l
// meet phi_m only after it; fused multiply-adds here, in the operator and in
// the packed x steps make up for that: on random FP32 fields the strain of a
// 64^3 cell is 2.49e-7 off its 64-bit value (2.61e-7 without them, 2.50e-7
// with all 18 fields through z).  The 12 values sit in the first slots of the point's 18, l-major (the four
// values of one l are 16-byte pieces).  Cells with N2 = 1 have no y
// pass; their z pass takes all 18.
//
// Every supported length has a compile-time plan of one to three Stockham
// stages (radices up to 18, the coprime ones without twiddles).  Tiles are whole
// columns, (col N + p) LN + c, loaded into shared memory in 16-byte asynchronous
// copies; the last stage of the y inverse and z passes stores to global memory
// from registers.
#pragma once

#include "mp_device.cuh"
#include "mp_fft.cuh"
#include "mp_green.cuh"
#include "mp_kernels.cuh"
#include "mp_tma.cuh"

namespace mp {

// Threads and blocks per SM of the line passes.  FP32: a tile of 256 points
// has 288 radix-16 butterflies of 18 lines (192 of 12), three (four) blocks of
// 72 (80) registers.  FP64: tiles of 128 points, so that three blocks share
// an SM and its FP64 pipe stays busy while one of them loads or waits.
template <class R>
struct LineCfg;
template <>
struct LineCfg<float> {
  static constexpr int y_threads = 288, y_blocks = 3, z_threads = 192, z_blocks = 4;
};
template <>
struct LineCfg<double> {
  static constexpr int y_threads = 160, y_blocks = 3, z_threads = 128, z_blocks = 4;
};

// ------------------------------------------------------------------ transforms
// The DFT of length N over the lines of `cols` columns, LN lines each.  The
// first stage takes its points from load, the last gives them to store:
// load(c, j, col) returns a reader whose (r) is point j + r N / RADIX, and
// store(c, p, col) a writer whose (r, value) is point p + r NS, so that each
// butterfly forms its addresses once and steps by a constant.  `a` holds the
// tile between the stages (`b` too in three-stage plans).
template <class R, int DIR, int RADIX, int NS, int N, int LN, class Load, class Store>
__device__ __forceinline__ void line_stage(int cols, const cpx<R>* tw, Load load, Store store) {
  constexpr int nb = N / RADIX, tstep = N / (NS * RADIX);
  const int total = cols * nb * LN;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int c = idx % LN, q = idx / LN;
    const int col = q / nb, j = q % nb;
    const int kk = j % NS;
    cpx<R> v[RADIX];
    const auto in = load(c, j, col);
#pragma unroll
    for (int r = 0; r < RADIX; ++r) v[r] = in(r);
    if constexpr (NS > 1) {
#pragma unroll
      for (int r = 1; r < RADIX; ++r) v[r] = cmul(v[r], twiddle<R, DIR>(tw, r * kk * tstep));
    }
    dft<R, DIR, RADIX>(v);
    const auto out = store(c, (j / NS) * NS * RADIX + kk, col);
#pragma unroll
    for (int r = 0; r < RADIX; ++r) out(r, v[r]);
  }
}

// Readers and writers of points `step` complex values apart (global memory:
// step_bytes, one wide multiply-add per point).  Tiles are loaded in 16-byte
// asynchronous copies: first stages that took their points straight from
// global memory (8 bytes a lane, 144-byte runs) kept the load queue full and
// the y pass of a 128^3 cell took 87 us instead of 61.
template <class R>
struct TileReader {
  const cpx<R>* p;
  int step;
  __device__ __forceinline__ cpx<R> operator()(int r) const { return p[r * step]; }
};
template <class R>
struct TileWriter {
  cpx<R>* p;
  int step;
  __device__ __forceinline__ void operator()(int r, cpx<R> v) const { p[r * step] = v; }
};
template <class R>
struct GlobalWriter {
  cpx<R>* p;
  unsigned step_bytes;
  __device__ __forceinline__ void operator()(int r, cpx<R> v) const {
    void* q = reinterpret_cast<char*>(p) + (unsigned long long)step_bytes * (unsigned)r;
    if constexpr (sizeof(R) == 4) *reinterpret_cast<float2*>(q) = make_float2(v.x, v.y);
    else *reinterpret_cast<double2*>(q) = make_double2(v.x, v.y);
  }
};

// Between two stages a gap follows every r0 points (line_gap): the first stage
// writes runs of r0 points a butterfly, and without the gap the butterflies of
// a warp would meet in the same banks.
template <class R, int DIR, int N, int LN, class Load, class Store>
__device__ __forceinline__ void line_dft(int cols, const cpx<R>* tw, cpx<R>* a, cpx<R>* b, Load load, Store store) {
  constexpr LinePlan P = line_plan(N);
  static_assert(P.count > 0 && P.r0 * P.r1 * P.r2 == N, "the plan's radices multiply to the length");
  if constexpr (P.count == 1) {
    line_stage<R, DIR, P.r0, 1, N, LN>(cols, tw, load, store);
  } else if constexpr (P.count == 2) {
    constexpr int G = line_gap(N, LN), NP = line_pitch(N, LN);
    line_stage<R, DIR, P.r0, 1, N, LN>(cols, tw, load, [=](int c, int p, int col) {
      return TileWriter<R>{a + col * NP + p * LN + p / P.r0 * G + c, LN};
    });
    __syncthreads();
    line_stage<R, DIR, P.r1, P.r0, N, LN>(
        cols, tw, [=](int c, int j, int col) { return TileReader<R>{a + col * NP + j * LN + c, P.r0 * LN + G}; },
        store);
  } else {
    line_stage<R, DIR, P.r0, 1, N, LN>(
        cols, tw, load, [=](int c, int p, int col) { return TileWriter<R>{a + (col * N + p) * LN + c, LN}; });
    __syncthreads();
    line_stage<R, DIR, P.r1, P.r0, N, LN>(
        cols, tw, [=](int c, int j, int col) { return TileReader<R>{a + (col * N + j) * LN + c, N / P.r1 * LN}; },
        [=](int c, int p, int col) { return TileWriter<R>{b + (col * N + p) * LN + c, P.r0 * LN}; });
    __syncthreads();
    line_stage<R, DIR, P.r2, P.r0 * P.r1, N, LN>(
        cols, tw, [=](int c, int j, int col) { return TileReader<R>{b + (col * N + j) * LN + c, N / P.r2 * LN}; },
        store);
  }
}
// Points between the outputs of a last-stage butterfly.
template <int N>
__host__ __device__ constexpr int last_step() {
  return N / (line_plan(N).count == 1 ? line_plan(N).r0 : line_plan(N).count == 2 ? line_plan(N).r1 : line_plan(N).r2);
}
template <int N>
__host__ __device__ constexpr int first_step() { return N / line_plan(N).r0; }
// The tile a transform that ends in shared memory leaves its result in, of
// the tiles a and b it was given (neither is read by its last stage).
template <int N>
__host__ __device__ constexpr bool ends_in_b() { return line_plan(N).count == 2; }

// 16-byte pieces: two (FP32) or one (FP64) complex values.
template <class R>
__device__ __forceinline__ void store4(cpx<R>* dst, const cpx<R>* v) {
  if constexpr (sizeof(R) == 4) {
    reinterpret_cast<float4*>(dst)[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    reinterpret_cast<float4*>(dst)[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) reinterpret_cast<double2*>(dst)[i] = make_double2(v[i].x, v[i].y);
  }
}

// ------------------------------------------------------------------ y pass
// Column col of a y tile is (kz, kx), index kz KX + kx; its point ky is point
// (kz N + ky) KX + kx of the spectrum.
template <class R, int N>
__device__ __forceinline__ long long y_column(const CellDev<R>& c, int col, int& kx) {
  const int kz = div_kx(c, col);
  kx = col - kz * c.kx;
  return (long long)(kz * N) * c.kx + kx;
}

// Spreads a tile's points (n rows of `units` items) over the block: body(u, p0,
// dp) handles item u of rows p0, p0 + dp, ..., so that addresses advance by a
// constant.
template <class Body>
__device__ __forceinline__ void for_rows(int units, Body body) {
  const int bd = (int)blockDim.x, t = (int)threadIdx.x;
  if (units <= bd) {
    const int rows = (int)((unsigned)bd / (unsigned)units), r = (int)((unsigned)t / (unsigned)units);
    if (r < rows) body(t - r * units, r, rows);
  } else {
    for (int u = t; u < units; u += bd) body(u, 0, 1);
  }
}

// The first LN values of every point of a tile of `cols` columns into t, in
// 16-byte pieces; `first(col)` is a column's first point, `step` the points
// between its points (neighbouring columns are neighbouring points).  Ends
// with a barrier.
template <class R, int N, int LN, class First>
__device__ __forceinline__ void load_tile(const cpx<R>* spec, int cols, long long step, cpx<R>* t, First first) {
  constexpr int W = LN * (int)sizeof(cpx<R>) / 16;
  for_rows(cols * W, [=](int u, int p0, int dp) {
    const int col = u / W, w = u - col * W;
    const cpx<R>* src = spec + (first(col) + p0 * step) * 18 + w * (16 / (int)sizeof(cpx<R>));
    cpx<R>* dst = t + (col * N + p0) * LN + w * (16 / (int)sizeof(cpx<R>));
    const long long ds = step * dp * 18;
    for (int p = p0; p < N; p += dp) {
      cp_async16(dst, src);
      src += ds;
      dst += dp * LN;
    }
  });
  cp_async_wait_all();
  __syncthreads();
}

// y forward, then the 12 values of each point (see the top of the file).
template <class R, int N>
__device__ __forceinline__ void y_forward_tile(const CellDev<R>& c, long long tile, cpx<R>* a, cpx<R>* b,
                                               const cpx<R>* tw, const R* xi) {
  const int ncols = c.n3 * c.kx, col0 = (int)tile * c.cols_y;
  const int cols = ncols - col0 < c.cols_y ? ncols - col0 : c.cols_y;
  cpx<R>* x = ends_in_b<N>() ? b : a;
  load_tile<R, N, 18>(c.spec, cols, c.kx, b, [&](int col) {
    int kx;
    return y_column<R, N>(c, col0 + col, kx);
  });
  line_dft<R, -1, N, 18>(
      cols, tw, a, b,
      [=](int ln, int j, int col) { return TileReader<R>{b + (col * N + j) * 18 + ln, first_step<N>() * 18}; },
      [=](int ln, int p, int col) { return TileWriter<R>{x + (col * N + p) * 18 + ln, last_step<N>() * 18}; });
  __syncthreads();
  for_rows(cols * 3, [=, &c](int u, int p0, int dp) {
    const int col = u / 3, l = u - 3 * col;
    int kx;
    const long long i0 = y_column<R, N>(c, col0 + col, kx);
    const R x1 = c.n1 == 1 ? R(0) : c.two_pi_over_L[0] * (R)kx;
    // (eps : tau)_l = tau_mn - tau_nm with (l, m, n) cyclic
    const int m = l == 2 ? 0 : l + 1, n = l == 0 ? 2 : l - 1;
    const cpx<R>* v = x + (col * N + p0) * 18;
    cpx<R>* dst = c.spec + (i0 + (long long)p0 * c.kx) * 18 + 4 * l;
    const long long ds = (long long)c.kx * dp * 18;
    for (int p = p0; p < N; p += dp) {
      const R x2 = xi[p];
      const cpx<R> ta = v[l], tb = v[3 + l], ma = v[9 + l], mb = v[12 + l];
      const cpx<R> rot = csub(v[3 * m + n], v[3 * n + m]);
      cpx<R> o[4];
      o[0] = cmake<R>(-(ta.y * x1 + tb.y * x2), ta.x * x1 + tb.x * x2);
      o[1] = v[6 + l];
      o[2] = cmake<R>(fma(-mb.y, x2, fma(-ma.y, x1, rot.x)), fma(mb.x, x2, fma(ma.x, x1, rot.y)));
      o[3] = v[15 + l];
      store4(dst, o);
      v += dp * 18;
      dst += ds;
    }
  });
  // the next tile is loaded into b, which a two-stage plan has just been read from
  if constexpr (ends_in_b<N>()) __syncthreads();
}

// One line's reader of the 12 values after the z pass:
//   e_kl = i xi_k u_l + eps_lkm phi_m,   gamma_kl = i xi_l phi_k,
// where slot 4l + 1 holds e_3l and slot 4k + 3 holds gamma_k3 as they are.  The
// kinds are selected, not branched on (a warp holds lines of every kind).
template <class R, int N>
struct StrainReader {
  const cpx<R>*w, *ph;  // u_l, phi_k or the value itself; phi_m
  const R* xi;          // x2 of the points
  R x1, sgn;            // sign of phi_m, 0 for none
  int der;              // axis of the derivative
  __device__ __forceinline__ cpx<R> operator()(int r) const {
    constexpr int step = first_step<N>();
    const cpx<R> a = w[r * step * 12], b = ph[r * step * 12];
    const R f = der == 0 ? x1 : xi[r * step];
    const cpx<R> d = cmake<R>(fma(-a.y, f, sgn * b.x), fma(a.x, f, sgn * b.y));
    return der == 2 ? a : d;
  }
};

// The 12 values after the z pass -> the 18 components, then y inverse.
template <class R, int N>
__device__ __forceinline__ void y_inverse_tile(const CellDev<R>& c, long long tile, cpx<R>* a, cpx<R>* b,
                                               const cpx<R>* tw, const R* xi) {
  const int ncols = c.n3 * c.kx, col0 = (int)tile * c.cols_y;
  const int cols = ncols - col0 < c.cols_y ? ncols - col0 : c.cols_y;
  const unsigned point = (unsigned)(c.kx * 18 * sizeof(cpx<R>));
  load_tile<R, N, 12>(c.spec, cols, c.kx, b, [&](int col) {
    int kx;
    return y_column<R, N>(c, col0 + col, kx);
  });
  line_dft<R, +1, N, 18>(
      cols, tw, a, b,
      [=, &c](int ln, int j, int col) {
        const bool is_e = ln < 9;
        const int q = is_e ? ln : ln - 9, k = q / 3, l = q - 3 * k;
        const int g = col0 + col, kx = g - div_kx(c, g) * c.kx;
        const cpx<R>* v = b + (col * N + j) * 12;
        StrainReader<R, N> s;
        s.der = is_e ? k : l;
        s.w = v + (is_e ? 4 * l : 4 * k + 2) + (s.der == 2 ? 1 : 0);
        const bool rot = is_e && k != l && k != 2;
        s.ph = rot ? v + 4 * (3 - k - l) + 2 : s.w;
        s.sgn = !rot ? R(0) : (l == (k + 1) % 3) ? R(-1) : R(1);
        s.x1 = c.n1 == 1 ? R(0) : c.two_pi_over_L[0] * (R)kx;
        s.xi = xi + j;
        return s;
      },
      [=, &c](int ln, int p, int col) {
        int kx;
        const long long i = y_column<R, N>(c, col0 + col, kx) + (long long)(p * c.kx);
        return GlobalWriter<R>{c.spec + i * 18 + ln, last_step<N>() * point};
      });
  // a one-stage plan still reads b, a three-stage one b in its last stage
  if constexpr (!ends_in_b<N>()) __syncthreads();
}

// ------------------------------------------------------------------ z pass
// Column col of a z tile is (ky, kx), index ky KX + kx; its point kz is point
// kz N2 KX + col of the spectrum.  LN = 12: the reduced fields; LN = 18
// (N2 = 1): all.
template <class R, int N, int LN>
__device__ __forceinline__ void z_tile(const CellDev<R>& c, long long tile, cpx<R>* a, cpx<R>* b, const cpx<R>* tw,
                                       const R* xi) {
  const int ncols = c.n2 * c.kx, col0 = (int)tile * c.cols_z;
  const int cols = ncols - col0 < c.cols_z ? ncols - col0 : c.cols_z;
  const unsigned point = (unsigned)ncols * (unsigned)(18 * sizeof(cpx<R>));
  cpx<R>* x = ends_in_b<N>() ? b : a;
  cpx<R>* y = ends_in_b<N>() ? a : b;
  load_tile<R, N, LN>(c.spec, cols, ncols, b, [=](int col) { return (long long)(col0 + col); });
  line_dft<R, -1, N, LN>(
      cols, tw, a, b,
      [=](int ln, int j, int col) { return TileReader<R>{b + (col * N + j) * LN + ln, first_step<N>() * LN}; },
      [=](int ln, int p, int col) { return TileWriter<R>{x + (col * N + p) * LN + ln, last_step<N>() * LN}; });
  __syncthreads();
  const R scale = (R)c.inv_nvox;
  for_rows(cols, [=, &c](int col, int p0, int dp) {
    const int ky = div_kx(c, col0 + col), kx = col0 + col - ky * c.kx;
    const R x1 = c.n1 == 1 ? R(0) : c.two_pi_over_L[0] * (R)kx;
    const R x2 = signed_freq_scale<R>(ky, c.n2, c.two_pi_over_L[1]);
    const bool nyq_y = c.n2 % 2 == 0 && ky == c.n2 / 2;
    for (int kz = p0; kz < N; kz += dp) {
      cpx<R>* pt = x + (col * N + kz) * LN;
      // zero fluctuation on the Nyquist planes of y and z and at k = 0
      if (nyq_y || (N % 2 == 0 && kz == N / 2) || (kx == 0 && ky == 0 && kz == 0)) {
#pragma unroll
        for (int q = 0; q < LN; ++q) pt[q] = cmake<R>(R(0), R(0));
      } else if constexpr (LN == 12) {
        green_point_reduced<R>(c.ref, x1, x2, xi[kz], pt, scale);
      } else {
        green_point<R>(c.ref, x1, x2, xi[kz], pt, scale);
      }
    }
  });
  __syncthreads();
  line_dft<R, +1, N, LN>(
      cols, tw, y, x,
      [=](int ln, int j, int col) { return TileReader<R>{x + (col * N + j) * LN + ln, first_step<N>() * LN}; },
      [=, &c](int ln, int p, int col) {
        const long long i = col0 + col + (long long)p * ncols;
        return GlobalWriter<R>{c.spec + i * 18 + ln, last_step<N>() * point};
      });
  __syncthreads();
}

// ------------------------------------------------------------------ kernels
template <class R>
__host__ __device__ constexpr int line_threads(int pass) {
  return pass < kZReduced ? LineCfg<R>::y_threads : LineCfg<R>::z_threads;
}
// (FP64 y passes of small radices fit four blocks' registers without spills.)
template <class R>
__host__ __device__ constexpr int line_blocks(int pass, int n) {
  return pass < kZReduced ? LineCfg<R>::y_blocks + (sizeof(R) == 8 && line_plan(n).r0 <= 9 ? 1 : 0)
         : pass == kZReduced ? LineCfg<R>::z_blocks
                             : 2;
}

template <class R, int PASS, int N>
__device__ __forceinline__ void line_tile(const CellDev<R>& c, long long tile, cpx<R>* smem, bool fresh) {
  constexpr int LN = PASS == kZReduced ? 12 : 18;
  const int cols = PASS < kZReduced ? c.cols_y : c.cols_z;
  // the axis' twiddles and angular frequencies, then the two tiles
  cpx<R>* tw = smem;
  R* xi = reinterpret_cast<R*>(tw + N);
  cpx<R>* a = tw + line_table(N);
  cpx<R>* b = a + line_pitch(N, LN) * cols;
  if (fresh) {
    const cpx<R>* t = PASS < kZReduced ? c.tw[1] : c.tw[2];
    const R f = c.two_pi_over_L[PASS < kZReduced ? 1 : 2];
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
      tw[k] = t[k];
      xi[k] = signed_freq_scale<R>(k, N, f);
    }
    // (both are read after the first barrier of the tile)
  }
  if constexpr (PASS == kYForward) y_forward_tile<R, N>(c, tile, a, b, tw, xi);
  else if constexpr (PASS == kYInverse) y_inverse_tile<R, N>(c, tile, a, b, tw, xi);
  else z_tile<R, N, LN>(c, tile, a, b, tw, xi);
}

// One cell, one length.
template <class R, int PASS, int N>
__global__ void __launch_bounds__(line_threads<R>(PASS), line_blocks<R>(PASS, N)) k_fft_y(CellDev<R> c) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  for (long long t = blockIdx.x; t < tiles_y(c); t += gridDim.x)
    line_tile<R, PASS, N>(c, t, reinterpret_cast<cpx<R>*>(smem_raw), t == (long long)blockIdx.x);
}
template <class R, int PASS, int N>
__global__ void __launch_bounds__(line_threads<R>(PASS), line_blocks<R>(PASS, N)) k_green_z(CellDev<R> c) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  for (long long t = blockIdx.x; t < tiles_z(c); t += gridDim.x)
    line_tile<R, PASS, N>(c, t, reinterpret_cast<cpx<R>*>(smem_raw), t == (long long)blockIdx.x);
}

#define MP_LINE_LENGTHS(X)                                                                                   \
  X(1) X(2) X(4) X(6) X(8) X(12) X(16) X(18) X(24) X(32) X(36) X(48) X(54) X(64) X(72) X(96) X(108) X(128) \
  X(144) X(162) X(192) X(216) X(256) X(288) X(324) X(384) X(432) X(486) X(512)

// Whether a pass meets a length: cells of one y point have no y pass, and FP64
// columns beyond 384 points do not fit a tile (sizes_fit).
template <class R>
__host__ __device__ constexpr bool line_exists(int pass, int n) {
  return (n > 1 || pass >= kZReduced) && (sizeof(R) == 4 || n <= 384);
}

// Several cells: the length is dispatched per tile.
template <class R, int PASS>
__device__ __forceinline__ void line_tile_any(const CellDev<R>& c, long long tile, cpx<R>* smem, bool fresh) {
  switch (PASS < kZReduced ? c.n2 : c.n3) {
#define MP_CASE(N) \
  case N:                                                                              \
    if constexpr (line_exists<R>(PASS, N)) line_tile<R, PASS, N>(c, tile, smem, fresh); \
    break;
    MP_LINE_LENGTHS(MP_CASE)
#undef MP_CASE
    default: break;  // refused by validation
  }
}
template <class R, int PASS>
__global__ void __launch_bounds__(line_threads<R>(PASS), line_blocks<R>(PASS, 256)) k_line_multi(Work<R> w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ CellDev<R> cs;
  for_items<R, true>(CellDev<R>{}, 0, w, cs, [&](const CellDev<R>& c, long long t, bool fresh) {
    cpx<R>* smem = reinterpret_cast<cpx<R>*>(smem_raw);
    if constexpr (PASS == kZReduced) {
      if (c.n2 == 1) line_tile_any<R, kZFull>(c, t, smem, fresh);
      else line_tile_any<R, kZReduced>(c, t, smem, fresh);
    } else {
      line_tile_any<R, PASS>(c, t, smem, fresh);
    }
  });
}

// ------------------------------------------------------------------ launches
template <class R, int PASS, int N>
const void* line_kernel() {
  if constexpr (!line_exists<R>(PASS, N)) return nullptr;
  else if constexpr (PASS < kZReduced) return (const void*)k_fft_y<R, PASS, N>;
  else return (const void*)k_green_z<R, PASS, N>;
}
template <class R, int PASS>
const void* line_kernel(int n) {
  switch (n) {
#define MP_CASE(N) \
  case N: return line_kernel<R, PASS, N>();
    MP_LINE_LENGTHS(MP_CASE)
#undef MP_CASE
    default: return nullptr;
  }
}

template <class R, int PASS>
int line_block(int n, int cols) {
  const int want = ((PASS == kZReduced ? 12 : 18) * n * cols / (sizeof(R) == 4 ? 16 : 12) + 31) / 32 * 32;
  return want < 64 ? 64 : want > line_threads<R>(PASS) ? line_threads<R>(PASS) : want;
}

template <class R, int PASS>
int line_grid(const CellDev<R>& c, int nsm) {
  const int n = PASS < kZReduced ? c.n2 : c.n3, cols = PASS < kZReduced ? c.cols_y : c.cols_z;
  const void* fn = line_kernel<R, PASS>(n);
  if (!fn) return 1;
  const int threads = line_block<R, PASS>(n, cols);
  const long long tiles = PASS < kZReduced ? tiles_y(c) : tiles_z(c);
  const long long most = (long long)resident_blocks(fn, threads, smem_line<R>(n, cols, PASS == kZReduced ? 12 : 18), true) * nsm;
  return (int)(tiles < most ? tiles : most);
}

template <class R, int PASS>
cudaError_t launch_line(const CellDev<R>& c, int grid, cudaStream_t st) {
  const int n = PASS < kZReduced ? c.n2 : c.n3, cols = PASS < kZReduced ? c.cols_y : c.cols_z;
  const void* fn = line_kernel<R, PASS>(n);
  if (!fn) return cudaErrorInvalidValue;
  CellDev<R> arg = c;
  void* args[] = {&arg};
  return cudaLaunchKernel(fn, dim3(grid), dim3(line_block<R, PASS>(n, cols)), args, smem_line<R>(n, cols, PASS == kZReduced ? 12 : 18), st);
}

template <class R, int PASS>
int line_multi_grid(long long items, size_t smem, int nsm) {
  const long long most =
      (long long)resident_blocks((const void*)k_line_multi<R, PASS>, line_threads<R>(PASS), smem, true) * nsm;
  return (int)(items < 1 ? 1 : items < most ? items : most);
}

template <class R, int PASS>
cudaError_t launch_line_multi(const Work<R>& w, int grid, size_t smem, cudaStream_t st) {
  k_line_multi<R, PASS><<<grid, line_threads<R>(PASS), smem, st>>>(w);
  return cudaGetLastError();
}

#define MP_INSTANTIATE_LINE(R, PASS, ...)                              \
  __VA_ARGS__ template int line_grid<R, PASS>(const CellDev<R>&, int); \
  __VA_ARGS__ template cudaError_t launch_line<R, PASS>(const CellDev<R>&, int, cudaStream_t);
#define MP_INSTANTIATE_LINE_MULTI(R, PASS, ...)                              \
  __VA_ARGS__ template int line_multi_grid<R, PASS>(long long, size_t, int); \
  __VA_ARGS__ template cudaError_t launch_line_multi<R, PASS>(const Work<R>&, int, size_t, cudaStream_t);

}  // namespace mp
