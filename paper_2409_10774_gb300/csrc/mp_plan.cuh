// Transform plans of one axis (host side): the radix sequence and the twiddle
// table W_N^k = exp(-2 pi i k / N).  Header-only, with no dependency on the
// library context, so that every entry point (allocating or not) builds its
// plans from the same code.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include "mp_common.cuh"

namespace mp {

// Columns of length n per y / z tile, of `ncols` in all, on `nsm` SMs.  Cells
// launched together (shared) take about 256 points (FP32) or 128 (FP64).  A
// cell alone takes, in FP64, fewer where that would not give every SM two
// tiles (16^3: the three passes took 106 us in 8 tiles of 16 columns, 40 us in
// 128 of one; fewer columns than that only leave lanes of the FP64 pipe idle),
// and in FP32 the size that ends soonest: the tiles run in waves of what the
// SMs hold - about 800 points each, in at most 32 blocks - and a wave costs its
// tile's points plus a fixed latency, about 100 points' worth (64^3: 11.9 us a
// pass in 512 tiles of four columns, which is one wave and an eighth, 10.6 us
// in 2048 of one; 256 x 128 x 8: the z pass 26 us in tiles of one column, 17 us
// in tiles of two, which an unlimited number of blocks would not be given).
constexpr int kTileBlocks = 32;  // blocks an SM holds at most
inline int tile_columns(int n, long long ncols, bool fp64, bool shared, int nsm) {
  const int full = n < (fp64 ? 128 : 256) ? (fp64 ? 128 : 256) / n : 1;
  if (shared) return full;
  if (fp64) {
    const long long most = ncols / (2 * nsm) > 1 ? ncols / (2 * nsm) : 1;
    return full < most ? full : (int)most;
  }
  int best = full;
  double best_cost = INFINITY;
  for (int cols = full; cols >= 1; --cols) {
    int blocks = 800 / (cols * n);
    blocks = blocks < 1 ? 1 : blocks > kTileBlocks ? kTileBlocks : blocks;
    const long long tiles = (ncols + cols - 1) / cols, slots = (long long)nsm * blocks;
    const double cost = (double)((tiles + slots - 1) / slots) * (cols * n + 100.0);
    if (cost < 0.97 * best_cost) {
      best = cols;
      best_cost = cost;
    }
  }
  return best;
}

// Radix sequence of the packed x axis' complex transform of length n1 / 2 = 2^a 3^b
// (for the lengths without compile-time stages): powers of two in as few
// radix-8 stages as possible, radix-3 stages last.
inline RadixPlan radix_plan(int n1) {
  RadixPlan p{};
  p.m = n1 > 1 ? n1 / 2 : 1;
  int m = p.m;
  int k2 = 0;
  while (m % 2 == 0) {
    m /= 2;
    ++k2;
  }
  int k3 = 0;
  while (m % 3 == 0) {
    m /= 3;
    ++k3;
  }
  static const int kPlan2[10][3] = {{0}, {2}, {4}, {8}, {4, 4}, {8, 4}, {8, 8}, {8, 4, 4}, {8, 8, 4}, {8, 8, 8}};
  static const int kLen2[10] = {0, 1, 1, 1, 2, 2, 2, 3, 3, 3};
  for (int i = 0; i < kLen2[k2]; ++i) p.radix[p.nstages++] = kPlan2[k2][i];
  for (int i = 0; i < k3; ++i) p.radix[p.nstages++] = 3;
  return p;
}

// Twiddle table of an axis, computed in FP64 and rounded to R (n entries).
template <class R>
void twiddle_table(int n, cpx<R>* tw) {
  for (int k = 0; k < n; ++k) {
    const double a = 2.0 * M_PI * (double)k / (double)n;
    tw[k].x = (R)std::cos(a);
    tw[k].y = (R)(-std::sin(a));
  }
}

// What a Green-operator call uploads, as one image: `words` zeroed 32-bit words
// (status and control), then the three axes' twiddle tables, 16-byte aligned.
// Fills `image` (kImageBytes) and the tables' byte offsets; returns the image's
// size.
constexpr size_t kImageBytes = 32 * 1024;
template <class R>
size_t operator_image(const int32_t n[3], size_t words, unsigned char* image, size_t table[3]) {
  size_t o = (words * 4 + 15) / 16 * 16;
  std::memset(image, 0, o);
  for (int a = 0; a < 3; ++a) {
    table[a] = o;
    twiddle_table<R>(n[a], reinterpret_cast<cpx<R>*>(image + o));
    o += ((size_t)n[a] * sizeof(cpx<R>) + 15) / 16 * 16;
  }
  return o;
}
static_assert(4 * (4 + 2 + 2 * 256) + 16 + 3 * 512 * sizeof(cpx<double>) <= kImageBytes,
              "the largest image: control words of 256 kx planes, three axes of 512 points");

}  // namespace mp
