// Launchers of the solver kernels (host-callable; defined in mp_kernels.cu).
#pragma once

#include "mp_common.cuh"
#include "mp_fft.cuh"

namespace mp {

struct LaunchCfg {
  int rows = 1;    // rows per pass-A work item
  long long items_a = 1;
  int threads_a = 256;  // threads of a pass-A block
  int grid_a = 1;  // pass-A grid (persistent, one error partial per block)
  int grid_max = 1;  // the largest grid_a of any configuration on this device
  int cols_y = 1, cols_z = 1;  // columns per tile of the y / z passes
  int grid_y = 1;
  int grid_z = 1;
  int grid_v = 1;  // per-voxel kernels (init, commit, fields)
};

// Most pass-A blocks per SM of any launch configuration (one error partial each).
constexpr int kPassABlocks = 4;
// rows_wanted > 0: that many rows per pass-A item (halved until the tile fits).
// shared: the cell's work is launched together with other cells' (full y / z
// tiles; a cell alone takes smaller ones rather than leave SMs idle).
template <class R>
LaunchCfg make_launch_cfg(const CellDev<R>& c, int nsm, int rows_wanted = 0, bool shared = false);
// Writes the configuration's item and tile sizes to the cell.
template <class R>
void use_launch_cfg(CellDev<R>& c, const LaunchCfg& L) {
  c.rows_a = L.rows;
  c.items_a = L.items_a;
  c.cols_y = L.cols_y;
  c.cols_z = L.cols_z;
  c.kx_magic = c.kx > 1 ? (unsigned)(((1ull << 32) + c.kx - 1) / c.kx) : 0u;
}
// Whether the kernels' shared-memory tiles fit for this grid in precision R.
template <class R>
bool sizes_fit(int n1, int n2, int n3);

// Lets `fn` use the shared memory its static part leaves of the opt-in maximum
// on the current device (KernelLimits; tiled: the static part must fit the
// reserve), and the blocks of it an SM holds, at least 1, with the limit raised.
cudaError_t raise_smem(const void* fn, bool tiled);
int resident_blocks(const void* fn, int threads, size_t smem, bool tiled);

// The line passes (mp_lines.cuh): y forward, y inverse, and z with the Green
// operator on the reduced 12 fields or, for cells without a y pass, on all 18.
enum LinePass { kYForward = 0, kYInverse = 1, kZReduced = 2, kZFull = 3 };
// Shared memory of a tile of `cols` columns of n points: tables and two tiles
// of `lines` lines (12 in the reduced z pass, else 18).
template <class R>
size_t smem_line(int n, int cols, int lines) {
  return ((size_t)line_table(n) + ((size_t)lines * n + line_pitch(n, lines)) * cols) * sizeof(cpx<R>);
}
template <class R, int PASS>
int line_grid(const CellDev<R>& c, int nsm);
template <class R, int PASS>
cudaError_t launch_line(const CellDev<R>& c, int grid, cudaStream_t st);
template <class R, int PASS>
int line_multi_grid(long long items, size_t smem, int nsm);
template <class R, int PASS>
cudaError_t launch_line_multi(const Work<R>& w, int grid, size_t smem, cudaStream_t st);

// The kernels of one fixed-point iteration, one launch each (y pass dir -1 forward, +1 inverse).
template <class R>
cudaError_t launch_fft_y(const LaunchCfg& L, const CellDev<R>& c, int dir, cudaStream_t st);
template <class R>
cudaError_t launch_green_z(const LaunchCfg& L, const CellDev<R>& c, cudaStream_t st);
// What pass A's last block does with the iteration's error: the error row
// `out` (err, the four per-field errors, status) and, with `loop`, the
// decision of a device-run loop for `handle` (a conditional WHILE node's) in
// out[6..10]: loop iterations, last low, its iteration, stopped by the watch,
// longest gap between lows (out[6..9] zeroed before the loop).
struct ErrTail {
  unsigned* counters;  // set by the launcher (in the partials buffer)
  double* out;
  int err_kind, loop;
  double tol, div_limit;
  int max_iter, stag, adapt;
  cudaGraphConditionalHandle handle;
};
// The partials buffer of a cell: group records, one record per block, arrival
// counters (zero before the first launch; every launch leaves them zero).
constexpr int kTailRecords = 64;
inline size_t partials_bytes(int nsm) {
  return sizeof(double) * kErrPartials * (size_t)(kTailRecords + kPassABlocks * nsm) + sizeof(unsigned) * (kTailRecords + 1);
}
template <class R>
cudaError_t launch_pass_a_iter(const LaunchCfg& L, const CellDev<R>& c, double* partials, const ErrTail& tail,
                               cudaStream_t st);
// Start of a load increment: (first ? zero state + e = E : predictor already in place),
// Algorithm 1 at the predictor, polarizations, forward x transform.
template <class R>
cudaError_t launch_start(const LaunchCfg& L, const CellDev<R>& c, int first, cudaStream_t st);
// Commit of a converged increment (c.predict / c.ratio select the predictor);
// avg_out[0..39] receives the homogenized averages.
template <class R>
cudaError_t launch_commit(const LaunchCfg& L, const CellDev<R>& c, double* partials, double* avg_out,
                          cudaStream_t st);

// Multi-cell launches: each Work lists the entries (cells) and their item
// prefix for one kernel family; the cells' descriptors live in device memory.
template <class R>
struct MultiCfg {
  Work<R> wy, wz, wa;   // iterating cells: y columns, z columns, pass-A items
  Work<R> ws;           // cells starting an increment: pass-A items
  Work<R> wv, wv0;      // 256-voxel chunks: commit, first-increment initialisation
  long long items_y = 0, items_z = 0, items_a = 0, items_s = 0, items_v = 0, items_v0 = 0;
  size_t smem_y = 0, smem_z = 0, smem_a = 0;  // largest tile over the entries (smem_a: pass A, both modes)
  int grid_y = 1, grid_z = 1, grid_a = 1, grid_s = 1, grid_v = 1, grid_v0 = 1;
};
template <class R>
void multi_grids(MultiCfg<R>& m, int nsm);
template <class R>
cudaError_t launch_multi_iteration(const MultiCfg<R>& m, cudaStream_t st);
template <class R>
cudaError_t launch_multi_start(const MultiCfg<R>& m, cudaStream_t st);
template <class R>
cudaError_t launch_multi_commit(const MultiCfg<R>& m, cudaStream_t st);
template <class R>
size_t smem_pass_a(int n1, int rows);
template <class R>
cudaError_t launch_fields(const LaunchCfg& L, const CellDev<R>& c, int from_elast, double* fe,
                          double* fg, double* ft, double* fm, double* fp, double* fq, cudaStream_t st);
// ctl (FP32 cells with spectral_fused_ok only; else NULL): the fused spectral
// pass's control words, which select it for the y / z work.
template <class R>
cudaError_t launch_green_apply(const LaunchCfg& L, const CellDev<R>& c, const R* tau, const R* mu,
                               R* e_out, R* g_out, cudaStream_t st, int* ctl = nullptr, int nsm = 0);
// Algorithm 1 at `count` points.  The phase table is passed by value from
// host_phases (n_phases <= max_table_phases()), or read from dev_phases.
template <class R>
cudaError_t launch_radial_return(int nsm, long long count, const uint16_t* phase, int n_phases,
                                 const PhaseDev<R>* host_phases, const PhaseDev<R>* dev_phases, const R* e,
                                 const R* g, const R* e_n, const R* g_n, const R* t_n, const R* m_n,
                                 const double* p_n, const double* q_n, R* t, R* m, double* p, double* q,
                                 cudaStream_t st);
int max_table_phases();

// Fused spectral pass (y forward, z forward, Green operator, z inverse, y
// inverse in one persistent launch; mp_spectral.cu) for FP32 cells whose y
// and z lengths are 256.  ctl: spectral_ctl_ints(c.kx) ints of device memory
// (zeroed by the launcher on `st`).
bool spectral_fused_ok(const CellDev<float>& c);
size_t spectral_ctl_ints(int kx);
cudaError_t launch_spectral(const CellDev<float>& c, int* ctl, int nsm, cudaStream_t st);

// dst[i] = (D) src[i], i < n (state of a cell changing precision).
template <class S, class D>
cudaError_t launch_convert(const S* src, D* dst, long long n, int nsm, cudaStream_t st);

}  // namespace mp
