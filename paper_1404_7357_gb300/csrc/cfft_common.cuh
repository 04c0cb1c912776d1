// Shared device/host helpers of the GB300 C-FFT kernels: a small complex type,
// precision-overloaded math, and the kernel argument structs.  Nothing here
// is specific to one stage; every formula lives in the kernel that uses it.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <vector>

namespace cfft {

// streaming multiprocessors of the current device (persistent grids and grid-stride caps
// are sized from it; the runtime caches the attribute)
inline int current_sm_count() {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) {
    cudaGetLastError();
    v = 1;
  }
  return v;
}

template <class T>
struct alignas(2 * sizeof(T)) cpx {
  T re, im;
};

template <class T>
__host__ __device__ __forceinline__ cpx<T> mk(T r, T i) {
  cpx<T> z;
  z.re = r;
  z.im = i;
  return z;
}
template <class T>
__host__ __device__ __forceinline__ cpx<T> operator+(cpx<T> a, cpx<T> b) {
  return mk(a.re + b.re, a.im + b.im);
}
template <class T>
__host__ __device__ __forceinline__ cpx<T> operator-(cpx<T> a, cpx<T> b) {
  return mk(a.re - b.re, a.im - b.im);
}
template <class T>
__host__ __device__ __forceinline__ cpx<T> operator*(cpx<T> a, cpx<T> b) {
  return mk(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
template <class T>
__host__ __device__ __forceinline__ cpx<T> operator*(T s, cpx<T> a) {
  return mk(s * a.re, s * a.im);
}
template <class T>
__host__ __device__ __forceinline__ cpx<T> conj(cpx<T> a) {
  return mk(a.re, -a.im);
}
// a += b * c
template <class T>
__host__ __device__ __forceinline__ void cmac(cpx<T>& a, cpx<T> b, cpx<T> c) {
  a.re = fma(b.re, c.re, fma(-b.im, c.im, a.re));
  a.im = fma(b.re, c.im, fma(b.im, c.re, a.im));
}
// a += conj(b) * c
template <class T>
__host__ __device__ __forceinline__ void cmac_conj(cpx<T>& a, cpx<T> b, cpx<T> c) {
  a.re = fma(b.re, c.re, fma(b.im, c.im, a.re));
  a.im = fma(b.re, c.im, fma(-b.im, c.re, a.im));
}
template <class T>
__host__ __device__ __forceinline__ cpx<T> cdiv(cpx<T> a, cpx<T> b) {
  // Smith's algorithm
  if (fabs(b.re) >= fabs(b.im)) {
    T r = b.im / b.re, d = b.re + b.im * r;
    return mk((a.re + a.im * r) / d, (a.im - a.re * r) / d);
  }
  T r = b.re / b.im, d = b.im + b.re * r;
  return mk((a.re * r + a.im) / d, (a.im * r - a.re) / d);
}
template <class TO, class TI>
__host__ __device__ __forceinline__ cpx<TO> ccast(cpx<TI> a) {
  return mk<TO>((TO)a.re, (TO)a.im);
}

// precision-overloaded accurate math (never the fast-math intrinsics)
__device__ __forceinline__ void sincospi_(float x, float* s, float* c) { sincospif(x, s, c); }
__device__ __forceinline__ void sincospi_(double x, double* s, double* c) { sincospi(x, s, c); }
__device__ __forceinline__ void sincos_(float x, float* s, float* c) { sincosf(x, s, c); }
__device__ __forceinline__ void sincos_(double x, double* s, double* c) { sincos(x, s, c); }
__device__ __forceinline__ float exp_(float x) { return expf(x); }
__device__ __forceinline__ double exp_(double x) { return exp(x); }
__device__ __forceinline__ float cospi_(float x) { return cospif(x); }
__device__ __forceinline__ double cospi_(double x) { return cospi(x); }

// e^{i pi x} with x reduced exactly modulo 2 in float64 first
template <class T>
__device__ __forceinline__ cpx<T> expipi(double x) {
  double r = x - 2.0 * floor(0.5 * x);  // [0, 2)
  T s, c;
  sincospi_((T)r, &s, &c);
  return mk(c, s);
}

__device__ __forceinline__ float sinh_(float x) { return sinhf(x); }
__device__ __forceinline__ double sinh_(double x) { return sinh(x); }
__device__ __forceinline__ float cosh_(float x) { return coshf(x); }
__device__ __forceinline__ double cosh_(double x) { return cosh(x); }

// sin(z), cos(z) for complex z.  sinh of the imaginary part comes from the library
// function, not from (e^y - e^-y)/2, whose cancellation for small y leaves an
// absolute error of one ulp of 1 in Im sin z (amplified by 1/|z| in sin(z)/z).
template <class T>
__device__ __forceinline__ void csincos(cpx<T> z, cpx<T>* sz, cpx<T>* cz) {
  T s, c;
  sincos_(z.re, &s, &c);
  const T ch = cosh_(z.im), sh = sinh_(z.im);
  *sz = mk(s * ch, c * sh);
  *cz = mk(c * ch, -s * sh);
}

// sin(z)/z for complex z (series near zero)
template <class T>
__device__ __forceinline__ cpx<T> csinc(cpx<T> z) {
  T a2 = z.re * z.re + z.im * z.im;
  if (a2 < (T)1e-4) {
    cpx<T> z2 = z * z;
    // 1 - z^2/6 + z^4/120 - z^6/5040
    cpx<T> t = mk((T)(-1.0 / 5040.0) * z2.re, (T)(-1.0 / 5040.0) * z2.im);
    t = mk(t.re + (T)(1.0 / 120.0), t.im);
    t = t * z2;
    t = mk(t.re - (T)(1.0 / 6.0), t.im);
    t = t * z2;
    return mk(t.re + (T)1, t.im);
  }
  cpx<T> s, c;
  csincos(z, &s, &c);
  return cdiv(s, z);
}

// principal complex square root
template <class T>
__device__ __forceinline__ cpx<T> csqrt_(cpx<T> z) {
  T r = hypot(z.re, z.im);
  if (r == (T)0) return mk((T)0, (T)0);
  if (z.re >= (T)0) {
    T t = sqrt((T)0.5 * (r + z.re));
    return mk(t, z.im / ((T)2 * t));
  }
  T t = sqrt((T)0.5 * (r - z.re));
  return mk(fabs(z.im) / ((T)2 * t), copysign(t, z.im));
}

// ---------------------------------------------------------------------------
// kernel arguments

struct ContourArgs {
  int n;
  double beta_max, beta_p, height, step;  // step = beta_max / n
  double eps_r, hs, k0;
  int extract;                            // 1: subtract the homogeneous medium and its image
  double eps_eff, deps_eff;               // its permittivity and d eps_eff / d eps_r
  int es_width;                           // > 0: ES precorrection of that kernel width
  double ds;                              // transform grid step (for the precorrection)
};

// per-node contour data written by the contour kernel (float64 throughout)
struct ContourData {
  double2* beta_c;  // beta_R + i beta_I
  double2* weight;  // step * (1 + i dbeta_I/dbeta_R)
  double2* bw;      // beta_c * weight  (the factor of Eq. 9's beta d beta)
  double* bi_rel;   // beta_I / height  (0 beyond beta_p); in [0, 1]
  float* bi_rel_f;  // the same in float32 (read by the float32 transform)
  double2* green_p; // G = P I - R k k^T  (P, R: functions of beta only)
  double2* green_r; // R * beta_c^2
  // optional (null to skip): derivatives of P and R beta_c^2 with respect to
  // eps_r and to the slab thickness h, contour held fixed
  double2* dp_eps;
  double2* dr_eps;
  double2* dp_h;
  double2* dr_h;
  // optional: 1 / phi_hat(omega_j) of the ES interpolation kernel, omega_j = (beta_c,j -
  // beta_max / 2) ds, the precorrection of the FP32-mixed transform input
  float2* prec;
};

struct ShapeClass {
  int kind;      // 0 = rooftop, 1 = cosine strip
  int dir;       // 0 = x, 1 = y
  int begin;     // basis range [begin, end) of this class (bases sorted by class)
  int end;
  double p1, p2; // rooftop: half-length, width; strip: length, width
};

constexpr int kMaxShapeClasses = 32;
constexpr int kMaxBasis = 4096;

template <class T>
struct IntegrandArgs {
  int n, n_alpha, q_max, n_cls;  // n_cls computed classes (1 or 3)
  int n_mbf;                      // real MBF count (q holds a padded column count)
  int n_shape, n_basis;
  int tables;                     // 1: the nodes are spectral_nodes' (real; D, then E on the same nodes)
  const ShapeClass* shapes;       // device, n_shape
  const T* bx;                    // device, basis centres x (sorted by class)
  const T* by;
  const cpx<T>* q;                // device, [n_basis][M padded]
  const double2* beta_c;
  const double2* bw;
  const double2* green_p;
  const double2* green_r;
  cpx<T>* y;                      // out [cls][pair][qi][n]
  // tensor-core spectra (FP32 rooftop elements): float centres, GEMM B operand (with the
  // mirrored columns of the opposite wave direction) and its width (both blocks)
  const float* tc_bx;
  const float* tc_by;
  const float* tc_bmat;
  int tc_ncol;
  float tc_rmax;                  // max |r_i| of the basis centres
  int* err;                       // bit 4: a tensor-core wait ran past its bound
};

template <class T>
struct FftArgs {
  int series, n, sub_len, log2_sub, n_sub;   // n_sub = D = P / sub_len
  int64_t fft_len;                            // P = sigma * n
  int grid_half;                              // K
  int taylor;                                 // highest term index N of the series
  int expansion;                              // contour-factor series: 0 Taylor (Eq. 22), 1 Chebyshev
  int n_active;                               // nodes with beta_I > 0 (prefix)
  int sigma;
  double ds_height;                           // delta_s * height  (series variable scale)
  const cpx<T>* y;                            // [series][n]
  const double* bi_rel;                       // [n]
  const float* bi_rel_f;                      // [n] float32 copy
  const cpx<T>* twiddle;                      // [sub_len] e^{-2 pi i t / sub_len}
  const cpx<T>* prec;                         // [n] input precorrection (null: none)
  cpx<T>* grid;                               // [series][2K+1]
  // gridded transform (null: the series of FFTs): y holds the coarse samples, fft_len their
  // FFT length, and output k is multiplied by out_factor[k + K]
  const cpx<T>* out_factor;
};

// ---- spectral tables and gridding (k_grid.cu)

// harmonics on the contour from the element's spectral tables D, E ([series][2][nc], sampled
// at beta0 + i / inv_d): y = bw (P D - R beta^2 E)
constexpr int kSpecOver = 8;   // samples per Nyquist step of the tables
template <class T>
struct SpecInterpArgs {
  int n, nc, series;
  double beta0, inv_d;
  const cpx<T>* tab;
  const double2* beta_c;
  const double2* bw;
  const double2* green_p;
  const double2* green_r;
  cpx<T>* y;               // out [series][n]
};

// shape of a gridded transform: coarse FFT length m, Gaussian exp(-a z^2) of half width hw
// cells, at most kmax nodes per cell, cells with nodes and with active nodes, coarse samples
struct GridShape {
  int m, hw, kmax, n_cells, act_cells, nc;
  double a, y_scale;
};
// Fills g and returns true when the gridded transform serves this contour and grid: height *
// rho_max <= 3.5, a coarse grid (m >= 2 (2K + 1), a power of two >= min_m) no finer than the contour's
// own transform (m <= fft_len), a contour that does not rise too many of its cells, and a Gaussian
// within the staging buffer.  Otherwise the series of FFTs runs.
bool grid_plan(bool fp64, int n, int64_t fft_len, int n_active, int grid_half, double ds, double height,
               double rho_max, int min_m, GridShape* g);

template <class T>
struct GridArgs {
  int n, series, grid_half, sigma;
  int m, hw, kmax, n_cells, act_cells, nc;
  int64_t fft_len;           // P: node j lies at (j + 1/2) m / P cells
  double a, y_scale, inv_norm;   // inv_norm = sqrt(a / pi)
  const double* bi_rel;      // [n]
  const cpx<T>* prec;        // [n] or null
  const cpx<T>* y;           // [series][n]
  T* wre;                    // [2 hw][kmax][n_cells]
  T* wim;                    // [2 hw][kmax][act_cells]
  cpx<T>* out_factor;        // [2K + 1]
  cpx<T>* coarse;            // out [series][nc]
};

template <class T>
struct BackprojArgs {
  int series_per_q;        // classes * pairs
  int n_harm, q_max, n_rho, grid_half, sigma, taps, group, rchunk;
  double d_rho, d_s;       // rho step, s step
  double beta_abs_max;     // max |beta_c| (angular content of the integrand)
  double alpha_margin;
  const cpx<T>* grid;      // [series][2K+1]   series = (cls*pairs + pair) * n_harm + qi
  cpx<T>* table;           // [series][n_rho]
  const int* chunk_nodes;  // [chunks] angular nodes of each chunk of rows
  const int64_t* chunk_off;// [chunks] offset of its cosines in cosv
  const double* cosv;      // node cosines
  int* err;                // tensor-core form: bit 5 set when a wait ran past its bound
  int kern;                // interpolation kernel: 0 Lagrange, 1 ES (precorrected grid)
  // > 0: only the rows below sum_first_row(low_h, |q|) are formed (the sample sums form the
  // others); the rho step in grid samples
  double low_h;
};

// The far part of the sample sums is interpolated over cells of rows (k_backproject_sum.cu), where
// the weights of harmonic q turn up to about sqrt(width) times from row q^2 on.  Up to |q| =
// kSumNarrow any width keeps the interpolation's error (single tones, times 2 pi) at 1.6e-7 in
// float32 and 5e-15 in float64; above, a cell is at most sum_cell_width samples wide (2e-7,
// 3e-14), where that leaves it kSumCellRows rows (of fewer, the far part's points would be as many
// as the rows).  Wider: |q| = 32 7e-6, 64 6e-4 in float32 (6e-13, 3e-10 in float64).
constexpr int kSumNarrow = 16, kSumCellRows = 16;
__host__ __device__ constexpr double sum_cell_width(bool fp64) { return fp64 ? 150.0 : 36.0; }

// first row that the sums over grid samples serve for harmonics +-p (k_backproject_sum.cu); h:
// the rho step in grid samples
__host__ __device__ inline int sum_first_row(double h, int p, bool fp64) {
  if (p > kSumNarrow && (kSumCellRows - 1) * h > sum_cell_width(fp64)) return 2000000000;   // none
  // end weights against Bessel functions there (single tones, times 2 pi): float32 1e-7,
  // float64 1e-13, falling like u^-3 and faster beyond
  const double u = (fp64 ? 1.0 : 0.5) * (double)p * (double)p;
  const double r = ceil((u > 40.0 ? u : 40.0) / h);
  return r < 2.0e9 ? (int)r : 2000000000;
}

// back-projection by sums over the grid samples
template <class T>
struct SumArgs {
  int series_per_q, n_harm, q_max, n_rho, grid_half, sigma;
  int n_cells, cell_rows;  // n_cells = 0: not in use
  int k_used, k_pad;       // samples k >= 0 the rows read, and the folded arrays' length
  int split;               // samples of a far block's share of a sum
  double d_rho, d_s;
  const cpx<T>* grid;      // [series][2K+1]
  cpx<T>* table;           // [series][n_rho]
  cpx<T>* wrow;            // [end sample][n_rho]
  T* fold;                 // [|q|][chunk of 16 or 4 series][G+, i G-][k_pad][64 or 16 columns]
  cpx<T>* far;             // [split][|q|][chunk][cell][point][32 or 8]
};
struct SumPlan {
  int cells, cell_rows, k_used, k_pad, split, splits, tiles;
  size_t fold, far, wrow;  // elements of the three buffers (real, complex, complex)
};
// false (and an empty plan) where the sums do not serve: another zero padding than the end
// weights were made for, a grid that ends before the end samples, no row far enough out
bool sum_plan(bool fp64, int n_rho, double d_rho, double d_s, int sigma, int grid_half, int taps, int kern, int q_max,
              int series_per_q, int sms, SumPlan* p);
int sum_grid_extra(bool fp64, int taps, int kern);
int sum_tile_rows();
int sum_fold_samples();
template <class T>
cudaError_t launch_backproject_sum(const SumArgs<T>& a, int taps, int kern, int splits, int tiles, cudaStream_t s);
template <class T>
cudaError_t launch_backproject_sum_batch(const SumArgs<T>* items, int first, int n_items, int n_rho, const int2* fold_map,
                                         int n_fold, const int2* far_map, int n_far, const int2* near_map, int n_near,
                                         int max_splits, int q_max, int series_per_q, int taps, int kern,
                                         cudaStream_t s);

// back-projection with the W x G+- product on the tensor cores (FP32-mixed)
size_t backproject_tc_smem(int max_nodes);
int backproject_tc_ktile();
cudaError_t launch_backproject_tc(const BackprojArgs<float>& a, int n_tiles, int max_nodes, cudaStream_t s);
cudaError_t launch_backproject_tc_batch(const BackprojArgs<float>* items, const int4* tasks, int n_tasks,
                                        int* counter, int taps, int kern, int max_nodes, int n_ctas,
                                        cudaStream_t s);

template <class T, class TO>
struct FillArgs {
  int n_el, n_mbf, q_max, n_harm, n_rho, taps, n_cls;
  double inv_d_rho, rho_max;
  int64_t ld;
  const cpx<T>* table;     // [cls][pair][qi][r]
  const double* pos;       // [2 * n_el]
  const int* rot;          // [n_el] or null
  cpx<TO>* z;              // [(m*M + a) * ld + n*M + b]
  int* err;                // set when a pair lies beyond rho_max
  // a lattice's displacements in place of element pairs (FP64, bucketed): "pair" (m, n), m < n_rows,
  // n < n_el, is the displacement (dx[m], dy[n]), and bad[m * n_el + n] is set in place of err
  int n_rows;              // 0: n_el
  const double* dx;        // null: element pairs
  const double* dy;
  unsigned char* bad;
};

// one coordinate of a lattice (k_fill_lattice.cu)
constexpr int kLatAxis = 96;   // different values at most
struct LatticeAxis {
  int* id;        // [n_el]
  int* did;       // [kLatAxis^2]
  double* ud;     // [kLatAxis^2]
  int* info;      // [2] different values (0: too many), different differences
};

// host launchers (one translation unit per stage)
void spectral_table_shape(bool fp64, double elem_radius, double beta_max, int* nc, double* beta0, double* d);
bool spectral_tables_serve(int nc, double d, int n, double height);
void launch_spectral_nodes(int nc, double beta0, double d, double2* beta, double2* bw, double2* gp, double2* gr,
                           cudaStream_t s);
template <class T>
cudaError_t launch_spectral_interp(const SpecInterpArgs<T>& a, cudaStream_t s);
// contour nodes per block of the batched interpolation
template <class T>
int spectral_interp_nodes();
template <class T>
cudaError_t launch_spectral_interp_batch(const SpecInterpArgs<T>* items, const int2* map, int n_blocks, int series,
                                         cudaStream_t s);
template <class T>
cudaError_t launch_grid_tables(const GridArgs<T>& a, cudaStream_t s);
template <class T>
cudaError_t launch_grid_tables_batch(const GridArgs<T>* items, int item0, int n_items, cudaStream_t s);
template <class T>
cudaError_t launch_spread(const GridArgs<T>& a, cudaStream_t s);
// coarse samples per block of the batched spreading
int spread_samples();
template <class T>
cudaError_t launch_spread_batch(const GridArgs<T>* items, const int2* map, int n_blocks, int series, int max_hw,
                                cudaStream_t s);
void launch_contour(const ContourArgs& a, const ContourData& d, cudaStream_t s);
template <class T>
void launch_twiddle(cpx<T>* tw, int len, cudaStream_t s);
template <class T>
cudaError_t launch_integrand(const IntegrandArgs<T>& a, int n_mbf_padded, cudaStream_t s);
template <class T>
cudaError_t launch_fft(const FftArgs<T>& a, cudaStream_t s);
template <class T>
int integrand_tile_nodes(const IntegrandArgs<T>& a, int n_mbf_padded);
// fused integrand with the MBF spectra on the tensor cores (FP32, N_alpha = 128 or 256,
// a.tc_* set); false when the form does not apply
bool integrand_tc_applies(const IntegrandArgs<float>& a);
cudaError_t launch_integrand_tc(const IntegrandArgs<float>& a, cudaStream_t s);
// contour nodes per CTA of the tensor-core integrand (n_alpha 128 or 256), and its batched launch
int integrand_tc_nodes(int n_alpha);
cudaError_t launch_integrand_tc_batch(const IntegrandArgs<float>& shape_args, const IntegrandArgs<float>* items,
                                      const int2* map, int n_blocks, cudaStream_t s);
template <class T>
cudaError_t launch_integrand_batch(const IntegrandArgs<T>& shape_args, const IntegrandArgs<T>* items,
                                   const int2* map, int n_blocks, int jt, int n_mbf_padded,
                                   cudaStream_t s);
void launch_contour_batch(const ContourArgs* items, const ContourData* data, const int2* map,
                          int n_blocks, cudaStream_t s);
// shared-memory bytes of one transform task beyond its FFT buffer
template <class T>
__host__ __device__ constexpr size_t fft_task_extra(int /*n_active_max*/, int n_out_max, int hi_max) {
  return (size_t)(128 + hi_max + 128 + 128) * sizeof(cpx<T>) +
         (size_t)n_out_max * (sizeof(cpx<T>) + sizeof(T)) + 64;
}

// max_n_out of a gridded batch, whose tasks keep no outputs in shared memory (others: less two)
constexpr int kNoOutputs = -2;
template <class T>
cudaError_t launch_fft_batch(const FftArgs<T>* items, const int4* tasks, int n_tasks, int* counter,
                             int log2_sub, int max_n_out, int max_active, int max_hi, int zt_arrays,
                             int n_ctas, cudaStream_t s);
template <class T>
size_t backproject_smem(int group, int max_seg, int max_nodes);
template <class T>
cudaError_t launch_backproject_impl(const BackprojArgs<T>& a, const int* chunk_nodes,
                                    const int64_t* chunk_off, const double* cosv,
                                    const double* lag_den, int n_chunks, int max_nodes,
                                    int max_seg, cudaStream_t s);
template <class T>
cudaError_t launch_backproject_batch(const BackprojArgs<T>* items, const int4* tasks, int n_tasks,
                                     int* counter, int taps, int group, int max_nodes, int max_seg,
                                     int n_ctas, cudaStream_t s);
cudaError_t launch_chunk_cosines(const int* n_nodes, const int64_t* offset, int n_chunks,
                                 int max_nodes, double* cosv, cudaStream_t s);
template <class T>
size_t backproject_w_smem(int rows, int max_nodes, int series);
// paired-harmonic matrix form (FP32-mixed, taps 8/12/16): tiles of backproject_pm_rows()
// rows, tasks (tile, |q|, chunk of backproject_pm_series_chunk() series per sign)
size_t backproject_pm_smem(int max_nodes);
int backproject_pm_rows();
int backproject_pm_series_chunk();
cudaError_t launch_backproject_pm(const BackprojArgs<float>& a, int n_tiles, int max_nodes, cudaStream_t s);
cudaError_t launch_backproject_pm_batch(const BackprojArgs<float>* items, const int4* tasks, int n_tasks,
                                        int* counter, int taps, int kern, int max_nodes, int n_ctas,
                                        cudaStream_t s);
int backproject_w_rows();
int backproject_w_low_rows(int n_rows, int n_harm);   // low rows beside the sums
template <class T>
cudaError_t launch_backproject_w(const BackprojArgs<T>& a, int n_tiles, int max_nodes, cudaStream_t s);
template <class T>
cudaError_t launch_backproject_w_batch(const BackprojArgs<T>* items, const int4* tasks, int n_tasks,
                                       int* counter, int taps, int max_nodes, int series, int n_ctas,
                                       cudaStream_t s);
template <class T>
void launch_class_phase(cpx<T>* table, int pairs, int n_harm, int q_max, int n_rho,
                        cudaStream_t s);
template <class T>
void launch_nonfinite(const cpx<T>* buf, int64_t count, int* flag, cudaStream_t s);
template <class T, class TG>
struct FillBackArgs {
  FillArgs<T, float> f;      // geometry and table (f.z unused)
  const cpx<T>* dtab_eps;    // d table / d eps_r  (null: no substrate gradient)
  const cpx<T>* dtab_h;      // d table / d h
  const cpx<TG>* grad;       // dL/dZ (torch convention: dL = Re sum conj(G) dZ)
  int64_t ld_g;
  double d_rho;
  double* grad_pos;          // [2 * n_el], accumulated
  double* grad_theta;        // [2], accumulated (eps_r, h)
};

// plan of the bucketed fill (pairs counting-sorted by rotation class and
// stencil row, table windows staged in shared memory); ok = false: per-row fill
struct FillBucketPlan {
  bool ok;
  bool tc;                 // the tensor-core form (FP32, M = 4, 8 taps)
  int win, n_cells, nb_bits, block_rows, rows_per_wave;
  size_t n_keys_max, smem, scratch;
  bool direct;             // few pairs: no sort, a block per pair (fill only)
  int parts;               // CTAs per window of the fill (0: by their number)
};
// pairs up to which fill_direct_kernel is the faster fill
constexpr int64_t direct_pairs(bool fp64) { return fp64 ? 2048 : 6144; }
template <class T>
FillBucketPlan plan_fill_bucketed(int n_el, int n_mbf, int n_harm, int n_rho, int taps, int n_cls,
                                  int block_rows, bool tc, bool lattice = false);
template <class T>
cudaError_t launch_fill_bucketed(const FillArgs<T, T>& a, const FillBucketPlan& plan, void* scratch,
                                 cudaStream_t s);
cudaError_t launch_lattice_axes(int n_el, const double* pos, const LatticeAxis& ax, const LatticeAxis& ay,
                                cudaStream_t s);
// counts: info of ax, then of ay; plan, scratch: those of max(counts[1], counts[3]) elements, one
// class; blocks: [n_cls][counts[1] M][counts[3] M]; bad: [counts[1]][counts[3]]
cudaError_t launch_fill_lattice(const FillArgs<double, double>& a, const LatticeAxis& ax, const LatticeAxis& ay,
                                const int (&counts)[4], const FillBucketPlan& plan, void* scratch, void* blocks,
                                unsigned char* bad, cudaStream_t s);
// adjoint of the bucketed fill: position gradient (grad_pos) and, with both
// derivative tables, the (eps_r, h) gradient (grad_theta[0..1]); both accumulated
template <class T>
struct FillAdjointArgs {
  const cpx<T>* grad;        // dL/dZ, same layout as the matrix, leading dimension ld_g
  int64_t ld_g;
  const cpx<T>* dtab_eps;    // d table / d eps_r, or null
  const cpx<T>* dtab_h;      // d table / d h, or null
  double* grad_pos;          // [2 * n_el] or null
  double* grad_theta;        // [2] or null
};
template <class T>
cudaError_t launch_fill_adjoint_bucketed(const FillArgs<T, T>& a, const FillAdjointArgs<T>& ad,
                                         const FillBucketPlan& plan, void* scratch, cudaStream_t s);

// the bounded mbarrier wait, run out on purpose: flag = 16 after `polls` tries
cudaError_t launch_wait_selftest(unsigned polls, int* flag, cudaStream_t s);

// MBF spectra on the tensor cores (FP32 with TF32 head/tail splitting)
int spectra_tc_columns(int n_shape, int n_mbf);
void spectra_tc_bmatrix(int n_basis, int n_shape, const int* basis_class, int n_mbf,
                        const double* q_re_im, int q_stride, bool mirror, std::vector<float>* out);
cudaError_t launch_spectra_tc(int n_points, int n_basis, int n_shape, int n_mbf, const ShapeClass* shapes,
                              const float* bx, const float* by, const float* bmat, const void* k, void* out,
                              int* err, cudaStream_t s);

template <class T, class TG>
cudaError_t launch_fill_backward(const FillBackArgs<T, TG>& a, cudaStream_t s);
// g[i][j] = 2 r_i conj(v_j), n x n row-major (dL/dZ' of sum |Z' v - t|^2 with r = Z' v - t)
template <class T>
cudaError_t launch_residual_outer(const void* r, const void* v, int n, void* g, cudaStream_t s);
// a posteriori interpolation-error estimate of the fill on a table's rho grid: per series
// (n_rho entries each) out = (max |Z|, max over interior windows of |p-th difference| *
// fac_c, the last window's |p-th difference| * fac_e, 0)
template <class T>
cudaError_t launch_fill_estimate(const void* table, int64_t n_series, int n_rho, int q_max, int taps,
                                 double fac_c, double fac_e, double4* out, cudaStream_t s);
// the 2-D Cartesian C-FFT (k_cartesian.cu): N x N spectral samples on [-k_max, k_max)^2
// (dk = 2 k_max / N), the contour (beta_p, height), the substrate and the element
template <class T>
struct CartArgs {
  int n, n_mbf, n_shape, q_stride;
  double k_max, dk, beta_p, height, eps_r, hs, k0;
  int extract;
  double eps_eff;
  const ShapeClass* shapes;
  const T* bx;
  const T* by;
  const cpx<T>* q;   // [n_basis][q_stride], bases sorted by shape class
};
// the refined table [pairs][2N][2N] (dx-major) up to Taylor order `order`; work: [pairs][N][2N]
// (row transforms of one power); im: [pairs][N][N]; gx, gy: [N][N]
template <class T>
cudaError_t cartesian_tabulate(const CartArgs<T>& a, int order, cpx<T>* table, cpx<T>* work, cpx<T>* im, T* gx,
                               T* gy, cudaStream_t s);
template <class T, class TO>
cudaError_t cartesian_fill(const cpx<T>* table, int p, int m, double x0, double step, double rho_max, int n_el,
                           const double* pos, void* z, int64_t ld, int* err, cudaStream_t s);

// dense LU of the reduced system (k_solve.cu): device work arrays of one factorization
struct LuWork {
  int2* moves;         // [panels][2][panel width] row moves (source, destination): a whole panel's
                       // list, or one list per half
  int* n_moves;        // [panels][2]
  double* cand_val;    // [2][SMs] 64-bit words: the panel CTAs' pivot keys with column tags
  int* perm;           // [n] the factors' row order
  void* cand_data;     // [2][SMs][panel width] complex, the element type: the candidates' entries
  unsigned long long* words;  // [2][n] solved entries with tags: 2 (complex64) or 4 words each
  int* err;            // bit 1: a key poll ran out; bit 2: zero pivot; bit 3: a tensor-core
                       // wait of the trailing update ran out; bit 4: a wait of a substitution
  int* diag;           // host: [5] panel grid, resident CTAs per SM, shared bytes of the last grid
                       // panel; panels run on one cluster, CTAs per cluster (0: none)
  cudaStream_t side;   // second stream and events of the look-ahead
  cudaEvent_t ev[3];
  bool (*fail_forked)();   // failure injection: a launch behind the fork is to fail
  int tc_update;       // complex64: the trailing update on the tensor cores
  int panel_cluster;   // 1: panels whose rows fit one cluster's shared memory run there
};
int lu_panel_width();
// the largest order whose panels fit the panel CTAs' shared memory on `sms` SMs
template <class T>
int lu_max_order(int sms);
template <class T>
cudaError_t lu_factor(cpx<T>* a, int64_t ld, int n, const LuWork& w, cudaStream_t s);
template <class T>
cudaError_t lu_solve(const cpx<T>* a, int64_t ld, int n, const LuWork& w, cpx<T>* x, cpx<T>* y, cudaStream_t s);
cudaError_t residual_f64(const void* z, int64_t ld, int n, const void* x, const void* b, void* r, double* sums,
                         cudaStream_t s);
cudaError_t residual_f32(const void* z, int64_t ld, int n, const void* x, const void* b, double* sums,
                         cudaStream_t s);
template <class TD, class TS>
cudaError_t copy_matrix(const void* src, int64_t ld, int n, void* dst, int64_t ld_dst, cudaStream_t s);
template <class TD, class TS>
cudaError_t copy_vector(const void* src, int n, void* dst, cudaStream_t s);
cudaError_t add_correction(void* x, const void* d, int n, double* sums, cudaStream_t s);
// kind 0: V' = Q^H V; 1: delta-gap port excitation; 2: port currents (q: complex128 [B][M])
template <class T>
cudaError_t launch_excitation(int kind, int n_el, int n_basis, int m, int port, const void* in, const double* q,
                              void* out, cudaStream_t s);

// plan.ok: bucketed fill with `scratch` of plan.scratch bytes; else the per-row fill
template <class T, class TO>
cudaError_t launch_fill(const FillArgs<T, TO>& a, const FillBucketPlan& plan, void* scratch, cudaStream_t s);

}  // namespace cfft
