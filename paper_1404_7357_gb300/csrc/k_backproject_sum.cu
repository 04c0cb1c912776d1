// Back-projection by sums over the grid samples themselves.
//
//   Z_q(rho) = 1/(2 pi^2) int_0^pi cos(q alpha) g_q(rho cos alpha) d alpha
//            = 1/(2 pi^2) int_{-rho}^{rho} T_q(t / rho) g_q(t) / sqrt(rho^2 - t^2) dt.
// g_q is known at the samples t = k ds, sigma times denser than its band needs, so away from
// the ends t = +-rho the trapezoidal rule over the samples is exact to all digits; the inverse
// square root at each end takes a fixed number of corrected weights that depend on the
// fractional part of u = rho / ds alone (end_weights.cuh, gen_end_weights.py):
//   Z = 1/(2 pi^2) sum_{k >= 0} A_k G+(k) + i B_k G-(k),  G+-(k) = g(k) +- (-1)^q g(-k),
//   A_k = T_q(k / u) / sqrt(u^2 - k^2)                        up to floor(u) - kIn
//   A_k + i B_k = w_j(u - floor(u)) T_q(k / u) / sqrt(u + k)  for the kIn + kOut end samples
// (k = 0 with half weight).  No interpolation stencils, no angular nodes, and a weight that is
// real and closed in form but for the end samples.  The part of a sum that lies far from a
// row's end is a smooth function of rho, so the rows are taken in cells of 64, 32 or less: with
// [ua, ub] a cell's extent in samples, the samples below kc = ua - (ub - ua) (and below the cell's
// end samples) are summed at kPts Chebyshev points of the cell only and interpolated (the nearest
// singularity lies three half widths from the cell's middle: the error falls by 5.8 per point).
//
// The weights' accuracy is that of the end weights while T_q(k / u) / sqrt(u + k) varies slowly
// over the end samples, that is from u of about q^2 / 2 (float32) or q^2 (float64) up
// (sum_first_row); the rows below keep the quadrature in alpha.  Errors against Bessel functions
// (single tones over the band, times 2 pi) at the first row: float32 form 1e-7 at |q| = 12 and 16,
// 2e-8 at 64, float64 form 1e-13 at 8, 2e-14 at 64; at twice that row a tenth.  The far part's
// interpolation adds at most 2e-7 (float32) and 3e-14 (float64): cells are narrowed for |q| beyond
// kSumNarrow, and where rows lie too far apart for that those |q| keep the quadrature.
//
// Kernels (q and -q share their weights; 16 series per sign and block column):
//   rows   end weights w_j of every row
//   fold   G+ and i G- as [|q|][chunk][k][64 columns] (with the ES kernel the grid holds
//          precorrected samples: g(k) is their ES interpolation at the integer offset 0)
//   far    the sums at the cells' points: tiles of 64 points, weights formed 32 samples at a time
//          in shared memory and multiplied by the folded samples in registers (4 x 4 per
//          thread); a sum is split over kSplit samples a block, then added in order
//   near   64 rows: the samples from kc up (real and, at the end samples, imaginary weights
//          formed together), and the interpolation of the far sums as one more short product
// A block column holds 16 series per sign, or 4 where there are no more than 4 (one or two
// MBFs: a column of 16 would mostly multiply zeros).  Bound by the FP32 (FP64) pipe: a weight
// (T_q from the binary power of e^{i alpha}, one reciprocal square root) costs about as much as
// its 64 products.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "cfft_common.cuh"
#include "end_weights.cuh"
#include "es_weights.cuh"

namespace cfft {

namespace {

constexpr int kSR = 64;        // rows (points) of a block's tile
constexpr int kSK = 32;        // samples per step
constexpr int kSThreads = 256;
constexpr int kSPitch = kSR + 4;

// series per sign of a block column (16 or 4), and its columns: both signs, (re, im)
inline int sum_chunk(int series_per_q) { return series_per_q <= 4 ? 4 : 16; }

template <class T>
constexpr int kPts = sizeof(T) == 4 ? 10 : 20;   // Chebyshev points per cell

template <class T>
struct SumShape {
  static constexpr int kIn = EndShape<T>::kIn, kOut = EndShape<T>::kOut, kEnd = kIn + kOut;
};

template <class T>
__device__ __forceinline__ T end_coef(int j, int d, int part) {
  if constexpr (sizeof(T) == 4) return kEndWeightsF[j][d][part];
  else return kEndWeightsD[j][d][part];
}

// extent of a cell, in samples: first row, width, first near sample (0: no far part), and its
// middle as an integer and an offset
template <class T>
struct SumCell {
  double ua, width;
  int kc;
  T o, mid, hh;
};

template <class T>
__device__ __forceinline__ SumCell<T> sum_cell(const SumArgs<T>& a, int cell) {
  const double h = a.d_rho / a.d_s;
  SumCell<T> c;
  c.ua = (double)cell * a.cell_rows * h;
  c.width = (a.cell_rows - 1) * h;
  // a width below the cell, and below every row's end samples
  c.kc = max(0, (int)floor(c.ua - fmax(c.width, (double)EndShape<T>::kIn)));
  const double m = c.ua + 0.5 * c.width, o = rint(m);
  c.o = (T)o;
  c.mid = (T)(m - o);
  c.hh = (T)(0.5 * c.width);
  return c;
}

template <class T>
__device__ __forceinline__ T sum_point(const SumCell<T>& c, int i) {   // offset from c.o
  return c.mid + c.hh * cospi_((T)(2 * i + 1) / (T)(2 * kPts<T>));
}

// T_p(cos) from x = cos alpha, y = sin alpha (p-th power of e^{i alpha}, by squaring)
template <class T>
__device__ __forceinline__ T cheb_in(T x, T y, int p) {
  cpx<T> z = mk(x, y), r = mk((T)1, (T)0);
  for (int e = p; e; e >>= 1) {
    if (e & 1) r = r * z;
    z = z * z;
  }
  return r.re;
}
// T_p outside [-1, 1]: z = x + sqrt(x^2 - 1), (z^p + z^-p) / 2
template <class T>
__device__ __forceinline__ T cheb_out(T z, int p) {
  T r = (T)1, b = z;
  for (int e = p; e; e >>= 1) {
    if (e & 1) r *= b;
    b *= b;
  }
  return (T)0.5 * (r + (T)1 / r);
}

// acc[4 rows][J columns] += x[4] y[J] (J = 4 or 1), 16-byte shared loads
template <class T, int J>
__device__ __forceinline__ void ld_vec(const T* p, T* v) {
  if constexpr (J == 1) {
    v[0] = p[0];
  } else if constexpr (sizeof(T) == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const double2 q0 = reinterpret_cast<const double2*>(p)[0], q1 = reinterpret_cast<const double2*>(p)[1];
    v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
  }
}
template <class T, int J>
__device__ __forceinline__ void fma4(T (&acc)[4][J], const T* x, const T* y) {
  T xv[4], yv[J];
  ld_vec<T, 4>(x, xv);
  ld_vec<T, J>(y, yv);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < J; ++j) acc[i][j] = fma(xv[i], yv[j], acc[i][j]);
}

// ---- end weights of the rows: [end sample][row]
template <class T>
__device__ __forceinline__ void sum_row_weights(const SumArgs<T>& a, int r) {
  if (r >= a.n_rho) return;
  const double u = (double)r * (a.d_rho / a.d_s);
  const T x = (T)(2.0 * (u - floor(u)) - 1.0);
  constexpr int D = EndShape<T>::kDeg;
#pragma unroll
  for (int j = 0; j < SumShape<T>::kEnd; ++j) {
    cpx<T> w = mk(end_coef<T>(j, D, 0), end_coef<T>(j, D, 1));
#pragma unroll
    for (int d = D - 1; d >= 0; --d) w = mk(fma(w.re, x, end_coef<T>(j, d, 0)), fma(w.im, x, end_coef<T>(j, d, 1)));
    a.wrow[(size_t)j * a.n_rho + r] = w;
  }
}

// ---- folded samples of kSK consecutive k of |q| = p, chunk sc
template <class T, int TAPS, int KERN, int kSS>
__device__ __forceinline__ void sum_fold_tile(const SumArgs<T>& a, int k0, int p, int sc) {
  constexpr int HALF = TAPS / 2 - 1;
  constexpr int NW = KERN == 1 ? TAPS : 1;
  constexpr int kSC = 4 * kSS;
  __shared__ T G[2][kSK][kSC + 1];
  const int tid = threadIdx.x;
  T cw[NW];
  if constexpr (KERN == 1) es_weights<TAPS>(0.f, cw);
  else cw[0] = (T)1;
  const int S = a.series_per_q, K = a.grid_half;
  const int qi_pos = a.q_max + p, qi_neg = a.q_max - p;
  const T par = (p & 1) ? (T)-1 : (T)1;
  const int kk = tid & (kSK - 1), k = k0 + kk;
  T s1, c1;   // exp(-i pi k / sigma): the grid is stored demodulated
  sincospi_(-(T)(k & (2 * a.sigma - 1)) / (T)a.sigma, &s1, &c1);
  for (int c = tid / kSK; c < 2 * kSS; c += kSThreads / kSK) {
    const int g = sc * kSS + (c & (kSS - 1));
    cpx<T> vp = mk((T)0, (T)0), vm = vp;
    if (g < S && (c < kSS || p > 0) && k < a.k_used) {
      const cpx<T>* src = a.grid + ((size_t)g * a.n_harm + (c < kSS ? qi_pos : qi_neg)) * (2 * K + 1) + K;
      cpx<T> x = vp, y = vp;
#pragma unroll
      for (int m = 0; m < NW; ++m) {
        const int dk = KERN == 1 ? m - HALF : 0;
        const cpx<T> gp = src[k + dk], gm = src[-k + dk];
        x.re = fma(cw[m], gp.re, x.re);
        x.im = fma(cw[m], gp.im, x.im);
        y.re = fma(cw[m], gm.re, y.re);
        y.im = fma(cw[m], gm.im, y.im);
      }
      // g(k) = x e^{-i pi k / sigma}, (-1)^p g(-k) = +-y e^{+i pi k / sigma}
      const cpx<T> gk = x * mk(c1, s1), gn = par * (y * mk(c1, -s1));
      vp = gk + gn;
      const cpx<T> d = gk - gn;
      vm = mk(-d.im, d.re);
    }
    G[0][kk][2 * c] = vp.re;
    G[0][kk][2 * c + 1] = vp.im;
    G[1][kk][2 * c] = vm.re;
    G[1][kk][2 * c + 1] = vm.im;
  }
  __syncthreads();
  const int n_sc = (S + kSS - 1) / kSS;
  T* dst = a.fold + ((size_t)p * n_sc + sc) * 2 * a.k_pad * kSC;
  for (int e = tid; e < 2 * kSK * kSC; e += kSThreads) {
    const int h = e / (kSK * kSC), r = e / kSC % kSK, c = e % kSC;
    dst[((size_t)h * a.k_pad + k0 + r) * kSC + c] = G[h][r][c];
  }
  __syncthreads();
}

// a step's samples into shared memory: 16-byte asynchronous copies
template <class T, int kSC>
__device__ __forceinline__ void sum_fetch(const T* src, T* dst, int n_k) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  const char* s = reinterpret_cast<const char*>(src);
  for (int e = threadIdx.x; e < n_k * kSC * (int)sizeof(T) / 16; e += kSThreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16u * e), "l"(s + 16 * e) : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
}

template <class T, int kSS>
struct SumSmem {
  T W[2][kSK][kSPitch];
  T G[2][kSK][4 * kSS];
};

// samples the far sums of the points of the tile starting at row0 reach
template <class T>
__device__ __forceinline__ int sum_reach(const SumArgs<T>& a, int row0) {
  const int n_pts = a.n_cells * kPts<T>;
  return sum_cell(a, min(row0 + kSR - 1, n_pts - 1) / kPts<T>).kc;
}

template <class T, int kSS>
__device__ __forceinline__ void sum_far_tile(const SumArgs<T>& a, int row0, int p, int sc, int split,
                                             SumSmem<T, kSS>& sm) {
  constexpr int kSC = 4 * kSS, J = kSC / 16;
  const int n_pts = a.n_cells * kPts<T>;
  const int tid = threadIdx.x;
  const int k_beg = split * a.split, k_end = min(sum_reach(a, row0), k_beg + a.split);
  // cells of rows below |q| = p's first row are not summed
  const int last = min(row0 + kSR - 1, n_pts - 1) / kPts<T>;
  if (k_beg >= k_end || (last + 1) * a.cell_rows <= sum_first_row(a.d_rho / a.d_s, p, sizeof(T) == 8)) return;
  const int wrow = tid & (kSR - 1), kw = tid / kSR;
  const int pt = min(row0 + wrow, n_pts - 1);
  const SumCell<T> c = sum_cell(a, pt / kPts<T>);
  const T off = sum_point(c, pt % kPts<T>);
  const T inv_u = (T)1 / (c.o + off);
  const int ty = tid >> 4, tx = tid & 15;
  T acc[4][J];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < J; ++j) acc[i][j] = (T)0;
  const int S = a.series_per_q, n_sc = (S + kSS - 1) / kSS;
  const T* fold = a.fold + ((size_t)p * n_sc + sc) * 2 * a.k_pad * kSC;
  sum_fetch<T, kSC>(fold + (size_t)k_beg * kSC, &sm.G[0][0][0], kSK);
  for (int k0 = k_beg, buf = 0; k0 < k_end; k0 += kSK, buf ^= 1) {
#pragma unroll
    for (int m = 0; m < kSK / 4; ++m) {
      const int kl = kw + 4 * m, k = k0 + kl;
      T w = (T)0;
      if (k < c.kc) {
        // u - k and u + k from the integer parts: no cancellation
        const T kf = (T)k, d = (c.o - kf) + off, e = (c.o + kf) + off, de = d * e;
        const T ir = rsqrt(de);
        w = cheb_in<T>(kf * inv_u, de * ir * inv_u, p) * ir;
        if (k == 0) w *= (T)0.5;
      }
      sm.W[0][kl][wrow] = w;
    }
    const bool more = k0 + kSK < k_end;
    if (more) sum_fetch<T, kSC>(fold + (size_t)(k0 + kSK) * kSC, &sm.G[buf ^ 1][0][0], kSK);
    if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < kSK; ++k) fma4<T, J>(acc, &sm.W[0][k][4 * ty], &sm.G[buf][k][J * tx]);
    __syncthreads();
  }
  T* out = reinterpret_cast<T*>(a.far) + ((((size_t)split * (a.q_max + 1) + p) * n_sc + sc) * n_pts) * kSC;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = row0 + 4 * ty + i;
    if (row >= n_pts) continue;
#pragma unroll
    for (int j = 0; j < J; ++j) out[(size_t)row * kSC + J * tx + j] = acc[i][j];
  }
}

// the far sums of kSR points: the splits added to the first
template <class T, int kSS>
__device__ __forceinline__ void sum_splits(const SumArgs<T>& a, int row0, int p, int sc) {
  const int n_pts = a.n_cells * kPts<T>, n_sc = (a.series_per_q + kSS - 1) / kSS;
  const int n = (sum_reach(a, row0) + a.split - 1) / a.split;
  const int last = min(row0 + kSR - 1, n_pts - 1) / kPts<T>;
  if (n < 2 || (last + 1) * a.cell_rows <= sum_first_row(a.d_rho / a.d_s, p, sizeof(T) == 8)) return;
  const size_t stride = (size_t)(a.q_max + 1) * n_sc * n_pts * (2 * kSS);
  cpx<T>* f = a.far + (((size_t)p * n_sc + sc) * n_pts + row0) * (2 * kSS);
  const int total = min(kSR, n_pts - row0) * 2 * kSS;
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    cpx<T> v = f[e];
    for (int s = 1; s < n; ++s) v = v + f[s * stride + e];
    f[e] = v;
  }
}

// kSR rows from row0 on: near sums, end samples, far interpolation, stores
template <class T, int kSS>
__device__ __forceinline__ void sum_near_tile(const SumArgs<T>& a, int row0, int p, int sc, SumSmem<T, kSS>& sm) {
  constexpr int kSC = 4 * kSS, J = kSC / 16;
  constexpr int IN = SumShape<T>::kIn, OUT = SumShape<T>::kOut, NE = SumShape<T>::kEnd;
  const int r_min = sum_first_row(a.d_rho / a.d_s, p, sizeof(T) == 8);
  if (row0 + kSR <= r_min || row0 >= a.n_rho) return;
  const int tid = threadIdx.x;
  const double h = a.d_rho / a.d_s;
  const int wrow = tid & (kSR - 1), kw = tid / kSR;
  const int r = min(row0 + wrow, a.n_rho - 1);
  const bool live = r >= r_min;                      // rows below r_min: not formed here
  const double u = (double)r * h, fl = floor(u);
  const int ku = (int)fl;
  const T f = (T)(u - fl);
  const SumCell<T> c = sum_cell(a, r / a.cell_rows);
  const SumCell<T> first = sum_cell(a, row0 / a.cell_rows);
  const int k_beg = first.kc / 4 * 4;
  const int k_end = (int)floor((double)min(row0 + kSR - 1, a.n_rho - 1) * h) + OUT + 1;
  const T kuf = (T)ku;
  const T inv_u = (T)1 / (kuf + f);
  const int ty = tid >> 4, tx = tid & 15;
  T acc[4][J];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < J; ++j) acc[i][j] = (T)0;
  const int S = a.series_per_q, n_sc = (S + kSS - 1) / kSS;
  const T* fold_p = a.fold + ((size_t)p * n_sc + sc) * 2 * a.k_pad * kSC;
  const T* fold_m = fold_p + (size_t)a.k_pad * kSC;
  // weight of sample k for this thread's row (imaginary at the end samples only)
  auto weight = [&](int k) -> cpx<T> {
    const int j = k - (ku + 1 - IN);
    if (!live || k < c.kc || j >= NE) return mk((T)0, (T)0);
    const T kf = (T)k, d = (kuf - kf) + f, e = (kuf + kf) + f;   // u - k, u + k
    if (j < 0) {
      const T de = d * e, ir = rsqrt(de);
      const T w = cheb_in<T>(kf * inv_u, de * ir * inv_u, p) * ir;
      return mk(k == 0 ? (T)0.5 * w : w, (T)0);
    }
    const T root = sqrt(fabs(d) * e) * inv_u;
    const T w = (d >= (T)0 ? cheb_in<T>(kf * inv_u, root, p) : cheb_out<T>(kf * inv_u + root, p)) * rsqrt(e);
    return w * a.wrow[(size_t)j * a.n_rho + r];
  };
  // steps below the tile's first end sample take the real weights alone
  const int b_beg = (int)floor((double)max(row0, r_min) * h) + 1 - IN;
  for (int k0 = k_beg; k0 < k_end; k0 += kSK) {
    const bool end = k0 + kSK > b_beg;
    sum_fetch<T, kSC>(fold_p + (size_t)k0 * kSC, &sm.G[0][0][0], kSK);
    if (end) sum_fetch<T, kSC>(fold_m + (size_t)k0 * kSC, &sm.G[1][0][0], kSK);
#pragma unroll
    for (int m = 0; m < kSK / 4; ++m) {
      const cpx<T> w = weight(k0 + kw + 4 * m);
      sm.W[0][kw + 4 * m][wrow] = w.re;
      if (end) sm.W[1][kw + 4 * m][wrow] = w.im;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int part = 0; part < (end ? 2 : 1); ++part)
#pragma unroll 8
      for (int k = 0; k < kSK; ++k) fma4<T, J>(acc, &sm.W[part][k][4 * ty], &sm.G[part][k][J * tx]);
    __syncthreads();
  }
  // far sums of the tile's cells, interpolated (barycentric weights of the Chebyshev points)
  constexpr int P = kPts<T>;
  const T* far = reinterpret_cast<const T*>(a.far) + (((size_t)p * n_sc + sc) * a.n_cells * P) * kSC;
  const int cell1 = min(row0 + kSR - 1, a.n_rho - 1) / a.cell_rows;
  for (int cell = row0 / a.cell_rows; cell <= cell1; ++cell) {
    if (sum_cell(a, cell).kc == 0 || (cell + 1) * a.cell_rows <= r_min) continue;
    sum_fetch<T, kSC>(far + (size_t)cell * P * kSC, &sm.G[0][0][0], P);
    if (kw == 0) {
      const bool mine = live && r / a.cell_rows == cell;
      const T x = (kuf - c.o) + f;
      T sum = (T)0;
      int at = -1;
#pragma unroll
      for (int i = 0; i < P; ++i) {
        const T dx = x - sum_point(c, i);
        T s1, c1;
        sincospi_((T)(2 * i + 1) / (T)(2 * P), &s1, &c1);
        if (dx == (T)0) at = i;
        const T b = ((i & 1) ? -s1 : s1) / (dx == (T)0 ? (T)1 : dx);
        sm.W[0][i][wrow] = b;
        sum += b;
      }
      const T inv = (T)1 / sum;
#pragma unroll
      for (int i = 0; i < P; ++i)
        sm.W[0][i][wrow] = !mine ? (T)0 : (at >= 0 ? (at == i ? (T)1 : (T)0) : sm.W[0][i][wrow] * inv);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll 5
    for (int k = 0; k < P; ++k) fma4<T, J>(acc, &sm.W[0][k][4 * ty], &sm.G[0][k][J * tx]);
    __syncthreads();
  }
  // stores through shared memory: 64 consecutive rows of a series
  const T norm = (T)(1.0 / (2.0 * 3.14159265358979323846 * 3.14159265358979323846));
  T* tile = &sm.G[0][0][0];                       // [column][kSR]
  static_assert(sizeof(sm.G) >= (size_t)kSC * kSR * sizeof(T), "output tile");
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < J; ++j) tile[(J * tx + j) * kSR + 4 * ty + i] = norm * acc[i][j];
  __syncthreads();
  for (int e = tid; e < 2 * kSS * kSR; e += kSThreads) {
    const int c2 = e / kSR, rr = e % kSR, row = row0 + rr;
    const int g = sc * kSS + (c2 & (kSS - 1));
    if (g >= S || row >= a.n_rho || row < r_min || (c2 >= kSS && p == 0)) continue;
    const int qi = c2 < kSS ? a.q_max + p : a.q_max - p;
    a.table[((size_t)g * a.n_harm + qi) * a.n_rho + row] = mk(tile[(2 * c2) * kSR + rr], tile[(2 * c2 + 1) * kSR + rr]);
  }
}

template <class T>
__global__ void __launch_bounds__(128) sum_rows_kernel(SumArgs<T> a) {
  sum_row_weights<T>(a, blockIdx.x * blockDim.x + threadIdx.x);
}
template <class T, int TAPS, int KERN, int kSS>
__global__ void __launch_bounds__(kSThreads) sum_fold_kernel(SumArgs<T> a) {
  sum_fold_tile<T, TAPS, KERN, kSS>(a, blockIdx.x * kSK, blockIdx.y, blockIdx.z);
}
template <class T, int kSS>
__global__ void __launch_bounds__(kSThreads) sum_far_kernel(SumArgs<T> a, int n_tiles, int n_p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int t = blockIdx.x;   // the largest rho (most splits) first
  sum_far_tile<T, kSS>(a, (n_tiles - 1 - t / n_p) * kSR, t % n_p, blockIdx.y, blockIdx.z,
                  *reinterpret_cast<SumSmem<T, kSS>*>(smem_raw));
}
template <class T, int kSS>
__global__ void __launch_bounds__(256) sum_splits_kernel(SumArgs<T> a) {
  sum_splits<T, kSS>(a, blockIdx.x * kSR, blockIdx.y, blockIdx.z);
}
template <class T, int kSS>
__global__ void __launch_bounds__(kSThreads) sum_near_kernel(SumArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  sum_near_tile<T, kSS>(a, blockIdx.x * kSR, blockIdx.y, blockIdx.z, *reinterpret_cast<SumSmem<T, kSS>*>(smem_raw));
}

// batched forms: maps of (item, first sample | point | row)
template <class T>
__global__ void __launch_bounds__(128) sum_rows_batch_kernel(const SumArgs<T>* items, int first) {
  const SumArgs<T> a = items[first + blockIdx.y];
  if (a.n_cells > 0) sum_row_weights<T>(a, blockIdx.x * blockDim.x + threadIdx.x);
}
template <class T, int TAPS, int KERN, int kSS>
__global__ void __launch_bounds__(kSThreads) sum_fold_batch_kernel(const SumArgs<T>* items, const int2* map) {
  const int2 bm = map[blockIdx.x];
  const SumArgs<T> a = items[bm.x];
  sum_fold_tile<T, TAPS, KERN, kSS>(a, bm.y, blockIdx.y, blockIdx.z);
}
template <class T, int kSS>
__global__ void __launch_bounds__(kSThreads) sum_far_batch_kernel(const SumArgs<T>* items, const int2* map, int n_p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int2 bm = map[blockIdx.x / n_p];
  const SumArgs<T> a = items[bm.x];
  sum_far_tile<T, kSS>(a, bm.y, blockIdx.x % n_p, blockIdx.y, blockIdx.z, *reinterpret_cast<SumSmem<T, kSS>*>(smem_raw));
}
template <class T, int kSS>
__global__ void __launch_bounds__(256) sum_splits_batch_kernel(const SumArgs<T>* items, const int2* map) {
  const int2 bm = map[blockIdx.x];
  const SumArgs<T> a = items[bm.x];
  sum_splits<T, kSS>(a, bm.y, blockIdx.y, blockIdx.z);
}
template <class T, int kSS>
__global__ void __launch_bounds__(kSThreads) sum_near_batch_kernel(const SumArgs<T>* items, const int2* map) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int2 bm = map[blockIdx.x];
  const SumArgs<T> a = items[bm.x];
  sum_near_tile<T, kSS>(a, bm.y, blockIdx.y, blockIdx.z, *reinterpret_cast<SumSmem<T, kSS>*>(smem_raw));
}

template <class T, class F>
cudaError_t by_kernel(int kern, int taps, F f) {
  if constexpr (sizeof(T) == 4) {
    if (kern == 1 && taps == 6) return f(std::integral_constant<int, 6>{}, std::integral_constant<int, 1>{});
    if (kern == 1 && taps == 8) return f(std::integral_constant<int, 8>{}, std::integral_constant<int, 1>{});
  }
  if (kern == 1) return cudaErrorInvalidValue;
  return f(std::integral_constant<int, 16>{}, std::integral_constant<int, 0>{});
}

template <class T, int kSS>
cudaError_t sum_smem_opt_in() {
  const int bytes = (int)sizeof(SumSmem<T, kSS>);
  for (const void* k : {(const void*)sum_far_kernel<T, kSS>, (const void*)sum_near_kernel<T, kSS>,
                        (const void*)sum_far_batch_kernel<T, kSS>, (const void*)sum_near_batch_kernel<T, kSS>}) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <class T, int kSS>
cudaError_t launch_sums(const SumArgs<T>& a, int taps, int kern, int splits, int tiles, cudaStream_t s) {
  cudaError_t e = sum_smem_opt_in<T, kSS>();
  if (e != cudaSuccess) return e;
  const size_t smem = sizeof(SumSmem<T, kSS>);
  const int n_p = a.q_max + 1, n_sc = (a.series_per_q + kSS - 1) / kSS;
  sum_rows_kernel<T><<<(a.n_rho + 31) / 32, 32, 0, s>>>(a);
  e = by_kernel<T>(kern, taps, [&](auto tp, auto kn) {
    sum_fold_kernel<T, decltype(tp)::value, decltype(kn)::value, kSS>
        <<<dim3(a.k_pad / kSK, n_p, n_sc), kSThreads, 0, s>>>(a);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  sum_far_kernel<T, kSS><<<dim3(tiles * n_p, n_sc, splits), kSThreads, smem, s>>>(a, tiles, n_p);
  if (splits > 1) sum_splits_kernel<T, kSS><<<dim3(tiles, n_p, n_sc), 256, 0, s>>>(a);
  sum_near_kernel<T, kSS><<<dim3((a.n_rho + kSR - 1) / kSR, n_p, n_sc), kSThreads, smem, s>>>(a);
  return cudaGetLastError();
}

template <class T, int kSS>
cudaError_t launch_sums_batch(const SumArgs<T>* items, int first, int n_items, int n_rho, const int2* fold_map,
                              int n_fold, const int2* far_map, int n_far, const int2* near_map, int n_near,
                              int max_splits, int q_max, int series_per_q, int taps, int kern, cudaStream_t s) {
  cudaError_t e = sum_smem_opt_in<T, kSS>();
  if (e != cudaSuccess) return e;
  const size_t smem = sizeof(SumSmem<T, kSS>);
  const int n_p = q_max + 1, n_sc = (series_per_q + kSS - 1) / kSS;
  for (int i = 0; i < n_items; i += 32768)
    sum_rows_batch_kernel<T><<<dim3((n_rho + 127) / 128, std::min(32768, n_items - i)), 128, 0, s>>>(items, first + i);
  e = by_kernel<T>(kern, taps, [&](auto tp, auto kn) {
    sum_fold_batch_kernel<T, decltype(tp)::value, decltype(kn)::value, kSS>
        <<<dim3(n_fold, n_p, n_sc), kSThreads, 0, s>>>(items, fold_map);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  sum_far_batch_kernel<T, kSS><<<dim3(n_far * n_p, n_sc, max_splits), kSThreads, smem, s>>>(items, far_map, n_p);
  if (max_splits > 1) sum_splits_batch_kernel<T, kSS><<<dim3(n_far, n_p, n_sc), 256, 0, s>>>(items, far_map);
  sum_near_batch_kernel<T, kSS><<<dim3(n_near, n_p, n_sc), kSThreads, smem, s>>>(items, near_map);
  return cudaGetLastError();
}

}  // namespace

// grid samples beyond ceil(u) that the end samples, and the ES interpolation around them, read
int sum_grid_extra(bool fp64, int taps, int kern) {
  return (fp64 ? SumShape<double>::kOut : SumShape<float>::kOut) + (kern == 1 ? taps / 2 : 0) + 1;
}

bool sum_plan(bool fp64, int n_rho, double d_rho, double d_s, int sigma, int grid_half, int taps, int kern, int q_max,
              int series_per_q, int sms, SumPlan* p) {
  *p = SumPlan{};
  const int out = fp64 ? EndShape<double>::kOut : EndShape<float>::kOut;
  if (sigma != (fp64 ? EndShape<double>::kSigma : EndShape<float>::kSigma)) return false;
  // Lagrange stencils narrower than the precision's target asks for (an option) keep the quadrature
  // that interpolates with them
  if (kern == 0 && taps < (fp64 ? 16 : 12)) return false;
  const double h = d_rho / d_s, top = (n_rho - 1) * h;
  if ((int)std::ceil(top) + sum_grid_extra(fp64, taps, kern) > grid_half) return false;
  if (sum_first_row(h, 0, fp64) >= n_rho) return false;
  // 64 rows to a cell, 32 where those are more than 40 samples wide: the near window (two
  // widths and the end samples) grows with the width, the far points with the number of cells
  p->cell_rows = 63.0 * h > 40.0 ? 32 : 64;
  // narrower for high harmonics, while sum_first_row has the sums serve them
  if (q_max > kSumNarrow && (kSumCellRows - 1) * h <= sum_cell_width(fp64))
    p->cell_rows = std::min(p->cell_rows, 1 + (int)(sum_cell_width(fp64) / h));
  p->cells = (n_rho + p->cell_rows - 1) / p->cell_rows;
  p->k_used = (int)std::floor(top) + out + 1;
  p->k_pad = (p->k_used + 4 + kSK) / kSK * kSK + kSK;   // steps may start at any multiple of 4
  const int pts = fp64 ? kPts<double> : kPts<float>;
  const int ss = sum_chunk(series_per_q);
  p->tiles = (p->cells * pts + kSR - 1) / kSR;
  const size_t blocks = (size_t)(q_max + 1) * ((series_per_q + ss - 1) / ss);
  // a far sum is split over blocks of 64 to 512 samples: about eight blocks per SM (half the
  // (tile, split) pairs lie beyond their tile's reach), at most 16 splits
  p->split = 512;
  while (p->split > 64 && (int64_t)p->tiles * blocks * (p->k_used / p->split + 1) < 16 * sms &&
         p->k_used / (p->split / 2) < 16)
    p->split /= 2;
  // ... and as large as it takes to keep the splits' sums, a sixth of the table each, to 256 MB
  const size_t per_split = blocks * p->cells * pts * 2 * ss;
  while (p->split < p->k_used && (size_t)((p->k_used + p->split - 1) / p->split) * per_split * (fp64 ? 16 : 8) > ((size_t)256 << 20))
    p->split *= 2;
  p->splits = std::max(1, (p->k_used + p->split - 1) / p->split);
  p->fold = blocks * 2 * p->k_pad * 4 * ss;
  p->far = p->splits * per_split;
  p->wrow = (size_t)(fp64 ? SumShape<double>::kEnd : SumShape<float>::kEnd) * n_rho;
  return true;
}

int sum_tile_rows() { return kSR; }
int sum_fold_samples() { return kSK; }

template <class T>
cudaError_t launch_backproject_sum(const SumArgs<T>& a, int taps, int kern, int splits, int tiles, cudaStream_t s) {
  return sum_chunk(a.series_per_q) == 4 ? launch_sums<T, 4>(a, taps, kern, splits, tiles, s)
                                        : launch_sums<T, 16>(a, taps, kern, splits, tiles, s);
}

template <class T>
cudaError_t launch_backproject_sum_batch(const SumArgs<T>* items, int first, int n_items, int n_rho, const int2* fold_map,
                                         int n_fold, const int2* far_map, int n_far, const int2* near_map, int n_near,
                                         int max_splits, int q_max, int series_per_q, int taps, int kern,
                                         cudaStream_t s) {
  auto run = sum_chunk(series_per_q) == 4 ? launch_sums_batch<T, 4> : launch_sums_batch<T, 16>;
  return run(items, first, n_items, n_rho, fold_map, n_fold, far_map, n_far, near_map, n_near, max_splits, q_max,
             series_per_q, taps, kern, s);
}

template cudaError_t launch_backproject_sum<float>(const SumArgs<float>&, int, int, int, int, cudaStream_t);
template cudaError_t launch_backproject_sum<double>(const SumArgs<double>&, int, int, int, int, cudaStream_t);
template cudaError_t launch_backproject_sum_batch<float>(const SumArgs<float>*, int, int, int, const int2*, int,
                                                         const int2*, int, const int2*, int, int, int, int, int, int,
                                                         cudaStream_t);
template cudaError_t launch_backproject_sum_batch<double>(const SumArgs<double>*, int, int, int, const int2*, int,
                                                          const int2*, int, const int2*, int, int, int, int, int, int,
                                                          cudaStream_t);

}  // namespace cfft
