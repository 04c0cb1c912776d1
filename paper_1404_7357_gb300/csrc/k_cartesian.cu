// The paper's own 2-D Cartesian C-FFT (Section III-B-2 and III-B-3, Eq. 21-24,
// Appendix I), as a second tabulation beside the harmonic one.
//
// On the real grid kx, ky = -k_m + n dk (n < N, dk = 2 k_m / N; Appendix I) the
// contour of Eq. 8 enters through the extension k (1 + i gamma), gamma =
// beta_I(beta_R) / beta_R (Eq. 20): per sample the kernel of Eq. 10 at that
// complex wavevector times the Jacobian (1 + i d beta_I / d beta_R)(1 + i gamma)
// gives I_M (Eq. 21); samples outside |k| <= k_m (the polar integral's limit)
// are zero.  The contour factor exp(gamma k.Delta) is expanded in Taylor
// monomials (Eq. 22): Z' = sum_{a, b} dx^a dy^b / (a! b!) F_ab with F_ab the 2-D
// Fourier sum of (gamma kx)^a (gamma ky)^b I_M (Eq. 23-24).  Each F_ab is one
// FFT2: the N x N samples, times (-1)^(n1 + n2) (Appendix I), sit in the middle
// of a 2N x 2N zero grid (the Whittaker-Shannon refinement that halves the
// table's step), and the output is multiplied by (-1)^(k1 + k2) dk^2 / (4 pi^2)
// on the lattice dx = -x_m + k1 pi / (2 k_m).
//
// Kernels: the spectrum (Green's function in float64; MBF spectra at the complex
// wavevector); then the monomials factored by direction,
//   Z' = sum_a (H dx)^a / a! F_x[ sum_b (H dy)^b / b! F_y[ (gamma kx/H)^a (gamma ky/H)^b I_M ] ],
// since (H dy)^b does not depend on kx: per power a one launch of row transforms, each of
// which sums its (order - a + 1) powers b in registers, and one launch of column
// transforms that adds into the table.  Against one FFT2 per monomial this runs order + 1
// column transforms instead of (order + 1)(order + 2) / 2, row transforms over the N
// sampled rows only (the padding rows are zero), and no transposes, padded inputs or
// per-monomial passes over the table.  The transforms are radix-4 Stockham passes in
// shared memory, p / 4 threads per line and several lines per block; the two of a line's
// four quarters that the centred zero padding leaves empty are never read.  Measured
// (GB300, N 128, 16 pairs, order 6, float32): transforms and accumulation 10.6 ms ->
// 0.29 ms (the passes' barriers bound them), tabulation and a 200-element fill 11.1 -> 0.59 ms.  The fill interpolates the table with three-point Lagrange stencils in x and y.
#include <algorithm>
#include <cmath>

#include "cfft_common.cuh"
#include "green_ext.cuh"
#include "shape_factor.cuh"

namespace cfft {

namespace {

constexpr double kEta0c = 376.730313668;   // free-space wave impedance, ohm
constexpr int kCartMaxM = 8;

// grounded-slab Green's function G = P I - R k k^T at the complex radial wavenumber
// beta_c (the TE/TM denominators and branches as in the contour kernel); returns P and
// R beta_c^2
__device__ void slab_green(cpx<double> bc, double eps_r, double hs, double k0, cpx<double>* p,
                           cpx<double>* rb2) {
  const cpx<double> b2 = bc * bc;
  const double k02 = k0 * k0;
  const cpx<double> k1 = csqrt_(mk(eps_r * k02 - b2.re, -b2.im));
  cpx<double> arg2 = mk(b2.re - k02, b2.im);
  if (arg2.im == 0.0) arg2.im = 0.0;   // +0: real beta < k0 gives k2 > 0 (outgoing)
  const cpx<double> r2 = csqrt_(arg2);
  const cpx<double> k2 = mk(r2.im, -r2.re);   // -j sqrt(.): Im k2 <= 0
  cpx<double> sn, cs;
  csincos(mk(k1.re * hs, k1.im * hs), &sn, &cs);
  const cpx<double> j1 = mk(0.0, 1.0);
  const cpx<double> te = k1 * cs + j1 * (k2 * sn);
  const cpx<double> tm = eps_r * (k2 * cs) + j1 * (k1 * sn);
  const cpx<double> cfac = cdiv(mk(0.0, -kEta0c / k0) * sn, te * tm);
  *p = cfac * ((eps_r * k02) * (k2 * cs) + j1 * (k02 * (k1 * sn)));
  *rb2 = cfac * (k2 * cs + j1 * (k1 * sn)) * b2;
}

// I_M (times the Appendix I sign) of every MBF pair at every sample, and gamma kx, gamma ky;
// M: the padded MBF count (the columns of Q), so that the spectra stay in registers
template <class T, int M>
__global__ void __launch_bounds__(64) cart_spectrum_kernel(CartArgs<T> a, cpx<T>* im, T* gx, T* gy) {
  const int64_t nn = (int64_t)a.n * a.n;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nn) return;
  const int n1 = (int)(e / a.n), n2 = (int)(e % a.n);
  const int pairs = a.n_mbf * a.n_mbf;
  const double kx = -a.k_max + n1 * a.dk, ky = -a.k_max + n2 * a.dk;
  const double br = hypot(kx, ky);
  if (br > a.k_max) {
    for (int pr = 0; pr < pairs; ++pr) im[pr * nn + e] = mk((T)0, (T)0);
    gx[e] = (T)0;
    gy[e] = (T)0;
    return;
  }
  double bi = 0.0, slope = 0.0;
  if (br < a.beta_p) {
    const double ip2 = 1.0 / (a.beta_p * a.beta_p);
    bi = 4.0 * a.height * br * (a.beta_p - br) * ip2;
    slope = 4.0 * a.height * (a.beta_p - 2.0 * br) * ip2;
  }
  const double gamma = br > 0.0 ? bi / br : 4.0 * a.height / a.beta_p;
  // gamma k / H: at most beta_I / H <= 1 (H moves to the spatial factor, as (H dx)^a)
  const double ih = a.height > 0.0 ? 1.0 / a.height : 0.0;
  gx[e] = (T)(gamma * kx * ih);
  gy[e] = (T)(gamma * ky * ih);
  cpx<double> p, rb2;
  slab_green(mk(br, bi), a.eps_r, a.hs, a.k0, &p, &rb2);
  if (a.extract) {
    const GreenExt ge = ext_green(mk(br, bi), a.eps_eff, 0.0, a.hs, a.k0, false);
    p = p - ge.p;
    rb2 = rb2 - ge.rb2;
  }
  const double ux = br > 0.0 ? kx / br : 1.0, uy = br > 0.0 ? ky / br : 0.0;
  // MBF spectra at k_c = k (1 + i gamma): both sides, x and y components
  const cpx<T> kcx = mk((T)kx, (T)(gamma * kx)), kcy = mk((T)ky, (T)(gamma * ky));
  cpx<T> mt[2][M], mb[2][M];
#pragma unroll
  for (int d = 0; d < 2; ++d)
#pragma unroll
    for (int m = 0; m < M; ++m) {
      mt[d][m] = mk((T)0, (T)0);
      mb[d][m] = mk((T)0, (T)0);
    }
  for (int c = 0; c < a.n_shape; ++c) {
    const ShapeClass sc = a.shapes[c];
    cpx<T> acct[M], accb[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
      acct[m] = mk((T)0, (T)0);
      accb[m] = mk((T)0, (T)0);
    }
    for (int i = sc.begin; i < sc.end; ++i) {
      const T xi = a.bx[i], yi = a.by[i];
      const T theta = kcx.re * xi + kcy.re * yi, psi = kcx.im * xi + kcy.im * yi;
      T sn, cs;
      sincos_(theta, &sn, &cs);
      const T ex = exp_(psi), iex = (T)1 / ex;
      const cpx<T> ph = mk(cs * ex, -sn * ex);    // exp(-i k_c.r)
      const cpx<T> pb = mk(cs * iex, sn * iex);   // exp(+i k_c.r)
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const cpx<T> qv = a.q[(size_t)i * M + m];
        cmac_conj(acct[m], qv, ph);
        cmac(accb[m], qv, pb);
      }
    }
    const cpx<T> sf = shape_factor<T>(sc, kcx, kcy);
#pragma unroll
    for (int m = 0; m < M; ++m) {
      if (sc.dir == 0) {
        mt[0][m] = mt[0][m] + sf * acct[m];
        mb[0][m] = mb[0][m] + sf * accb[m];
      } else {
        mt[1][m] = mt[1][m] + sf * acct[m];
        mb[1][m] = mb[1][m] + sf * accb[m];
      }
    }
  }
  // Jacobian (1 + i slope)(1 + i gamma) and the Appendix I input sign (-1)^(n1 + n2)
  cpx<double> jac = mk(1.0, slope) * mk(1.0, gamma);
  if ((n1 + n2) & 1) jac = mk(-jac.re, -jac.im);
#pragma unroll
  for (int ia = 0; ia < M; ++ia)
#pragma unroll
    for (int ib = 0; ib < M; ++ib) {
      if (ia >= a.n_mbf || ib >= a.n_mbf) continue;
      const cpx<double> tx = ccast<double>(mt[0][ia]), ty = ccast<double>(mt[1][ia]);
      const cpx<double> bx = ccast<double>(mb[0][ib]), by = ccast<double>(mb[1][ib]);
      const cpx<double> dot = tx * bx + ty * by;
      const cpx<double> ut = ux * tx + uy * ty, ub = ux * bx + uy * by;
      const cpx<double> h = p * dot - rb2 * (ut * ub);
      im[(ia * a.n_mbf + ib) * nn + e] = ccast<T>(jac * h);
    }
}

// ---- line transforms (exp(-2 pi i n k / p)), p = 2 n a power of two, p / 4 threads per line.
// A line's buffer is padded by one entry in 16 (the strided writes of the first passes).
__device__ __forceinline__ int lidx(int e) { return e + (e >> 4); }

template <class T>
__device__ __forceinline__ void line_twiddles(cpx<T>* tw, int p) {
  for (int t = threadIdx.x; t < p; t += blockDim.x) {
    T sv, cv;
    sincospi_((T)(-2.0 * (double)t / (double)p), &sv, &cv);
    tw[t] = mk(cv, sv);
  }
}

// One transform of every line of the block.  The input sits in the middle half of the line
// (the N samples of the padded 2N grid): thread i brings x1 = sample i (entry i + p/4) and
// x2 = sample i + p/4 (entry i + p/2); the first and last quarters are zero.  Natural order
// in `buf` on return (after a barrier); the caller synchronises before the next call.
template <class T>
__device__ __forceinline__ void line_fft(cpx<T>* buf, const cpx<T>* tw, int p, int i, cpx<T> x1, cpx<T> x2) {
  const int q = p >> 2;
  {  // span 1: (0, x1, x2, 0)
    const cpx<T> mid = mk(x1.im, -x1.re);   // -i x1
    buf[lidx(4 * i)] = x2 + x1;
    buf[lidx(4 * i + 1)] = mid - x2;
    buf[lidx(4 * i + 2)] = x2 - x1;
    buf[lidx(4 * i + 3)] = mk((T)0, (T)0) - x2 - mid;
  }
  __syncthreads();
  int sp = 4;
  for (; 4 * sp <= p; sp *= 4) {
    const int k = i & (sp - 1), st = q / sp;   // p / (4 sp)
    cpx<T> v0 = buf[lidx(i)], v1 = buf[lidx(i + q)] * tw[k * st], v2 = buf[lidx(i + 2 * q)] * tw[2 * k * st],
           v3 = buf[lidx(i + 3 * q)] * tw[3 * k * st];
    __syncthreads();
    const cpx<T> s02 = v0 + v2, d02 = v0 - v2, s13 = v1 + v3, d13 = v1 - v3;
    const cpx<T> mid = mk(d13.im, -d13.re);
    const int j = (i - k) * 4 + k;
    buf[lidx(j)] = s02 + s13;
    buf[lidx(j + sp)] = d02 + mid;
    buf[lidx(j + 2 * sp)] = s02 - s13;
    buf[lidx(j + 3 * sp)] = d02 - mid;
    __syncthreads();
  }
  if (sp < p) {   // p an odd power of two: a last radix-2 pass, span p / 2, two butterflies per thread
    const int h = p >> 1;
    const cpx<T> a0 = buf[lidx(i)], a1 = buf[lidx(i + h)] * tw[i];
    const cpx<T> b0 = buf[lidx(i + q)], b1 = buf[lidx(i + q + h)] * tw[i + q];
    __syncthreads();
    buf[lidx(i)] = a0 + a1;
    buf[lidx(i + h)] = a0 - a1;
    buf[lidx(i + q)] = b0 + b1;
    buf[lidx(i + q + h)] = b0 - b1;
    __syncthreads();
  }
}

// Row transforms of power a: out[pair][n1][k2] = sum_b (H y(k2))^b / b! F_y[(gx)^a (gy)^b I_M],
// b = 0 .. nb - 1; one line per (pair, sampled row n1)
template <class T>
__global__ void __launch_bounds__(1024) cart_row_kernel(const cpx<T>* im, const T* gx, const T* gy, int n, int pa, int nb, int n_lines,
                                double hx0, double hstep, cpx<T>* out) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int p = 2 * n, tpl = p >> 2;
  cpx<T>* tw = reinterpret_cast<cpx<T>*>(sm);
  const int ll = threadIdx.x / tpl, i = threadIdx.x - ll * tpl;
  cpx<T>* buf = tw + p + (size_t)ll * (p + p / 16);
  const int line = blockIdx.x * (blockDim.x / tpl) + ll;
  line_twiddles(tw, p);
  cpx<T> z[2];
  T g[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    z[u] = mk((T)0, (T)0);
    g[u] = (T)0;
    if (line < n_lines) {
      const int n2 = i + u * tpl;
      const int64_t s = (int64_t)(line % n) * n + n2;
      z[u] = im[(int64_t)line * n + n2];
      const T x = gx[s];
      for (int t = 0; t < pa; ++t) z[u] = x * z[u];
      g[u] = gy[s];
    }
  }
  cpx<T> acc[4];
  T cf[4], hy[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    acc[u] = mk((T)0, (T)0);
    cf[u] = (T)1;
    hy[u] = (T)(hx0 + (i + u * tpl) * hstep);
  }
  __syncthreads();
  for (int b = 0; b < nb; ++b) {
    line_fft(buf, tw, p, i, z[0], z[1]);
    const T inv = (T)1 / (T)(b + 1);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      acc[u] = acc[u] + cf[u] * buf[lidx(i + u * tpl)];
      cf[u] *= hy[u] * inv;
    }
    z[0] = g[0] * z[0];
    z[1] = g[1] * z[1];
    __syncthreads();
  }
  if (line < n_lines)
#pragma unroll
    for (int u = 0; u < 4; ++u) out[(int64_t)line * p + i + u * tpl] = acc[u];
}

// Column transforms of power a, added into the table: table[pair][k1][k2] (+)= (-1)^(k1 + k2)
// K' (H x(k1))^a / a! F_x[in[pair][.][k2]]; a block takes consecutive columns k2
template <class T>
__global__ void __launch_bounds__(1024) cart_column_kernel(const cpx<T>* in, int n, int pa, double hx0, double hstep, double scale,
                                   cpx<T>* table) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int p = 2 * n, tpl = p >> 2, cols = blockDim.x / tpl;
  cpx<T>* tw = reinterpret_cast<cpx<T>*>(sm);
  line_twiddles(tw, p);
  // consecutive threads take consecutive columns (their global accesses are one segment)
  const int ll = threadIdx.x % cols, i = threadIdx.x / cols;
  cpx<T>* buf = tw + p + (size_t)ll * (p + p / 16);
  const int k2 = blockIdx.x * cols + ll;   // cols divides p
  const cpx<T>* src = in + (int64_t)blockIdx.y * n * p + k2;
  const cpx<T> x1 = src[(int64_t)i * p], x2 = src[(int64_t)(i + tpl) * p];
  __syncthreads();
  line_fft(buf, tw, p, i, x1, x2);
  cpx<T>* dst = table + (int64_t)blockIdx.y * p * p + k2;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int k1 = i + u * tpl;
    const T x = (T)(hx0 + k1 * hstep);
    T c = (T)(((k1 + k2) & 1) ? -scale : scale);
    for (int t = 1; t <= pa; ++t) c *= x / (T)t;
    const cpx<T> v = c * buf[lidx(k1)];
    cpx<T>& z = dst[(int64_t)k1 * p];
    z = pa == 0 ? v : z + v;
  }
}

// reduced matrix by three-point Lagrange interpolation in the refined table: a block forms the
// float64 stencils of kFillPairs element pairs once (one thread each), then all its threads
// take the pairs' M^2 entries.  Bound by the float64 pipe (27 operations an entry); 200
// elements, M 4: 45 us, with one thread per pair 101 us.  err bit 1 when a pair lies outside the valid region
constexpr int kFillPairs = 64;

template <class T, class TO>
__global__ void __launch_bounds__(256) cart_fill_kernel(const cpx<T>* table, int p, int m, double x0, double step,
                                                        double rho_max, int n_el, const double* pos, cpx<TO>* z,
                                                        int64_t ld, int* err) {
  __shared__ double w[kFillPairs][9];
  __shared__ int64_t at[kFillPairs];     // table entry of the stencil's first node, -1 outside
  __shared__ int64_t dst[kFillPairs];    // the pair's first matrix entry
  const int mm = m * m;
  const int64_t total = (int64_t)n_el * n_el;
  for (int64_t e0 = (int64_t)blockIdx.x * kFillPairs; e0 < total; e0 += (int64_t)gridDim.x * kFillPairs) {
    const int np = (int)min((int64_t)kFillPairs, total - e0);
    if ((int)threadIdx.x < np) {
      const int64_t e = e0 + threadIdx.x;
      const int i = (int)(e / n_el), j = (int)(e % n_el);
      const double dx = pos[2 * i] - pos[2 * j], dy = pos[2 * i + 1] - pos[2 * j + 1];
      const double u = (dx - x0) / step, v = (dy - x0) / step;
      const int i0 = (int)floor(u + 0.5), j0 = (int)floor(v + 0.5);
      const bool ok = hypot(dx, dy) <= rho_max * (1.0 + 1e-12) && i0 >= 1 && i0 <= p - 2 && j0 >= 1 && j0 <= p - 2;
      if (!ok) atomicOr(err, 1);
      const double fu = u - i0, fv = v - j0;
      const double wu[3] = {0.5 * fu * (fu - 1.0), 1.0 - fu * fu, 0.5 * fu * (fu + 1.0)};
      const double wv[3] = {0.5 * fv * (fv - 1.0), 1.0 - fv * fv, 0.5 * fv * (fv + 1.0)};
#pragma unroll
      for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int r = 0; r < 3; ++r) w[threadIdx.x][3 * s + r] = wu[s] * wv[r];
      at[threadIdx.x] = ok ? (int64_t)(i0 - 1) * p + (j0 - 1) : -1;
      dst[threadIdx.x] = (int64_t)i * m * ld + (int64_t)j * m;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < np * mm; t += blockDim.x) {
      const int q = t / mm, ab = t - q * mm, a = ab / m, b = ab - a * m;
      cpx<double> acc = mk(0.0, 0.0);
      if (at[q] >= 0) {
        const cpx<T>* tp = table + (int64_t)ab * p * p + at[q];
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const cpx<T> v = tp[(int64_t)s * p + r];
            acc.re = fma(w[q][3 * s + r], (double)v.re, acc.re);
            acc.im = fma(w[q][3 * s + r], (double)v.im, acc.im);
          }
      }
      z[dst[q] + (int64_t)a * ld + b] = ccast<TO>(acc);
    }
    __syncthreads();
  }
}

}  // namespace

template <class T>
cudaError_t cartesian_tabulate(const CartArgs<T>& a, int order, cpx<T>* table, cpx<T>* work, cpx<T>* im, T* gx,
                               T* gy, cudaStream_t s) {
  if (a.n < 2 || (a.n & 1) || a.n_mbf < 1 || a.n_mbf > kCartMaxM) return cudaErrorInvalidValue;
  const int p = 2 * a.n;
  if (p & (p - 1) || p < 16 || p > 4096) return cudaErrorInvalidValue;
  const int pairs = a.n_mbf * a.n_mbf;
  const int64_t nn = (int64_t)a.n * a.n;
  cudaError_t e;
  const unsigned sblocks = (unsigned)((nn + 63) / 64);
  switch (a.q_stride) {
    case 1: cart_spectrum_kernel<T, 1><<<sblocks, 64, 0, s>>>(a, im, gx, gy); break;
    case 2: cart_spectrum_kernel<T, 2><<<sblocks, 64, 0, s>>>(a, im, gx, gy); break;
    case 4: cart_spectrum_kernel<T, 4><<<sblocks, 64, 0, s>>>(a, im, gx, gy); break;
    case 8: cart_spectrum_kernel<T, 8><<<sblocks, 64, 0, s>>>(a, im, gx, gy); break;
    default: return cudaErrorInvalidValue;
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // lines per block: about 128 threads for the rows; four columns (one 32-byte segment in
  // float32, two in float64) where 1024 threads allow
  const int tpl = p / 4;
  const int rows = std::max(1, 128 / tpl), cols = std::max(1, std::min(std::min(4, p), 1024 / tpl));
  const size_t line = (size_t)(p + p / 16) * sizeof(cpx<T>), twb = (size_t)p * sizeof(cpx<T>);
  const size_t rsmem = twb + rows * line, csmem = twb + cols * line;
  if ((e = cudaFuncSetAttribute(cart_row_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsmem)) !=
          cudaSuccess ||
      (e = cudaFuncSetAttribute(cart_column_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csmem)) !=
          cudaSuccess)
    return e;
  const double step = 3.14159265358979323846 / (2.0 * a.k_max);
  const double x0 = -(double)a.n * 3.14159265358979323846 / (2.0 * a.k_max);
  const double kprime = a.dk * a.dk / (4.0 * 3.14159265358979323846 * 3.14159265358979323846);
  const int n_lines = pairs * a.n;
  for (int pa = 0; pa <= order; ++pa) {
    cart_row_kernel<T><<<(n_lines + rows - 1) / rows, rows * tpl, rsmem, s>>>(
        im, gx, gy, a.n, pa, order - pa + 1, n_lines, a.height * x0, a.height * step, work);
    cart_column_kernel<T><<<dim3(p / cols, pairs), cols * tpl, csmem, s>>>(work, a.n, pa, a.height * x0,
                                                                          a.height * step, kprime, table);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <class T, class TO>
cudaError_t cartesian_fill(const cpx<T>* table, int p, int m, double x0, double step, double rho_max, int n_el,
                           const double* pos, void* z, int64_t ld, int* err, cudaStream_t s) {
  const int64_t total = (int64_t)n_el * n_el;
  const int blocks = (int)std::max<int64_t>(
      1, std::min<int64_t>((total + kFillPairs - 1) / kFillPairs, (int64_t)current_sm_count() * 16));
  cart_fill_kernel<T, TO><<<blocks, 256, 0, s>>>(table, p, m, x0, step, rho_max, n_el, pos,
                                                 reinterpret_cast<cpx<TO>*>(z), ld, err);
  return cudaGetLastError();
}

template cudaError_t cartesian_tabulate<float>(const CartArgs<float>&, int, cpx<float>*, cpx<float>*, cpx<float>*,
                                               float*, float*, cudaStream_t);
template cudaError_t cartesian_tabulate<double>(const CartArgs<double>&, int, cpx<double>*, cpx<double>*,
                                                cpx<double>*, double*, double*, cudaStream_t);
template cudaError_t cartesian_fill<float, float>(const cpx<float>*, int, int, double, double, double, int,
                                                  const double*, void*, int64_t, int*, cudaStream_t);
template cudaError_t cartesian_fill<float, double>(const cpx<float>*, int, int, double, double, double, int,
                                                   const double*, void*, int64_t, int*, cudaStream_t);
template cudaError_t cartesian_fill<double, double>(const cpx<double>*, int, int, double, double, double, int,
                                                    const double*, void*, int64_t, int*, cudaStream_t);
template cudaError_t cartesian_fill<double, float>(const cpx<double>*, int, int, double, double, double, int,
                                                   const double*, void*, int64_t, int*, cudaStream_t);

}  // namespace cfft
