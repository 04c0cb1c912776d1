// From the element's spectra to the transform grid, without evaluating the spectra at
// every contour node and without one FFT per term of the contour factor's series.
//
// 1. Spectral tables.  With G = P I - R k k^T the kernel of Eq. 10 is, per harmonic,
//      H_ab,q(beta) = P(beta) D_ab,q(beta) - R(beta) beta^2 E_ab,q(beta),
//    D, E = the azimuthal harmonics of M_a . Mbar_b and of (u.M_a)(u.Mbar_b), u = k / beta.
//    Only P and R carry the substrate (poles, branch points); D and E are entire functions
//    of beta of exponential type tau = 2 (element radius), because the element's currents
//    have compact support.  They are sampled on a uniform real grid of step pi / (tau os)
//    (os = kSpecOver times denser than their Nyquist step; a few samples beyond both ends:
//    D and E continue through beta = 0 and beta_max) and interpolated at every contour
//    node, complex ones included, with Lagrange stencils.  An entire function of type tau
//    interpolated by w central taps has the error |prod (x - t)| / w! (pi / os)^w: on the real
//    axis below 1e-9 of the table for w = 8, os = 8 (float32), 2e-15 for w = 16, os = 8
//    (float64), measured on the 200-rooftop patch.  Off the axis that product grows, and so do
//    the weights, which carry the table's rounding (sum |weight| of 8 taps: 50 two steps off
//    the axis, 12,000 six steps off), so contours rising more than kSpecRise steps keep the
//    spectra at every node (spectral_tables_serve).  The paper tabulates the MBFs' Fourier
//    transforms before its FFTs in the same spirit (Table II, "FT tabulation").
// 2. Gridding.  The transform in beta, g_q(s_k) = sum_j Y_j exp(-i beta_c,j s_k), is wanted
//    on |k| <= K only, a small part of the period 2 pi / step that the contour's nodes
//    resolve.  The nodes are spread onto a coarser grid in beta (spacing 2 pi / (M ds),
//    M >= 2 (2K + 1) a power of two) with the Gaussian exp(-a z^2) (fast Gaussian gridding:
//    Greengard & Lee, SIAM Rev. 46, 2004), one FFT of length M follows, and every output is
//    divided by the Gaussian's transform.  The Gaussian is entire, so a node at complex
//    u = x + i y (y = beta_I in grid units) is spread with the complex weights
//    exp(-a (x - m + i y)^2): the Poisson sum then carries exp(-i u theta) itself, contour
//    factor exp(beta_I s) included, and no series of it is needed.  With theta_c = 2 pi K / M
//    the aliasing error is exp(-((2 pi - theta_c)^2 - theta_c^2) / 4a + y (2 pi - theta_c))
//    and the truncation error exp(-a hw^2) at half width hw: both are held to
//    exp(-17) in float32 (4e-8) and exp(-37) in float64 (1e-16) by the choice of a and hw
//    (float32 on the full-size patch: hw = 8; float64: 16 .. 18).  One FFT then stands for
//    the 8 (float32) or 14 (float64) terms of the contour factor's series, and it is as long
//    as the wanted outputs need, not as the contour's nodes do.
//
// Measured (GB300, before -> now, same table error): the 16-pair patch table (n 16384, 8192 rho
// points, float32) integrand 1247 -> 126 us (tables 77, interpolation 49; one serial chain on 72
// blocks and float32 issue bound them), transform 1170 -> 157 us (spreading 65: shared-memory
// bandwidth, 16 bytes per node, tap and pair of series; FFT 75: one 512-thread CTA per SM; spreading
// weights 17); float64 (n 4096) integrand 19.5 -> 0.82 ms (tables 0.37, interpolation 0.46),
// transform 24.4 -> 1.13 ms (FP64 pipe).
#include <algorithm>
#include <cmath>

#include "cfft_common.cuh"

namespace cfft {

namespace {

constexpr int kInterpThreads = 128;

// Lagrange weights of the nodes 0..W-1 at x, real or complex, from prefix and suffix products
template <class V, int W, class Sub>
__device__ __forceinline__ void lagrange_weights(V* wt, V one, Sub sub) {
  V pre = one;
#pragma unroll
  for (int t = 0; t < W; ++t) {
    wt[t] = pre;
    pre = pre * sub(t);
  }
  V suf = one;
#pragma unroll
  for (int t = W - 1; t >= 0; --t) {
    wt[t] = wt[t] * suf;
    suf = suf * sub(t);
  }
}

template <int W>
__device__ __forceinline__ double lagrange_den(int t) {   // 1 / prod_{j != t} (t - j)
  double d = 1.0;
#pragma unroll
  for (int j = 0; j < W; ++j)
    if (j != t) d *= (double)(t - j);
  return 1.0 / d;
}

// nodes [0, nc) carry (P, R beta^2) = (1, 0) and give D, nodes [nc, 2 nc) carry (0, -1) and
// give E: the integrand kernels evaluate both tables in one launch
__global__ void spectral_nodes_kernel(int nc, double beta0, double d, double2* beta, double2* bw, double2* gp,
                                      double2* gr) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * nc) return;
  const int half = i >= nc;
  beta[i] = make_double2(beta0 + (i - half * nc) * d, 0.0);
  bw[i] = make_double2(1.0, 0.0);
  gp[i] = make_double2(half ? 0.0 : 1.0, 0.0);
  gr[i] = make_double2(half ? -1.0 : 0.0, 0.0);
}

// Y = bw (P D - R beta^2 E) for R consecutive nodes per thread and the series [s0, s1).  All
// nodes of a thread use the stencil of their middle one, so a loaded table entry serves R
// nodes; CPLX: at least one node of the warp lies off the real axis.
template <class T, int W, int R, bool CPLX>
__device__ __forceinline__ void interp_series(const SpecInterpArgs<T>& a, int j, int c0, const double2* x, int s0,
                                              int s1) {
  cpx<T> w[R][CPLX ? W : 1];
  T wr[R][CPLX ? 1 : W];
  cpx<T> pb[R], rb[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const T xr = (T)(x[r].x - (double)c0), xi = (T)x[r].y;
    if constexpr (CPLX) {
      lagrange_weights<cpx<T>, W>(w[r], mk((T)1, (T)0), [&](int t) { return mk(xr - (T)t, xi); });
#pragma unroll
      for (int t = 0; t < W; ++t) w[r][t] = (T)lagrange_den<W>(t) * w[r][t];
    } else {
      lagrange_weights<T, W>(wr[r], (T)1, [&](int t) { return xr - (T)t; });
#pragma unroll
      for (int t = 0; t < W; ++t) wr[r][t] *= (T)lagrange_den<W>(t);
    }
    pb[r] = rb[r] = mk((T)0, (T)0);
    if (j + r < a.n) {
      const double2 b = a.bw[j + r], p = a.green_p[j + r], q = a.green_r[j + r];
      pb[r] = mk((T)(b.x * p.x - b.y * p.y), (T)(b.x * p.y + b.y * p.x));
      rb[r] = mk((T)(b.x * q.x - b.y * q.y), (T)(b.x * q.y + b.y * q.x));
    }
  }
  for (int s = s0; s < s1; ++s) {
    const cpx<T>* d = a.tab + (size_t)s * 2 * a.nc + c0;
    const cpx<T>* e = d + a.nc;
    cpx<T> sd[R], se[R];
#pragma unroll
    for (int r = 0; r < R; ++r) sd[r] = se[r] = mk((T)0, (T)0);
#pragma unroll
    for (int t = 0; t < W; ++t) {
      const cpx<T> dv = d[t], ev = e[t];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (CPLX) {
          cmac(sd[r], w[r][t], dv);
          cmac(se[r], w[r][t], ev);
        } else {
          sd[r].re = fma(wr[r][t], dv.re, sd[r].re);
          sd[r].im = fma(wr[r][t], dv.im, sd[r].im);
          se[r].re = fma(wr[r][t], ev.re, se[r].re);
          se[r].im = fma(wr[r][t], ev.im, se[r].im);
        }
      }
    }
    cpx<T>* y = a.y + (size_t)s * a.n + j;
    if constexpr (sizeof(T) == 4 && R == 2) {
      // n is a multiple of 32 and j even: both nodes are in range or neither, 16-byte aligned
      if (j < a.n) {
        const cpx<T> y0 = pb[0] * sd[0] - rb[0] * se[0], y1 = pb[1] * sd[1] - rb[1] * se[1];
        *reinterpret_cast<float4*>(y) = make_float4(y0.re, y0.im, y1.re, y1.im);
      }
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (j + r < a.n) y[r] = pb[r] * sd[r] - rb[r] * se[r];
    }
  }
}

template <class T>
struct InterpShape {
  static constexpr int W = sizeof(T) == 4 ? 8 : 16;
  static constexpr int R = sizeof(T) == 4 ? 2 : 1;
  static constexpr int kNodes = kInterpThreads * R;   // nodes of a block
};

template <class T>
__device__ __forceinline__ void interp_tile(const SpecInterpArgs<T>& a, int j0, int s0, int s1) {
  constexpr int W = InterpShape<T>::W, R = InterpShape<T>::R;
  const int j = j0 + R * (int)threadIdx.x;
  double2 x[R];
  bool off_axis = false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const double2 b = a.beta_c[min(j + r, a.n - 1)];
    x[r] = make_double2((b.x - a.beta0) * a.inv_d, b.y * a.inv_d);
    off_axis = off_axis || b.y != 0.0;
  }
  const int c0 = max(0, min((int)floor(x[R / 2].x) - W / 2 + 1, a.nc - W));
  if (__any_sync(0xffffffffu, off_axis)) interp_series<T, W, R, true>(a, j, c0, x, s0, s1);
  else interp_series<T, W, R, false>(a, j, c0, x, s0, s1);
}

template <class T>
__global__ void __launch_bounds__(kInterpThreads) spectral_interp_kernel(SpecInterpArgs<T> a, int chunk) {
  const int s0 = blockIdx.y * chunk;
  interp_tile<T>(a, blockIdx.x * InterpShape<T>::kNodes, s0, min(s0 + chunk, a.series));
}

// batched form: block b covers the nodes from map[b].y on of item map[b].x
template <class T>
__global__ void __launch_bounds__(kInterpThreads) spectral_interp_batch_kernel(const SpecInterpArgs<T>* items,
                                                                               const int2* map, int chunk) {
  const int2 bm = map[blockIdx.x];
  const SpecInterpArgs<T> a = items[bm.x];
  const int s0 = blockIdx.y * chunk;
  interp_tile<T>(a, bm.y, s0, min(s0 + chunk, a.series));
}

// ---- gridding

__device__ __forceinline__ float exp_t(float x) { return expf(x); }
__device__ __forceinline__ double exp_t(double x) { return exp(x); }

// first node of coarse cell c: the smallest j with (j + 1/2) M / P >= c
__host__ __device__ __forceinline__ int first_node(int64_t p, int m, int c) {
  return c <= 0 ? 0 : (int)((2 * p * c - m + 2 * (int64_t)m - 1) / (2 * (int64_t)m));
}

// entry e of an item's tables: the spreading weights [2 hw][kmax][cells] (im only for the
// cells with active nodes), then the output factors [2K + 1]
template <class T>
__device__ __forceinline__ void grid_table_entry(const GridArgs<T>& a, int64_t e) {
  const int64_t nw = (int64_t)2 * a.hw * a.kmax * a.n_cells;
  if (e < nw) {
    const int c = (int)(e % a.n_cells);
    const int rest = (int)(e / a.n_cells), k = rest % a.kmax, t = rest / a.kmax;
    const int j0 = first_node(a.fft_len, a.m, c), j1 = min(first_node(a.fft_len, a.m, c + 1), a.n);
    const int j = j0 + k;
    T wre = (T)0, wim = (T)0;
    if (j < j1) {
      const int64_t num = (2 * (int64_t)j + 1) * a.m - (int64_t)c * 2 * a.fft_len;
      const T f = (T)num / (T)(2 * a.fft_len);            // in [0, 1)
      const T u = f - (T)(t - a.hw + 1);
      const T y = (T)(a.bi_rel[j] * a.y_scale);
      const T g = exp_t((T)(-a.a) * (u - y) * (u + y));
      if (y != (T)0) {
        T s, co;
        sincos_((T)(2.0 * a.a) * u * y, &s, &co);
        wre = g * co;
        wim = -g * s;
      } else {
        wre = g;
      }
    }
    a.wre[e] = wre;
    if (c < a.act_cells) a.wim[((int64_t)t * a.kmax + k) * a.act_cells + c] = wim;
    return;
  }
  const int64_t o = e - nw;
  if (o > 2 * (int64_t)a.grid_half) return;
  // exp(i theta (hw - 1)) (the coarse array starts hw - 1 cells before beta = 0), the
  // demodulation exp(i pi k / sigma) and the division by sqrt(pi / a) exp(-theta^2 / 4a)
  const int k = (int)o - a.grid_half;
  const double theta = 6.283185307179586476925 * (double)k / (double)a.m;
  const double mag = exp(theta * theta / (4.0 * a.a)) * a.inv_norm;
  double s1, c1, s2, c2;
  sincospi(2.0 * (double)(((int64_t)k * (a.hw - 1)) % a.m) / (double)a.m, &s1, &c1);
  sincospi((double)(k % (2 * a.sigma)) / (double)a.sigma, &s2, &c2);
  a.out_factor[o] = mk((T)(mag * (c1 * c2 - s1 * s2)), (T)(mag * (s1 * c2 + c1 * s2)));
}

template <class T>
__global__ void grid_table_kernel(GridArgs<T> a) {
  const int64_t total = (int64_t)2 * a.hw * a.kmax * a.n_cells + 2 * a.grid_half + 1;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
    grid_table_entry<T>(a, e);
}

template <class T>
__global__ void grid_table_batch_kernel(const GridArgs<T>* items, int item0) {
  const GridArgs<T> a = items[item0 + blockIdx.y];
  const int64_t total = (int64_t)2 * a.hw * a.kmax * a.n_cells + 2 * a.grid_half + 1;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
    grid_table_entry<T>(a, e);
}

// Spreading as a gather: a thread owns one coarse sample i of kSb series and sums the nodes
// of the 2 hw cells that reach it (coarse i takes cell c = i - t with the weights of tap t).
// The block's nodes are staged in shared memory as [vector][k][cell] (k the node's place in
// its cell, absent ones zero), 16 bytes per vector (two series in float32, one in float64):
// consecutive threads read consecutive cells of the nodes and of the weight tables, and a
// weight serves kSb series.  Cells with many nodes go through in chunks of kKc nodes.  With SUB
// tap groups a block has 1 / SUB as many samples and SUB threads for each, every SUB-th tap: for
// few series, whose blocks are fewer than the SMs and serial (strip, FP64: 15 blocks 112 us ->
// 33 us).
constexpr int kSpreadThreads = 128;
constexpr int kSpreadVec = 4;        // 16-byte vectors per node
constexpr int kKc = 4;               // nodes of a cell staged at a time
constexpr int kMaxHw = 24;           // half width limit of the staging buffer

template <class T>
struct SpreadShape {
  static constexpr int kPer = sizeof(T) == 4 ? 2 : 1;   // series per 16-byte vector
  static constexpr int kSb = kSpreadVec * kPer;
};

template <class T, int SUB>
__device__ __forceinline__ void spread_tile(const GridArgs<T>& a, int i0, int s0, unsigned char* smem_raw,
                                            int* s_first) {
  constexpr int PER = SpreadShape<T>::kPer, SB = SpreadShape<T>::kSb;
  const int tid = threadIdx.x;
  const int taps = 2 * a.hw;
  const int c_lo = i0 - taps + 1;                       // first cell that reaches this tile
  constexpr int kSamples = kSpreadThreads / SUB;
  const int ncell = kSamples + taps - 1;                // cells of the tile
  const int pitch = ncell | 1;
  float4* ys = reinterpret_cast<float4*>(smem_raw);     // [vector][kKc][pitch]
  for (int c = tid; c <= ncell; c += kSpreadThreads)
    s_first[c] = min(first_node(a.fft_len, a.m, c_lo + c), a.n);
  __syncthreads();
  const int i = i0 + tid % kSamples, sub = tid / kSamples;
  cpx<T> acc[SB];
#pragma unroll
  for (int u = 0; u < SB; ++u) acc[u] = mk((T)0, (T)0);
  for (int k0 = 0; k0 < a.kmax; k0 += kKc) {
    const int kc = min(kKc, a.kmax - k0);
    for (int e = tid; e < ncell * kKc; e += kSpreadThreads) {
      const int c = e / kKc, k = e - c * kKc;
      const int j = s_first[c] + k0 + k;
      const bool in = c_lo + c >= 0 && j < s_first[c + 1];
      cpx<T> pr = mk((T)1, (T)0);
      if (in && a.prec) pr = a.prec[j];
#pragma unroll
      for (int v = 0; v < kSpreadVec; ++v) {
        cpx<T> y[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          const int s = s0 + v * PER + u;
          y[u] = in && s < a.series ? a.y[(size_t)s * a.n + j] : mk((T)0, (T)0);
          if (a.prec) y[u] = y[u] * pr;
        }
        if constexpr (sizeof(T) == 4)
          ys[(v * kKc + k) * pitch + c] = make_float4(y[0].re, y[0].im, y[1].re, y[1].im);
        else
          *reinterpret_cast<double2*>(&ys[(v * kKc + k) * pitch + c]) = make_double2(y[0].re, y[0].im);
      }
    }
    __syncthreads();
#pragma unroll 2
    for (int t = sub; t < taps; t += SUB) {
      const int c = i - t;
      if (c < 0 || c >= a.n_cells) continue;
      const bool act = c < a.act_cells;
      const T* wr = a.wre + ((int64_t)t * a.kmax + k0) * a.n_cells + c;
      const T* wi = a.wim + ((int64_t)t * a.kmax + k0) * a.act_cells + c;
      const float4* yp = ys + (c - c_lo);
      // a cell's weights first (independent loads in flight), then its nodes
      T w[kKc], q[kKc];
#pragma unroll
      for (int k = 0; k < kKc; ++k) {
        w[k] = k < kc ? wr[(int64_t)k * a.n_cells] : (T)0;
        q[k] = act && k < kc ? wi[(int64_t)k * a.act_cells] : (T)0;
      }
#pragma unroll
      for (int k = 0; k < kKc; ++k) {
#pragma unroll
        for (int v = 0; v < kSpreadVec; ++v) {
          cpx<T> y[PER];
          if constexpr (sizeof(T) == 4) {
            const float4 f = yp[(v * kKc + k) * pitch];
            y[0] = mk(f.x, f.y);
            y[1] = mk(f.z, f.w);
          } else {
            const double2 f = *reinterpret_cast<const double2*>(&yp[(v * kKc + k) * pitch]);
            y[0] = mk(f.x, f.y);
          }
#pragma unroll
          for (int u = 0; u < PER; ++u) {
            cpx<T>& z = acc[v * PER + u];
            z.re = fma(w[k], y[u].re, z.re);
            z.im = fma(w[k], y[u].im, z.im);
            if (act) {
              z.re = fma(-q[k], y[u].im, z.re);
              z.im = fma(q[k], y[u].re, z.im);
            }
          }
        }
      }
    }
    __syncthreads();
  }
  if constexpr (SUB > 1) {
    // the tap groups' sums, in order (the staging buffer holds kSpreadThreads SB entries)
    cpx<T>* part = reinterpret_cast<cpx<T>*>(smem_raw);
#pragma unroll
    for (int u = 0; u < SB; ++u) part[u * kSpreadThreads + tid] = acc[u];
    __syncthreads();
    if (sub > 0) return;
#pragma unroll
    for (int u = 0; u < SB; ++u)
#pragma unroll
      for (int g = 1; g < SUB; ++g) acc[u] = acc[u] + part[u * kSpreadThreads + g * kSamples + tid];
  }
  if (i < a.nc) {
#pragma unroll
    for (int u = 0; u < SB; ++u)
      if (s0 + u < a.series) a.coarse[(size_t)(s0 + u) * a.nc + i] = acc[u];
  }
}

template <class T, int SUB>
__global__ void __launch_bounds__(kSpreadThreads) spread_kernel(GridArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_first[kSpreadThreads + 2 * kMaxHw + 1];
  spread_tile<T, SUB>(a, blockIdx.x * (kSpreadThreads / SUB), blockIdx.y * SpreadShape<T>::kSb, smem_raw, s_first);
}

template <class T>
__global__ void __launch_bounds__(kSpreadThreads) spread_batch_kernel(const GridArgs<T>* items, const int2* map) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_first[kSpreadThreads + 2 * kMaxHw + 1];
  const int2 bm = map[blockIdx.x];
  const GridArgs<T> a = items[bm.x];
  spread_tile<T, 1>(a, bm.y, blockIdx.y * SpreadShape<T>::kSb, smem_raw, s_first);
}

size_t spread_smem(int hw, int samples) { return (size_t)kSpreadVec * kKc * ((samples + 2 * hw - 1) | 1) * 16; }

int series_chunk(int series, int tiles) {
  // about sixteen blocks per SM (the table loads' latency needs that many warps: 72 us with
  // four on the full-size patch), at least four series per block (its weights are formed once)
  const int want = std::max(1, 16 * current_sm_count() / std::max(1, tiles));
  return std::max(std::min(series, 4), (series + want - 1) / want);
}

}  // namespace

void spectral_table_shape(bool fp64, double elem_radius, double beta_max, int* nc, double* beta0, double* d) {
  const int w = fp64 ? InterpShape<double>::W : InterpShape<float>::W;
  // 1.06: the corner of the outermost rooftop lies a little beyond the element radius
  const double step = 3.14159265358979323846 / (2.0 * 1.06 * elem_radius * kSpecOver);
  // samples at half-integer steps (none at beta = 0), w / 2 + 1 of them beyond either end;
  // a multiple of 8, so that no group of equally spaced nodes straddles the two tables
  const int need = (int)std::ceil(std::min(beta_max / step, 1e8)) + w + 4;
  *nc = (need + 7) / 8 * 8;
  *d = step;
  *beta0 = (0.5 - (w / 2 + 1)) * step;
}

// Where the tables serve a contour of n nodes: far fewer table nodes than contour nodes, and a
// contour that stays within kSpecRise table steps of the real axis.  Functions of the full type
// (all weight at the ends of the support, the worst case), float32 / float64 error over their
// maximum, by the rise in steps: 0: 3e-7 / 1e-13, 1: 2e-6 / 1e-12, 1.5: 5e-6 / 5e-12,
// 2: 2e-5 / 2e-11, 3: 1e-4 / 3e-10, 6: 1e-2 / 2e-7 (an element's spectrum: a tenth of that).  A
// contour six of its own node spacings high, the workloads' choice, rises at most 1.5 steps
// wherever the first condition holds.
constexpr double kSpecRise = 1.5;
bool spectral_tables_serve(int nc, double d, int n, double height) {
  return 4 * (int64_t)nc <= n && height <= kSpecRise * d;
}

void launch_spectral_nodes(int nc, double beta0, double d, double2* beta, double2* bw, double2* gp, double2* gr,
                           cudaStream_t s) {
  spectral_nodes_kernel<<<(2 * nc + 127) / 128, 128, 0, s>>>(nc, beta0, d, beta, bw, gp, gr);
}

template <class T>
cudaError_t launch_spectral_interp(const SpecInterpArgs<T>& a, cudaStream_t s) {
  const int tiles = (a.n + InterpShape<T>::kNodes - 1) / InterpShape<T>::kNodes;
  const int chunk = series_chunk(a.series, tiles);
  spectral_interp_kernel<T><<<dim3(tiles, (a.series + chunk - 1) / chunk), kInterpThreads, 0, s>>>(a, chunk);
  return cudaGetLastError();
}

template <class T>
int spectral_interp_nodes() { return InterpShape<T>::kNodes; }

template <class T>
cudaError_t launch_spectral_interp_batch(const SpecInterpArgs<T>* items, const int2* map, int n_blocks, int series,
                                         cudaStream_t s) {
  const int chunk = series_chunk(series, n_blocks);
  spectral_interp_batch_kernel<T><<<dim3(n_blocks, (series + chunk - 1) / chunk), kInterpThreads, 0, s>>>(items, map,
                                                                                                         chunk);
  return cudaGetLastError();
}

// the gridding of one transform; false where the series of FFTs serves it (see grid_plan's
// declaration)
bool grid_plan(bool fp64, int n, int64_t fft_len, int n_active, int grid_half, double ds, double height,
               double rho_max, int min_m, GridShape* g) {
  // height rho_max up to 3 is the documented range of float32
  if (!(height * rho_max <= 3.5)) return false;
  int64_t m = min_m;
  while (m < 2 * (2 * (int64_t)grid_half + 1)) m *= 2;
  if (m > fft_len) return false;
  const double pi = 3.14159265358979323846, e = fp64 ? 37.0 : 17.0;
  const double db = 2.0 * pi / ((double)m * ds), thc = 2.0 * pi * (grid_half + 1) / (double)m;
  const double y = n_active > 0 ? height / db : 0.0, far = 2.0 * pi - thc;
  g->a = (far * far - thc * thc) / 4.0 / (e + y * far);
  // The complex weights grow to exp(a y^2) and must cancel.  A grid as fine as the outputs ask
  // for (m below 8 K) keeps a y^2 below 4 up to height rho_max = 3.5; the shortest grid, min_m,
  // with few outputs does not.  Error of the transform over its maximum by a y^2, float32: up to
  // 5 below 1e-6 (that of a y^2 = 1), 8: 4e-6, 10: 3e-5, 13: 5e-4, 21: 4; float64: up to 7 below
  // 2e-14, 8: 5e-14, 14: 2e-11.
  if (g->a * y * y > (fp64 ? 7.0 : 5.0)) return false;
  g->hw = (int)std::ceil(std::sqrt(e / g->a));
  if (g->hw > kMaxHw) return false;
  g->m = (int)m;
  g->kmax = (int)((fft_len + m - 1) / m);
  g->n_cells = (int)((((int64_t)2 * n - 1) * m) / (2 * fft_len)) + 1;
  g->act_cells = n_active > 0 ? (int)((((int64_t)2 * n_active - 1) * m) / (2 * fft_len)) + 1 : 0;
  g->nc = g->n_cells + 2 * g->hw - 1;
  g->y_scale = n_active > 0 ? height / db : 0.0;
  return g->nc <= g->m;
}

template <class T>
cudaError_t launch_grid_tables(const GridArgs<T>& a, cudaStream_t s) {
  const int64_t total = (int64_t)2 * a.hw * a.kmax * a.n_cells + 2 * a.grid_half + 1;
  const int blocks = (int)std::min<int64_t>((total + 127) / 128, 16 * current_sm_count());
  grid_table_kernel<T><<<blocks, 128, 0, s>>>(a);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_grid_tables_batch(const GridArgs<T>* items, int item0, int n_items, cudaStream_t s) {
  for (int i = 0; i < n_items; i += 32768) {
    const int m = std::min(32768, n_items - i);
    grid_table_batch_kernel<T><<<dim3(std::max(1, 16 * current_sm_count() / m + 1), m), 128, 0, s>>>(items, item0 + i);
  }
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_spread(const GridArgs<T>& a, cudaStream_t s) {
  constexpr int kSub = 4;
  const int chunks = (a.series + SpreadShape<T>::kSb - 1) / SpreadShape<T>::kSb;
  const int tiles = (a.nc + kSpreadThreads - 1) / kSpreadThreads;
  if ((int64_t)tiles * chunks < current_sm_count()) {
    constexpr int n = kSpreadThreads / kSub;
    spread_kernel<T, kSub><<<dim3((a.nc + n - 1) / n, chunks), kSpreadThreads, spread_smem(a.hw, n), s>>>(a);
  } else {
    spread_kernel<T, 1><<<dim3(tiles, chunks), kSpreadThreads, spread_smem(a.hw, kSpreadThreads), s>>>(a);
  }
  return cudaGetLastError();
}

int spread_samples() { return kSpreadThreads; }

template <class T>
cudaError_t launch_spread_batch(const GridArgs<T>* items, const int2* map, int n_blocks, int series, int max_hw,
                                cudaStream_t s) {
  spread_batch_kernel<T><<<dim3(n_blocks, (series + SpreadShape<T>::kSb - 1) / SpreadShape<T>::kSb), kSpreadThreads,
                           spread_smem(max_hw, kSpreadThreads), s>>>(items, map);
  return cudaGetLastError();
}

#define CFFT_GRID_INSTANCES(T)                                                                                   \
  template cudaError_t launch_spectral_interp<T>(const SpecInterpArgs<T>&, cudaStream_t);                        \
  template int spectral_interp_nodes<T>();                                                                       \
  template cudaError_t launch_spectral_interp_batch<T>(const SpecInterpArgs<T>*, const int2*, int, int, cudaStream_t); \
  template cudaError_t launch_grid_tables<T>(const GridArgs<T>&, cudaStream_t);                                  \
  template cudaError_t launch_grid_tables_batch<T>(const GridArgs<T>*, int, int, cudaStream_t);                  \
  template cudaError_t launch_spread<T>(const GridArgs<T>&, cudaStream_t);                                       \
  template cudaError_t launch_spread_batch<T>(const GridArgs<T>*, const int2*, int, int, int, cudaStream_t);
CFFT_GRID_INSTANCES(float)
CFFT_GRID_INSTANCES(double)

}  // namespace cfft
