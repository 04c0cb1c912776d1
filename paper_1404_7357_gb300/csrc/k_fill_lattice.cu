// The FP64 fill of arrays whose element pairs repeat their displacements (lattices).
//
// Z_mn depends on the pair only through r_m - r_n (and the rotation class), so an array whose
// coordinates take few values has few different displacements: n_x and n_y different
// coordinates make at most U_x U_y pairs of coordinate differences, compared bit for bit.  When
// those are a small part of the pairs, the bucketed fill evaluates each (difference in x,
// difference in y, class) once, as the matrix of a U_x by U_y array of displacements, and the
// blocks are copied to the pairs.  The fill's arithmetic sees the same differences, so every
// entry equals the general path's to the bit.
//
// The general path is bound by the FP64 pipe (10,000 DFMA per pair of M = 4, 17 harmonics, 16 taps),
// the copy by writing the matrix.  GB300, 25 x 25 elements (about 20,000 displacements of
// 390,625 pairs; the differences of one pitch round to a few values each): 23 ms -> 0.60 ms.
// FP64 only: the float32 fill takes 0.28 ms for 500 elements where this one's general path takes
// 4.9, so the search, the displacements' sort and the copy (0.2 ms) would leave little.
#include <algorithm>

#include "cfft_common.cuh"

namespace cfft {

namespace {

constexpr int kLatSlots = 16384;   // hash slots: more than kLatAxis^2
constexpr unsigned long long kLatEmpty = ~0ull;   // (a NaN: no coordinate or difference)

__device__ __forceinline__ unsigned lat_hash(unsigned long long key) {
  return (unsigned)((key * 0x9E3779B97F4A7C15ull) >> 50);   // 14 bits
}

// The different values of one coordinate and of its differences, one block per axis (x, y):
//   id[i]             value of element i          did[u * n + v]   difference value u - value v
//   ud[d]             the differences             info[0 .. 1]     values (0: too many), differences
__global__ void __launch_bounds__(1024) lattice_axes_kernel(int n_el, const double* pos, LatticeAxis ax, LatticeAxis ay) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* tab = reinterpret_cast<unsigned long long*>(smem_raw);   // [kLatSlots]
  __shared__ double val[kLatAxis];
  __shared__ int count, many;
  const LatticeAxis& a = blockIdx.x ? ay : ax;
  unsigned short* slot_id = reinterpret_cast<unsigned short*>(tab + kLatSlots);   // [kLatSlots]
  // the slot of a key, inserted if it is new (then numbered); at most kLatAxis^2 < kLatSlots keys
  auto insert = [&](unsigned long long key, double v, double* out, int cap) {
    unsigned h = lat_hash(key);
    for (int probe = 0; probe < kLatSlots; ++probe, h = (h + 1) & (kLatSlots - 1)) {
      const unsigned long long old = atomicCAS(&tab[h], kLatEmpty, key);
      if (old == key) break;
      if (old == kLatEmpty) {
        const int c = atomicAdd(&count, 1);
        if (c >= cap) {
          many = 1;
        } else {
          slot_id[h] = (unsigned short)c;
          out[c] = v;
        }
        break;
      }
      if (*reinterpret_cast<volatile int*>(&many)) break;
    }
    return (int)h;
  };
  for (int h = threadIdx.x; h < kLatSlots; h += blockDim.x) tab[h] = kLatEmpty;
  if (threadIdx.x == 0) count = many = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < n_el && !*reinterpret_cast<volatile int*>(&many); i += blockDim.x) {
    const double v = pos[2 * i + blockIdx.x];
    if (!(v - v == 0.0)) many = 1;   // not finite: the general path reports it
    else a.id[i] = insert((unsigned long long)__double_as_longlong(v), v, val, kLatAxis);
  }
  __syncthreads();
  if (many) {
    if (threadIdx.x == 0) a.info[0] = a.info[1] = 0;
    return;
  }
  for (int i = threadIdx.x; i < n_el; i += blockDim.x) a.id[i] = slot_id[a.id[i]];
  const int n = count;
  __syncthreads();
  for (int h = threadIdx.x; h < kLatSlots; h += blockDim.x) tab[h] = kLatEmpty;
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const double d = __dsub_rn(val[e / n], val[e % n]);
    a.did[e] = insert((unsigned long long)__double_as_longlong(d), d, a.ud, kLatAxis * kLatAxis);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) a.did[e] = slot_id[a.did[e]];
  if (threadIdx.x == 0) {
    a.info[0] = n;
    a.info[1] = count;
  }
}

// Z of every pair from its displacement's block; a pair whose displacement lies beyond the
// table sets err (its block is zero)
template <int M>
__global__ void __launch_bounds__(256) lattice_expand_kernel(FillArgs<double, double> a, LatticeAxis ax, LatticeAxis ay,
                                                             int nx, int ny, int ux, int uy, const cpx<double>* blocks,
                                                             const unsigned char* bad) {
  const int e = blockIdx.x * 256 + threadIdx.x, n = e / M, b = e % M;
  if (n >= a.n_el) return;
  const int xn = ax.id[n], yn = ay.id[n], rn = a.rot && a.n_cls > 1 ? (a.rot[n] != 0) : 0;
  for (int m = blockIdx.y; m < a.n_el; m += gridDim.y) {
    const int gx = ax.did[ax.id[m] * nx + xn], gy = ay.did[ay.id[m] * ny + yn];
    const int cls = a.rot && a.n_cls > 1 ? 2 * (a.rot[m] != 0) + rn : 0;
    if (b == 0 && bad[(size_t)gx * uy + gy]) atomicOr(a.err, 1);
    const double2* src = reinterpret_cast<const double2*>(blocks) +
                         (((size_t)cls * ux + gx) * M * uy + gy) * M + b;
    double2* dst = reinterpret_cast<double2*>(a.z) + (size_t)m * M * a.ld + (size_t)n * M + b;
#pragma unroll
    for (int r = 0; r < M; ++r) dst[(size_t)r * a.ld] = __ldg(src + (size_t)r * uy * M);
  }
}

}  // namespace

cudaError_t launch_lattice_axes(int n_el, const double* pos, const LatticeAxis& ax, const LatticeAxis& ay,
                                cudaStream_t s) {
  constexpr int smem = kLatSlots * (int)(sizeof(unsigned long long) + sizeof(unsigned short));
  cudaError_t e = cudaFuncSetAttribute(lattice_axes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  lattice_axes_kernel<<<2, 1024, smem, s>>>(n_el, pos, ax, ay);
  return cudaGetLastError();
}

cudaError_t launch_fill_lattice(const FillArgs<double, double>& a, const LatticeAxis& ax, const LatticeAxis& ay,
                                const int (&counts)[4], const FillBucketPlan& plan, void* scratch, void* blocks,
                                unsigned char* bad, cudaStream_t s) {
  const int nx = counts[0], ux = counts[1], ny = counts[2], uy = counts[3], M = a.n_mbf;
  cudaError_t e = cudaMemsetAsync(bad, 0, (size_t)ux * uy, s);
  if (e != cudaSuccess) return e;
  for (int c = 0; c < a.n_cls; ++c) {
    FillArgs<double, double> g = a;
    g.n_el = uy;
    g.n_rows = ux;
    g.n_cls = 1;
    g.rot = nullptr;
    g.table = a.table + (size_t)c * M * M * a.n_harm * a.n_rho;
    g.z = reinterpret_cast<cpx<double>*>(blocks) + (size_t)c * ux * M * uy * M;
    g.ld = (int64_t)uy * M;
    g.dx = ax.ud;
    g.dy = ay.ud;
    g.bad = bad;
    if ((e = launch_fill_bucketed<double>(g, plan, scratch, s)) != cudaSuccess) return e;
  }
  const dim3 grid((a.n_el * M + 255) / 256, std::min(a.n_el, 65535));
  const cpx<double>* z = reinterpret_cast<const cpx<double>*>(blocks);
  switch (M) {
    case 1: lattice_expand_kernel<1><<<grid, 256, 0, s>>>(a, ax, ay, nx, ny, ux, uy, z, bad); break;
    case 2: lattice_expand_kernel<2><<<grid, 256, 0, s>>>(a, ax, ay, nx, ny, ux, uy, z, bad); break;
    case 4: lattice_expand_kernel<4><<<grid, 256, 0, s>>>(a, ax, ay, nx, ny, ux, uy, z, bad); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace cfft
