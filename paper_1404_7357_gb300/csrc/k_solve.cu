// Reduced MBF system on the GPU (Section II): the reduced excitation V' = Q^H V
// (Eq. 4), the direct solution of Z' I' = V' by a blocked LU factorization with
// partial pivoting, and the port currents (Q I'_m)[port].  The paper solves the
// reduced system directly because the MBF reduction makes it small (Table II,
// "Solving time"); this is that step, dense, on one GPU.
//
// LU (right-looking, row-major, panels of kNb columns):
//   panel    one launch over the panel's rows: per column, every CTA proposes its
//            largest |re| + |im| among the rows not yet chosen (complex64 compared
//            as floats, complex128 on the leading 32 bits; ties: lowest row), a
//            barrier, every CTA takes the same pivot, gets the pivot row and
//            eliminates the column from its own rows, the next column's entries
//            first, so that the exchange of its candidates overlaps the rest.
//            Pivoting is logical: rows stay where they are and the chosen rows are
//            recorded; one barrier per column.  A panel of more than 2048 rows runs
//            as two halves of 32 columns.  What fits the shared memory of one
//            thread-block cluster (16 CTAs, else 8) runs there: the CTAs send
//            their candidate rows into each other's shared memory.  Longer panels
//            run cooperatively over the grid: each CTA publishes its candidate's
//            key with a column tag in global memory, and polling the keys (with
//            a bound) is the grid barrier.
//   moves    the panel's pivot rows go to rows k..k+kb-1 and the rows they
//            displace to the vacated places, as a list of (source, destination)
//            row moves applied to every column of the matrix.
//   trsm     U12 = L11^-1 A12 (unit lower L11), four columns per warp at once.
//   gemm     A22 -= L21 U12, K = the panel: in complex64 on the tensor cores (the
//            complex product as a real GEMM, three TF32 products), otherwise
//            64 x 64 tiles of complex entries on the FP32 / FP64 pipe.
// With the tensor-core update the next panel runs ahead on a second stream beside the rest of
// the update (look-ahead).
// The solve takes the right-hand side in the factors' row order, then forward (unit L)
// and backward (U) substitution, one cooperative launch each: block rows of 64 dealt to
// the CTAs, solved entries passed on through tagged words in global memory.
//
// Every wait is bounded: one that runs out sets an error bit, and the CTAs leave the
// kernel (the host then returns CFFT_ERR_TIMEOUT).  The cluster barriers before and
// behind a cluster panel are the hardware's own: every CTA of the cluster is resident
// by construction and takes both.
#include <cuda.h>

#include <algorithm>

#include "cfft_common.cuh"
#include "spectra_tc.cuh"
#include "tc_sm100.cuh"

namespace cfft {

namespace {

constexpr int kNb = 64;                 // panel width
constexpr int kPanelThreads = 256;
constexpr unsigned kBarrierPolls = 1u << 22;

template <class T>
__device__ __forceinline__ cpx<T> ldcg(const cpx<T>* p);
template <>
__device__ __forceinline__ cpx<float> ldcg(const cpx<float>* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return mk(v.x, v.y);
}
template <>
__device__ __forceinline__ cpx<double> ldcg(const cpx<double>* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return mk(v.x, v.y);
}

template <class T>
__device__ __forceinline__ cpx<T> crecip(cpx<T> z) {
  return cdiv(mk((T)1, (T)0), z);
}

// a panel row's pitch in shared memory: odd, so that a column's entries lie in different banks
__host__ __device__ constexpr int cl_pitch(int kb) { return kb | 1; }

template <class T>
struct PanelArgs {
  cpx<T>* a;
  int64_t ld;
  int n, k, kb;
  unsigned long long* slot;  // [2][grid] per-CTA pivot key | column tag, by column parity
  cpx<T>* cand_data;  // [2][grid][kNb] the candidate rows' remaining panel entries
  int2* moves;        // (source row, destination row), at most 2 kb
  int* n_moves;
  int* err;           // bit 1: a barrier wait ran out; bit 2: zero pivot
};

// pivot key of row `row` with entry v: the leading 32 bits of |re| + |im| (non-negative, so its
// bits order like its value; a float whole, a double's exponent and 20 mantissa bits), then the
// lower row (rows below 65535); the low 16 bits stay free for a column tag.  The largest key is
// the pivot, so the choice does not depend on how the rows are split between CTAs; 0 stands for
// no candidate.  (complex64 in its own type: three conversions and an addition on the FP64 pipe
// per entry were most of a column's 1,100 cycles in the cluster form.)
__device__ __forceinline__ unsigned long long pivot_key(cpx<float> v, int row) {
  return ((unsigned long long)__float_as_uint(fabsf(v.re) + fabsf(v.im)) << 32) |
         ((unsigned long long)(0xFFFFu - (unsigned)row) << 16);
}
__device__ __forceinline__ unsigned long long pivot_key(cpx<double> v, int row) {
  return (((unsigned long long)__double_as_longlong(fabs(v.re) + fabs(v.im)) >> 32) << 32) |
         ((unsigned long long)(0xFFFFu - (unsigned)row) << 16);
}
__device__ __forceinline__ int key_row(unsigned long long key) { return 0xFFFF - (int)((key >> 16) & 0xFFFFu); }
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}

// the largest of the CTA's keys (every thread gets it); `wk` is not written again before the
// caller's next barrier
template <int kWarps>
__device__ __forceinline__ unsigned long long cta_max_key(unsigned long long best, unsigned long long* wk) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) best = umax64(best, __shfl_xor_sync(0xffffffffu, best, off));
  if (lane == 0) wk[warp] = best;
  __syncthreads();
  unsigned long long b = wk[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) b = umax64(b, wk[w]);
  return b;
}

// A panel column, both forms.  Column j's elimination is split so that the exchange of column
// j + 1's candidates overlaps most of it:
//   panel_column   the multipliers of column j and the new entries of column j + 1 (one thread
//                  per row), and the CTA's best key of column j + 1;
//   panel_row      the remaining entries of that best row (warp 0), which is then published;
//   panel_rest     the remaining entries of the other rows (the other warps), while warp 0
//                  exchanges keys and reads the pivot row.
// Every entry takes the same operations in the same order as an elimination column by column.

// column j with pivot row `pr` (entries j.. in prow): returns this thread's best key of j + 1
template <class T>
__device__ __forceinline__ unsigned long long panel_column(cpx<T>* rows, unsigned char* chosen, int nr, int kb, int j,
                                                           int lo, int pr, const cpx<T>* prow) {
  const cpx<T> inv = crecip(prow[0]);
  unsigned long long best = 0;
  for (int i = threadIdx.x; i < nr; i += blockDim.x) {
    if (lo + i == pr) chosen[i] = 1;
    if (chosen[i]) continue;
    cpx<T>* row = rows + (size_t)i * cl_pitch(kb) + j;
    const cpx<T> l = row[0] * inv;
    row[0] = l;
    if (j + 1 < kb) {
      cpx<T> v = row[1];
      cmac(v, mk(-l.re, -l.im), prow[1]);
      row[1] = v;
      best = umax64(best, pivot_key(v, lo + i));
    }
  }
  return best;
}

// entries j + 2.. of local row i, one warp
template <class T>
__device__ __forceinline__ void panel_row(cpx<T>* rows, int i, int kb, int j, const cpx<T>* prow) {
  cpx<T>* row = rows + (size_t)i * cl_pitch(kb) + j;
  const cpx<T> l = row[0];
  const cpx<T> ml = mk(-l.re, -l.im);
  for (int t = 2 + (int)(threadIdx.x & 31); t < kb - j; t += 32) cmac(row[t], ml, prow[t]);
}

// entries j + 2.. of every row not chosen but `skip`, warps 1 .. kWarps - 1
template <class T, int kWarps>
__device__ __forceinline__ void panel_rest(cpx<T>* rows, const unsigned char* chosen, int nr, int kb, int j, int skip,
                                           const cpx<T>* prow) {
  constexpr int kBatch = sizeof(T) == 4 ? 4 : 2;   // rows in flight per warp
  const int lane = threadIdx.x & 31, pitch = cl_pitch(kb);
  for (int t = 2 + lane; t - lane < kb - j; t += 32) {
    const bool in = t < kb - j;
    const cpx<T> pt = in ? prow[t] : mk((T)0, (T)0);
    for (int i0 = (int)(threadIdx.x >> 5) - 1; i0 < nr; i0 += kBatch * (kWarps - 1)) {
      cpx<T> l[kBatch], v[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const cpx<T>* row = rows + (size_t)min(i0 + u * (kWarps - 1), nr - 1) * pitch + j;
        l[u] = row[0];
        v[u] = in ? row[t] : mk((T)0, (T)0);
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) cmac(v[u], mk(-l[u].re, -l[u].im), pt);
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int i = i0 + u * (kWarps - 1);
        if (in && i < nr && i != skip && !chosen[i]) rows[(size_t)i * pitch + j + t] = v[u];
      }
    }
  }
}

// the panel's row moves from its pivots (every thread of the CTA, at least kNb): pivot j to row
// k + j, and the rows of the block that no column chose, in ascending order, to the rows that
// pivots from below the block left, in ascending order.  Every source is read before any
// destination is written, so the order of the list does not matter.
template <class T>
__device__ void panel_record_moves(const PanelArgs<T>& p, const int* s_piv) {
  __shared__ int displaced[kNb], vacated[kNb], taken[kNb], nm, nd;
  const int kb = p.kb, t = threadIdx.x;
  if (t < kNb) taken[t] = 0;
  if (t == 0) nm = nd = 0;
  __syncthreads();
  const int pr = t < kb ? s_piv[t] : -1;
  if (pr >= p.k && pr < p.k + kb) taken[pr - p.k] = 1;
  __syncthreads();
  if (t < kb) {
    if (pr != p.k + t) p.moves[atomicAdd(&nm, 1)] = make_int2(pr, p.k + t);
    int d = 0, v = 0;
    for (int u = 0; u < kb; ++u) {
      d += u < t && !taken[u];
      v += s_piv[u] >= p.k + kb && s_piv[u] < pr;
    }
    if (!taken[t]) {
      displaced[d] = p.k + t;
      atomicAdd(&nd, 1);
    }
    if (pr >= p.k + kb) vacated[v] = pr;   // as many as there are displaced rows
  }
  __syncthreads();
  if (t < nd) p.moves[nm + t] = make_int2(displaced[t], vacated[t]);
  if (t == 0) *p.n_moves = nm + nd;
}

// One panel of kb columns on rows k..n-1, cooperative over the grid.  Each CTA holds its
// slice of rows in shared memory for the whole panel.  Per column warp 0 completes its CTA's
// best candidate row, stages its remaining entries in global memory, publishes its pivot key
// tagged with the column (one 64-bit store after a fence) and polls the G keys of the column
// until all carry the tag (the poll is the grid barrier, and it delivers the candidates), takes
// the largest as the pivot and reads that row's entries; the other warps meanwhile finish the
// previous column's elimination.  Keys and entries are double-buffered by column parity: a CTA
// publishes column j + 2 only after it has seen every key of column j + 1, which each CTA
// publishes after its reads of column j.  Every poll is bounded; a CTA whose poll runs out
// leaves the panel, and the others then run out on its missing keys.  Bound by two trips
// through L2 per column (key, row).
template <class T>
__global__ void __launch_bounds__(kPanelThreads) lu_panel_kernel(PanelArgs<T> p) {
  constexpr int kWarps = kPanelThreads / 32;
  constexpr int kSlots = 8;   // keys per lane: at most 256 CTAs
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int R = p.n - p.k, kb = p.kb, pitch = cl_pitch(kb);
  const int per = (R + G - 1) / G;
  const int lo = p.k + min(g * per, R), hi = p.k + min((g + 1) * per, R), nr = hi - lo;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* rows = reinterpret_cast<cpx<T>*>(smem_raw);                       // [per][pitch]
  unsigned char* chosen = smem_raw + (size_t)per * pitch * sizeof(cpx<T>);  // [per]
  __shared__ cpx<T> prow[2][kNb];                                           // by column parity
  __shared__ unsigned long long wk[kWarps];
  __shared__ unsigned long long s_win;
  __shared__ int s_piv[kNb];
  __shared__ int s_fail;
  for (int e = tid; e < nr * kb; e += blockDim.x)
    rows[(size_t)(e / kb) * pitch + e % kb] = p.a[(int64_t)(lo + e / kb) * p.ld + p.k + e % kb];
  for (int i = tid; i < per; i += blockDim.x) chosen[i] = 0;
  if (tid == 0) s_fail = 0;
  __syncthreads();
  unsigned long long mine = 0;
  for (int i = tid; i < nr; i += blockDim.x) {
    const cpx<T> v = rows[(size_t)i * pitch];
    mine = umax64(mine, pivot_key(v, lo + i));
  }
  mine = cta_max_key<kWarps>(mine, wk);
  bool ok = true;
  for (int j = 0; j < kb; ++j) {
    const int buf = (p.k + j) & 1;
    const unsigned long long tag = (unsigned long long)((p.k + j) & 0xFFFF);
    const int bl = mine != 0 ? key_row(mine) - lo : -1;
    const cpx<T>* prev = prow[(j & 1) ^ 1];     // pivot row of column j - 1
    if (warp == 0) {
      if (bl >= 0) {
        if (j > 0) panel_row(rows, bl, kb, j - 1, prev);
        __syncwarp();
        for (int t = lane; t < kb - j; t += 32)
          p.cand_data[((size_t)buf * G + g) * kNb + t] = rows[(size_t)bl * pitch + j + t];
      }
      __threadfence();   // the entries before the key
      __syncwarp();
      if (lane == 0) *reinterpret_cast<volatile unsigned long long*>(p.slot + buf * G + g) = mine | tag;
      const volatile unsigned long long* sp = reinterpret_cast<const volatile unsigned long long*>(p.slot + buf * G);
      unsigned long long kmax = 0;
      bool fine = false;
      for (unsigned polls = 0; polls <= kBarrierPolls && !fine; ++polls) {
        unsigned long long x[kSlots];
#pragma unroll
        for (int u = 0; u < kSlots; ++u) x[u] = lane + 32 * u < G ? sp[lane + 32 * u] : tag;
        fine = true;
        kmax = 0;
#pragma unroll
        for (int u = 0; u < kSlots; ++u) {
          fine = fine && (x[u] & 0xFFFFull) == tag;
          kmax = umax64(kmax, x[u] & ~0xFFFFull);
        }
        if (polls > 256) __nanosleep(32);
      }
      const bool all_fine = __all_sync(0xffffffffu, fine);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) kmax = umax64(kmax, __shfl_xor_sync(0xffffffffu, kmax, off));
      __threadfence();   // the winner's entries after its key
      const int w_row = kmax != 0 ? key_row(kmax) : -1;
      if (all_fine && w_row >= p.k && w_row < p.n) {
        const int w = (w_row - p.k) / per;   // the CTA whose candidate it is
        for (int t = lane; t < kb - j; t += 32) prow[j & 1][t] = ldcg(p.cand_data + ((size_t)buf * G + w) * kNb + t);
      }
      if (lane == 0) {
        s_win = kmax;
        if (!all_fine) s_fail = 1;
      }
    } else if (j > 0) {
      panel_rest<T, kWarps>(rows, chosen, nr, kb, j - 1, bl, prev);
    }
    __syncthreads();
    if (s_fail) {
      ok = false;
      break;
    }
    const unsigned long long win = s_win;
    const int pr = win != 0 ? key_row(win) : -1;
    if (!(pr >= p.k && pr < p.n)) {   // no row left (cannot happen with n - k >= kb)
      if (tid == 0 && g == 0) atomicOr(p.err, 4);
      ok = false;
      break;
    }
    if ((win >> 32) == 0 && tid == 0 && g == 0) atomicOr(p.err, 4);   // a zero pivot
    if (tid == 0) s_piv[j] = pr;
    mine = cta_max_key<kWarps>(panel_column(rows, chosen, nr, kb, j, lo, pr, prow[j & 1]), wk);
  }
  __syncthreads();
  if (!ok) {
    // the panel stopped (a zero pivot or a wait that ran out): no row moves for it
    if (tid == 0 && s_fail) atomicOr(p.err, 2);
    if (tid == 0 && g == 0) *p.n_moves = 0;
    return;
  }
  for (int e = tid; e < nr * kb; e += blockDim.x)
    p.a[(int64_t)(lo + e / kb) * p.ld + p.k + e % kb] = rows[(size_t)(e / kb) * pitch + e % kb];
  if (g == 0) panel_record_moves(p, s_piv);
}

// ---- the panel inside one thread-block cluster (distributed shared memory)
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// all threads of all CTAs of the cluster; orders this CTA's shared-memory writes before
// the peers' reads after the barrier
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the shared-memory address `a` of this CTA in the shared memory of cluster CTA `rank`
__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// `bytes` (a multiple of 16) of this CTA's shared memory to a peer's (a cluster address), counted
// by the peer's mbarrier
__device__ __forceinline__ void bulk_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "r"(src), "r"(bytes), "r"(mbar)
               : "memory");
}
// the largest of the lanes' keys: the two halves in turn
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
  return (unsigned long long)hi << 32 | lo;
}

constexpr int kClWarps = 16;             // warps of a cluster panel's CTA that hold rows
constexpr int kClSenders = 4;            // warps that send its candidates
constexpr int kClThreads = 32 * (kClWarps + kClSenders);
constexpr int kClSlots = 3;              // columns of candidates held
constexpr unsigned kClPolls = 1u << 20;  // bound of a wait for a column's candidates
// bytes of one candidate: its key, the reciprocal of its first entry (at 16), its entries (at 32)
template <class T>
__host__ __device__ constexpr uint32_t cand_bytes(int kb) {
  return 32u + (uint32_t)((kb * sizeof(cpx<T>) + 15) & ~(size_t)15);
}
template <class T>
__host__ __device__ constexpr int cl_batch() {   // rows a warp has in flight
  return sizeof(T) == 4 ? 4 : 2;
}
// shared bytes of a CTA of `per` rows in a cluster of G: received candidates, own candidates,
// rows (and what a batch reads past the last)
template <class T>
__host__ __device__ constexpr size_t cl_smem(int G, int per, int kb) {
  return (size_t)kClSlots * (G + 1) * cand_bytes<T>(kb) + (size_t)(per + cl_batch<T>()) * cl_pitch(kb) * sizeof(cpx<T>);
}

// One panel of kb columns on rows k..n-1, the grid being one cluster of G CTAs.  Each CTA
// holds its slice of rows in shared memory for the whole panel, each of its row warps a share of
// them.  Per column the sending warps bring the CTA's best candidate row up to date and send its
// key, its entries and the reciprocal of the first to all G CTAs (one bulk copy each, counted by
// the receivers' mbarriers); meanwhile the row warps finish the previous column on their other
// rows.  All wait for the G candidates in their own shared memory and take the largest key (the
// same pivot as the grid form); the row warps divide the column of their rows, form their next
// column and that column's best key.  One trip between SMs and one block barrier per column; no
// row warp reads another's rows.  Three columns of candidates are held: a CTA sends column j + 3
// after it has column j + 2 of every peer, which a peer sends after the block barrier behind its
// last use of column j.  Every wait is bounded; a last cluster barrier keeps every CTA's shared
// memory in place until all have stopped sending.
//
// A serial chain per column: the CTA's best key, its row, the copies, the pivot, the column.
// Sending by 16-byte remote stores took 220 cycles per peer, by bulk copies of one warp 65;
// a cluster barrier, then reads of the keys and of the pivot row from the peers, 3,400.
template <class T>
__global__ void __launch_bounds__(kClThreads) lu_panel_cluster_kernel(PanelArgs<T> p) {
  constexpr int kBatch = cl_batch<T>();
  const int G = gridDim.x, g = (int)cluster_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int R = p.n - p.k, kb = p.kb;
  const int per = (R + G - 1) / G;
  const int lo = p.k + min(g * per, R), hi = p.k + min((g + 1) * per, R), nr = hi - lo;
  const int pitch = cl_pitch(kb);
  const uint32_t slot = cand_bytes<T>(kb);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* recv = smem_raw;                            // [kClSlots][G][slot]
  unsigned char* own = recv + kClSlots * G * slot;           // [kClSlots][slot]
  cpx<T>* rows = reinterpret_cast<cpx<T>*>(own + kClSlots * slot);   // [per + kBatch][pitch]
  __shared__ uint64_t mbar[kClSlots];
  __shared__ unsigned long long wk[2][kClWarps];   // the row warps' best keys, by column parity
  __shared__ int s_piv[kNb];
  __shared__ int s_fail[2];   // error bits, by column parity: every warp leaves at the same column
  for (int e = tid; e < nr * kb; e += kClThreads)
    rows[(size_t)(e / kb) * pitch + e % kb] = p.a[(int64_t)(lo + e / kb) * p.ld + p.k + e % kb];
  if (tid == 0) {
    s_fail[0] = s_fail[1] = 0;
    for (int i = 0; i < kClSlots; ++i) tc::mbar_init(&mbar[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cluster_sync_all();
  // this warp's rows r0 .. r0 + nw - 1 of the CTA's (at most 64: a bit each while not chosen)
  const int q = (per + kClWarps - 1) / kClWarps;
  const int r0 = min(warp * q, nr), nw = warp < kClWarps ? min(q, nr - r0) : 0;
  unsigned long long alive = nw == 64 ? ~0ull : (1ull << nw) - 1;
  {
    unsigned long long best = 0;
    for (int i = lane; i < nw; i += 32) {
      const cpx<T> v = rows[(size_t)(r0 + i) * pitch];
      best = umax64(best, pivot_key(v, lo + r0 + i));
    }
    best = warp_max_key(best);
    if (lane == 0 && warp < kClWarps) wk[0][warp] = best;
  }
  __syncthreads();
  uint32_t prev_at = 0;   // where recv holds the pivot row of column j - 1, from that column on
  int fail = 0, b = 0;
  uint32_t phase = 0;
  for (int j = 0; j < kb; ++j) {
    const int cnt = kb - j;
    const int nv = (int)((cnt * sizeof(cpx<T>) + 15) / 16);   // 16-byte pieces of a candidate's entries
    if (tid == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(&mbar[b])),
                   "r"((uint32_t)G * (32u + 16u * (uint32_t)nv))
                   : "memory");
    const unsigned long long mine = warp_max_key(lane < kClWarps ? wk[j & 1][lane] : 0ull);
    const int bl = mine != 0 ? key_row(mine) - lo : -1;
    const cpx<T>* prev = reinterpret_cast<const cpx<T>*>(recv + prev_at);
    if (warp >= kClWarps) {
      const cpx<T>* row = rows + max(bl, 0) * pitch + j;
      unsigned char* out = own + b * slot;
      if (warp == kClWarps) {
        // the candidate row's entries j.., with column j - 1's elimination (not written back:
        // its warp takes them from what arrives)
        const bool upd = j > 0 && bl >= 0;
        const cpx<T> l = upd ? row[-1] : mk((T)0, (T)0);
        const cpx<T> ml = mk(-l.re, -l.im);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int e = lane + 32 * u;
          if (e < cnt) {
            cpx<T> v = row[e];
            if (upd && e >= 1) cmac(v, ml, prev[e + 1]);
            reinterpret_cast<cpx<T>*>(out + 32)[e] = v;
          }
        }
      } else if (warp == kClWarps + 1 && lane == 0) {
        *reinterpret_cast<unsigned long long*>(out) = mine;
        *reinterpret_cast<cpx<T>*>(out + 16) = crecip(row[0]);
      }
      tc::fence_proxy_async();
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kClSenders) : "memory");
      const int c = (warp - kClWarps) + kClSenders * lane;
      if (c < G)
        bulk_to_peer(cluster_addr(tc::smem_u32(recv + (b * G + g) * slot), c), tc::smem_u32(out),
                     32u + 16u * (uint32_t)nv, cluster_addr(tc::smem_u32(&mbar[b]), c));
    }
    if (j > 0) {
      // entries j + 1.. of column j - 1's elimination on the warp's other rows: lanes over
      // columns, kBatch rows in flight (the rows a batch reads past the warp's are not stored)
      unsigned long long todo = alive;
      if (bl >= r0 && bl < r0 + nw) todo &= ~(1ull << (bl - r0));
      for (int c = 1 + lane; c - lane < cnt; c += 32) {
        const bool in = c < cnt;
        const int cc = in ? c : 0;
        const cpx<T> pc = prev[cc + 1];
        cpx<T>* row = rows + r0 * pitch + j;
        for (int i0 = 0; i0 < nw; i0 += kBatch, row += kBatch * pitch) {
          cpx<T> l[kBatch], v[kBatch];
#pragma unroll
          for (int u = 0; u < kBatch; ++u) {
            l[u] = row[u * pitch - 1];
            v[u] = row[u * pitch + cc];
          }
#pragma unroll
          for (int u = 0; u < kBatch; ++u) cmac(v[u], mk(-l[u].re, -l[u].im), pc);
          const unsigned bits = in ? (unsigned)(todo >> i0) : 0u;
#pragma unroll
          for (int u = 0; u < kBatch; ++u)
            if ((bits >> u) & 1) row[u * pitch + cc] = v[u];
        }
      }
    }
    __syncwarp();
    // the candidates of column j, and the pivot
    const bool got = tc::mbar_wait(&mbar[b], phase, kClPolls);
    const unsigned char* at = recv + b * G * slot;
    const unsigned long long key = got && lane < G ? *reinterpret_cast<const unsigned long long*>(at + lane * slot) : 0ull;
    const unsigned long long win = warp_max_key(key);
    const int pr = win != 0 ? key_row(win) : -1;
    const bool ok = pr >= p.k && pr < p.n;   // no row left cannot happen with n - k >= kb
    unsigned long long best = 0;
    if (ok) {
      const int who = __ffs((int)__ballot_sync(0xffffffffu, key == win)) - 1;   // the CTA whose candidate it is
      const unsigned char* cand = at + who * slot;
      const cpx<T> inv = *reinterpret_cast<const cpx<T>*>(cand + 16);
      prev_at = (b * G + who) * slot + 32;
      const int mine_pr = pr - lo - r0;
      if (mine_pr >= 0 && mine_pr < nw) alive &= ~(1ull << mine_pr);
      if (bl >= r0 && bl < r0 + nw) {   // the entries of the CTA's candidate, back into its row
        const cpx<T>* mc = reinterpret_cast<const cpx<T>*>(at + g * slot + 32);
        for (int e = 1 + lane; e < cnt; e += 32) rows[bl * pitch + j + e] = mc[e];
        __syncwarp();
      }
      const cpx<T> p1 = j + 1 < kb ? reinterpret_cast<const cpx<T>*>(cand + 32)[1] : mk((T)0, (T)0);
      for (int i = lane; i < nw; i += 32) {
        if (!((alive >> i) & 1)) continue;
        cpx<T>* row = rows + (r0 + i) * pitch + j;
        const cpx<T> l = row[0] * inv;
        row[0] = l;
        if (j + 1 < kb) {
          cpx<T> v = row[1];
          cmac(v, mk(-l.re, -l.im), p1);
          row[1] = v;
          best = umax64(best, pivot_key(v, lo + r0 + i));
        }
      }
      best = warp_max_key(best);
    }
    if (lane == 0) {
      if (warp < kClWarps) wk[(j + 1) & 1][warp] = best;
      if (!ok) s_fail[j & 1] = got ? 4 : 2;
    }
    if (tid == 0) {
      s_piv[j] = pr;
      if (ok && (win >> 32) == 0 && g == 0) atomicOr(p.err, 4);   // a zero pivot
    }
    __syncthreads();
    fail = s_fail[j & 1];
    if (fail != 0) break;
    if (++b == kClSlots) {
      b = 0;
      phase ^= 1;
    }
  }
  if (fail == 0) {
    for (int e = tid; e < nr * kb; e += kClThreads)
      p.a[(int64_t)(lo + e / kb) * p.ld + p.k + e % kb] = rows[(size_t)(e / kb) * pitch + e % kb];
    if (g == 0) panel_record_moves(p, s_piv);
  } else if (warp == 0) {
    if (lane == 0) {
      atomicOr(p.err, fail);
      if (g == 0) *p.n_moves = 0;   // the panel stopped: no row moves for it
    }
    // once more, with the same bound, for candidates still on their way here: no CTA's shared
    // memory goes while a copy into it or out of it may be in flight
    tc::mbar_wait(&mbar[b], phase, kClPolls);
  }
  cluster_sync_all();
}

// n_lists lists of row moves (kNb apart) in turn, on n_cols columns from c0 on, those from `skip`
// on kNb further: all sources of a list read before any destination is written (16 columns per
// block, every move)
template <class T>
__global__ void __launch_bounds__(256) lu_moves_kernel(cpx<T>* a, int64_t ld, int n, int c0, int n_cols, int skip,
                                                       const int2* moves, const int* n_moves, int n_lists) {
  __shared__ cpx<T> buf[2 * kNb][16];
  __shared__ int2 mv[2 * kNb];
  const int tid = threadIdx.x, cl = tid & 15, mr = tid >> 4;
  const int idx = blockIdx.x * 16 + cl;
  int col = c0 + idx;
  if (col >= skip) col += kNb;
  const bool in = idx < n_cols && col < n;
  for (int h = 0; h < n_lists; ++h) {
    const int nm = max(0, min(n_moves[h], n_lists > 1 && h > 0 ? kNb : 2 * kNb));
    if (nm == 0) continue;
    __syncthreads();
    // a move outside the matrix (none is written; checked all the same) is dropped
    for (int m = tid; m < nm; m += blockDim.x) {
      const int2 v = moves[h * kNb + m];
      mv[m] = (v.x >= 0 && v.x < n && v.y >= 0 && v.y < n) ? v : make_int2(-1, -1);
    }
    __syncthreads();
    for (int m = mr; m < nm; m += 16)
      if (in && mv[m].x >= 0) buf[m][cl] = a[(int64_t)mv[m].x * ld + col];
    __syncthreads();
    for (int m = mr; m < nm; m += 16)
      if (in && mv[m].x >= 0) a[(int64_t)mv[m].y * ld + col] = buf[m][cl];
  }
}

// Column-oriented substitution with one warp, NC right-hand sides in flight: their entries of
// rows lane and lane + 32 stay in the lane's registers; at step j the solved entries x_j are
// shuffled to every lane, and the rows below (lower, unit diagonal) or above (upper, rd the
// diagonal's reciprocals) subtract their coefficient times x_j.  M: the kb x kb diagonal block
// in shared memory (row stride ms).
template <class T, bool UPPER, int NC>
__device__ __forceinline__ void warp_substitute(const cpx<T>* M, int ms, int kb, const cpx<T>* rd, cpx<T> (&x0)[NC],
                                                cpx<T> (&x1)[NC]) {
  const int lane = threadIdx.x & 31;
  for (int s = 0; s < kb; ++s) {
    const int j = UPPER ? kb - 1 - s : s;
    const bool t0 = UPPER ? lane < j : (lane > j && lane < kb);
    const bool t1 = UPPER ? lane + 32 < j : (lane + 32 > j && lane + 32 < kb);
    const cpx<T> m0 = t0 ? M[lane * ms + j] : mk((T)0, (T)0), m1 = t1 ? M[(lane + 32) * ms + j] : mk((T)0, (T)0);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      cpx<T> xj = mk(__shfl_sync(0xffffffffu, j < 32 ? x0[c].re : x1[c].re, j & 31),
                     __shfl_sync(0xffffffffu, j < 32 ? x0[c].im : x1[c].im, j & 31));
      if (UPPER) {
        const cpx<T> y = xj;
        xj = y * rd[j];
        if constexpr (sizeof(T) == 8 || NC == 1) {   // the quotient's last bits, as a division would have them
          cpx<T> r = y;
          const cpx<T> d = M[j * ms + j];
          cmac(r, mk(-xj.re, -xj.im), d);
          cmac(xj, r, rd[j]);
        }
        if (lane == j) x0[c] = xj;
        if (lane + 32 == j) x1[c] = xj;
      }
      xj = mk(-xj.re, -xj.im);
      if ((UPPER || j < 31) && t0) cmac(x0[c], m0, xj);
      if ((!UPPER || j > 32) && t1) cmac(x1[c], m1, xj);
    }
  }
}

// U12 = L11^-1 A12 on rows k..k+kb-1 and columns k+kb..nc-1: L11 and a tile of 32 columns in
// shared memory, four columns per warp at once (lanes over rows; a serial chain of kb steps,
// so the columns of a warp share it), the tile stored back coalesced
template <class T>
__global__ void __launch_bounds__(256) lu_trsm_kernel(cpx<T>* a, int64_t ld, int nc, int k, int kb) {
  constexpr int TC = 32, LS = kNb + 1, NC = TC / 8;
  extern __shared__ __align__(16) unsigned char sm[];
  cpx<T>* L = reinterpret_cast<cpx<T>*>(sm);          // [kNb][LS]
  cpx<T>* X = L + kNb * LS;                            // [kNb][TC]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c0 = k + kb + blockIdx.x * TC;
  // (every load of a thread in flight at once)
  cpx<T> vl[kNb * kNb / 256], vx[kNb * TC / 256];
#pragma unroll
  for (int u = 0; u < kNb * kNb / 256; ++u) {
    const int r = (tid + 256 * u) / kNb, c = tid % kNb;
    vl[u] = r < kb && c < kb ? a[(int64_t)(k + r) * ld + k + c] : mk((T)0, (T)0);
  }
#pragma unroll
  for (int u = 0; u < kNb * TC / 256; ++u) {
    const int r = (tid + 256 * u) / TC, c = tid % TC;
    vx[u] = r < kb && c0 + c < nc ? a[(int64_t)(k + r) * ld + c0 + c] : mk((T)0, (T)0);
  }
#pragma unroll
  for (int u = 0; u < kNb * kNb / 256; ++u) L[((tid + 256 * u) / kNb) * LS + tid % kNb] = vl[u];
#pragma unroll
  for (int u = 0; u < kNb * TC / 256; ++u) X[((tid + 256 * u) / TC) * TC + tid % TC] = vx[u];
  __syncthreads();
  cpx<T> x0[NC], x1[NC];
#pragma unroll
  for (int u = 0; u < NC; ++u) {
    x0[u] = lane < kb ? X[lane * TC + warp * NC + u] : mk((T)0, (T)0);
    x1[u] = lane + 32 < kb ? X[(lane + 32) * TC + warp * NC + u] : mk((T)0, (T)0);
  }
  warp_substitute<T, false, NC>(L, LS, kb, nullptr, x0, x1);
#pragma unroll
  for (int u = 0; u < NC; ++u) {
    if (lane < kb) X[lane * TC + warp * NC + u] = x0[u];
    if (lane + 32 < kb) X[(lane + 32) * TC + warp * NC + u] = x1[u];
  }
  __syncthreads();
  for (int e = tid; e < kb * TC; e += blockDim.x) {
    const int r = e / TC, c = e % TC;
    if (c0 + c < nc) a[(int64_t)(k + r) * ld + c0 + c] = X[r * TC + c];
  }
}

// A22 -= L21 U12 (columns below nc): a 64 x 64 tile of complex entries per block, 256 threads with 4 x 4 each,
// the whole K (the panel width) staged in shared memory (A transposed, padded)
template <class T>
__global__ void __launch_bounds__(256) lu_gemm_kernel(cpx<T>* a, int64_t ld, int n, int nc, int k, int kb) {
  constexpr int BM = 64, BN = 64, PA = BM + 1;
  extern __shared__ unsigned char sm[];
  cpx<T>* As = reinterpret_cast<cpx<T>*>(sm);   // [kb][PA]
  cpx<T>* Bs = As + kb * PA;                    // [kb][BN]
  const int tid = threadIdx.x;
  const int r0 = k + kb + blockIdx.y * BM, c0 = k + kb + blockIdx.x * BN;
  for (int e = tid; e < BM * kb; e += 256) {
    const int row = e / kb, kk = e % kb;
    As[kk * PA + row] = r0 + row < n ? a[(int64_t)(r0 + row) * ld + k + kk] : mk((T)0, (T)0);
  }
  for (int e = tid; e < kb * BN; e += 256) {
    const int kk = e / BN, col = e % BN;
    Bs[kk * BN + col] = c0 + col < nc ? a[(int64_t)(k + kk) * ld + c0 + col] : mk((T)0, (T)0);
  }
  __syncthreads();
  const int ty = tid >> 4, tx = tid & 15;
  cpx<T> acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = mk((T)0, (T)0);
  for (int kk = 0; kk < kb; ++kk) {
    cpx<T> av[4], bv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) av[i] = As[kk * PA + ty * 4 + i];
#pragma unroll
    for (int j = 0; j < 4; ++j) bv[j] = Bs[kk * BN + tx * 4 + j];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) cmac(acc[i][j], av[i], bv[j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty * 4 + i;
    if (r >= n) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int cc = c0 + tx * 4 + j;
      if (cc < nc) {
        cpx<T>& z = a[(int64_t)r * ld + cc];
        z = z - acc[i][j];
      }
    }
  }
}

// ---- A22 -= L21 U12 on the tensor cores (complex64).  With the rows of L21 and of A22
// stored interleaved (re, im), one tile
//   D (128 rows x 128 reals = 64 complex columns) = A' (128 x 2 kb) B' (2 kb x 128)
// with A' the rows of L21 as stored (k' = 2 c + part) and
//   B'^T[j][2c] = Re U_cj, B'^T[j][2c+1] = -Im U_cj,
//   B'^T[64+j][2c] = Im U_cj, B'^T[64+j][2c+1] = Re U_cj
// holds the 64 columns' real parts of L21 U12, then their imaginary parts.  Three TF32
// products (head x head into one tensor-memory accumulator, the two corrections into a
// second, added in FP32 registers).
//
// Persistent, one CTA per SM, tiles dealt out row by row in equal contiguous runs:
//   producers  (4 warps) split L21's block into A' once per row of tiles, which stays in tensor
//              memory (from shared memory the two operands took 119 of its 128 bytes a clock
//              and starved the epilogue: 16,000 cycles per tile), and U12's into B' in shared
//              memory, 32 reals per stage, a tile ahead, with two more stages' loads in flight;
//   issuer     (1 warp) the tensor core's products;
//   epilogue   (16 warps) subtracts the products from A22's tile, which TMA brings into shared
//              memory one tile ahead and takes back: four boxes of 128 rows x 128 bytes, each with
//              its four warps, swizzled so that a lane per row meets no bank conflict.  (As loads
//              and stores of the warps it held up the producers: 12,000 cycles per tile.)
// A22 is read and written once per panel, which bounds it (16 bytes per entry); the products
// take about three quarters of that time.  The rows of `a` are 16-byte aligned (ld even).
// GB300, 8,000^2, all panels: 19.9 ms with a tile per CTA, which loaded, split, multiplied
// and stored in turn (two CTAs per SM) -> 12.4 ms.
constexpr int kUM = 128, kUN = 128, kUK = 32;   // tile rows, tile real columns, reals per stage
constexpr int kUStages = 2 * kNb / kUK;          // stages per tile
constexpr int kUProd = 4, kUEpi = 16;            // producer and epilogue warps
constexpr int kUThreads = 32 * (kUProd + kUEpi + 1);
constexpr uint32_t kUSbo = (kUK / 4) * 128;      // 8-row group stride of B' (K-major)
constexpr uint32_t kUB = kUN * kUK * 4;          // bytes of a stage's head or correction
constexpr unsigned kUPolls = 1u << 22;           // bound of a wait
constexpr uint32_t kUColA = 2 * kUN;             // tensor-memory columns: products, corrections, then A'
constexpr int kUBox = 32;                        // floats of a box's rows
constexpr uint32_t kUBoxBytes = kUM * kUBox * 4;
constexpr size_t kUSmem = 1024 + 2 * kUStages * kUB + (kUN / kUBox) * kUBoxBytes;
static_assert(kUSmem <= 227 * 1024 - 1024, "update: one CTA's shared memory");
static_assert(kUColA + 4 * kNb <= 512 && kUProd * 32 == kUM, "update: A' in tensor memory");

// panel of kNb columns at k; rows k + kNb .. n - 1, ct tiles of columns from cf on.  map: a as n rows of 2 n floats
// (ld apart), boxes of kUBox x kUM, 128-byte swizzle
__global__ void __launch_bounds__(kUThreads, 1) lu_gemm_tc_kernel(const __grid_constant__ CUtensorMap map, cpx<float>* a,
                                                                   int64_t ld, int n, int k, int cf, int ct, int* err) {
  extern __shared__ __align__(1024) unsigned char sm_raw[];
  __shared__ uint64_t full_c[kUN / kUBox], full_b[kUStages], empty_b[kUStages], full_t, empty_t, drain;
  __shared__ uint32_t taddr_s;
  __shared__ int s_fail;
  unsigned char* Bs = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int k1 = k + kNb, rt = (n - k1 + kUM - 1) / kUM;
  const int64_t tiles = (int64_t)rt * ct;
  const int t0 = (int)(tiles * blockIdx.x / gridDim.x), t1 = (int)(tiles * (blockIdx.x + 1) / gridDim.x);
  if (tid == 0) {
    s_fail = 0;
    for (int i = 0; i < kUStages; ++i) {
      tc::mbar_init(&full_b[i], kUProd);
      tc::mbar_init(&empty_b[i], 1);
    }
    for (int i = 0; i < kUN / kUBox; ++i) tc::mbar_init(&full_c[i], 1);
    tc::mbar_init(&full_t, 1);
    tc::mbar_init(&empty_t, kUEpi);
    tc::mbar_init(&drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    tc::tmem_alloc(&taddr_s, 512);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = taddr_s;
  auto failed = [&]() { return *reinterpret_cast<volatile int*>(&s_fail) != 0; };
  // one lane per warp polls, the others wait for it
  auto wait = [&](uint64_t* m, int parity) {
    if (lane == 0 && !failed() && !tc::mbar_wait(m, (uint32_t)parity & 1u, kUPolls)) atomicOr(&s_fail, 1);
    __syncwarp();
  };
  if (warp < kUEpi) {
    // ---- epilogue: tensor-memory lanes 32 (warp mod 4).., columns 16 (warp / 4).. (a box)
    const int lq = warp & 3, cg = warp >> 2, r = 32 * lq + lane;
    unsigned char* box = Bs + 2 * kUStages * kUB + cg * kUBoxBytes;
    float4* row = reinterpret_cast<float4*>(box + r * kUBox * 4);
    const bool lead = lq == 0 && lane == 0;
    int loads = 0;
    auto load = [&](int t) {
      ++loads;
      tc::mbar_expect(&full_c[cg], kUBoxBytes);
      tc::tma_load2(box, &map, 2 * (cf + (t % ct) * (kUN / 2)) + kUBox * cg, k1 + (t / ct) * kUM, &full_c[cg]);
    };
    if (lead && t0 < t1) load(t0);
    for (int t = t0, it = 0; t < t1; ++t, ++it) {
      wait(&full_t, it);
      tc::fence_after_sync();
      const uint32_t at = tmem + ((uint32_t)(32 * lq) << 16) + 16u * cg;
      float4 d[8];   // 16 complex columns
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[4][8];   // real parts, their corrections, imaginary parts, theirs: 8 columns
        const uint32_t re = at + 8u * h, im = re + kUN / 2;
        tc::tmem_ld8x4(re, re + kUN, im, im + kUN, v);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          d[4 * h + i] = make_float4(v[0][2 * i] + v[1][2 * i], v[2][2 * i] + v[3][2 * i],
                                     v[0][2 * i + 1] + v[1][2 * i + 1], v[2][2 * i + 1] + v[3][2 * i + 1]);
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&empty_t);   // the accumulators are read
      wait(&full_c[cg], it);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float4* z = row + (i ^ (r & 7));
        const float4 c = *z;
        *z = make_float4(c.x - d[i].x, c.y - d[i].y, c.z - d[i].z, c.w - d[i].w);
      }
      tc::fence_proxy_async();
      asm volatile("bar.sync %0, 128;" ::"r"(1 + cg) : "memory");   // the box's four warps
      if (lead) {
        const int x = 2 * (cf + (t % ct) * (kUN / 2)) + kUBox * cg;
        if (!failed() && x < 2 * n) tc::tma_store2(&map, x, k1 + (t / ct) * kUM, box);
        tc::tma_store_wait_read();
        if (t + 1 < t1) load(t + 1);
      }
      __syncwarp();
    }
    if (lead) {
      if (loads > 0) tc::mbar_wait(&full_c[cg], (loads - 1) & 1, kUPolls);   // (in flight after a failure)
      tc::tma_store_wait();
    }
  } else if (warp < kUEpi + kUProd) {
    // ---- producers
    const int w = warp - kUEpi;   // (its tensor-memory lanes: kUEpi is a multiple of 4)
    const int n_stages = (t1 - t0) * kUStages;
    // B': two adjacent panel rows of one column give whole 16-byte rows of a core matrix, eight
    // lanes a whole one; warp w takes row pairs 2 w, 2 w + 1 of the stage's 8, lanes over 32 columns
    float2 bv[2][8];
    int lt = t0 % ct, ls = 0;   // tile column and stage of the next load
    const float2* const x0 = reinterpret_cast<const float2*>(a + (int64_t)(k + 4 * w) * ld + cf + lane);
    auto load = [&](float2 (&v)[8]) {
      const float2* x = x0 + (int64_t)ls * (kUK / 2) * ld + lt * (kUN / 2);
      const int cols = n - (cf + lt * (kUN / 2) + lane);
#pragma unroll
      for (int r = 0; r < 4; ++r, x += ld) {
        v[2 * r] = 0 < cols ? __ldcg(x) : make_float2(0.f, 0.f);
        v[2 * r + 1] = 32 < cols ? __ldcg(x + 32) : make_float2(0.f, 0.f);
      }
      if (++ls == kUStages) {
        ls = 0;
        if (++lt == ct) lt = 0;
      }
    };
    unsigned char* const B0 = Bs + tc::kmajor_offset(lane, 8 * w, kUK);
    constexpr uint32_t kPair = 128, kHalf = 4 * kUSbo, kIm = 8 * kUSbo;   // next row pair; columns + 32; imaginary
    if (n_stages > 0) {
      load(bv[0]);
      load(bv[1]);
    }
    for (int t = t0, it = 0; t < t1; ++t, ++it) {
      if (it == 0 || t % ct == 0) {
        // A' of this row of tiles, once no product reads the last one's: a lane per row, the
        // panel's 128 reals as tensor-memory columns (heads, then corrections)
        if (it > 0) {
          wait(&full_t, it - 1);
          tc::fence_after_sync();
        }
        const int R = k1 + (t / ct) * kUM + 32 * w + lane;
        const float4* x = reinterpret_cast<const float4*>(a + (int64_t)R * ld + k);
        const uint32_t to = tmem + ((uint32_t)(32 * w) << 16) + kUColA;
#pragma unroll 2
        for (int c = 0; c < 2 * kNb; c += 16) {
          float hi[16], lo[16];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 v = R < n ? __ldcg(x + c / 4 + u) : make_float4(0.f, 0.f, 0.f, 0.f);
            tf32_split(v.x, hi[4 * u], lo[4 * u]);
            tf32_split(v.y, hi[4 * u + 1], lo[4 * u + 1]);
            tf32_split(v.z, hi[4 * u + 2], lo[4 * u + 2]);
            tf32_split(v.w, hi[4 * u + 3], lo[4 * u + 3]);
          }
          tc::tmem_st16(to + c, hi);
          tc::tmem_st16(to + 2 * kNb + c, lo);
        }
        tc::tmem_wait_st();
        tc::fence_before_sync();
      }
#pragma unroll 2
      for (int st = 0; st < kUStages; ++st) {
        const int gs = it * kUStages + st, buf = st & 1;
        if (it > 0) wait(&empty_b[st], it - 1);
#pragma unroll
        for (int rp = 0; rp < 2; ++rp)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float2 x = bv[buf][4 * rp + h], y = bv[buf][4 * rp + 2 + h];
            float xh, xl, xih, xil, yh, yl, yih, yil;
            tf32_split(x.x, xh, xl);
            tf32_split(x.y, xih, xil);
            tf32_split(y.x, yh, yl);
            tf32_split(y.y, yih, yil);
            unsigned char* B = B0 + st * 2 * kUB + rp * kPair + h * kHalf;
            *reinterpret_cast<float4*>(B) = make_float4(xh, -xih, yh, -yih);
            *reinterpret_cast<float4*>(B + kIm) = make_float4(xih, xh, yih, yh);
            *reinterpret_cast<float4*>(B + kUB) = make_float4(xl, -xil, yl, -yil);
            *reinterpret_cast<float4*>(B + kUB + kIm) = make_float4(xil, xl, yil, yl);
          }
        if (gs + 2 < n_stages) load(bv[buf]);
        tc::fence_proxy_async();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&full_b[st]);
      }
    }
  } else {
    // ---- issuer
    const uint32_t idesc = tc::idesc_tf32(kUM, kUN), b0 = tc::smem_u32(Bs);
    bool issued = false;
    for (int t = t0, it = 0; t < t1; ++t, ++it) {
      if (it > 0) wait(&empty_t, it - 1);
      for (int st = 0; st < kUStages; ++st) {
        wait(&full_b[st], it);
        tc::fence_after_sync();
        if (lane == 0 && !failed()) {
          const uint32_t bh = b0 + st * 2 * kUB, bl = bh + kUB;
#pragma unroll
          for (int s2 = 0; s2 < kUK / 8; ++s2) {
            const uint32_t ah = tmem + kUColA + st * kUK + 8 * s2, al = ah + 2 * kNb;
            const uint64_t dbh = tc::sdesc(bh + s2 * 256, 128, kUSbo), dbl = tc::sdesc(bl + s2 * 256, 128, kUSbo);
            const uint32_t accf = (st > 0 || s2 > 0) ? 1u : 0u;
            tc::mma_tf32_ta(tmem + kUN, ah, dbl, idesc, accf);
            tc::mma_tf32_ta(tmem + kUN, al, dbh, idesc, 1u);
            tc::mma_tf32_ta(tmem, ah, dbh, idesc, accf);
          }
          tc::mma_commit(&empty_b[st]);
          if (st == kUStages - 1) tc::mma_commit(&full_t);
          issued = true;
        }
        __syncwarp();
      }
    }
    if (lane == 0 && issued) {
      // every product done before the tensor memory is freed
      tc::mma_commit(&drain);
      if (!tc::mbar_wait(&drain, 0, kUPolls)) atomicOr(&s_fail, 1);
    }
    __syncwarp();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
  if (tid == 0 && failed()) atomicOr(err, 8);
}

// the row order of the factors: row i holds the matrix's row perm[i], every panel's row moves
// applied in panel order (two lists per panel, the second that of the panel's second half where
// it ran in two).  One block, the order in shared memory (n <= 65535), kPermLists lists at a
// time: on a vector in global memory the lists took 1 us each (8,000: 0.25 ms per right-hand
// side); once per factorization
constexpr int kPermLists = 32;
__global__ void __launch_bounds__(256) lu_order_kernel(int n, int n_lists, const int2* moves, const int* n_moves,
                                                       int* perm) {
  extern __shared__ __align__(16) unsigned char sm[];
  unsigned short* p = reinterpret_cast<unsigned short*>(sm);
  __shared__ int2 mv[kPermLists * kNb];
  __shared__ int nm[kPermLists];
  for (int i = threadIdx.x; i < n; i += 256) p[i] = (unsigned short)i;
  for (int h0 = 0; h0 < n_lists; h0 += kPermLists) {
    const int cnt = min(kPermLists, n_lists - h0);
    __syncthreads();
    if ((int)threadIdx.x < cnt)
      nm[threadIdx.x] = max(0, min(n_moves[h0 + threadIdx.x], ((h0 + threadIdx.x) & 1) ? kNb : 2 * kNb));
    for (int e = threadIdx.x; e < cnt * kNb; e += 256) mv[e] = moves[(size_t)h0 * kNb + e];
    __syncthreads();
    for (int h = 0; h < cnt; ++h) {
      if (nm[h] == 0) continue;   // the same in every thread
      const int m = threadIdx.x;  // at most 2 kNb moves; a whole panel's list runs on into its second place
      int2 v = make_int2(-1, -1);
      unsigned short r = 0;
      if (m < nm[h]) {
        v = mv[h * kNb + m];
        if (v.x >= 0 && v.x < n && v.y >= 0 && v.y < n) r = p[v.x];
        else v.x = -1;
      }
      __syncthreads();
      if (v.x >= 0) p[v.y] = r;
      __syncthreads();
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += 256) perm[i] = p[i];
}
static_assert(kPermLists % 2 == 0, "a panel's two lists are staged together");

// A solved entry on its way to the other CTAs: 32 bits of value under a tag per 64-bit word, so
// that a reader that finds the tag has the value (no flag, no fence)
constexpr unsigned kSolvedTag = 1;
__device__ __forceinline__ unsigned long long tag_word(unsigned v) {
  return (unsigned long long)kSolvedTag << 32 | v;
}
template <class T>
struct Solved;
template <>
struct Solved<float> {
  static constexpr int kWords = 2;
  static __device__ __forceinline__ void put(volatile unsigned long long* w, cpx<float> v) {
    w[0] = tag_word(__float_as_uint(v.re));
    w[1] = tag_word(__float_as_uint(v.im));
  }
  static __device__ __forceinline__ cpx<float> value(const unsigned long long* w) {
    return mk(__uint_as_float((unsigned)w[0]), __uint_as_float((unsigned)w[1]));
  }
};
template <>
struct Solved<double> {
  static constexpr int kWords = 4;
  static __device__ __forceinline__ void put(volatile unsigned long long* w, cpx<double> v) {
    w[0] = tag_word((unsigned)__double2loint(v.re));
    w[1] = tag_word((unsigned)__double2hiint(v.re));
    w[2] = tag_word((unsigned)__double2loint(v.im));
    w[3] = tag_word((unsigned)__double2hiint(v.im));
  }
  static __device__ __forceinline__ cpx<double> value(const unsigned long long* w) {
    return mk(__hiloint2double((int)(unsigned)w[1], (int)(unsigned)w[0]),
              __hiloint2double((int)(unsigned)w[3], (int)(unsigned)w[2]));
  }
};

// acc[u] (row 8 warp + u, u < 8) summed over the warp's lanes: halving exchanges, after which
// lane 4 u' holds a whole row; returns that row's sum and its index in the warp (all lanes)
template <class T>
__device__ __forceinline__ cpx<T> rows_sum(cpx<T> (&acc)[8], int& row) {
  const int lane = threadIdx.x & 31;
  row = 0;
#pragma unroll
  for (int half = 4, off = 16; half > 0; half >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
    row += up ? half : 0;
#pragma unroll
    for (int u = 0; u < half; ++u) {
      const cpx<T> keep = up ? acc[u + half] : acc[u], give = up ? acc[u] : acc[u + half];
      acc[u].re = keep.re + __shfl_xor_sync(0xffffffffu, give.re, off);
      acc[u].im = keep.im + __shfl_xor_sync(0xffffffffu, give.im, off);
    }
  }
  cpx<T> v = acc[0];
#pragma unroll
  for (int off = 2; off > 0; off >>= 1) {
    v.re += __shfl_xor_sync(0xffffffffu, v.re, off);
    v.im += __shfl_xor_sync(0xffffffffu, v.im, off);
  }
  return v;
}

// One row of a kNb x kNb matrix (row stride kNb + 1, shared) times a vector: four threads per
// row, the sum in all four
template <class T>
__device__ __forceinline__ cpx<T> row_times(const cpx<T>* M, const cpx<T>* v) {
  const int r = threadIdx.x >> 2, part = threadIdx.x & 3;
  cpx<T> s = mk((T)0, (T)0);
#pragma unroll
  for (int q = 0; q < kNb / 4; ++q) cmac(s, M[r * (kNb + 1) + part + 4 * q], v[part + 4 * q]);
#pragma unroll
  for (int off = 1; off < 4; off <<= 1) {
    s.re += __shfl_xor_sync(0xffffffffu, s.re, off);
    s.im += __shfl_xor_sync(0xffffffffu, s.im, off);
  }
  return s;
}

template <class T>
constexpr size_t subst_smem() {   // the diagonal block, and its inverse (complex64)
  return (size_t)(sizeof(T) == 4 ? 2 : 1) * kNb * (kNb + 1) * sizeof(cpx<T>);
}

// x with L x = b[order] (unit lower) or U x = b (UPPER), one cooperative launch: block rows of
// kNb, dealt to the CTAs in the order in which they are solved, so the lowest unsolved one always
// has a CTA at work on it.  A CTA subtracts the solved blocks as they appear (its next tile's
// loads in flight meanwhile), solves its diagonal block and publishes the entries.  complex64
// inverts the diagonal block while it waits and multiplies by the inverse, with one step of
// refinement against the block itself, so that the error is that of a substitution; in complex128
// the FP64 pipe makes the three products (13 us) and the inverse (50 us and more) dearer than a
// substitution of 64 serial steps, and so is the first block's, which waits for nothing (two
// substitutions of 24 unknowns: 39 us with the inverses, 12 us without).  Bound by the chain of blocks:
// publish, poll, one tile, the diagonal block.  One launch per block row with a serial substitution
// in every CTA took 15 us (forward) and 25 us (backward) per block in complex64.
template <class T, bool UPPER>
__global__ void __launch_bounds__(256) lu_substitute_kernel(const cpx<T>* a, int64_t ld, int n, const int* order,
                                                            const cpx<T>* b, cpx<T>* x, unsigned long long* words,
                                                            int* err) {
  constexpr int LS = kNb + 1, W = Solved<T>::kWords;
  extern __shared__ __align__(16) unsigned char sm[];
  cpx<T>* D = reinterpret_cast<cpx<T>*>(sm);   // the diagonal block
  cpx<T>* V = D + kNb * LS;                     // its inverse (complex64)
  __shared__ cpx<T> xs[2][kNb], rhs[kNb], sol[kNb], rd[kNb];
  __shared__ int s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nb = (n + kNb - 1) / kNb;
  const cpx<T> zero = mk((T)0, (T)0);
  if (tid == 0) s_fail = 0;
  for (int t = blockIdx.x; t < nb; t += gridDim.x) {
    const int k = kNb * (UPPER ? nb - 1 - t : t), kb = min(kNb, n - k);
    __syncthreads();
    cpx<T> v[kNb * kNb / 256];
#pragma unroll
    for (int u = 0; u < kNb * kNb / 256; ++u) {
      const int r = (tid >> 6) + 4 * u, c = tid & 63;
      v[u] = r < kb && c < kb ? a[(int64_t)(k + r) * ld + k + c] : mk(r == c ? (T)1 : (T)0, (T)0);
      if (UPPER ? r > c : r < c) v[u] = zero;
      if (!UPPER && r == c) v[u] = mk((T)1, (T)0);
    }
#pragma unroll
    for (int u = 0; u < kNb * kNb / 256; ++u) D[((tid >> 6) + 4 * u) * LS + (tid & 63)] = v[u];
    if (tid < kb) rhs[tid] = b[order ? order[k + tid] : k + tid];
    if (tid >= kb && tid < kNb) rhs[tid] = zero;
    __syncthreads();
    if (UPPER) {
      if (tid < kNb) rd[tid] = crecip(D[tid * LS + tid]);
      __syncthreads();
    }
    const bool invert = sizeof(T) == 4 && t > 0;
    if (invert) {
      cpx<T> x0[8], x1[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        x0[u] = mk(lane == 8 * warp + u ? (T)1 : (T)0, (T)0);
        x1[u] = mk(lane + 32 == 8 * warp + u ? (T)1 : (T)0, (T)0);
      }
      warp_substitute<T, UPPER, 8>(D, LS, kNb, rd, x0, x1);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        V[lane * LS + 8 * warp + u] = x0[u];
        V[(lane + 32) * LS + 8 * warp + u] = x1[u];
      }
    }
    // the solved blocks: rows k + 8 warp + u, columns lane and lane + 32 of each
    cpx<T> acc[8], m0[8], m1[8];
    auto load = [&](int s) {
      const int c = kNb * (UPPER ? nb - 1 - s : s) + lane;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = k + 8 * warp + u;
        const cpx<T>* p = a + (int64_t)r * ld + c;
        m0[u] = r < n && c < n ? ldcg(p) : zero;
        m1[u] = r < n && c + 32 < n ? ldcg(p + 32) : zero;
      }
    };
#pragma unroll
    for (int u = 0; u < 8; ++u) acc[u] = zero;
    if (t > 0) load(0);
    for (int s = 0; s < t; ++s) {
      if (warp == 0) {
        const int c = kNb * (UPPER ? nb - 1 - s : s) + lane;
        const volatile unsigned long long* p = words + (size_t)c * W;
        unsigned long long w[2][W];
        bool have = false;
        for (unsigned polls = 0; polls <= kBarrierPolls && !have; ++polls) {
          if (polls > 0 && t - s > 2) __nanosleep(200);   // the next blocks first
          have = true;
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < W; ++q) {
              w[h][q] = c + 32 * h < n ? p[32 * h * W + q] : tag_word(0);
              have = have && (unsigned)(w[h][q] >> 32) == kSolvedTag;
            }
        }
        if (!have) s_fail = 1;
        xs[s & 1][lane] = Solved<T>::value(w[0]);
        xs[s & 1][lane + 32] = Solved<T>::value(w[1]);
      }
      __syncthreads();
      if (s_fail) break;
      const cpx<T> y0 = xs[s & 1][lane], y1 = xs[s & 1][lane + 32];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        cmac(acc[u], m0[u], y0);
        cmac(acc[u], m1[u], y1);
      }
      if (s + 1 < t) load(s + 1);
    }
    int row;
    const cpx<T> sum = rows_sum(acc, row);
    if ((lane & 3) == 0) rhs[8 * warp + row] = rhs[8 * warp + row] - sum;
    __syncthreads();
    if (s_fail) break;
    if (!invert) {
      if (warp == 0) {
        cpx<T> x0[1] = {rhs[lane]}, x1[1] = {rhs[lane + 32]};
        warp_substitute<T, UPPER, 1>(D, LS, kb, rd, x0, x1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = lane + 32 * h;
          const cpx<T> z = h ? x1[0] : x0[0];
          if (r < kb) {
            Solved<T>::put(words + (size_t)(k + r) * W, z);
            x[k + r] = z;
          }
        }
      }
      continue;
    }
    const int r = tid >> 2;
    const cpx<T> y = row_times(V, rhs);
    if ((tid & 3) == 0) sol[r] = y;
    __syncthreads();
    const cpx<T> dy = row_times(D, sol);
    if ((tid & 3) == 0) xs[0][r] = rhs[r] - dy;
    __syncthreads();
    const cpx<T> z = y + row_times(V, xs[0]);
    if ((tid & 3) == 0 && r < kb) {
      Solved<T>::put(words + (size_t)(k + r) * W, z);
      x[k + r] = z;
    }
  }
  if (tid == 0 && s_fail) atomicOr(err, 16);
}

// r = b - Z x in float64 from the float64 matrix (one warp per row), and |r|^2, |b|^2 sums
__global__ void __launch_bounds__(256) residual_kernel(const cpx<double>* z, int64_t ld, int n, const cpx<double>* x,
                                                       const cpx<double>* b, cpx<double>* r, double* sums) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  double rr = 0.0, bb = 0.0;
  for (int i = blockIdx.x * nw + warp; i < n; i += gridDim.x * nw) {
    cpx<double> acc = mk(0.0, 0.0);
    for (int j = lane; j < n; j += 32) cmac(acc, z[(int64_t)i * ld + j], x[j]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      acc.re += __shfl_xor_sync(0xffffffffu, acc.re, off);
      acc.im += __shfl_xor_sync(0xffffffffu, acc.im, off);
    }
    if (lane == 0) {
      const cpx<double> v = b[i] - acc;
      if (r) r[i] = v;
      rr += v.re * v.re + v.im * v.im;
      bb += b[i].re * b[i].re + b[i].im * b[i].im;
    }
  }
  if (lane == 0) {
    atomicAdd(sums, rr);
    atomicAdd(sums + 1, bb);
  }
}

// the same residual from a complex64 matrix and vectors (accumulated in float64)
__global__ void __launch_bounds__(256) residual32_kernel(const cpx<float>* z, int64_t ld, int n, const cpx<float>* x,
                                                         const cpx<float>* b, double* sums) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  double rr = 0.0, bb = 0.0;
  for (int i = blockIdx.x * nw + warp; i < n; i += gridDim.x * nw) {
    cpx<double> acc = mk(0.0, 0.0);
    for (int j = lane; j < n; j += 32) cmac(acc, ccast<double>(z[(int64_t)i * ld + j]), ccast<double>(x[j]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      acc.re += __shfl_xor_sync(0xffffffffu, acc.re, off);
      acc.im += __shfl_xor_sync(0xffffffffu, acc.im, off);
    }
    if (lane == 0) {
      const cpx<double> v = ccast<double>(b[i]) - acc;
      rr += v.re * v.re + v.im * v.im;
      bb += (double)b[i].re * b[i].re + (double)b[i].im * b[i].im;
    }
  }
  if (lane == 0) {
    atomicAdd(sums, rr);
    atomicAdd(sums + 1, bb);
  }
}

// copy an n x n block (row stride ld) into one of row stride ld_dst, changing precision: a
// block of rows per CTA, lanes over columns
template <class TD, class TS>
__global__ void __launch_bounds__(256) copy_matrix_kernel(const cpx<TS>* src, int64_t ld, int n, cpx<TD>* dst,
                                                          int64_t ld_dst) {
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y)
    for (int j = blockIdx.x * 256 + threadIdx.x; j < n; j += gridDim.x * 256)
      dst[i * ld_dst + j] = ccast<TD>(src[i * ld + j]);
}

template <class TD, class TS>
__global__ void copy_vector_kernel(const cpx<TS>* src, int n, cpx<TD>* dst) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = ccast<TD>(src[i]);
}

// x += d (float64 + float32 correction); sums[0] += |d|^2, sums[1] += |x|^2
__global__ void add_correction_kernel(cpx<double>* x, const cpx<float>* d, int n, double* sums) {
  double dd = 0.0, xx = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const cpx<double> di = ccast<double>(d[i]);
    const cpx<double> v = x[i] + di;
    x[i] = v;
    dd += di.re * di.re + di.im * di.im;
    xx += v.re * v.re + v.im * v.im;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    dd += __shfl_xor_sync(0xffffffffu, dd, off);
    xx += __shfl_xor_sync(0xffffffffu, xx, off);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(sums, dd);
    atomicAdd(sums + 1, xx);
  }
}

// V'_{e,a} = sum_i conj(Q_ia) V_{e,i}  (Eq. 4), one thread per (element, MBF)
template <class T>
__global__ void reduced_excitation_kernel(int n_el, int n_basis, int m, const cpx<T>* v, const cpx<double>* q,
                                          cpx<T>* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_el * m) return;
  const int e = t / m, a = t % m;
  cpx<double> acc = mk(0.0, 0.0);
  for (int i = 0; i < n_basis; ++i) cmac_conj(acc, q[(size_t)i * m + a], ccast<double>(v[(size_t)e * n_basis + i]));
  out[t] = ccast<T>(acc);
}

// delta-gap port across basis function `port`: V'_{e,a} = amp_e conj(Q_port,a)
template <class T>
__global__ void port_excitation_kernel(int n_el, int m, int port, const cpx<T>* amp, const cpx<double>* q,
                                       cpx<T>* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_el * m) return;
  const int e = t / m, a = t % m;
  out[t] = ccast<T>(conj(q[(size_t)port * m + a]) * ccast<double>(amp[e]));
}

// port current of element e: (Q I'_e)[port] = sum_a Q_port,a I'_{e,a}
template <class T>
__global__ void port_currents_kernel(int n_el, int m, int port, const cpx<T>* ired, const cpx<double>* q,
                                     cpx<T>* out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_el) return;
  cpx<double> acc = mk(0.0, 0.0);
  for (int a = 0; a < m; ++a) cmac(acc, q[(size_t)port * m + a], ccast<double>(ired[(size_t)e * m + a]));
  out[e] = ccast<T>(acc);
}

int grid_for(int64_t items, int per_block, int cap) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((items + per_block - 1) / per_block, cap));
}

}  // namespace

int lu_panel_width() { return kNb; }

// panel CTAs: enough that each CTA's rows fit kPanelSmem bytes of shared memory, and about
// kPanelRows rows each (the per-column elimination is short; the grid barrier's cost grows
// slowly with the CTA count), at most one per SM
constexpr size_t kPanelSmem = 160 * 1024;
constexpr int kPanelRows = 64;

template <class T>
int lu_panel_grid(int rows, int sms) {
  const int64_t row_bytes = (int64_t)kNb * sizeof(cpx<T>);
  const int64_t need = (rows * row_bytes + (int64_t)kPanelSmem - 1) / (int64_t)kPanelSmem;
  const int64_t g = std::max<int64_t>(need, std::min<int64_t>(sms, (rows + kPanelRows - 1) / kPanelRows));
  return (int)std::max<int64_t>(1, g);
}

// the most rows of a panel of kb columns that one cluster of cs CTAs holds in shared
// memory (the opt-in limit per CTA less room for the kernel's static words), at most 64 per warp
template <class T>
int cluster_panel_rows(int cs, int kb, int smem_optin) {
  const int64_t avail = std::max<int64_t>(0, (int64_t)smem_optin - 4096 - (int64_t)cl_smem<T>(cs, 0, kb));
  const int64_t per = std::min<int64_t>(avail / ((int64_t)cl_pitch(kb) * (int64_t)sizeof(cpx<T>)), 64 * kClWarps);
  return (int)(cs * per);
}

// panels of more than this many rows run as two halves of kNb / 2 columns (the second after
// the first's update of its columns): half the elimination per column, and twice the rows fit
// the cluster (12,880 in complex64, 6,032 in complex128 with 16 CTAs; beyond, the grid form).
// Below, a half's own launches and narrow update (about 15 us) cost more than that gives.
// GB300, 8,000^2 complex64, every panel: 42.2 ms (2,048 rows and more on the grid, whole; the
// cluster's CTAs reading each other's candidates behind its barrier, one row per warp at a
// time) -> 19 ms
constexpr int kWholePanelRows = 2048;
constexpr int kLookRows = 3072;

// cluster size of the cluster panels on this device: 16 CTAs where the device schedules
// such a cluster with the shared memory it needs, else 8, else 0 (grid panels only)
template <class T>
int choose_panel_cluster(int smem_optin, cudaStream_t s) {
  const int dyn = std::max(0, smem_optin - 4096);
  if (cudaFuncSetAttribute(lu_panel_cluster_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) !=
          cudaSuccess ||
      cudaFuncSetAttribute(lu_panel_cluster_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
          cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  for (int c : {16, 8}) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = (size_t)dyn;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, lu_panel_cluster_kernel<T>, &cfg) == cudaSuccess && nc >= 1) return c;
    cudaGetLastError();
  }
  return 0;
}

template <class T>
int lu_max_order(int sms) {
  return (int)((int64_t)sms * (int64_t)kPanelSmem / ((int64_t)kNb * sizeof(cpx<T>)));
}

// the update's tensor map of a (n rows of 2 n floats, 2 ld floats apart)
cudaError_t update_map(float* a, int64_t ld, int n, CUtensorMap* map) {
  void* f = nullptr;
  cudaDriverEntryPointQueryResult found;
  cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &found);
  if (e != cudaSuccess) return e;
  if (found != cudaDriverEntryPointSuccess || !f) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {(cuuint64_t)2 * n, (cuuint64_t)n}, strides[1] = {(cuuint64_t)ld * sizeof(cpx<float>)};
  const cuuint32_t box[2] = {kUBox, kUM}, step[2] = {1, 1};
  const CUresult r = reinterpret_cast<decltype(&cuTensorMapEncodeTiled)>(f)(
      map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, a, dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
      CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <class T>
cudaError_t lu_factor(cpx<T>* a, int64_t ld, int n, const LuWork& w, cudaStream_t s) {
  const int sms = std::min(current_sm_count(), 256);   // lu_panel_kernel polls up to 256 CTAs' keys
  const int n_panels = (n + kNb - 1) / kNb;
  if (lu_panel_grid<T>(n, sms) > sms) return cudaErrorInvalidValue;
  if (n > 65535) return cudaErrorInvalidValue;   // rows and column tags are 16-bit fields of the pivot keys
  // every panel CTA's key slots start with a tag no column has (0xFFFF)
  cudaError_t e = cudaMemsetAsync(w.cand_val, 0xFF, (size_t)2 * sms * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(w.err, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  // no row moves until a panel records its own (a panel that stops early records none)
  e = cudaMemsetAsync(w.n_moves, 0, (size_t)2 * n_panels * sizeof(int), s);
  if (e != cudaSuccess) return e;
  const size_t trsm_smem = (size_t)kNb * (kNb + 1 + 32) * sizeof(cpx<T>);
  const size_t gemm_smem = (size_t)kNb * (65 + 64) * sizeof(cpx<T>);
  // the most shared memory any panel's CTAs take (the grid shrinks in steps as the rows do)
  size_t panel_smem0 = 0;
  for (int pnl = 0; pnl < n_panels; ++pnl) {
    const int R = n - pnl * kNb, G = lu_panel_grid<T>(R, sms), per = (R + G - 1) / G;
    panel_smem0 = std::max(panel_smem0, (size_t)per * cl_pitch(kNb) * sizeof(cpx<T>) + (size_t)per + 16);
  }
  if ((e = cudaFuncSetAttribute(lu_panel_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)panel_smem0)) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(lu_panel_kernel<T>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared)) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(lu_trsm_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)trsm_smem)) !=
      cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(lu_gemm_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem)) !=
      cudaSuccess)
    return e;
  const bool tc_update = sizeof(T) == 4 && w.tc_update;
  if (tc_update && (e = cudaFuncSetAttribute(lu_gemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kUSmem)) != cudaSuccess)
    return e;
  CUtensorMap map = {};
  if (tc_update && n > kNb && (e = update_map(reinterpret_cast<float*>(a), ld, n, &map)) != cudaSuccess) return e;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lu_panel_kernel<T>, kPanelThreads,
                                                         panel_smem0)) != cudaSuccess)
    return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  int smem_optin = 0, dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess)
    return e;
  const int cs = w.panel_cluster ? choose_panel_cluster<T>(smem_optin, s) : 0;
  w.diag[3] = 0;
  w.diag[4] = cs;
  // columns k .. k + kb - 1 as panel list h on stream st; `begun` (or null) is recorded when every
  // CTA of a cluster panel has begun
  auto panel = [&](int k, int kb, int h, bool whole, cudaStream_t st, cudaEvent_t begun) -> cudaError_t {
    const int R = n - k;
    PanelArgs<T> pa{a, ld, n, k, kb, reinterpret_cast<unsigned long long*>(w.cand_val),
                    reinterpret_cast<cpx<T>*>(w.cand_data), w.moves + (size_t)h * kNb, w.n_moves + h, w.err};
    cudaError_t e;
    if (cs > 0 && R <= cluster_panel_rows<T>(cs, kb, smem_optin)) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(kClThreads);
      cfg.dynamicSmemBytes = cl_smem<T>(cs, (R + cs - 1) / cs, kb);
      cfg.stream = st;
      cudaLaunchAttribute at[2];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cs;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      at[1].id = cudaLaunchAttributeLaunchCompletionEvent;
      at[1].val.launchCompletionEvent.event = begun;
      at[1].val.launchCompletionEvent.flags = 0;
      cfg.attrs = at;
      cfg.numAttrs = begun ? 2 : 1;
      if ((e = cudaLaunchKernelEx(&cfg, lu_panel_cluster_kernel<T>, pa)) != cudaSuccess) return e;
      if (whole) ++w.diag[3];
      return cudaSuccess;
    }
    const int G = std::min(lu_panel_grid<T>(R, sms), per_sm * sms);   // all CTAs resident
    const int per = (R + G - 1) / G;
    const size_t psmem = (size_t)per * cl_pitch(kb) * sizeof(cpx<T>) + (size_t)per + 16;
    void* args[] = {&pa};
    w.diag[0] = G;
    w.diag[1] = per_sm;
    w.diag[2] = (int)psmem;
    return cudaLaunchCooperativeKernel((const void*)lu_panel_kernel<T>, dim3(G), dim3(kPanelThreads), args, psmem, st);
  };
  // row moves of `lists` lists from h on: on columns c0 .. c0 + cols - 1, from `skip` on kNb further
  auto moves = [&](int h, int lists, int c0, int cols, int skip, cudaStream_t st) {
    if (cols > 0)
      lu_moves_kernel<T><<<(cols + 15) / 16, 256, 0, st>>>(a, ld, n, c0, cols, skip, w.moves + (size_t)h * kNb,
                                                           w.n_moves + h, lists);
  };
  // block column pnl, whole or in halves, its row moves on its own columns (own) or on all
  auto block = [&](int pnl, bool own, cudaStream_t st, cudaEvent_t begun) -> cudaError_t {
    const int k = pnl * kNb, kb = std::min(kNb, n - k), hb = kNb / 2, c0 = own ? k : 0, cols = own ? kb : n;
    cudaError_t e;
    if (n - k <= kWholePanelRows) {
      if ((e = panel(k, kb, 2 * pnl, true, st, begun)) != cudaSuccess) return e;
      moves(2 * pnl, 1, c0, cols, n, st);
    } else {   // kb = kNb
      if ((e = panel(k, hb, 2 * pnl, false, st, begun)) != cudaSuccess) return e;
      moves(2 * pnl, 1, c0, cols, n, st);
      lu_trsm_kernel<T><<<1, 256, trsm_smem, st>>>(a, ld, k + kb, k, hb);
      lu_gemm_kernel<T><<<dim3(1, (n - k - hb + 63) / 64), 256, gemm_smem, st>>>(a, ld, n, k + kb, k, hb);
      if ((e = panel(k + hb, hb, 2 * pnl + 1, false, st, nullptr)) != cudaSuccess) return e;
      moves(2 * pnl + 1, 1, c0, cols, n, st);
    }
    return cudaGetLastError();
  };
  // the update of ct tiles of columns from cf on by panel k, on at most `ctas` CTAs
  auto update = [&](int k, int cf, int ct, int ctas, cudaStream_t st) {
    const int rt = (n - k - kNb + kUM - 1) / kUM;
    if constexpr (sizeof(T) == 4)
      lu_gemm_tc_kernel<<<grid_for((int64_t)rt * ct, 1, ctas), kUThreads, kUSmem, st>>>(map, a, ld, n, k, cf, ct, w.err);
  };
  // the second stream joined again when the factorization stops between its fork and its join
  struct Fork {
    const LuWork& w;
    cudaStream_t s;
    bool open = false;
    ~Fork() {
      if (open && cudaEventRecord(w.ev[2], w.side) == cudaSuccess) cudaStreamWaitEvent(s, w.ev[2], 0);
    }
  } fork{w, s};
  bool done = false;   // block column pnl was factored ahead
  for (int pnl = 0; pnl < n_panels; ++pnl) {
    const int k = pnl * kNb, kb = std::min(kNb, n - k), k1 = k + kb, rest = n - k1;
    if (!done) {
      if ((e = block(pnl, false, s, nullptr)) != cudaSuccess) return e;
    } else {
      moves(2 * pnl, 2, 0, n - kb, k, s);   // the other columns, behind their update
    }
    done = false;
    if (rest > 0) {   // kb = kNb
      lu_trsm_kernel<T><<<(rest + 31) / 32, 256, trsm_smem, s>>>(a, ld, n, k, kb);
      const int ct = (rest + kNb - 1) / kNb;
      // Look-ahead: the next block column's update and factorization on the second stream, on one
      // cluster, beside the rest of the update on the other SMs, which starts when the panel's
      // CTAs have begun: a cluster needs its SMs in one place, before the update's CTAs take them.
      // (The update reads nothing that the panel writes.)  From kLookRows rows, below which the
      // hand-over costs what the overlap gives.  GB300, 8,000^2: 35.3 -> 29.2 ms (32.9 with the
      // update released by the narrow update's end instead).
      done = tc_update && cs > 0 && rest >= kLookRows && rest <= cluster_panel_rows<T>(cs, kNb / 2, smem_optin);
      if (done) {
        if ((e = cudaEventRecord(w.ev[0], s)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(w.side, w.ev[0], 0)) != cudaSuccess)
          return e;
        fork.open = true;
        update(k, k1, 1, sms, w.side);
        if (w.fail_forked()) return cudaErrorLaunchOutOfResources;
        if ((e = block(pnl + 1, true, w.side, w.ev[1])) != cudaSuccess ||
            (e = cudaEventRecord(w.ev[2], w.side)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(s, w.ev[1], 0)) != cudaSuccess)
          return e;
        update(k, k1 + kNb, ct - 1, sms - cs, s);
        if ((e = cudaStreamWaitEvent(s, w.ev[2], 0)) != cudaSuccess) return e;
        fork.open = false;
      } else if (tc_update) {
        update(k, k1, ct, sms, s);
      } else {
        lu_gemm_kernel<T><<<dim3((rest + 63) / 64, (rest + 63) / 64), 256, gemm_smem, s>>>(a, ld, n, n, k, kb);
      }
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const size_t osmem = (size_t)n * sizeof(unsigned short);
  if ((e = cudaFuncSetAttribute(lu_order_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)osmem)) !=
      cudaSuccess)
    return e;
  lu_order_kernel<<<1, 256, osmem, s>>>(n, 2 * n_panels, w.moves, w.n_moves, w.perm);
  return cudaGetLastError();
}

template <class T>
cudaError_t lu_solve(const cpx<T>* a, int64_t ld, int n, const LuWork& w, cpx<T>* x, cpx<T>* y, cudaStream_t s) {
  constexpr size_t smem = subst_smem<T>();
  const size_t bytes = (size_t)n * Solved<T>::kWords * sizeof(unsigned long long);
  unsigned long long* words[2] = {w.words, w.words + (size_t)n * Solved<T>::kWords};
  int G = std::min((n + kNb - 1) / kNb, current_sm_count());
  const int* order = w.perm;
  const int* none = nullptr;
  const cpx<T>* xc = x;
  const cpx<T>* yc = y;
  int* err = w.err;
  cudaError_t e;
  // one block row: no CTA waits for another, and no word is read
  const bool coop = G > 1;
  if (coop && (e = cudaMemsetAsync(w.words, 0, 2 * bytes, s)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(lu_substitute_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(lu_substitute_kernel<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem)) != cudaSuccess)
    return e;
  auto launch = [&](const void* f, void** args) {
    return coop ? cudaLaunchCooperativeKernel(f, dim3(G), dim3(256), args, smem, s)
                : cudaLaunchKernel(f, dim3(G), dim3(256), args, smem, s);
  };
  void* fwd[] = {&a, &ld, &n, &order, &xc, &y, &words[0], &err};
  if ((e = launch((const void*)lu_substitute_kernel<T, false>, fwd)) != cudaSuccess) return e;
  void* bwd[] = {&a, &ld, &n, &none, &yc, &x, &words[1], &err};
  return launch((const void*)lu_substitute_kernel<T, true>, bwd);
}

cudaError_t residual_f64(const void* z, int64_t ld, int n, const void* x, const void* b, void* r, double* sums,
                         cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(sums, 0, 2 * sizeof(double), s);
  if (e != cudaSuccess) return e;
  residual_kernel<<<grid_for(n, 8, 8 * current_sm_count()), 256, 0, s>>>(
      reinterpret_cast<const cpx<double>*>(z), ld, n, reinterpret_cast<const cpx<double>*>(x),
      reinterpret_cast<const cpx<double>*>(b), reinterpret_cast<cpx<double>*>(r), sums);
  return cudaGetLastError();
}

cudaError_t residual_f32(const void* z, int64_t ld, int n, const void* x, const void* b, double* sums,
                         cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(sums, 0, 2 * sizeof(double), s);
  if (e != cudaSuccess) return e;
  residual32_kernel<<<grid_for(n, 8, 8 * current_sm_count()), 256, 0, s>>>(
      reinterpret_cast<const cpx<float>*>(z), ld, n, reinterpret_cast<const cpx<float>*>(x),
      reinterpret_cast<const cpx<float>*>(b), sums);
  return cudaGetLastError();
}

template <class TD, class TS>
cudaError_t copy_matrix(const void* src, int64_t ld, int n, void* dst, int64_t ld_dst, cudaStream_t s) {
  copy_matrix_kernel<TD, TS><<<dim3(grid_for(n, 256, 64), std::min(n, 65535)), 256, 0, s>>>(
      reinterpret_cast<const cpx<TS>*>(src), ld, n, reinterpret_cast<cpx<TD>*>(dst), ld_dst);
  return cudaGetLastError();
}

template <class TD, class TS>
cudaError_t copy_vector(const void* src, int n, void* dst, cudaStream_t s) {
  copy_vector_kernel<TD, TS><<<grid_for(n, 256, 4 * current_sm_count()), 256, 0, s>>>(
      reinterpret_cast<const cpx<TS>*>(src), n, reinterpret_cast<cpx<TD>*>(dst));
  return cudaGetLastError();
}

cudaError_t add_correction(void* x, const void* d, int n, double* sums, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(sums, 0, 2 * sizeof(double), s);
  if (e != cudaSuccess) return e;
  add_correction_kernel<<<grid_for(n, 256, 4 * current_sm_count()), 256, 0, s>>>(
      reinterpret_cast<cpx<double>*>(x), reinterpret_cast<const cpx<float>*>(d), n, sums);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_excitation(int kind, int n_el, int n_basis, int m, int port, const void* in, const double* q,
                              void* out, cudaStream_t s) {
  const cpx<double>* qd = reinterpret_cast<const cpx<double>*>(q);
  const int items = kind == 2 ? n_el : n_el * m;
  const int blocks = (items + 255) / 256;
  if (kind == 0)
    reduced_excitation_kernel<T><<<blocks, 256, 0, s>>>(n_el, n_basis, m, reinterpret_cast<const cpx<T>*>(in), qd,
                                                        reinterpret_cast<cpx<T>*>(out));
  else if (kind == 1)
    port_excitation_kernel<T><<<blocks, 256, 0, s>>>(n_el, m, port, reinterpret_cast<const cpx<T>*>(in), qd,
                                                     reinterpret_cast<cpx<T>*>(out));
  else
    port_currents_kernel<T><<<blocks, 256, 0, s>>>(n_el, m, port, reinterpret_cast<const cpx<T>*>(in), qd,
                                                   reinterpret_cast<cpx<T>*>(out));
  return cudaGetLastError();
}

template int lu_max_order<float>(int);
template int lu_max_order<double>(int);
template cudaError_t lu_factor<float>(cpx<float>*, int64_t, int, const LuWork&, cudaStream_t);
template cudaError_t lu_factor<double>(cpx<double>*, int64_t, int, const LuWork&, cudaStream_t);
template cudaError_t lu_solve<float>(const cpx<float>*, int64_t, int, const LuWork&, cpx<float>*, cpx<float>*,
                                     cudaStream_t);
template cudaError_t lu_solve<double>(const cpx<double>*, int64_t, int, const LuWork&, cpx<double>*, cpx<double>*,
                                      cudaStream_t);
template cudaError_t copy_matrix<float, double>(const void*, int64_t, int, void*, int64_t, cudaStream_t);
template cudaError_t copy_matrix<float, float>(const void*, int64_t, int, void*, int64_t, cudaStream_t);
template cudaError_t copy_matrix<double, double>(const void*, int64_t, int, void*, int64_t, cudaStream_t);
template cudaError_t copy_vector<float, double>(const void*, int, void*, cudaStream_t);
template cudaError_t copy_vector<double, float>(const void*, int, void*, cudaStream_t);
template cudaError_t copy_vector<float, float>(const void*, int, void*, cudaStream_t);
template cudaError_t copy_vector<double, double>(const void*, int, void*, cudaStream_t);
template cudaError_t launch_excitation<float>(int, int, int, int, int, const void*, const double*, void*,
                                              cudaStream_t);
template cudaError_t launch_excitation<double>(int, int, int, int, int, const void*, const double*, void*,
                                               cudaStream_t);

}  // namespace cfft
