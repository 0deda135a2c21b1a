// Dense inverse of the coarsest AMG level: Gauss-Jordan elimination with partial
// pivoting, in place, in panels of kNb columns.
//
// The elimination works on [M | I].  After step p, column p of M is a unit vector and
// column orig(p) of X (the row of I that the pivot swap brought to row p) is the only new
// nonzero one, so one n x n array W holds all that changes: column j is M's column j
// before step j and X's column orig(j) from then on; the columns are put in order at the
// end.  A panel of kNb steps is one launch of a thread-block cluster (k_gj_panel), which
// leaves the kNb multipliers of every row, and one launch over the whole GPU
// (k_gj_update), which applies the panel's swaps and its kNb rank-1 updates to the other
// columns.  Every entry sees the operations of the column-by-column elimination in the
// same order with the same rounding (one fused multiply-add per step), so the inverse of a matrix whose
// pivot rows stay finite is the one that a launch per pivot gave, up to the signs of zeros.
//
// Why panels: one launch per pivot took 11 us (n = 300) to 40 us (n = 1100) because each
// read and wrote 2 n^2 entries and ended with one CTA's search for the next pivot.  The
// four inverses of a 32x16x16 preconditioner (3,315 pivots) went from 133 to 21 ms, those
// of a 256x128 one (1,139 pivots) from 20 to 5 ms.
#include "sparse_util.cuh"

#include <cooperative_groups.h>
#include <algorithm>

namespace fsi {
namespace {

namespace cg = cooperative_groups;

constexpr int kNb = 16;               // panel columns
constexpr int kPanelThreads = 256;
constexpr int kMaxCluster = 16;
constexpr int kLd = kNb + 1;          // row stride of the panel in shared memory

// Magnitudes compared on the bits: an FP64 comparison would take the FP64 pipe as long as
// a multiply-add does.  (For the same reason a zero multiplier is not tested for: fma(-0, u, w)
// is w for every finite pivot row u, up to the sign of a zero.)
// Orders like |x|, 0 for NaN (never a pivot), at least 1 otherwise
__device__ __forceinline__ unsigned long long pivot_key(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
  return b > 0x7FF0000000000000ull ? 0ull : b + 1;
}

// What a CTA tells the others about its pivot candidate (and row p's owner about row p).
struct Offer {
  unsigned long long key;             // pivot_key of the candidate, 0: none
  double inv;                         // 1 / candidate
  int idx;                            // its row
  double w[kNb], l[kNb];              // the row's panel entries and multipliers
};
struct Mail {
  Offer from[kMaxCluster];
  double w[kNb], l[kNb];              // row p
};

// Steps [P0, P0 + nb) on the panel's columns.  The rows are dealt to the cluster's CTAs
// cyclically and stay in shared memory; one cluster barrier per step (the mailboxes
// alternate: a CTA writes those of step s + 2 only after every CTA has arrived at step
// s + 1, that is, has read those of step s).  A step is bound by that barrier and the
// candidate search: 3.4 us a pivot with the panel's loads and stores (11.2 ms for the 3,315 pivots of
// a 32x16x16 build); the panel's own updates are n kNb FP64 FMAs per step,
// which one SM alone could not hide (1.7 FMAs per clock), hence the cluster.
__global__ void __launch_bounds__(kPanelThreads) k_gj_panel(int n, int P0, int nb, const double* __restrict__ Win,
                                                            double* __restrict__ Wout, double* __restrict__ Lg,
                                                            double* __restrict__ sg, int* __restrict__ piv,
                                                            int* __restrict__ fail) {
  extern __shared__ __align__(16) double panel_sm[];
  __shared__ Mail mail[2];
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks(), me = (int)cluster.block_rank();
  const int t = threadIdx.x;
  const int nl = n > me ? (n - me + cs - 1) / cs : 0;   // local row i is row me + i cs
  double* W = panel_sm;
  double* L = panel_sm + (size_t)((n + cs - 1) / cs) * kLd;
  for (int e = t; e < nl * kNb; e += kPanelThreads) {
    const int i = e / kNb, c = e % kNb;
    W[i * kLd + c] = c < nb ? Win[(int64_t)(me + i * cs) * n + P0 + c] : 0.0;
    L[i * kLd + c] = 0.0;
  }
  cluster.sync();   // every CTA has started and holds its rows
  for (int s = 0; s < nb; ++s) {
    const int p = P0 + s;
    Mail& box = mail[s & 1];
    if (t < 32) {
      // largest |W(r, p)| over this CTA's rows r >= p, ties to the lowest row
      const int first = p > me ? (p - me + cs - 1) / cs : 0;
      unsigned long long best = 0;
      int bi = n;
      for (int i = first + t; i < nl; i += 32) {
        const unsigned long long v = pivot_key(W[i * kLd + s]);
        if (v > best) { best = v; bi = me + i * cs; }
      }
      for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long ov = __shfl_xor_sync(0xffffffffu, best, off);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
      }
      const int ci = bi < n ? (bi - me) / cs : -1;
      const int c = t & (kNb - 1);
      const double mine = ci < 0 ? 0.0 : (t < kNb ? W : L)[ci * kLd + c];
      const bool own_p = p % cs == me;
      const double rowp = own_p ? (t < kNb ? W : L)[(p - me) / cs * kLd + c] : 0.0;
      const double inv = 1.0 / __shfl_sync(0xffffffffu, mine, s);
      for (int d = 0; d < cs; ++d) {
        Mail* to = cluster.map_shared_rank(&box, d);
        (t < kNb ? to->from[me].w : to->from[me].l)[c] = mine;
        if (own_p) (t < kNb ? to->w : to->l)[c] = rowp;
      }
      if (t < cs) {
        Mail* to = cluster.map_shared_rank(&box, t);
        to->from[me].key = best;
        to->from[me].idx = bi;
        to->from[me].inv = inv;
      }
    }
    cluster.sync();
    unsigned long long bv = 0;
    int pr = p, who = p % cs;
    for (int d = 0; d < cs; ++d) {
      const unsigned long long v = box.from[d].key;
      const int i = box.from[d].idx;
      if (v > bv || (v == bv && v && i < pr)) { bv = v; pr = i; who = d; }
    }
    const Offer& o = box.from[who];
    const int c = t & (kNb - 1);
    const bool none = bv == 0;   // a NaN column: row p itself, as without a swap; the inverse is refused below
    const double wc = none ? box.w[c] : o.w[c];
    const double inv = none ? 1.0 / box.w[s] : o.inv;
    const double u = c == s ? inv : __dmul_rn(wc, inv);       // the scaled pivot row; X's new column holds 1 / pivot
    if (me == 0 && t == 0) {
      piv[p] = pr;
      sg[s] = inv;
      if (bv <= 1) *fail = 1;                                 // no pivot above 0
    }
    for (int i = t / kNb; i < nl; i += kPanelThreads / kNb) {   // a row's kNb entries are in one warp
      const int r = me + i * cs;
      double* w = W + i * kLd;
      double* l = L + i * kLd;
      const bool swapped = r == pr && pr != p;
      const double f = swapped ? box.w[s] : w[s];
      const double x = swapped ? box.w[c] : w[c];
      __syncwarp(0xffffu << (t & 16));
      if (r == p) {
        w[c] = u;
        l[c] = c == s ? 0.0 : (none ? box.l[c] : o.l[c]);
      } else {
        const double y = c == s ? 0.0 : x;
        w[c] = __fma_rn(-f, u, y);
        if (c == s) l[c] = f;
        else if (swapped) l[c] = box.l[c];
      }
      __syncwarp(0xffffu << (t & 16));
    }
    __syncthreads();
  }
  for (int e = t; e < nl * kNb; e += kPanelThreads) {
    const int i = e / kNb, c = e % kNb;
    const int64_t r = me + i * cs;
    if (c < nb) Wout[r * n + P0 + c] = W[i * kLd + c];
    Lg[r * kNb + c] = L[i * kLd + c];
  }
  cluster.sync();   // no CTA leaves while another may still read what it was sent
}

// The row that the panel's swaps (step p exchanges rows p and piv[p]) brought to row r.
__device__ __forceinline__ int row_before(int r, int P0, int nb, const int* pv) {
  for (int q = nb - 1; q >= 0; --q) {
    const int a = P0 + q, b = pv[q];
    r = r == a ? b : (r == b ? a : r);
  }
  return r;   // for r >= n (a pivot row past the last column) unchanged: no swap names it
}

// The panel's swaps and updates on the other columns: Win -> Wout, one lane per column,
// kRowsPerThread rows per thread.  FP64 bound (kNb n^2 FMAs); each CTA first repeats the kNb
// steps on its columns of the pivot rows (kNb^2 / 2 FMAs per column), so the tile grows
// with n: 64 rows when that still gives several CTAs per SM, 16 for small matrices, which
// would otherwise leave SMs idle.
constexpr int kUpThreads = 128;
template <int RT>
__global__ void __launch_bounds__(kUpThreads) k_gj_update(int n, int P0, int nb, const double* __restrict__ Win,
                                                          double* __restrict__ Wout, const double* __restrict__ Lg,
                                                          const double* __restrict__ sg, const int* __restrict__ piv) {
  __shared__ double U[kNb][32];
  __shared__ double Lp[kNb][kNb], Ls[RT][kNb], sc[kNb];
  __shared__ int pv[kNb], src[RT + kNb];   // source rows of the tile's rows, then of the pivot rows
  const int t = threadIdx.x, lane = t & 31, wq = t >> 5;
  const int c = blockIdx.x * 32 + lane;
  const int r0 = blockIdx.y * RT;
  const int nr = n - r0 < RT ? n - r0 : RT;
  const bool on = c < n && (c < P0 || c >= P0 + nb);
  if (t < kNb) {
    pv[t] = t < nb ? piv[P0 + t] : -1;
    sc[t] = t < nb ? sg[t] : 0.0;
  }
  for (int e = t; e < kNb * kNb; e += kUpThreads)
    Lp[e / kNb][e % kNb] = e / kNb < nb ? Lg[(int64_t)(P0 + e / kNb) * kNb + e % kNb] : 0.0;
  for (int e = t; e < nr * kNb; e += kUpThreads) {
    // a pivot row starts from its value after its own step: its earlier multipliers are masked
    const int r = r0 + e / kNb;
    const bool done = r >= P0 && r < P0 + nb && e % kNb <= r - P0;
    Ls[e / kNb][e % kNb] = done ? 0.0 : Lg[(int64_t)r * kNb + e % kNb];
  }
  __syncthreads();
  for (int i = t; i < nr + kNb; i += kUpThreads)
    src[i < nr ? i : RT + i - nr] = row_before(i < nr ? r0 + i : P0 + i - nr, P0, nb, pv);
  __syncthreads();
  if (wq == 0) {
    double u[kNb];
#pragma unroll
    for (int p = 0; p < kNb; ++p) u[p] = on && p < nb ? Win[(int64_t)src[RT + p] * n + c] : 0.0;
#pragma unroll
    for (int p = 0; p < kNb; ++p) {
      u[p] = __dmul_rn(u[p], sc[p]);
      U[p][lane] = u[p];
#pragma unroll
      for (int q = p + 1; q < kNb; ++q) {
        u[q] = __fma_rn(-Lp[q][p], u[p], u[q]);
      }
    }
  }
  __syncthreads();
  double u[kNb];
#pragma unroll
  for (int p = 0; p < kNb; ++p) u[p] = U[p][lane];
#pragma unroll 4
  for (int i = wq; i < nr; i += kUpThreads / 32) {
    const int in_panel = r0 + i - P0;
    double w = in_panel >= 0 && in_panel < nb ? U[in_panel][lane] : (on ? Win[(int64_t)src[i] * n + c] : 0.0);
#pragma unroll
    for (int p = 0; p < kNb; ++p) {
      w = __fma_rn(-Ls[i][p], u[p], w);
    }
    if (on) Wout[(int64_t)(r0 + i) * n + c] = w;
  }
}

// Rows that are entirely zero become identity rows (one warp per row).
__global__ void k_gj_init(int n, double* __restrict__ M) {
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= n) return;
  bool nz = false;
  for (int c = lane; c < n; c += 32) nz |= M[r * n + c] != 0.0;
  if (!__any_sync(0xffffffffu, nz) && lane == 0) M[r * n + r] = 1.0;
}

// orig[j]: the row of the identity that step j's swap brought to row j (all swaps before undone).
__global__ void k_gj_orig(int n, const int* __restrict__ piv, int* __restrict__ orig) {
  extern __shared__ int gj_pv[];
  for (int i = threadIdx.x; i < n; i += blockDim.x) gj_pv[i] = piv[i];
  __syncthreads();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  int x = gj_pv[j];
  for (int q = j - 1; q >= 0; --q) {
    const int b = gj_pv[q];
    x = x == q ? b : (x == b ? q : x);
  }
  orig[j] = x;
}

// X(r, orig(j)) = W(r, j)
__global__ void k_gj_finish(int n, const double* __restrict__ W, const int* __restrict__ orig, double* __restrict__ X) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n * n) return;
  const int64_t r = e / n;
  X[r * n + orig[e - r * n]] = W[e];
}

size_t panel_smem(int n, int cs) { return sizeof(double) * 2 * (size_t)((n + cs - 1) / cs) * kLd; }

cudaLaunchConfig_t panel_config(int n, int cs, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs);
  cfg.blockDim = dim3(kPanelThreads);
  cfg.dynamicSmemBytes = panel_smem(n, cs);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Cluster size for an n x n inverse: 16 CTAs where the device takes such a cluster (more than
// 8 is opt-in), else 8.  n <= 8192 needs 143 KB of shared memory in a 16-CTA cluster.
int panel_cluster(int n) {
  constexpr int kMaxN16 = 8192;
  static OncePerDevice done;
  static std::atomic<int> big[64];
  once_per_device(done, [](int dev) {
    FSI_CUDA(cudaFuncSetAttribute(k_gj_panel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)panel_smem(kMaxN16, kMaxCluster)));
    int ok = 0;
    if (cudaFuncSetAttribute(k_gj_panel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      cudaLaunchAttribute attr[1];
      cudaLaunchConfig_t cfg = panel_config(kMaxN16, kMaxCluster, attr, nullptr);
      int k = 0;
      ok = cudaOccupancyMaxActiveClusters(&k, k_gj_panel, &cfg) == cudaSuccess && k > 0;
    }
    cudaGetLastError();
    big[dev].store(ok, std::memory_order_relaxed);
  });
  int dev = 0;
  FSI_CUDA(cudaGetDevice(&dev));
  require(big[dev].load(std::memory_order_relaxed) || n <= kMaxN16 / 2, "dense_inverse: matrix too large for this device");
  return big[dev].load(std::memory_order_relaxed) && n > 256 ? kMaxCluster : 8;
}

}  // namespace

bool dense_inverse(int n, double* M, double* Minv, cudaStream_t s) {
  if (n <= 0) return true;
  DBuf<int> flag(1), piv(n), orig(n);
  DBuf<double> W1((size_t)n * n), L((size_t)n * kNb), sc(kNb);
  FSI_CUDA(cudaMemsetAsync(flag.p, 0, sizeof(int), s));
  k_gj_init<<<div_up((int64_t)n * 32, 256), 256, 0, s>>>(n, M);
  FSI_CHECK_LAUNCH();
  const int cs = panel_cluster(n);
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = panel_config(n, cs, attr, s);
  double* in = M;
  double* out = W1.p;
  for (int P0 = 0; P0 < n; P0 += kNb) {
    const int nb = std::min(kNb, n - P0);
    FSI_CUDA(cudaLaunchKernelEx(&cfg, k_gj_panel, n, P0, nb, (const double*)in, out, L.p, sc.p, piv.p, flag.p));
    FSI_CHECK_LAUNCH();
    const unsigned ct = (unsigned)div_up(n, 32);
    if (n >= 1024)
      k_gj_update<64><<<dim3(ct, div_up(n, 64)), kUpThreads, 0, s>>>(n, P0, nb, in, out, L.p, sc.p, piv.p);
    else if (n >= 512)
      k_gj_update<32><<<dim3(ct, div_up(n, 32)), kUpThreads, 0, s>>>(n, P0, nb, in, out, L.p, sc.p, piv.p);
    else
      k_gj_update<16><<<dim3(ct, div_up(n, 16)), kUpThreads, 0, s>>>(n, P0, nb, in, out, L.p, sc.p, piv.p);
    FSI_CHECK_LAUNCH();
    std::swap(in, out);
  }
  k_gj_orig<<<div_up(n, 256), 256, sizeof(int) * n, s>>>(n, piv.p, orig.p);
  FSI_CHECK_LAUNCH();
  k_gj_finish<<<div_up((int64_t)n * n, 256), 256, 0, s>>>(n, in, orig.p, Minv);
  FSI_CHECK_LAUNCH();
  int failed = 0;
  FSI_CUDA(cudaMemcpyAsync(&failed, flag.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  FSI_CUDA(cudaStreamSynchronize(s));
  return failed == 0;
}

}  // namespace fsi
