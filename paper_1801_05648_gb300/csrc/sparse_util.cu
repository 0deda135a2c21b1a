#include "sparse_util.cuh"

#include <algorithm>
#include <climits>
#include <type_traits>

namespace fsi {

namespace {

constexpr int kScanBlock = 1024;

__device__ __forceinline__ long long warp_incl_scan(long long v, int lane) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    long long t = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += t;
  }
  return v;
}

// Exclusive scan of a 1024-element tile; writes block totals.
__global__ void __launch_bounds__(kScanBlock) k_scan_tile(const int* __restrict__ in, int* __restrict__ out, int64_t n,
                                                          long long* __restrict__ bsum) {
  __shared__ long long wsum[32];
  const int64_t i = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  long long v = i < n ? (long long)in[i] : 0;
  long long inc = warp_incl_scan(v, lane);
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    long long t = wsum[lane];
    t = warp_incl_scan(t, lane);
    wsum[lane] = t;
  }
  __syncthreads();
  long long base = w ? wsum[w - 1] : 0;
  if (i < n) out[i] = (int)(base + inc - v);   // total < 2^31, checked on the host
  if (threadIdx.x == kScanBlock - 1) bsum[blockIdx.x] = base + inc;
}

// Exclusive scan of the nb tile totals in place, by one block; bsum[nb] = the total.
__global__ void __launch_bounds__(kScanBlock) k_scan_totals(long long* __restrict__ bsum, int nb) {
  __shared__ long long wsum[32];
  __shared__ long long carry;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int b0 = 0; b0 < nb; b0 += kScanBlock) {
    const int i = b0 + threadIdx.x;
    const long long v = i < nb ? bsum[i] : 0;
    const long long inc = warp_incl_scan(v, lane);
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) wsum[lane] = warp_incl_scan(wsum[lane], lane);
    __syncthreads();
    const long long ex = carry + (w ? wsum[w - 1] : 0) + inc - v;
    if (i < nb) bsum[i] = ex;
    __syncthreads();
    if (threadIdx.x == kScanBlock - 1) carry = ex + v;
    __syncthreads();
  }
  if (threadIdx.x == 0) bsum[nb] = carry;
}

// Tile offsets added, out[n] = the total.
__global__ void __launch_bounds__(kScanBlock) k_scan_add(int* __restrict__ out, int64_t n,
                                                         const long long* __restrict__ bsum, int nb) {
  const int64_t i = (int64_t)blockIdx.x * kScanBlock + threadIdx.x;
  if (i < n) out[i] = (int)(out[i] + bsum[blockIdx.x]);
  if (i == n) out[n] = (int)bsum[nb];
}

// exclusive scan of n ints into out (n + 1 entries); returns the total on the host (three launches,
// one wait)
long long scan_ints(const int* in, int* out, int64_t n, cudaStream_t s) {
  const int nb = div_up(n, kScanBlock);
  DBuf<long long> bsum(nb + 1);
  if (n > 0) {
    k_scan_tile<<<nb, kScanBlock, 0, s>>>(in, out, n, bsum.p);
    FSI_CHECK_LAUNCH();
  }
  k_scan_totals<<<1, kScanBlock, 0, s>>>(bsum.p, nb);
  FSI_CHECK_LAUNCH();
  k_scan_add<<<div_up(n + 1, kScanBlock), kScanBlock, 0, s>>>(out, n, bsum.p, nb);
  FSI_CHECK_LAUNCH();
  long long total = 0;
  FSI_CUDA(cudaMemcpyAsync(&total, bsum.p + nb, sizeof(long long), cudaMemcpyDeviceToHost, s));
  FSI_CUDA(cudaStreamSynchronize(s));
  return total;
}

__device__ __forceinline__ int lower_bound_i(const int* a, int lo, int hi, int key) {
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (a[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}
__device__ __forceinline__ int64_t lower_bound_l(const int* a, int64_t lo, int64_t hi, int key) {
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (a[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// --------------------------------------------------------------- extraction
// One warp per block row.  Rows of a node share their columns as a rule, and the columns
// of a node come together: then the br scalar rows, restricted to the column window, are
// the same list of whole blocks, and the lanes read and write them side by side.  Any
// other block row (a Dirichlet node's identity rows, say) is merged entry by entry by one
// lane.  (One thread per block row merging every row took 22 ms for the 18 class blocks of
// the 32x16x16 operator.)
template <bool FILL>
__global__ void __launch_bounds__(128) k_extract(const int64_t* __restrict__ rp, const int* __restrict__ ci,
                                                 const double* __restrict__ va, int64_t r0, int nbr, int br,
                                                 int64_t c0, int64_t c1, int bc, int* __restrict__ cnt,
                                                 const int* __restrict__ orp, int* __restrict__ oci,
                                                 double* __restrict__ ova) {
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= nbr) return;
  // lanes 0 .. br - 1: the window [from, to) of their scalar row
  int64_t from = 0;
  int len = 0;
  if (lane < br) {
    const int64_t r = r0 + (int64_t)row * br + lane;
    from = lower_bound_l(ci, rp[r], rp[r + 1], (int)c0);
    len = (int)(lower_bound_l(ci, from, rp[r + 1], (int)c1) - from);
  }
  const int64_t f0 = __shfl_sync(0xffffffffu, from, 0);
  const int n0 = __shfl_sync(0xffffffffu, len, 0);
  bool same = !__any_sync(0xffffffffu, lane < br && len != n0) && n0 % bc == 0;
  for (int q = 0; q < br && same; ++q) {
    const int64_t f = __shfl_sync(0xffffffffu, from, q);
    bool ok = true;
    for (int e = lane; e < n0; e += 32) {
      const int c = ci[f + e];
      // row 0: blocks of consecutive, aligned columns; other rows: row 0's columns
      ok = ok && (q == 0 ? (c - (int)c0) % bc == e % bc && c == ci[f0 + e - e % bc] + e % bc : c == ci[f0 + e]);
    }
    same = __all_sync(0xffffffffu, ok);
  }
  if (same) {
    const int nb = n0 / bc;
    if (!FILL) {
      if (lane == 0) cnt[row] = nb;
      return;
    }
    const int64_t o = orp[row];
    for (int e = lane; e < nb; e += 32) oci[o + e] = (int)((ci[f0 + (int64_t)e * bc] - c0) / bc);
    for (int q = 0; q < br; ++q) {
      const int64_t f = __shfl_sync(0xffffffffu, from, q);
      for (int e = lane; e < n0; e += 32) ova[(o + e / bc) * (br * bc) + q * bc + e % bc] = va[f + e];
    }
    return;
  }
  int64_t ptr[6], end[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    ptr[q] = __shfl_sync(0xffffffffu, from, q);
    end[q] = ptr[q] + __shfl_sync(0xffffffffu, len, q);
  }
  if (lane != 0) return;
  int count = 0;
  int64_t outpos = FILL ? orp[row] : 0;
  while (true) {
    int best = INT_MAX;
    for (int q = 0; q < br; ++q)
      if (ptr[q] < end[q]) {
        int b = (int)((ci[ptr[q]] - c0) / bc);
        if (b < best) best = b;
      }
    if (best == INT_MAX) break;
    if (FILL) {
      double* blk = ova + outpos * (int64_t)(br * bc);
      for (int t = 0; t < br * bc; ++t) blk[t] = 0.0;
      oci[outpos] = best;
      for (int q = 0; q < br; ++q)
        while (ptr[q] < end[q] && (int)((ci[ptr[q]] - c0) / bc) == best) {
          blk[q * bc + (int)((ci[ptr[q]] - c0) % bc)] = va[ptr[q]];
          ++ptr[q];
        }
      ++outpos;
    } else {
      for (int q = 0; q < br; ++q)
        while (ptr[q] < end[q] && (int)((ci[ptr[q]] - c0) / bc) == best) ++ptr[q];
    }
    ++count;
  }
  if (!FILL) cnt[row] = count;
}

// --------------------------------------------------------------- add
// One warp per block row: equal patterns side by side, others merged by one lane.
template <bool FILL>
__global__ void __launch_bounds__(128) k_add(int nbr, int bsz, const int* __restrict__ arp,
                                             const int* __restrict__ aci, const double* __restrict__ ava,
                                             const int* __restrict__ brp, const int* __restrict__ bci,
                                             const double* __restrict__ bva, double alpha, int* __restrict__ cnt,
                                             const int* __restrict__ crp, int* __restrict__ cci,
                                             double* __restrict__ cva) {
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= nbr) return;
  int ia = arp[row], ea = arp[row + 1], ib = brp[row], eb = brp[row + 1];
  bool same = ea - ia == eb - ib;
  if (same) {
    for (int e = lane; e < ea - ia; e += 32) same = same && aci[ia + e] == bci[ib + e];
    same = __all_sync(0xffffffffu, same);
  }
  if (same) {
    if (!FILL) {
      if (lane == 0) cnt[row] = ea - ia;
      return;
    }
    const int64_t o = crp[row];
    for (int e = lane; e < ea - ia; e += 32) cci[o + e] = aci[ia + e];
    for (int64_t e = lane; e < (int64_t)(ea - ia) * bsz; e += 32)
      cva[o * bsz + e] = ava[(int64_t)ia * bsz + e] + alpha * bva[(int64_t)ib * bsz + e];
    return;
  }
  if (lane != 0) return;
  int count = 0;
  int pos = FILL ? crp[row] : 0;
  while (ia < ea || ib < eb) {
    int ca = ia < ea ? aci[ia] : INT_MAX;
    int cb = ib < eb ? bci[ib] : INT_MAX;
    int c = ca < cb ? ca : cb;
    if (FILL) {
      double* o = cva + (int64_t)pos * bsz;
      for (int t = 0; t < bsz; ++t) o[t] = 0.0;
      if (ca == c) for (int t = 0; t < bsz; ++t) o[t] += ava[(int64_t)ia * bsz + t];
      if (cb == c) for (int t = 0; t < bsz; ++t) o[t] += alpha * bva[(int64_t)ib * bsz + t];
      cci[pos] = c;
      ++pos;
    }
    if (ca == c) ++ia;
    if (cb == c) ++ib;
    ++count;
  }
  if (!FILL) cnt[row] = count;
}

// --------------------------------------------------------------- transpose
__global__ void k_count_cols(int64_t nnzb, const int* __restrict__ ci, int* __restrict__ cnt) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < nnzb) atomicAdd(cnt + ci[k], 1);
}
__global__ void k_row_of_block(int nbr, const int* __restrict__ rp, int* __restrict__ rowof) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= nbr) return;
  for (int k = rp[row]; k < rp[row + 1]; ++k) rowof[k] = row;
}
__global__ void k_scatter_t(int64_t nnzb, const int* __restrict__ ci, const int* __restrict__ rowof,
                            const int* __restrict__ trp, int* __restrict__ cursor, int* __restrict__ trow,
                            int* __restrict__ tsrc) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nnzb) return;
  const int c = ci[k];
  const int pos = trp[c] + atomicAdd(cursor + c, 1);
  trow[pos] = rowof[k];
  tsrc[pos] = (int)k;
}
// Each segment of (distinct) keys sorted with its payload, from (key, pay) to (okey, opay):
// an entry's place is the number of smaller keys.  `group` threads (a warp or the block)
// per segment, the keys in shared memory where they fit.  (An insertion sort per thread
// took 49 ms for the transposes of the 32x16x16 hierarchies.)
constexpr int kSortThreads = 128, kSortKeys = 2048;
__global__ void __launch_bounds__(kSortThreads) k_sort_segments(int nseg, int group, const int* __restrict__ off,
                                                                const int* __restrict__ key,
                                                                const int* __restrict__ pay, int* __restrict__ okey,
                                                                int* __restrict__ opay) {
  __shared__ __align__(16) int sk[kSortKeys];
  const int per = kSortThreads / group, g = threadIdx.x / group, t = threadIdx.x % group;
  const int cap = kSortKeys / per;
  const int seg = blockIdx.x * per + g;
  int lo = 0, n = 0;
  if (seg < nseg) {
    lo = off[seg];
    n = off[seg + 1] - lo;
  }
  const bool fits = n <= cap;
  int* k = sk + g * cap;
  if (fits)
    for (int e = t; e < n; e += group) k[e] = key[lo + e];
  __syncthreads();
  for (int e = t; e < n; e += group) {
    const int v = fits ? k[e] : key[lo + e];
    int rank = 0;
    if (fits) for (int f = 0; f < n; ++f) rank += k[f] < v;
    else for (int f = 0; f < n; ++f) rank += __ldg(key + lo + f) < v;
    okey[lo + rank] = v;
    if (pay) opay[lo + rank] = pay[lo + e];
  }
}
__global__ void k_gather_t(int64_t nnzb, int br, int bc, const int* __restrict__ tsrc, const double* __restrict__ va,
                           double* __restrict__ tva) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nnzb) return;
  const double* s = va + (int64_t)tsrc[k] * br * bc;
  double* d = tva + k * br * bc;
  // source block br x bc row-major -> destination bc x br row-major
  for (int i = 0; i < br; ++i)
    for (int j = 0; j < bc; ++j) d[j * br + i] = s[i * bc + j];
}

// --------------------------------------------------------------- SpGEMM
constexpr int kHashSize = 1024;      // per warp, shared memory (2 x 4 x 4 KB per block)
constexpr int kWarpsPerBlock = 4;

__device__ __forceinline__ unsigned hash_slot(int key) { return ((unsigned)key * 2654435761u) & (kHashSize - 1); }

// returns 1 when key was newly inserted, 0 when present, -1 when the table is
// full (every slot probed once: the loop always ends)
__device__ __forceinline__ int hash_insert(int* table, int key) {
  unsigned h = hash_slot(key);
  for (int probe = 0; probe < kHashSize; ++probe) {
    int prev = atomicCAS(table + h, -1, key);
    if (prev == -1) return 1;
    if (prev == key) return 0;
    h = (h + 1) & (kHashSize - 1);
  }
  return -1;
}

// Symbolic pass, WPR warps per row of A (the whole block, for products of few long
// rows, or one).  FILL = false: count unique block columns (flag overflow; info[1] = the
// longest row).  FILL = true: write them sorted.  Each warp takes batches of 32 entries of
// A's row and reads their B rows' bounds together; `sub` lanes then take one B row each
// time (about its mean length), so that several short B rows are inserted at once.
template <bool FILL, int WPR>
__global__ void __launch_bounds__(kWarpsPerBlock * 32) k_spgemm_sym(int nbr, int sub, const int* __restrict__ arp,
                                                                    const int* __restrict__ aci,
                                                                    const int* __restrict__ brp,
                                                                    const int* __restrict__ bci, int* __restrict__ cnt,
                                                                    const int* __restrict__ crp, int* __restrict__ cci,
                                                                    int* __restrict__ info) {
  static_assert(WPR == 1 || WPR == kWarpsPerBlock, "a warp or the block per row");
  constexpr int ROWS = kWarpsPerBlock / WPR, T = WPR * 32;
  __shared__ int table[ROWS][kHashSize];
  __shared__ __align__(16) int list[ROWS][FILL ? kHashSize : 4];
  __shared__ int found[ROWS], wide[ROWS], place[ROWS];
  const int g = threadIdx.x / T, t = threadIdx.x % T, lane = threadIdx.x & 31, wr = t / 32;
  const int row = blockIdx.x * ROWS + g;
  if (row >= nbr) return;   // a row's threads leave together
  auto sync = [] { if constexpr (WPR == 1) __syncwarp(); else __syncthreads(); };
  int* tb = table[g];
  for (int e = t; e < kHashSize; e += T) tb[e] = -1;
  if (t == 0) found[g] = wide[g] = place[g] = 0;
  sync();
  const int ka = arp[row], ke = arp[row + 1];
  const int groups = 32 / sub, q0 = lane / sub, l = lane % sub;
  for (int k0 = ka + 32 * wr; k0 < ke; k0 += T) {
    int lo = 0, hi = 0;
    if (k0 + lane < ke) {
      const int kk = aci[k0 + lane];
      lo = brp[kk];
      hi = brp[kk + 1];
    }
    const int nk = ke - k0 < 32 ? ke - k0 : 32;
    bool stop = false;
    for (int j = 0; j < nk && !stop; j += groups) {
      int a = __shfl_sync(0xffffffffu, lo, (j + q0) & 31), b = __shfl_sync(0xffffffffu, hi, (j + q0) & 31);
      if (j + q0 >= nk) b = a;
      int fresh = 0, full = 0;
      for (int q = a + l; q < b; q += sub) {
        const int r = hash_insert(tb, bci[q]);
        if (r < 0) { full = 1; break; }
        fresh += r;
      }
      fresh = __reduce_add_sync(0xffffffffu, fresh);
      full = __any_sync(0xffffffffu, full);
      // over 3/4 of the table in use, or a failed insert: the row does not fit
      int total = 0;
      if (lane == 0) {
        total = (fresh ? atomicAdd(&found[g], fresh) : *(volatile int*)&found[g]) + fresh;
        if (full || total > kHashSize * 3 / 4) *(volatile int*)&wide[g] = 1;
      }
      stop = __shfl_sync(0xffffffffu, lane == 0 && (full || total > kHashSize * 3 / 4), 0);
    }
    // another warp of the row may be setting the flag: the lanes' looks at it are pooled, so that all 32 leave
    // here or none does
    if (__any_sync(0xffffffffu, stop || *(volatile int*)&wide[g])) break;
  }
  sync();
  if (wide[g]) {
    if (t == 0) atomicExch(info, 1);
    return;
  }
  if (!FILL) {
    if (t == 0) {
      const int total = found[g];
      cnt[row] = total;
      if (total > __ldcg(info + 1)) atomicMax(info + 1, total);
    }
    return;
  }
  // compact the table (in any order: the ranks put it in order)
  int* ls = list[g];
  for (int t0 = 32 * wr; t0 < kHashSize; t0 += T) {
    const int v = tb[t0 + lane];
    const unsigned m = __ballot_sync(0xffffffffu, v != -1);
    int base = 0;
    if (lane == 0) base = atomicAdd(&place[g], __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (v != -1) ls[base + __popc(m & ((1u << lane) - 1))] = v;
  }
  sync();
  const int n = found[g];
  if (t < 4 && n + t < kHashSize) ls[n + t] = INT_MAX;   // pad the last group of four
  sync();
  const int out0 = crp[row];
  for (int e = t; e < n; e += T) {
    const int v = ls[e];
    int rank = 0;
    for (int f = 0; f < n; f += 4) {
      const int4 x = *reinterpret_cast<const int4*>(ls + f);
      rank += (x.x < v) + (x.y < v) + (x.z < v) + (x.w < v);
    }
    cci[out0 + rank] = v;
  }
}

// Numeric pass: C(row, J) = sum over k of A(row, k) B(k, J), every entry summed over k in
// increasing order.  One warp takes a chunk (blockIdx.y) of `cap` consecutive block
// columns of a row, with the sums in shared memory.  For a batch of up to 32 entries k the
// lanes first cut each B row to the chunk's columns, then find where each of the batch's
// remaining entries goes (binary search in the chunk's columns, all lanes on different
// entries), and then add the B rows one after the other, lanes side by side on (entry,
// component), several loads ahead of the sums.  Bound by the FP64 pipe (BK FMAs per match
// and component) as long as an SM holds enough warps to hide the loads: about 5 KB of sums a warp let 32 of them
// fit, and chunks are cut smaller where rows x chunks would make fewer than 16.  All products of a 32x16x16 preconditioner build:
// 24 ms; one lane per C entry searching every B row took 125 ms, whole rows per warp (two
// CTAs' worth of sums per SM) 66 ms.
constexpr int kSlots = 256;          // matches placed at a time
constexpr int kNumWarps = 4;
struct NumScratch {
  int pref[33], start[32];
  short slot[kSlots];
};
template <int BR, int BC>
__host__ __device__ constexpr size_t num_smem_per_warp(int cap) {
  return ((size_t)cap * BR * BC * sizeof(double) + sizeof(int) * (size_t)cap + sizeof(NumScratch) + 15) / 16 * 16;
}

template <int BR, int BK, int BC>
__global__ void __launch_bounds__(kNumWarps * 32) k_spgemm_num(int nbr, int cap, const int* __restrict__ arp,
                                                               const int* __restrict__ aci,
                                                               const double* __restrict__ ava,
                                                               const int* __restrict__ brp,
                                                               const int* __restrict__ bci,
                                                               const double* __restrict__ bva,
                                                               const int* __restrict__ crp,
                                                               const int* __restrict__ cci,
                                                               double* __restrict__ cva) {
  constexpr int BS = BR * BC, U = BK <= 3 ? 4 : 2;   // U items per lane loaded before their sums
  extern __shared__ __align__(16) unsigned char num_sm[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * kNumWarps + w;
  if (row >= nbr) return;
  const int c0 = crp[row] + blockIdx.y * cap;
  const int nc = min(crp[row + 1] - c0, cap);
  if (nc <= 0) return;
  unsigned char* base = num_sm + (size_t)w * num_smem_per_warp<BR, BC>(cap);
  double* acc = reinterpret_cast<double*>(base);
  int* cols = reinterpret_cast<int*>(acc + (size_t)cap * BS);
  NumScratch& sc = *reinterpret_cast<NumScratch*>(cols + cap);
  for (int e = lane; e < nc; e += 32) cols[e] = cci[c0 + e];
  for (int e = lane; e < nc * BS; e += 32) acc[e] = 0.0;
  __syncwarp();
  const int first = cols[0], last = cols[nc - 1];
  const bool part = nc < crp[row + 1] - crp[row];
  const int ka = arp[row], ke = arp[row + 1];
  for (int k0 = ka; k0 < ke; k0 += 32) {
    const int nk = ke - k0 < 32 ? ke - k0 : 32;
    int len = 0;
    if (lane < nk) {
      const int kk = aci[k0 + lane];
      int lo = brp[kk], hi = brp[kk + 1];
      if (part) {
        lo = lower_bound_i(bci, lo, hi, first);
        hi = lower_bound_i(bci, lo, hi, last + 1);
      }
      len = hi - lo;
      sc.start[lane] = lo;
    }
    int inc = len;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc += t;
    }
    sc.pref[lane + 1] = inc;
    if (lane == 0) sc.pref[0] = 0;
    __syncwarp();
    const int tot = sc.pref[32];
    int k = 0;                                     // the B row that the first match of the part belongs to
    for (int m0 = 0; m0 < tot; m0 += kSlots) {
      const int m1 = min(m0 + kSlots, tot);
      for (int m = m0 + lane; m < m1; m += 32) {
        int lo = 0, hi = nk;                       // last k with pref[k] <= m
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (sc.pref[mid] <= m) lo = mid; else hi = mid;
        }
        const int J = __ldg(bci + sc.start[lo] + (m - sc.pref[lo]));
        sc.slot[m - m0] = (short)lower_bound_i(cols, 0, nc, J);   // present: C's pattern covers every match
      }
      __syncwarp();
      for (; k < nk; ++k) {
        const int f = max(sc.pref[k], m0), l = min(sc.pref[k + 1], m1);
        const double* a = ava + (int64_t)(k0 + k) * BR * BK;
        const double* b = bva + ((int64_t)sc.start[k] + (f - sc.pref[k])) * BK * BC;
        const int ne = (l - f) * BS;
        for (int e0 = lane; e0 < ne; e0 += 32 * U) {
          double av[U][BK], bv[U][BK];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int e = e0 + 32 * u;
            if (e < ne) {
              const int m = e / BS, t = e % BS, i = t / BC, j = t % BC;
#pragma unroll
              for (int q = 0; q < BK; ++q) {
                av[u][q] = __ldg(a + i * BK + q);
                bv[u][q] = __ldg(b + (m * BK + q) * BC + j);
              }
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int e = e0 + 32 * u;
            if (e < ne) {
              double* s = acc + sc.slot[f - m0 + e / BS] * BS + e % BS;
              double sum = *s;
#pragma unroll
              for (int q = 0; q < BK; ++q) sum += av[u][q] * bv[u][q];
              *s = sum;
            }
          }
        }
        __syncwarp();
        if (sc.pref[k + 1] > m1) break;            // the row goes on in the next part
      }
    }
    __syncwarp();
  }
  for (int e = lane; e < nc * BS; e += 32) cva[(int64_t)c0 * BS + e] = acc[e];
}

// --------------------------------------------------------------- misc
__global__ void k_scale_rows(int nbr, int br, int bc, const int* __restrict__ rp, double* __restrict__ va,
                             const double* __restrict__ w) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= nbr) return;
  for (int k = rp[row]; k < rp[row + 1]; ++k)
    for (int i = 0; i < br; ++i)
      for (int j = 0; j < bc; ++j) va[((int64_t)k * br + i) * bc + j] *= w[(int64_t)row * br + i];
}
__global__ void k_scale_all(int64_t n, double alpha, double* __restrict__ va) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) va[i] *= alpha;
}
__global__ void k_delta16(int nbr, const int* __restrict__ rp, const int* __restrict__ ci, int16_t* __restrict__ d,
                          int* __restrict__ overflow) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= nbr) return;
  for (int k = rp[row]; k < rp[row + 1]; ++k) {
    const int off = ci[k] - row;
    if (off < -32768 || off > 32767) { atomicExch(overflow, 1); return; }
    d[k] = (int16_t)off;
  }
}
// Slot table of a two-matrix SpMV (block rows of A1 next to those of A2): within
// each window of 32 block rows, the rows by decreasing A1 length, then decreasing A2
// length, ties in row order; record {row | len1 << 24, first A1 block, first A2 block,
// len2}.  One warp per window ranks its rows by counting.  *bad = 1 if an A1 row is
// longer than 255 blocks (the record cannot hold it).
__global__ void k_pair_order(int nbr, const int* __restrict__ rp1, const int* __restrict__ rp2,
                             int4* __restrict__ ord, int* __restrict__ bad) {
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int kb1 = 0, kb2 = 0, l1 = -1, l2 = -1;     // lanes past the end rank last and write nothing
  if (row < nbr) {
    kb1 = rp1[row];
    l1 = rp1[row + 1] - kb1;
    kb2 = rp2[row];
    l2 = rp2[row + 1] - kb2;
    if (l1 > 255) atomicExch(bad, 1);
  }
  int rank = 0;
  for (int j = 0; j < 32; ++j) {
    const int a = __shfl_sync(0xffffffffu, l1, j), b = __shfl_sync(0xffffffffu, l2, j);
    rank += (a > l1 || (a == l1 && (b > l2 || (b == l2 && j < lane)))) ? 1 : 0;
  }
  if (row < nbr && l1 <= 255) ord[row - lane + rank] = make_int4((int)row | (l1 << 24), kb1, kb2, l2);
}
__global__ void k_point_diag(int nbr, int b, const int* __restrict__ rp, const int* __restrict__ ci,
                             const double* __restrict__ va, double* __restrict__ diag) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= nbr) return;
  const int pos = lower_bound_i(ci, rp[row], rp[row + 1], row);
  const bool has = pos < rp[row + 1] && ci[pos] == row;
  for (int i = 0; i < b; ++i) diag[(int64_t)row * b + i] = has ? va[((int64_t)pos * b + i) * b + i] : 0.0;
}
__global__ void k_invert_nonzero(int64_t n, const double* __restrict__ d, double* __restrict__ o) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) o[i] = d[i] != 0.0 ? 1.0 / d[i] : 0.0;
}
__global__ void k_to_f32(int64_t n, const double* __restrict__ a, float* __restrict__ b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (float)a[i];
}
// FP32 copy of 3 x 3 blocks in the planar layout: value t of block k goes to
// 4k + t (t < 4), 4 nnzb + 4k + t - 4 (t < 8) or 8 nnzb + k (t = 8).
__global__ void k_to_f32_planar9(int64_t nnzb, const double* __restrict__ a, float* __restrict__ b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 9 * nnzb) return;
  const int64_t k = i / 9;
  const int t = (int)(i - 9 * k);
  const int64_t o = t < 4 ? 4 * k + t : (t < 8 ? 4 * nnzb + 4 * k + (t - 4) : 8 * nnzb + k);
  b[o] = (float)a[i];
}
// one warp per block row
__global__ void k_to_dense(int nbr, int br, int bc, int ncols, const int* __restrict__ rp, const int* __restrict__ ci,
                           const double* __restrict__ va, double* __restrict__ D) {
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= nbr) return;
  const int k0 = rp[row], bs = br * bc, cnt = (rp[row + 1] - k0) * bs;
  for (int e = lane; e < cnt; e += 32) {
    const int k = k0 + e / bs, i = e % bs / bc, j = e % bc;
    D[((int64_t)row * br + i) * ncols + (int64_t)ci[k] * bc + j] = va[(int64_t)k0 * bs + e];
  }
}

template <class F>
void spgemm_dispatch(int br, int bk, int bc, F&& f) {
#define FSI_G(a, b, c) if (br == a && bk == b && bc == c) { f.template operator()<a, b, c>(); return; }
  // A * P_tent / A * P (b x b times b x k)
  FSI_G(1, 1, 1) FSI_G(2, 2, 2) FSI_G(3, 3, 3) FSI_G(2, 2, 3) FSI_G(3, 3, 6) FSI_G(6, 6, 6)
  // R * (A P)  (k x b times b x k)
  FSI_G(3, 2, 3) FSI_G(6, 3, 6)
  // R * A on the first level of the rigid-body solid hierarchy (k x b times b x b)
  FSI_G(3, 2, 2) FSI_G(6, 3, 3)
  // pressure Schur: (1 x d) * (d x 1)
  FSI_G(1, 2, 1) FSI_G(1, 3, 1)
#undef FSI_G
  throw Error(EINVAL_, "unsupported SpGEMM block shape " + std::to_string(br) + "x" + std::to_string(bk) + "x" +
                           std::to_string(bc));
}

// row pointers from the row lengths, and the index array
void finalize_rowptr(const int* cnt, Bsr& C, cudaStream_t s) {
  C.rowptr.alloc(C.nbr + 1);
  const long long total = scan_ints(cnt, C.rowptr.p, C.nbr, s);
  require(total < INT_MAX, "sparse matrix too large for 32-bit block indices");
  C.nnzb = total;
  C.colind.alloc(total > 0 ? total : 1);
}
void alloc_values(Bsr& C) { C.v64.alloc(C.nnzb > 0 ? C.nnzb * C.br * C.bc : 1); }

}  // namespace

int64_t exclusive_scan(const int* in, int* out, int64_t n, cudaStream_t s) {
  const long long total = scan_ints(in, out, n, s);
  require(total < INT_MAX, "scan overflow");
  return total;
}

void extract_bsr(const CsrView& A, int64_t r0, int nbr, int br, int64_t c0, int nbc, int bc, Bsr& out, bool keep,
                 cudaStream_t s) {
  require(br <= 6, "extract_bsr: block rows > 6");
  const int64_t c1 = c0 + (int64_t)nbc * bc;
  const int grid = div_up((int64_t)nbr * 32, 128);
  keep = keep && out.rowptr.p && out.colind.p && out.nbr == nbr && out.nbc == nbc && out.br == br && out.bc == bc;
  if (!keep) {
    out = Bsr();
    out.nbr = nbr; out.nbc = nbc; out.br = br; out.bc = bc;
    DBuf<int> cnt(nbr > 0 ? nbr : 1);
    if (nbr > 0) {
      k_extract<false><<<grid, 128, 0, s>>>(A.rowptr, A.colind, A.vals, r0, nbr, br, c0, c1, bc, cnt.p, nullptr,
                                            nullptr, nullptr);
      FSI_CHECK_LAUNCH();
    }
    finalize_rowptr(cnt.p, out, s);
  }
  if (!out.v64.p) alloc_values(out);
  // copies of the old values go: what is decided from a block's bytes must not depend on an earlier build
  out.v32.release();
  out.cd16.release();
  out.stage_rows = out.stage_max = 0;
  if (nbr > 0) {
    k_extract<true><<<grid, 128, 0, s>>>(A.rowptr, A.colind, A.vals, r0, nbr, br, c0, c1, bc, nullptr, out.rowptr.p,
                                         out.colind.p, out.v64.p);
    FSI_CHECK_LAUNCH();
  }
  set_tpr(out);
}

void bsr_add(const Bsr& A, const Bsr& B, double alpha, Bsr& C, cudaStream_t s) {
  require(A.nbr == B.nbr && A.nbc == B.nbc && A.br == B.br && A.bc == B.bc, "bsr_add: shape mismatch");
  C = Bsr();
  C.nbr = A.nbr; C.nbc = A.nbc; C.br = A.br; C.bc = A.bc;
  DBuf<int> cnt(A.nbr > 0 ? A.nbr : 1);
  const int bsz = A.br * A.bc;
  if (A.nbr > 0) {
    k_add<false><<<div_up((int64_t)A.nbr * 32, 128), 128, 0, s>>>(A.nbr, bsz, A.rowptr.p, A.colind.p, A.v64.p, B.rowptr.p,
                                                   B.colind.p, B.v64.p, alpha, cnt.p, nullptr, nullptr, nullptr);
    FSI_CHECK_LAUNCH();
  }
  finalize_rowptr(cnt.p, C, s);
  alloc_values(C);
  if (A.nbr > 0) {
    k_add<true><<<div_up((int64_t)A.nbr * 32, 128), 128, 0, s>>>(A.nbr, bsz, A.rowptr.p, A.colind.p, A.v64.p, B.rowptr.p,
                                                  B.colind.p, B.v64.p, alpha, nullptr, C.rowptr.p, C.colind.p,
                                                  C.v64.p);
    FSI_CHECK_LAUNCH();
  }
  set_tpr(C);
}

void bsr_transpose(const Bsr& A, Bsr& C, cudaStream_t s) {
  C = Bsr();
  C.nbr = A.nbc; C.nbc = A.nbr; C.br = A.bc; C.bc = A.br;
  DBuf<int> cnt(C.nbr + 1), cursor(C.nbr + 1);
  FSI_CUDA(cudaMemsetAsync(cnt.p, 0, sizeof(int) * (C.nbr + 1), s));
  FSI_CUDA(cudaMemsetAsync(cursor.p, 0, sizeof(int) * (C.nbr + 1), s));
  if (A.nnzb > 0) {
    k_count_cols<<<div_up(A.nnzb, 256), 256, 0, s>>>(A.nnzb, A.colind.p, cnt.p);
    FSI_CHECK_LAUNCH();
  }
  finalize_rowptr(cnt.p, C, s);
  alloc_values(C);
  if (A.nnzb == 0) { set_tpr(C); return; }
  DBuf<int> rowof(A.nnzb), trow(A.nnzb), tsrc(A.nnzb), src(A.nnzb);
  k_row_of_block<<<div_up(A.nbr, 128), 128, 0, s>>>(A.nbr, A.rowptr.p, rowof.p);
  FSI_CHECK_LAUNCH();
  k_scatter_t<<<div_up(A.nnzb, 256), 256, 0, s>>>(A.nnzb, A.colind.p, rowof.p, C.rowptr.p, cursor.p, trow.p, tsrc.p);
  FSI_CHECK_LAUNCH();
  sort_segments(C.nbr, A.nnzb, C.rowptr.p, trow.p, tsrc.p, C.colind.p, src.p, s);
  k_gather_t<<<div_up(A.nnzb, 256), 256, 0, s>>>(A.nnzb, A.br, A.bc, src.p, A.v64.p, C.v64.p);
  FSI_CHECK_LAUNCH();
  set_tpr(C);
}

void bsr_spgemm(const Bsr& A, const Bsr& B, Bsr& C, cudaStream_t s) {
  int longest = 0;
  require(bsr_spgemm_pattern(A, B, C, longest, s), "bsr_spgemm: a product row has more than 768 block columns");
  bsr_spgemm_values(A, B, C, longest, s);
}

bool bsr_spgemm_pattern(const Bsr& A, const Bsr& B, Bsr& C, int& longest, cudaStream_t s) {
  require(A.bc == B.br && A.nbc == B.nbr, "bsr_spgemm: inner dimensions differ");
  C = Bsr();
  C.nbr = A.nbr; C.nbc = B.nbc; C.br = A.br; C.bc = B.bc;
  DBuf<int> cnt(A.nbr > 0 ? A.nbr : 1), info(2);
  FSI_CUDA(cudaMemsetAsync(info.p, 0, 2 * sizeof(int), s));
  int sub = 4;
  while (sub < 32 && B.nbr > 0 && (double)B.nnzb / B.nbr > sub) sub *= 2;
  // a block per row when a warp per row would leave an SM fewer than 16 warps
  const bool wide = A.nbr < 16 * device_sms();
  const int grid = wide ? A.nbr : div_up(A.nbr, kWarpsPerBlock);
  auto pass = [&](auto fill) {
    constexpr bool FILL = decltype(fill)::value;
    if (A.nbr == 0) return;
    (wide ? k_spgemm_sym<FILL, kWarpsPerBlock> : k_spgemm_sym<FILL, 1>)<<<grid, kWarpsPerBlock * 32, 0, s>>>(
        A.nbr, sub, A.rowptr.p, A.colind.p, B.rowptr.p, B.colind.p, cnt.p, C.rowptr.p, C.colind.p, info.p);
    FSI_CHECK_LAUNCH();
  };
  pass(std::false_type());
  int h[2] = {0, 0};
  FSI_CUDA(cudaMemcpyAsync(h, info.p, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
  FSI_CUDA(cudaStreamSynchronize(s));
  if (h[0]) {
    C = Bsr();
    return false;
  }
  longest = h[1];
  finalize_rowptr(cnt.p, C, s);
  pass(std::true_type());
  set_tpr(C);
  return true;
}

void bsr_spgemm_values(const Bsr& A, const Bsr& B, Bsr& C, int longest, cudaStream_t s) {
  alloc_values(C);
  if (A.nbr == 0 || longest == 0) return;
  spgemm_dispatch(A.br, A.bc, B.bc, [&]<int BR, int BK, int BC>() {
    // columns per warp: about 5 KB of sums (a row a little longer is not split), fewer when
    // rows x chunks would leave an SM fewer than 16 warps, at least 12
    const int most = (int)(5 * 1024 / (BR * BC * sizeof(double)));
    int cap = longest <= most + most / 2 ? longest : most;
    const int64_t tasks = (int64_t)16 * device_sms();
    if ((int64_t)A.nbr * div_up(longest, cap) < tasks)
      cap = std::min(cap, std::max(12, (int)((int64_t)A.nbr * longest / tasks)));
    const int chunks = div_up(longest, cap);
    const size_t sm = kNumWarps * num_smem_per_warp<BR, BC>(cap);
    k_spgemm_num<BR, BK, BC><<<dim3(div_up(A.nbr, kNumWarps), chunks), kNumWarps * 32, sm, s>>>(
        A.nbr, cap, A.rowptr.p, A.colind.p, A.v64.p, B.rowptr.p, B.colind.p, B.v64.p, C.rowptr.p, C.colind.p, C.v64.p);
    FSI_CHECK_LAUNCH();
  });
}

void sort_segments(int nseg, int64_t n, const int* off, const int* key, const int* pay, int* okey, int* opay,
                   cudaStream_t s) {
  if (nseg <= 0) return;
  const int group = n / nseg > 96 ? kSortThreads : 32;   // long segments: the block's threads share one
  k_sort_segments<<<div_up(nseg, kSortThreads / group), kSortThreads, 0, s>>>(nseg, group, off, key, pay, okey, opay);
  FSI_CHECK_LAUNCH();
}

void bsr_scale_rows(Bsr& A, const double* w, cudaStream_t s) {
  if (A.nbr == 0) return;
  k_scale_rows<<<div_up(A.nbr, 128), 128, 0, s>>>(A.nbr, A.br, A.bc, A.rowptr.p, A.v64.p, w);
  FSI_CHECK_LAUNCH();
}

void bsr_scale(Bsr& A, double alpha, cudaStream_t s) {
  const int64_t n = A.nnzb * A.br * A.bc;
  if (n == 0) return;
  k_scale_all<<<div_up(n, 256), 256, 0, s>>>(n, alpha, A.v64.p);
  FSI_CHECK_LAUNCH();
}

void bsr_point_diagonal(const Bsr& A, double* diag, cudaStream_t s) {
  require(A.br == A.bc && A.nbr == A.nbc, "point diagonal of a non-square matrix");
  if (A.nbr == 0) return;
  k_point_diag<<<div_up(A.nbr, 128), 128, 0, s>>>(A.nbr, A.br, A.rowptr.p, A.colind.p, A.v64.p, diag);
  FSI_CHECK_LAUNCH();
}

void invert_nonzero(int64_t n, const double* diag, double* dinv, cudaStream_t s) {
  if (n == 0) return;
  k_invert_nonzero<<<div_up(n, 256), 256, 0, s>>>(n, diag, dinv);
  FSI_CHECK_LAUNCH();
}

void bsr_make_fp32(Bsr& A, cudaStream_t s) {
  const int64_t n = A.nnzb * A.br * A.bc;
  A.v32.alloc(n > 0 ? n : 1);
  if (n > 0) {
    if (planar_fp32_shape(A.br, A.bc))
      k_to_f32_planar9<<<div_up(n, 256), 256, 0, s>>>(A.nnzb, A.v64.p, A.v32.p);
    else
      k_to_f32<<<div_up(n, 256), 256, 0, s>>>(n, A.v64.p, A.v32.p);
    FSI_CHECK_LAUNCH();
  }
}

// Largest slice (in blocks, counted from the 8-entry boundary below it) of the CTAs
// that take R consecutive block rows each: the shared-memory size of the staged
// Chebyshev kernel.
__global__ void k_stage_max(int nbr, const int* __restrict__ rp, int R, int* __restrict__ out) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t r0 = c * R;
  if (r0 >= nbr) return;
  const int64_t r1 = r0 + R < nbr ? r0 + R : nbr;
  atomicMax(out, rp[r1] - (rp[r0] & ~7));
}

void bsr_make_pair_order(Bsr& A1, const Bsr& A2, cudaStream_t s) {
  A1.ord2.release();
  A1.ord2_rp2 = nullptr;
  if (A1.nbr == 0 || A2.nbr != A1.nbr || A1.nbr >= (1 << 24)) return;
  DBuf<int> bad(1);
  FSI_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), s));
  A1.ord2.alloc(A1.nbr);
  k_pair_order<<<div_up(A1.nbr, 256), 256, 0, s>>>(A1.nbr, A1.rowptr.p, A2.rowptr.p, A1.ord2.p, bad.p);
  FSI_CHECK_LAUNCH();
  int h = 0;
  FSI_CUDA(cudaMemcpyAsync(&h, bad.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  FSI_CUDA(cudaStreamSynchronize(s));
  if (h) A1.ord2.release();
  else A1.ord2_rp2 = A2.rowptr.p;
}

bool bsr_make_delta16(Bsr& A, cudaStream_t s) {
  A.cd16.release();
  A.stage_rows = A.stage_max = 0;
  if (A.nbr == 0 || A.nbr != A.nbc || A.nnzb == 0) return false;
  DBuf<int> of(2);
  FSI_CUDA(cudaMemsetAsync(of.p, 0, 2 * sizeof(int), s));
  // 8 spare entries: the staged kernel copies whole 16-byte groups of offsets
  A.cd16.alloc(A.nnzb + 8);
  FSI_CUDA(cudaMemsetAsync(A.cd16.p + A.nnzb, 0, 8 * sizeof(int16_t), s));
  k_delta16<<<div_up(A.nbr, 128), 128, 0, s>>>(A.nbr, A.rowptr.p, A.colind.p, A.cd16.p, of.p);
  FSI_CHECK_LAUNCH();
  const int R = A.br == 2 && A.bc == 2 ? 256 / A.tpr : 0;
  if (R > 0) {
    k_stage_max<<<div_up(div_up(A.nbr, R), 128), 128, 0, s>>>(A.nbr, A.rowptr.p, R, of.p + 1);
    FSI_CHECK_LAUNCH();
  }
  int h[2] = {0, 0};
  FSI_CUDA(cudaMemcpyAsync(h, of.p, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
  FSI_CUDA(cudaStreamSynchronize(s));
  if (h[0]) {
    A.cd16.release();
    return false;
  }
  if (R > 0) {
    A.stage_rows = R;
    A.stage_max = h[1];
  }
  return true;
}

void bsr_to_dense(const Bsr& A, double* dense, cudaStream_t s) {
  const int64_t nr = A.rows(), nc = A.cols();
  FSI_CUDA(cudaMemsetAsync(dense, 0, sizeof(double) * nr * nc, s));
  if (A.nbr == 0) return;
  k_to_dense<<<div_up((int64_t)A.nbr * 32, 128), 128, 0, s>>>(A.nbr, A.br, A.bc, (int)nc, A.rowptr.p, A.colind.p, A.v64.p, dense);
  FSI_CHECK_LAUNCH();
}

}  // namespace fsi
