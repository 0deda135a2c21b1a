// Shared device-side definitions of the FSI solver library: dependent launches,
// launch knobs, the block-sparse-row (BSR) matrix type and small helpers.
#pragma once
#include "error.cuh"
#include "mempool.cuh"

#include <cuda.h>
#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>
#include <cstdio>
#include <memory>
#include <string>
#include <vector>
#include <utility>

namespace fsi {

// Kernel launches issued by this thread (captured launches are re-counted per
// graph replay by the solver).
inline thread_local int64_t g_kernel_launches = 0;

#define FSI_CHECK_LAUNCH()        \
  do {                            \
    ++::fsi::g_kernel_launches;   \
    FSI_CUDA(cudaGetLastError()); \
  } while (0)

// Programmatic dependent launch (sm_90 and later).  A kernel started with
// launch_k() may be scheduled before the previous kernel of its stream has finished:
// once every block of that kernel has called dep_trigger() or ended, its blocks become
// resident where there is room, and dep_wait_only() returns when that kernel (and with
// it all before it) has completed and its writes are visible.  Before that wait a
// kernel touches only what no queued kernel writes: the launch's arguments, and, outside
// set-up, matrices and weights, which every call that writes them leaves with a
// stream synchronisation.  Every kernel launched through launch_k() waits, as its first
// act (dep_wait: trigger and wait) or after such loads.  Triggering first takes the
// launch itself out of the chain of short dependent kernels: 256x128 solve 9.5 -> 9.2 ms.
// A kernel that precedes or is a product bound by the FP64 pipe does not trigger: blocks that
// arrive early settle where there happens to be room, and the fullest SM's FP64 pipe then sets
// the pace (64x32 solve 1.99 ms with such triggers, 1.92 without; training step 800 / 762 us).
// Off for the whole process when a context was set up with FSI_NO_PDL.
// Such a kernel's lifetime overlaps writes of the kernels before it, so nothing that a queued kernel
// may write counts as read-only in it: those arguments carry no __restrict__ and are read by ordinary loads
// behind the wait, not by __ldg or ld.global.nc, which the compiler may move ahead of it and which
// need not see the write.  Matrices, patterns, weights and the arguments themselves may be.
__device__ __forceinline__ void dep_trigger() {
#if defined(__CUDA_ARCH__) && (__CUDA_ARCH__ >= 900)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}
__device__ __forceinline__ void dep_wait_only() {
#if defined(__CUDA_ARCH__) && (__CUDA_ARCH__ >= 900)
  asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}
__device__ __forceinline__ void dep_wait() {
  dep_trigger();
  dep_wait_only();
}

// Launch knobs (programmatic dependent launch here; the SpMV shape and the coarse
// V-cycle threshold below) are per thread: every entry point that takes a context
// applies that context's values for the duration of the call (KnobScope in
// fsi_api.cu), so contexts with different parameters do not interfere.
inline bool& pdl_enabled() {
  thread_local bool on = true;
  return on;
}
// Learned-stage MLP on the tensor cores (else on the CUDA cores).
inline bool& mlp_tensor_cores() {
  thread_local bool on = true;
  return on;
}
// Host-side fault injection for the tests of the bounded waits (0 in normal use):
// kInjectCoarseBarrier: the coarse V-cycle's grid barrier waits for one CTA more than
// the launch has; kInjectMlpCommit: the tensor-core MLP does not commit its first
// layer's MMAs to the barrier it then waits on.  Either wait then runs out.
enum { kInjectCoarseBarrier = 1, kInjectMlpCommit = 2 };
inline int& fault_inject() {
  thread_local int v = 0;
  return v;
}

// Streaming multiprocessors of the current device (looked up once per device).
inline int device_sms() {
  constexpr int kMaxDev = 64;
  static int cache[kMaxDev] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 152;
  int v = __atomic_load_n(&cache[dev], __ATOMIC_RELAXED);
  if (v == 0) {
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 152;
    __atomic_store_n(&cache[dev], v, __ATOMIC_RELAXED);
  }
  return v;
}

template <class... KArgs, class... Args>
void launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args);

// Makes `dev` the calling thread's current CUDA device while the guard lives and
// restores the previous device afterwards (nothing to do when dev < 0 or when it
// is current already).  A context's streams and memory belong to the device that
// was current at fsi_setup; every entry point runs under a guard for it, so a
// caller whose thread has since switched devices still launches on the right one.
struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (dev < 0) return;
    int cur = -1;
    FSI_CUDA(cudaGetDevice(&cur));
    if (cur == dev) return;
    FSI_CUDA(cudaSetDevice(dev));
    prev = cur;
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
  DeviceGuard(const DeviceGuard&) = delete;
  DeviceGuard& operator=(const DeviceGuard&) = delete;
};

// A number of the current CUDA context that no other one of this process has or had: a device that was reset
// gets another.  (0 where the driver does not tell.)
inline unsigned long long cuda_context_id() {
  using GetCurrent = CUresult (*)(CUcontext*);
  using GetId = CUresult (*)(CUcontext, unsigned long long*);
  struct Entry {
    void* current = nullptr;
    void* id = nullptr;
    Entry() {
      cudaDriverEntryPointQueryResult r;
      if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &current, 12000, cudaEnableDefault, &r) != cudaSuccess ||
          cudaGetDriverEntryPointByVersion("cuCtxGetId", &id, 12000, cudaEnableDefault, &r) != cudaSuccess)
        current = nullptr;
      cudaGetLastError();
    }
  };
  static const Entry e;
  if (!e.current || !e.id) return 0;
  CUcontext c = nullptr;
  unsigned long long v = 0;
  if (reinterpret_cast<GetCurrent>(e.current)(&c) != CUDA_SUCCESS || !c) {
    FSI_CUDA(cudaFree(nullptr));   // makes the device's context, where this thread has none yet
    if (reinterpret_cast<GetCurrent>(e.current)(&c) != CUDA_SUCCESS || !c) return 0;
  }
  return reinterpret_cast<GetId>(e.id)(c, &v) == CUDA_SUCCESS ? v : 0;
}

// cuda_context_id() + 1 of each device, as of the last solver context or assembler made on it (0: none yet).
// The driver is asked there and not in once_per_device, which short calls pass through.
inline std::atomic<unsigned long long>& device_context(int dev) {
  static std::atomic<unsigned long long> id[64];
  return id[dev];
}
inline unsigned long long note_device_context() {
  int dev = 0;
  FSI_CUDA(cudaGetDevice(&dev));
  require(dev >= 0 && dev < 64, "device ordinal above 63");
  const unsigned long long id = cuda_context_id() + 1;
  device_context(dev).store(id, std::memory_order_release);
  return id;
}

// Runs setup(dev) once per device dev, on the current one, and again for solver contexts and assemblers made
// after the device was reset: a kernel's function attributes, a __device__ variable's address and a stream
// belong to one CUDA context of one device, so what was set up in one does not hold in another.  `done` is the
// call site's record: the CUDA context that each device was set up in.  Two threads may both run it for the
// same device; it must be idempotent.
struct OncePerDevice {
  std::atomic<unsigned long long> context[64] = {};   // as device_context, 0: not yet
};
template <class F>
void once_per_device(OncePerDevice& done, F&& setup) {
  int dev = 0;
  FSI_CUDA(cudaGetDevice(&dev));
  require(dev >= 0 && dev < 64, "device ordinal above 63");
  unsigned long long now = device_context(dev).load(std::memory_order_acquire);
  if (now == 0) now = note_device_context();
  if (done.context[dev].load(std::memory_order_acquire) == now) return;
  setup(dev);
  done.context[dev].store(now, std::memory_order_release);
}

// Block sparse row matrix on the device: nbr x nbc blocks of br x bc values,
// block values row-major, blocks of a row stored consecutively with sorted
// block-column indices.  Values may exist in FP64, FP32 or both.
struct Bsr {
  int nbr = 0, nbc = 0, br = 1, bc = 1;
  int64_t nnzb = 0;
  DBuf<int> rowptr;     // nbr + 1
  DBuf<int> colind;     // nnzb
  DBuf<double> v64;     // nnzb * br * bc
  DBuf<float> v32;      // optional FP32 copy
  DBuf<int16_t> cd16;   // optional, square matrices: block column minus block row as int16 (read by the
                        // FP32 Chebyshev steps when every offset fits; 2 bytes per block instead of 4)
  DBuf<int4> ord2;      // optional: the slot table of the two-matrix SpMV with the partner whose row
  const int* ord2_rp2 = nullptr;   // pointers these are: block rows sorted by (length here, length
                        // there) within 32-row windows, {row | length << 24, first block, first
                        // partner block, partner length} per slot (k_pair_order)
  int stage_rows = 0;   // 2 x 2 FP32 with cd16: block rows per CTA the staged Chebyshev kernel was sized for
  int stage_max = 0;    // ... and the largest CTA slice in blocks, from the 8-entry boundary below it
  int tpr = 32;         // threads per block row of the FP32 SpMV, from the mean row length
  int tpr64 = 2;        // ... of the FP64 SpMV (fewer lanes: FP64 issue slots are scarce)
  int64_t rows() const { return (int64_t)nbr * br; }
  int64_t cols() const { return (int64_t)nbc * bc; }
  template <class T> const T* vals() const;
  // algorithmic bytes of one SpMV: values + column indices + row pointers + x + y
  // (FP32 products of a matrix with 16-bit column offsets read 2 bytes per block index)
  double spmv_bytes(int value_bytes) const {
    const int ib = (value_bytes == 4 && cd16.p) ? 2 : 4;
    return (double)nnzb * (br * bc * value_bytes + ib) + 4.0 * (nbr + 1) + (double)value_bytes * (cols() + rows());
  }
};
// FP32 copies of blocks with 9 values (3 x 3) are stored planar (values 0-3 of
// every block, then 4-7, then 8; see load_block in spmv.cuh); all other copies are
// row-major blocks.
__host__ __device__ constexpr bool planar_fp32_shape(int br, int bc) { return br * bc == 9; }

template <> inline const double* Bsr::vals<double>() const { return v64.p; }
template <> inline const float* Bsr::vals<float>() const { return v32.p; }

// Lanes per block row: the most lanes (a power of two, at most 32) that leave
// each lane at least `min_per_lane` blocks of an average row, so a row's blocks
// are read by neighbouring lanes (coalesced) in about one pass per lane,
// whatever the number of rows.  FP32 rows keep two blocks per lane.  FP64 rows
// keep at least eight: the FP64 pipe of this GPU retires a small fraction of the
// FP32 rate, and the shuffle reduction across a wide lane group would cost more
// FP64 instructions than the products themselves.
inline int lanes_for(int64_t nnzb, int nbr, double min_per_lane) {
  const double mean = nbr ? (double)nnzb / nbr : 0.0;
  int t = 1;
  while (t < 32 && mean / (2 * t) >= min_per_lane) t *= 2;
  return t;
}

// SpMV launch shape knobs (fsi_params: spmv_unroll, spmv_prefetch).
struct SpmvTuning {
  int unroll = 4;      // blocks each lane loads before multiplying: 4 or 8 (8 only for small blocks)
  int prefetch = 1;    // 0 none, 1 L2 bulk prefetch of each CTA's matrix slice, 2 also persistent CTAs
  int ctas_per_sm = 5; // persistent grid size per SM (prefetch 2)
  int lane_shift = 0;  // FP32 launches: lanes per block row divided by 2^lane_shift (at least 1)
  int stage = 0;       // 2 x 2 FP32 Chebyshev steps with the column offsets staged in shared memory
  int order = 1;       // two-matrix launches take their rows in the order of Bsr::ord2 when it is built
  int wide64 = 0;      // FP64 launches take more lanes per row on small matrices (see WideRows64)
  int setup_depth = 0; // > 0 while matrices are being built: no reads before the dependency wait
};
inline SpmvTuning& spmv_tuning() {
  thread_local SpmvTuning t;
  return t;
}

// Marks the set-up phase (context set-up, preconditioner build): an SpMV may then
// be launched right after the kernel that writes its matrix, so it reads no matrix
// memory before its dependency wait, and buffers come from the context's pool.
struct SetupPhase {
  std::shared_ptr<MemPool> saved;
  explicit SetupPhase(const std::shared_ptr<MemPool>& pool) : saved(current_pool()) {
    ++spmv_tuning().setup_depth;
    current_pool() = pool;
  }
  ~SetupPhase() {
    --spmv_tuning().setup_depth;
    current_pool() = saved;
  }
  SetupPhase(const SetupPhase&) = delete;
  SetupPhase& operator=(const SetupPhase&) = delete;
};

// The FP64 preconditioner's launches spread a row over more lanes where its matrix would
// otherwise leave the GPU a few warps per SM (widened() in spmv_inst.cuh).  That changes the order of a
// row's sum, so only the FP64 preconditioner takes it: the outer operator and the set-up,
// which the FP32 form shares, keep theirs.
struct WideRows64 {
  int saved;
  explicit WideRows64(bool on) : saved(spmv_tuning().wide64) { spmv_tuning().wide64 = on ? 1 : 0; }
  ~WideRows64() { spmv_tuning().wide64 = saved; }
  WideRows64(const WideRows64&) = delete;
  WideRows64& operator=(const WideRows64&) = delete;
};

inline void set_tpr(Bsr& A) {
  A.tpr = lanes_for(A.nnzb, A.nbr, 2.0);
  A.tpr64 = lanes_for(A.nnzb, A.nbr, 8.0);
}

inline int div_up(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

template <class... KArgs, class... Args>
void launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  FSI_CUDA(cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...));
  ++g_kernel_launches;
}


}  // namespace fsi
