// Errors inside the library and their conversion from CUDA's.
#pragma once
#include <cuda_runtime.h>
#include <stdexcept>
#include <string>

namespace fsi {

// Error raised inside the library; converted to a status code at the C ABI.
struct Error : std::runtime_error {
  int code;
  Error(int c, const std::string& m) : std::runtime_error(m), code(c) {}
};

enum Status { OK = 0, EINVAL_ = -1, ENOMEM_ = -2, ECUDA_ = -3, ENOTCONV_ = -4, EBREAKDOWN_ = -5, ENONFINITE_ = -6 };

#define FSI_CUDA(call)                                                                          \
  do {                                                                                          \
    cudaError_t e_ = (call);                                                                    \
    if (e_ != cudaSuccess) {                                                                    \
      if (e_ == cudaErrorMemoryAllocation)                                                      \
        throw ::fsi::Error(::fsi::ENOMEM_, std::string("out of device memory at ") + #call);    \
      throw ::fsi::Error(::fsi::ECUDA_, std::string(cudaGetErrorString(e_)) + " at " + #call);  \
    }                                                                                           \
  } while (0)

inline void require(bool ok, const std::string& msg) {
  if (!ok) throw Error(EINVAL_, msg);
}

}  // namespace fsi
