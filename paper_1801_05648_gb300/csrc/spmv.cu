// The FP32 SpMV kernels and the staged steps' error flag.
#include "spmv_inst.cuh"

namespace fsi {

bool spmv_stage_failed(cudaStream_t s) {
  int h = 0;
  FSI_CUDA(cudaMemcpyAsync(&h, stage_err_ptr(), sizeof(int), cudaMemcpyDeviceToHost, s));
  FSI_CUDA(cudaStreamSynchronize(s));
  if (h) FSI_CUDA(cudaMemsetAsync(stage_err_ptr(), 0, sizeof(int), s));
  return h != 0;
}

FSI_INST(float)

}  // namespace fsi
