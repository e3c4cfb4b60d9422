// launch.cu -- what the kernel launchers ask of the runtime, kept per plan.
//
// A launch used to set two function attributes and ask for five device and function
// attributes; with a dozen launches a pass, and a memset of the queue counter before
// each queue kernel, that was a third of a short record's pass (2^20 samples, T = 256).
#include <algorithm>

#include "internal.cuh"

namespace ss {

cudaError_t sm_count(LaunchCache* lc, int* nsm) {
  if (lc && lc->nsm > 0) {
    *nsm = lc->nsm;
    return cudaSuccess;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && lc) lc->nsm = *nsm;
  return e;
}

cudaError_t prepare_kernel(const void* kern, int threads, size_t smem, size_t limit, int max_ctas,
                           LaunchCache* lc, int slot, int* occ) {
  if (lc && lc->occ[slot] > 0) {
    *occ = lc->occ[slot];
    return cudaSuccess;
  }
  // The dynamic shared-memory limit of a kernel is an attribute of the function, shared
  // by every plan, stream and captured graph that launches it; each kernel therefore
  // has one fixed limit, the largest amount any of its launches can ask for, so that no
  // launch depends on which launch set it last.
  cudaFuncAttributes fa;
  int dev = 0, sm_smem = 0, sm_regs = 0, rsv = 0;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&sm_regs, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&rsv, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  if (e != cudaSuccess) return e;
  const int by_smem = sm_smem / (int)(smem + fa.sharedSizeBytes + rsv);
  const int by_regs = sm_regs / std::max(1, ((fa.numRegs + 7) & ~7) * threads);
  *occ = std::max(1, std::min(max_ctas, std::min(by_smem, by_regs)));
  if (lc) lc->occ[slot] = *occ;
  return cudaSuccess;
}

}  // namespace ss
