// The batched Rosenbrock integrator with 4 warps per cell (see integrator_impl.cuh).
#include "integrator_impl.cuh"

namespace dlb {

cudaError_t launch_rosenbrock_w4(unsigned grid, int threads, int smem, cudaStream_t s, const KernelArgs& a) {
  rosenbrock_kernel<4, false><<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

const void* rosenbrock_kernel_ptr_w4() { return reinterpret_cast<const void*>(&rosenbrock_kernel<4, false>); }

const void* gate_kernel_ptr_w4() { return reinterpret_cast<const void*>(&gate_kernel<4>); }

cudaError_t launch_gate_w4(unsigned grid, int threads, int smem, cudaStream_t s, const GateArgs& a) {
  gate_kernel<4><<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_rhs_w4(unsigned grid, int threads, int smem, cudaStream_t s, const RhsArgs& a) {
  if (general_kernel(a.m)) rhs_kernel<4, true><<<grid, threads, smem, s>>>(a);
  else rhs_kernel<4, false><<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

const void* rhs_kernel_ptr_w4(bool general) {
  return general ? reinterpret_cast<const void*>(&rhs_kernel<4, true>) : reinterpret_cast<const void*>(&rhs_kernel<4, false>);
}

}  // namespace dlb
