// The kernels of rr_route_quad.cuh at d = 128.
#include "rr_route_quad.cuh"

rr_quad_kernel rr_quad_kernel_d128(int variant, bool test) { return test ? quad_kernels<128, true>(variant) : quad_kernels<128, false>(variant); }

#ifdef RR_PHASE_TIMING
extern "C" int rr_debug_quad_phase_counters(unsigned long long* out32, int reset) {
  cudaDeviceSynchronize();
  if (cudaMemcpyFromSymbol(out32, g_quad_phase, sizeof(unsigned long long) * 32) != cudaSuccess) return -1;
  if (reset) {
    unsigned long long z[32] = {};
    cudaMemcpyToSymbol(g_quad_phase, z, sizeof z);
  }
  return 0;
}
#endif
