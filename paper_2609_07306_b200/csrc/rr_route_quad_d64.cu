// The kernels of rr_route_quad.cuh at d = 64.
#include "rr_route_quad.cuh"

rr_quad_kernel rr_quad_kernel_d64(int variant, bool test) { return test ? quad_kernels<64, true>(variant) : quad_kernels<64, false>(variant); }
