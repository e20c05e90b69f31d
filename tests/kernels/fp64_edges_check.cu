// Test kernel: the FP64 saturation temperature of the tabulated curves (physics.cuh), and logexp.cuh's
// halving where the exponent field runs out.
#include <cuda_runtime.h>

#include "../../paper_2504_20742_gb300/csrc/physics.cuh"

__global__ void k_edges(int which, const double* __restrict__ x, const double* __restrict__ tab, double* __restrict__ r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  ct::SrcCase sc{};
  sc.tables = 1;
  sc.tab = tab;
  if (which == 0) r[i] = ct::prop_tsat<double, false>(sc, x[i]);
  else if (which == 1) r[i] = ct::prop_tsat<double, true>(sc, x[i]);
  else r[i] = ct::half_bits(x[i]);
}

extern "C" int fp64_edges(int which, const double* x, const double* tab, double* r, int n) {
  k_edges<<<(n + 255) / 256, 256>>>(which, x, tab, r, n);
  return (int)cudaDeviceSynchronize();
}
