// Test kernel: logexp.cuh's functions and the FP64 saturation temperature of physics.cuh, with
// CUDA's own functions and the six-step Newton iteration beside them.
#include <cuda_runtime.h>

#include "../../paper_2504_20742_gb300/csrc/physics.cuh"

__global__ void k_check(int which, const double* __restrict__ x, const double* __restrict__ y, double* __restrict__ r,
                        double* __restrict__ ref, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double a = x[i], b = y[i];
  switch (which) {
    case 0: r[i] = ct::log_t(a); ref[i] = log(a); break;
    case 1: r[i] = ct::exp_t(a); ref[i] = exp(a); break;
    case 2: r[i] = ct::expm1_t(a); ref[i] = expm1(a); break;
    case 3: r[i] = ct::sqrt_t(a); ref[i] = sqrt(a); break;
    case 4: r[i] = ct::quot_t(a, b); ref[i] = a / b; break;
    case 5: r[i] = ct::to_d((float)a); ref[i] = (double)(float)a; break;
    case 6: r[i] = ct::half_bits(a); ref[i] = 0.5 * a; break;
    case 7: {
      ct::SrcCase sc{};
      r[i] = ct::prop_tsat<double, false>(sc, a);
      ref[i] = ct::t_sat<double, false>(a);
      break;
    }
    default: {
      ct::SrcCase sc{};
      r[i] = ct::prop_tsat<double, true>(sc, a);
      ref[i] = ct::t_sat<double, true>(a);
      break;
    }
  }
}

extern "C" int logexp_check(int which, const double* x, const double* y, double* r, double* ref, int n) {
  k_check<<<(n + 255) / 256, 256>>>(which, x, y, r, ref, n);
  return (int)cudaDeviceSynchronize();
}
