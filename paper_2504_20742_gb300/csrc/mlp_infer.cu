// mlp_infer.cu -- packing of a trained surrogate into its device blob, and a standalone
// persistent tensor-core inference kernel over a batch of raw inputs (the same tile routine
// as the fused FP32_MLP step).
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include "../../include/contrail.h"
#include "mlp_tc.cuh"

extern "C" ct_status ct__set_error(ct_status s, const char* msg);

namespace ct {
namespace mlp {

// params: flat FP32 (per layer W out x in, then b); stats: 16-float arrays.
__global__ void k_pack(const float* __restrict__ params, const float* __restrict__ x_mean,
                       const float* __restrict__ x_sd, const float* __restrict__ x_min, const float* __restrict__ x_max,
                       const float* __restrict__ y_mean, const float* __restrict__ y_sd, const float* __restrict__ y_min,
                       const float* __restrict__ y_max, unsigned char* __restrict__ blob) {
  float* hdr = reinterpret_cast<float*>(blob);
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
  for (int i = tid; i < 16; i += nt) {
    hdr[F_XMEAN + i] = x_mean[i];
    hdr[F_XISD + i] = x_sd[i] > 0.0f ? 1.0f / x_sd[i] : 1.0f;
    hdr[F_YMEAN + i] = i < CT_MLP_OUT ? y_mean[i] : 0.0f;
    hdr[F_YSD + i] = i < CT_MLP_OUT ? y_sd[i] : 0.0f;
    hdr[F_HMIN + i] = x_min[i];
    hdr[F_HMAX + i] = x_max[i];
    hdr[F_YMIN + i] = i < CT_MLP_OUT ? y_min[i] : 0.0f;
    hdr[F_YMAX + i] = i < CT_MLP_OUT ? y_max[i] : 0.0f;
  }
  // flat parameter offsets
  int po = 0;
  for (int l = 0; l < 5; ++l) {
    const int K = kdim(l), Nout = l == 4 ? CT_MLP_OUT : 128, Np = ndim(l);
    const float* Wl = params + po;
    const float* bl = Wl + Nout * K;
    __nv_bfloat16* wb = reinterpret_cast<__nv_bfloat16*>(blob + WOFF + woff(l));
    for (int e = tid; e < Np * K; e += nt) {
      const int n = e / K, k = e % K;
      const float v = n < Nout ? Wl[n * K + k] : 0.0f;
      wb[tc::cm_offset(n, k, K) / 2] = __float2bfloat16_rn(v);
    }
    for (int n = tid; n < Np; n += nt) hdr[F_BIAS + 128 * l + n] = n < Nout ? bl[n] : 0.0f;
    po += Nout * K + Nout;
  }
}

// Three warpgroups per CTA, one CTA per SM with all weights resident, each group on tiles of its own
// (run_group): 60 us for 200,000 rows (GB300), 106 us with one tile at a time per SM, four warps
// waiting on each layer in turn.
__global__ void __launch_bounds__(128 * GROUPS, 1) k_infer(const unsigned char* __restrict__ blob,
                                                          const float* __restrict__ X, int n, float* __restrict__ Y,
                                                          int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ GroupTc tcs;
  const uint32_t tmem = group_acquire(&tcs);
  load_net(sm, blob);
  const float* hdr = reinterpret_cast<const float*>(sm + GS_HDR);
  const int g = threadIdx.x >> 7, t = threadIdx.x & 127;
  const uint32_t mbar = tc::smem_addr(&tcs.bar[g]);
  uint32_t phase = 0;
  const int ntiles = (n + 127) / 128;
  const bool vec = ((uintptr_t)X & 15) == 0;
  // tiles blockIdx.x + gridDim.x * (g + GROUPS k): the groups of all SMs fill evenly
  for (long long tile = blockIdx.x + (long long)gridDim.x * g; tile < ntiles; tile += (long long)gridDim.x * GROUPS) {
    const long long row = tile * 128 + t;
    float v[16], o[10];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (row < n) {
        const float* p = X + (size_t)row * 16 + 4 * c;
        x = vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
      }
      v[4 * c] = x.x;
      v[4 * c + 1] = x.y;
      v[4 * c + 2] = x.z;
      v[4 * c + 3] = x.w;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = row < n ? (v[i] - hdr[F_XMEAN + i]) * hdr[F_XISD + i] : 0.0f;
    if (!run_group(sm, g, v, tmem + 128u * g, mbar, phase, o)) {
      if (t == 0) atomicExch(err, 1);
      break;
    }
    if (row < n) {
#pragma unroll
      for (int i = 0; i < 10; ++i) Y[(size_t)row * 10 + i] = o[i] * hdr[F_YSD + i] + hdr[F_YMEAN + i];
    }
  }
  group_release(tmem);
}

}  // namespace mlp
}  // namespace ct

using namespace ct::mlp;

extern "C" {

size_t ct_mlp_blob_bytes(void) { return (size_t)BLOB_BYTES; }

ct_status ct_mlp_pack(const float* params, const float* x_mean, const float* x_sd, const float* x_min,
                      const float* x_max, const float* y_mean, const float* y_sd, const float* y_min,
                      const float* y_max, void* blob, void* stream) {
  if (!params || !x_mean || !x_sd || !x_min || !x_max || !y_mean || !y_sd || !y_min || !y_max || !blob)
    return ct__set_error(CT_ERR_ARG, "ct_mlp_pack: null pointer");
  if (((uintptr_t)blob & 15) != 0) return ct__set_error(CT_ERR_ARG, "ct_mlp_pack: blob must be 16-byte aligned");
  k_pack<<<64, 256, 0, (cudaStream_t)stream>>>(params, x_mean, x_sd, x_min, x_max, y_mean, y_sd, y_min, y_max,
                                                (unsigned char*)blob);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? CT_OK : ct__set_error(CT_ERR_CUDA, cudaGetErrorString(e));
}

ct_status ct_mlp_infer(const void* blob, const float* X, int n, float* Y, int* err_flag, void* stream) {
  if (!blob || !X || !Y || !err_flag || n < 0) return ct__set_error(CT_ERR_ARG, "ct_mlp_infer: bad argument");
  if (((uintptr_t)blob & 15) != 0) return ct__set_error(CT_ERR_ARG, "ct_mlp_infer: blob must be 16-byte aligned");
  if (n == 0) return CT_OK;
  // on every call: the limit belongs to the current device
  cudaError_t e = cudaFuncSetAttribute(k_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GROUP_SMEM);
  if (e != cudaSuccess) return ct__set_error(CT_ERR_CUDA, cudaGetErrorString(e));
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int ntiles = (n + 127) / 128;
  const int grid = ntiles < nsm ? ntiles : nsm;
  k_infer<<<grid, 128 * GROUPS, GROUP_SMEM, (cudaStream_t)stream>>>((const unsigned char*)blob, X, n, Y, err_flag);
  e = cudaGetLastError();
  return e == cudaSuccess ? CT_OK : ct__set_error(CT_ERR_CUDA, cudaGetErrorString(e));
}

}  // extern "C"
