// mlp_tc.cuh -- BF16 tensor-core inference of the source surrogate (16 -> 4x128 SiLU -> 10)
// on tiles of 128 rows: the five layers run as tcgen05.mma chains (M = 128, K = 16 or 128,
// N = 128 or 16) with FP32 accumulation in TMEM; between layers, one warpgroup reads the
// accumulator back (tcgen05.ld), adds the bias, applies SiLU, rounds to BF16 and writes the
// next layer's operand into shared memory.
#pragma once
#include <cuda_bf16.h>

#include "tc.cuh"

namespace ct {
namespace mlp {

// Device blob: a float header, then the BF16 weights in K-major core-matrix order.
constexpr int F_XMEAN = 0, F_XISD = 16, F_YMEAN = 32, F_YSD = 48, F_HMIN = 64, F_HMAX = 80, F_YMIN = 96,
              F_YMAX = 112, F_BIAS = 128;
constexpr int NFLOAT = F_BIAS + 4 * 128 + 16;   // 656
constexpr int WOFF = 2688;                      // byte offset of the weights (128-byte aligned)
__host__ __device__ constexpr int kdim(int l) { return l == 0 ? 16 : 128; }
__host__ __device__ constexpr int ndim(int l) { return l == 4 ? 16 : 128; }      // padded output width
__host__ __device__ constexpr int wbytes(int l) { return ndim(l) * kdim(l) * 2; }
__host__ __device__ constexpr int woff(int l) {
  int o = 0;
  for (int q = 0; q < l; ++q) o += wbytes(q);
  return o;
}
constexpr int WBYTES = woff(5);                 // 106,496
constexpr int BLOB_BYTES = WOFF + WBYTES;       // 109,184
constexpr int ABYTES = 128 * 128 * 2;           // activation operand, 32 KB

// SiLU of 16 accumulators: z sigmoid(z) = (z/2)(1 + tanh(z/2)), z = v + bias, with the hardware
// tanh approximation (one special-function operation; its relative error, below 2^-10, is under the
// BF16 rounding that follows).  hb: half the biases (16-byte aligned shared memory): z/2 is then one
// fused operation, with the bits of the halved sum.  Two values per instruction but for the tanh.
__device__ __forceinline__ void silu16(float* v, const float* hb) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 b = *reinterpret_cast<const float4*>(hb + 4 * i);
    const float2 h0 = __ffma2_rn(make_float2(v[4 * i], v[4 * i + 1]), make_float2(0.5f, 0.5f), make_float2(b.x, b.y));
    const float2 h1 = __ffma2_rn(make_float2(v[4 * i + 2], v[4 * i + 3]), make_float2(0.5f, 0.5f), make_float2(b.z, b.w));
    float2 t0, t1;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t0.x) : "f"(h0.x));
    asm("tanh.approx.f32 %0, %1;" : "=f"(t0.y) : "f"(h0.y));
    asm("tanh.approx.f32 %0, %1;" : "=f"(t1.x) : "f"(h1.x));
    asm("tanh.approx.f32 %0, %1;" : "=f"(t1.y) : "f"(h1.y));
    const float2 r0 = __ffma2_rn(h0, t0, h0), r1 = __ffma2_rn(h1, t1, h1);
    v[4 * i] = r0.x;
    v[4 * i + 1] = r0.y;
    v[4 * i + 2] = r1.x;
    v[4 * i + 3] = r1.y;
  }
}
// The blob's header in shared memory: entry i, the biases of the hidden layers halved for silu16.
__device__ __forceinline__ float hdr_entry(int i, float v) { return i >= F_BIAS && i < F_BIAS + 512 ? 0.5f * v : v; }

// Write 16 values of row `row` (columns c16*16 .. +15) as BF16 into a K-major operand with K
// columns (two 16-byte core-matrix rows).
__device__ __forceinline__ void store_row16(unsigned char* buf, int row, int c16, int K, const float* v) {
  uint4 a, b;
  __nv_bfloat162 t;
  t = __floats2bfloat162_rn(v[0], v[1]);   a.x = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(v[2], v[3]);   a.y = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(v[4], v[5]);   a.z = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(v[6], v[7]);   a.w = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(v[8], v[9]);   b.x = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(v[10], v[11]); b.y = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(v[12], v[13]); b.z = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(v[14], v[15]); b.w = *reinterpret_cast<uint32_t*>(&t);
  *reinterpret_cast<uint4*>(buf + tc::cm_offset(row, c16 * 16, K)) = a;
  *reinterpret_cast<uint4*>(buf + tc::cm_offset(row, c16 * 16 + 8, K)) = b;
}

// one thread: layer l's weights from the global blob weights Wg into the 32 KB buffer W, completion on wbar
__device__ __forceinline__ void fetch_layer(unsigned char* W, const unsigned char* __restrict__ Wg, int l, uint32_t wbar) {
  tc::mbar_arrive_expect_tx(wbar, (uint32_t)wbytes(l));
  tc::bulk_g2s(tc::smem_addr(W), Wg + woff(l), (uint32_t)wbytes(l), wbar);
}

// Run the network on up to 256 rows (one or two 128-row tiles) whose standardised inputs are
// already in A (K = 16 layout; the second tile's operand ABYTES further).  All threads of the CTA
// (at least 8 warps) call this; `out` gets the 10 standardised outputs of a row: with one tile in
// threads 0..127 (row = thread), with two in threads 0..255.  W: a 32 KB shared buffer that layer 0's
// weights are on their way to (fetch_layer); each further layer's arrive by one bulk copy (completion on
// `wbar`/`wphase`), issued as soon as the previous layer's products have finished, so that the copy
// overlaps that layer's epilogue (keeps the fused step at 2 CTAs per SM); `more`: layer 0's again at
// the end, for the next call.  `bias`: the 4x128 (halved) + 16 biases; `tmem`: 256 allocated TMEM
// columns; `mbar`/`phase`: the completion barrier of the products.  nrows: rows that carry data; 32-row
// groups beyond them skip the epilogue.  One tile: warps w and w + 4 share a lane quarter of TMEM and
// split the columns; two tiles: each takes its own.  Returns false if a wait timed out.  Two tiles at a
// time halve the weight traffic and the chain of waits of a full 256-cell stage tile.
__device__ __forceinline__ bool run_tiles(unsigned char* A, unsigned char* W, const float* bias, uint32_t tmem, uint32_t mbar,
                                          uint32_t& phase, float* out, const unsigned char* __restrict__ Wg, int nrows,
                                          uint32_t wbar, uint32_t* wphase, bool more) {
  const int tid = threadIdx.x, warp = tid >> 5;
  const bool two = nrows > 128;
  const int quarter = warp & 3, half = warp >> 2;      // half: the tile (two), else the column half
  const int row = 32 * quarter + (tid & 31);
  const bool epi = warp < 8 && 32 * quarter + (two && half ? 128 : 0) < nrows;
  unsigned char* At = A + (two && half == 1 ? ABYTES : 0);
  const uint32_t lane_addr = tmem + (two && half == 1 ? 128u : 0u) + ((uint32_t)(32 * quarter) << 16);
  const int c_lo = two ? 0 : 4 * half, c_hi = two ? 8 : c_lo + 4;
  bool ok = true;
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  for (int l = 0; l < 5; ++l) {
    const int K = kdim(l), N = ndim(l);
    if (tid == 0) {
      if (!tc::mbar_wait(wbar, *wphase)) ok = false;
      *wphase ^= 1u;
      const uint32_t b0 = tc::smem_addr(W), sbo = (uint32_t)(K / 8) * 128u, idesc = tc::idesc_bf16_f32(128, N);
      for (int t = 0; t < (two ? 2 : 1); ++t) {
        const uint32_t a0 = tc::smem_addr(A) + (uint32_t)(t * ABYTES);
        for (int s = 0; s < K / 16; ++s)
          tc::mma_bf16(tmem + 128u * t, tc::smem_desc(a0 + 256u * s, 128u, sbo), tc::smem_desc(b0 + 256u * s, 128u, sbo), idesc,
                       s > 0 ? 1u : 0u);
      }
      tc::mma_commit(mbar);
    }
    if (!tc::mbar_wait(mbar, phase)) ok = false;
    phase ^= 1u;
    tc::fence_after_sync();
    if (tid == 0 && (l < 4 || more)) fetch_layer(W, Wg, l < 4 ? l + 1 : 0, wbar);   // W is free again
    if (epi) {
      if (l < 4) {
#pragma unroll 1
        for (int c = c_lo; c < c_hi; ++c) {
          float v[16];
          tc::tmem_ld16(lane_addr + 16u * c, v);
          silu16(v, bias + l * 128 + 16 * c);
          store_row16(At, row, c, 128, v);
        }
      } else if (two || half == 0) {
        float v[16];
        tc::tmem_ld16(lane_addr, v);
#pragma unroll
        for (int i = 0; i < 10; ++i) out[i] = v[i] + bias[4 * 128 + i];
      }
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
  }
  return ok;
}

// ---- one warpgroup, one 128-row tile ---------------------------------------------------------------
// The same network on a tile that belongs to a group of 128 threads (four warps, the first of
// them a multiple of four in the CTA, so that thread t of the group reads TMEM lane t): the kernels
// that keep all weights in shared memory run GROUPS such tiles side by side on an SM, each on its
// own operand buffer, TMEM columns, mbarrier and named barrier, so that one group's epilogue (the
// SiLUs, 16,384 hardware tanh per layer at 16 per cycle: 4,096 cycles per tile, what bounds it) runs
// under the other groups' products and waits.  The products, the epilogue's arithmetic and so the
// outputs are run_tiles', bit for bit.
constexpr int GROUPS = 3;            // 106 KB of weights and 3 x 32 KB of operands fill an SM's shared memory
constexpr int GROUP_TMEM = 512;      // TMEM columns of a CTA (3 x 128, a power of two)
constexpr size_t GS_A = WBYTES, GS_HDR = GS_A + (size_t)GROUPS * ABYTES, GROUP_SMEM = GS_HDR + NFLOAT * sizeof(float);

__device__ __forceinline__ void group_sync(int g) { asm volatile("barrier.sync %0, 128;" ::"r"(g + 1) : "memory"); }
// true in every thread of the group when p holds in one of them
__device__ __forceinline__ bool group_any(int g, bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.red.or.pred q, %2, 128, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(p ? 1u : 0u), "r"(g + 1)
      : "memory");
  return r != 0;
}

// Weights and header into shared memory (all threads; smem: GROUP_SMEM bytes).  Ends with a barrier.
__device__ __forceinline__ void load_net(unsigned char* smem, const unsigned char* __restrict__ blob) {
  const uint4* src = reinterpret_cast<const uint4*>(blob + WOFF);
  uint4* dst = reinterpret_cast<uint4*>(smem);
  for (int i = threadIdx.x; i < WBYTES / 16; i += blockDim.x) dst[i] = __ldg(src + i);
  float* hdr = reinterpret_cast<float*>(smem + GS_HDR);
  for (int i = threadIdx.x; i < NFLOAT; i += blockDim.x) hdr[i] = hdr_entry(i, __ldg(reinterpret_cast<const float*>(blob) + i));
  tc::fence_async_smem();
  __syncthreads();
}

// Network on the group's tile.  x: this thread's 16 standardised inputs; out: its 10 standardised
// outputs.  tmem: the group's 128 columns; mbar, phase: its completion barrier.  Returns false, in every
// thread of the group, if a wait gave up.
__device__ __forceinline__ bool run_group(unsigned char* smem, int g, const float* x, uint32_t tmem, uint32_t mbar,
                                          uint32_t& phase, float* out) {
  const int t = threadIdx.x & 127;
  unsigned char* A = smem + GS_A + (size_t)g * ABYTES;
  const float* bias = reinterpret_cast<const float*>(smem + GS_HDR) + F_BIAS;
  const uint32_t lane_addr = tmem + ((uint32_t)(t & 96) << 16);
  store_row16(A, t, 0, 16, x);
  for (int l = 0; l < 5; ++l) {
    tc::fence_async_smem();
    tc::fence_before_sync();
    group_sync(g);
    tc::fence_after_sync();
    if (t == 0) {
      const int K = kdim(l), N = ndim(l);
      const uint32_t a0 = tc::smem_addr(A), b0 = tc::smem_addr(smem + woff(l));
      const uint32_t sbo = (uint32_t)(K / 8) * 128u, idesc = tc::idesc_bf16_f32(128, N);
      for (int s = 0; s < K / 16; ++s)
        tc::mma_bf16(tmem, tc::smem_desc(a0 + 256u * s, 128u, sbo), tc::smem_desc(b0 + 256u * s, 128u, sbo), idesc,
                     s > 0 ? 1u : 0u);
      tc::mma_commit(mbar);
    }
    const bool mine = tc::mbar_wait(mbar, phase);
    phase ^= 1u;
    tc::fence_after_sync();
    if (group_any(g, !mine)) {
      tc::mbar_wait(mbar, phase ^ 1u);   // give the abandoned products a bounded time to land
      return false;
    }
    if (l < 4) {
#pragma unroll 1
      for (int c = 0; c < 8; c += 2) {   // two loads in flight
        uint32_t r0[16], r1[16];
        tc::tmem_ld16_issue(lane_addr + 16u * c, r0);
        tc::tmem_ld16_issue(lane_addr + 16u * c + 16u, r1);
        tc::tmem_wait_ld();
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r0[i]);
        silu16(v, bias + l * 128 + 16 * c);
        store_row16(A, t, c, 128, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r1[i]);
        silu16(v, bias + l * 128 + 16 * c + 16);
        store_row16(A, t, c + 1, 128, v);
      }
    } else {
      float v[16];
      tc::tmem_ld16(lane_addr, v);
#pragma unroll
      for (int i = 0; i < 10; ++i) out[i] = v[i] + bias[4 * 128 + i];
      tc::fence_before_sync();
    }
  }
  return true;
}

// Tensor-core resources of a CTA of GROUPS warpgroups: 512 TMEM columns and a barrier per group.
struct GroupTc {
  uint64_t bar[GROUPS];
  uint32_t slot;
};
__device__ __forceinline__ uint32_t group_acquire(GroupTc* tcs) {
  if (threadIdx.x < 32) {
    tc::tmem_alloc(tc::smem_addr(&tcs->slot), GROUP_TMEM);
    tc::tmem_relinquish();
  }
  if (threadIdx.x == 0) {
    for (int g = 0; g < GROUPS; ++g) tc::mbar_init(tc::smem_addr(&tcs->bar[g]), 1);
    tc::fence_mbar_init();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  return tcs->slot;
}
__device__ __forceinline__ void group_release(uint32_t tmem) {
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (threadIdx.x < 32) tc::tmem_dealloc(tmem, GROUP_TMEM);
}

}  // namespace mlp
}  // namespace ct
