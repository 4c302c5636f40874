// The feature map of the linear heads on packed bf16, as the tensor-core kernels apply it.
#pragma once

#include "common.cuh"
#include "sm100.cuh"

namespace gf {

// phi(x) = elu(x) + 1 = max(x, 0) + exp(min(x, 0)) on two packed bf16 values (branch free; the
// result is needed in bf16 anyway).  log2(e) is split in two bf16 terms so that the exponent
// argument carries only the rounding of one bf16 product.
__device__ __forceinline__ uint32_t phi_bf16x2(uint32_t w) {
  constexpr float kLog2e = 1.4426950408889634f;
  const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162*>(&w);
  const __nv_bfloat162 zero = __float2bfloat162_rn(0.f);
  const __nv_bfloat162 l2e_hi = __float2bfloat162_rn(1.4453125f);
  const __nv_bfloat162 l2e_lo = __float2bfloat162_rn(kLog2e - 1.4453125f);
  const __nv_bfloat162 t = __hmin2(__hfma2(x, l2e_lo, __hmul2(x, l2e_hi)), zero);
  uint32_t e;  // native packed exponential (the header's h2exp2 goes through two fp32 ex2 + converts)
  asm("ex2.approx.ftz.bf16x2 %0, %1;" : "=r"(e) : "r"(*reinterpret_cast<const uint32_t*>(&t)));
  const __nv_bfloat162 f = __hadd2(__hmax2(x, zero), *reinterpret_cast<const __nv_bfloat162*>(&e));
  return *reinterpret_cast<const uint32_t*>(&f);
}

// kId: the tensors the kernel reads as Q and K already hold features (positive random features
// computed by a kernel of their own): the feature map here is the identity.
template <bool kId>
__device__ __forceinline__ uint32_t phi_sel(uint32_t w) {
  if constexpr (kId) return w;
  else return phi_bf16x2(w);
}

// phi on a K tile (128 rows in boxes of 64 columns, 128-byte swizzle) in place in shared memory, by NT threads: a
// thread (number tt) takes one 16-byte column chunk of rows sixteen apart, so that the tile is spread over all of them
// whatever D is (with four rows per thread half of 512 threads had nothing to do at D = 64: 832 chains of 4096 tokens
// 388 -> 364 us).  Rows from n_valid on (past the end of the sequence) become zero.
template <int D, int NT>
__device__ __forceinline__ void transform_k_tile(uint8_t* tile, int tt, int n_valid) {
  constexpr int kBox = 16384, kChunks = D / 8, kRows = 8 * 16 * kChunks / NT;
  const int cc = (tt >> 4) % kChunks, row0 = (tt & 15) + 16 * kRows * ((tt >> 4) / kChunks), cin = cc & 7;
  uint8_t* kb = tile + (cc >> 3) * kBox;
  uint4 raw[kRows];
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int row = row0 + 16 * k;
    raw[k] = *reinterpret_cast<const uint4*>(kb + row * 128 + ((cin ^ (row & 7)) << 4));
  }
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    raw[k].x = phi_bf16x2(raw[k].x);
    raw[k].y = phi_bf16x2(raw[k].y);
    raw[k].z = phi_bf16x2(raw[k].z);
    raw[k].w = phi_bf16x2(raw[k].w);
  }
  if (n_valid < 128) {
#pragma unroll
    for (int k = 0; k < kRows; ++k)
      if (row0 + 16 * k >= n_valid) raw[k] = make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int row = row0 + 16 * k;
    *reinterpret_cast<uint4*>(kb + row * 128 + ((cin ^ (row & 7)) << 4)) = raw[k];
  }
  sm100::fence_proxy_async_smem();
}

}  // namespace gf
