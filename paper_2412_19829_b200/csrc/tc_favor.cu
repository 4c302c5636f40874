// Positive random features of the linear heads (Sec. III-A / III-C: "positive orthogonal random
// features"; the formula is the cited Performer paper's):
//     phi_W(x)[a] = exp(<w_a, x> - |x|^2 / 2) / sqrt(d),   a = 0 .. d-1,
// for every token of Q and of K of the linear heads, written as bf16 tensors [B, heads, N, d] that the
// chunked linear-attention kernels then read in place of Q and K (with their own feature map
// switched off).  A positive factor common to all features of one query cancels in
// o_i = phi(q_i)^T S / <phi(q_i), z>, so the query features are taken relative to the row's largest
// projection, exp(<w_a, q> - max_a <w_a, q>) (no |q|^2 / 2, no 1 / sqrt(d)): they then lie in (0, 1]
// and their products with the state stay inside the range of fp32 however small the key features
// are.  The key features (and with them the state S, z) are the definition's.
//
// A CTA (one per SM) takes a run of consecutive 128-token tiles of Q, then of K, in (head, tile) order, so that a head's
// projection W (d x d, row a = w_a) is loaded once for many tiles.  Per tile X (128 x d, by TMA into a ring of 6 buffers, 12
// at d = 64): one tcgen05.mma group computes Y = X W^T (M = 128, N = d, K = d, both operands K-major from shared memory) into
// one of four TMEM buffers; 128 threads, one per token (a group of four warps for each of those), take the exponentials and
// write the features over the tile, which a TMA store ships (rows past the end of the sequence are clipped).  Bound by the
// memory system: X in and features out once each, 26 heads of 32K tokens, d = 128: 148 us = 5.9 TB/s.  A buffer is away for
// about 7 us (load, product, exponentials, store), so what counts is how many there are: with two CTAs per SM of two
// buffers and a copy of W each it took 156 us, and the layer of 16 heads x 4 x 2048 tokens 71 against 66; with one CTA per
// tile, which did load, product, exponentials and store one after the other, 181.  L2 eviction hints make it slower.
#include "common.cuh"
#include "sm100.cuh"

namespace gf {
namespace {

using namespace sm100;

constexpr int kFavorThreads = 19 * 32;  // warps 0-15: four groups of one thread per token, 16: loads, 17: products, 18: stores
constexpr float kLog2eF = 1.4426950408889634f;

struct FavorParams {
  int h_begin, h_count;  // heads [h_begin, h_begin + h_count) of the input tensors
  int ntile;             // 128-token tiles of a head
  long long rows;        // (batch, head) pairs; tiles are numbered Q first, then K: 2 x rows x ntile
  unsigned int* status;
};

template <int D>
struct FavorCfg {
  static constexpr int kTile = 128 * D * 2, kW = D * D * 2;
  static constexpr int kX = (D == 128) ? 6 : 12;  // tiles in shared memory
  static constexpr int kBytes = kX * kTile + kW + 1024;
};

template <int D>
__global__ void __launch_bounds__(kFavorThreads, 1)
favor_tc_kernel(const __grid_constant__ CUtensorMap mxq, const __grid_constant__ CUtensorMap mxk,
                const __grid_constant__ CUtensorMap mw, const __grid_constant__ CUtensorMap mfq,
                const __grid_constant__ CUtensorMap mfk, const FavorParams p) {
  using C = FavorCfg<D>;
  extern __shared__ __align__(1024) uint8_t raw_smem[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw_smem) + 1023) & ~(uintptr_t)1023);
  constexpr int NX = C::kX;
  uint8_t* sW = sm + NX * C::kTile;
  __shared__ __align__(8) uint64_t x_full[NX], x_free[NX], staged[NX], w_full, w_free, y_full[4], y_free[4];
  __shared__ uint32_t tmem_base_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < NX; ++i) {
      mbar_init(&x_full[i], 1);
      mbar_init(&x_free[i], 1);
      mbar_init(&staged[i], 128);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(&y_full[i], 1);
      mbar_init(&y_free[i], 128);
    }
    mbar_init(&w_full, 1);
    mbar_init(&w_free, 1);
    mbar_fence_init();
    tma_prefetch_desc(&mxq);
    tma_prefetch_desc(&mxk);
    tma_prefetch_desc(&mw);
    tma_prefetch_desc(&mfq);
    tma_prefetch_desc(&mfk);
  }
  if (warp == 17) {
    tmem_alloc(&tmem_base_s, 4 * D);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_s;
  grid_dep_wait();
  grid_dep_launch();

  // This CTA's tiles [t0, t1); tile number n of the CTA lives in buffer n % NX of shared memory and n & 3 of TMEM.
  const long long total = 2 * p.rows * p.ntile;
  const long long t0 = total * blockIdx.x / gridDim.x, t1 = total * (blockIdx.x + 1) / gridDim.x;
  struct Tile {
    bool is_k;
    int row, hl, b, i0;  // row: (batch, head) pair; W changes with hl
  };
  auto tile_at = [&](long long t) {
    Tile x;
    const long long r = t / p.ntile;
    x.is_k = r >= p.rows;
    x.row = (int)(x.is_k ? r - p.rows : r);
    x.hl = x.row % p.h_count;
    x.b = x.row / p.h_count;
    x.i0 = (int)(t - r * p.ntile) * 128;
    return x;
  };
  if (warp == 16) {
    if (elect_one()) {
      int have = -1;       // head whose W is loaded
      uint32_t loads = 0;  // of W
      uint32_t n = 0;
      for (long long t = t0; t < t1; ++t, ++n) {
        const Tile x = tile_at(t);
        const uint32_t s = n % NX;
        if (n >= NX && !mbar_wait(&x_free[s], (n / NX + 1) & 1, p.status, 900)) break;
        mbar_arrive_expect_tx(&x_full[s], C::kTile);
        for (int c = 0; c < D / 64; ++c)
          tma_load_4d(sm + s * C::kTile + c * 16384, x.is_k ? &mxk : &mxq, &x_full[s], c * 64, x.i0, p.h_begin + x.hl, x.b);
        if (x.hl != have) {  // the products with the old one are done
          if (loads >= 1 && !mbar_wait(&w_free, (loads - 1) & 1, p.status, 901)) break;
          mbar_arrive_expect_tx(&w_full, C::kW);
          for (int c = 0; c < D / 64; ++c) tma_load_4d(sW + c * (D * 128), &mw, &w_full, c * 64, 0, x.hl, 0);
          have = x.hl;
          ++loads;
        }
      }
    }
  } else if (warp == 17) {
    if (elect_one()) {
      constexpr uint32_t idesc = umma_idesc_bf16(128, D, false, false);
      int have = -1;
      uint32_t loads = 0, n = 0;
      for (long long t = t0; t < t1; ++t, ++n) {
        const int hl = tile_at(t).hl;
        const uint32_t s = n % NX, sy = n & 3;
        if (hl != have) {
          if (!mbar_wait(&w_full, loads & 1, p.status, 902)) break;
          have = hl;
          ++loads;
        }
        if (!mbar_wait(&x_full[s], (n / NX) & 1, p.status, 903)) break;
        if (n >= 4 && !mbar_wait(&y_free[sy], ((n >> 2) + 1) & 1, p.status, 904)) break;
        tc_fence_after_sync();
        const uint64_t dx = umma_smem_desc(smem_u32(sm) + s * C::kTile, 16, 1024), dw = umma_smem_desc(smem_u32(sW), 16, 1024);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          umma_ss(tmem + sy * D, umma_desc_add(dx, (ks >> 2) * 16384 + (ks & 3) * 32),
                  umma_desc_add(dw, (ks >> 2) * (D * 128) + (ks & 3) * 32), idesc, ks > 0);
        umma_commit(&y_full[sy]);
        if (t + 1 < t1 && tile_at(t + 1).hl != hl) umma_commit(&w_free);
      }
    }
  } else if (warp == 18) {
    if (elect_one()) {
      uint32_t n = 0;
      for (long long t = t0; t < t1; ++t, ++n) {
        const Tile x = tile_at(t);
        const uint32_t s = n % NX;
        if (!mbar_wait(&staged[s], (n / NX) & 1, p.status, 905)) break;
        for (int c = 0; c < D / 64; ++c)
          tma_store_4d(x.is_k ? &mfk : &mfq, sm + s * C::kTile + c * 16384, c * 64, x.i0, x.hl, x.b);
        tma_store_commit();
        tma_store_wait_read<1>();  // the one before has been read out
        if (n >= 1) mbar_arrive(&x_free[(n - 1) % NX]);
      }
      tma_store_wait_all<0>();
    }
  } else {
    const uint32_t sy = warp >> 2;  // this group's TMEM buffer: every fourth tile of the CTA
    const int quarter = warp & 3;  // TMEM lane quarter this warp may touch
    const int r = quarter * 32 + lane;
    const uint32_t ty = tmem + sy * D + ((uint32_t)(quarter * 32) << 16);
    uint32_t n = sy;
    for (long long t = t0 + sy; t < t1; t += 4, n += 4) {
      uint8_t* sX = sm + (n % NX) * C::kTile;
      const bool is_k = tile_at(t).is_k;
      // the products are done: X is no longer read by the tensor core
      const bool ok = mbar_wait(&y_full[sy], (n >> 2) & 1, p.status, 906);
      if (__any_sync(0xffffffffu, !ok)) break;
      tc_fence_after_sync();
      // keys: exp(y - |x|^2 / 2) / sqrt(d) = 2^((y - |x|^2 / 2) log2(e) - log2(d) / 2);
      // queries: exp(y - max_a y) (the row's factor cancels in the output)
      float shift;
      if (is_k) {  // |x|^2 of this thread's token from the tile (128-byte swizzle: 16-byte chunks)
        // One running sum in column order: the last bit of a bf16 feature depends on the order.  In two halves (even and
        // odd columns) 3 of 1000 features were the neighbouring bf16 value, which moved the outputs by 1.4e-4.
        float n2 = 0.f;
#pragma unroll
        for (int c8 = 0; c8 < D / 8; ++c8) {
          const uint4 v4 = *reinterpret_cast<const uint4*>(sX + (c8 >> 3) * 16384 + swz128_offset(r, (c8 & 7) * 8));
          const uint32_t w4[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w4[e]));
            n2 = fmaf(f.x, f.x, n2);
            n2 = fmaf(f.y, f.y, n2);
          }
        }
        shift = -0.5f * n2 * kLog2eF - 0.5f * log2f((float)D);
      } else {
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
          uint32_t y[32];
          tmem_ld32(ty + c * 32, y);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; ++e) mx[e & 3] = fmaxf(mx[e & 3], __uint_as_float(y[e]));
        }
        shift = -fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * kLog2eF;
      }
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        uint32_t y[32];
        tmem_ld32(ty + c * 32, y);
        tmem_wait_ld();
        uint8_t* box = sX + (c >> 1) * 16384;
#pragma unroll
        for (int g = 0; g < 4; ++g) {  // 4 chunks of 8 features
          float f[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) f[e] = exp2f(fmaf(__uint_as_float(y[8 * g + e]), kLog2eF, shift));
          uint4 val;
          val.x = pack_bf16(f[0], f[1]);
          val.y = pack_bf16(f[2], f[3]);
          val.z = pack_bf16(f[4], f[5]);
          val.w = pack_bf16(f[6], f[7]);
          *reinterpret_cast<uint4*>(box + swz128_offset(r, (c & 1) * 32 + g * 8)) = val;
        }
      }
      tc_fence_before_sync();
      mbar_arrive(&y_free[sy]);
      fence_proxy_async_smem();
      mbar_arrive(&staged[n % NX]);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 17) tmem_dealloc(tmem, 4 * D);
}

}  // namespace

cudaError_t launch_favor_features_tc(const void* q, const void* k, const void* W, void* fq, void* fk, int B, int H,
                                     int N, int d, int layout, int h_begin, int h_count, WsHeader* ws,
                                     cudaStream_t stream) {
  if (h_count <= 0) return cudaSuccess;
  CUtensorMap mxq, mxk, mw, mfq, mfk;
  if (!make_qkv_tensor_map(&mxq, q, B, H, N, d, layout, 128) || !make_qkv_tensor_map(&mxk, k, B, H, N, d, layout, 128) ||
      !make_qkv_tensor_map(&mfq, fq, B, h_count, N, d, GF_BHND, 128) ||
      !make_qkv_tensor_map(&mfk, fk, B, h_count, N, d, GF_BHND, 128) ||
      !make_qkv_tensor_map(&mw, W, 1, h_count, d, d, GF_BHND, d))  // [1, heads, d features, d inputs]: box of d rows
    return cudaErrorInvalidValue;
  FavorParams p;
  p.h_begin = h_begin;
  p.h_count = h_count;
  p.status = &ws->status;
  p.rows = (long long)B * h_count;
  p.ntile = (N + 127) / 128;
  const long long total = 2 * p.rows * p.ntile;
  if (p.rows > 0x7fffffffLL || p.ntile > 65535) return cudaErrorInvalidValue;  // (tiles: more than 8 million tokens)
  auto launch = [&](auto kern, int smem) -> cudaError_t {
    int dev = 0, sms = 0;
    cudaError_t err = device_info(&dev, &sms);
    if (err == cudaSuccess) err = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), dev, smem);
    if (err != cudaSuccess) return err;
    const unsigned grid = (unsigned)(total < sms ? total : sms);
    return launch_link(kern, dim3(grid), dim3(kFavorThreads), smem, stream, mxq, mxk, mw, mfq, mfk, p);
  };
  return d == 64 ? launch(favor_tc_kernel<64>, FavorCfg<64>::kBytes) : launch(favor_tc_kernel<128>, FavorCfg<128>::kBytes);
}

}  // namespace gf
