// FFMA kernels (fp32 arithmetic) of libgformer.
//
// The linear heads of fp32 tensors where neither the tcgen05 kernels nor those of split tf32 products apply (the
// bidirectional layer's sums, positive random features), and the memory-bound decode step and ring export, which have
// no dense contraction worth a tensor core.  Plain data-parallel kernels: no inter-CTA communication, no spin waits.
#include <cooperative_groups.h>

#include "common.cuh"

namespace gf {
namespace {

template <typename T> struct Vec4;
template <> struct Vec4<float> {
  static __device__ __forceinline__ float4 load(const float* p) { return *reinterpret_cast<const float4*>(p); }
  static __device__ __forceinline__ void store(float* p, float4 x) { *reinterpret_cast<float4*>(p) = x; }
};
template <> struct Vec4<__nv_bfloat16> {
  static __device__ __forceinline__ float4 load(const __nv_bfloat16* p) {
    uint2 raw = *reinterpret_cast<const uint2*>(p);
    __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162*>(&raw.x);
    __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162*>(&raw.y);
    float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
    return make_float4(fa.x, fa.y, fb.x, fb.y);
  }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, float4 x) {
    __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y);
    __nv_bfloat162 b = __floats2bfloat162_rn(x.z, x.w);
    uint2 raw;
    raw.x = *reinterpret_cast<uint32_t*>(&a);
    raw.y = *reinterpret_cast<uint32_t*>(&b);
    *reinterpret_cast<uint2*>(p) = raw;
  }
};

// ------------------------------------------------------------------------------------
// Linear attention token by token: Algorithm 1 with positive random features, and both feature maps of the bidirectional
// layer (the causal heads with elu + 1 are linear_walk_kernel).
// One CTA = one head x one slice of 32 value columns.  Warp g owns features
// a in [g*D/8, (g+1)*D/8); lane c owns value column c of the slice.  S lives in registers
// (D/8 per thread), z is replicated per lane.  Tokens are staged 16 at a time.
// global_sum != 0: the unmasked form of the bidirectional layer (Sec. II-B) -- a first sweep over
// the tokens only accumulates S and z, a second one only reads them out.
// ------------------------------------------------------------------------------------
template <typename T, int D>
__global__ void __launch_bounds__(256)
linear_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                   T* __restrict__ o, int N, Strides st, int h_begin, int h_count,
                   float* __restrict__ S_io, float* __restrict__ z_io, int zero_init, int global_sum,
                   const T* __restrict__ W /* [h_count, D, D] or null: elu + 1 */, Place place) {
  constexpr int TB = 16;
  constexpr int AR = D / 8;
  __shared__ float qs[TB][D];
  __shared__ float ks[TB][D];
  __shared__ float xr[TB][D + 1];  // raw rows while the positive random features are taken (W != null)
  __shared__ float vs[TB][32];
  __shared__ float red[TB][8][33];
  __shared__ float redden[TB][8];

  begin(place);
  const int slice = blockIdx.x, hl = blockIdx.y, b = blockIdx.z;
  const int h = h_begin + hl;
  const long long base = (long long)b * st.b + (long long)h * st.h;
  const int tid = threadIdx.x, c = tid & 31, g = tid >> 5;
  const long long sidx = (long long)b * h_count + hl;

  float S[AR], zr[AR];
#pragma unroll
  for (int a = 0; a < AR; ++a) {
    S[a] = 0.f;
    zr[a] = 0.f;
  }
  if (S_io != nullptr && !zero_init) {
#pragma unroll
    for (int a = 0; a < AR; ++a) {
      S[a] = S_io[(sidx * D + (g * AR + a)) * D + slice * 32 + c];
      zr[a] = z_io[sidx * D + g * AR + a];
    }
    // the slices of a chain are one cluster: the one that overwrites z waits until all have read it
    cooperative_groups::this_cluster().sync();
  }

  for (int sweep = global_sum ? 0 : 1; sweep < 2; ++sweep) {
  const bool accumulate = !global_sum || sweep == 0, readout = !global_sum || sweep == 1;
  for (int n0 = 0; n0 < N; n0 += TB) {
    __syncthreads();
    if (W == nullptr) {
      for (int idx = tid; idx < TB * D; idx += 256) {
        const int tok = idx / D, a = idx % D;
        const int n = n0 + tok;
        float qq = 0.f, kk = 0.f;
        if (n < N) {
          qq = phi_elu1(to_f32(q[base + (long long)n * st.n + a]));
          kk = phi_elu1(to_f32(k[base + (long long)n * st.n + a]));
        }
        qs[tok][a] = qq;
        ks[tok][a] = kk;  // 0 for rows past N: they must not enter the state
      }
    } else {
      // phi_W(x)[a] = exp(<w_a, x> - |x|^2 / 2) / sqrt(D) (Sec. III-A / III-C), Q rows first, then K rows.
      // A factor common to all features of a query cancels in the output: the query features are taken
      // relative to the row's largest projection, exp(<w_a, q> - max_a <w_a, q>), which keeps their
      // products with the state inside the range of fp32.
      const T* Wh = W + (long long)hl * D * D;
      for (int which = 0; which < 2; ++which) {
        const T* src = which ? k : q;
        float (*dst)[D] = which ? ks : qs;
        for (int idx = tid; idx < TB * D; idx += 256) {
          const int tok = idx / D, a = idx % D;
          const int n = n0 + tok;
          xr[tok][a] = (n < N) ? to_f32(src[base + (long long)n * st.n + a]) : 0.f;
        }
        __syncthreads();
        for (int idx = tid; idx < TB * D; idx += 256) {
          const int tok = idx / D, a = idx % D;
          float proj = 0.f, n2 = 0.f;
          for (int cc = 0; cc < D; ++cc) {
            const float x = xr[tok][cc];
            proj = fmaf(to_f32(Wh[(long long)a * D + cc]), x, proj);
            n2 = fmaf(x, x, n2);
          }
          if (which) dst[tok][a] = (n0 + tok < N) ? expf(proj - 0.5f * n2) * rsqrtf((float)D) : 0.f;
          else dst[tok][a] = proj;
        }
        __syncthreads();
        if (which == 0) {  // queries: relative to the row maximum
          float e[TB * D / 256];
          for (int i = 0; i < TB * D / 256; ++i) {
            const int idx = tid + 256 * i, tok = idx / D, a = idx % D;
            float mx = -INFINITY;
            for (int cc = 0; cc < D; ++cc) mx = fmaxf(mx, qs[tok][cc]);
            e[i] = expf(qs[tok][a] - mx);
          }
          __syncthreads();
          for (int i = 0; i < TB * D / 256; ++i) {
            const int idx = tid + 256 * i;
            qs[idx / D][idx % D] = e[i];
          }
          __syncthreads();
        }
      }
    }
    for (int idx = tid; idx < TB * 32; idx += 256) {
      const int tok = idx >> 5, cc = idx & 31;
      const int n = n0 + tok;
      vs[tok][cc] = (n < N) ? to_f32(v[base + (long long)n * st.n + slice * 32 + cc]) : 0.f;
    }
    __syncthreads();
#pragma unroll 1
    for (int tok = 0; tok < TB; ++tok) {
      const float vv = vs[tok][c];
      float num = 0.f, den = 0.f;
#pragma unroll
      for (int a = 0; a < AR; ++a) {
        const float kk = accumulate ? ks[tok][g * AR + a] : 0.f;
        const float qq = qs[tok][g * AR + a];
        S[a] = fmaf(kk, vv, S[a]);
        zr[a] += kk;
        num = fmaf(qq, S[a], num);
        den = fmaf(qq, zr[a], den);
      }
      red[tok][g][c] = num;
      if (c == 0) redden[tok][g] = den;
    }
    __syncthreads();
    for (int idx = tid; idx < TB * 32; idx += 256) {
      const int tok = idx >> 5, cc = idx & 31;
      const int n = n0 + tok;
      float num = 0.f, den = 0.f;
#pragma unroll
      for (int gg = 0; gg < 8; ++gg) {
        num += red[tok][gg][cc];
        den += redden[tok][gg];
      }
      if (n < N && readout) o[base + (long long)n * st.n + slice * 32 + cc] = from_f32<T>(num / den);
    }
  }
  }
  if (S_io != nullptr) {
#pragma unroll
    for (int a = 0; a < AR; ++a) {
      S_io[(sidx * D + (g * AR + a)) * D + slice * 32 + c] = S[a];
      if (slice == 0 && c == 0) z_io[sidx * D + g * AR + a] = zr[a];
    }
  }
}

// ------------------------------------------------------------------------------------
// Ring export: the last min(N, w) keys/values of the windowed heads into slot j mod w.
// It runs beside the linear heads, whose kernel leaves 4096 registers of an SM: 128 threads of 32.  A thread moves two 16-byte
// pieces of K and two of V, all four loads in flight at once.
// ------------------------------------------------------------------------------------
constexpr int kExportThreads = 128;
__global__ void __launch_bounds__(kExportThreads, 16)
export_ring_kernel(const uint4* __restrict__ k, const uint4* __restrict__ v, uint4* __restrict__ kc, uint4* __restrict__ vc,
                   int N, int d16, int w, int wn, Strides st16, int h_sparse, unsigned int total) {
  // d16, st16: row length and strides in 16-byte pieces
  grid_dep_launch();
  uint4 x[2], y[2];
  long long dst[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const unsigned int idx = (blockIdx.x * 2u + e) * kExportThreads + threadIdx.x;
    dst[e] = -1;
    if (idx < total) {
      const unsigned int row = idx / (unsigned)d16, c = idx - row * d16;
      const unsigned int bh = row / (unsigned)wn, b = bh / (unsigned)h_sparse;
      const int j = N - wn + (int)(row - bh * wn);
      const long long src = b * st16.b + (bh - b * h_sparse) * st16.h + j * st16.n + c;
      x[e] = k[src];
      y[e] = v[src];
      dst[e] = ((long long)bh * w + j % w) * d16 + c;
    }
  }
#pragma unroll
  for (int e = 0; e < 2; ++e)
    if (dst[e] >= 0) {
      kc[dst[e]] = x[e];
      vc[dst[e]] = y[e];
    }
  if (blockIdx.x == 0) grid_dep_wait();
}

// ------------------------------------------------------------------------------------
// Decode step: one CTA per (b, h).
// ------------------------------------------------------------------------------------
// A 16-byte load that stays where it is written: several in a row are all in flight before the first use (left to
// itself the compiler, short of registers, pairs every load with its use).
__device__ __forceinline__ uint4 ld16_in_order(const void* p) {
  uint4 r;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p) : "memory");
  return r;
}
// 16 bytes of a ring row (4 floats or 8 bf16) against the matching entries of a vector in shared memory
template <typename T> struct Row16;
template <> struct Row16<float> {
  static constexpr int kElems = 4;
  static __device__ __forceinline__ float dot(uint4 raw, const float* qv) {
    const float4 q4 = *reinterpret_cast<const float4*>(qv);
    return __uint_as_float(raw.x) * q4.x + __uint_as_float(raw.y) * q4.y + __uint_as_float(raw.z) * q4.z +
           __uint_as_float(raw.w) * q4.w;
  }
  static __device__ __forceinline__ void axpy(uint4 raw, float p, float* acc) {
    acc[0] = fmaf(p, __uint_as_float(raw.x), acc[0]);
    acc[1] = fmaf(p, __uint_as_float(raw.y), acc[1]);
    acc[2] = fmaf(p, __uint_as_float(raw.z), acc[2]);
    acc[3] = fmaf(p, __uint_as_float(raw.w), acc[3]);
  }
};
template <> struct Row16<__nv_bfloat16> {
  static constexpr int kElems = 8;
  static __device__ __forceinline__ float dot(uint4 raw, const float* qv) {
    const float4 qa = *reinterpret_cast<const float4*>(qv), qb = *reinterpret_cast<const float4*>(qv + 4);
    float a0 = __uint_as_float(raw.x << 16) * qa.x, a1 = __uint_as_float(raw.x & 0xffff0000u) * qa.y;
    a0 = fmaf(__uint_as_float(raw.y << 16), qa.z, a0);
    a1 = fmaf(__uint_as_float(raw.y & 0xffff0000u), qa.w, a1);
    a0 = fmaf(__uint_as_float(raw.z << 16), qb.x, a0);
    a1 = fmaf(__uint_as_float(raw.z & 0xffff0000u), qb.y, a1);
    a0 = fmaf(__uint_as_float(raw.w << 16), qb.z, a0);
    a1 = fmaf(__uint_as_float(raw.w & 0xffff0000u), qb.w, a1);
    return a0 + a1;
  }
  static __device__ __forceinline__ void axpy(uint4 raw, float p, float* acc) {
    acc[0] = fmaf(p, __uint_as_float(raw.x << 16), acc[0]);
    acc[1] = fmaf(p, __uint_as_float(raw.x & 0xffff0000u), acc[1]);
    acc[2] = fmaf(p, __uint_as_float(raw.y << 16), acc[2]);
    acc[3] = fmaf(p, __uint_as_float(raw.y & 0xffff0000u), acc[3]);
    acc[4] = fmaf(p, __uint_as_float(raw.z << 16), acc[4]);
    acc[5] = fmaf(p, __uint_as_float(raw.z & 0xffff0000u), acc[5]);
    acc[6] = fmaf(p, __uint_as_float(raw.w << 16), acc[6]);
    acc[7] = fmaf(p, __uint_as_float(raw.w & 0xffff0000u), acc[7]);
  }
};

// fmaxf drops a NaN
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

__device__ __forceinline__ float block_reduce(float x, bool is_max, float* scratch /* 33 floats */) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float y = __shfl_xor_sync(0xffffffffu, x, off);
    x = is_max ? fmaxf(x, y) : x + y;
  }
  __syncthreads();
  if (lane == 0) scratch[wid] = x;
  __syncthreads();
  if (wid == 0) {
    float y = (lane < nw) ? scratch[lane] : (is_max ? -INFINITY : 0.f);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float u = __shfl_xor_sync(0xffffffffu, y, off);
      y = is_max ? fmaxf(y, u) : y + u;
    }
    if (lane == 0) scratch[32] = y;
  }
  __syncthreads();
  return scratch[32];
}

// One CTA per (batch, head).  What bounds a step is round trips to L2 or HBM, so a thread has as many loads in flight as
// its registers hold: NW key pieces and the NW value pieces of the same slots (windowed heads), or four pieces of S, the
// first of them asked for before q and k have arrived.
//   windowed heads  a group of threads that share a slot keeps a running maximum, sum and output of its own over the
//                   slots it meets; the groups are combined once at the end, so that no barrier stands between keys
//                   and values.
// CTAS per SM and NW go together (registers): four with NW = 4, six with NW = 2 (decode_dispatch says which when).
// Measured at B = 64, H = 16, d = 64, w = 256: 8.3 us a step (two loads in flight, scores and values apart by two
// block-wide reductions: 10.3); B = 8, H = 32, d = 128, w = 512: 12.3 (18.6); B = 128, H = 32, d = 128, w = 512: 98 us =
// 5.8 TB/s (110).
template <typename T, int D, int CTAS, int NW>
__global__ void __launch_bounds__(256, CTAS)
decode_step_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                   T* __restrict__ o, T* __restrict__ kc, T* __restrict__ vc, float* __restrict__ S,
                   float* __restrict__ z, long long t_all, long long* __restrict__ t_seq, int H, int w,
                   int h_sparse, float scale, const T* __restrict__ W /* [H - h_sparse, D, D] or null: elu + 1 */) {
  constexpr int NB = 4;
  constexpr int D4 = D / 4;
  constexpr int G = 256 / D4;  // thread groups along the reduced dimension
  // windowed heads: a ring row is read 16 bytes per thread: TPS threads per slot (8, 16 or 32: a group never straddles
  // a warp), GW slots at a time
  constexpr int EPT = Row16<T>::kElems, TPS = D / EPT, GW = 256 / TPS;
  __shared__ __align__(16) float qs[D];
  __shared__ __align__(16) float ks[D];
  __shared__ float scratch[33];
  __shared__ float gm[GW], gl[GW];
  __shared__ __align__(16) float part[GW][D];  // GW >= G

  grid_dep_wait();  // (nothing is read or written before the kernel before this one is complete)
  // the windowed heads of the whole batch come first: they take longest, so none of them should start late
  const int tid = threadIdx.x, id = blockIdx.x, n_win = (int)(gridDim.x / (unsigned)H) * h_sparse;
  int h, b;
  if (id < n_win) {
    b = id / h_sparse;
    h = id - b * h_sparse;
  } else {
    const int h_lin = H - h_sparse;
    b = (id - n_win) / h_lin;
    h = h_sparse + (id - n_win) - b * h_lin;
  }
  const long long io = ((long long)b * H + h) * D;
  // Position of this sequence: the whole batch in lock step, or its own entry of t_seq (a negative
  // entry marks an idle slot of the batch: state untouched, output row zero).  The sequence's H
  // CTAs count their arrivals in bits 48..62 of the entry; the last one clears the count and moves
  // the position on, so the step needs no second launch.
  // (A thread that loads none of the step's inputs fetches the position, so that the two global
  // round trips overlap.)
  float qv = 0.f;
  T kin = from_f32<T>(0.f), vin = from_f32<T>(0.f);
  long long t = t_all;
  if (tid < D) {
    qv = to_f32(q[io + tid]);
    kin = k[io + tid];
    vin = v[io + tid];
  }
  if (t_seq != nullptr) {
    __shared__ long long t_sh;
    if (tid == 255) {
      long long cur = *reinterpret_cast<const volatile long long*>(t_seq + b);
      if (cur >= 0) {
        unsigned long long* slot = reinterpret_cast<unsigned long long*>(t_seq + b);
        const unsigned long long old = atomicAdd(slot, 1ull << 48);
        cur = (long long)(old & ((1ull << 48) - 1));
        if ((old >> 48) + 1 == (unsigned long long)H) atomicAdd(slot, 1ull - ((unsigned long long)H << 48));
      }
      t_sh = cur;
    }
    __syncthreads();
    t = t_sh;
  }
  if (t < 0) {
    if (tid < D) o[io + tid] = from_f32<T>(0.f);
    return;
  }

  if (h < h_sparse) {
    T* kcb = kc + ((long long)b * h_sparse + h) * (long long)w * D;
    T* vcb = vc + ((long long)b * h_sparse + h) * (long long)w * D;
    const int cur = (int)(t % w);
    const int nvalid = (t + 1 < (long long)w) ? (int)(t + 1) : w;
    if (tid < D) {
      qs[tid] = qv;
      kcb[(long long)cur * D + tid] = kin;
      vcb[(long long)cur * D + tid] = vin;
    }
    // slot `cur` is read from the step input (same values)
    const int cw = tid % TPS, gw = tid / TPS;
    float m = -INFINITY, l = 0.f, acc[EPT];
#pragma unroll
    for (int e = 0; e < EPT; ++e) acc[e] = 0.f;
    for (int s0 = 0; s0 < nvalid; s0 += NW * GW) {  // uniform trip count: the shuffles below are warp-wide
      uint4 rk[NW], rv[NW];
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        const int sl = s0 + i * GW + gw;
        rk[i] = make_uint4(0u, 0u, 0u, 0u);
        if (sl < nvalid) rk[i] = ld16_in_order(((sl == cur) ? (k + io) : (kcb + (long long)sl * D)) + EPT * cw);
      }
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        const int sl = s0 + i * GW + gw;
        rv[i] = make_uint4(0u, 0u, 0u, 0u);
        if (sl < nvalid) rv[i] = ld16_in_order(((sl == cur) ? (v + io) : (vcb + (long long)sl * D)) + EPT * cw);
      }
      if (s0 == 0) __syncthreads();  // qs
      float s[NW], mx = m;
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        s[i] = Row16<T>::dot(rk[i], &qs[EPT * cw]);
#pragma unroll
        for (int off = TPS / 2; off > 0; off >>= 1) s[i] += __shfl_xor_sync(0xffffffffu, s[i], off);
        s[i] = (s0 + i * GW + gw < nvalid) ? s[i] * scale : -INFINITY;
        mx = max_nan(mx, s[i]);
      }
      if (mx != -INFINITY) {  // (a group that has met no slot yet keeps l = 0; a NaN goes on into l and the output)
        const float corr = expf(m - mx);
        m = mx;
        l *= corr;
#pragma unroll
        for (int e = 0; e < EPT; ++e) acc[e] *= corr;
#pragma unroll
        for (int i = 0; i < NW; ++i) {
          const float p = expf(s[i] - mx);
          l += p;
          Row16<T>::axpy(rv[i], p, acc);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < EPT; e += 4)
      *reinterpret_cast<float4*>(&part[gw][EPT * cw + e]) = make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
    if (cw == 0) {
      gm[gw] = m;
      gl[gw] = l;
    }
    grid_dep_launch();
    __syncthreads();
    if (tid < D) {
      float mx = -INFINITY, sum = 0.f, lsum = 0.f;
#pragma unroll
      for (int gi = 0; gi < GW; ++gi) mx = fmaxf(mx, gm[gi]);
#pragma unroll 8
      for (int gi = 0; gi < GW; ++gi) {
        const float f = expf(gm[gi] - mx);
        sum = fmaf(f, part[gi][tid], sum);
        lsum = fmaf(f, gl[gi], lsum);
      }
      o[io + tid] = from_f32<T>(sum / lsum);
    }
  } else {
    const int c4 = tid % D4, grp = tid / D4;
    const long long sidx = (long long)b * (H - h_sparse) + (h - h_sparse);
    float* Sb = S + sidx * D * D + 4 * c4;
    float* zb = z + sidx * D;
    uint4 raw[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) raw[i] = ld16_in_order(Sb + (grp + i * G) * D);
    const float4 vv = Vec4<T>::load(v + io + 4 * c4);
    const float zin = tid < D ? zb[tid] : 0.f;
    if (W != nullptr) {
      // positive random features of q_t and k_t (Sec. III-A / III-C): exp(<w_a, x> - |x|^2 / 2) / sqrt(D)
      // for the key; for the query exp(<w_a, q> - max_a <w_a, q>) (a factor common to its features cancels
      // in the output).  A warp per feature, lanes along the input dimension.
      if (tid < D) {
        part[0][tid] = qv;
        part[1][tid] = to_f32(kin);
      }
      const float n2k = block_reduce(tid < D ? to_f32(kin) * to_f32(kin) : 0.f, false, scratch);  // barriers inside publish part[]
      const T* Wh = W + (long long)(h - h_sparse) * D * D;
      const int lane = tid & 31, wid = tid >> 5;
      for (int a = wid; a < D; a += 8) {
        float pq = 0.f, pk = 0.f;
        for (int cc = lane; cc < D; cc += 32) {
          const float wv = to_f32(Wh[(long long)a * D + cc]);
          pq = fmaf(wv, part[0][cc], pq);
          pk = fmaf(wv, part[1][cc], pk);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          pq += __shfl_xor_sync(0xffffffffu, pq, off);
          pk += __shfl_xor_sync(0xffffffffu, pk, off);
        }
        if (lane == 0) {
          qs[a] = pq;
          ks[a] = expf(pk - 0.5f * n2k) * rsqrtf((float)D);
        }
      }
      __syncthreads();
      const float pmax = block_reduce(tid < D ? qs[tid] : -INFINITY, true, scratch);
      if (tid < D) qs[tid] = expf(qs[tid] - pmax);
      __syncthreads();
    }
    if (tid < D) {
      const float qp = W != nullptr ? qs[tid] : phi_elu1(qv);
      const float kp = W != nullptr ? ks[tid] : phi_elu1(to_f32(kin));
      qs[tid] = qp;
      ks[tid] = kp;
      const float zn = zin + kp;
      zb[tid] = zn;
      float den = qp * zn;  // the denominator: D/32 partial sums, one per warp
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
      if ((tid & 31) == 0) scratch[tid >> 5] = den;
    }
    __syncthreads();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int a0 = grp; a0 < D; a0 += NB * G) {
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const int a = a0 + i * G;
        const float kp = ks[a], qp = qs[a];
        float4 s4;
        s4.x = fmaf(kp, vv.x, __uint_as_float(raw[i].x));
        s4.y = fmaf(kp, vv.y, __uint_as_float(raw[i].y));
        s4.z = fmaf(kp, vv.z, __uint_as_float(raw[i].z));
        s4.w = fmaf(kp, vv.w, __uint_as_float(raw[i].w));
        *reinterpret_cast<float4*>(Sb + a * D) = s4;
        acc.x = fmaf(qp, s4.x, acc.x);
        acc.y = fmaf(qp, s4.y, acc.y);
        acc.z = fmaf(qp, s4.z, acc.z);
        acc.w = fmaf(qp, s4.w, acc.w);
      }
      if (a0 + NB * G < D) {
#pragma unroll
        for (int i = 0; i < NB; ++i) raw[i] = ld16_in_order(Sb + (a0 + (NB + i) * G) * D);
      }
    }
    *reinterpret_cast<float4*>(&part[grp][4 * c4]) = acc;
    grid_dep_launch();
    __syncthreads();
    if (tid < D) {
      float sum = 0.f, den = 0.f;
#pragma unroll
      for (int gi = 0; gi < G; ++gi) sum += part[gi][tid];
#pragma unroll
      for (int i = 0; i < D / 32; ++i) den += scratch[i];
      o[io + tid] = from_f32<T>(sum / den);
    }
  }
}

template <typename T>
cudaError_t linear_dispatch(const void* q, const void* k, const void* v, void* o, int B, int N, int d,
                            Strides st, int h_begin, int h_count, float* S_io, float* z_io, bool zero_init,
                            bool global_sum, cudaStream_t stream, Place place, const void* W) {
  return launch_link_clusters(S_io != nullptr && !zero_init ? d / 32 : 1,
                              d == 64 ? linear_simt_kernel<T, 64> : linear_simt_kernel<T, 128>, dim3(d / 32, h_count, B),
                              dim3(256), 0, stream, (const T*)q, (const T*)k, (const T*)v, (T*)o, N, st, h_begin, h_count, S_io,
                              z_io, zero_init ? 1 : 0, global_sum ? 1 : 0, (const T*)W, place);
}

template <typename T>
cudaError_t decode_dispatch(const void* q, const void* k, const void* v, void* o, void* kc, void* vc, float* S,
                            float* z, long long t, long long* t_seq, int B, int H, int d, int w, int h_sparse,
                            float scale, cudaStream_t stream, const void* W) {
  int dev = 0, sms = 0;
  const cudaError_t e = device_info(&dev, &sms);
  if (e != cudaSuccess) return e;
  // Four CTAs per SM with twice the loads in flight, unless heads of d = 64 (16 KB of state, or 256 bytes per slot) are
  // more than that makes one wave of: then six, 8.3 against 9.2 us at B = 64, H = 16 and 20.5 against 22.7 at 128 x 32.
  // Few or large ones want the loads: 4.2 against 5.2 us at 1 x 12, 70 against 84 at 32 x 12 with w = 4096, and at d = 128
  // 12.3 against 14.4 us at 8 x 32 (at 128 x 32, bound by HBM, there is no difference).
  auto* kern = d == 128                          ? decode_step_kernel<T, 128, 4, 4>
               : (long long)B * H <= 4LL * sms ? decode_step_kernel<T, 64, 4, 4>
                                                 : decode_step_kernel<T, 64, 6, 2>;
  return launch_link(kern, dim3((unsigned)(B * H)), dim3(256), 0, stream, (const T*)q, (const T*)k, (const T*)v, (T*)o,
                     (T*)kc, (T*)vc, S, z, t, t_seq, H, w, h_sparse, scale, (const T*)W);
}

}  // namespace

cudaError_t launch_linear_simt(const void* q, const void* k, const void* v, void* o, int B, int N, int d,
                               int dtype, Strides st, int h_begin, int h_count, float* S_io, float* z_io,
                               bool zero_init, cudaStream_t stream, Place place, bool global_sum, const void* W) {
  if (h_count <= 0 || B <= 0) return cudaSuccess;
  if (!global_sum && W == nullptr)
    return launch_linear_tiled(q, k, v, o, B, N, d, dtype, st, h_begin, h_count, S_io, z_io, zero_init, stream, place);
  if (dtype == GF_F32)
    return linear_dispatch<float>(q, k, v, o, B, N, d, st, h_begin, h_count, S_io, z_io, zero_init, global_sum,
                                  stream, place, W);
  return linear_dispatch<__nv_bfloat16>(q, k, v, o, B, N, d, st, h_begin, h_count, S_io, z_io, zero_init, global_sum,
                                        stream, place, W);
}

// (32-bit indices of 16-byte pieces: 64 GB of keys)
bool export_ring_fits(int B, int N, int d, int w, int dtype, int h_sparse) {
  const long long rows = (long long)B * h_sparse * (N < w ? N : w);
  return rows * (d / (dtype == GF_F32 ? 4 : 8)) <= 0xffffffffLL - 2 * kExportThreads;
}

cudaError_t launch_export_ring(const void* k, const void* v, void* k_cache, void* v_cache, int B, int N, int d,
                               int w, int dtype, Strides st, int h_sparse, cudaStream_t stream) {
  if (h_sparse <= 0 || B <= 0) return cudaSuccess;
  const int wn = N < w ? N : w, per16 = dtype == GF_F32 ? 4 : 8;  // elements of 16 bytes
  const long long total = (long long)B * h_sparse * wn * (d / per16);
  if (!export_ring_fits(B, N, d, w, dtype, h_sparse)) return cudaErrorInvalidValue;
  const Strides st16 = {st.b / per16, st.h / per16, st.n / per16};
  return launch_link(export_ring_kernel, dim3((unsigned)((total + 2 * kExportThreads - 1) / (2 * kExportThreads))),
                     dim3(kExportThreads), 0, stream, (const uint4*)k, (const uint4*)v, (uint4*)k_cache, (uint4*)v_cache, N,
                     d / per16, w, wn, st16, h_sparse, (unsigned)total);
}

namespace {
__global__ void clear_ws_kernel(Place place, unsigned int n16) {
  begin(place);
  const unsigned int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= sizeof(WsHeader) / 16 && i < n16) place.ws[i] = make_uint4(0u, 0u, 0u, 0u);
}
}  // namespace

cudaError_t launch_clear_ws(Place place, size_t bytes, cudaStream_t stream) {
  const size_t n16 = bytes / 16;
  if (n16 > 0x7fffffffu) return cudaErrorInvalidValue;
  return launch_link(clear_ws_kernel, dim3((unsigned)((n16 + 255) / 256)), dim3(256), 0, stream, place, (unsigned)n16);
}

cudaError_t launch_decode_step(const void* q, const void* k, const void* v, void* o, void* k_cache,
                               void* v_cache, float* S, float* z, long long t, long long* t_seq, int B, int H,
                               int d, int w, int h_sparse, float scale, int dtype, cudaStream_t stream,
                               const void* W) {
  if (dtype == GF_F32)
    return decode_dispatch<float>(q, k, v, o, k_cache, v_cache, S, z, t, t_seq, B, H, d, w, h_sparse, scale,
                                  stream, W);
  return decode_dispatch<__nv_bfloat16>(q, k, v, o, k_cache, v_cache, S, z, t, t_seq, B, H, d, w, h_sparse, scale,
                                        stream, W);
}

}  // namespace gf
