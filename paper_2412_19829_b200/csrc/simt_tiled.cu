// Attention in fp32 arithmetic: the windowed heads and the causal linear heads of fp32 tensors (and of bf16 ones when the
// tcgen05 kernels are switched off).
//
// The products run on the tensor cores as mma.sync with tf32 operands, each operand split in two (x = hi + lo, hi rounded to
// tf32's 11 bits, lo the exact rest, of which the tensor core reads 11 bits: a quarter of all operands lose their last one):
// hi hi + hi lo + lo hi, at most 2^-21.1 of a product away from it, 2^-23.7 in the mean square.  Sums of many terms come out nearer
// than with FFMA, which rounds after each; those of fewer than kFewKeys stay FFMA's.  The tensor core rounds towards zero when it adds to an accumulator, so no sum runs through it: the 8 products of
// an instruction (windowed heads: of two) start from zero and are added to the running sum on the CUDA cores, rounded to
// nearest.  Against 64 bits (2 x 12 heads of 2048 tokens, d = 64, w = 128; relative error, windowed and linear heads) that is
// 2.0e-7 and 1.1e-7, all sums in the accumulators 1.2e-6 and 1.1e-6, FFMA products 3.1e-7 and 1.5e-7.  (tcgen05.mma, four times
// as fast, could only add up in its accumulators.)
// Register-tiled FFMA products, which this replaced, were bound by shared memory (us, before and now): 8 x 12 heads of 2048
// tokens, d = 64, windowed (w = 128) 296 and 212, linear 240 and 172; d = 128 548 and 470, 843 and 686; the layer with 2
// windowed heads 246 and 171.  What bounds these is the latency of their instructions and the issue of them: 1400 a warp for a block of 32
// tokens, a quarter of them splitting operands, at 49 % of the issue slots (windowed 48 %); tensor pipe 36 % (42 %).  Not faster: operands split once
// and kept as pairs in shared memory (10 to 25 % slower), cvt.rna (8 %), the three products of a split apart (3 %).
#include <cooperative_groups.h>

#include <atomic>
#include <type_traits>

#include "common.cuh"

namespace gf {
namespace {

constexpr int kC = 32;    // tokens per block
constexpr int kLinThreads = 256;
constexpr int kW = 64;    // value columns per CTA of the linear heads
// Row strides in shared memory: the fragments are read 8 bytes (rows g, columns 2 t) or 4 bytes (rows t, columns g) per lane,
// both without bank conflicts when the stride is 8 mod 32; rows 2 t and 2 t + 1, or rows g and columns t, when it is 4.
constexpr int kLdV = kW + 8, kLdP = kC + 4;

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u), __uint_as_float(raw.y << 16),
                     __uint_as_float(raw.y & 0xffff0000u));
}
__device__ __forceinline__ void store4(float* p, float4 x) { *reinterpret_cast<float4*>(p) = x; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 x) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), b = __floats2bfloat162_rn(x.z, x.w);
  uint2 raw;
  raw.x = *reinterpret_cast<const uint32_t*>(&a);
  raw.y = *reinterpret_cast<const uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = raw;
}
__device__ __forceinline__ void store2(float* p, float x, float y) { *reinterpret_cast<float2*>(p) = make_float2(x, y); }
__device__ __forceinline__ void store2(__nv_bfloat16* p, float x, float y) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(x, y);
}
__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float2 lds2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float4 phi4(float4 x) {
  return make_float4(phi_elu1(x.x), phi_elu1(x.y), phi_elu1(x.z), phi_elu1(x.w));
}
// acc += a * b, element by element of b
__device__ __forceinline__ void axpy4(float4& acc, float a, float4 b) {
  acc.x = fmaf(a, b.x, acc.x);
  acc.y = fmaf(a, b.y, acc.y);
  acc.z = fmaf(a, b.z, acc.z);
  acc.w = fmaf(a, b.w, acc.w);
}
__device__ __forceinline__ float dot4(float4 a, float4 b, float acc) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}
__device__ __forceinline__ bool is_nan(float x) { return x != x; }
__device__ __forceinline__ bool is_finite(float x) { return (__float_as_uint(x) & 0x7f800000u) != 0x7f800000u; }

// ------------------------------------------------------------------------------------ products
struct Split {
  uint32_t hi, lo;
};
__device__ __forceinline__ Split split(float x) {
  const uint32_t hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  return {hi, __float_as_uint(x - __uint_as_float(hi))};
}
// Lane (g, t) = (lane / 4, lane % 4) of an m16n8k8 product holds A[g | g + 8][t | t + 4], B[t | t + 4][g] and
// C[g | g + 8][2 t | 2 t + 1].  The order of the contracted index is free as long as A and B agree.
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t a0, const uint32_t a1, const uint32_t a2, const uint32_t a3,
                                         const uint32_t b0, const uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// d += the 8 (or, small: the corrections of the 8) products of an element
__device__ __forceinline__ void product_small(float (&d)[4], const Split (&a)[4], const Split b0, const Split b1) {
  mma_tf32(d, a[0].lo, a[1].lo, a[2].lo, a[3].lo, b0.hi, b1.hi);
  mma_tf32(d, a[0].hi, a[1].hi, a[2].hi, a[3].hi, b0.lo, b1.lo);
}
__device__ __forceinline__ void product_big(float (&d)[4], const Split (&a)[4], const Split b0, const Split b1) {
  mma_tf32(d, a[0].hi, a[1].hi, a[2].hi, a[3].hi, b0.hi, b1.hi);
}
// acc += A B over 8 contracted elements, or 16
__device__ __forceinline__ void product8(float (&acc)[4], const Split (&a)[4], const Split b0, const Split b1) {
  float d[4] = {0.f, 0.f, 0.f, 0.f};
  product_small(d, a, b0, b1);
  product_big(d, a, b0, b1);
#pragma unroll
  for (int e = 0; e < 4; ++e) acc[e] += d[e];
}
__device__ __forceinline__ void product16(float (&acc)[4], const Split (&a)[2][4], const Split (&b)[2][2]) {
  float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int x = 0; x < 2; ++x) product_small(d, a[x], b[x][0], b[x][1]);
#pragma unroll
  for (int x = 0; x < 2; ++x) product_big(d, a[x], b[x][0], b[x][1]);
#pragma unroll
  for (int e = 0; e < 4; ++e) acc[e] += d[e];
}
__device__ __forceinline__ void lds_split2(Split& x, Split& y, const float* p) {
  const float2 v = lds2(p);
  x = split(v.x);
  y = split(v.y);
}
// A from rows row, row + 8 of a row-major array (a pair of columns per lane)
__device__ __forceinline__ void rows_a(Split (&a)[4], const float* p, int ld8) {
  lds_split2(a[0], a[2], p);
  lds_split2(a[1], a[3], p + ld8);
}

// A block's rows on their way from global to shared memory: COLS columns of 32 tokens, all loads of a thread in
// flight at once and issued a block ahead of their use.  Rows past the end are zero.
template <typename T, int COLS, int THREADS>
struct BlockRegs {
  static constexpr int C4 = COLS / 4, kN = kC * C4 / THREADS, kStep = THREADS / C4;
  float4 x[kN];
  __device__ __forceinline__ void load(const T* p, long long stride, int n0, int n_end, int tid) {
    const T* src = p + (long long)(n0 + tid / C4) * stride + 4 * (tid % C4);
#pragma unroll
    for (int e = 0; e < kN; ++e)
      x[e] = (n0 + tid / C4 + kStep * e < n_end) ? load4<T>(src + e * kStep * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ __forceinline__ void store(float* dst, int ld, int tid) const {
#pragma unroll
    for (int e = 0; e < kN; ++e) *reinterpret_cast<float4*>(dst + (tid / C4 + kStep * e) * ld + 4 * (tid % C4)) = x[e];
  }
  // with phi; rows past the end stay zero
  __device__ __forceinline__ void store_phi(float* dst, int ld, int n0, int n_end, int tid) const {
#pragma unroll
    for (int e = 0; e < kN; ++e)
      *reinterpret_cast<float4*>(dst + (tid / C4 + kStep * e) * ld + 4 * (tid % C4)) =
          (n0 + tid / C4 + kStep * e < n_end) ? phi4(x[e]) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};

// ------------------------------------------------------------------------------------ windowed heads
// One CTA = 64 query rows of one head, 16 per warp, as two groups of four warps that take every other block of 32 keys and
// values; online softmax in registers, a row shared by four lanes.  Weights go from the scores' accumulators to the operand
// of the second product as they are (its contracted index in the accumulators' order).  The groups' sums meet at the end.
// (One group: 12 heads of 100 tokens, w = 512, 16.4 us against 12.3, 8 of 1000, d = 128, w = 64, 25.0 and 18.5.)
constexpr int kWinRows = 64, kWinGroup = 128, kWinThreads = 2 * kWinGroup;
template <int D>
constexpr int window_smem() { return (kWinRows * (D + 8) + 2 * kC * (D + 8) + 2 * kC * (D + 4)) * 4; }

// The output row of query i with FFMA products, by the four lanes that share it, over the keys it sees and no others.
// For rows in which a sum came out NaN: masked keys have weight 0 in the products above, which is nothing unless their value
// is infinite or NaN (0 x inf = NaN), and an infinite operand's rest is NaN.  And, kShort, for windows of fewer than kFewKeys keys, in
// which the errors of split operands do not average out (relative
// error of split operands at d = 64, FFMA's = 1: w = 2 1.21, 4 1.05, 8 0.91; us, 8 x 12 heads of 2048 tokens, w = 4 split 120, so 68).
constexpr int kFewKeys = 6;
template <typename T, int D, bool kShort>
__device__ __noinline__ void window_row(const T* q, const T* k, const T* v, T* o, int i, int j_begin, int j_end, float scale,
                                        long long stride, int part, unsigned int quad) {
  constexpr int kAhead = kShort ? kFewKeys - 2 : 1, kCols = kShort ? D / 16 : 1;
  auto score = [&](int j) {
    float s = 0.f;
#pragma unroll(kCols)
    for (int c = 0; c < D / 16; ++c)
      s = dot4(load4<T>(q + i * stride + 4 * (part + 4 * c)), load4<T>(k + j * stride + 4 * (part + 4 * c)), s);
    s += __shfl_xor_sync(quad, s, 1);
    s += __shfl_xor_sync(quad, s, 2);
    return s * scale;
  };
  float m = -INFINITY, l = 0.f;
#pragma unroll(kAhead)
  for (int j = j_begin; j < j_end; ++j) m = fmaxf(m, score(j));
  const float ref = m == -INFINITY ? 0.f : m;
  float4 acc[D / 16];
#pragma unroll
  for (int c = 0; c < D / 16; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll(kAhead)
  for (int j = j_begin; j < j_end; ++j) {
    const float p = expf(score(j) - ref);
    l += p;
#pragma unroll
    for (int c = 0; c < D / 16; ++c) axpy4(acc[c], p, load4<T>(v + j * stride + 4 * (part + 4 * c)));
  }
#pragma unroll
  for (int c = 0; c < D / 16; ++c)
    store4(o + i * stride + 4 * (part + 4 * c), make_float4(acc[c].x / l, acc[c].y / l, acc[c].z / l, acc[c].w / l));
}

template <typename T>
struct WindowArgs {
  const T *q, *k, *v;
  T* o;
  int N, w, fwd;  // fwd: keys after the query that it may see (0: the causal window; w - 1: the two-sided one)
  float scale;
  Strides st;
  int h_begin;
};

// The causal row that sees one key, over what the tile has stored: that key's value as it is, NaN unless the score is finite.  By a warp
// of the group that has no part in the tile's end, and behind the tile, since anything within it cost other tiles 1 to 4 %.
template <typename T, int D>
__device__ __noinline__ void window_first_row(const T* q, const T* k, const T* v, T* o, float scale) {
  const int lane = (int)threadIdx.x - kWinGroup;
  const bool part = lane >= 0 && 4 * lane < D;
  float4 value = make_float4(0.f, 0.f, 0.f, 0.f);
  if (lane >= 0 && lane < 32) {
    float s = 0.f;
    if (part) {
      value = load4<T>(v + 4 * lane);
      s = dot4(load4<T>(q + 4 * lane), load4<T>(k + 4 * lane), 0.f);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (!is_finite(s * scale)) value = make_float4(NAN, NAN, NAN, NAN);
  }
  __syncthreads();
  if (part) store4(o + 4 * lane, value);
}
template <typename T, int D>
__device__ __forceinline__ void window_short_tile(const WindowArgs<T>& p, int tile, int head, int b) {
  const long long base = (long long)b * p.st.b + (long long)(p.h_begin + head) * p.st.h;
  if (const int i = tile * kWinRows + (int)threadIdx.x / 4; i < p.N)
    window_row<T, D, true>(p.q + base, p.k + base, p.v + base, p.o + base, i, max(i - p.w + 1, 0), min(i + p.fwd, p.N - 1) + 1, p.scale,
                           p.st.n, threadIdx.x & 3, 0xfu << (threadIdx.x & 28));
}
template <typename T, int D>
__device__ __forceinline__ void window_tile(const WindowArgs<T>& p, int tile, int head, int b, float* sm) {
  constexpr int LD = D + 8, LDV = D + 4, NT = D / 8;
  const int group = threadIdx.x / kWinGroup, tid = threadIdx.x % kWinGroup, lane = tid & 31, warp = tid >> 5;
  float *Qs = sm, *Ks = Qs + kWinRows * LD + group * kC * (LD + LDV), *Vs = Ks + kC * LD;
  const int N = p.N;
  const long long base = (long long)b * p.st.b + (long long)(p.h_begin + head) * p.st.h;
  const int i0 = tile * kWinRows;
  const int g = lane >> 2, t = lane & 3;
  const int iw = i0 + 16 * warp;  // the warp's first row
  auto sync_group = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kWinGroup) : "memory"); };

  const int jlo = max(i0 - p.w + 1, 0) + kC * group, jhi = min(min(i0 + kWinRows, N) - 1 + p.fwd, N - 1);
  BlockRegs<T, D, kWinGroup> rk, rv;
  {
    BlockRegs<T, D, kWinGroup> rq;
    rq.load(p.q + base, p.st.n, i0 + kC * group, N, tid);
    rk.load(p.k + base, p.st.n, jlo, N, tid);
    rv.load(p.v + base, p.st.n, jlo, N, tid);
    rq.store(Qs + kC * group * LD, LD, tid);
  }
  __syncthreads();
  float acc[NT][4];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};  // rows iw + g, iw + g + 8

  for (int j0 = jlo; j0 <= jhi; j0 += 2 * kC) {
    rk.store(Ks, LD, tid);
    rv.store(Vs, LDV, tid);
    sync_group();
    if (j0 + 2 * kC <= jhi) {
      rk.load(p.k + base, p.st.n, j0 + 2 * kC, N, tid);
      rv.load(p.v + base, p.st.n, j0 + 2 * kC, N, tid);
    }
    // keys that a row of the warp can see
    if (iw < N && j0 <= iw + 15 + p.fwd && j0 + kC - 1 >= iw - p.w + 1) {
      float s[4][4];
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) s[n][e] = 0.f;
#pragma unroll(D == 64 ? NT / 2 : 1)  // (212 -> 208 us for 96 chains of 2048; d = 128 has no registers left: 470, and 492 unrolled)
      for (int kk = 0; kk < NT; kk += 2) {
        Split a[2][4];
        rows_a(a[0], Qs + (16 * warp + g) * LD + 8 * kk + 2 * t, 8 * LD);
        rows_a(a[1], Qs + (16 * warp + g) * LD + 8 * kk + 8 + 2 * t, 8 * LD);
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          Split k2[2][2];
          lds_split2(k2[0][0], k2[0][1], Ks + (8 * n + g) * LD + 8 * kk + 2 * t);
          lds_split2(k2[1][0], k2[1][1], Ks + (8 * n + g) * LD + 8 * kk + 8 + 2 * t);
          product16(s[n], a, k2);
        }
      }
      // some row does not see some key of the block
      const bool edge = j0 <= iw + 15 - p.w || j0 + kC - 1 > min(iw + p.fwd, N - 1);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int i = iw + g + 8 * r;
        if (edge) {
          const int lo = i - p.w - j0 - 2 * t, hi = min(i + p.fwd, N - 1) - j0 - 2 * t;  // lo < 8 n + e <= hi
#pragma unroll
          for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e)
              if (!(8 * n + e > lo && 8 * n + e <= hi)) s[n][2 * r + e] = -INFINITY;
        }
        float mx = -INFINITY;
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float& x = s[n][2 * r + e];
            x *= p.scale;
            mx = fmaxf(mx, x);
          }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m[r], mx);
        const float ref = (m_new == -INFINITY) ? 0.f : m_new;  // a row that has seen no key yet
        const float corr = expf(m[r] - ref);
        float sum = 0.f;
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float& x = s[n][2 * r + e];
            x = expf(x - ref);
            sum += x;
          }
        l[r] = l[r] * corr + sum;  // (of this lane's keys)
        m[r] = m_new;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          acc[n][2 * r] *= corr;
          acc[n][2 * r + 1] *= corr;
        }
      }
#pragma unroll
      for (int kk = 0; kk < 4; kk += 2) {
        const Split a[2][4] = {{split(s[kk][0]), split(s[kk][2]), split(s[kk][1]), split(s[kk][3])},
                               {split(s[kk + 1][0]), split(s[kk + 1][2]), split(s[kk + 1][1]), split(s[kk + 1][3])}};
        const float* vp = Vs + (8 * kk + 2 * t) * LDV + g;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const Split v2[2][2] = {{split(vp[8 * n]), split(vp[8 * n + LDV])},
                                  {split(vp[8 * n + 8 * LDV]), split(vp[8 * n + 9 * LDV])}};
          product16(acc[n], a, v2);
        }
      }
    }
    sync_group();
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
  }
  // the second group's sums, element by element of a lane, through the room of the keys and values
  static_assert((NT * 4 + 4) * kWinGroup <= 2 * kC * (LD + LDV), "room of the sums");
  float* part = Qs + kWinRows * LD + tid;
  __syncthreads();
  if (group == 1) {
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) part[(4 * n + e) * kWinGroup] = acc[n][e];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      part[(4 * NT + r) * kWinGroup] = m[r];
      part[(4 * NT + 2 + r) * kWinGroup] = l[r];
    }
  }
  __syncthreads();
  if (group == 1) return;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int i = iw + g + 8 * r;
    const float m1 = part[(4 * NT + r) * kWinGroup], mx = fmaxf(m[r], m1), ref = mx == -INFINITY ? 0.f : mx;
    const float f0 = expf(m[r] - ref), f1 = expf(m1 - ref);
    const float inv = 1.f / (l[r] * f0 + part[(4 * NT + 2 + r) * kWinGroup] * f1);
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 2; ++e)
        acc[n][2 * r + e] = acc[n][2 * r + e] * f0 + part[(4 * n + 2 * r + e) * kWinGroup] * f1;
    bool bad = false;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      bad |= is_nan(acc[n][2 * r]) || is_nan(acc[n][2 * r + 1]);
      if (i < N)
        store2(p.o + base + (long long)i * p.st.n + 8 * n + 2 * t, acc[n][2 * r] * inv, acc[n][2 * r + 1] * inv);
    }
    const unsigned int quad = 0xfu << (lane & 28);
    if ((__ballot_sync(0xffffffffu, bad) & quad) != 0u && i < N) {
      __syncwarp(quad);  // (the row's stores above come first)
      window_row<T, D, false>(p.q + base, p.k + base, p.v + base, p.o + base, i, max(i - p.w + 1, 0), min(i + p.fwd, N - 1) + 1,
                              p.scale, p.st.n, t, quad);
    }
    __syncwarp();
  }
}

template <typename T, int D>
__device__ __forceinline__ void any_window_tile(const WindowArgs<T>& p, int tile, int head, int b, float* sm) {
  if (p.w < kFewKeys) {
    window_short_tile<T, D>(p, tile, head, b);
    return;
  }
  window_tile<T, D>(p, tile, head, b, sm);
  if (tile == 0 && p.fwd == 0) {
    const long long base = (long long)b * p.st.b + (long long)(p.h_begin + head) * p.st.h;
    window_first_row<T, D>(p.q + base, p.k + base, p.v + base, p.o + base, p.scale);
  }
}

template <typename T, int D>
__global__ void __launch_bounds__(kWinThreads, D == 64 ? 2 : 1)
window_tiled_kernel(const WindowArgs<T> p, Place place) {
  extern __shared__ __align__(16) float sm[];
  begin(place);
  any_window_tile<T, D>(p, blockIdx.x, blockIdx.y, blockIdx.z, sm);
  grid_dep_launch();
  if (blockIdx.x + blockIdx.y + blockIdx.z == 0) grid_dep_wait();
}

// ------------------------------------------------------------------------------------ causal linear heads
// Algorithm 1 regrouped in blocks of 32 tokens (exactly equal by associativity): with S, z the sums before a block,
//   P = phi(Q) phi(K)^T masked to j <= i,   O = (P V + phi(Q) S) / (rowsum(P) + phi(Q) z),
//   S += phi(K)^T V,   z += colsum(phi(K)).
// A CTA owns 64 value columns of a chain, a warp 16 of them and half of the features.  S lives in the warps' registers as the
// accumulators of S^T += V^T phi(K) (a lane: columns g, g + 8, features 8 n + 2 t, + 1 of its half), which are at the same
// time its operand in phi(Q) S; the two halves of O meet in shared memory.  (Four warps with all features each need 168
// registers a lane, three CTAs per SM, and take 5.2 us for a block when alone on one, eight 3.6.)
//
// With few chains a chain is cut into G segments, so that every SM has work.  Up to kMaxCluster of them are a cluster of
// CTAs in one launch (kCluster): each sums its own segment; every CTA then turns its share of the elements, read from all
// CTAs' shared memory at once, into running sums and puts those back; then they walk.  Where a chain has two CTAs per segment
// (D = 128) and brings a state, both are in the cluster: both read the caller's z, and one of them overwrites it, which has
// to wait until the other has started.  Longer chains in smaller numbers take three launches, with segments of a little
// more than D tokens:
//   contribution   the sums of every segment but the last, each alone
//   prefix         running sums over the segments of a chain
//   walk           the segments' outputs, each from its own starting state
// The states wait in the rows of the OUTPUT tensor that their own segment will later overwrite (row a of S in the
// row of token a of the segment, z in the next row or two, one per 64 columns): no workspace, and a CTA of the walk
// reads only rows and columns that itself will write.
constexpr int kMaxCluster = 8;
template <int D> struct LinT {
  static constexpr int LD = D + 8;
  static constexpr int ZROWS = D / 64;  // rows z takes behind S
  // shortest segment: D + ZROWS rows, also when the last segment's last block is a single token
  static constexpr int kMinSeg = D + 32 * ZROWS;
  static constexpr int kSmem = (2 * kC * LD + kC * kLdV + kC * kLdP + D * kW + kC * kW + D + 2 * kC) * 4;
  static constexpr int kSmemSum = (kC * LD + kC * kLdV) * 4;
};
struct Segs {  // tokens [begin(g), begin(g + 1)) of segment g, whole blocks but for the last
  int N, G, base, rem;  // blocks per segment: base, one more for the first rem
  __host__ __device__ int begin(int g) const { return g >= G ? N : kC * (g * base + (g < rem ? g : rem)); }
};

// The lane's share of S: S[n][0 | 1] column g, S[n][2 | 3] column g + 8 of the warp's 16; features 8 n + 2 t, + 1 of its half.
template <int D> using State = float[D / 16][4];
struct Lane {
  int g, t, c0, half;  // c0: the warp's first column
};
__device__ __forceinline__ Lane lane_of() {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  return {lane >> 2, lane & 3, 16 * (warp & 3), warp >> 2};
}
// f(feature, column of the CTA's 64, element)
template <int D, typename F>
__device__ __forceinline__ void for_state(State<D>& S, F f) {
  const Lane l = lane_of();
#pragma unroll
  for (int n = 0; n < D / 16; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) f(l.half * (D / 2) + 8 * n + 2 * l.t + (e & 1), l.c0 + l.g + 8 * (e >> 1), S[n][e]);
}
// kSane: values that are not finite count as 0
template <bool kSane>
__device__ __forceinline__ Split split_value(float v) { return split(kSane && !is_finite(v) ? 0.f : v); }

// S += phi(K)^T V
template <int D, bool kSane>
__device__ __forceinline__ void add_outer(const float* Ks, const float* Vs, State<D>& S) {
  constexpr int LD = LinT<D>::LD;
  const Lane l = lane_of();
#pragma unroll(D == 64 ? 4 : 2)
  for (int kk = 0; kk < kC / 8; ++kk) {
    const float *v = Vs + (8 * kk + l.t) * kLdV + l.c0 + l.g, *k = Ks + (8 * kk + l.t) * LD + l.half * (D / 2) + l.g;
    const Split a[4] = {split_value<kSane>(v[0]), split_value<kSane>(v[8]), split_value<kSane>(v[4 * kLdV]),
                        split_value<kSane>(v[4 * kLdV + 8])};
#pragma unroll
    for (int n = 0; n < D / 16; ++n) product8(S[n], a, split(k[8 * n]), split(k[8 * n + 4 * LD]));
  }
}
// This half's part of phi(Q) S + P V (its features; half of the keys): rows 16 m + g | + 8, columns 8 n + 2 t | + 1 of the warp's
template <int D, bool kSane>
__device__ __forceinline__ void readout(const float* Qs, const float* Vs, const float* Ps, const State<D>& S, float (&acc)[2][2][4]) {
  constexpr int LD = LinT<D>::LD;
  const Lane l = lane_of();
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.f;
#pragma unroll
  for (int kk = 0; kk < D / 16; ++kk) {
    const Split b[4] = {split(S[kk][0]), split(S[kk][1]), split(S[kk][2]), split(S[kk][3])};
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      Split a[4];
      rows_a(a, Qs + (16 * m + l.g) * LD + l.half * (D / 2) + 8 * kk + 2 * l.t, 8 * LD);
      product8(acc[m][0], a, b[0], b[1]);
      product8(acc[m][1], a, b[2], b[3]);
    }
  }
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int key = 8 * (2 * l.half + x) + l.t;
    const float* v = Vs + key * kLdV + l.c0 + l.g;
    const Split b[4] = {split_value<kSane>(v[0]), split_value<kSane>(v[4 * kLdV]), split_value<kSane>(v[8]),
                        split_value<kSane>(v[4 * kLdV + 8])};
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      if (m == 0 && l.half == 1) continue;  // masked
      const float* p = Ps + (16 * m + l.g) * kLdP + key;
      const Split a[4] = {split(p[0]), split(p[8 * kLdP]), split(p[4]), split(p[8 * kLdP + 4])};
      product8(acc[m][0], a, b[0], b[1]);
      product8(acc[m][1], a, b[2], b[3]);
    }
  }
}
// The six tiles of P that are not all masked, 16 rows x 8 keys each, by six warps ...
template <int D>
__device__ __forceinline__ void score_block(const float* Qs, const float* Ks, float* Ps) {
  constexpr int LD = LinT<D>::LD;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, warp = threadIdx.x >> 5;
  if (warp < 6) {
    const int m = warp < 2 ? 0 : 1, n = warp < 2 ? warp : warp - 2;
    float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};  // (two sums: half the chain)
#pragma unroll(D == 64 ? 8 : 4)
    for (int kk = 0; kk < D / 8; ++kk) {
      Split a[4], b0, b1;
      lds_split2(b0, b1, Ks + (8 * n + g) * LD + 8 * kk + 2 * t);
      rows_a(a, Qs + (16 * m + g) * LD + 8 * kk + 2 * t, 8 * LD);
      product8(s[kk & 1], a, b0, b1);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int row = 16 * m + g + 8 * r, key = 8 * n + 2 * t;
      store2(Ps + row * kLdP + key, key <= row ? s[0][2 * r] + s[1][2 * r] : 0.f,
             key + 1 <= row ? s[0][2 * r + 1] + s[1][2 * r + 1] : 0.f);
    }
  }
}
// ... and phi(Q) z by the other two.
template <int D>
__device__ __forceinline__ void dot_z(const float* Qs, const float* zs, float* qz_s) {
  constexpr int LD = LinT<D>::LD;
  if (threadIdx.x >= 192) {
    const int row = (threadIdx.x - 192) >> 1, part = threadIdx.x & 1;
    float d[2] = {0.f, 0.f};
#pragma unroll 4
    for (int a = 0; a < D; a += 8)
      d[(a >> 3) & 1] = dot4(lds4(Qs + row * LD + a + 4 * part), lds4(zs + a + 4 * part), d[(a >> 3) & 1]);
    float q = d[0] + d[1];
    q += __shfl_xor_sync(0xffffffffu, q, 1);
    if (part == 0) qz_s[row] = q;
  }
}
template <int D>
__device__ __forceinline__ float column_sum(const float* col) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
  for (int j = 0; j < kC; ++j) s[j & 3] += (col[j * LinT<D>::LD]);
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// Below 2^-112 tf32 has fewer than 11 bits for the rest of an operand.  Features are that small under inputs of -77.6, their
// products sooner, and what comes out is a quotient, in which the size of all features cancels: of rows whose denominators, and
// segments whose feature sums, are all under kLow the products are FFMA's.  (Above it such operands are lost beside the others.  Values
// below 2^-112 keep an error of 2^-136.)  Error beside FFMA's with keys around -84, d = 64: 11 times without this, equal with it.  Such
// blocks take five times as long; the question costs the others 0.5 to 1.5 % (8 x 12 heads of 2048 tokens 170 -> 172 us).
constexpr float kLow = 0x1p-84f;

// S += phi(K)^T V with FFMA products
template <int D>
__device__ __forceinline__ void add_outer_ffma(const float* Ks, const float* Vs, State<D>& S) {
  const Lane l = lane_of();
  const float *k = Ks + l.half * (D / 2) + 2 * l.t, *v = Vs + l.c0 + l.g;
#pragma unroll 1
  for (int j = 0; j < kC; ++j, k += LinT<D>::LD, v += kLdV) {
    const float v0 = v[0], v1 = v[8];
#pragma unroll
    for (int n = 0; n < D / 16; ++n) {
      const float2 x = lds2(k + 8 * n);
      S[n][0] = fmaf(x.x, v0, S[n][0]);
      S[n][1] = fmaf(x.y, v0, S[n][1]);
      S[n][2] = fmaf(x.x, v1, S[n][2]);
      S[n][3] = fmaf(x.y, v1, S[n][3]);
    }
  }
}

// Adds tokens [n_begin, n_end) to S = 0 and z = 0 (thread tid < D: feature tid).
template <typename T, int D>
__device__ __forceinline__ void sum_segment(const T* k, const T* v, long long stride, int n_begin, int n_end, float* Ks,
                                            float* Vs, int tid, State<D>& S, float& z) {
  BlockRegs<T, D, kLinThreads> rk;
  BlockRegs<T, kW, kLinThreads> rv;
  rk.load(k, stride, n_begin, n_end, tid);
  rv.load(v, stride, n_begin, n_end, tid);
  int big = 0;  // some feature's sum is not under kLow
  for (int n0 = n_begin; n0 < n_end; n0 += kC) {
    rk.store_phi(Ks, LinT<D>::LD, n0, n_end, tid);
    rv.store(Vs, kLdV, tid);
    __syncthreads();
    rk.load(k, stride, n0 + kC, n_end, tid);
    rv.load(v, stride, n0 + kC, n_end, tid);
    add_outer<D, false>(Ks, Vs, S);
    if (tid < D) z += column_sum<D>(Ks + tid);
    big = __syncthreads_or(tid < D && !(z < kLow));
  }
  if (!big && __syncthreads_or(tid < D && z > 0.f)) {
    for_state<D>(S, [](int, int, float& x) { x = 0.f; });
    for (int n0 = n_begin; n0 < n_end; n0 += kC) {
      rk.load(k, stride, n0, n_end, tid);
      rv.load(v, stride, n0, n_end, tid);
      rk.store_phi(Ks, LinT<D>::LD, n0, n_end, tid);
      rv.store(Vs, kLdV, tid);
      __syncthreads();
      add_outer_ffma<D>(Ks, Vs, S);
      __syncthreads();
    }
  }
  // (an infinite operand's rest is NaN)
  bool bad = false;
  for_state<D>(S, [&](int, int, float& x) { bad |= is_nan(x); });
  if (bad) {
    const Lane l = lane_of();
    for (int n = 0; n < D / 16; ++n)
      for (int e = 0; e < 4; ++e) {
        const int a = l.half * (D / 2) + 8 * n + 2 * l.t + (e & 1), c = l.c0 + l.g + 8 * (e >> 1);
        float x = 0.f;
        for (int j = n_begin; j < n_end; ++j) x = fmaf(phi_elu1(to_f32(k[j * stride + a])), to_f32(v[j * stride + c]), x);
#pragma unroll
        for (int n1 = 0; n1 < D / 16; ++n1)
#pragma unroll
          for (int e1 = 0; e1 < 4; ++e1)
            if (n1 == n && e1 == e && is_nan(S[n1][e1])) S[n1][e1] = x;
      }
  }
}

template <int D>
__global__ void __launch_bounds__(kLinThreads, 2)
linear_contribution_kernel(const float* __restrict__ k, const float* __restrict__ v, float* __restrict__ o, Segs sg,
                           Strides st, int h_begin, Place place) {
  extern __shared__ __align__(16) float sm[];
  begin(place);
  float *Ks = sm, *Vs = Ks + kC * LinT<D>::LD;
  const int g = blockIdx.x / (D / kW), col0 = (blockIdx.x % (D / kW)) * kW;
  const long long base = (long long)blockIdx.z * st.b + (long long)(h_begin + blockIdx.y) * st.h;
  const int tid = threadIdx.x;
  State<D> S;
  for_state<D>(S, [](int, int, float& x) { x = 0.f; });
  float z = 0.f;
  const int n_end = sg.begin(g + 1);
  sum_segment<float, D>(k + base, v + base + col0, st.n, sg.begin(g), n_end, Ks, Vs, tid, S, z);
  float* slot = o + base + (long long)n_end * st.n + col0;  // the state before segment g + 1, once summed
  for_state<D>(S, [&](int a, int c, float& x) { slot[(long long)a * st.n + c] = x; });
  if (tid < D) slot[(long long)(D + tid / kW) * st.n + tid % kW] = z;
  if (blockIdx.x + blockIdx.y + blockIdx.z == 0) grid_dep_wait();
}

// The slots of segments 1 .. G - 1 hold contributions; turned into running sums from the caller's initial state
// (which also goes to segment 0's slot: the walk's last segment may overwrite the caller's copy).
template <int D>
__global__ void linear_prefix_kernel(float* __restrict__ o, Segs sg, Strides st, int h_begin, int h_count,
                                     const float* __restrict__ S_in, const float* __restrict__ z_in) {
  constexpr int D4 = D / 4, kRows = D + LinT<D>::ZROWS, kAhead = 8;
  grid_dep_wait();
  grid_dep_launch();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= kRows * D4) return;
  const int row = idx / D4, c = 4 * (idx % D4);
  float* slot = o + (long long)blockIdx.z * st.b + (long long)(h_begin + blockIdx.y) * st.h + (long long)row * st.n + c;
  const long long sidx = (long long)blockIdx.z * h_count + blockIdx.y;
  float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
  if (S_in != nullptr) {
    run = row < D ? lds4(S_in + (sidx * D + row) * D + c) : lds4(z_in + sidx * D + (row - D) * kW + c % kW);
    store4(slot, run);
  }
  for (int g0 = 1; g0 < sg.G; g0 += kAhead) {
    float4 x[kAhead];
#pragma unroll
    for (int e = 0; e < kAhead; ++e)
      if (g0 + e < sg.G) x[e] = load4<float>(slot + (long long)sg.begin(g0 + e) * st.n);
#pragma unroll
    for (int e = 0; e < kAhead; ++e)
      if (g0 + e < sg.G) {
        run.x += x[e].x;
        run.y += x[e].y;
        run.z += x[e].z;
        run.w += x[e].w;
        store4(slot + (long long)sg.begin(g0 + e) * st.n, run);
      }
  }
}

// 1 / (row sums of P + phi(Q) z), eight threads per row.  Whether the thread has found one under kLow (past the end they are 0)
__device__ __forceinline__ bool invert_denominators(const float* Ps, const float* qz_s, float* inv_s) {
  const int row = threadIdx.x >> 3, part8 = threadIdx.x & 7;
  float den = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) den += Ps[row * kLdP + part8 + 8 * e];
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
  den += qz_s[row];
  if (part8 == 0) inv_s[row] = 1.f / den;
  return den > 0.f && den < kLow;
}

// A block with a row whose denominator is under kLow: all of it with FFMA products.
template <int D>
__device__ __noinline__ void low_block(const float* Qs, const float* Ks, const float* Vs, float* Ps, float* Ss, const float* qz_s,
                                       float* inv_s, State<D>& S, float (&acc)[2][2][4], bool more) {
  constexpr int LD = LinT<D>::LD;
  const Lane l = lane_of();
  for_state<D>(S, [&](int a, int c, float& x) { Ss[a * kW + c] = x; });
  for (int e = 0; e < 4; ++e) {
    const int row = threadIdx.x >> 3, key = (threadIdx.x & 7) + 8 * e;
    float x = 0.f;
    if (key <= row)
      for (int a = 0; a < D; a += 4) x = dot4(lds4(Qs + row * LD + a), lds4(Ks + key * LD + a), x);
    Ps[row * kLdP + key] = x;
  }
  __syncthreads();
  (void)invert_denominators(Ps, qz_s, inv_s);
  if (l.half == 0)
    for (int i = 0; i < 16; ++i) {
      const int m = i >> 3, n = (i >> 2) & 1, e = i & 3;
      const int row = 16 * m + l.g + 8 * (e >> 1), c = l.c0 + 8 * n + 2 * l.t + (e & 1);
      float x = 0.f;
      for (int a = 0; a < D; ++a) x = fmaf(Qs[row * LD + a], Ss[a * kW + c], x);
      for (int j = 0; j <= row; ++j) x = fmaf(Ps[row * kLdP + j], Vs[j * kLdV + c], x);
      acc[m][n][e] = x;
    }
  if (more) add_outer_ffma<D>(Ks, Vs, S);
  __syncthreads();
}

// A block in which a sum came out NaN: a masked weight is 0, which is nothing unless the value is infinite or NaN (0 x inf
// = NaN), and an infinite operand's rest is NaN.  The same products with such values left out (so that what does not see them
// keeps its bits), and the elements that see one of them, or are NaN even so, once more by plain multiply-adds.
template <int D>
__device__ __noinline__ void mend_block(const float* Qs, const float* Ks, const float* Vs, const float* Ps, float* Ss, float* Os,
                                        State<D>& S, float (&acc)[2][2][4], bool more) {
  constexpr int LD = LinT<D>::LD;
  const Lane l = lane_of();
  for_state<D>(S, [&](int a, int c, float& x) { Ss[a * kW + c] = x; });
  readout<D, true>(Qs, Vs, Ps, S, acc);
  if (l.half == 1)
    for (int i = 0; i < 16; ++i) Os[i * 128 + (threadIdx.x & 127)] = acc[i >> 3][(i >> 2) & 1][i & 3];
  __syncthreads();
  if (l.half == 0)
    for (int i = 0; i < 16; ++i) {
      const int m = i >> 3, n = (i >> 2) & 1, e = i & 3;
      acc[m][n][e] += Os[i * 128 + threadIdx.x];
      const int row = 16 * m + l.g + 8 * (e >> 1), c = l.c0 + 8 * n + 2 * l.t + (e & 1);
      bool bad = is_nan(acc[m][n][e]);
      for (int j = 0; j <= row; ++j) bad |= !is_finite(Vs[j * kLdV + c]);
      if (!bad) continue;
      float x = 0.f;
      for (int a = 0; a < D; ++a) x = fmaf(Qs[row * LD + a], Ss[a * kW + c], x);
      for (int j = 0; j <= row; ++j) {
        float p = Ps[row * kLdP + j];
        if (is_nan(p)) {
          p = 0.f;
          for (int a = 0; a < D; ++a) p = fmaf(Qs[row * LD + a], Ks[j * LD + a], p);
        }
        x = fmaf(p, Vs[j * kLdV + c], x);
      }
      acc[m][n][e] = x;
    }
  if (!more) return;
  add_outer<D, true>(Ks, Vs, S);
  for (int n = 0; n < D / 16; ++n)
    for (int e = 0; e < 4; ++e) {
      const int a = l.half * (D / 2) + 8 * n + 2 * l.t + (e & 1), c = l.c0 + l.g + 8 * (e >> 1);
      bool bad = is_nan(S[n][e]);
      for (int j = 0; j < kC; ++j) bad |= !is_finite(Vs[j * kLdV + c]);
      if (!bad) continue;
      float x = Ss[a * kW + c];
      for (int j = 0; j < kC; ++j) x = fmaf(Ks[j * LD + a], Vs[j * kLdV + c], x);
      S[n][e] = x;
    }
}

// Without cuts (G == 1) the state before token 0 comes from S_io; with cuts from the segment's slot (segment 0 has
// one only when there is an initial state), or, kCluster, from S_io and the cluster's CTAs before this one.  A chain that
// brings a state and has several slices is one cluster (G x D / kW CTAs), also when it is not cut.
template <typename T>
struct WalkArgs {
  const T *q, *k, *v;
  T* o;
  Segs sg;
  Strides st;
  int h_begin, h_count;
  float *S_io, *z_io;
  int zero_init;
};

template <typename T, int D, bool kCluster>
__device__ __forceinline__ void linear_walk(const WalkArgs<T>& p, int part, int head, int b, float* sm) {
  constexpr int LD = LinT<D>::LD;
  float *Qs = sm, *Ks = Qs + kC * LD, *Vs = Ks + kC * LD, *Ps = Vs + kC * kLdV, *Ss = Ps + kC * kLdP,
        *Os = Ss + D * kW, *zs = Os + kC * kW, *inv_s = zs + D, *qz_s = inv_s + kC;
  const Segs& sg = p.sg;
  // (a cluster's CTAs are neighbours in x: the segments of one slice, then those of the next)
  const int g = kCluster ? part % sg.G : part / (D / kW);
  const int col0 = (kCluster ? part / sg.G : part % (D / kW)) * kW;
  const long long base = (long long)b * p.st.b + (long long)(p.h_begin + head) * p.st.h;
  const long long sidx = (long long)b * p.h_count + head;
  const int tid = threadIdx.x, lane = tid & 31;
  const int n_begin = sg.begin(g), n_end = sg.begin(g + 1);
  const T *q = p.q + base, *k = p.k + base, *v = p.v + base + col0;
  T* o = p.o + base + col0;
  float* S_io = p.S_io;

  BlockRegs<T, D, kLinThreads> rq, rk;
  BlockRegs<T, kW, kLinThreads> rv;
  auto load_first = [&]() {
    rq.load(q, p.st.n, n_begin, n_end, tid);
    rk.load(k, p.st.n, n_begin, n_end, tid);
    rv.load(v, p.st.n, n_begin, n_end, tid);
  };
  // phi(Q), phi(K) and V of the block at n0 into shared memory, the next block's on their way
  auto store_block = [&](int n0) {
    rq.store_phi(Qs, LD, n0, n_end, tid);
    rk.store_phi(Ks, LD, n0, n_end, tid);
    rv.store(Vs, kLdV, tid);
    __syncthreads();  // (also: every thread has read its state out of the rows this CTA writes)
    rq.load(q, p.st.n, n0 + kC, n_end, tid);
    rk.load(k, p.st.n, n0 + kC, n_end, tid);
    rv.load(v, p.st.n, n0 + kC, n_end, tid);
  };
  Ps[(tid >> 4) * kLdP + 16 + (tid & 15)] = 0.f;  // (masked, and nobody computes them)
  State<D> S;
  if constexpr (kCluster) {
    auto cluster = cooperative_groups::this_cluster();
    for_state<D>(S, [](int, int, float& x) { x = 0.f; });
    float z = 0.f;
    float4* frag = reinterpret_cast<float4*>(Ss) + tid;  // S of this lane, element n at frag[n * kLinThreads]
    if (g < sg.G - 1) {  // nobody needs the last segment's sum
      sum_segment<T, D>(k, v, p.st.n, n_begin, n_end, Ks, Vs, tid, S, z);
#pragma unroll
      for (int n = 0; n < D / 16; ++n) frag[n * kLinThreads] = make_float4(S[n][0], S[n][1], S[n][2], S[n][3]);
      if (tid < D) zs[tid] = z;
    }
    load_first();
    const bool from_caller = S_io != nullptr && !p.zero_init;
    for_state<D>(S, [&](int a, int c, float& x) { x = from_caller ? S_io[(sidx * D + a) * D + col0 + c] : 0.f; });
    z = (from_caller && tid < D) ? p.z_io[sidx * D + tid] : 0.f;
    // the first block's scores while the sums of the others arrive (a layer of 8 x 12 chains of 300 tokens 35.5 -> 34.1 us,
    // one of 256 9.4 -> 9.0)
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    store_block(n_begin);
    score_block<D>(Qs, Ks, Ps);
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    // running sums: of S[n] by segment n mod G, of z by segment 0, for all segments, read and put back in place
    const int rank0 = (int)cluster.block_rank() - g;  // first segment of this slice
    for (int n = g; n < D / 16; n += sg.G) {
      float4 x[kMaxCluster - 1];
#pragma unroll
      for (int gg = 0; gg < kMaxCluster - 1; ++gg)
        if (gg < sg.G - 1) x[gg] = *cluster.map_shared_rank(frag + n * kLinThreads, rank0 + gg);
      float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int gg = 0; gg < kMaxCluster - 1; ++gg)
        if (gg < sg.G - 1) {
          axpy4(run, 1.f, x[gg]);
          *cluster.map_shared_rank(frag + n * kLinThreads, rank0 + gg + 1) = run;
        }
    }
    if (g == 0 && tid < D) {
      float x[kMaxCluster - 1], run = 0.f;
#pragma unroll
      for (int gg = 0; gg < kMaxCluster - 1; ++gg)
        if (gg < sg.G - 1) x[gg] = *cluster.map_shared_rank(zs + tid, rank0 + gg);
#pragma unroll
      for (int gg = 0; gg < kMaxCluster - 1; ++gg)
        if (gg < sg.G - 1) {
          run += x[gg];
          *cluster.map_shared_rank(zs + tid, rank0 + gg + 1) = run;
        }
    }
    cluster.sync();  // (also: everybody has read the caller's state, which the last CTAs will overwrite)
    if (g > 0) {
#pragma unroll
      for (int n = 0; n < D / 16; ++n) {
        const float4 x = frag[n * kLinThreads];
        S[n][0] += x.x;
        S[n][1] += x.y;
        S[n][2] += x.z;
        S[n][3] += x.w;
      }
      if (tid < D) z += zs[tid];
    }
    if (tid < D) zs[tid] = z;
    __syncthreads();
  } else {
    load_first();
    const float* Sp = nullptr;  // row a of the starting state at Sp + a * stride
    long long stride = D;
    const float* zp = nullptr;
    if (sg.G > 1 && (g > 0 || (S_io != nullptr && !p.zero_init))) {
      if constexpr (sizeof(T) == 4) {
        Sp = reinterpret_cast<const float*>(o) + (long long)n_begin * p.st.n;
        stride = p.st.n;
      }
    } else if (g == 0 && S_io != nullptr && !p.zero_init) {
      Sp = S_io + sidx * D * D + col0;
      zp = p.z_io + sidx * D;
    }
    for_state<D>(S, [&](int a, int c, float& x) { x = Sp != nullptr ? Sp[a * stride + c] : 0.f; });
    if (tid < D)
      zs[tid] = Sp == nullptr ? 0.f : zp != nullptr ? zp[tid] : Sp[(long long)(D + tid / kW) * stride + tid % kW];
  }
  // Whether the chain starts from nothing, so that its first rows see few keys: kept in a column of P that nobody uses.
  if (g == 0) {
    bool any = false;
    if (S_io != nullptr && !p.zero_init) {
      any = tid < D && zs[tid] != 0.f;
      for_state<D>(S, [&](int, int, float& x) { any |= x != 0.f; });
      any = __syncthreads_or(any);
    }
    if (tid == 0) Ps[kC] = any ? 0.f : 1.f;
  }
  for (int n0 = n_begin; n0 < n_end; n0 += kC) {
    if (!kCluster || n0 > n_begin) {
      store_block(n0);
      score_block<D>(Qs, Ks, Ps);
    }
    dot_z<D>(Qs, zs, qz_s);
    __syncthreads();
    const bool low = invert_denominators(Ps, qz_s, inv_s);
    float acc[2][2][4];
    readout<D, false>(Qs, Vs, Ps, S, acc);
    bool bad = low;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) bad |= is_nan(acc[m][n][e]);
    if (tid >= 128) {
#pragma unroll
      for (int i = 0; i < 16; ++i) Os[i * 128 + tid - 128] = acc[i >> 3][(i >> 2) & 1][i & 3];
    }
    const bool more = n0 + kC < n_end || (g == sg.G - 1 && S_io != nullptr);  // somebody wants the state after this block
    if (__syncthreads_or(bad)) {
      State<D> Sx;
      float ax[2][2][4];
#pragma unroll
      for (int n = 0; n < D / 16; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) Sx[n][e] = S[n][e];
      if (__syncthreads_or(low)) low_block<D>(Qs, Ks, Vs, Ps, Ss, qz_s, inv_s, Sx, ax, more);
      else mend_block<D>(Qs, Ks, Vs, Ps, Ss, Os, Sx, ax, more);
#pragma unroll
      for (int n = 0; n < D / 16; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) S[n][e] = Sx[n][e];
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[i >> 3][(i >> 2) & 1][i & 3] = ax[i >> 3][(i >> 2) & 1][i & 3];
    } else {
      if (tid < 128) {
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i >> 3][(i >> 2) & 1][i & 3] += Os[i * 128 + tid];
      }
      if (more) add_outer<D, false>(Ks, Vs, S);
    }
    if (tid < 128) {
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int row = 16 * m + (lane >> 2) + 8 * r;
          if (n0 + row >= n_end) continue;
          const float inv = inv_s[row];
#pragma unroll
          for (int n = 0; n < 2; ++n)
            store2(o + (long long)(n0 + row) * p.st.n + 16 * (tid >> 5) + 8 * n + 2 * (lane & 3), acc[m][n][2 * r] * inv,
                   acc[m][n][2 * r + 1] * inv);
        }
    }
    // Rows that see fewer than kFewKeys keys, with FFMA products, over what was just stored (largest error of chains of 64 to 2048
    // tokens, d = 64, FFMA's = 1: 1.39 without this, 0.73 with it; 0.2 us of a chain).
    if (n0 == 0 && Ps[kC] != 0.f) {
      __syncthreads();
      if (const int row = tid >> 4, c = 4 * (tid & 15); row < kFewKeys - 1 && row < n_end) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int j = 0; j <= row; ++j) axpy4(x, Ps[row * kLdP + j], lds4(Vs + j * kLdV + c));
        const float inv = inv_s[row];
        store4(o + (long long)row * p.st.n + c, make_float4(x.x * inv, x.y * inv, x.z * inv, x.w * inv));
      }
    }
    if (more && tid >= kLinThreads - D) zs[tid - (kLinThreads - D)] += column_sum<D>(Ks + tid - (kLinThreads - D));
    __syncthreads();
  }
  if (g == sg.G - 1 && S_io != nullptr) {
    for_state<D>(S, [&](int a, int c, float& x) { S_io[(sidx * D + a) * D + col0 + c] = x; });
    if (col0 == 0 && tid < D) p.z_io[sidx * D + tid] = zs[tid];
  }
}

template <typename T, int D, bool kCluster>
__global__ void __launch_bounds__(kLinThreads, 2)
linear_walk_kernel(const WalkArgs<T> p, int after, Place place) {
  extern __shared__ __align__(16) float sm[];
  if (after) grid_dep_wait();  // the segments' starting states
  begin(place);
  linear_walk<T, D, kCluster>(p, blockIdx.x, blockIdx.y, blockIdx.z, sm);
  grid_dep_launch();
  if (blockIdx.x + blockIdx.y + blockIdx.z == 0) grid_dep_wait();
}

template <typename T, int D>
cudaError_t window_launch(const WindowArgs<T>& p, int B, int h_count, cudaStream_t stream, Place place) {
  int dev = 0, sms = 0;
  cudaError_t e = device_info(&dev, &sms);
  if (e != cudaSuccess) return e;
  auto kern = window_tiled_kernel<T, D>;
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), dev, window_smem<D>())) != cudaSuccess) return e;
  return launch_link(kern, dim3((p.N + kWinRows - 1) / kWinRows, h_count, B), dim3(kWinThreads),
                     window_smem<D>(), stream, p, place);
}

// Shared memory that a launch of few CTAs asks for so that no SM takes more than its share of them (the scheduler packs the
// CTAs of a cluster onto as few SMs as hold them: 20 chains of 1588 tokens, clusters of 8, 64 -> 53 us).
constexpr int kSmemPerSM = 228 * 1024, kSmemReserved = 1024;
int spread_smem(int need, long long ctas, int sms) {
  const long long per_sm = (ctas + sms - 1) / sms;
  const long long least = kSmemPerSM / (per_sm + 1) - kSmemReserved + 256;  // one CTA more does not fit
  return least > need ? (int)least : need;
}

// Clusters of that many CTAs of the walk that the device holds at a time (asked once for each number of CTAs that the shared
// memory asked for leaves an SM).
template <typename T, int D>
int resident_clusters(int size, int smem, int dev) {
  constexpr int kMost = 4;  // (of the CTAs with the least shared memory)
  static_assert(kSmemPerSM / (LinT<D>::kSmem + kSmemReserved) <= kMost, "a slot for each number");
  static std::atomic<int> known[64][kMaxCluster + 1][kMost + 1];
  if (dev < 0 || dev >= 64) return 0;
  std::atomic<int>& slot = known[dev][size][kSmemPerSM / (smem + kSmemReserved)];
  int n = slot.load(std::memory_order_relaxed);
  if (n == 0) {
    auto kern = linear_walk_kernel<T, D, true>;
    if (ensure_dynamic_smem(reinterpret_cast<const void*>(kern), dev, smem) != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(kLinThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = size;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
    if (e != cudaSuccess) {
      (void)cudaGetLastError();
      return 0;
    }
    slot.store(n > 0 ? n : -1, std::memory_order_relaxed);
  }
  return n > 0 ? n : 0;
}

// Segments per chain: as a cluster, or (three > 1) in three launches.
struct LinearPlan {
  int cluster, slices, three;
  long long ctas;  // of one segment per chain
};
template <typename T, int D>
LinearPlan linear_plan(int B, int N, int h_count, bool brings_state, int dev, int sms) {
  using C = LinT<D>;
  // How many segments, and whether as one cluster per chain or in three launches: the least time of the CTA that takes longest, in
  // blocks of a CTA that has an SM to itself (3.6 us at d = 64).  Both sweeps over a block cost 1.37 of the walk alone; two
  // CTAs on an SM take 1.6 times as long; the exchange in a cluster costs about one block, the two other launches 3.5.
  // Measured (us, layers with w = 64 or 128 and 12 heads, clusters of c | three launches with G): 80 chains of 2048 tokens 234 (c =
  // 1) 246 (2) 177 (3) 196 (4) | 180 (4) 187 (12); 40 of 2048 111 (3) 103 (6) 119 (8) | 107 (5); 20 of 2048 60 (6) 66 (8) | 61 (12);
  // 10 of 2048 45 (8) | 37 (20); 40 of 500 35 (4) 29 (6) 46 (8); d = 128, 12 of 300 27 (5) 35 (8).  With powers of two only, sized
  // to fill the device once, 80 of 2048 took 187, 40 of 500 46.
  const int blocks = (N + kC - 1) / kC;
  const long long ctas = (long long)B * h_count * (D / kW);
  // (Of a chain that brings a state all slices are one cluster: both read the caller's z, and one of them overwrites it.)
  const int slices = brings_state ? D / kW : 1;
  auto cost = [&](int segments, double waves) {
    const double per_block = (segments > 1 ? 1.37 : 1.0) * (ctas * segments > sms ? 1.6 : 1.0);
    return waves * ((blocks + segments - 1) / segments) * per_block;
  };
  int cluster = 1, G3 = 1;
  double best = cost(1, (double)((ctas + 2 * sms - 1) / (2 * sms)));
  for (int c = 2; c * slices <= kMaxCluster && c <= blocks; ++c) {
    const long long fit = (long long)resident_clusters<T, D>(c * slices, spread_smem(C::kSmem, c * ctas, sms), dev) * slices;
    if (fit < 1) continue;
    const double x = cost(c, (double)((ctas + fit - 1) / fit)) + 1.0;
    if (x < best) {
      best = x;
      cluster = c;
    }
  }
  if constexpr (sizeof(T) == 4) {
    for (int g = 2; g <= N / C::kMinSeg && (g == 2 || ctas * g <= 2LL * sms); ++g) {
      const double x = cost(g, (double)((ctas * g + 2 * sms - 1) / (2 * sms))) + 3.5;
      if (x < best) {
        best = x;
        G3 = g;
      }
    }
  }
  return {cluster, slices, G3, ctas};
}

template <typename T, int D>
cudaError_t linear_launch(const LinearPlan& plan, WalkArgs<T> p, int B, int N, int dev, int sms, cudaStream_t stream, Place place) {
  using C = LinT<D>;
  cudaError_t e;
  const int blocks = (N + kC - 1) / kC;
  if constexpr (sizeof(T) == 4) {
    if (plan.three > 1) {
      const int G = plan.three;
      const Segs sg = p.sg = {N, G, blocks / G, blocks % G};
      auto sum = linear_contribution_kernel<D>;
      if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(sum), dev, C::kSmemSum)) != cudaSuccess) return e;
      if ((e = launch_link(sum, dim3((G - 1) * (D / kW), p.h_count, B), dim3(kLinThreads), C::kSmemSum, stream, p.k, p.v, p.o,
                           sg, p.st, p.h_begin, Place{place.ws, place.wait_kcycles, place.drop_flag, 0})) != cudaSuccess)
        return e;
      constexpr int kItems = (D + C::ZROWS) * (D / 4);
      if ((e = launch_link(linear_prefix_kernel<D>, dim3((kItems + 127) / 128, p.h_count, B), dim3(128), 0, stream, p.o, sg,
                           p.st, p.h_begin, p.h_count, p.zero_init ? nullptr : p.S_io, p.z_io)) != cudaSuccess)
        return e;
      auto walk = linear_walk_kernel<float, D, false>;
      if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(walk), dev, spread_smem(C::kSmem, 1, sms))) != cudaSuccess) return e;
      return launch_link(walk, dim3(G * (D / kW), p.h_count, B), dim3(kLinThreads), C::kSmem, stream, p, 1, Place{nullptr, 0, 0, place.last});
    }
  }
  p.sg = {N, plan.cluster, blocks / plan.cluster, blocks % plan.cluster};
  const int cluster_ctas = plan.cluster * plan.slices;
  auto walk = cluster_ctas > 1 ? linear_walk_kernel<T, D, true> : linear_walk_kernel<T, D, false>;
  const int smem = spread_smem(C::kSmem, plan.cluster * plan.ctas, sms);
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(walk), dev, spread_smem(C::kSmem, 1, sms))) != cudaSuccess) return e;
  return launch_link_clusters(cluster_ctas, walk, dim3(plan.cluster * (D / kW), p.h_count, B), dim3(kLinThreads), smem, stream, p,
                              0, place);
}

// Both head groups in one launch: first the CTAs of the linear heads, `parts` per chain, then those of the windowed heads.
template <typename T, int D, bool kCluster>
__global__ void __launch_bounds__(kLinThreads, D == 64 ? 2 : 1)
layer_kernel(const WalkArgs<T> lp, const WindowArgs<T> wp, int parts, int n_lin, int h_sparse, int n_win, Place place) {
  static_assert(kLinThreads == kWinThreads, "one block size for both");
  extern __shared__ __align__(16) float sm[];
  begin(place);
  const int id = blockIdx.x;
  if (id < n_lin) {
    const int chain = id / parts, b = chain / lp.h_count;
    linear_walk<T, D, kCluster>(lp, id - chain * parts, chain - b * lp.h_count, b, sm);
  } else if (id - n_lin < n_win) {  // (the grid is a multiple of the cluster size)
    const int tiles = (wp.N + kWinRows - 1) / kWinRows, row = (id - n_lin) / tiles, b = row / h_sparse;
    any_window_tile<T, D>(wp, id - n_lin - row * tiles, row - b * h_sparse, b, sm);
  }
  grid_dep_launch();
}

template <typename T, int D>
cudaError_t layer_launch(WalkArgs<T> lp, const WindowArgs<T>& wp, int B, int h_sparse, cudaStream_t stream, Place place) {
  using C = LinT<D>;
  int dev = 0, sms = 0;
  cudaError_t e = device_info(&dev, &sms);
  if (e != cudaSuccess) return e;
  const int N = wp.N;
  const LinearPlan plan = linear_plan<T, D>(B, N, lp.h_count, false, dev, sms);
  const long long n_lin = plan.ctas * plan.cluster, n_win = (long long)B * h_sparse * ((N + kWinRows - 1) / kWinRows);
  // One launch for both unless the linear heads take three, or the device does not hold all CTAs at a time (two per SM, at d =
  // 128, by the windowed heads' registers, one; us, one launch and two: 1 x 2 heads of 1030 tokens, d = 128, 44.6 and 51.5, 1 x 8 of
  // 64 14.3 and 16.4; but 8 x 12 of 2048, d = 64, 189 and 181, 32 x 12 of 1024 330 and 321).
  if (plan.three > 1 || n_lin + n_win > (D == 64 ? 2LL : 1LL) * sms) {
    const Place first = {place.ws, place.wait_kcycles, place.drop_flag, 0};
    if ((e = linear_launch<T, D>(plan, lp, B, N, dev, sms, stream, first)) != cudaSuccess) return e;
    return window_launch<T, D>(wp, B, h_sparse, stream, Place{nullptr, 0, 0, place.last});
  }
  const int blocks = (N + kC - 1) / kC;
  lp.sg = {N, plan.cluster, blocks / plan.cluster, blocks % plan.cluster};
  auto kern = plan.cluster > 1 ? layer_kernel<T, D, true> : layer_kernel<T, D, false>;
  constexpr int kNeed = C::kSmem > window_smem<D>() ? C::kSmem : window_smem<D>();
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), dev, spread_smem(kNeed, 1, sms))) != cudaSuccess) return e;
  const long long grid = (n_lin + n_win + plan.cluster - 1) / plan.cluster * plan.cluster;
  return launch_link_clusters(plan.cluster, kern, dim3((unsigned)grid), dim3(kLinThreads),
                              spread_smem(kNeed, grid, sms), stream, lp, wp, plan.cluster * (D / kW), (int)n_lin, h_sparse,
                              (int)n_win, place);
}

template <typename F>
cudaError_t dispatch(int dtype, int d, F f) {
  if (dtype == GF_F32) return d == 64 ? f(float(), std::integral_constant<int, 64>()) : f(float(), std::integral_constant<int, 128>());
  return d == 64 ? f(__nv_bfloat16(), std::integral_constant<int, 64>()) : f(__nv_bfloat16(), std::integral_constant<int, 128>());
}

}  // namespace

cudaError_t launch_window_simt(const void* q, const void* k, const void* v, void* o, int B, int N, int d, int w, int fwd,
                               float scale, int dtype, Strides st, int h_begin, int h_count, cudaStream_t stream, Place place) {
  if (h_count <= 0 || B <= 0) return cudaSuccess;
  return dispatch(dtype, d, [&](auto t, auto dd) {
    using T = decltype(t);
    const WindowArgs<T> p = {(const T*)q, (const T*)k, (const T*)v, (T*)o, N, w, fwd, scale, st, h_begin};
    return window_launch<T, decltype(dd)::value>(p, B, h_count, stream, place);
  });
}

cudaError_t launch_linear_tiled(const void* q, const void* k, const void* v, void* o, int B, int N, int d, int dtype,
                                Strides st, int h_begin, int h_count, float* S_io, float* z_io, bool zero_init,
                                cudaStream_t stream, Place place) {
  if (h_count <= 0 || B <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  const cudaError_t e = device_info(&dev, &sms);
  if (e != cudaSuccess) return e;
  return dispatch(dtype, d, [&](auto t, auto dd) {
    using T = decltype(t);
    constexpr int D = decltype(dd)::value;
    const WalkArgs<T> p = {(const T*)q, (const T*)k, (const T*)v, (T*)o, Segs{}, st, h_begin, h_count, S_io, z_io, zero_init ? 1 : 0};
    const LinearPlan plan = linear_plan<T, D>(B, N, h_count, S_io != nullptr && !zero_init, dev, sms);
    return linear_launch<T, D>(plan, p, B, N, dev, sms, stream, place);
  });
}

cudaError_t launch_layer_tiled(const void* q, const void* k, const void* v, void* o, int B, int N, int d, int w, float scale,
                               int dtype, Strides st, int h_sparse, int h_lin, float* S_io, float* z_io, cudaStream_t stream,
                               Place place) {
  return dispatch(dtype, d, [&](auto t, auto dd) {
    using T = decltype(t);
    const WalkArgs<T> lp = {(const T*)q, (const T*)k, (const T*)v, (T*)o, Segs{}, st, h_sparse, h_lin, S_io, z_io, 1};
    const WindowArgs<T> wp = {(const T*)q, (const T*)k, (const T*)v, (T*)o, N, w, 0, scale, st, 0};
    return layer_launch<T, decltype(dd)::value>(lp, wp, B, h_sparse, stream, place);
  });
}

}  // namespace gf
