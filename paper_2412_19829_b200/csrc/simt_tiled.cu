// Attention in fp32 arithmetic on the CUDA cores, as register-tiled products: the windowed heads and the causal
// linear heads of fp32 tensors (and of bf16 ones when the tensor-core kernels are switched off).
//
// Both kernels walk 32-token blocks with 128 threads.  A thread's tile of a product is 4 rows x 4 columns (4 x 2 of a
// score block, D/8 x 4 of the state).  Rows are i + 8 r of a block, so that the eight row groups of a warp read eight
// different padded rows of shared memory without bank conflicts; operands are read 16 bytes at a time, along the
// contracted dimension for A and along the columns for B.  The next block's rows are loaded into registers while one
// is worked on: loaded when they are needed, a block waited about 5 us for them.
// What bounds both is shared memory: for these tiles the 16-byte loads take 1.5 to 3 times the cycles of the
// multiply-adds (ncu at 8 x 12 heads x 2048 tokens, d = 64, w = 128: shared-memory pipe 60-75 % busy, FMA pipe 40-49 %).
// Larger tiles (64 threads, 4 x 8, 4 x 4 and 8 x 8) need a third fewer loads but leave 8 warps per SM: no faster there
// (244 us for the layer either way).  Token by token, with a block-wide reduction per 16 tokens and no reuse of K, it took
// 756 us, and 2 heads of 256 tokens 57 us, now 17.
#include <cooperative_groups.h>

#include "common.cuh"

namespace gf {
namespace {

constexpr int kC = 32;    // tokens per block
constexpr int kNT = 128;  // threads per CTA
constexpr int kW = 64;    // value columns per CTA of the linear heads
constexpr int kLdP = kC + 4;

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
__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
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

// (also of infinities of both signs)
__device__ __forceinline__ bool has_nan(float4 x) {
  const float s = (x.x + x.y) + (x.z + x.w);
  return s != s;
}

// A block's rows on their way from global to shared memory: COLS columns of 32 tokens, all loads of a thread in
// flight at once and issued a block ahead of their use.  Rows past the end are zero.
template <typename T, int COLS>
struct BlockRegs {
  static constexpr int C4 = COLS / 4, kN = kC * C4 / kNT, kStep = kNT / C4;
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

// Scores of a 32 x 32 block: rows i + 8 r of A against rows jg + 16 s of B, both [32][D + 4].
template <int D>
__device__ __forceinline__ void score_block(const float* A, const float* B, int i, int jg, float (&acc)[4][2]) {
  constexpr int LD = D + 4;
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = 0.f;
#pragma unroll 4
  for (int a = 0; a < D; a += 4) {
    const float4 b0 = lds4(B + jg * LD + a), b1 = lds4(B + (jg + 16) * LD + a);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 x = lds4(A + (i + 8 * r) * LD + a);
      acc[r][0] = dot4(x, b0, acc[r][0]);
      acc[r][1] = dot4(x, b1, acc[r][1]);
    }
  }
}
// acc[r][c] += rows i + 8 r of A (K entries each, row stride lda) times B, four columns at col(k, c)
template <int K, int NG, typename Col>
__device__ __forceinline__ void product(float4 (&acc)[4][NG], const float* A, int lda, int i, Col col) {
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    float4 x[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) x[r] = lds4(A + (i + 8 * r) * lda + k);
#pragma unroll
    for (int c = 0; c < NG; ++c) {
      const float4 b0 = lds4(col(k, c)), b1 = lds4(col(k + 1, c)), b2 = lds4(col(k + 2, c)), b3 = lds4(col(k + 3, c));
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        axpy4(acc[r][c], x[r].x, b0);
        axpy4(acc[r][c], x[r].y, b1);
        axpy4(acc[r][c], x[r].z, b2);
        axpy4(acc[r][c], x[r].w, b3);
      }
    }
  }
}

// ------------------------------------------------------------------------------------ windowed heads
// One CTA = 32 query rows of one head; keys and values pass through shared memory 32 at a time; online softmax
// with the running maximum and sum of a row kept by the four threads that share it.
template <int D>
constexpr int window_smem() { return (2 * kC * (D + 4) + kC * D + kC * kLdP + kC) * 4; }

// Masked keys have weight 0 in the products above, which is nothing unless their value is infinite or NaN (0 x inf = NaN):
// the output row of query i once more, by the four threads that share it, over the keys it sees and no others.  m, l: its
// final maximum and sum.
template <typename T, int D>
__device__ __forceinline__ void window_row(const T* q, const T* k, const T* v, T* o, int i, int j_begin, int j_end, float scale,
                                        long long stride, int part, unsigned int quad, float m, float l) {
  float4 acc[D / 16];
#pragma unroll
  for (int c = 0; c < D / 16; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int j = j_begin; j < j_end; ++j) {
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < D / 16; ++c)
      s = dot4(load4<T>(q + i * stride + 4 * (part + 4 * c)), load4<T>(k + j * stride + 4 * (part + 4 * c)), s);
    s += __shfl_xor_sync(quad, s, 1);
    s += __shfl_xor_sync(quad, s, 2);
    const float p = expf(s * scale - m);
#pragma unroll
    for (int c = 0; c < D / 16; ++c) axpy4(acc[c], p, load4<T>(v + j * stride + 4 * (part + 4 * c)));
  }
#pragma unroll
  for (int c = 0; c < D / 16; ++c)
    store4(o + i * stride + 4 * (part + 4 * c), make_float4(acc[c].x / l, acc[c].y / l, acc[c].z / l, acc[c].w / l));
}

template <typename T, int D>
__global__ void __launch_bounds__(kNT, D == 64 ? 5 : 3)  // (else the rare path at the end takes registers from the rest)
window_tiled_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, T* __restrict__ o,
                    int N, int w, int fwd, float scale, Strides st, int h_begin) {
  // fwd: keys after the query that it may see (0: the causal window; w - 1: the two-sided one)
  grid_dep_launch();
  constexpr int LD = D + 4, NC = D / 64;  // NC: groups of four output columns per thread, 64 apart
  extern __shared__ __align__(16) float sm[];
  float *Qs = sm, *Ks = Qs + kC * LD, *Vs = Ks + kC * LD, *Ps = Vs + kC * D, *As = Ps + kC * kLdP;

  const long long base = (long long)blockIdx.z * st.b + (long long)(h_begin + blockIdx.y) * st.h;
  const int i0 = blockIdx.x * kC, tid = threadIdx.x, lane = tid & 31;
  const int i = lane & 7, cg = (tid >> 5) * 4 + (lane >> 3);  // row group, column group of the products
  const int t = tid >> 2, part = tid & 3;                     // row and quarter of it in the softmax

  const int jlo = max(i0 - w + 1, 0), jhi = min(i0 + kC - 1 + fwd, N - 1);
  BlockRegs<T, D> rk, rv;
  rk.load(q + base, st.n, i0, N, tid);
  rk.store(Qs, LD, tid);
  rk.load(k + base, st.n, jlo, N, tid);
  rv.load(v + base, st.n, jlo, N, tid);
  float4 acc[4][NC];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[r][c] = make_float4(0.f, 0.f, 0.f, 0.f);
  float m = -INFINITY, l = 0.f;

  for (int j0 = jlo; j0 <= jhi; j0 += kC) {
    rk.store(Ks, LD, tid);
    rv.store(Vs, D, tid);
    __syncthreads();
    if (j0 + kC <= jhi) {
      rk.load(k + base, st.n, j0 + kC, N, tid);
      rv.load(v + base, st.n, j0 + kC, N, tid);
    }
    {
      float s[4][2];
      score_block<D>(Qs, Ks, i, cg, s);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        Ps[(i + 8 * r) * kLdP + cg] = s[r][0];
        Ps[(i + 8 * r) * kLdP + cg + 16] = s[r][1];
      }
    }
    __syncthreads();
    {
      float* row = Ps + t * kLdP + part * 8;
      const float4 x0 = lds4(row), x1 = lds4(row + 4);
      float s[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      const int lo = i0 + t - w - (j0 + part * 8), hi = min(i0 + t + fwd, N - 1) - (j0 + part * 8);  // lo < e <= hi
      float mx = -INFINITY;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        s[e] = (e > lo && e <= hi) ? s[e] * scale : -INFINITY;
        mx = fmaxf(mx, s[e]);
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float m_new = fmaxf(m, mx);
      const float ref = (m_new == -INFINITY) ? 0.f : m_new;  // a row that has seen no key yet
      const float corr = expf(m - ref);
      float sum = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        s[e] = expf(s[e] - ref);
        sum += s[e];
      }
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      l = l * corr + sum;
      m = m_new;
      *reinterpret_cast<float4*>(row) = make_float4(s[0], s[1], s[2], s[3]);
      *reinterpret_cast<float4*>(row + 4) = make_float4(s[4], s[5], s[6], s[7]);
      if (part == 0) As[t] = corr;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float corr = As[i + 8 * r];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        acc[r][c].x *= corr;
        acc[r][c].y *= corr;
        acc[r][c].z *= corr;
        acc[r][c].w *= corr;
      }
    }
    product<kC, NC>(acc, Ps, kLdP, i, [&](int j, int c) { return Vs + j * D + c * 64 + 4 * cg; });
    __syncthreads();
  }
  if (part == 0) {
    As[t] = 1.f / l;
    Ps[t] = 0.f;  // 1: the row has a NaN
  }
  __syncthreads();
  bool any = false;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = i + 8 * r;
    if (i0 + row >= N) continue;
    const float inv = As[row];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (has_nan(acc[r][c])) {
        Ps[row] = 1.f;
        any = true;
      }
      store4(o + base + (long long)(i0 + row) * st.n + c * 64 + 4 * cg,
             make_float4(acc[r][c].x * inv, acc[r][c].y * inv, acc[r][c].z * inv, acc[r][c].w * inv));
    }
  }
  if (__syncthreads_or(any) && Ps[t] != 0.f)
    window_row<T, D>(q + base, k + base, v + base, o + base, i0 + t, max(i0 + t - w + 1, 0), min(i0 + t + fwd, N - 1) + 1, scale,
                     st.n, part, 0xfu << (lane & 28), m, l);
  if (blockIdx.x + blockIdx.y + blockIdx.z == 0) grid_dep_wait();
}

// ------------------------------------------------------------------------------------ causal linear heads
// Algorithm 1 regrouped in blocks of 32 tokens (exactly equal by associativity): with S, z the sums before a block,
//   P = phi(Q) phi(K)^T masked to j <= i,   O = (P V + phi(Q) S) / (rowsum(P) + phi(Q) z),
//   S += phi(K)^T V,   z += colsum(phi(K)).
// A CTA owns 64 value columns of a chain; S lives in its registers (a thread: D/8 features x 4 columns) with a copy
// in shared memory for the readout.
//
// With few chains a chain is cut into G segments, so that every SM has work.  Up to kMaxCluster of them are a cluster of
// CTAs in one launch (kCluster): each sums its own segment, then adds up the sums of those before it from their shared
// memory, then walks.  Where a chain has two CTAs per segment (D = 128) and brings a state, both are in the cluster: both read
// the caller's z, and one of them overwrites it, which has to wait until the other has started.  Longer chains in smaller numbers take three launches, with segments of a little more than D tokens:
//   contribution   the sums of every segment but the last, each alone
//   prefix         running sums over the segments of a chain
//   walk           the segments' outputs, each from its own starting state
// The states wait in the rows of the OUTPUT tensor that their own segment will later overwrite (row a of S in the
// row of token a of the segment, z in the next row or two, one per 64 columns): no workspace, and a CTA of the walk
// reads only rows and columns that itself will write.
constexpr int kMaxCluster = 8;
template <int D> struct LinT {
  static constexpr int LD = D + 4;
  static constexpr int ZROWS = D / 64;  // rows z takes behind S
  // shortest segment: D + ZROWS rows, also when the last segment's last block is a single token
  static constexpr int kMinSeg = D + 32 * ZROWS;
  static constexpr int kSmem = (2 * kC * LD + kC * kW + D * kW + kC * kLdP + D + kC) * 4;
  static constexpr int kSmemSum = (kC * LD + kC * kW) * 4;
};
struct Segs {  // tokens [begin(g), begin(g + 1)) of segment g, whole blocks but for the last
  int N, G, base, rem;  // blocks per segment: base, one more for the first rem
  __host__ __device__ int begin(int g) const { return g >= G ? N : kC * (g * base + (g < rem ? g : rem)); }
};

// The 16-byte column groups of row a of the shared copy of S are swizzled, so that the eight feature groups of a warp
// store without bank conflicts.
__device__ __forceinline__ int s_off(int a, int col) { return a * kW + (col ^ (a & 28)); }

// S += phi(K)^T V: features 4 ag .. 4 ag + 3 of every 32, columns 4 cg .. 4 cg + 3
template <int D>
__device__ __forceinline__ void add_outer(const float* Ks, const float* Vs, int ag, int cg, float4 (&S)[D / 8]) {
#pragma unroll 2
  for (int j = 0; j < kC; ++j) {
    const float4 vv = lds4(Vs + j * kW + 4 * cg);
#pragma unroll
    for (int e = 0; e < D / 32; ++e) {
      const float4 kk = lds4(Ks + j * (D + 4) + 32 * e + 4 * ag);
      axpy4(S[4 * e + 0], kk.x, vv);
      axpy4(S[4 * e + 1], kk.y, vv);
      axpy4(S[4 * e + 2], kk.z, vv);
      axpy4(S[4 * e + 3], kk.w, vv);
    }
  }
}
// f(feature, element) for the thread's 4-column pieces of S
template <int D, typename F>
__device__ __forceinline__ void for_state(int ag, float4 (&S)[D / 8], F f) {
#pragma unroll
  for (int e = 0; e < D / 32; ++e)
#pragma unroll
    for (int x = 0; x < 4; ++x) f(32 * e + 4 * ag + x, S[4 * e + x]);
}
template <int D>
__device__ __forceinline__ float column_sum(const float* col) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < kC; ++j) s[j & 3] += col[j * (D + 4)];
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// Adds tokens [n_begin, n_end) to S and z (thread tid < D: feature tid).
template <typename T, int D>
__device__ __forceinline__ void sum_segment(const T* k, const T* v, long long stride, int n_begin, int n_end, float* Ks,
                                            float* Vs, int tid, int ag, int cg, float4 (&S)[D / 8], float& z) {
  BlockRegs<T, D> rk;
  BlockRegs<T, kW> rv;
  rk.load(k, stride, n_begin, n_end, tid);
  rv.load(v, stride, n_begin, n_end, tid);
  for (int n0 = n_begin; n0 < n_end; n0 += kC) {
    rk.store_phi(Ks, D + 4, n0, n_end, tid);
    rv.store(Vs, kW, tid);
    __syncthreads();
    rk.load(k, stride, n0 + kC, n_end, tid);
    rv.load(v, stride, n0 + kC, n_end, tid);
    add_outer<D>(Ks, Vs, ag, cg, S);
    if (tid < D) z += column_sum<D>(Ks + tid);
    __syncthreads();
  }
}

template <int D>
__global__ void __launch_bounds__(kNT)
linear_contribution_kernel(const float* __restrict__ k, const float* __restrict__ v, float* __restrict__ o, Segs sg,
                           Strides st, int h_begin) {
  extern __shared__ __align__(16) float sm[];
  grid_dep_launch();
  float *Ks = sm, *Vs = Ks + kC * (D + 4);
  const int g = blockIdx.x / (D / kW), col0 = (blockIdx.x % (D / kW)) * kW;
  const long long base = (long long)blockIdx.z * st.b + (long long)(h_begin + blockIdx.y) * st.h;
  const int tid = threadIdx.x, lane = tid & 31, ag = lane & 7, cg = (tid >> 5) * 4 + (lane >> 3);
  float4 S[D / 8];
  for_state<D>(ag, S, [](int, float4& x) { x = make_float4(0.f, 0.f, 0.f, 0.f); });
  float z = 0.f;
  const int n_end = sg.begin(g + 1);
  sum_segment<float, D>(k + base, v + base + col0, st.n, sg.begin(g), n_end, Ks, Vs, tid, ag, cg, S, z);
  float* slot = o + base + (long long)n_end * st.n + col0;  // the state before segment g + 1, once summed
  for_state<D>(ag, S, [&](int a, float4& x) { store4(slot + (long long)a * st.n + 4 * cg, x); });
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

// Without cuts (G == 1) the state before token 0 comes from S_io; with cuts from the segment's slot (segment 0 has
// one only when there is an initial state), or, kCluster, from S_io and the cluster's CTAs before this one.  A chain that
// brings a state and has several slices is one cluster (G x D / kW CTAs), also when it is not cut.
template <typename T, int D, bool kCluster>
__global__ void __launch_bounds__(kNT)
linear_walk_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, T* o, Segs sg, Strides st,
                   int h_begin, int h_count, float* S_io, float* z_io, int zero_init, int after) {
  constexpr int LD = LinT<D>::LD;
  if (after) grid_dep_wait();  // the segments' starting states
  grid_dep_launch();
  extern __shared__ __align__(16) float sm[];
  float *Qs = sm, *Ks = Qs + kC * LD, *Vs = Ks + kC * LD, *Ss = Vs + kC * kW, *Ps = Ss + D * kW, *zs = Ps + kC * kLdP,
        *inv_s = zs + D;
  // (a cluster's CTAs are neighbours in x: the segments of one slice, then those of the next)
  const int g = kCluster ? blockIdx.x % sg.G : blockIdx.x / (D / kW);
  const int col0 = (kCluster ? blockIdx.x / sg.G : blockIdx.x % (D / kW)) * kW;
  const long long base = (long long)blockIdx.z * st.b + (long long)(h_begin + blockIdx.y) * st.h;
  const long long sidx = (long long)blockIdx.z * h_count + blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31;
  const int i = lane & 7, cg = (tid >> 5) * 4 + (lane >> 3);
  const int n_begin = sg.begin(g), n_end = sg.begin(g + 1);

  float4 S[D / 8];
  if constexpr (kCluster) {
    auto cluster = cooperative_groups::this_cluster();
    for_state<D>(i, S, [](int, float4& x) { x = make_float4(0.f, 0.f, 0.f, 0.f); });
    float z = 0.f;
    if (g < sg.G - 1) {  // nobody needs the last segment's sum
      sum_segment<T, D>(k + base, v + base + col0, st.n, n_begin, n_end, Ks, Vs, tid, i, cg, S, z);
      for_state<D>(i, S, [&](int a, float4& x) { *reinterpret_cast<float4*>(Ss + s_off(a, 4 * cg)) = x; });
      if (tid < D) zs[tid] = z;
    }
    const bool from_caller = S_io != nullptr && !zero_init;
    for_state<D>(i, S, [&](int a, float4& x) {
      x = from_caller ? load4<float>(S_io + (sidx * D + a) * D + col0 + 4 * cg) : make_float4(0.f, 0.f, 0.f, 0.f);
    });
    z = (from_caller && tid < D) ? z_io[sidx * D + tid] : 0.f;
    cluster.sync();
    const int rank0 = (int)cluster.block_rank() - g;  // first segment of this slice
    for (int gg = 0; gg < g; ++gg) {
      const float* Sr = cluster.map_shared_rank(Ss, rank0 + gg);
      for_state<D>(i, S, [&](int a, float4& x) {
        const float4 y = lds4(Sr + s_off(a, 4 * cg));
        x.x += y.x;
        x.y += y.y;
        x.z += y.z;
        x.w += y.w;
      });
      if (tid < D) z += *cluster.map_shared_rank(zs + tid, rank0 + gg);
    }
    cluster.sync();  // everybody has read what is overwritten now, and the caller's state, which the last CTAs will overwrite
    for_state<D>(i, S, [&](int a, float4& x) { *reinterpret_cast<float4*>(Ss + s_off(a, 4 * cg)) = x; });
    if (tid < D) zs[tid] = z;
  } else {
    const float* Sp = nullptr;  // row a of the starting state at Sp + a * stride
    long long stride = D;
    const float* zp = nullptr;
    if (sg.G > 1 && (g > 0 || (S_io != nullptr && !zero_init))) {
      if constexpr (sizeof(T) == 4) {
        Sp = reinterpret_cast<const float*>(o) + base + (long long)n_begin * st.n + col0;
        stride = st.n;
      }
    } else if (g == 0 && S_io != nullptr && !zero_init) {
      Sp = S_io + sidx * D * D + col0;
      zp = z_io + sidx * D;
    }
    for_state<D>(i, S, [&](int a, float4& x) {
      x = Sp != nullptr ? load4<float>(Sp + a * stride + 4 * cg) : make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(Ss + s_off(a, 4 * cg)) = x;
    });
    if (tid < D)
      zs[tid] = Sp == nullptr ? 0.f : zp != nullptr ? zp[tid] : Sp[(long long)(D + tid / kW) * stride + tid % kW];
  }
  BlockRegs<T, D> rq, rk;
  BlockRegs<T, kW> rv;
  rq.load(q + base, st.n, n_begin, n_end, tid);
  rk.load(k + base, st.n, n_begin, n_end, tid);
  rv.load(v + base + col0, st.n, n_begin, n_end, tid);
  for (int n0 = n_begin; n0 < n_end; n0 += kC) {
    rq.store_phi(Qs, LD, n0, n_end, tid);
    rk.store_phi(Ks, LD, n0, n_end, tid);
    rv.store(Vs, kW, tid);
    __syncthreads();  // (also: every thread has read its state out of the rows this CTA writes)
    rq.load(q + base, st.n, n0 + kC, n_end, tid);
    rk.load(k + base, st.n, n0 + kC, n_end, tid);
    rv.load(v + base + col0, st.n, n0 + kC, n_end, tid);
    {
      float p[4][2];
      score_block<D>(Qs, Ks, i, cg, p);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int row = i + 8 * r;
        Ps[row * kLdP + cg] = cg <= row ? p[r][0] : 0.f;
        Ps[row * kLdP + cg + 16] = cg + 16 <= row ? p[r][1] : 0.f;
      }
    }
    __syncthreads();
    {  // denominators: four threads per row
      const int t = tid >> 2, part = tid & 3;
      float den = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) den += Ps[t * kLdP + part + 4 * e];
#pragma unroll 4
      for (int a = 4 * part; a < D; a += 16) den = dot4(lds4(Qs + t * LD + a), lds4(zs + a), den);
      den += __shfl_xor_sync(0xffffffffu, den, 1);
      den += __shfl_xor_sync(0xffffffffu, den, 2);
      if (part == 0) inv_s[t] = 1.f / den;
    }
    float4 acc[4][1];
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r][0] = make_float4(0.f, 0.f, 0.f, 0.f);
    product<D, 1>(acc, Qs, LD, i, [&](int a, int) { return Ss + s_off(a, 4 * cg); });
    product<kC, 1>(acc, Ps, kLdP, i, [&](int j, int) { return Vs + j * kW + 4 * cg; });
    const bool more = n0 + kC < n_end || (g == sg.G - 1 && S_io != nullptr);  // somebody wants the state after this block
    if (more) add_outer<D>(Ks, Vs, i, cg, S);
    if (__syncthreads_or(has_nan(acc[0][0]) || has_nan(acc[1][0]) || has_nan(acc[2][0]) || has_nan(acc[3][0]))) {
      // a masked weight is 0, which is nothing unless the value is infinite or NaN (0 x inf = NaN): the same sums without
      // the masked ones, so that a row sees no later value
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int row = i + 8 * r;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int a = 0; a < D; ++a) axpy4(x, Qs[row * LD + a], lds4(Ss + s_off(a, 4 * cg)));
#pragma unroll 1
        for (int j = 0; j <= row; ++j) axpy4(x, Ps[row * kLdP + j], lds4(Vs + j * kW + 4 * cg));
        acc[r][0] = x;
      }
      __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = i + 8 * r;
      if (n0 + row >= n_end) continue;
      const float inv = inv_s[row];
      store4(o + base + (long long)(n0 + row) * st.n + col0 + 4 * cg,
             make_float4(acc[r][0].x * inv, acc[r][0].y * inv, acc[r][0].z * inv, acc[r][0].w * inv));
    }
    if (more) {
      for_state<D>(i, S, [&](int a, float4& x) { *reinterpret_cast<float4*>(Ss + s_off(a, 4 * cg)) = x; });
      if (tid < D) zs[tid] += column_sum<D>(Ks + tid);
    }
    __syncthreads();
  }
  if (g == sg.G - 1 && S_io != nullptr) {
    for_state<D>(i, S, [&](int a, float4& x) { store4(S_io + (sidx * D + a) * D + col0 + 4 * cg, x); });
    if (col0 == 0 && tid < D) z_io[sidx * D + tid] = zs[tid];
  }
  if (blockIdx.x + blockIdx.y + blockIdx.z == 0) grid_dep_wait();
}

template <typename T, int D>
cudaError_t window_launch(const void* q, const void* k, const void* v, void* o, int B, int N, int w, int fwd, float scale,
                          Strides st, int h_begin, int h_count, cudaStream_t stream, Link link) {
  int dev = 0, sms = 0;
  cudaError_t e = device_info(&dev, &sms);
  if (e != cudaSuccess) return e;
  auto kern = window_tiled_kernel<T, D>;
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), dev, window_smem<D>())) != cudaSuccess) return e;
  return launch_link(link, kern, dim3((N + kC - 1) / kC, h_count, B), dim3(kNT), window_smem<D>(), stream, (const T*)q,
                     (const T*)k, (const T*)v, (T*)o, N, w, fwd, scale, st, h_begin);
}

template <typename T, int D>
cudaError_t linear_launch(const void* q, const void* k, const void* v, void* o, int B, int N, Strides st, int h_begin,
                          int h_count, float* S_io, float* z_io, bool zero_init, cudaStream_t stream, Link link) {
  using C = LinT<D>;
  int dev = 0, sms = 0;
  cudaError_t e = device_info(&dev, &sms);
  if (e != cudaSuccess) return e;
  // Clusters as large as one wave allows (three CTAs per SM at d = 64, two at 128, by registers), unless three launches
  // can cut a chain into clearly more segments.  Measured (us, clusters of 8 | of 4 | three launches): 1 chain of 256
  // tokens 17 | 21 | 39, 8 of 300 24.6 | 28.7 | 39, 6 of 1000 (d = 128) 74 | 107 | 100, 80 of 500 93 | 70.5 | 71, 80 of
  // 2048 267 | 248 | 244, 1 of 2048 (d = 128) 113 | 203 | 99.  Clusters of 16 are no faster, and with 80 KB of shared
  // memory per CTA slower (6 of 1000: 135).
  const int blocks = (N + kC - 1) / kC;
  const long long ctas = (long long)B * h_count * (D / kW), wave = (D == 64 ? 3LL : 2LL) * sms;
  // (Of a chain that brings a state all slices are one cluster, which at d = 128 leaves room for four segments: 6 of 1000 then
  // take the three launches, 76 -> 100 us, 17 of 1000 165 -> 134, 18 of 500 118 -> 91.  Clusters of 16 CTAs take 76 us for
  // 6 of 1000 but 189 for 17.)
  const int slices = (S_io != nullptr && !zero_init) ? D / kW : 1;
  int cluster = 1;
  while (2 * cluster * slices <= kMaxCluster && 2 * cluster <= blocks && 2 * cluster * ctas <= wave) cluster *= 2;
  if constexpr (sizeof(T) == 4) {
    long long G3 = ctas < 4LL * sms ? (8LL * sms + ctas - 1) / ctas : 1;
    if (G3 > N / C::kMinSeg) G3 = N / C::kMinSeg;
    if (5 * G3 > 6 * cluster) {
      const int G = (int)G3;
      const Segs sg = {N, G, blocks / G, blocks % G};
      auto sum = linear_contribution_kernel<D>;
      if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(sum), dev, C::kSmemSum)) != cudaSuccess) return e;
      if ((e = launch_link(link, sum, dim3((G - 1) * (D / kW), h_count, B), dim3(kNT), C::kSmemSum, stream, (const float*)k,
                           (const float*)v, (float*)o, sg, st, h_begin)) != cudaSuccess)
        return e;
      constexpr int kItems = (D + C::ZROWS) * (D / 4);
      if ((e = launch_link(kAfter, linear_prefix_kernel<D>, dim3((kItems + 127) / 128, h_count, B), dim3(128), 0, stream,
                           (float*)o, sg, st, h_begin, h_count, zero_init ? nullptr : S_io, z_io)) != cudaSuccess)
        return e;
      auto walk = linear_walk_kernel<float, D, false>;
      if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(walk), dev, C::kSmem)) != cudaSuccess) return e;
      return launch_link(kAfter, walk, dim3(G * (D / kW), h_count, B), dim3(kNT), C::kSmem, stream, (const float*)q,
                         (const float*)k, (const float*)v, (float*)o, sg, st, h_begin, h_count, S_io, z_io, zero_init ? 1 : 0, 1);
    }
  }
  const Segs sg = {N, cluster, blocks / cluster, blocks % cluster};
  const int cluster_ctas = cluster * slices;
  auto walk = cluster_ctas > 1 ? linear_walk_kernel<T, D, true> : linear_walk_kernel<T, D, false>;
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(walk), dev, C::kSmem)) != cudaSuccess) return e;
  return launch_link_clusters(link, cluster_ctas, walk, dim3(cluster * (D / kW), h_count, B), dim3(kNT), C::kSmem, stream,
                              (const T*)q, (const T*)k, (const T*)v, (T*)o, sg, st, h_begin, h_count, S_io, z_io,
                              zero_init ? 1 : 0, 0);
}

}  // namespace

cudaError_t launch_window_simt(const void* q, const void* k, const void* v, void* o, int B, int N, int d, int w, int fwd,
                               float scale, int dtype, Strides st, int h_begin, int h_count, cudaStream_t stream,
                               Link link) {
  if (h_count <= 0 || B <= 0) return cudaSuccess;
  auto* f = dtype == GF_F32 ? (d == 64 ? window_launch<float, 64> : window_launch<float, 128>)
                            : (d == 64 ? window_launch<__nv_bfloat16, 64> : window_launch<__nv_bfloat16, 128>);
  return f(q, k, v, o, B, N, w, fwd, scale, st, h_begin, h_count, stream, link);
}

cudaError_t launch_linear_tiled(const void* q, const void* k, const void* v, void* o, int B, int N, int d, int dtype,
                                Strides st, int h_begin, int h_count, float* S_io, float* z_io, bool zero_init,
                                cudaStream_t stream, Link link) {
  if (h_count <= 0 || B <= 0) return cudaSuccess;
  auto* f = dtype == GF_F32 ? (d == 64 ? linear_launch<float, 64> : linear_launch<float, 128>)
                            : (d == 64 ? linear_launch<__nv_bfloat16, 64> : linear_launch<__nv_bfloat16, 128>);
  return f(q, k, v, o, B, N, st, h_begin, h_count, S_io, z_io, zero_init, stream, link);
}

}  // namespace gf
