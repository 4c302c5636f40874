// Global (unmasked) linear attention on the tensor cores: the linear heads of the bidirectional
// ("self") layer.  Sec. II-B without the causal mask:
//   S = sum_j phi(K_j) (x) V_j,  z = sum_j phi(K_j)   over the whole sequence,
//   out_i = phi(Q_i)^T S / (phi(Q_i) . z).
// Three launches, bf16 in, fp32 accumulate:
//   reduce   a chain is cut into segments; a CTA walks a segment's 128-row chunks: K and V tiles by
//            TMA, phi(K) in place in shared memory (16 warps), [S | z] += phi(K)^T [V | 1] as one
//            tcgen05.mma per 16 keys with N = D + 16 (V's B operand is followed by a constant box
//            whose column 0 is all ones, so z is column D of the accumulator); the segment's sum
//            goes from TMEM to a scratch slot of its own.
//   sum      adds the segments' slots of a chain in a fixed order (CUDA cores): deterministic totals.
//   readout  a CTA loads a chain's totals once per item as the bf16 B operand [Sb | hi(z) lo(z)],
//            then per chunk: Q tile by TMA, phi(Q) into TMEM (8 warps), one product with
//            N = D + 16 leaves the numerators and, in columns D and D + 1, the denominator split
//            in two; 4 epilogue warps divide, pack and stage the tile for a TMA store.
// At D = 64, where shared memory has room for both halves, and with chains enough for the SMs (or chains that are
// short), one launch does it all:
//   whole    a CTA takes whole chains; it sums chain c + 1 while it reads out chain c
// Every wait is bounded; on expiry the kernel records a status word and drains.
#include "common.cuh"
#include "linear_phi.cuh"
#include "sm100.cuh"

namespace gf {
namespace {

using namespace sm100;

constexpr int kBox = 16384;  // one 128-row x 64-column bf16 box (what one TMA copy moves)

struct SelfParams {
  int N, nch, h_begin, h_count, nchains;
  int G, seg_base, seg_rem, nitems;  // segments per chain (balanced lengths), nchains * G
  float* partial;                    // [nitems][D*D + D]: a segment's sums (S row-major [feature][column], then z)
  float* total;                      // [nchains][D*D + D]
  unsigned int* status;
  // What the launches hand on is counted per chain, because the windowed heads of a layer run between them: warps that have
  // written their rows of a segment's sums (4 G), then blocks of the totals (sum_blocks, with more than one segment).
  // Zero at launch.
  unsigned int *summed, *totalled;
  unsigned int sum_blocks;
  int totals_of_one;  // the sums were formed in one segment per chain: no totals
  LetGo let_go;       // of the kernel for whole chains
};
constexpr int kSumThreads = 64;

__device__ __forceinline__ void count_up(unsigned int* counter) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
}
// Bounded poll (acquire) until the counter has reached the target.
__device__ __forceinline__ bool wait_count(const unsigned int* counter, unsigned int target, unsigned int* status,
                                           unsigned int where) {
  const long long t0 = clock64();
  for (unsigned int n = 0;; ++n) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    if (v >= target) return true;
    if (n > 0 && clock64() - t0 > wait_limit_cycles(status)) {
      if (atomicCAS(status, 0u, 1u) == 0u) status[1] = where;
      return false;
    }
    __nanosleep(100);
  }
}

struct SelfItem {
  int chain, g, b, hl, h, c_begin, nC;
};

__device__ __forceinline__ SelfItem self_item(const SelfParams& p, int item) {
  SelfItem it;
  it.chain = item / p.G;
  it.g = item - it.chain * p.G;
  it.b = it.chain / p.h_count;
  it.hl = it.chain - it.b * p.h_count;
  it.h = p.h_begin + it.hl;
  it.c_begin = it.g * p.seg_base + (it.g < p.seg_rem ? it.g : p.seg_rem);
  it.nC = p.seg_base + (it.g < p.seg_rem ? 1 : 0);
  return it;
}

// ------------------------------------------------------------------------------------ reduce
template <int D>
struct RedCfg {
  static constexpr int kTile = 128 * D * 2;
  // V | ones: one constant box serves every V slot, a box distance past the slot's last box:
  //   D = 128:  V0a . V1a V0b V1b . ONES   (slot 0: distance 3 boxes, slot 1: 2; two boxes unused)
  //   D = 64:   V0 V1 V2 V3 ONES           (slot s: distance 4 - s)
  static constexpr int kVSlots = (D == 128) ? 2 : 4;
  __host__ __device__ static constexpr int v_off(int s) { return (D == 128) ? (s ? 2 : 0) * kBox : s * kBox; }
  __host__ __device__ static constexpr int v_lbo(int s) { return (D == 128) ? (s ? 2 : 3) * kBox : (4 - s) * kBox; }
  static constexpr int kOnes = (D == 128) ? 6 * kBox : 4 * kBox;
  static constexpr int kK = kOnes + kBox;  // three K slots, contiguous
  static constexpr int kKSlots = 3;
  static constexpr int kBytes = kK + kKSlots * kTile + 1024;
  static constexpr int kAcc = D + 16;  // accumulator columns: S, then z in column D
  static constexpr int kThreads = 22 * 32;
};

template <int D, bool kId>
__global__ void __launch_bounds__(RedCfg<D>::kThreads, 1)
linear_self_reduce_kernel(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv,
                          const SelfParams p) {
  using C = RedCfg<D>;
  constexpr int VS = C::kVSlots, KS = C::kKSlots;
  extern __shared__ uint8_t raw_smem[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw_smem) + 1023) & ~(uintptr_t)1023);
  uint8_t* sK = sm + C::kK;
  uint8_t* sOnes = sm + C::kOnes;
  __shared__ __align__(8) uint64_t k_full[KS], kphi[KS], k_free[KS], v_full[4], v_free[4], acc_done[2], acc_free[2];
  __shared__ uint32_t tmem_base_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int i = 0; i < KS; ++i) {
      mbar_init(&k_full[i], 1);
      mbar_init(&kphi[i], 16);
      mbar_init(&k_free[i], 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(&v_full[i], 1);
      mbar_init(&v_free[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_done[i], 1);
      mbar_init(&acc_free[i], 128);
    }
    mbar_fence_init();
    tma_prefetch_desc(&mk);
    tma_prefetch_desc(&mv);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base_s, 512);
    tmem_relinquish();
  } else if (warp >= 2) {
    // constant ones box: column 0 of every key row is 1 (128B swizzle: the row's first 16-byte
    // chunk sits at position row & 7), all else 0
    for (int i = tid - 64; i < kBox / 4; i += C::kThreads - 64) {
      const int row = i >> 5, w = i & 31;
      reinterpret_cast<uint32_t*>(sOnes)[i] = (w == ((row & 7) << 2)) ? 0x00003F80u : 0u;
    }
    fence_proxy_async_smem();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_s;
  grid_dep_wait();
  grid_dep_launch();

  // Every role walks the same items and keeps the same running counters: nk = K tiles so far
  // (slot nk % KS, phase nk / KS), nv likewise for V, na = items so far (accumulator na & 1).
  if (warp == 0) {
    if (elect_one()) {
      uint32_t nk = 0, nv = 0;
      bool ok = true;
      const uint64_t pol = l2_policy_evict_first();
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
        const SelfItem it = self_item(p, item);
        for (int j = 0; j < it.nC && ok; ++j) {
          const int n0 = (it.c_begin + j) * 128;
          const uint32_t sk = nk % KS, sv = nv % VS;
          if (nk >= KS && !mbar_wait(&k_free[sk], ((nk / KS) + 1) & 1, p.status, 700)) { ok = false; break; }
          mbar_arrive_expect_tx(&k_full[sk], C::kTile);
          for (int x = 0; x < D / 64; ++x)
            tma_load_4d_hint(sK + sk * C::kTile + x * kBox, &mk, &k_full[sk], x * 64, n0, kId ? it.hl : it.h, it.b, pol);
          ++nk;
          if (nv >= VS && !mbar_wait(&v_free[sv], ((nv / VS) + 1) & 1, p.status, 701)) { ok = false; break; }
          mbar_arrive_expect_tx(&v_full[sv], C::kTile);
          for (int x = 0; x < D / 64; ++x)
            tma_load_4d_hint(sm + C::v_off(sv) + x * C::v_lbo(sv), &mv, &v_full[sv], x * 64, n0, it.h, it.b, pol);
          ++nv;
        }
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      constexpr uint32_t id_s = umma_idesc_bf16(128, C::kAcc, true, true);  // [S | z] += Kc^T [V | 1]
      constexpr uint32_t kLboA = (D == 128) ? kBox : 0;                     // D=64: rows 64..127 mirror 0..63
      uint32_t nk = 0, nv = 0, na = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x, ++na) {
        const SelfItem it = self_item(p, item);
        const uint32_t acc = tmem + (na & 1) * C::kAcc;
        // the accumulator's previous sum has left TMEM
        if (na >= 2 && !mbar_wait(&acc_free[na & 1], ((na >> 1) + 1) & 1, p.status, 710)) break;
        for (int j = 0; j < it.nC; ++j) {
          const uint32_t sk = nk % KS, sv = nv % VS;
          if (!mbar_wait(kId ? &k_full[sk] : &kphi[sk], (nk / KS) & 1, p.status, 711) ||
              !mbar_wait(&v_full[sv], (nv / VS) & 1, p.status, 712)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          const uint64_t dk = umma_smem_desc(smem_u32(sK) + sk * C::kTile, kLboA, 1024),
                         dv = umma_smem_desc(smem_u32(sm) + C::v_off(sv), C::v_lbo(sv), 1024);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            umma_ss(acc, umma_desc_add(dk, ks * 2048), umma_desc_add(dv, ks * 2048), id_s, (j > 0) || (ks > 0));
          umma_commit(&k_free[sk]);
          umma_commit(&v_free[sv]);
          ++nk;
          ++nv;
        }
        if (!ok) break;
        umma_commit(&acc_done[na & 1]);
      }
    }
  } else if (warp < 6) {
    // drain: one thread per feature row writes the segment's sums to its scratch slot
    const int quarter = warp & 3, r = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    uint32_t na = 0;
    for (int item = blockIdx.x; item < p.nitems; item += gridDim.x, ++na) {
      const SelfItem it = self_item(p, item);
      if (!mbar_wait(&acc_done[na & 1], (na >> 1) & 1, p.status, 720)) break;
      tc_fence_after_sync();
      const uint32_t acc = tmem + (na & 1) * C::kAcc + lane_off;
      float* dst = p.partial + (long long)item * (D * D + D);
#pragma unroll 1
      for (int cc = 0; cc < D / 32; ++cc) {
        uint32_t v[32];
        tmem_ld32(acc + cc * 32, v);
        tmem_wait_ld();
        if (r < D) {
#pragma unroll
          for (int jj = 0; jj < 32; jj += 4)
            *reinterpret_cast<float4*>(dst + (long long)r * D + cc * 32 + jj) =
                make_float4(__uint_as_float(v[jj]), __uint_as_float(v[jj + 1]), __uint_as_float(v[jj + 2]),
                            __uint_as_float(v[jj + 3]));
        }
      }
      const uint32_t zc = tmem_ld1(acc + D);
      tmem_wait_ld();
      if (r < D) dst[D * D + r] = __uint_as_float(zc);
      tc_fence_before_sync();
      mbar_arrive(&acc_free[na & 1]);
      __syncwarp();
      if (lane == 0) count_up(p.summed + it.chain);
    }
  } else if (!kId) {
    // phi on the K tiles, in place, by 16 warps (features given: a tile is ready as it lands, rows past the end of the
    // sequence filled with zeros by the copy)
    const int tt = tid - 6 * 32;
    uint32_t nk = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
      const SelfItem it = self_item(p, item);
      for (int j = 0; j < it.nC; ++j) {
        const uint32_t sk = nk % KS;
        ok = ok && mbar_wait(&k_full[sk], (nk / KS) & 1, p.status, 730);
        if (ok) transform_k_tile<D, 512>(sK + sk * C::kTile, tt, p.N - (it.c_begin + j) * 128);
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(&kphi[sk]);
        ++nk;
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------ sum
// total[chain] = sum over the chain's segments, in segment order (deterministic).  It is launched behind the windowed heads
// and runs beside them: they leave 4096 registers of an SM, room for one block of 64 threads.  Eight loads in flight per
// thread (one after the other, and with the device to itself, it took 6 us for 26 chains of 11 segments at d = 128).
__global__ void __launch_bounds__(kSumThreads, 16)
linear_self_sum_kernel(const SelfParams p, int state_floats) {
  constexpr int kAhead = 8;
  grid_dep_launch();
  __shared__ int ready;
  const int chain = blockIdx.y;
  if (threadIdx.x == 0) ready = wait_count(p.summed + chain, 4u * p.G, p.status, 790);
  __syncthreads();
  const int i = (blockIdx.x * kSumThreads + threadIdx.x) * 4;
  if (ready && i < state_floats) {
    const float* src = p.partial + (long long)chain * p.G * state_floats + i;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int g0 = 0; g0 < p.G; g0 += kAhead) {
      float4 x[kAhead];
#pragma unroll
      for (int e = 0; e < kAhead; ++e)
        x[e] = g0 + e < p.G ? __ldcg(reinterpret_cast<const float4*>(src + (long long)(g0 + e) * state_floats))
                          : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int e = 0; e < kAhead; ++e) {
        acc.x += x[e].x;
        acc.y += x[e].y;
        acc.z += x[e].z;
        acc.w += x[e].w;
      }
    }
    *reinterpret_cast<float4*>(p.total + (long long)chain * state_floats + i) = acc;
  }
  __syncthreads();
  if (threadIdx.x == 0 && ready) count_up(p.totalled + chain);
  if (blockIdx.x + blockIdx.y == 0) grid_dep_wait();
}

// ------------------------------------------------------------------------------------ readout
template <int D>
struct OutCfg {
  static constexpr int kTile = 128 * D * 2;
  static constexpr int kSbBox = D * 128;  // one D-row x 64-column box of the B operand
  static constexpr int kQ = 0;            // two raw Q tiles
  static constexpr int kSb = 2 * kTile;   // bf16 totals [D rows][D columns] in 64-column boxes ...
  static constexpr int kZb = kSb + D * D * 2;  // ... followed by one more box: columns 0, 1 = hi(z), lo(z)
  static constexpr int kStage = kZb + kSbBox;  // two output tiles staged for the TMA store
  // One CTA per SM, also at d = 64, where the tiles take 81 KB: its launch comes early, and CTAs that found room beside another
  // one's (of either kernel: both take all of the tensor memory) waited for it while other SMs stood idle (160 chains of 4096
  // tokens with random features: 74 us, 43 with this).
  static constexpr int kTiles = kStage + 2 * kTile + 1024, kBytes = kTiles > 120 * 1024 ? kTiles : 120 * 1024;
  static constexpr int kAcc = D + 16;
  static constexpr uint32_t tQ = 0, tO = D;  // phi(Q): 2 x D/2 columns; O | den: 2 x (D + 16)
  static constexpr int kThreads = 15 * 32;
};

template <int D, bool kId>
__global__ void __launch_bounds__(OutCfg<D>::kThreads, 1)
linear_self_readout_kernel(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mo,
                           const SelfParams p) {
  using C = OutCfg<D>;
  extern __shared__ uint8_t raw_smem[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw_smem) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = sm + C::kQ;
  uint8_t* sSb = sm + C::kSb;
  uint8_t* sZb = sm + C::kZb;
  uint8_t* sStage = sm + C::kStage;
  __shared__ __align__(8) uint64_t q_full[2], q_free[2], qphi_full[2], tq_free[2], o_full[2], o_free[2], sb_ready,
      o_staged[2], stage_free[2];
  __shared__ uint32_t tmem_base_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&q_full[i], 1);
      mbar_init(&q_free[i], 8);
      mbar_init(&qphi_full[i], 8);
      mbar_init(&tq_free[i], 1);
      mbar_init(&o_full[i], 1);
      mbar_init(&o_free[i], 128);
    }
    mbar_init(&sb_ready, 128);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&o_staged[i], 128);
      mbar_init(&stage_free[i], 1);
    }
    mbar_fence_init();
    tma_prefetch_desc(&mq);
    tma_prefetch_desc(&mo);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base_s, 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_s;

  // Running counters shared by all roles: nq = chunks so far (Q slot, phi(Q) slot and O buffer
  // nq & 1, phase nq >> 1; staging buffer phase nq), ni = items so far.
  if (warp == 0) {
    if (elect_one()) {
      uint32_t nq = 0;
      bool ok = true;
      const uint64_t pol = l2_policy_evict_first();
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
        const SelfItem it = self_item(p, item);
        for (int j = 0; j < it.nC; ++j, ++nq) {
          const uint32_t s = nq & 1;
          if (nq >= 2 && !mbar_wait(&q_free[s], ((nq >> 1) + 1) & 1, p.status, 800)) { ok = false; break; }
          mbar_arrive_expect_tx(&q_full[s], C::kTile);
          for (int x = 0; x < D / 64; ++x)
            tma_load_4d_hint(sQ + s * C::kTile + x * kBox, &mq, &q_full[s], x * 64, (it.c_begin + j) * 128, kId ? it.hl : it.h, it.b,
                             pol);
        }
      }
      grid_dep_launch();
    }
  } else if (warp == 1) {
    if (elect_one()) {
      constexpr uint32_t id_o = umma_idesc_bf16(128, C::kAcc, false, true);  // [O | den] = Qc [Sb | Zb]
      uint32_t nq = 0, ni = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x, ++ni) {
        const SelfItem it = self_item(p, item);
        if (!mbar_wait(&sb_ready, ni & 1, p.status, 810)) break;  // this item's totals are in shared memory
        for (int j = 0; j < it.nC; ++j, ++nq) {
          const uint32_t s = nq & 1;
          if (!mbar_wait(&qphi_full[s], (nq >> 1) & 1, p.status, 811) ||
              (nq >= 2 && !mbar_wait(&o_free[s], ((nq >> 1) + 1) & 1, p.status, 812))) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          const uint32_t tq = tmem + C::tQ + s * (D / 2), to = tmem + C::tO + s * C::kAcc;
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks)
            umma_ts(to, tq + ks * 8, umma_smem_desc(smem_u32(sSb) + ks * 2048, C::kSbBox, 1024), id_o, ks > 0);
          umma_commit(&o_full[s]);
          umma_commit(&tq_free[s]);
        }
      }
    }
  } else if (warp < 6) {
    // epilogue warps (one thread per row): load the chain's totals as the B operand at the start of an
    // item; per chunk divide the numerators by the denominator and stage the tile
    const int quarter = warp & 3, r = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const bool s_row = r < D;
    uint32_t nq = 0, ni = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x, ++ni) {
      const SelfItem it = self_item(p, item);
      if (lane == 0)
        ok = p.totals_of_one ? wait_count(p.summed + it.chain, 4u, p.status, 823)
                             : wait_count(p.totalled + it.chain, p.sum_blocks, p.status, 822);
      if (__any_sync(0xffffffffu, !ok)) break;
      __syncwarp();  // (a vote orders no memory)
      // (the previous item's last product has completed: its o_full was seen below)
      if (s_row) {
        const float* src = p.total + (long long)it.chain * (D * D + D);
#pragma unroll 1
        for (int cc = 0; cc < D / 32; ++cc) {
          float4 in[8];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) in[jj] = __ldcg(reinterpret_cast<const float4*>(src + (long long)r * D + cc * 32) + jj);
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            uint4 val;
            val.x = pack_bf16(in[2 * g].x, in[2 * g].y);
            val.y = pack_bf16(in[2 * g].z, in[2 * g].w);
            val.z = pack_bf16(in[2 * g + 1].x, in[2 * g + 1].y);
            val.w = pack_bf16(in[2 * g + 1].z, in[2 * g + 1].w);
            *reinterpret_cast<uint4*>(sSb + (cc >> 1) * C::kSbBox + swz128_offset(r, (cc & 1) * 32 + g * 8)) = val;
          }
        }
        const float z = __ldcg(src + D * D + r);
        const float hi = __bfloat162float(__float2bfloat16_rn(z));
        // row r of the extra box: columns 0, 1 = hi(z), lo(z); the other 14 columns the product reads are zero
        uint4 zrow[2] = {make_uint4(pack_bf16(hi, z - hi), 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
        *reinterpret_cast<uint4*>(sZb + swz128_offset(r, 0)) = zrow[0];
        *reinterpret_cast<uint4*>(sZb + swz128_offset(r, 8)) = zrow[1];
      }
      fence_proxy_async_smem();
      mbar_arrive(&sb_ready);
      for (int j = 0; j < it.nC; ++j, ++nq) {
        const uint32_t s = nq & 1;
        if (!mbar_wait(&o_full[s], (nq >> 1) & 1, p.status, 820) ||
            (nq >= 2 && !mbar_wait(&stage_free[s], ((nq >> 1) + 1) & 1, p.status, 821))) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        const uint32_t to = tmem + C::tO + s * C::kAcc + lane_off;
        uint32_t den_hi, den_lo;
        tmem_ld2(to + D, den_hi, den_lo);
        tmem_wait_ld();
        const float inv = 1.f / (__uint_as_float(den_hi) + __uint_as_float(den_lo));
#pragma unroll 1
        for (int cc = 0; cc < D / 32; ++cc) {
          uint32_t v[32];
          tmem_ld32(to + cc * 32, v);
          tmem_wait_ld();
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            uint4 val;
            val.x = pack_bf16(__uint_as_float(v[8 * g + 0]) * inv, __uint_as_float(v[8 * g + 1]) * inv);
            val.y = pack_bf16(__uint_as_float(v[8 * g + 2]) * inv, __uint_as_float(v[8 * g + 3]) * inv);
            val.z = pack_bf16(__uint_as_float(v[8 * g + 4]) * inv, __uint_as_float(v[8 * g + 5]) * inv);
            val.w = pack_bf16(__uint_as_float(v[8 * g + 6]) * inv, __uint_as_float(v[8 * g + 7]) * inv);
            *reinterpret_cast<uint4*>(sStage + s * C::kTile + (cc >> 1) * kBox + swz128_offset(r, (cc & 1) * 32 + g * 8)) = val;
          }
        }
        tc_fence_before_sync();
        mbar_arrive(&o_free[s]);
        fence_proxy_async_smem();
        mbar_arrive(&o_staged[s]);
      }
    }
  } else if (warp < 14) {
    // phi(Q): thread = (row, half of the head dimension); the result is the A operand in TMEM
    const int quarter = warp & 3, half = ((warp - 6) >> 2) & 1, r = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    constexpr int kChunks = D / 16;  // 16-byte chunks of one row half
    uint32_t nq = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
      const SelfItem it = self_item(p, item);
      for (int j = 0; j < it.nC && ok; ++j, ++nq) {
        const uint32_t s = nq & 1;
        ok = mbar_wait(&q_full[s], (nq >> 1) & 1, p.status, 830);
        uint32_t pk[kChunks * 4];
        if (ok) {
#pragma unroll
          for (int g = 0; g < kChunks; ++g) {
            const int gl = half * kChunks + g, box = gl >> 3, cin = gl & 7;
            const uint4 rawv = *reinterpret_cast<const uint4*>(sQ + s * C::kTile + box * kBox + r * 128 +
                                                               ((cin ^ (r & 7)) << 4));
            pk[g * 4 + 0] = rawv.x;
            pk[g * 4 + 1] = rawv.y;
            pk[g * 4 + 2] = rawv.z;
            pk[g * 4 + 3] = rawv.w;
          }
        }
        // the buffer goes back to the TMA engine: these reads (generic proxy) must be ordered before its
        // next write (async proxy), which a barrier arrival alone does not do
        __threadfence_block();
        fence_proxy_async_smem();
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(&q_free[s]);  // this warp has its part of the raw tile in registers
        if (ok) {
#pragma unroll
          for (int w = 0; w < kChunks * 4; ++w) pk[w] = phi_sel<kId>(pk[w]);
          if (nq >= 2) ok = mbar_wait(&tq_free[s], ((nq >> 1) + 1) & 1, p.status, 831);
        }
        tc_fence_after_sync();
        if (ok) {
          if constexpr (D == 128) {
            uint32_t(&pk32)[32] = *reinterpret_cast<uint32_t(*)[32]>(pk);
            tmem_st32(tmem + C::tQ + s * (D / 2) + lane_off + half * 32, pk32);
          } else {
            tmem_st16(tmem + C::tQ + s * (D / 2) + lane_off + half * 16, pk);
          }
          tmem_wait_st();
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&qphi_full[s]);
        }
        ok = !__any_sync(0xffffffffu, !ok);
      }
    }
  } else {
    // TMA stores of the staged output tiles
    if (elect_one()) {
      uint32_t nq = 0;
      bool ok = true;
      const uint64_t pol = l2_policy_evict_first();
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
        const SelfItem it = self_item(p, item);
        for (int j = 0; j < it.nC; ++j, ++nq) {
          const uint32_t s = nq & 1;
          if (!mbar_wait(&o_staged[s], (nq >> 1) & 1, p.status, 840)) { ok = false; break; }
          for (int x = 0; x < D / 64; ++x)
            tma_store_4d_hint(&mo, sStage + s * C::kTile + x * kBox, x * 64, (it.c_begin + j) * 128, it.h, it.b, pol);
          tma_store_commit();
          // the other buffer's store (the previous chunk's) has read its tile: hand that buffer back
          if (nq >= 1) {
            tma_store_wait_read<1>();
            mbar_arrive(&stage_free[s ^ 1]);
          }
        }
      }
      tma_store_wait_all<0>();
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
  if (blockIdx.x == 0) grid_dep_wait();
}

// ------------------------------------------------------------------------------------ whole
// Both halves in one CTA, D = 64: the sums of a chain never leave the SM.  Warps: 0 K/V producer, 1 issuer of the
// sums, 2-5 epilogue, 6-13 phi(Q), 14-21 phi(K), 22 Q producer, 23 issuer of the readout, 24-25 totals from TMEM into
// the bf16 B operand (D = 64 feature rows: TMEM lane quarters 0 and 1), 26 output stores.  Accumulators, totals, Q,
// phi(Q), O and staging are all double-buffered, so the two halves run side by side, a chain apart.
// What bounds it is the memory system, as in the kernels above, but a chain's start-up and its totals are hidden
// behind the chain before: 640 chains of 197 tokens take 20.5 us, in three launches 46.5 (16, 6 and 24: the totals of
// an item are loaded when it begins, which for items of two chunks is most of their time).
struct WholeCfg {
  static constexpr int D = 64, kTile = 128 * D * 2;
  static constexpr int kVSlots = 4, kKSlots = 3;  // V0 V1 V2 V3 ONES, as in RedCfg<64>
  static constexpr int kOnes = 4 * kBox, kK = 5 * kBox, kQ = kK + kKSlots * kTile;
  static constexpr int kSb = kQ + 2 * kTile;      // two times [64 rows][64 columns] of totals + the box of hi(z), lo(z)
  static constexpr int kSbBox = D * 128, kSbSlot = 2 * kSbBox;
  static constexpr int kStage = kSb + 2 * kSbSlot;
  static constexpr int kBytes = kStage + 2 * kTile + 1024;
  static constexpr int kAcc = D + 16;
  static constexpr uint32_t tAcc = 0, tQ = 2 * kAcc, tO = tQ + D;  // two accumulators, two phi(Q), two O
  static constexpr int kThreads = 27 * 32;
};

template <bool kId>
__global__ void __launch_bounds__(WholeCfg::kThreads, 1)
linear_self_whole_kernel(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mk,
                         const __grid_constant__ CUtensorMap mv, const __grid_constant__ CUtensorMap mo,
                         const SelfParams p) {
  using C = WholeCfg;
  constexpr int D = C::D, VS = C::kVSlots, KS = C::kKSlots;
  extern __shared__ uint8_t raw_smem[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw_smem) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t k_full[KS], kphi[KS], k_free[KS], v_full[VS], v_free[VS], acc_done[2], acc_free[2],
      q_full[2], q_free[2], qphi_full[2], tq_free[2], o_full[2], o_free[2], sb_ready[2], sb_free[2], o_staged[2],
      stage_free[2];
  __shared__ uint32_t tmem_base_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int i = 0; i < KS; ++i) {
      mbar_init(&k_full[i], 1);
      mbar_init(&kphi[i], 8);
      mbar_init(&k_free[i], 1);
    }
    for (int i = 0; i < VS; ++i) {
      mbar_init(&v_full[i], 1);
      mbar_init(&v_free[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_done[i], 1);
      mbar_init(&acc_free[i], 2);
      mbar_init(&q_full[i], 1);
      mbar_init(&q_free[i], 8);
      mbar_init(&qphi_full[i], 8);
      mbar_init(&tq_free[i], 1);
      mbar_init(&o_full[i], 1);
      mbar_init(&o_free[i], 128);
      mbar_init(&sb_ready[i], 64);
      mbar_init(&sb_free[i], 1);
      mbar_init(&o_staged[i], 128);
      mbar_init(&stage_free[i], 1);
    }
    mbar_fence_init();
    tma_prefetch_desc(&mq);
    tma_prefetch_desc(&mk);
    tma_prefetch_desc(&mv);
    tma_prefetch_desc(&mo);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base_s, 512);
    tmem_relinquish();
  } else if (warp >= 2) {
    // constant ones box, as in the reduce kernel
    for (int i = tid - 64; i < kBox / 4; i += C::kThreads - 64) {
      const int row = i >> 5, w = i & 31;
      reinterpret_cast<uint32_t*>(sm + C::kOnes)[i] = (w == ((row & 7) << 2)) ? 0x00003F80u : 0u;
    }
    fence_proxy_async_smem();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_base_s;
  grid_dep_wait();
  if (p.let_go == kAtStart) grid_dep_launch();

  // Every role walks the chains blockIdx.x, blockIdx.x + gridDim.x, ... (an item is a whole chain) and keeps the same
  // running counters: n = chunks so far, c = chains so far.
  if (warp == 0 || warp == 22) {
    if (elect_one()) {
      const bool kv = warp == 0;
      const uint64_t pol = l2_policy_evict_first();
      uint32_t n = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
        const SelfItem it = self_item(p, item);
        for (int j = 0; j < it.nC; ++j, ++n) {
          if (kv) {
            const uint32_t sk = n % KS, sv = n % VS;
            if (n >= KS && !mbar_wait(&k_free[sk], ((n / KS) + 1) & 1, p.status, 900)) { ok = false; break; }
            mbar_arrive_expect_tx(&k_full[sk], C::kTile);
            tma_load_4d_hint(sm + C::kK + sk * C::kTile, &mk, &k_full[sk], 0, j * 128, kId ? it.hl : it.h, it.b, pol);
            if (n >= VS && !mbar_wait(&v_free[sv], ((n / VS) + 1) & 1, p.status, 901)) { ok = false; break; }
            mbar_arrive_expect_tx(&v_full[sv], C::kTile);
            tma_load_4d_hint(sm + sv * kBox, &mv, &v_full[sv], 0, j * 128, it.h, it.b, pol);
          } else {
            const uint32_t s = n & 1;
            if (n >= 2 && !mbar_wait(&q_free[s], ((n >> 1) + 1) & 1, p.status, 902)) { ok = false; break; }
            mbar_arrive_expect_tx(&q_full[s], C::kTile);
            tma_load_4d_hint(sm + C::kQ + s * C::kTile, &mq, &q_full[s], 0, j * 128, kId ? it.hl : it.h, it.b, pol);
          }
        }
      }
      if (!kv && p.let_go == kAtEnd) grid_dep_launch();
    }
  } else if (warp == 1) {
    if (elect_one()) {
      constexpr uint32_t id_s = umma_idesc_bf16(128, C::kAcc, true, true);  // [S | z] += Kc^T [V | 1]
      uint32_t n = 0, c = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x, ++c) {
        const SelfItem it = self_item(p, item);
        const uint32_t acc = tmem + C::tAcc + (c & 1) * C::kAcc;
        if (c >= 2 && !mbar_wait(&acc_free[c & 1], ((c >> 1) + 1) & 1, p.status, 910)) break;
        for (int j = 0; j < it.nC; ++j, ++n) {
          const uint32_t sk = n % KS, sv = n % VS;
          if (!mbar_wait(kId ? &k_full[sk] : &kphi[sk], (n / KS) & 1, p.status, 911) ||
              !mbar_wait(&v_full[sv], (n / VS) & 1, p.status, 912)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          const uint64_t dk = umma_smem_desc(smem_u32(sm) + C::kK + sk * C::kTile, 0, 1024),
                         dv = umma_smem_desc(smem_u32(sm) + sv * kBox, (4 - sv) * kBox, 1024);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)  // (rows 64..127 of the product mirror 0..63)
            umma_ss(acc, umma_desc_add(dk, ks * 2048), umma_desc_add(dv, ks * 2048), id_s, (j > 0) || (ks > 0));
          umma_commit(&k_free[sk]);
          umma_commit(&v_free[sv]);
        }
        if (!ok) break;
        umma_commit(&acc_done[c & 1]);
      }
    }
  } else if (warp == 23) {
    if (elect_one()) {
      constexpr uint32_t id_o = umma_idesc_bf16(128, C::kAcc, false, true);  // [O | den] = Qc [Sb | Zb]
      uint32_t n = 0, c = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x, ++c) {
        const SelfItem it = self_item(p, item);
        if (!mbar_wait(&sb_ready[c & 1], (c >> 1) & 1, p.status, 920)) break;
        const uint32_t sb = smem_u32(sm) + C::kSb + (c & 1) * C::kSbSlot;
        for (int j = 0; j < it.nC; ++j, ++n) {
          const uint32_t s = n & 1;
          if (!mbar_wait(&qphi_full[s], (n >> 1) & 1, p.status, 921) ||
              (n >= 2 && !mbar_wait(&o_free[s], ((n >> 1) + 1) & 1, p.status, 922))) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          const uint32_t tq = tmem + C::tQ + s * (D / 2), to = tmem + C::tO + s * C::kAcc;
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks)
            umma_ts(to, tq + ks * 8, umma_smem_desc(sb + ks * 2048, C::kSbBox, 1024), id_o, ks > 0);
          umma_commit(&o_full[s]);
          umma_commit(&tq_free[s]);
        }
        if (!ok) break;
        umma_commit(&sb_free[c & 1]);
      }
    }
  } else if (warp < 6) {
    // epilogue: one thread per row
    const int quarter = warp & 3, r = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    uint32_t n = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
      for (int j = 0; j < p.nch; ++j, ++n) {
        const uint32_t s = n & 1;
        if (!mbar_wait(&o_full[s], (n >> 1) & 1, p.status, 930) ||
            (n >= 2 && !mbar_wait(&stage_free[s], ((n >> 1) + 1) & 1, p.status, 931))) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        const uint32_t to = tmem + C::tO + s * C::kAcc + lane_off;
        uint32_t den_hi, den_lo;
        tmem_ld2(to + D, den_hi, den_lo);
        tmem_wait_ld();
        const float inv = 1.f / (__uint_as_float(den_hi) + __uint_as_float(den_lo));
#pragma unroll 1
        for (int cc = 0; cc < D / 32; ++cc) {
          uint32_t v[32];
          tmem_ld32(to + cc * 32, v);
          tmem_wait_ld();
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            uint4 val;
            val.x = pack_bf16(__uint_as_float(v[8 * g + 0]) * inv, __uint_as_float(v[8 * g + 1]) * inv);
            val.y = pack_bf16(__uint_as_float(v[8 * g + 2]) * inv, __uint_as_float(v[8 * g + 3]) * inv);
            val.z = pack_bf16(__uint_as_float(v[8 * g + 4]) * inv, __uint_as_float(v[8 * g + 5]) * inv);
            val.w = pack_bf16(__uint_as_float(v[8 * g + 6]) * inv, __uint_as_float(v[8 * g + 7]) * inv);
            *reinterpret_cast<uint4*>(sm + C::kStage + s * C::kTile + swz128_offset(r, cc * 32 + g * 8)) = val;
          }
        }
        tc_fence_before_sync();
        mbar_arrive(&o_free[s]);
        fence_proxy_async_smem();
        mbar_arrive(&o_staged[s]);
      }
    }
  } else if (warp < 14) {
    // phi(Q): thread = (row, half of the head dimension); the result is the A operand in TMEM
    const int quarter = warp & 3, half = ((warp - 6) >> 2) & 1, r = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    constexpr int kChunks = D / 16;  // 16-byte chunks of one row half
    uint32_t n = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
      for (int j = 0; j < p.nch && ok; ++j, ++n) {
        const uint32_t s = n & 1;
        ok = mbar_wait(&q_full[s], (n >> 1) & 1, p.status, 940);
        uint32_t pk[kChunks * 4];
        if (ok) {
#pragma unroll
          for (int g = 0; g < kChunks; ++g) {
            const int cin = half * kChunks + g;
            const uint4 rawv =
                *reinterpret_cast<const uint4*>(sm + C::kQ + s * C::kTile + r * 128 + ((cin ^ (r & 7)) << 4));
            pk[g * 4 + 0] = rawv.x;
            pk[g * 4 + 1] = rawv.y;
            pk[g * 4 + 2] = rawv.z;
            pk[g * 4 + 3] = rawv.w;
          }
        }
        // the buffer goes back to the TMA engine: these reads (generic proxy) must be ordered before its
        // next write (async proxy), which a barrier arrival alone does not do
        __threadfence_block();
        fence_proxy_async_smem();
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(&q_free[s]);
        if (ok) {
#pragma unroll
          for (int w = 0; w < kChunks * 4; ++w) pk[w] = phi_sel<kId>(pk[w]);
          if (n >= 2) ok = mbar_wait(&tq_free[s], ((n >> 1) + 1) & 1, p.status, 941);
        }
        tc_fence_after_sync();
        if (ok) {
          tmem_st16(tmem + C::tQ + s * (D / 2) + lane_off + half * 16, pk);
          tmem_wait_st();
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&qphi_full[s]);
        }
        ok = !__any_sync(0xffffffffu, !ok);
      }
    }
  } else if (warp < 22) {
    if constexpr (!kId) {  // phi on the K tiles, in place (features given: a tile is ready as it lands)
    uint32_t n = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
      for (int j = 0; j < p.nch; ++j, ++n) {
        const uint32_t sk = n % KS;
        ok = ok && mbar_wait(&k_full[sk], (n / KS) & 1, p.status, 950);
        if (ok) transform_k_tile<D, 256>(sm + C::kK + sk * C::kTile, tid - 14 * 32, p.N - j * 128);
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(&kphi[sk]);
      }
    }
    }
  } else if (warp < 26) {
    // totals: one thread per feature row
    const int quarter = warp & 3, r = quarter * 32 + lane;  // 0..63
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    uint32_t c = 0;
    for (int item = blockIdx.x; item < p.nitems; item += gridDim.x, ++c) {
      const uint32_t s = c & 1;
      bool ok = mbar_wait(&acc_done[s], (c >> 1) & 1, p.status, 960) &&
                (c < 2 || mbar_wait(&sb_free[s], ((c >> 1) + 1) & 1, p.status, 961));
      if (__any_sync(0xffffffffu, !ok)) break;
      tc_fence_after_sync();
      const uint32_t acc = tmem + C::tAcc + s * C::kAcc + lane_off;
      uint8_t* sb = sm + C::kSb + s * C::kSbSlot;
#pragma unroll 1
      for (int cc = 0; cc < D / 32; ++cc) {
        uint32_t v[32];
        tmem_ld32(acc + cc * 32, v);
        tmem_wait_ld();
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint4 val;
          val.x = pack_bf16(__uint_as_float(v[8 * g + 0]), __uint_as_float(v[8 * g + 1]));
          val.y = pack_bf16(__uint_as_float(v[8 * g + 2]), __uint_as_float(v[8 * g + 3]));
          val.z = pack_bf16(__uint_as_float(v[8 * g + 4]), __uint_as_float(v[8 * g + 5]));
          val.w = pack_bf16(__uint_as_float(v[8 * g + 6]), __uint_as_float(v[8 * g + 7]));
          *reinterpret_cast<uint4*>(sb + swz128_offset(r, cc * 32 + g * 8)) = val;
        }
      }
      const float z = __uint_as_float(tmem_ld1(acc + D));
      tmem_wait_ld();
      const float hi = __bfloat162float(__float2bfloat16_rn(z));
      // row r of the box behind: columns 0, 1 = hi(z), lo(z); the other 14 columns the product reads are zero
      *reinterpret_cast<uint4*>(sb + C::kSbBox + swz128_offset(r, 0)) = make_uint4(pack_bf16(hi, z - hi), 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(sb + C::kSbBox + swz128_offset(r, 8)) = make_uint4(0u, 0u, 0u, 0u);
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_free[s]);
      fence_proxy_async_smem();
      mbar_arrive(&sb_ready[s]);
    }
  } else {
    // TMA stores of the staged output tiles
    if (elect_one()) {
      uint32_t n = 0;
      bool ok = true;
      const uint64_t pol = l2_policy_evict_first();
      for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
        const SelfItem it = self_item(p, item);
        for (int j = 0; j < it.nC; ++j, ++n) {
          const uint32_t s = n & 1;
          if (!mbar_wait(&o_staged[s], (n >> 1) & 1, p.status, 970)) { ok = false; break; }
          tma_store_4d_hint(&mo, sm + C::kStage + s * C::kTile, 0, j * 128, it.h, it.b, pol);
          tma_store_commit();
          tma_store_wait_read<0>();
          mbar_arrive(&stage_free[s]);
        }
      }
      tma_store_wait_all<0>();
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}
// Segments per chain.  CTAs take items (segments) round-robin, so a launch lasts ceil(items / CTAs)
// rounds of one item each: among the segment counts that keep segments at least four chunks long
// (and the scratch within 64 slots per chain, more when the chains are few), take the one with the least rounds x (chunks of the
// longest segment + about one chunk of fixed cost per item).  The plan must not depend on the
// device that is current when the workspace size is asked for: it assumes the 148 SMs of a B200.
int self_segments(int nchains, int nch) {
  constexpr int kPlanSMs = 148;
  int g_max = (nch + 3) / 4;
  int cap = (2 * kPlanSMs + nchains - 1) / nchains;  // few chains: as many segments as fill two rounds
  if (cap < 64) cap = 64;
  if (g_max > cap) g_max = cap;
  int best_g = 1;
  long long best = -1;
  for (int g = 1; g <= g_max; ++g) {
    const long long rounds = ((long long)nchains * g + kPlanSMs - 1) / kPlanSMs;
    const long long cost = rounds * ((nch + g - 1) / g + 1);
    if (best < 0 || cost < best) {
      best = cost;
      best_g = g;
    }
  }
  return best_g;
}

// Segments that the sums are formed in, at most self_segments.  Where windowed heads run behind the first launch (beside_us)
// they fill the SMs that it leaves idle, so that only what they do not fill counts, in microseconds, beside the work itself; more segments
// are more slots to add up, beside the windowed heads at 0.7 TB/s.
int self_sum_segments(int nchains, int nch, int d, int sms, double beside_us) {
  const int g_max = self_segments(nchains, nch);
  if (beside_us <= 0.0) return g_max;
  const double chunk_us = d == 128 ? 1.5 : 0.8, state = ((double)d * d + d) * sizeof(float);
  int best_g = 1;
  double best = 1e300;
  for (int g = 1; g <= g_max; ++g) {
    const double rounds = (double)(((long long)nchains * g + sms - 1) / sms);
    const double work = nchains * (double)(nch + g) / sms * chunk_us, span = rounds * ((nch + g - 1) / g + 1) * chunk_us;
    const double idle = span - work - beside_us, sum = g > 1 ? 1.0 + nchains * g * state / 0.7e6 - 0.7 * beside_us : 0.0;
    const double cost = work + (idle > 0.0 ? idle : 0.0) + (g > 1 ? (sum > 1.0 ? sum : 1.0) : 0.0);
    if (cost < best) {
      best = cost;
      best_g = g;
    }
  }
  return best_g;
}

// Whether whole chains go through linear_self_whole_kernel, by estimates of both forms in microseconds, within 8 % of what was
// measured over 20 to 640 chains of 1024 to 8192 tokens.
// Whole: while a CTA reads one chain out it sums up its next, so R rounds of chains are R + 1 phases of nch chunks each; a chunk
// takes 0.72 where few CTAs are at work, 0.92 where each has one chain in hand and 1.5, HBM's pace, where each has two.
// Three launches: 1.83 a chunk of both passes, spread evenly, with one more chunk per segment, and 10 for their starts;
// behind a pre-pass of random features 5 more and 0.15 a chunk.
// Windowed heads add what they take of the whole device (beside_us); behind whole chains less what the SMs without a chain in the
// last round leave idle, and up to 8 for coming late.
// us, whole | three: where the rule takes whole chains 128 of 1024 tokens 20.5 | 30.8, 160 of 2048 48.2 | 50.5, 300 of 2048 69.7 |
// 77.2, 448 of 4096 187 | 210, with windowed heads of w = 128 160 of 4096 96.7 | 106, 320 of 4096 166 | 204; where it takes three
// launches 40 of 1536 22.4 | 17.6, 100 of 4096 55.6 | 53.4, 160 of 4096 90.5 | 76.4, 220 of 8192 192 | 186.
bool self_whole(int nchains, int nch, int d, int sms, double beside_us, bool features) {
  if (d != WholeCfg::D) return false;
  const int rounds = (nchains + sms - 1) / sms, last = nchains - (rounds - 1) * sms;
  auto chunk_us = [&](int streams) {  // (chains being summed up and chains being read out)
    const double x = (double)streams / sms;
    return x <= 1.0 ? 0.72 + 0.2 * x * x : 0.92 + 0.58 * (x - 1.0);
  };
  double whole = 5.0 + 2.0 * nch * chunk_us(last);
  if (rounds > 1) whole = 5.0 + nch * (chunk_us(sms) + (rounds - 2) * chunk_us(2 * sms) + chunk_us(sms + last) + chunk_us(last));
  const double work = (double)nchains * (nch + self_segments(nchains, nch)) / sms;
  const double three = 10.0 + 1.83 * work + (features ? 5.0 + 0.15 * work : 0.0);
  const double idle = (1.0 - (double)last / sms) * nch * chunk_us(last) * (rounds > 1 ? 1 : 2), late = 0.4 * beside_us;
  return whole + (beside_us > idle ? beside_us - idle : 0.0) + (late < 8.0 ? late : 8.0) <= three + beside_us;
}

}  // namespace

// Counters at the start of the scratch, cleared by the caller with the workspace header.
size_t linear_self_count_bytes(int nchains) { return ((size_t)nchains * 2 * sizeof(unsigned int) + 255) & ~(size_t)255; }

size_t linear_self_workspace_bytes(int nchains, int N, int d) {
  const int nch = (N + 127) / 128;
  const size_t state = ((size_t)d * d + d) * sizeof(float);
  const int G = self_segments(nchains, nch);
  // One segment: its sum is the total, and the counters take less than the room that totals would (what fits the fixed
  // scratch of the allocation-free call depends on this: 252 chains of up to 512 tokens, d = 64).
  if (G == 1) return 2 * (size_t)nchains * state;
  return linear_self_count_bytes(nchains) + (size_t)nchains * (G + 1) * state;
}

cudaError_t launch_linear_self_tc(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                                  int layout, int h_begin, int h_count, WsHeader* ws, size_t scratch_offset,
                                  cudaStream_t stream, const std::function<cudaError_t(LetGo)>& beside, double beside_us, const void* fq,
                                  const void* fk) {
  if (h_count <= 0) return beside(kAtEnd);
  // fq, fk: feature tensors [B, h_count, N, d] that stand in for Q and K (feature map: identity);
  // their heads are counted from the first linear one
  const bool features = fq != nullptr;
  CUtensorMap mq, mk, mv, mo;
  if (features ? (!make_qkv_tensor_map(&mq, fq, B, h_count, N, d, GF_BHND, 128) ||
                  !make_qkv_tensor_map(&mk, fk, B, h_count, N, d, GF_BHND, 128))
               : (!make_qkv_tensor_map(&mq, q, B, H, N, d, layout, 128) ||
                  !make_qkv_tensor_map(&mk, k, B, H, N, d, layout, 128)))
    return cudaErrorInvalidValue;
  if (!make_qkv_tensor_map(&mv, v, B, H, N, d, layout, 128) || !make_qkv_tensor_map(&mo, o, B, H, N, d, layout, 128))
    return cudaErrorInvalidValue;
  SelfParams p;
  p.N = N;
  p.nch = (N + 127) / 128;
  p.h_begin = h_begin;
  p.h_count = h_count;
  p.nchains = B * h_count;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = device_info(&dev, &sms)) != cudaSuccess) return e;
  const bool whole = self_whole(p.nchains, p.nch, d, sms, beside_us, features);
  auto cut = [&](int G) {
    p.G = G;
    p.seg_base = p.nch / G;
    p.seg_rem = p.nch % G;
    p.nitems = p.nchains * G;
    return dim3(p.nitems < sms ? p.nitems : sms);
  };
  dim3 grid = cut(whole ? 1 : self_sum_segments(p.nchains, p.nch, d, sms, beside_us));
  const int state_floats = d * d + d;
  uint8_t* scratch = reinterpret_cast<uint8_t*>(ws) + scratch_offset;
  p.summed = reinterpret_cast<unsigned int*>(scratch);
  p.totalled = p.summed + p.nchains;
  p.sum_blocks = (unsigned)((state_floats / 4 + kSumThreads - 1) / kSumThreads);
  p.partial = reinterpret_cast<float*>(scratch + linear_self_count_bytes(p.nchains));
  p.total = p.G == 1 ? p.partial : p.partial + (size_t)p.nitems * state_floats;  // one segment: its sum is the total
  p.status = &ws->status;
  p.let_go = h_begin > 0 ? kAtStart : kAtEnd;  // (the windowed heads, where there are any, run beside it)
  if (whole) {
    auto kern = features ? linear_self_whole_kernel<true> : linear_self_whole_kernel<false>;
    if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), dev, WholeCfg::kBytes)) != cudaSuccess) return e;
    e = launch_link(kern, grid, dim3(WholeCfg::kThreads), WholeCfg::kBytes, stream, mq, mk, mv, mo, p);
    return e == cudaSuccess ? beside(kAtEnd) : e;
  }
  auto launch_red = [&](auto kern, int smem, int threads) -> cudaError_t {
    cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), dev, smem);
    if (err != cudaSuccess) return err;
    return launch_link(kern, grid, dim3(threads), smem, stream, mk, mv, p);
  };
  auto launch_out = [&](auto kern, int smem, int threads) -> cudaError_t {
    cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), dev, smem);
    if (err != cudaSuccess) return err;
    return launch_link(kern, grid, dim3(threads), smem, stream, mq, mo, p);
  };
  if (features)
    e = (d == 64) ? launch_red(linear_self_reduce_kernel<64, true>, RedCfg<64>::kBytes, RedCfg<64>::kThreads)
                  : launch_red(linear_self_reduce_kernel<128, true>, RedCfg<128>::kBytes, RedCfg<128>::kThreads);
  else
    e = (d == 64) ? launch_red(linear_self_reduce_kernel<64, false>, RedCfg<64>::kBytes, RedCfg<64>::kThreads)
                  : launch_red(linear_self_reduce_kernel<128, false>, RedCfg<128>::kBytes, RedCfg<128>::kThreads);
  if (e != cudaSuccess) return e;
  // The windowed heads between the two: they start on the SMs that the first kernel leaves, and the readout on those that they
  // leave.
  if ((e = beside(kAtStart)) != cudaSuccess) return e;
  if (p.G > 1 && (e = launch_link(linear_self_sum_kernel, dim3(p.sum_blocks, p.nchains), dim3(kSumThreads), 0, stream, p,
                                  state_floats)) != cudaSuccess)
    return e;
  p.totals_of_one = p.G == 1;
  grid = cut(self_segments(p.nchains, p.nch));  // (the readout goes by the segments that fill the device best by themselves)
  if (features)
    return (d == 64) ? launch_out(linear_self_readout_kernel<64, true>, OutCfg<64>::kBytes, OutCfg<64>::kThreads)
                     : launch_out(linear_self_readout_kernel<128, true>, OutCfg<128>::kBytes, OutCfg<128>::kThreads);
  return (d == 64) ? launch_out(linear_self_readout_kernel<64, false>, OutCfg<64>::kBytes, OutCfg<64>::kThreads)
                   : launch_out(linear_self_readout_kernel<128, false>, OutCfg<128>::kBytes, OutCfg<128>::kThreads);
}

}  // namespace gf
