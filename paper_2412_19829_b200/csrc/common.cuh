// Shared declarations of the libgformer CUDA sources (host-side launch interfaces and a
// few device helpers).  Not part of the public ABI.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <functional>

#include "gformer.h"
#include "host_state.h"

namespace gf {

// Element strides of a logical [B, H, N, d] tensor (innermost stride is 1).
struct Strides {
  long long b, h, n;
};

inline Strides make_strides(int layout, int H, int N, int d) {
  Strides s;
  if (layout == GF_BNHD) {
    s.b = (long long)N * H * d;
    s.n = (long long)H * d;
    s.h = d;
  } else {
    s.b = (long long)H * N * d;
    s.h = (long long)N * d;
    s.n = d;
  }
  return s;
}

// Layout of the first bytes of the caller's workspace.
struct WsHeader {
  unsigned int status;   // 0 = fine, else a code written by a kernel whose bounded wait expired
  unsigned int where;    // which wait gave up (diagnostic)
  unsigned int ticket;   // work counter of the persistent kernels
  unsigned int wait_kcycles;  // limit of every bounded wait in units of 1024 cycles; 0 = default (about 2 s)
  unsigned int drop_flag;     // failure injection for tests: the linear kernel skips the flag of segment n - 1
  unsigned int pad[59];
};
static_assert(sizeof(WsHeader) == 256, "workspace header is 256 bytes");

// Counts kernel launches (reported by gformer_launch_count).
void note_launch(int n = 1);

// ---- The kernels of a stream as a chain of programmatic dependent launches.
//
// A kernel of the chain is launched as soon as every CTA of the kernel before it has started and has called
// grid_dep_launch() (or has ended), and its CTAs are placed wherever an SM has room for them.  Two kinds of link:
//   kAfter   the kernel reads what the one before it writes, or is the first of its call: its CTAs set themselves up, then
//            grid_dep_wait(), which returns when all kernels before it are complete
//   kBeside  it depends on nothing that the kernel before it does, only on what that one had itself waited for before it
//            let go of its dependents.  It starts at once, on the SMs that are free or become so.  One of its CTAs waits
//            before it ends, so that what follows the call in the stream follows all of its kernels.
// The last kernel of a call lets go when its CTAs run out of work: the next call's CTAs, which only wait, would otherwise fill the
// SMs unevenly (8 x 32 heads decoding, d = 128, 12.3 us a step launched the ordinary way, 19.5 let go at the start, 9.9 at the end).
// Launched the ordinary way kernels of a few microseconds also start on a grid of about 2 us (8.2, 10.2, 12.3 us a call).
enum Link { kAfter, kBeside };
// When the kernels that have a choice let go: as soon as they have waited themselves; when the kernel before them is complete
// (what follows kBeside needs what that one writes); at the end of their work (the last of a call).
enum LetGo { kAtStart, kWhenPreviousDone, kAtEnd };
template <typename... P, typename... A>
cudaError_t launch_link_clusters(int cluster /* CTAs along x; 1: none */, void (*kern)(P...), dim3 grid, dim3 block,
                                 size_t smem, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2] = {};
  attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cluster;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
  if (e != cudaSuccess) return e;
  note_launch();
  return cudaGetLastError();
}
template <typename... P, typename... A>
cudaError_t launch_link(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
  return launch_link_clusters(1, kern, grid, block, smem, stream, args...);
}

// What a kernel that does not use the workspace has to know of its place in its call.
struct Place {
  uint4* ws;  // its first kernel (kAfter) writes the workspace header, all zero but for the test knobs; null: kBeside
  unsigned int wait_kcycles, drop_flag;
  int last;   // nothing of the call follows
};

// Writes the header and zeroes the rest of the first `bytes` bytes (a multiple of 16) of a workspace: the first launch of a
// call whose kernels use it.
cudaError_t launch_clear_ws(Place place, size_t bytes, cudaStream_t stream);

// ---- fp32 arithmetic (split tf32 products by mma.sync, or FFMA): any w, d in {64,128}, f32 or bf16 storage.
// Heads [h_begin, h_begin + h_count) of the [B, H, N, d] tensors are processed.
// fwd: keys after the query it may see: 0 = the causal window, w - 1 = the two-sided window |i - j| < w.
cudaError_t launch_window_simt(const void* q, const void* k, const void* v, void* o, int B, int N, int d,
                               int w, int fwd, float scale, int dtype, Strides st, int h_begin, int h_count,
                               cudaStream_t stream, Place place);
// S_io/z_io: [B, h_count, d, d] / [B, h_count, d] or null.  zero_init: ignore their contents on entry.
// global_sum: the unmasked linear attention of the bidirectional layer (sum over all tokens, then readout).
cudaError_t launch_linear_simt(const void* q, const void* k, const void* v, void* o, int B, int N, int d,
                               int dtype, Strides st, int h_begin, int h_count, float* S_io, float* z_io,
                               bool zero_init, cudaStream_t stream, Place place, bool global_sum = false,
                               const void* W = nullptr /* [h_count, d, d] storage dtype: positive random features */);
// The causal heads with phi = elu + 1: register-tiled blocks of 32 tokens (launch_linear_simt comes here by itself).
cudaError_t launch_linear_tiled(const void* q, const void* k, const void* v, void* o, int B, int N, int d, int dtype,
                                Strides st, int h_begin, int h_count, float* S_io, float* z_io, bool zero_init,
                                cudaStream_t stream, Place place);
// The causal layer with phi = elu + 1: heads [0, h_sparse) windowed, the h_lin behind them linear from a zero state (their
// final one goes to S_io, z_io unless null); one launch for both where that is not slower.
cudaError_t launch_layer_tiled(const void* q, const void* k, const void* v, void* o, int B, int N, int d, int w, float scale,
                               int dtype, Strides st, int h_sparse, int h_lin, float* S_io, float* z_io, cudaStream_t stream,
                               Place place);
bool export_ring_fits(int B, int N, int d, int w, int dtype, int h_sparse);
cudaError_t launch_export_ring(const void* k, const void* v, void* k_cache, void* v_cache, int B, int N, int d,
                               int w, int dtype, Strides st, int h_sparse, cudaStream_t stream);  // kBeside
// t_seq == nullptr: every sequence is at position t; else sequence b is at t_seq[b] (device array,
// negative = idle slot, otherwise below 2^48) and the kernel itself moves the positions on.
cudaError_t launch_decode_step(const void* q, const void* k, const void* v, void* o, void* k_cache,
                               void* v_cache, float* S, float* z, long long t, long long* t_seq, int B, int H,
                               int d, int w, int h_sparse, float scale, int dtype, cudaStream_t stream,
                               const void* W = nullptr /* [H - h_sparse, d, d] storage dtype */);

// The current device and its SM count (asked of the driver once per device).
cudaError_t device_info(int* dev, int* sms);

// ---- tensor-core (tcgen05 / TMEM / TMA) path: bf16 storage, d in {64,128}.
bool tc_window_supported(int N, int d, int w, int dtype);
bool tc_linear_supported(int N, int d, int dtype);
cudaError_t launch_window_tc(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                             int w, int fwd, float scale, int layout, int h_begin, int h_count, WsHeader* ws,
                             cudaStream_t stream, Link link, LetGo let_go);
// Global (unmasked) linear attention of the bidirectional layer, heads [h_begin, h_begin + h_count): one launch, or three
// (segment sums, totals, readout), kAfter the kernel before them; its scratch starts scratch_offset bytes into ws, with
// linear_self_count_bytes that must be zero.  beside() launches, kBeside, what is to run between the first launch and
// the others (the windowed heads), and takes about beside_us microseconds of the whole device.
size_t linear_self_count_bytes(int nchains);
size_t linear_self_workspace_bytes(int nchains, int N, int d);
cudaError_t launch_linear_self_tc(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                                  int layout, int h_begin, int h_count, WsHeader* ws, size_t scratch_offset,
                                  cudaStream_t stream, const std::function<cudaError_t(LetGo)>& beside, double beside_us,
                                  const void* fq = nullptr,
                                  const void* fk = nullptr);
// Segmentation used by the tensor-core linear kernel (split: 0 = automatic, else chunks per segment;
// ctas: CTAs the kernel will run with, 0 = one per SM of a B200) and the scratch it needs beyond
// the workspace header (sized for the largest segment count the plan may pick for any ctas).
void linear_tc_plan(int nchains, int N, int d, int split, int ctas, int* chunks_per_segment, int* segments_per_chain);
// The same plan with its two parts named: the first *whole_chains chains are left whole, the others cut
// (with somewhat more chains than CTAs the full rounds go whole and the leftover chains are cut, in a
// second launch); *whole_chains = nchains and one segment per chain when nothing is cut.
// shared: other kernels run beside this one and fill the SMs a thin round of whole chains leaves idle.
void linear_tc_plan_parts(int nchains, int N, int d, int split, int ctas, int* whole_chains, int* chunks_per_segment,
                          int* segments_per_chain, bool shared = false);
size_t linear_tc_workspace_bytes(int nchains, int N, int d, int split);
// Bytes at the start of that scratch (right after the workspace header) that must be zero when the
// kernel starts: the hand-over flags.  The caller clears them (together with the header).
size_t linear_tc_flag_bytes(int nchains, int N, int split);
cudaError_t launch_linear_tc(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                             int layout, int h_begin, int h_count, float* S_io, float* z_io, bool zero_init,
                             int split, int max_ctas, WsHeader* ws, cudaStream_t stream, Link link, LetGo let_go, bool shared = false,
                             const void* fq = nullptr, const void* fk = nullptr);
// Positive random features phi_W of Q and K of heads [h_begin, h_begin + h_count) (bf16 storage) into the
// contiguous bf16 tensors fq, fk [B, h_count, N, d]; W: [h_count, d, d] bf16, row a of a head's matrix is
// its projection vector w_a.  With fq, fk given, the two linear-attention launchers read them in place
// of Q and K and leave their own feature map out.
cudaError_t launch_favor_features_tc(const void* q, const void* k, const void* W, void* fq, void* fk, int B, int H,
                                     int N, int d, int layout, int h_begin, int h_count, WsHeader* ws,
                                     cudaStream_t stream);  // kAfter

// ---- device helpers
// All kernels before this one in the stream are complete and what they wrote can be read.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The kernel that follows in the stream may be launched once every CTA of this one has said so.
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void begin(const Place& place) {
  static_assert(offsetof(WsHeader, wait_kcycles) == 12 && offsetof(WsHeader, drop_flag) == 16, "what is written here");
  if (place.ws != nullptr) {
    grid_dep_wait();
    if (blockIdx.x + blockIdx.y + blockIdx.z == 0 && threadIdx.x < sizeof(WsHeader) / 16) {
      uint4 x = make_uint4(0u, 0u, 0u, 0u);
      if (threadIdx.x == 0) x.w = place.wait_kcycles;
      if (threadIdx.x == 1) x.x = place.drop_flag;
      place.ws[threadIdx.x] = x;
    }
  }
  if (!place.last) grid_dep_launch();
}

// Cycles a bounded wait may take; `status` points at the first word of the workspace header.
__device__ __forceinline__ long long wait_limit_cycles(const unsigned int* status) {
  const unsigned int kc = reinterpret_cast<const volatile unsigned int*>(status)[3];
  return kc ? (long long)kc * 1024 : 4000000000LL;
}

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}

// phi(x) = elu(x) + 1 (Sec. II-B), without a branch: max(x, 0) + exp(min(x, 0)), and NaN of a NaN (a selection, because
// fminf drops it).
__device__ __forceinline__ float phi_elu1(float x) { return fmaxf(x, 0.f) + expf(x > 0.f ? 0.f : x); }

}  // namespace gf
