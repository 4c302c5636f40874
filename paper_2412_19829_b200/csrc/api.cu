// C ABI of libgformer: argument validation, path selection and launches.
#include <math.h>
#include <stdint.h>

#include <atomic>

#include "common.cuh"

namespace gf {
static std::atomic<unsigned long long> g_launches{0};
void note_launch(int n) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }
}  // namespace gf

namespace {

using gf::Strides;
using gf::WsHeader;

// Process-wide knobs (gformer_set_tuning).  An entry point takes one snapshot when it is called
// and works from that, so a knob changed by another thread meanwhile cannot make the parts of one
// call disagree (the cleared flag bytes, the plan, the launch).
std::atomic<int> g_force_simt{0}, g_linear_split{0}, g_linear_ctas{0}, g_wait_kcycles{0}, g_drop_flag{0};
struct Tuning {
  int force_simt, linear_split, linear_ctas, wait_kcycles, drop_flag;
};
Tuning tuning_now() {
  Tuning t;
  t.force_simt = g_force_simt.load(std::memory_order_relaxed);
  t.linear_split = g_linear_split.load(std::memory_order_relaxed);
  t.linear_ctas = g_linear_ctas.load(std::memory_order_relaxed);
  t.wait_kcycles = g_wait_kcycles.load(std::memory_order_relaxed);
  t.drop_flag = g_drop_flag.load(std::memory_order_relaxed);
  return t;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool overlaps(const void* a, const void* b, size_t bytes) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
  return x < y + bytes && y < x + bytes;
}

size_t elem_size(int dtype) { return dtype == GF_F32 ? 4 : 2; }

int check_common(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d, int dtype,
                 int layout) {
  if (!q || !k || !v || !o) return GF_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o)) return GF_ERR_INVALID_ARG;
  if (B < 1 || H < 1 || N < 1 || d < 1) return GF_ERR_INVALID_ARG;
  if (dtype != GF_F32 && dtype != GF_BF16) return GF_ERR_INVALID_ARG;
  if (layout != GF_BHND && layout != GF_BNHD) return GF_ERR_INVALID_ARG;
  if (d != 64 && d != 128) return GF_ERR_UNSUPPORTED;
  if ((long long)B * H > 65535LL * 65535LL || B > 65535 || H > 65535) return GF_ERR_UNSUPPORTED;
  const size_t bytes = (size_t)B * H * N * d * elem_size(dtype);
  if (overlaps(o, q, bytes) || overlaps(o, k, bytes) || overlaps(o, v, bytes)) return GF_ERR_INVALID_ARG;
  return GF_OK;
}

int check_ws(void* ws, size_t ws_bytes, size_t need) {
  if (!ws || ws_bytes < need) return GF_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return GF_ERR_INVALID_ARG;
  return GF_OK;
}

int cuda_status(cudaError_t e) { return e == cudaSuccess ? GF_OK : GF_ERR_CUDA; }

// Window heads [h_begin, h_begin+h_count) on `stream`.
int run_window(const Tuning& tn, const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d, int w,
               float scale, int dtype, int layout, int h_begin, int h_count, WsHeader* ws,
               cudaStream_t stream, gf::Link link, gf::LetGo let_go, bool two_sided = false, gf::Place place = {}) {
  if (h_count <= 0) return GF_OK;
  const int w_eff = w > N ? N : w;  // keys before token 0 (or after the last one) do not exist
  const int fwd = two_sided ? w_eff - 1 : 0;
  if (!tn.force_simt && gf::tc_window_supported(N, d, w_eff, dtype))
    return cuda_status(
        gf::launch_window_tc(q, k, v, o, B, H, N, d, w_eff, fwd, scale, layout, h_begin, h_count, ws, stream, link, let_go));
  return cuda_status(gf::launch_window_simt(q, k, v, o, B, N, d, w_eff, fwd, scale, dtype,
                                            gf::make_strides(layout, H, N, d), h_begin, h_count, stream, place));
}

// Feature map of the linear heads of one call: elu + 1 (W null), or positive random features under
// the projections W [h_count, d, d].  On the tensor-core path those are computed first, into the two
// feature tensors at the end of the workspace (feat_offset bytes in): fq, fk once run_features has launched that.
struct Phi {
  const void* W = nullptr;
  size_t feat_offset = 0;
  void *fq = nullptr, *fk = nullptr;
};

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
size_t feature_bytes(int B, int h_lin, int N, int d) { return align256((size_t)B * h_lin * N * d * 2); }

int check_phi(int phi, const void* W) {
  if (phi == GF_PHI_ELU1) return W == nullptr ? GF_OK : GF_ERR_INVALID_ARG;
  if (phi == GF_PHI_FAVOR_POS) return (W != nullptr && aligned16(W)) ? GF_OK : GF_ERR_INVALID_ARG;
  return GF_ERR_UNSUPPORTED;
}

// The pre-pass of the positive random features.
int run_features(const Tuning& tn, const void* q, const void* k, int B, int H, int N, int d, int dtype, int layout,
                 int h_begin, int h_count, WsHeader* ws, cudaStream_t stream, Phi* phi) {
  if (h_count <= 0 || phi->W == nullptr || tn.force_simt || !gf::tc_linear_supported(N, d, dtype)) return GF_OK;
  phi->fq = reinterpret_cast<uint8_t*>(ws) + phi->feat_offset;
  phi->fk = reinterpret_cast<uint8_t*>(phi->fq) + feature_bytes(B, h_count, N, d);
  return cuda_status(gf::launch_favor_features_tc(q, k, phi->W, phi->fq, phi->fk, B, H, N, d, layout, h_begin, h_count, ws,
                                                  stream));
}

int run_linear(const Tuning& tn, const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d, int dtype,
               int layout, int h_begin, int h_count, float* S_io, float* z_io, bool zero_init, int max_ctas,
               WsHeader* ws, cudaStream_t stream, gf::Link link, gf::LetGo let_go, bool shared = false, const Phi& phi = Phi(), gf::Place place = {}) {
  if (h_count <= 0) return GF_OK;
  if (!tn.force_simt && gf::tc_linear_supported(N, d, dtype)) {
    return cuda_status(gf::launch_linear_tc(q, k, v, o, B, H, N, d, layout, h_begin, h_count, S_io, z_io,
                                            zero_init, tn.linear_split, max_ctas, ws, stream, link, let_go, shared, phi.fq, phi.fk));
  }
  return cuda_status(gf::launch_linear_simt(q, k, v, o, B, N, d, dtype, gf::make_strides(layout, H, N, d),
                                            h_begin, h_count, S_io, z_io, zero_init, stream, place, false, phi.W));
}

// The first launch of the calls whose kernels use the workspace: writes its header and zeroes the flags or counters of a
// linear kernel behind it.  What follows in the call's chain of kernels (launch_link) runs kAfter it or, behind one that is
// kAfter it, kBeside that.  The kernels that use no workspace (fp32 arithmetic) have the first of them write the header.
// A memset and two streams with events for the two head groups, which this chain replaced, took 11 driver calls for a layer
// instead of three and left the device idle for 2 to 4 us behind the memset and again at the end: 64 x 12 heads of 197 tokens
// (d = 64, both directions) 33.0 -> 26.7 us, 8 x 12 of 2048 34.0 -> 32.7, 1 x 32 of 32 768 (d = 128, w = 512) 343 -> 336.
gf::Place first_of_call(const Tuning& tn, void* ws, bool last) {
  return {(uint4*)ws, (unsigned int)tn.wait_kcycles, (unsigned int)tn.drop_flag, last};
}
constexpr gf::Place kLastOfCall = {nullptr, 0, 0, 1};
int clear_ws(const Tuning& tn, void* ws, cudaStream_t stream, size_t flag_bytes = 0) {
  return cuda_status(gf::launch_clear_ws(first_of_call(tn, ws, false), sizeof(WsHeader) + flag_bytes, stream));
}

// How the tensor-core kernel of the causal linear heads will run a call's chains: max_ctas as for launch_linear_tc, bytes of
// flags, the order among cut-chain calls entered where there are any.
int plan_linear(const Tuning& tn, int chains, int N, int d, int dtype, bool shared, cudaStream_t stream, int* max_ctas,
                size_t* flag_bytes, gf::CutChainOrder* order) {
  *max_ctas = 0;
  *flag_bytes = 0;
  if (chains <= 0 || tn.force_simt || !gf::tc_linear_supported(N, d, dtype)) return GF_OK;
  int L = 0, G = 0, whole = 0, dev = 0, sms = 0;
  if (gf::device_info(&dev, &sms) != cudaSuccess) return GF_ERR_CUDA;
  if (shared && tn.linear_ctas > 0 && tn.linear_ctas < sms) {
    gf::linear_tc_plan_parts(chains, N, d, tn.linear_split, 0, &whole, &L, &G, true);
    // (leaving SMs to the windowed heads from the start only makes sense where there is work for every SM)
    if ((long long)chains * (whole > 0 ? 1 : G) >= sms) *max_ctas = sms = tn.linear_ctas;
  }
  gf::linear_tc_plan_parts(chains, N, d, tn.linear_split, sms, &whole, &L, &G, shared);
  if (whole == chains) return GF_OK;  // (whole chains hand nothing on)
  *flag_bytes = gf::linear_tc_flag_bytes(chains, N, tn.linear_split);
  return cuda_status(order->enter(dev, stream));
}

size_t workspace_bytes(const Tuning& tn, int B, int H, int N, int d, int h_sparse, int dtype, int phi = GF_PHI_ELU1,
                       size_t* feat_offset = nullptr);

}  // namespace

extern "C" {

const char* gformer_status_string(int status) {
  switch (status) {
    case GF_OK: return "ok";
    case GF_ERR_INVALID_ARG: return "invalid argument";
    case GF_ERR_UNSUPPORTED: return "unsupported configuration";
    case GF_ERR_WORKSPACE: return "workspace missing or too small";
    case GF_ERR_CUDA: return "CUDA error";
    case GF_ERR_TIMEOUT: return "device-side wait timed out";
    default: return "unknown status";
  }
}

int gformer_version(void) { return 100; }

unsigned long long gformer_launch_count(void) { return gf::g_launches.load(std::memory_order_relaxed); }

int gformer_default_h_sparse(int H) {
  if (H < 1) return 0;
  int h0 = (int)floor(3.0 * H / 16.0 + 0.5);
  if (h0 < 1) h0 = 1;
  if (h0 > H) h0 = H;
  return h0;
}

int gformer_set_tuning(int key, int value) {
  switch (key) {
    case GF_TUNE_FORCE_SIMT:
      g_force_simt.store(value ? 1 : 0);
      return GF_OK;
    case GF_TUNE_WAIT_KCYCLES:
      if (value < 0) return GF_ERR_INVALID_ARG;
      g_wait_kcycles.store(value);
      return GF_OK;
    case GF_TUNE_TEST_DROP_FLAG:
      if (value < 0) return GF_ERR_INVALID_ARG;
      g_drop_flag.store(value);
      return GF_OK;
    case GF_TUNE_LINEAR_SPLIT:
      if (value < -1 || value > 4096) return GF_ERR_INVALID_ARG;
      g_linear_split.store(value);
      return GF_OK;
    case GF_TUNE_LINEAR_CTAS:
      if (value < 0 || value > 65535) return GF_ERR_INVALID_ARG;
      g_linear_ctas.store(value);
      return GF_OK;
    default:
      return GF_ERR_INVALID_ARG;
  }
}

int gformer_linear_plan(int chains, int N, int d, int ctas, int* segments, int* chunks_per_segment) {
  if (chains < 1 || N < 1 || ctas < 0 || segments == nullptr || chunks_per_segment == nullptr) return GF_ERR_INVALID_ARG;
  if (!gf::tc_linear_supported(N, d, GF_BF16)) return GF_ERR_UNSUPPORTED;
  gf::linear_tc_plan(chains, N, d, g_linear_split.load(), ctas, chunks_per_segment, segments);
  return GF_OK;
}

int gformer_linear_plan_parts(int chains, int N, int d, int ctas, int* whole_chains, int* segments,
                              int* chunks_per_segment) {
  if (chains < 1 || N < 1 || ctas < 0 || whole_chains == nullptr || segments == nullptr || chunks_per_segment == nullptr)
    return GF_ERR_INVALID_ARG;
  if (!gf::tc_linear_supported(N, d, GF_BF16)) return GF_ERR_UNSUPPORTED;
  gf::linear_tc_plan_parts(chains, N, d, g_linear_split.load(), ctas, whole_chains, chunks_per_segment, segments);
  return GF_OK;
}

size_t gformer_workspace_bytes(int B, int H, int N, int d, int w, int h_sparse, int dtype) {
  (void)w;
  return workspace_bytes(tuning_now(), B, H, N, d, h_sparse, dtype);
}

size_t gformer_workspace_bytes_phi(int B, int H, int N, int d, int w, int h_sparse, int dtype, int phi) {
  (void)w;
  return workspace_bytes(tuning_now(), B, H, N, d, h_sparse, dtype, phi);
}
}  // extern "C"

namespace {
size_t workspace_bytes(const Tuning& tn, int B, int H, int N, int d, int h_sparse, int dtype, int phi,
                       size_t* feat_offset) {
  size_t bytes = sizeof(WsHeader);
  if (feat_offset) *feat_offset = 0;
  if (B < 1 || H < 1 || N < 1) return bytes;
  if (h_sparse < 0) h_sparse = gformer_default_h_sparse(H);
  if (h_sparse > H) h_sparse = H;
  const int h_lin = H - h_sparse;
  if (h_lin > 0 && !tn.force_simt && gf::tc_linear_supported(N, d, dtype)) {
    // the causal kernel's hand-over scratch, or the bidirectional layer's segment sums: whichever is larger
    const size_t causal = gf::linear_tc_workspace_bytes(B * h_lin, N, d, tn.linear_split);
    const size_t self = gf::linear_self_workspace_bytes(B * h_lin, N, d);
    bytes += causal > self ? causal : self;
    if (phi == GF_PHI_FAVOR_POS) {  // the features of Q and K of the linear heads, behind everything else
      bytes = align256(bytes);
      if (feat_offset) *feat_offset = bytes;
      bytes += 2 * feature_bytes(B, h_lin, N, d);
    }
  }
  return bytes;
}
}  // namespace

extern "C" {

int gformer_last_device_status(void* ws, void* cuda_stream) {
  if (!ws) return GF_ERR_INVALID_ARG;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  WsHeader hdr;
  if (cudaMemcpyAsync(&hdr, ws, sizeof(hdr), cudaMemcpyDeviceToHost, stream) != cudaSuccess) return GF_ERR_CUDA;
  if (cudaStreamSynchronize(stream) != cudaSuccess) return GF_ERR_CUDA;
  return hdr.status == 0 ? GF_OK : GF_ERR_TIMEOUT;
}

int gformer_window_attn(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d, int w,
                        float scale, int dtype, int layout, void* ws, size_t ws_bytes, void* cuda_stream) {
  int rc = check_common(q, k, v, o, B, H, N, d, dtype, layout);
  if (rc != GF_OK) return rc;
  const Tuning tn = tuning_now();
  if (w < 1) return GF_ERR_INVALID_ARG;
  rc = check_ws(ws, ws_bytes, workspace_bytes(tn, B, H, N, d, H, dtype));
  if (rc != GF_OK) return rc;
  if (!(scale > 0.f)) scale = 1.0f / sqrtf((float)d);
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  const bool tc = !tn.force_simt && gf::tc_window_supported(N, d, w, dtype);
  if (tc && (rc = clear_ws(tn, ws, stream)) != GF_OK) return rc;
  return run_window(tn, q, k, v, o, B, H, N, d, w, scale, dtype, layout, 0, H, (WsHeader*)ws, stream, gf::kAfter, gf::kAtEnd,
                    false, first_of_call(tn, ws, true));
}

int gformer_window_attn_self(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                             int w, float scale, int dtype, int layout, void* ws, size_t ws_bytes,
                             void* cuda_stream) {
  int rc = check_common(q, k, v, o, B, H, N, d, dtype, layout);
  if (rc != GF_OK) return rc;
  const Tuning tn = tuning_now();
  if (w < 1) return GF_ERR_INVALID_ARG;
  rc = check_ws(ws, ws_bytes, workspace_bytes(tn, B, H, N, d, H, dtype));
  if (rc != GF_OK) return rc;
  if (!(scale > 0.f)) scale = 1.0f / sqrtf((float)d);
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  const bool tc = !tn.force_simt && gf::tc_window_supported(N, d, w, dtype);
  if (tc && (rc = clear_ws(tn, ws, stream)) != GF_OK) return rc;
  return run_window(tn, q, k, v, o, B, H, N, d, w, scale, dtype, layout, 0, H, (WsHeader*)ws, stream, gf::kAfter, gf::kAtEnd,
                    true, first_of_call(tn, ws, true));
}

int gformer_hybrid_attn_self(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                             int w, int h_sparse, float scale, int phi, int dtype, int layout, void* ws,
                             size_t ws_bytes, void* cuda_stream) {
  if (phi == GF_PHI_FAVOR_POS) return GF_ERR_INVALID_ARG;  // needs its projections: gformer_hybrid_attn_self_w
  return gformer_hybrid_attn_self_w(q, k, v, o, B, H, N, d, w, h_sparse, scale, phi, nullptr, dtype, layout, ws, ws_bytes,
                                    cuda_stream);
}

int gformer_hybrid_attn_self_w(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                               int w, int h_sparse, float scale, int phi, const void* W, int dtype, int layout,
                               void* ws, size_t ws_bytes, void* cuda_stream) {
  int rc = check_common(q, k, v, o, B, H, N, d, dtype, layout);
  if (rc != GF_OK) return rc;
  const Tuning tn = tuning_now();
  if (w < 1) return GF_ERR_INVALID_ARG;
  if ((rc = check_phi(phi, W)) != GF_OK) return rc;
  size_t feat_offset = 0;
  if (h_sparse < 0) h_sparse = gformer_default_h_sparse(H);
  if (h_sparse > H) return GF_ERR_INVALID_ARG;
  rc = check_ws(ws, ws_bytes, workspace_bytes(tn, B, H, N, d, h_sparse, dtype, phi, &feat_offset));
  if (rc != GF_OK) return rc;
  if (!(scale > 0.f)) scale = 1.0f / sqrtf((float)d);
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  const bool tc_linear = !tn.force_simt && gf::tc_linear_supported(N, d, dtype);
  if (tc_linear && (rc = clear_ws(tn, ws, stream, gf::linear_self_count_bytes(B * (H - h_sparse)))) != GF_OK) return rc;
  Phi fm;
  fm.W = W;
  fm.feat_offset = feat_offset;
  if ((rc = run_features(tn, q, k, B, H, N, d, dtype, layout, h_sparse, H - h_sparse, (WsHeader*)ws, stream, &fm)) != GF_OK)
    return rc;
  if (h_sparse == H)
    return run_window(tn, q, k, v, o, B, H, N, d, w, scale, dtype, layout, 0, H, (WsHeader*)ws, stream, gf::kAfter, gf::kAtEnd,
                      true, first_of_call(tn, ws, true));
  int wrc = GF_OK;  // of the windowed heads: on the SMs that the linear heads leave idle, and between their kernels
  auto window = [&](gf::LetGo let_go) -> cudaError_t {
    if (h_sparse == 0) return cudaSuccess;
    wrc = run_window(tn, q, k, v, o, B, H, N, d, w, scale, dtype, layout, 0, h_sparse, (WsHeader*)ws, stream, gf::kBeside, let_go, true,
                     kLastOfCall);
    return wrc == GF_OK ? cudaSuccess : cudaErrorUnknown;
  };
  if (tc_linear) {
    // (half tiles of 64 keys, 0.6 us each on an SM: tc_window.cu)
    const int tiles = (N + 127) / 128, seen = 2 * (((w < N ? w : N) + 126) / 128) + 1;  // (key tiles that a query tile sees)
    int dev = 0, sms = 0;
    if (gf::device_info(&dev, &sms) != cudaSuccess) return GF_ERR_CUDA;
    const double window_us = 1.0 * B * h_sparse * tiles * (seen < tiles ? seen : tiles) / sms;
    rc = cuda_status(gf::launch_linear_self_tc(q, k, v, o, B, H, N, d, layout, h_sparse, H - h_sparse, (WsHeader*)ws,
                                               sizeof(WsHeader), stream, window, window_us, fm.fq, fm.fk));
  } else {  // fp32 storage (or GF_TUNE_FORCE_SIMT): token by token, a summing sweep and a readout sweep
    rc = cuda_status(gf::launch_linear_simt(q, k, v, o, B, N, d, dtype, gf::make_strides(layout, H, N, d), h_sparse,
                                            H - h_sparse, nullptr, nullptr, true, stream, first_of_call(tn, ws, h_sparse == 0), true, W));
    if (rc == GF_OK) (void)window(gf::kAtEnd);
  }
  return wrc != GF_OK ? wrc : rc;
}

int gformer_causal_linear_attn(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                               int phi, int chunk, float* S_io, float* z_io, int dtype, int layout, void* ws,
                               size_t ws_bytes, void* cuda_stream) {
  if (phi == GF_PHI_FAVOR_POS) return GF_ERR_INVALID_ARG;  // needs its projections: gformer_causal_linear_attn_w
  return gformer_causal_linear_attn_w(q, k, v, o, B, H, N, d, phi, nullptr, chunk, S_io, z_io, dtype, layout, ws,
                                      ws_bytes, cuda_stream);
}

int gformer_causal_linear_attn_w(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d,
                                 int phi, const void* W, int chunk, float* S_io, float* z_io, int dtype, int layout,
                                 void* ws, size_t ws_bytes, void* cuda_stream) {
  int rc = check_common(q, k, v, o, B, H, N, d, dtype, layout);
  if (rc != GF_OK) return rc;
  const Tuning tn = tuning_now();
  if ((rc = check_phi(phi, W)) != GF_OK) return rc;
  Phi fm;
  fm.W = W;
  if (chunk != 0 && chunk != 128) return chunk < 0 || chunk % 64 ? GF_ERR_INVALID_ARG : GF_ERR_UNSUPPORTED;
  if ((S_io == nullptr) != (z_io == nullptr)) return GF_ERR_INVALID_ARG;
  if (S_io && (!aligned16(S_io) || !aligned16(z_io))) return GF_ERR_INVALID_ARG;
  rc = check_ws(ws, ws_bytes, workspace_bytes(tn, B, H, N, d, 0, dtype, phi, &fm.feat_offset));
  if (rc != GF_OK) return rc;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  gf::CutChainOrder order;
  int max_ctas = 0;
  size_t flags = 0;
  if ((rc = plan_linear(tn, B * H, N, d, dtype, false, stream, &max_ctas, &flags, &order)) != GF_OK) return rc;
  const bool tc = !tn.force_simt && gf::tc_linear_supported(N, d, dtype);
  if (tc && (rc = clear_ws(tn, ws, stream, flags)) != GF_OK) return rc;
  if ((rc = run_features(tn, q, k, B, H, N, d, dtype, layout, 0, H, (WsHeader*)ws, stream, &fm)) != GF_OK) return rc;
  if ((rc = run_linear(tn, q, k, v, o, B, H, N, d, dtype, layout, 0, H, S_io, z_io, false, max_ctas, (WsHeader*)ws, stream,
                       gf::kAfter, gf::kAtEnd, false, fm, first_of_call(tn, ws, true))) != GF_OK)
    return rc;
  return cuda_status(order.leave());
}

int gformer_hybrid_attn(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d, int w,
                        int h_sparse, float scale, int phi, int chunk, int dtype, int layout,
                        gf_decode_state* state_out, void* ws, size_t ws_bytes, void* cuda_stream) {
  if (phi == GF_PHI_FAVOR_POS) return GF_ERR_INVALID_ARG;  // needs its projections: gformer_hybrid_attn_w
  return gformer_hybrid_attn_w(q, k, v, o, B, H, N, d, w, h_sparse, scale, phi, nullptr, chunk, dtype, layout, state_out,
                               ws, ws_bytes, cuda_stream);
}

int gformer_hybrid_attn_w(const void* q, const void* k, const void* v, void* o, int B, int H, int N, int d, int w,
                          int h_sparse, float scale, int phi, const void* W, int chunk, int dtype, int layout,
                          gf_decode_state* state_out, void* ws, size_t ws_bytes, void* cuda_stream) {
  int rc = check_common(q, k, v, o, B, H, N, d, dtype, layout);
  if (rc != GF_OK) return rc;
  const Tuning tn = tuning_now();
  if (w < 1) return GF_ERR_INVALID_ARG;
  if ((rc = check_phi(phi, W)) != GF_OK) return rc;
  Phi fm;
  fm.W = W;
  if (chunk != 0 && chunk != 128) return chunk < 0 || chunk % 64 ? GF_ERR_INVALID_ARG : GF_ERR_UNSUPPORTED;
  if (h_sparse < 0) h_sparse = gformer_default_h_sparse(H);
  if (h_sparse > H) return GF_ERR_INVALID_ARG;
  const int h_lin = H - h_sparse;
  if (state_out) {
    gf_decode_state* s = state_out;
    if (s->B != B || s->H != H || s->d != d || s->w != w || s->h_sparse != h_sparse || s->dtype != dtype)
      return GF_ERR_INVALID_ARG;
    if (h_sparse > 0 && (!s->k_cache || !s->v_cache || !aligned16(s->k_cache) || !aligned16(s->v_cache)))
      return GF_ERR_INVALID_ARG;
    if (h_lin > 0 && (!s->S || !s->z || !aligned16(s->S) || !aligned16(s->z))) return GF_ERR_INVALID_ARG;
    if (h_sparse > 0 && !gf::export_ring_fits(B, N, d, w, dtype, h_sparse)) return GF_ERR_CUDA;
  }
  rc = check_ws(ws, ws_bytes, workspace_bytes(tn, B, H, N, d, h_sparse, dtype, phi, &fm.feat_offset));
  if (rc != GF_OK) return rc;
  if (!(scale > 0.f)) scale = 1.0f / sqrtf((float)d);
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  float* S_out = state_out ? state_out->S : nullptr;
  float* z_out = state_out ? state_out->z : nullptr;
  // The two head groups run side by side.  The linear heads (long serial chains, one CTA per SM, which takes all of the
  // SM's shared memory) come first and take every SM that they have work for (leaving some to the windowed heads from the start
  // was no faster and less steady); the windowed heads' CTAs fill the SMs that are free or that linear CTAs leave at different
  // times towards the end.  They are launched when all linear CTAs, which wait for one another, have started.  The export of the
  // ring, which only needs K and V, runs beside the linear heads: its CTAs fit into what those leave of an SM.
  const bool both = h_sparse > 0 && h_lin > 0;
  gf::CutChainOrder order;
  int max_ctas = 0;
  size_t flags = 0;
  if ((rc = plan_linear(tn, B * h_lin, N, d, dtype, both, stream, &max_ctas, &flags, &order)) != GF_OK) return rc;
  const bool tc = !tn.force_simt && gf::tc_linear_supported(N, d, dtype);
  const gf::Strides st = gf::make_strides(layout, H, N, d);
  const bool layer = both && !tc && W == nullptr;  // the fp32-arithmetic kernels take both head groups in one launch
  if (tc && (rc = clear_ws(tn, ws, stream, flags)) != GF_OK) return rc;
  if ((rc = run_features(tn, q, k, B, H, N, d, dtype, layout, h_sparse, h_lin, (WsHeader*)ws, stream, &fm)) != GF_OK) return rc;
  auto linear = [&](gf::Link link, gf::LetGo let_go) {
    return run_linear(tn, q, k, v, o, B, H, N, d, dtype, layout, h_sparse, h_lin, S_out, z_out, true, max_ctas, (WsHeader*)ws,
                      stream, link, let_go, both, fm, first_of_call(tn, ws, let_go == gf::kAtEnd));
  };
  auto window = [&](gf::Link link, gf::LetGo let_go) {
    return run_window(tn, q, k, v, o, B, H, N, d, w, scale, dtype, layout, 0, h_sparse, (WsHeader*)ws, stream, link, let_go, false,
                      h_lin > 0 ? kLastOfCall : first_of_call(tn, ws, let_go == gf::kAtEnd));
  };
  // Behind a pre-pass of random features the windowed heads come first and fill its tail, and the linear heads theirs (us, after
  // the linear heads and ahead of them: 32 heads of 32 768 tokens, d = 128, 461 and 444; 8 x 8 of 3217, d = 64, 62.0 and 57.9;
  // 32 x 12 of 1024 87.8 and 86.1; without features ahead of them is slower, 8 x 12 of 2048 32.6 and 39.6).
  const bool window_first = both && fm.fq != nullptr;
  const bool ring = state_out && h_sparse > 0;
  auto export_ring = [&]() {
    return ring ? cuda_status(gf::launch_export_ring(k, v, state_out->k_cache, state_out->v_cache, B, N, d, w, dtype, st, h_sparse,
                                                     stream))
                : GF_OK;
  };
  if (layer) {
    if ((rc = cuda_status(gf::launch_layer_tiled(q, k, v, o, B, N, d, w < N ? w : N, scale, dtype, st, h_sparse, h_lin, S_out, z_out,
                                                 stream, first_of_call(tn, ws, !ring)))) != GF_OK ||
        (rc = export_ring()) != GF_OK)
      return rc;
  } else if (window_first) {
    // (the windowed heads let go of the linear ones when the features are complete)
    if ((rc = window(gf::kBeside, gf::kWhenPreviousDone)) != GF_OK ||
        (rc = linear(gf::kBeside, ring ? gf::kAtStart : gf::kAtEnd)) != GF_OK || (rc = export_ring()) != GF_OK)
      return rc;
  } else if (h_lin > 0) {
    if ((rc = linear(gf::kAfter, both ? gf::kAtStart : gf::kAtEnd)) != GF_OK || (rc = export_ring()) != GF_OK ||
        (both && (rc = window(gf::kBeside, gf::kAtEnd)) != GF_OK))
      return rc;
  } else {
    // (windowed heads alone wait for the cleared header themselves, and the export runs beside them)
    if ((rc = window(gf::kAfter, ring ? gf::kAtStart : gf::kAtEnd)) != GF_OK || (rc = export_ring()) != GF_OK) return rc;
  }
  if ((rc = cuda_status(order.leave())) != GF_OK) return rc;
  if (state_out) state_out->t = N;
  return GF_OK;
}

static int decode_step_impl(const void* q, const void* k, const void* v, void* o, gf_decode_state* st,
                            long long* t_seq, float scale, int phi, const void* W, void* cuda_stream);

int gformer_decode_step(const void* q, const void* k, const void* v, void* o, gf_decode_state* st, float scale,
                        int phi, void* cuda_stream) {
  if (phi == GF_PHI_FAVOR_POS) return GF_ERR_INVALID_ARG;  // needs its projections: gformer_decode_step_w
  return decode_step_impl(q, k, v, o, st, nullptr, scale, phi, nullptr, cuda_stream);
}

int gformer_decode_step_w(const void* q, const void* k, const void* v, void* o, gf_decode_state* st, float scale,
                          int phi, const void* W, void* cuda_stream) {
  return decode_step_impl(q, k, v, o, st, nullptr, scale, phi, W, cuda_stream);
}

int gformer_decode_step_ragged(const void* q, const void* k, const void* v, void* o, gf_decode_state* st,
                               long long* t_seq, float scale, int phi, void* cuda_stream) {
  if (phi == GF_PHI_FAVOR_POS) return GF_ERR_INVALID_ARG;  // needs its projections: gformer_decode_step_ragged_w
  return gformer_decode_step_ragged_w(q, k, v, o, st, t_seq, scale, phi, nullptr, cuda_stream);
}

int gformer_decode_step_ragged_w(const void* q, const void* k, const void* v, void* o, gf_decode_state* st,
                                 long long* t_seq, float scale, int phi, const void* W, void* cuda_stream) {
  if (!t_seq || (reinterpret_cast<uintptr_t>(t_seq) & 7u) != 0) return GF_ERR_INVALID_ARG;
  if (st && st->H > 4096) return GF_ERR_UNSUPPORTED;  // the arrival count of a sequence's heads has 15 bits
  return decode_step_impl(q, k, v, o, st, t_seq, scale, phi, W, cuda_stream);
}

static int decode_step_impl(const void* q, const void* k, const void* v, void* o, gf_decode_state* st,
                            long long* t_seq, float scale, int phi, const void* W, void* cuda_stream) {
  if (!q || !k || !v || !o || !st) return GF_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o)) return GF_ERR_INVALID_ARG;
  {
    const int rc = check_phi(phi, W);
    if (rc != GF_OK) return rc;
  }
  if (st->B < 1 || st->H < 1 || st->w < 1 || st->h_sparse < 0 || st->h_sparse > st->H || st->t < 0)
    return GF_ERR_INVALID_ARG;
  if (st->dtype != GF_F32 && st->dtype != GF_BF16) return GF_ERR_INVALID_ARG;
  if (st->d != 64 && st->d != 128) return GF_ERR_UNSUPPORTED;
  if (st->B > 65535) return GF_ERR_UNSUPPORTED;
  // (rings of more than 40 960 slots are refused since the scores of a window were kept in shared memory; the kernel has no
  // such limit any more, and nothing above it is tested)
  if ((size_t)st->w * sizeof(float) > 160 * 1024) return GF_ERR_UNSUPPORTED;
  if (st->h_sparse > 0 &&
      (!st->k_cache || !st->v_cache || !aligned16(st->k_cache) || !aligned16(st->v_cache)))
    return GF_ERR_INVALID_ARG;
  if (st->h_sparse < st->H && (!st->S || !st->z || !aligned16(st->S) || !aligned16(st->z)))
    return GF_ERR_INVALID_ARG;
  const size_t bytes = (size_t)st->B * st->H * st->d * elem_size(st->dtype);
  if (overlaps(o, q, bytes) || overlaps(o, k, bytes) || overlaps(o, v, bytes)) return GF_ERR_INVALID_ARG;
  if (!(scale > 0.f)) scale = 1.0f / sqrtf((float)st->d);
  cudaError_t e = gf::launch_decode_step(q, k, v, o, st->k_cache, st->v_cache, st->S, st->z, st->t, t_seq, st->B,
                                         st->H, st->d, st->w, st->h_sparse, scale, st->dtype,
                                         (cudaStream_t)cuda_stream, W);
  if (e != cudaSuccess) return GF_ERR_CUDA;
  if (t_seq == nullptr) st->t += 1;
  return GF_OK;
}

}  // extern "C"
