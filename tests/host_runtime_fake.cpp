// Fakes of the CUDA runtime calls, the NVTX calls and the kernel launchers that csrc/api.cu makes, for
// tests of its host side without a GPU: every call is written to a log, a named call can be made to
// fail, and the current device is what the test says.
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

#include "../paper_2507_19608_b200/csrc/delta_internal.cuh"
#include "../paper_2507_19608_b200/csrc/k2_tc.cuh"

namespace {
std::mutex g_mu;
std::string g_log;
std::map<std::string, int> g_fail;      // call -> error of its next run
int g_device = 0, g_capturing = 0, g_fill = -1;
size_t g_handle = 0x1000;

cudaError_t call(const char* name, const std::string& args = "") {
  std::lock_guard<std::mutex> lock(g_mu);
  g_log += std::string(name) + args + "\n";
  auto it = g_fail.find(name);
  if (it == g_fail.end()) return cudaSuccess;
  const int e = it->second;
  g_fail.erase(it);
  return (cudaError_t)e;
}
std::string num(const char* key, long v) { return std::string(" ") + key + "=" + std::to_string(v); }
template <typename H> cudaError_t make(const char* name, H* out) {
  const cudaError_t e = call(name, num("dev", g_device));
  *out = e == cudaSuccess ? (H)(g_handle += 16) : nullptr;
  return e;
}
}  // namespace

extern "C" {
#define EXPORT __attribute__((visibility("default")))
EXPORT const char* fake_log() { return g_log.c_str(); }
EXPORT void fake_clear() { g_log.clear(); g_fail.clear(); }
EXPORT void fake_fail(const char* name, int error) { g_fail[name] = error; }
EXPORT void fake_fill(int byte) { g_fill = byte; }      // what copies leave at their destination (-1: nothing)
EXPORT void fake_capturing(int on) { g_capturing = on; }
EXPORT void fake_device(int dev) { g_device = dev; }

const char* cudaGetErrorName(cudaError_t e) { return e == cudaSuccess ? "cudaSuccess" : "fakeError"; }
const char* cudaGetErrorString(cudaError_t e) {
  static thread_local char text[32];
  snprintf(text, sizeof(text), "code %d", (int)e);
  return text;
}
cudaError_t cudaGetDevice(int* dev) { *dev = g_device; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return call("memset"); }
cudaError_t cudaMemcpyAsync(void* dst, const void*, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  if (g_fill >= 0) memset(dst, g_fill, n);
  return call("memcpy", num("kind", kind));
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind kind, cudaStream_t) {
  return call("memcpy", num("kind", kind));
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return make("stream_create", s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return call("stream_destroy"); }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return call("synchronize"); }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return call("wait_event"); }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return make("event_create", e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return make("event_create", e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return call("event_destroy"); }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return call("event_record"); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return call("event_synchronize"); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.0f; return cudaSuccess; }
int nvtxRangePushA(const char* name) { call("push", std::string(" ") + name); return 0; }
int nvtxRangePop() { call("pop"); return 0; }
}

namespace delta {
bool tc_kernel_available(int) { return true; }
bool tc_kernel_shape(int d) { return d == 64; }
bool tcq_kernel_shape(int d) { return d == 64 || d == 128; }
bool decode_mma_applies(const Shape&, int dtype) { return dtype == DELTA_BF16; }
size_t keypack_capacity(int T_max, int d) { return (size_t)T_max * d + 8u * ((size_t)T_max / 32 + 2); }
int keypack_segments(int T_max) { return (T_max + 31) / 32; }
cudaError_t launch_delta_chain(const Shape& s, const Workspace&, const void*, const SeqBatch&, float, int, int, bool, bool, void*,
                               size_t, cudaStream_t) { return call("chain", num("heads", s.B * s.H)); }
cudaError_t launch_delta_finish(const Shape& s, const Workspace&, const void*, const void*, const SeqBatch&, float, int, int, int, bool,
                                bool, bool, int, cudaStream_t) { return call("finish", num("heads", s.B * s.H)); }
cudaError_t launch_hybrid_attn_tc(const Shape& s, const Workspace&, const void*, const void*, const void*, void*, int, int, int,
                                  cudaStream_t) { return call("attn_tc", num("heads", s.B * s.H)); }
cudaError_t launch_hybrid_attn_tcq(const Shape& s, const Workspace&, const void*, const void*, const void*, void*, const SeqBatch& q,
                                   float, int, int, bool, bool, int, cudaStream_t) {
  return call("attn", num("heads", s.B * s.H) + num("form_heads", q.form_heads(s)));
}
cudaError_t launch_hybrid_attn_f32(const Shape& s, const Workspace&, const void*, const void*, const void*, void*,
                                       const SeqBatch& q, float, int, int, int, cudaStream_t) {
  return call("attn", num("heads", s.B * s.H) + num("form_heads", q.form_heads(s)));
}
cudaError_t launch_pack_keys(const Shape&, const Workspace&, const void*, int, cudaStream_t) { return call("pack"); }
cudaError_t launch_decode_step(const Shape&, const Workspace&, const void*, const void*, const void*, void*, void*, void*, int, float,
                               int, int, int, cudaStream_t) { return call("decode"); }
cudaError_t launch_decode_step_mma(const Shape&, const Workspace&, const void*, const void*, const void*, void*, void*, void*, int,
                                   const int*, float, int, int, bool, bool, bool behind_step, DecodeTmapCache*, cudaStream_t) {
  return call("decode_mma", num("behind_step", behind_step));
}
cudaError_t launch_decode_step_f32(const Shape&, const Workspace&, const void*, const void*, const void*, void*, void*, void*, int,
                                   const int*, float, int, int, DecodeTmapCache*, cudaStream_t) { return call("decode_f32"); }
cudaError_t launch_decode_step_key(const Shape&, const Workspace&, const void*, const void*, const void*, void*, void*, void*, int,
                                   float, int, int, cudaStream_t) { return call("decode_key"); }
}  // namespace delta
