// The host side of the no-allocation entry point on a fake CUDA runtime, for tests/test_static_host.py: which kernels a call
// launches while pinning the status page fails, works, or must not be tried.
#include <cstdarg>
#include <cstring>

#include "snn_static.cu"

namespace {
int g_register_fails = 0, g_registers = 0, g_capturing = 0, g_tensor_core = 0, g_popcount = 0, g_device = 0, g_asked = 0, g_plans_made = 0,
    g_planned_for = 0;
unsigned char g_device_memory[kStaticScratchBytes];
int* g_reported = nullptr;
}  // namespace

extern "C" {
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = g_device_memory; return cudaSuccess; }
cudaError_t cudaHostRegister(void*, size_t, unsigned int) {
  ++g_registers;
  if (g_register_fails <= 0) return cudaSuccess;
  --g_register_fails;
  return cudaErrorMemoryAllocation;
}
cudaError_t cudaHostGetDevicePointer(void** p, void* host, unsigned int) { *p = host; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) { ++g_asked; *v = d ? 132 : 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  memset(a, 0, sizeof(*a));
  a->type = cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
}

namespace snn {
snn_status_t api_fail(snn_status_t st, const char*, ...) { return st; }
void api_count_launches(int) {}
bool tcg_static_plan(const Geom&, TcgStatic* out) {
  ++g_plans_made;
  out->bytes = 1024;
  const int sms = sm_count();
  memcpy(out->opaque, &sms, sizeof(sms));
  return true;
}
cudaError_t tcg_static_forward(const TcgStatic& plan, const Geom&, const uint8_t*, const uint16_t*, const float*, uint8_t*, const Launch&,
                               int* status, int*) {
  ++g_tensor_core;
  memcpy(&g_planned_for, plan.opaque, sizeof(g_planned_for));
  g_reported = status;
  return cudaSuccess;
}
cudaError_t decode_layer(const LayerDev&, const uint8_t*, const Geom&, int, cudaStream_t, int*) { return cudaSuccess; }
cudaError_t popc_forward(const LayerDev&, const Geom&, const Launch&, int*) { ++g_popcount; return cudaSuccess; }
}  // namespace snn

extern "C" {
// One call; register_fails: the next so many attempts to pin fail.  out: attempts to pin, tensor-core and popcount launches so far.
int static_call(int register_fails, int capturing, int* out, int device) {
  if (register_fails >= 0) g_register_fails = register_fails;
  g_capturing = capturing;
  uint16_t codebook[2] = {1, 2};
  uint8_t stream[16 * 16 / 8] = {0};
  float alpha[16] = {0};
  alignas(16) static unsigned char buffer[16];
  snn_conv_desc_t d{};
  d.c_in = d.c_out = 16; d.tau = 1; d.stride = 1; d.pad = 1; d.act_type = SNN_ACT_BIN; d.ksize = 3; d.device = device;
  d.codebook = codebook; d.idx_packed = stream; d.alpha = alpha;
  const int st = snn_conv_forward_static(&d, buffer, 1, 8, 8, buffer, SNN_OUT_F32, nullptr);
  out[0] = g_registers; out[1] = g_tensor_core; out[2] = g_popcount;
  return st;
}
// SMs the last tensor-core launch was planned for, plans made, questions for a device's SMs
void static_planned(int* out) { out[0] = g_planned_for; out[1] = g_plans_made; out[2] = g_asked; }
// What a kernel does whose bounded wait ran out.
void static_report(int code) { *g_reported = code; }
}
