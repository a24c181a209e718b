// A runtime without a device, for the host side of the library (spd_api.cu built as C++): "device" memory is host memory,
// kernels do nothing, and a call of the test's choice fails.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstring>

#include "spd_prefill_tc.h"

namespace {
int copies_until_failure = -1, waits_until_failure = -1, enqueued = 0, capturing = 0;
bool due(int &left) { return left >= 0 && left-- == 0; }
CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
cudaError_t launched() {
  ++enqueued;
  return cudaSuccess;
}
}  // namespace

extern "C" {

// The copy (wait) behind the next `copies` (`waits`) fails; -1: none.
void fake_fail(int copies, int waits) {
  copies_until_failure = copies;
  waits_until_failure = waits;
}
int fake_enqueued() { return enqueued; }
// Whether the stream is being captured; a wait for it fails then.
void fake_capture(int on) { capturing = on; }

cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties_v2(cudaDeviceProp *p, int) {
  std::memset(p, 0, sizeof *p);
  p->multiProcessorCount = 148;
  p->cooperativeLaunch = 1;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char *, void **fn, unsigned long long, cudaDriverEntryPointQueryResult *found) {
  *fn = reinterpret_cast<void *>(&encode);
  *found = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (due(copies_until_failure)) return cudaErrorLaunchFailure;
  ++enqueued;
  std::memcpy(dst, src, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind) {
  std::memcpy(dst, src, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2D(void *, size_t, const void *, size_t, size_t, size_t, cudaMemcpyKind) { return cudaErrorNotSupported; }
cudaError_t cudaMemsetAsync(void *dst, int v, size_t n, cudaStream_t) {
  ++enqueued;
  std::memset(dst, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  if (capturing) return cudaErrorStreamCaptureUnsupported;
  return due(waits_until_failure) ? cudaErrorLaunchFailure : cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
  *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}

cudaError_t spd_internal_prepare(size_t, int *per_sm) {
  *per_sm = 1;
  return cudaSuccess;
}
cudaError_t spd_internal_prefill_prepare(int *per_sm) {
  *per_sm = 1;
  return cudaSuccess;
}
cudaError_t spd_internal_tc_prepare() { return cudaSuccess; }
cudaError_t spd_internal_job_prepare() { return cudaSuccess; }
cudaError_t spd_internal_pack_image(const void *, void *, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t spd_internal_launch(const spd::KParams *, int, size_t, cudaStream_t) { return launched(); }
cudaError_t spd_internal_prefill_launch(const spd::KParams *, int, cudaStream_t) { return launched(); }
cudaError_t spd_internal_tc_prefill(const spd::TcJob *, const spd::KParams *, cudaStream_t, int *n) {
  *n = 1;
  return launched();
}
cudaError_t spd_internal_tc_stall(const spd::TcJob *, int, cudaStream_t) { return launched(); }
cudaError_t spd_internal_batch_step(const spd::TcJob *, const spd::KParams *, int, int, int, const __nv_bfloat16 *, float *, int32_t *, cudaStream_t,
                                    int *n) {
  *n = 1;
  return launched();
}

}  // extern "C"
