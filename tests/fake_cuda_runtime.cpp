// A CUDA runtime that runs nothing and writes down what it is asked, and launchers that do the same: what the step driver
// (csrc/ctx.cu) is linked with in tests/test_step_driver_host.py.  Streams and events are numbers; the n-th call that can
// fail inside a step does so when the test asks for it.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <string>

#include "adapm_internal.h"

namespace {
std::string g_log;
long g_countdown = -1;        // calls until one fails; < 0: none does
intptr_t g_next = 100;        // handles of streams and events

void note(const char* what, const void* a, const void* b) {
  char line[96];
  std::snprintf(line, sizeof(line), "%s %ld %ld\n", what, (long)(intptr_t)a, (long)(intptr_t)b);
  g_log += line;
}
bool fails() { return g_countdown >= 0 && g_countdown-- == 0; }
cudaError_t answer(const char* what, const void* a, const void* b) {
  if (fails()) { note("failed", nullptr, nullptr); return cudaErrorUnknown; }
  note(what, a, b);
  return cudaSuccess;
}
int launch(cudaStream_t s) { return answer("launch", s, nullptr) == cudaSuccess ? ADAPM_OK : ADAPM_ECUDA; }
}  // namespace

extern "C" {
void fake_begin(long fail_at) { g_log.clear(); g_countdown = fail_at; }
const char* fake_log() { g_countdown = -1; return g_log.c_str(); }

cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorName(cudaError_t) { return "fake"; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) { return answer("memset", s, nullptr); }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t s) { return answer("copy", s, nullptr); }
cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) { *lo = 0; *hi = -1; return cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { *s = (cudaStream_t)++g_next; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { note("sync", s, nullptr); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)++g_next; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)++g_next; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return answer("record", e, s); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return answer("wait", s, e); }
}

namespace adapm {
int launch_stream(const StreamBlk*, const int32_t*, int64_t, bool, const Bases&, const StepScalars&, int, cudaStream_t s) { return launch(s); }
int launch_reduce_partial(const ReduceJob*, const int32_t*, int64_t, int64_t, const void*, float*, int, const int32_t*, cudaStream_t s) { return launch(s); }
int launch_reduce_final(const ReduceJob*, int64_t, int64_t, float*, const float*, float, const int32_t*, const float*, bool, cudaStream_t s) { return launch(s); }
int launch_gradnorm(const NormRange*, const int32_t*, int64_t, const void*, int, float*, float, int, float*, int32_t*, cudaStream_t s) { return launch(s); }
int launch_gemm(const GemmProb*, int64_t, int64_t, const Bases&, int, cudaStream_t s) { return launch(s); }
int launch_fp32_gram(const Fp32Gram*, const int32_t*, int64_t, const Bases&, int32_t*, cudaStream_t s) { return launch(s); }
int launch_fp32_refit(const Fp32Refit*, const int32_t*, int64_t, const Bases&, int, int32_t*, cudaStream_t s) { return launch(s); }
int launch_apply_simt(const ApplyBlk*, const int32_t*, int64_t, const Bases&, const StepScalars&, int, cudaStream_t s) { return launch(s); }
int launch_spd_inverse(const InverseJob*, int64_t, float*, float, const int32_t*, cudaStream_t s) { return launch(s); }
int launch_copy_ranges(const NormRange*, const int32_t*, int64_t, float*, const float*, const int32_t*, cudaStream_t s) { return launch(s); }
int launch_meansq_partial(const void*, int, int64_t, int64_t, int, float*, cudaStream_t s) { return launch(s); }
int launch_meansq_final(const float*, int64_t, int64_t, int, float*, cudaStream_t s) { return launch(s); }
int launch_init_L0(const InitJob*, int64_t, float*, uint64_t, int, cudaStream_t s) { return launch(s); }

// no block takes the tensor path here
bool tensor_path_block_ok(const adapm_hparams&, const adapm_block&) { return false; }
int build_tensor_program(adapm_ctx*, const std::vector<int64_t>&, const std::vector<double>&, int64_t&, std::vector<ReduceJob>&, int64_t&) { return ADAPM_EUNSUPPORTED; }
int tensor_prepare_step(adapm_ctx*, const Bases&, int64_t, cudaStream_t, int*, int*) { return ADAPM_EUNSUPPORTED; }
int run_tensor_launch(adapm_ctx*, const Launch&, const Bases&, const StepScalars&, int, cudaStream_t) { return ADAPM_EUNSUPPORTED; }
void destroy_tensor_program(adapm_ctx*) {}
void tensor_state_changed(adapm_ctx*) { note("rebuild", nullptr, nullptr); }
int run_expired_wait_probe(adapm_ctx*, cudaStream_t) { return ADAPM_EUNSUPPORTED; }
size_t probe_table(std::vector<unsigned char>& out) { out.resize(16); return 16; }
}  // namespace adapm
