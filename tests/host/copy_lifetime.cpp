// Plan creation and trajectory updates against a stand-in for the CUDA runtime in
// which an asynchronous copy from host memory reads its source only when something
// waits for it, as the runtime's contract allows.  Freed memory is overwritten and
// never reused, so a copy whose source died before the wait shows as a change.
// Kernels do nothing; the tile starts that the host reads back are a ramp, so that
// every tile has points.  Prints "late <copies whose source changed> of <copies>".
#include <malloc.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/nufft_gb300.h"

void* operator new(size_t n) { return malloc(n ? n : 1); }
void operator delete(void* p) noexcept {
  if (p) memset(p, 0xA5, malloc_usable_size(p));
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }

namespace {
struct Copy {
  void* dst;
  const void* src;
  size_t n;
  char* then;   // the source when the copy was asked for
};
Copy queue[64];
int queued = 0, copies = 0, late = 0;
size_t last = 1;                // bytes of the previous copy to the host
int64_t bins = 0, points = 0;   // of the plan in the making
int fail_after = -1;            // launch checks to pass after a queued copy before one fails

void run_queue() {
  for (int i = 0; i < queued; ++i) {
    Copy& c = queue[i];
    late += memcmp(c.then, c.src, c.n) != 0;
    memcpy(c.dst, c.src, c.n);
    free(c.then);
  }
  queued = 0;
}
}  // namespace

extern "C" {
int cudaMemcpyAsync(void* dst, const void* src, size_t n, int kind, void*) {
  if (kind == 1) {   // host to device: later
    char* then = (char*)malloc(n ? n : 1);
    memcpy(then, src, n);
    if (queued == 64) abort();
    queue[queued++] = {dst, src, n, then};
    ++copies;
    return 0;
  }
  memmove(dst, src, n);
  // the tile starts (with one tile as long as the plan's two flags, which follow
  // the errors of the coefficient tables)
  const bool flags = kind == 2 && n == 8 && last % 32 == 0;
  if (kind == 2) last = n;
  if (kind == 2 && !flags && n == (size_t)(bins + 1) * 4)
    for (int64_t b = 0; b <= bins; ++b) ((int32_t*)dst)[b] = (int32_t)(points * b / bins);
  return 0;
}
int cudaMemcpy(void* dst, const void* src, size_t n, int) { run_queue(); memmove(dst, src, n); return 0; }
int cudaStreamSynchronize(void*) { run_queue(); return 0; }
int cudaMalloc(void** p, size_t n) { *p = calloc(1, n ? n : 1); return 0; }
int cudaFree(void* p) { run_queue(); free(p); return 0; }
int cudaGetLastError() { return queued > 0 && fail_after >= 0 && fail_after-- == 0 ? 1 : 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
const char* cudaGetErrorString(int) { return "failed on purpose"; }
int cudaStreamIsCapturing(void*, int* s) { *s = 0; return 0; }
#define STUB(name) int name() { return 0; }
STUB(cudaMemsetAsync) STUB(cudaFuncSetAttribute) STUB(cudaEventCreate) STUB(cudaEventCreateWithFlags)
STUB(cudaEventDestroy) STUB(cudaEventElapsedTime) STUB(cudaEventRecord) STUB(cudaEventSynchronize)
STUB(cudaGetSymbolAddress) STUB(cudaGraphDestroy) STUB(cudaGraphExecDestroy) STUB(cudaGraphInstantiate)
STUB(cudaGraphLaunch) STUB(cudaPointerGetAttributes) STUB(cudaSetDevice) STUB(cudaStreamBeginCapture)
STUB(cudaStreamCreateWithFlags) STUB(cudaStreamDestroy) STUB(cudaStreamEndCapture) STUB(cudaStreamWaitEvent)
STUB(__cudaGetKernel) STUB(__cudaLaunchKernel) STUB(__cudaPopCallConfiguration) STUB(__cudaPushCallConfiguration)
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaRegisterFunction() {}
void __cudaRegisterVar() {}
void __cudaUnregisterFatBinary(void**) {}
}

// copy_lifetime d K J M fail_after
int main(int, char** argv) {
  const int d = atoi(argv[1]), k = atoi(argv[2]), j = atoi(argv[3]);
  const int64_t m = atoll(argv[4]);
  const int N[3] = {k / 2, k / 2, k / 2}, K[3] = {k, k, k}, J[3] = {j, j, j};
  float* om = (float*)calloc(m * d, sizeof(float));
  // the number of tiles, from a plan without points
  nufft_plan_t* p = nullptr;
  bins = 1;
  if (nufft_plan(d, N, K, J, 0, nullptr, nullptr, &p) != 0) return 2;
  int64_t info[16];
  nufft_plan_info(p, info);
  nufft_plan_destroy(p);
  bins = info[11];
  points = m;
  fail_after = atoi(argv[5]);
  copies = late = 0;
  const bool fails = fail_after >= 0;
  if ((nufft_plan(d, N, K, J, m, om, nullptr, &p) != 0) != fails) return 3;
  if (!fails) {
    if (nufft_plan_set_trajectory(p, om) != 0) return 4;
    points = m / 2;   // other tile starts, still within the capacity
    if (nufft_plan_set_trajectory(p, om) != 0) return 5;
    fail_after = 0;
    if (nufft_plan_set_trajectory(p, om) == 0) return 6;
    nufft_plan_destroy(p);
  }
  printf("late %d of %d\n", late, copies);
  return 0;
}
