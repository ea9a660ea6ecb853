// The library's host side on a stand-in CUDA runtime, for what no GPU test can
// show: which launches a second device would refuse, whether the sources of
// asynchronous copies live until they are read, and what shapes are launched.
// Linked with the library's own objects and no libcudart: kernels are recorded
// and not run, device memory is host memory, a device-to-host copy reads zeros.
// Prints one "name value" line per result; argv[1] picks the scenario.
#include <cuda_runtime_api.h>
#include <malloc.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include "../include/xmgn.h"

namespace {
int g_device = 0;
cudaError_t g_last = cudaSuccess;
std::map<const void*, std::string>& names() {  // filled by static constructors
  static std::map<const void*, std::string> m;
  return m;
}
std::map<std::pair<int, const void*>, int> g_smem;  // dynamic shared memory granted to (device, kernel)
struct Launch {
  std::string kernel;
  dim3 grid;
  std::vector<uint64_t> args;  // the first words of some kernels' arguments
};
std::vector<Launch> g_launches;
int g_refused = 0, g_changed = 0;
struct Copy {
  const void* src;
  std::vector<char> seen;
};
std::vector<Copy> g_pending;  // host sources that the device has not read yet

void settle() {
  for (const Copy& c : g_pending) g_changed += memcmp(c.src, c.seen.data(), c.seen.size()) != 0;
  g_pending.clear();
}
int encode_tiled(...) { return 0; }
}  // namespace

// Freed memory does not keep its contents.
void operator delete(void* p) noexcept {
  if (p) memset(p, 0xdd, malloc_usable_size(p));
  free(p);
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }
void* operator new(size_t n) {
  void* p = malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}

extern "C" {
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {
  names()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  const auto it = g_smem.find({g_device, f});
  const size_t may = it == g_smem.end() ? 48 * 1024 : size_t(it->second);
  if (c->dynamicSmemBytes > may) {
    ++g_refused;
    return g_last = cudaErrorInvalidValue;
  }
  Launch l{names()[f], c->gridDim, {}};
  if (l.kernel.find("sum_parts_kernel") != std::string::npos)  // (partial sums, how many, of what length)
    l.args = {*static_cast<uint64_t*>(args[0]), *static_cast<uint32_t*>(args[1]), *static_cast<uint32_t*>(args[2])};
  g_launches.push_back(l);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = g_device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 232448;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "refused by the stand-in"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static uint64_t word[8];
  *p = word;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind k, cudaStream_t) {
  const char* s = static_cast<const char*>(src);
  if (k == cudaMemcpyHostToDevice) g_pending.push_back({src, std::vector<char>(s, s + n)});
  if (k == cudaMemcpyDeviceToHost) memset(dst, 0, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  settle();
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode_tiled);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
#define UNUSED_CALL(name, ...) \
  cudaError_t name(__VA_ARGS__) { return cudaSuccess; }
UNUSED_CALL(cudaEventCreate, cudaEvent_t*)
UNUSED_CALL(cudaEventCreateWithFlags, cudaEvent_t*, unsigned)
UNUSED_CALL(cudaEventDestroy, cudaEvent_t)
UNUSED_CALL(cudaEventElapsedTime, float*, cudaEvent_t, cudaEvent_t)
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) {
  g_launches.push_back({"event", dim3(), {}});
  return cudaSuccess;
}
UNUSED_CALL(cudaEventRecordWithFlags, cudaEvent_t, cudaStream_t, unsigned)
UNUSED_CALL(cudaEventSynchronize, cudaEvent_t)
UNUSED_CALL(cudaGraphDestroy, cudaGraph_t)
UNUSED_CALL(cudaGraphExecDestroy, cudaGraphExec_t)
UNUSED_CALL(cudaGraphInstantiate, cudaGraphExec_t*, cudaGraph_t, unsigned long long)
UNUSED_CALL(cudaGraphLaunch, cudaGraphExec_t, cudaStream_t)
UNUSED_CALL(cudaStreamBeginCapture, cudaStream_t, cudaStreamCaptureMode)
UNUSED_CALL(cudaStreamCreateWithFlags, cudaStream_t*, unsigned)
UNUSED_CALL(cudaStreamDestroy, cudaStream_t)
UNUSED_CALL(cudaStreamEndCapture, cudaStream_t, cudaGraph_t*)
UNUSED_CALL(cudaStreamWaitEvent, cudaStream_t, cudaEvent_t, unsigned)
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
}

namespace xmgn {
void tune_time(int op);  // tune.cuh
}

namespace {
// Any address the library only hands on.
template <class T>
T* fake(int i) {
  return reinterpret_cast<T*>(uintptr_t(0x700000000000) + (uintptr_t(i) << 32));
}

int partition(int32_t P) {
  const int64_t n = 4096, e = 30000;
  size_t bytes = 0;
  xmgn_partition_halo_ws(n, e, P, &bytes);
  std::vector<int64_t> a(P + 1), b(P + 1), c(P);
  return xmgn_partition_halo(fake<int64_t>(0), fake<int32_t>(1), n, e, fake<float>(2), 2097152.0, P, 3, nullptr,
                             fake<void>(3), bytes, nullptr, a.data(), b.data(), c.data(), nullptr, nullptr, nullptr,
                             nullptr, nullptr, nullptr, 0, 0, nullptr);
}

int step(int H, xmgn_dtype dtype, int64_t n = 3000, int64_t e = 20000) {
  const xmgn_model_desc d{H, 2, 6, 4, dtype, 0};
  const xmgn_graph g{n,     e,      fake<int64_t>(0), fake<int32_t>(1), fake<int32_t>(2), fake<int32_t>(3), nullptr,
                     nullptr, n, n};
  size_t ws = 0, ck = 0;
  xmgn_model_ws(&d, n, e, &ws, &ck);
  int rc = xmgn_forward(&d, fake<float>(4), &g, fake<float>(5), fake<float>(6), fake<float>(7), fake<float>(8),
                        fake<float>(9), fake<void>(10), fake<void>(20), ws, nullptr);
  if (rc == 0)
    rc = xmgn_backward(&d, fake<float>(4), &g, fake<float>(5), fake<float>(6), fake<float>(7), fake<void>(10),
                       fake<float>(11), nullptr, fake<void>(20), ws, nullptr);
  return rc;
}
}  // namespace

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  if (what == "copies") {
    for (int P : {2, 24, 300}) printf("status_%d %d\n", P, partition(P));
    settle();
    printf("changed %d\n", g_changed);
  } else if (what == "devices") {
    for (g_device = 0; g_device < 3; ++g_device) {
      printf("partition_%d %d\n", g_device, partition(24));
      printf("bf16_%d %d\n", g_device, step(128, XMGN_BF16));
      printf("wide_%d %d\n", g_device, step(256, XMGN_BF16));
      printf("fp32_%d %d\n", g_device, step(128, XMGN_FP32));
    }
    printf("refused %d\n", g_refused);
  } else if (what == "timed") {  // what is launched while the tuner times a class, and where its events stand
    xmgn::tune_time(atoi(argv[2]));
    printf("status %d\n", step(128, XMGN_BF16, atoll(argv[3]), 8 * atoll(argv[3])));
    for (const Launch& l : g_launches) printf("launch %s\n", l.kernel.c_str());
  } else if (what == "products") {  // row chunks of the FP32 weight-gradient products; every sum of partials
    printf("status %d\n", step(atoi(argv[2]), XMGN_FP32, atoll(argv[3]), atoll(argv[3])));
    for (const Launch& l : g_launches) {
      if (l.kernel.find("sgemm_kernelILi2E") != std::string::npos) printf("chunks %u\n", l.grid.y);
      if (!l.args.empty())
        printf("parts %llu %llu %llu\n", (unsigned long long)l.args[0], (unsigned long long)l.args[1],
               (unsigned long long)l.args[2]);
    }
  }
  return 0;
}
