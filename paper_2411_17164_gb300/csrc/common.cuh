// Shared host/device utilities of libxmgn (errors, workspace carving, launch
// helpers).  Everything here is internal; the public surface is include/xmgn.h.
#pragma once

#include <atomic>
#include <utility>

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include <string>

#include "../../include/xmgn.h"

namespace xmgn {

// ---------------------------------------------------------------- errors
void set_error(const char* fmt, ...);
xmgn_status fail(xmgn_status s, const char* fmt, ...);

#define XMGN_CUDA(call)                                                                  \
  do {                                                                                   \
    cudaError_t e_ = (call);                                                             \
    if (e_ != cudaSuccess)                                                               \
      return ::xmgn::fail(XMGN_ERR_CUDA, "%s:%d %s: %s", __FILE__, __LINE__, #call,        \
                          cudaGetErrorString(e_));                                       \
  } while (0)

#define XMGN_TRY(expr)                     \
  do {                                     \
    xmgn_status s_ = (expr);               \
    if (s_ != XMGN_OK) return s_;          \
  } while (0)

// Every kernel launch is followed by exactly one XMGN_LAUNCH_CHECK(), which
// also counts the launch (xmgn_launch_count).
#define XMGN_LAUNCH_CHECK()          \
  do {                               \
    ::xmgn::count_launch();          \
    XMGN_CUDA(cudaGetLastError());   \
  } while (0)

void count_launch();

// CUDA-event probes around the launches of one kernel class (xmgn_probe_*).
enum ProbeKind : int {
  PROBE_EDGE_FWD = 0,
  PROBE_EDGE_BWD = 1,
  PROBE_NODE_FWD = 2,
  PROBE_NODE_BWD = 3,
  PROBE_WIDE_GEMM = 4,
  PROBE_KINDS = 5
};
void probe_begin(int kind, cudaStream_t s);
void probe_end(int kind, cudaStream_t s);

// Device error word (one per device, lives in api.cu).  Kernels OR a code
// into it instead of trapping; xmgn_check_device reads and clears it.
enum : uint32_t {
  DEV_ERR_RANGE = 1u,    // coordinate off the lattice
  DEV_ERR_GRAPH = 2u,    // id out of range in a graph array
  DEV_ERR_TIMEOUT = 4u,  // bounded wait gave up
  DEV_ERR_CAP = 8u,      // an output capacity was exceeded
};
uint32_t* device_error_word();  // device address for the current device

// ---------------------------------------------------------------- workspace
// Bump allocator over a caller-provided buffer; all carve-outs 256-B aligned.
struct Arena {
  char* base = nullptr;
  size_t cap = 0;
  size_t used = 0;
  bool dry = false;  // size-only pass
  template <class T>
  T* take(size_t count) {
    size_t off = (used + 255) & ~size_t(255);
    used = off + count * sizeof(T);
    if (dry) return nullptr;
    return reinterpret_cast<T*>(base + off);
  }
  bool ok() const { return dry || used <= cap; }
};

inline int num_sms() {
  static int cached[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) dev = 0;
  if (!cached[dev]) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    cached[dev] = n > 0 ? n : 1;
  }
  return cached[dev];
}

// Runs set() when a launch site is first reached on the current device: what it
// sets (the limit of a kernel's dynamic shared memory) belongs to the device.
// `done`, a bit per device, belongs to the site.
template <class F>
inline xmgn_status once_per_device(std::atomic<uint64_t>& done, F set) {
  int dev = 0;
  XMGN_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = dev < 64 ? uint64_t(1) << dev : 0;
  if (done.load(std::memory_order_acquire) & bit) return XMGN_OK;
  XMGN_TRY(set());
  done.fetch_or(bit, std::memory_order_release);
  return XMGN_OK;
}

inline unsigned grid_for(int64_t n, int threads, int64_t cap_blocks = 0) {
  int64_t b = (n + threads - 1) / threads;
  if (cap_blocks <= 0) cap_blocks = int64_t(num_sms()) * 32;
  if (b > cap_blocks) b = cap_blocks;
  if (b < 1) b = 1;
  return unsigned(b);
}

// ---------------------------------------------------------------- scans
// Exclusive prefix sum of n int32 values into int64 or int32 out[0..n]
// (out[n] = total).  Uses `tmp` scratch of scan_tmp_elems(n) int64.  When a
// device flag `skip` is given and set (and n > 0), out is left as it is.
size_t scan_tmp_elems(int64_t n);
xmgn_status exclusive_scan_i32(const int32_t* in, int64_t* out, int64_t n, int64_t* tmp, cudaStream_t s,
                               const int32_t* skip = nullptr);
xmgn_status exclusive_scan_i32(const int32_t* in, int32_t* out, int64_t n, int64_t* tmp, cudaStream_t s);

// ---------------------------------------------------------------- launches
// Programmatic dependent launch.  A kernel started with launch_pdl may begin
// while the kernel before it on the stream still runs: it sets itself up
// (barriers, TMEM, weights that no kernel of the call writes), calls pdl_wait()
// before it touches anything else in global memory, and then pdl_trigger() to
// let the next one begin.  As the trigger comes after the wait, whatever ran
// before the predecessor is complete when a kernel begins: only the
// predecessor's own results must wait for pdl_wait().  Without it a launch costs
// a drain, a start and the set-up in sequence: on a 2k-node graph, where a
// kernel runs 4 to 20 us, a training step (274 launches) went from 2.57 to 1.92 ms.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
inline void launch_pdl_if(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                          A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = early ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // errors: the XMGN_LAUNCH_CHECK that follows
}
template <class... P, class... A>
inline void launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  launch_pdl_if(true, kernel, grid, block, smem, s, std::forward<A>(args)...);
}
// Row kernels (LayerNorm, operand rounding, SiLU', segment sums) begin early only
// while their rows are this few bytes: over more, each takes 100 us and up and an
// early start costs more than the 2 us it saves (H = 512, 50k nodes, 725 MB a
// pass: 14.95 ms a step without, 15.55 with; H = 256, 30k nodes, 217 MB: 1.71
// without, 1.68 with).
inline bool rows_early(int64_t rows, int cols) { return rows * cols * 4 <= (int64_t(256) << 20); }

// ---------------------------------------------------------------- device helpers
__device__ __forceinline__ void dev_flag(uint32_t* err, uint32_t code) {
  if (err) atomicOr(err, code);
}

}  // namespace xmgn
