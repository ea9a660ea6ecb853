// Exclusive prefix sums (int32 counts -> int32 or int64 offsets) used to turn
// counts into CSR offsets.  Deterministic (integer arithmetic).
//
// Two launches: sums of 4096-element tiles, then a scan of each tile that
// starts from the sum of the tiles before it, which the tile's block adds up
// itself (a few loads per thread while there are at most kDirectTiles tiles;
// beyond that the tile sums are scanned first, recursively).  One launch when
// everything fits one tile.  Latency-bound at the sizes of a graph build: the
// three-launch form it replaced took 9-10 us per scan at 200k points in a
// launch list, against about 6 us.  Elements travel through shared memory so
// that global loads and stores are coalesced while each thread scans 16
// consecutive elements (row padding: no bank conflicts).
#include "common.cuh"

namespace xmgn {

namespace {
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr int64_t kDirectTiles = 2048;

__device__ __forceinline__ int64_t warp_sum64(int64_t x) {
#pragma unroll
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Sum over the block's threads, returned to all of them (red: 8 entries).
__device__ __forceinline__ int64_t block_sum64(int64_t x, int64_t* red) {
  x = warp_sum64(x);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  int64_t t = 0;
#pragma unroll
  for (int w = 0; w < kScanThreads / 32; ++w) t += red[w];
  return t;
}

template <class T>
__global__ void __launch_bounds__(kScanThreads) tile_sum_kernel(const T* __restrict__ in, int64_t n,
                                                                int64_t* __restrict__ sums) {
  pdl_wait();
  pdl_trigger();
  __shared__ int64_t red[kScanThreads / 32];
  const int64_t base = int64_t(blockIdx.x) * kScanTile;
  int64_t s = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    const int64_t i = base + j * kScanThreads + threadIdx.x;
    if (i < n) s += int64_t(in[i]);
  }
  s = block_sum64(s, red);
  if (threadIdx.x == 0) sums[blockIdx.x] = s;
}

// Scan of tile blockIdx.x.  sums: null (a single tile), the tile sums, or
// (scanned) their exclusive prefix.  The last tile also writes out[n].  Nothing
// is written when `skip` is given and set.
template <class T, class O>
__global__ void __launch_bounds__(kScanThreads) tile_scan_kernel(const T* __restrict__ in, O* __restrict__ out,
                                                                 int64_t n, const int64_t* __restrict__ sums,
                                                                 int scanned, const int32_t* __restrict__ skip) {
  pdl_wait();
  pdl_trigger();
  if (skip && *skip) return;
  __shared__ int64_t red[kScanThreads / 32];
  __shared__ int64_t tile[kScanTile + kScanTile / kScanItems];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t base = int64_t(blockIdx.x) * kScanTile;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    const int k = j * kScanThreads + tid;
    tile[k + k / kScanItems] = base + k < n ? int64_t(in[base + k]) : 0;
  }
  int64_t off = 0;
  if (sums && scanned) {
    off = sums[blockIdx.x];
  } else if (sums) {
    for (int64_t i = tid; i < int64_t(blockIdx.x); i += kScanThreads) off += sums[i];
    off = block_sum64(off, red);
  }
  __syncthreads();
  int64_t* mine = tile + tid * (kScanItems + 1);
  int64_t run = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) run += mine[j];
  int64_t x = run;  // inclusive warp scan of the threads' totals
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) red[wid] = x;
  __syncthreads();
  for (int w = 0; w < wid; ++w) off += red[w];
  off += x - run;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    const int64_t v = mine[j];
    mine[j] = off;
    off += v;
  }
  if (tid == kScanThreads - 1 && blockIdx.x == gridDim.x - 1) out[n] = O(off);
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    const int k = j * kScanThreads + tid;
    if (base + k < n) out[base + k] = O(tile[k + k / kScanItems]);
  }
}

template <class T, class O>
xmgn_status scan_impl(const T* in, O* out, int64_t n, int64_t* tmp, cudaStream_t s, const int32_t* skip = nullptr) {
  if (n <= 0) {
    XMGN_CUDA(cudaMemsetAsync(out, 0, sizeof(O), s));
    return XMGN_OK;
  }
  const int64_t nt = (n + kScanTile - 1) / kScanTile;
  const int64_t* sums = nullptr;
  if (nt > 1) {
    launch_pdl(tile_sum_kernel<T>, unsigned(nt), kScanThreads, 0, s, in, n, tmp);
    XMGN_LAUNCH_CHECK();
    sums = tmp;
    if (nt > kDirectTiles) {
      XMGN_TRY((scan_impl<int64_t, int64_t>(tmp, tmp + nt, nt, tmp + 2 * nt + 1, s)));
      sums = tmp + nt;
    }
  }
  launch_pdl(tile_scan_kernel<T, O>, unsigned(nt), kScanThreads, 0, s, in, out, n, sums, nt > kDirectTiles ? 1 : 0,
             skip);
  XMGN_LAUNCH_CHECK();
  return XMGN_OK;
}
}  // namespace

size_t scan_tmp_elems(int64_t n) {
  const int64_t nt = (n + kScanTile - 1) / kScanTile;
  if (nt <= 1) return 1;
  return size_t(2 * nt + 1) + scan_tmp_elems(nt);
}

xmgn_status exclusive_scan_i32(const int32_t* in, int64_t* out, int64_t n, int64_t* tmp, cudaStream_t s,
                               const int32_t* skip) {
  return scan_impl<int32_t, int64_t>(in, out, n, tmp, s, skip);
}
xmgn_status exclusive_scan_i32(const int32_t* in, int32_t* out, int64_t n, int64_t* tmp, cudaStream_t s) {
  return scan_impl<int32_t, int32_t>(in, out, n, tmp, s);
}

}  // namespace xmgn
