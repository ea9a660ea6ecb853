// Halo partitioning (Sec. III-A "Graph Partitioning", "Message Passing Across
// Partitions").
//
// Parts: recursive coordinate bisection (the paper uses METIS).  A level only
// needs the key (lattice coordinate on the segment's split axis, node id) of
// the first node that goes right, so every segment's key is found by radix
// selection -- a digit histogram and a bin search per pass -- and no node is
// moved or sorted.  Sizes and numbering of all levels follow from N and P, so
// the host writes one plan in advance and reads nothing back between levels.
//
// Halos: one multi-source BFS per part, all parts advanced together one hop
// per launch; a (part, node) pair is claimed exactly once through a bit in a
// P x N bitmask, and the part's map row takes the hop.  The batch order
// (part-major, inner nodes by id, then halo nodes by (hop, id)) is a stable
// counting sort of the mask's set bits, which are already in id order, by
// hop: per-block hop counts, one scan in (part, hop, block) order, and each
// set bit knows its place.
//
// Measured, 2M points in 16 parts with 15 hops, both calls: 28.9 -> 1.01 ms
// (bisection by sorting all keys per level, with six extent atomics per node,
// was 27 ms of it); 64 given regions of a 1M-point cloud: 2.48 -> 0.72 ms
// (the bitonic member sort was 0.8 ms of it).  What is left is bound by the L2
// traffic of the edge pass (147 us) and of the reverse-edge search (99 us),
// and by the launches of the levels and hops.
#include <math.h>

#include <vector>

#include "common.cuh"

namespace xmgn {

__global__ void csc_perm_kernel(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                const int32_t* __restrict__ recv, const int32_t* __restrict__ key,
                                int64_t n, int64_t e, int64_t cap, const int32_t* __restrict__ bad,
                                int32_t* __restrict__ perm, uint32_t* err);
xmgn_status quantize_launch(const float* xyz, int64_t n, double scale, int32_t* q, int32_t* bbox,
                            uint32_t* err, cudaStream_t s);

namespace {

constexpr int kIdBits = 28;          // node ids < 2^28
constexpr int kCoordBias = 1 << 24;  // lattice coordinate + bias is in [0, 2^25)
constexpr int kHistSmem = 16384;     // histogram words a block may keep in shared memory
constexpr int kMaxBins = 1024;

// ---- recursive coordinate bisection
// One segment of a level's plan: its first nl nodes in (coordinate, id) order
// go to segment `child` of the next level and the others to child + 1; a
// segment of one part (split = 0) moves to `child` whole.
struct RcbSeg {
  int64_t nl;
  int32_t child, split;
};
// Selection state: the key digits found so far and the rank still to go
// among the nodes that match them.  rank 0 ends it: no matching node is to go
// left, so the remaining (lower) digits stay zero.
struct RcbState {
  int64_t rank;
  int32_t axis, coord, id, split;
};

__global__ void rcb_begin_kernel(const int32_t* __restrict__ ext, const RcbSeg* __restrict__ plan, int nseg,
                                 RcbState* __restrict__ st, int32_t* __restrict__ next_ext, int nnext) {
  pdl_wait();
  pdl_trigger();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nnext; i += gridDim.x * blockDim.x)
    for (int a = 0; a < 3; ++a) {
      next_ext[6 * i + a] = INT32_MAX;
      next_ext[6 * i + 3 + a] = INT32_MIN;
    }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nseg; i += gridDim.x * blockDim.x) {
    RcbState t;
    t.rank = plan[i].nl;
    t.split = plan[i].split;
    t.coord = t.id = t.axis = 0;
    int64_t best = -1;
    for (int a = 0; a < 3; ++a) {  // the axis of largest extent, the lowest on ties
      const int64_t e = int64_t(ext[6 * i + 3 + a]) - ext[6 * i + a];
      if (e > best) best = e, t.axis = a;
    }
    st[i] = t;
  }
}

// Histogram of one key digit over the nodes of every segment that match the
// digits found so far.  Equal bins within a warp (neighbouring ids are
// neighbouring points) are added at once.  Small histograms are summed per
// block in shared memory first.
template <bool SMEM>
__global__ void __launch_bounds__(1024) rcb_hist_kernel(const int32_t* __restrict__ seg, int64_t n,
                                                        const int32_t* __restrict__ q,
                                                        const RcbState* __restrict__ st, int nseg, int on_id,
                                                        int shift, int bits, uint32_t* __restrict__ hist) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ uint32_t sh[];
  const int nb = 1 << bits;
  if (SMEM) {
    bool any = false;
    for (int i = threadIdx.x; i < nseg; i += blockDim.x) any |= st[i].split && st[i].rank > 0;
    if (!__syncthreads_or(any)) return;  // every key is found
    for (int i = threadIdx.x; i < nseg * nb; i += blockDim.x) sh[i] = 0u;
    __syncthreads();
  }
  for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n; v += int64_t(gridDim.x) * blockDim.x) {
    const int s = seg ? seg[v] : 0;
    const RcbState t = st[s];
    int bin = -1;
    if (t.split && t.rank > 0) {
      const int c = q[3 * v + t.axis] + kCoordBias;
      if (on_id) {
        if (c == t.coord && (int(v) >> (shift + bits)) == (t.id >> (shift + bits))) bin = (int(v) >> shift) & (nb - 1);
      } else if ((c >> (shift + bits)) == (t.coord >> (shift + bits))) {
        bin = (c >> shift) & (nb - 1);
      }
    }
    if (bin >= 0) {
      const uint32_t at = uint32_t(s) * uint32_t(nb) + uint32_t(bin);
      const unsigned same = __match_any_sync(__activemask(), at);
      if ((threadIdx.x & 31) == unsigned(__ffs(same) - 1))
        atomicAdd(SMEM ? &sh[at] : &hist[at], uint32_t(__popc(same)));
    }
  }
  if (SMEM) {
    __syncthreads();
    for (int i = threadIdx.x; i < nseg * nb; i += blockDim.x)
      if (sh[i]) atomicAdd(&hist[i], sh[i]);
  }
}

// A block per segment: the bin that holds the wanted rank becomes the next
// digit.  Leaves the histogram zeroed for the next pass.
__global__ void __launch_bounds__(256) rcb_find_kernel(RcbState* __restrict__ st, int on_id, int shift, int bits,
                                                       uint32_t* __restrict__ hist) {
  pdl_wait();
  pdl_trigger();
  __shared__ uint32_t wsum[8];
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const RcbState t = st[s];
  if (!t.split || t.rank <= 0) return;
  const int nb = 1 << bits, per = nb > 256 ? nb / 256 : 1;
  uint32_t* h = hist + int64_t(s) * nb;
  uint32_t c[kMaxBins / 256], sum = 0;
#pragma unroll
  for (int j = 0; j < kMaxBins / 256; ++j) {
    const int b = tid * per + j;
    c[j] = (j < per && b < nb) ? h[b] : 0u;
    if (j < per && b < nb) h[b] = 0u;
    sum += c[j];
  }
  uint32_t x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  uint32_t before = x - sum;
  for (int i = 0; i < w; ++i) before += wsum[i];
  const uint32_t rank = uint32_t(t.rank);
#pragma unroll
  for (int j = 0; j < kMaxBins / 256; ++j) {
    if (before <= rank && rank < before + c[j]) {  // true for exactly one bin
      if (on_id) st[s].id = t.id | ((tid * per + j) << shift);
      else st[s].coord = t.coord | ((tid * per + j) << shift);
      st[s].rank = int64_t(rank - before);
    }
    before += c[j];
  }
}

// Nodes take their segment of the next level (or, at the last level, their
// part), and the next level's extents are formed: warps whose nodes share a
// segment reduce first, up to 256 segments are summed per block.
__global__ void __launch_bounds__(512) rcb_split_kernel(int32_t* __restrict__ seg, int first, int64_t n,
                                                        const int32_t* __restrict__ q,
                                                        const RcbState* __restrict__ st,
                                                        const RcbSeg* __restrict__ plan, int nnext,
                                                        int32_t* __restrict__ ext, const int32_t* __restrict__ base,
                                                        int32_t* __restrict__ part) {
  pdl_wait();
  pdl_trigger();
  __shared__ int32_t sx[256 * 6];
  const bool sm = !part && nnext <= 256;
  if (sm) {
    for (int i = threadIdx.x; i < nnext * 6; i += blockDim.x) sx[i] = (i % 6) < 3 ? INT32_MAX : INT32_MIN;
    __syncthreads();
  }
  int32_t* const e = sm ? sx : ext;
  const int64_t step = int64_t(gridDim.x) * blockDim.x;
  const int64_t n32 = (n + 31) & ~int64_t(31);
  for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n32; v += step) {  // whole warps
    int ns = -1;
    int c[3] = {0, 0, 0};
    if (v < n) {
      const int s = first ? 0 : seg[v];
      const RcbState t = st[s];
      const RcbSeg g = plan[s];
#pragma unroll
      for (int a = 0; a < 3; ++a) c[a] = q[3 * v + a];
      const int k = c[t.axis] + kCoordBias;
      ns = g.child + ((g.split && (k > t.coord || (k == t.coord && int(v) >= t.id))) ? 1 : 0);
      if (part) part[v] = base[ns];
      else seg[v] = ns;
    }
    if (part) continue;
    int same;
    __match_all_sync(0xffffffffu, ns, &same);
    if (same && ns >= 0) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int lo = __reduce_min_sync(0xffffffffu, c[a]), hi = __reduce_max_sync(0xffffffffu, c[a]);
        if ((threadIdx.x & 31) == 0) {
          if (lo < *(volatile int32_t*)&e[6 * ns + a]) atomicMin(&e[6 * ns + a], lo);
          if (hi > *(volatile int32_t*)&e[6 * ns + 3 + a]) atomicMax(&e[6 * ns + 3 + a], hi);
        }
      }
    } else if (ns >= 0) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (c[a] < *(volatile int32_t*)&e[6 * ns + a]) atomicMin(&e[6 * ns + a], c[a]);
        if (c[a] > *(volatile int32_t*)&e[6 * ns + 3 + a]) atomicMax(&e[6 * ns + 3 + a], c[a]);
      }
    }
  }
  if (sm) {
    __syncthreads();
    for (int i = threadIdx.x; i < nnext * 6; i += blockDim.x) {
      if ((i % 6) < 3) {
        if (sx[i] != INT32_MAX) atomicMin(&ext[i], sx[i]);
      } else {
        if (sx[i] != INT32_MIN) atomicMax(&ext[i], sx[i]);
      }
    }
  }
}

// ---- halo BFS
__device__ __forceinline__ uint64_t mkey(uint32_t p, uint32_t hop, uint32_t v) {
  return (uint64_t(p) << 40) | (uint64_t(hop) << 32) | uint64_t(v);
}

// Hop 0: a warp's 32 nodes are one mask word of each part among them, which
// this warp alone writes (no atomics).
__global__ void bfs_seed_kernel(const int32_t* __restrict__ part, int64_t n, int P, uint32_t* __restrict__ bits,
                                int64_t words, int32_t* __restrict__ map, uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  const int64_t n32 = (n + 31) & ~int64_t(31);
  for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n32; v += int64_t(gridDim.x) * blockDim.x) {
    int p = v < n ? part[v] : -1;
    if (p < -1 || p >= P) {
      dev_flag(err, DEV_ERR_GRAPH);
      p = -1;
    }
    const unsigned same = __match_any_sync(0xffffffffu, p);
    if (p < 0) continue;  // inner in no part (may still be another part's halo)
    map[int64_t(p) * n + v] = 0;
    if ((threadIdx.x & 31) == unsigned(__ffs(same) - 1)) bits[int64_t(p) * words + (v >> 5)] = same;
  }
}

// Claims of one hop go to consecutive positions of `list`, counted in cnt[h].
// A block collects them in shared memory and takes room with one counter
// update: one update per claim, or per warp, serialises on the counter (22-25
// us per hop at 25-50k claims, 7-8 us this way).
constexpr int kFound = 1024;
struct Claims {
  uint64_t* found;  // shared, kFound
  int* nfound;      // shared
  unsigned long long* pos0;  // shared
  uint64_t* list;
  unsigned long long* cnt;   // this hop's counter
  unsigned long long out;    // list position of this hop's run
  int64_t cap;
  uint32_t* err;
  __device__ __forceinline__ void store(unsigned long long pos, uint64_t key) const {
    if (int64_t(pos) < cap) list[pos] = key;
    else dev_flag(err, DEV_ERR_CAP);
  }
  __device__ __forceinline__ void add(uint64_t key) const {
    const int k = atomicAdd(nfound, 1);
    if (k < kFound) found[k] = key;
    else store(out + atomicAdd(cnt, 1ull), key);  // a step of many long rows: straight to the list
  }
  // By all threads of the block, after every add.  No thread passes the second
  // barrier, and so claims for the next step, before every thread has read the
  // count: with the barriers only where there is something to store, a thread
  // held back would read a claim of the next step and wait in them alone.
  __device__ __forceinline__ void flush() const {
    __syncthreads();
    const int k = *nfound < kFound ? *nfound : kFound;
    __syncthreads();
    if (k > 0) {  // the same in every thread
      if (threadIdx.x == 0) {
        *pos0 = out + atomicAdd(cnt, (unsigned long long)k);
        *nfound = 0;
      }
      __syncthreads();
      for (int i = threadIdx.x; i < k; i += blockDim.x) store(*pos0 + i, found[i]);
      __syncthreads();
    }
  }
};

// Claims node w for part p at hop h unless it already is a member.
__device__ __forceinline__ void claim(const Claims& c, uint32_t* bits, int64_t words, int32_t* map, int64_t n, int p,
                                      int32_t w, int h) {
  uint32_t* word = &bits[int64_t(p) * words + (w >> 5)];
  const uint32_t m = 1u << (w & 31);
  if ((__ldcg(word) & m) || (atomicOr(word, m) & m)) return;
  map[int64_t(p) * n + w] = h;
  c.add(mkey(uint32_t(p), uint32_t(h), uint32_t(w)));
}

// Hop 1 looks at every inner node, most of which have no neighbour outside
// their part: a thread per node, eight neighbours' parts read at once.
__global__ void __launch_bounds__(256) bfs_first_kernel(const int64_t* __restrict__ row_ptr,
                                                        const int32_t* __restrict__ col, int64_t n,
                                                        const int32_t* __restrict__ part, int P,
                                                        uint32_t* __restrict__ bits, int64_t words,
                                                        int32_t* __restrict__ map, uint64_t* __restrict__ list,
                                                        unsigned long long* __restrict__ cnt, int64_t cap,
                                                        uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  __shared__ uint64_t found[kFound];
  __shared__ int nfound;
  __shared__ unsigned long long pos0;
  const Claims c{found, &nfound, &pos0, list, cnt + 1, 0ull, cap, err};
  if (threadIdx.x == 0) nfound = 0;
  __syncthreads();
  for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n; v += int64_t(gridDim.x) * blockDim.x) {
    const int p = part[v];
    const int64_t e0 = row_ptr[v], e1 = row_ptr[v + 1];
    if (p < 0 || p >= P) continue;
    for (int64_t e = e0; e < e1; e += 8) {
      int32_t w[8], pw[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) w[q] = e + q < e1 ? col[e + q] : int32_t(v);
#pragma unroll
      for (int q = 0; q < 8; ++q) pw[q] = (w[q] >= 0 && w[q] < n) ? part[w[q]] : -2;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (pw[q] == p) continue;
        if (w[q] < 0 || w[q] >= n) dev_flag(err, DEV_ERR_GRAPH);
        else claim(c, bits, words, map, n, p, w[q], 1);
      }
    }
  }
  c.flush();
}

// Hop h >= 2: eight lanes per node of the last hop, a lane per neighbour.
// The nodes claimed in hop g are the g-th run of `list`, cnt[g] of them.
// Bound by a chain of five dependent L2 accesses.
__global__ void __launch_bounds__(256) bfs_round_kernel(const int64_t* __restrict__ row_ptr,
                                                        const int32_t* __restrict__ col, int64_t n,
                                                        uint32_t* __restrict__ bits, int64_t words,
                                                        int32_t* __restrict__ map, uint64_t* __restrict__ list,
                                                        unsigned long long* __restrict__ cnt, int h, int64_t cap,
                                                        uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  __shared__ uint64_t found[kFound];
  __shared__ int nfound;
  __shared__ unsigned long long pos0;
  const int lane = threadIdx.x & 31, l = threadIdx.x & 7;
  unsigned long long prev = 0, out = 0;  // list positions of hop h-1's and hop h's runs
  for (int g = 1 + lane; g < h; g += 32) {
    const unsigned long long k = cnt[g];
    if (g < h - 1) prev += k;
    out += k;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    prev += __shfl_xor_sync(0xffffffffu, prev, o);
    out += __shfl_xor_sync(0xffffffffu, out, o);
  }
  int64_t total = int64_t(out - prev);
  if (int64_t(prev) + total > cap) total = cap > int64_t(prev) ? cap - int64_t(prev) : 0;
  const Claims c{found, &nfound, &pos0, list, cnt + h, out, cap, err};
  if (threadIdx.x == 0) nfound = 0;
  __syncthreads();
  for (int64_t t0 = int64_t(blockIdx.x) * 32; t0 < total; t0 += int64_t(gridDim.x) * 32) {  // uniform over the block
    const int64_t t = t0 + (threadIdx.x >> 3);
    if (t < total) {
      const uint64_t key = list[prev + t];
      const int p = int(key >> 40);
      const uint32_t u = uint32_t(key);
      const int64_t ee = row_ptr[u + 1];
      for (int64_t e = row_ptr[u] + l; e < ee; e += 8) {
        const int32_t w = col[e];
        if (w < 0 || w >= n) dev_flag(err, DEV_ERR_GRAPH);
        else claim(c, bits, words, map, n, p, w, h);
      }
    }
    c.flush();
  }
}

// ---- batch order: stable counting sort of part p's set bits by hop
// A block covers 256 mask words (8192 ids) of part blockIdx.y, a warp 32 of
// them.  Counts go out in (part, hop, block) order, so that their scan gives
// every (part, hop, block) its first batch position.
__device__ __forceinline__ void count_hops(const uint32_t* __restrict__ bits, const int32_t* __restrict__ map,
                                           int64_t words, int64_t n, int L, uint32_t (*hist)[256], uint32_t& word) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t p = blockIdx.y, w0 = int64_t(blockIdx.x) * 256 + 32 * w;
  for (int i = lane; i <= L; i += 32) hist[w][i] = 0u;
  __syncwarp();
  word = w0 + lane < words ? bits[p * words + w0 + lane] : 0u;
  unsigned todo = __ballot_sync(0xffffffffu, word != 0u);
  while (todo) {
    const int k = __ffs(todo) - 1;
    todo &= todo - 1;
    const uint32_t m = __shfl_sync(0xffffffffu, word, k);
    const bool in = (m >> lane) & 1u;
    const int hop = in ? map[p * n + (w0 + k) * 32 + lane] : -1;
    const unsigned same = __match_any_sync(0xffffffffu, hop);
    if (in && lane == __ffs(same) - 1) hist[w][hop] += uint32_t(__popc(same));
    __syncwarp();
  }
}

__global__ void __launch_bounds__(256) hop_count_kernel(const uint32_t* __restrict__ bits,
                                                        const int32_t* __restrict__ map, int64_t words, int64_t n,
                                                        int L, int32_t* __restrict__ cnt) {
  pdl_wait();
  pdl_trigger();
  __shared__ uint32_t hist[8][256];
  uint32_t word;
  count_hops(bits, map, words, n, L, hist, word);
  __syncthreads();
  for (int h = threadIdx.x; h <= L; h += 256) {
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += hist[w][h];
    cnt[(int64_t(blockIdx.y) * (L + 1) + h) * gridDim.x + blockIdx.x] = int32_t(s);
  }
}

// Each member takes its batch position: map[p][v] = position (over the hop),
// members[position] = key, and the ids and hops when asked for.
__global__ void __launch_bounds__(256) hop_place_kernel(const uint32_t* __restrict__ bits, int32_t* __restrict__ map,
                                                        int64_t words, int64_t n, int L,
                                                        const int64_t* __restrict__ base,
                                                        uint64_t* __restrict__ members, int32_t* __restrict__ gid,
                                                        uint8_t* __restrict__ hops) {
  pdl_wait();
  pdl_trigger();
  __shared__ uint32_t hist[8][256];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t p = blockIdx.y, w0 = int64_t(blockIdx.x) * 256 + 32 * w;
  uint32_t word;
  count_hops(bits, map, words, n, L, hist, word);
  __syncthreads();
  for (int h = threadIdx.x; h <= L; h += 256) {  // first position of each warp's members of hop h
    uint32_t s = uint32_t(base[(p * (L + 1) + h) * gridDim.x + blockIdx.x]);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t c = hist[i][h];
      hist[i][h] = s;
      s += c;
    }
  }
  __syncthreads();
  unsigned todo = __ballot_sync(0xffffffffu, word != 0u);
  while (todo) {
    const int k = __ffs(todo) - 1;
    todo &= todo - 1;
    const uint32_t m = __shfl_sync(0xffffffffu, word, k);
    const bool in = (m >> lane) & 1u;
    const int64_t v = (w0 + k) * 32 + lane;
    const int hop = in ? map[p * n + v] : -1;
    const unsigned same = __match_any_sync(0xffffffffu, hop);
    uint32_t t = 0;
    if (in) t = hist[w][hop] + uint32_t(__popc(same & ((1u << lane) - 1u)));
    __syncwarp();
    if (in && lane == __ffs(same) - 1) hist[w][hop] += uint32_t(__popc(same));
    __syncwarp();
    if (in) {
      map[p * n + v] = int32_t(t);
      members[t] = mkey(uint32_t(p), uint32_t(hop), uint32_t(v));
      if (gid) gid[t] = int32_t(v);
      if (hops) hops[t] = uint8_t(hop);
    }
  }
}

// info = [members, error word, node_ptr of every part, inner nodes of every part]
__global__ void part_sizes_kernel(const int64_t* __restrict__ base, int64_t nblk, int P, int L,
                                  const uint32_t* __restrict__ err, int64_t* __restrict__ info) {
  pdl_wait();
  pdl_trigger();
  const int64_t row = int64_t(L + 1) * nblk;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p <= P; p += gridDim.x * blockDim.x) {
    info[2 + p] = base[p * row];
    if (p < P) info[2 + P + 1 + p] = base[p * row + nblk] - base[p * row];
    if (p == 0) {
      info[0] = base[P * row];
      info[1] = int64_t(*err);
    }
  }
}

__global__ void part_edges_kernel(const int64_t* __restrict__ brp, const int64_t* __restrict__ node_ptr, int P,
                                  int64_t* __restrict__ edge_ptr) {
  pdl_wait();
  pdl_trigger();
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p <= P; p += gridDim.x * blockDim.x)
    edge_ptr[p] = brp[node_ptr[p]];
}

__global__ void batch_ids_kernel(const uint64_t* __restrict__ members, int64_t nb, int32_t* __restrict__ gid,
                                 uint8_t* __restrict__ hop) {
  pdl_wait();
  pdl_trigger();
  for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < nb; t += int64_t(gridDim.x) * blockDim.x) {
    const uint64_t key = members[t];
    gid[t] = int32_t(uint32_t(key));
    hop[t] = uint8_t(key >> 32);
  }
}

// Whether w is in part p (its bit; out-of-range ids are flagged and in no part).
__device__ __forceinline__ bool is_member(const uint32_t* __restrict__ bits, int64_t words, int64_t n, int64_t p,
                                          int32_t w, uint32_t* err) {
  if (w < 0 || w >= n) {
    dev_flag(err, DEV_ERR_GRAPH);
    return false;
  }
  return (bits[p * words + (w >> 5)] >> (w & 31)) & 1u;
}

// Degrees in the batch: every neighbour of a node short of the last hop is a
// member, so only last-hop rows are tested.
__global__ void batch_deg_kernel(const uint64_t* __restrict__ members, int64_t nb, int64_t n, int L,
                                 const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                 const uint32_t* __restrict__ bits, int64_t words, int32_t* __restrict__ deg,
                                 uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < nb; t += int64_t(gridDim.x) * blockDim.x) {
    const uint64_t key = members[t];
    const uint32_t v = uint32_t(key);
    const int64_t p = int64_t(key >> 40);
    const int64_t e0 = row_ptr[v], e1 = row_ptr[v + 1];
    int32_t d = int32_t(e1 - e0);
    if (int((key >> 32) & 0xff) == L) {
      d = 0;
      for (int64_t e = e0; e < e1; ++e) d += is_member(bits, words, n, p, col[e], err);
    }
    deg[t] = d;
  }
}

// Edges of the batch, eight lanes per node: its neighbours that are members,
// in row order.  Two nodes in flight per group of lanes (a chain of four
// dependent reads each).
__global__ void __launch_bounds__(256) batch_edges_kernel(const uint64_t* __restrict__ members, int64_t nb, int64_t n,
                                                          const int64_t* __restrict__ row_ptr,
                                                          const int32_t* __restrict__ col,
                                                          const int32_t* __restrict__ map,
                                                          const uint32_t* __restrict__ bits, int64_t words, int L,
                                                          const int64_t* __restrict__ brp, int32_t* __restrict__ bcol,
                                                          int32_t* __restrict__ brecv, uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  constexpr int U = 2;
  const int lane = threadIdx.x & 31, sub = lane >> 3, l = lane & 7;
  const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t t0 = warp * 4 * U; t0 < nb; t0 += nw * 4 * U) {
    uint64_t key[U];
    int64_t e[U], ee[U], o[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t t = t0 + 4 * u + sub;
      key[u] = t < nb ? members[t] : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t t = t0 + 4 * u + sub;
      const uint32_t v = uint32_t(key[u]);
      e[u] = t < nb ? row_ptr[v] + l : 0;
      ee[u] = t < nb ? row_ptr[v + 1] : 0;
      o[u] = t < nb ? brp[t] : 0;
    }
    bool more = true;
    while (more) {  // 16 neighbours per node and step (a row seldom has more)
      int32_t w[U][2], b[U][2];
      bool in[U][2];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < 2; ++k) w[u][k] = e[u] + 8 * k < ee[u] ? col[e[u] + 8 * k] : -1;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t p = int64_t(key[u] >> 40);
        const bool last = int((key[u] >> 32) & 0xff) == L;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          in[u][k] = e[u] + 8 * k < ee[u];
          if (in[u][k]) in[u][k] = last ? is_member(bits, words, n, p, w[u][k], err) : (w[u][k] >= 0 && w[u][k] < n);
          b[u][k] = in[u][k] ? map[p * n + w[u][k]] : 0;
        }
      }
      more = false;
#pragma unroll
      for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const unsigned got = (__ballot_sync(0xffffffffu, in[u][k]) >> (8 * sub)) & 0xffu;
          if (in[u][k]) {
            const int64_t at = o[u] + __popc(got & ((1u << l) - 1u));
            bcol[at] = b[u][k];
            brecv[at] = int32_t(t0 + 4 * u + sub);
          }
          o[u] += __popc(got);
        }
        e[u] += 16;
        more |= e[u] < ee[u];
      }
      more = __any_sync(0xffffffffu, more);
    }
  }
}

struct PartLayout {
  int32_t* q;
  int32_t* bbox;
  int32_t* part;       // part ids of the bisection
  int32_t* seg;        // bisection segment of each node
  int32_t* ext[2];     // 6 per segment, of this level and the next
  RcbSeg* plan;        // all levels
  RcbState* state;     // per segment
  int32_t* base;       // part of each last-level segment
  uint32_t* hist;      // kMaxBins per segment
  uint32_t* bits;      // P x words
  uint64_t* members;   // cap (during the search: the halo claims in hop order)
  unsigned long long* counters;  // claims of each hop
  int32_t* map;        // P x N: hop, then batch position (valid where the bit is set)
  int32_t* hcnt;       // P x (L + 1) x blocks
  int64_t* hbase;
  int64_t* info;       // part_sizes_kernel, then P + 1 edge offsets
  int32_t* deg;        // cap
  int64_t* brp;        // cap + 1
  int64_t* scan_tmp;
  int64_t* stamp;      // [8]: what the last sizing pass left in this workspace (see kStampMagic)
  int64_t cap;
};

// Written by a completed sizing pass, checked by the emit pass that resumes
// from it: magic, N, E, P, hops, batch nodes, batch edges, part_in given.
constexpr int64_t kStampMagic = 0x78686c6f73697a65;

int64_t member_cap(int64_t N, int32_t P) {
  int64_t c = int64_t(P) * N;
  int64_t lim = 8 * N + 4096;
  return c < lim ? c : lim;
}

int64_t hop_blocks(int64_t N) { return ((N + 31) / 32 + 255) / 256; }

void part_layout(Arena& A, int64_t N, int32_t P, PartLayout& w) {
  const int64_t words = (N + 31) / 32;
  const int64_t hc = int64_t(P) * 256 * hop_blocks(N);  // any halo depth
  w.cap = member_cap(N, P);
  w.q = A.take<int32_t>(size_t(3 * N));
  w.bbox = A.take<int32_t>(8);
  w.part = A.take<int32_t>(size_t(N));
  w.seg = A.take<int32_t>(size_t(N));
  for (int i = 0; i < 2; ++i) w.ext[i] = A.take<int32_t>(size_t(6) * (P + 1));
  w.plan = A.take<RcbSeg>(size_t(3) * P + 64);
  w.state = A.take<RcbState>(size_t(P + 1));
  w.base = A.take<int32_t>(size_t(P + 1));
  w.hist = A.take<uint32_t>(size_t(P) * kMaxBins);
  w.bits = A.take<uint32_t>(size_t(int64_t(P) * words));
  w.members = A.take<uint64_t>(size_t(w.cap));
  w.counters = A.take<unsigned long long>(260);
  w.map = A.take<int32_t>(size_t(int64_t(P) * N));
  w.hcnt = A.take<int32_t>(size_t(hc));
  w.hbase = A.take<int64_t>(size_t(hc + 1));
  w.info = A.take<int64_t>(size_t(3) * P + 8);
  w.deg = A.take<int32_t>(size_t(w.cap));
  w.brp = A.take<int64_t>(size_t(w.cap + 1));
  w.scan_tmp = A.take<int64_t>(scan_tmp_elems((w.cap > hc ? w.cap : hc) + 1) + 16);
  w.stamp = A.take<int64_t>(8);
}

struct Seg {
  int64_t size;
  int32_t parts, base;
};

// The host side of a bisection's plan.  The copies of it are asynchronous, and
// where the GPU reads pageable memory itself nothing stages them: the arrays live
// until the stream has been waited for.
struct HostPlan {
  std::vector<RcbSeg> plan;
  std::vector<int32_t> base;
  cudaStream_t s = nullptr;
  bool pending = false;
  ~HostPlan() {
    if (pending) cudaStreamSynchronize(s);  // an error on the way to the caller's wait
  }
};

// Parts by recursive coordinate bisection: part ids of all nodes into `part`,
// no host synchronisation (a coordinate off the lattice is flagged in err).  The
// caller keeps `host` and clears its `pending` once it has waited for the stream.
xmgn_status bisect(const float* xyz, int64_t N, double scale, int32_t P, PartLayout& w, int32_t* part, uint32_t* err,
                   HostPlan& host, cudaStream_t s) {
  XMGN_TRY(quantize_launch(xyz, N, scale, w.q, w.bbox, err, s));
  if (P == 1) {
    XMGN_CUDA(cudaMemsetAsync(part, 0, sizeof(int32_t) * size_t(N), s));
    return XMGN_OK;
  }
  std::vector<RcbSeg>& plan = host.plan;
  std::vector<int> level;  // first plan entry of each level
  std::vector<Seg> segs{{N, P, 0}};
  for (bool any = true; any;) {
    any = false;
    std::vector<Seg> next;
    level.push_back(int(plan.size()));
    for (const Seg& g : segs) {
      RcbSeg r{0, int32_t(next.size()), g.parts > 1 ? 1 : 0};
      if (g.parts == 1) {
        next.push_back(g);
      } else {
        const int32_t pl = g.parts / 2;
        r.nl = (g.size * pl) / g.parts;
        next.push_back({r.nl, pl, g.base});
        next.push_back({g.size - r.nl, g.parts - pl, g.base + pl});
      }
      plan.push_back(r);
    }
    segs.swap(next);
    for (const Seg& g : segs) any |= g.parts > 1;
  }
  level.push_back(int(plan.size()));
  std::vector<int32_t>& base = host.base;
  base.resize(segs.size());
  for (size_t i = 0; i < segs.size(); ++i) base[i] = segs[i].base;
  host.s = s;
  host.pending = true;
  XMGN_CUDA(cudaMemcpyAsync(w.plan, plan.data(), sizeof(RcbSeg) * plan.size(), cudaMemcpyHostToDevice, s));
  XMGN_CUDA(cudaMemcpyAsync(w.base, base.data(), sizeof(int32_t) * base.size(), cudaMemcpyHostToDevice, s));
  XMGN_CUDA(cudaMemsetAsync(w.hist, 0, sizeof(uint32_t) * size_t(P) * kMaxBins, s));
  static std::atomic<uint64_t> attr{0};  // devices
  XMGN_TRY(once_per_device(attr, [] {
    XMGN_CUDA(cudaFuncSetAttribute(rcb_hist_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kHistSmem * 4));
    return XMGN_OK;
  }));
  // digits of the 53-bit key, high to low: 25 coordinate bits, then as many id bits as N needs
  struct Digit {
    int on_id, shift, bits;
  };
  std::vector<Digit> digits = {{0, 16, 9}, {0, 8, 8}, {0, 0, 8}};
  int idb = 1;
  while ((int64_t(1) << idb) < N) ++idb;
  for (int hi = idb; hi > 0;) {
    const int b = hi > 10 ? 10 : hi;
    digits.push_back({1, hi - b, b});
    hi -= b;
  }
  const int nl = int(level.size()) - 1;
  for (int l = 0; l < nl; ++l) {
    const int nseg = level[l + 1] - level[l];
    const int nnext = l + 1 < nl ? level[l + 2] - level[l + 1] : int(segs.size());
    const RcbSeg* pl = w.plan + level[l];
    const int32_t* ext = l ? w.ext[l & 1] : w.bbox;
    const bool last = l + 1 == nl;
    launch_pdl(rcb_begin_kernel, grid_for(nnext, 256), 256, 0, s, ext, pl, nseg, w.state, w.ext[(l + 1) & 1], nnext);
    XMGN_LAUNCH_CHECK();
    for (const Digit& d : digits) {
      const int words = nseg << d.bits;
      const int32_t* seg = l ? w.seg : nullptr;
      // one histogram per block in shared memory while all segments' fit; with more segments the
      // atomics spread over that many more addresses and go to memory
      if (words <= kHistSmem)
        launch_pdl(rcb_hist_kernel<true>, grid_for(N, 1024, int64_t(num_sms()) * 2), 1024, size_t(words) * 4, s, seg, N,
                   w.q, w.state, nseg, d.on_id, d.shift, d.bits, w.hist);
      else
        launch_pdl(rcb_hist_kernel<false>, grid_for(N, 1024, int64_t(num_sms()) * 2), 1024, 0, s, seg, N, w.q, w.state,
                   nseg, d.on_id, d.shift, d.bits, w.hist);
      XMGN_LAUNCH_CHECK();
      launch_pdl(rcb_find_kernel, unsigned(nseg), 256, 0, s, w.state, d.on_id, d.shift, d.bits, w.hist);
      XMGN_LAUNCH_CHECK();
    }
    launch_pdl(rcb_split_kernel, grid_for(N, 512, int64_t(num_sms()) * 4), 512, 0, s, w.seg, l == 0 ? 1 : 0, N, w.q,
               w.state, pl, nnext, w.ext[(l + 1) & 1], w.base, last ? part : nullptr);
    XMGN_LAUNCH_CHECK();
  }
  return XMGN_OK;
}

}  // namespace

xmgn_status partition_halo_ws(int64_t N, int64_t E, int32_t P, size_t* ws_bytes) {
  (void)E;
  Arena A;
  A.dry = true;
  PartLayout w;
  part_layout(A, N, P, w);
  *ws_bytes = A.used + 256;
  return XMGN_OK;
}

xmgn_status partition_halo(const int64_t* row_ptr, const int32_t* col, int64_t N, int64_t E,
                           const float* xyz, double scale, int32_t P, int32_t L,
                           const int32_t* part_in, void* ws, size_t ws_bytes, int32_t* part_out,
                           int64_t* node_ptr, int64_t* edge_ptr, int64_t* inner_cnt, int32_t* gid,
                           uint8_t* hop, int64_t* b_row_ptr, int32_t* b_col, int32_t* b_recv,
                           int32_t* b_csc_perm, int64_t cap_nodes, int64_t cap_edges,
                           cudaStream_t s, bool resume) {
  if (!row_ptr || !col || !ws || !node_ptr || !edge_ptr || !inner_cnt)
    return fail(XMGN_ERR_ARG, "null pointer");
  if (P < 1 || P > 65535 || int64_t(P) > N) return fail(XMGN_ERR_ARG, "need 1 <= P <= min(N, 65535)");
  if (L < 0 || L > 255) return fail(XMGN_ERR_ARG, "halo_hops must be in [0, 255]");
  if (N < 1 || N >= (int64_t(1) << kIdBits)) return fail(XMGN_ERR_ARG, "N must be in [1, 2^28)");
  if (!part_in && !xyz) return fail(XMGN_ERR_ARG, "xyz required for RCB");
  const bool emit = gid != nullptr;
  if (emit && (!b_row_ptr || !b_col || !b_recv || !hop))
    return fail(XMGN_ERR_ARG, "emit pass needs gid, hop, b_row_ptr, b_col, b_recv");

  Arena A;
  A.base = static_cast<char*>(ws);
  A.cap = ws_bytes;
  PartLayout w;
  part_layout(A, N, P, w);
  if (!A.ok()) return fail(XMGN_ERR_WORKSPACE, "partition workspace too small: need %zu", A.used);
  uint32_t* err = device_error_word();
  const int32_t* part = part_in ? part_in : w.part;
  const int64_t words = (N + 31) / 32;
  // edges and the CSC permutation, once ids and row offsets are in place
  auto emit_edges = [&](int64_t nb, int64_t eb) -> xmgn_status {
    if (nb > 0) {
      launch_pdl(batch_edges_kernel, grid_for(nb * 4, 256), 256, 0, s, w.members, nb, N, row_ptr, col, w.map, w.bits,
                 words, L, b_row_ptr, b_col, b_recv, err);
      XMGN_LAUNCH_CHECK();
    }
    if (b_csc_perm && eb > 0) {
      launch_pdl(csc_perm_kernel, grid_for((eb + 3) / 4, 256), 256, 0, s, b_row_ptr, b_col, b_recv, gid, nb, eb, eb,
                 nullptr, b_csc_perm, err);
      XMGN_LAUNCH_CHECK();
    }
    XMGN_CUDA(cudaMemsetAsync(w.stamp, 0, sizeof(int64_t) * 8, s));  // one emit per sizing pass
    XMGN_CUDA(cudaStreamSynchronize(s));
    return XMGN_OK;
  };
  if (resume) {
    if (!emit) return fail(XMGN_ERR_ARG, "the emit pass needs gid, hop, b_row_ptr, b_col, b_recv");
    int64_t st[8];
    XMGN_CUDA(cudaMemcpyAsync(st, w.stamp, sizeof(st), cudaMemcpyDeviceToHost, s));
    XMGN_CUDA(cudaStreamSynchronize(s));
    if (st[0] != kStampMagic || st[1] != N || st[2] != E || st[3] != P || st[4] != L || st[5] != node_ptr[P] ||
        st[6] != edge_ptr[P] || st[7] != (part_in ? 1 : 0))
      return fail(XMGN_ERR_ARG, "partition emit pass: the workspace holds no sizing pass of these inputs");
    const int64_t nb = node_ptr[P], eb = edge_ptr[P];
    if (cap_nodes < nb) return fail(XMGN_ERR_WORKSPACE, "cap_nodes %lld < %lld", (long long)cap_nodes, (long long)nb);
    if (cap_edges < eb) return fail(XMGN_ERR_WORKSPACE, "cap_edges %lld < %lld", (long long)cap_edges, (long long)eb);
    if (nb > 0) {  // the sizing pass left members, map, mask and row offsets
      launch_pdl(batch_ids_kernel, grid_for(nb, 256), 256, 0, s, w.members, nb, gid, hop);
      XMGN_LAUNCH_CHECK();
    }
    XMGN_CUDA(cudaMemcpyAsync(b_row_ptr, w.brp, sizeof(int64_t) * size_t(nb + 1), cudaMemcpyDeviceToDevice, s));
    return emit_edges(nb, eb);
  }

  XMGN_CUDA(cudaMemsetAsync(w.stamp, 0, sizeof(int64_t) * 8, s));  // this pass replaces what an earlier one left
  // ---------------- parts
  HostPlan host;
  if (!part_in) XMGN_TRY(bisect(xyz, N, scale, P, w, w.part, err, host, s));

  // ---------------- halo BFS
  XMGN_CUDA(cudaMemsetAsync(w.bits, 0, sizeof(uint32_t) * size_t(int64_t(P) * words), s));
  XMGN_CUDA(cudaMemsetAsync(w.counters, 0, sizeof(unsigned long long) * 260, s));
  launch_pdl(bfs_seed_kernel, grid_for(N, 256), 256, 0, s, part, N, P, w.bits, words, w.map, err);
  XMGN_LAUNCH_CHECK();
  if (L > 0) {
    launch_pdl(bfs_first_kernel, grid_for(N, 256, int64_t(num_sms()) * 8), 256, 0, s, row_ptr, col, N, part, P, w.bits,
               words, w.map, w.members, w.counters, w.cap, err);
    XMGN_LAUNCH_CHECK();
  }
  for (int h = 2; h <= L; ++h) {
    launch_pdl(bfs_round_kernel, grid_for(N * 8, 256, int64_t(num_sms()) * 8), 256, 0, s, row_ptr, col, N, w.bits,
               words, w.map, w.members, w.counters, h, w.cap, err);
    XMGN_LAUNCH_CHECK();
  }

  // ---------------- batch order and sizes
  const int64_t nblk = hop_blocks(N), hc = int64_t(P) * (L + 1) * nblk;
  const dim3 hgrid(static_cast<unsigned>(nblk), static_cast<unsigned>(P));
  launch_pdl(hop_count_kernel, hgrid, 256, 0, s, w.bits, w.map, words, N, L, w.hcnt);
  XMGN_LAUNCH_CHECK();
  XMGN_TRY(exclusive_scan_i32(w.hcnt, w.hbase, hc, w.scan_tmp, s));
  launch_pdl(part_sizes_kernel, grid_for(P + 1, 256), 256, 0, s, w.hbase, nblk, P, L, err, w.info);
  XMGN_LAUNCH_CHECK();
  std::vector<int64_t> info(size_t(2) * P + 3);
  XMGN_CUDA(cudaMemcpyAsync(info.data(), w.info, sizeof(int64_t) * info.size(), cudaMemcpyDeviceToHost, s));
  XMGN_CUDA(cudaStreamSynchronize(s));
  host.pending = false;
  const int64_t nb = info[0];
  const uint32_t herr = uint32_t(info[1]) & (DEV_ERR_CAP | DEV_ERR_GRAPH | (part_in ? 0u : DEV_ERR_RANGE));
  if (herr || nb > w.cap) {
    XMGN_CUDA(cudaMemsetAsync(err, 0, sizeof(uint32_t), s));
    if (herr & DEV_ERR_RANGE) return fail(XMGN_ERR_RANGE, "coordinate outside the lattice range");
    if (herr & DEV_ERR_GRAPH) return fail(XMGN_ERR_GRAPH, "part id or sender id out of range");
    return fail(XMGN_ERR_WORKSPACE, "halo members exceed the workspace capacity (%lld)", (long long)w.cap);
  }
  if (part_out && part_out != part)  // only now: bad coordinates or ids leave it alone
    XMGN_CUDA(cudaMemcpyAsync(part_out, part, sizeof(int32_t) * size_t(N), cudaMemcpyDeviceToDevice, s));
  if (emit && cap_nodes < nb) return fail(XMGN_ERR_WORKSPACE, "cap_nodes %lld < %lld", (long long)cap_nodes, (long long)nb);
  for (int p = 0; p <= P; ++p) node_ptr[p] = info[2 + p];
  for (int p = 0; p < P; ++p) inner_cnt[p] = info[3 + P + p];

  // ---------------- batch nodes and degrees
  launch_pdl(hop_place_kernel, hgrid, 256, 0, s, w.bits, w.map, words, N, L, w.hbase, w.members, emit ? gid : nullptr,
             emit ? hop : nullptr);
  XMGN_LAUNCH_CHECK();
  if (nb > 0) {
    launch_pdl(batch_deg_kernel, grid_for(nb, 256), 256, 0, s, w.members, nb, N, L, row_ptr, col, w.bits, words, w.deg,
               err);
    XMGN_LAUNCH_CHECK();
  }
  int64_t* brp = emit ? b_row_ptr : w.brp;
  XMGN_TRY(exclusive_scan_i32(w.deg, brp, nb, w.scan_tmp, s));
  int64_t* d_edge_ptr = w.info + 2 * int64_t(P) + 3;
  launch_pdl(part_edges_kernel, grid_for(P + 1, 256), 256, 0, s, brp, w.info + 2, P, d_edge_ptr);
  XMGN_LAUNCH_CHECK();
  XMGN_CUDA(cudaMemcpyAsync(edge_ptr, d_edge_ptr, sizeof(int64_t) * size_t(P + 1), cudaMemcpyDeviceToHost, s));
  XMGN_CUDA(cudaStreamSynchronize(s));
  if (!emit) {  // leave the stamp that lets an emit pass resume from this one
    const int64_t st[8] = {kStampMagic, N, E, P, L, node_ptr[P], edge_ptr[P], part_in ? 1 : 0};
    XMGN_CUDA(cudaMemcpyAsync(w.stamp, st, sizeof(st), cudaMemcpyHostToDevice, s));
    XMGN_CUDA(cudaStreamSynchronize(s));
    return XMGN_OK;
  }
  const int64_t eb = edge_ptr[P];
  if (cap_edges < eb) return fail(XMGN_ERR_WORKSPACE, "cap_edges %lld < %lld", (long long)cap_edges, (long long)eb);
  return emit_edges(nb, eb);
}

}  // namespace xmgn
