// kNN graph construction (Sec. III-B "K-Nearest Neighbor Connectivity") and
// symmetrisation into receiver-major CSR.
//
// Exactness: coordinates are mapped to the integer lattice q = rint(x*s) with
// s a power of two, so x*s is exact in float32 and rintf gives the same
// round-half-even result as any exact reference; squared distances are int64.
// Candidates are ranked by (d^2, index), so the result is unique and
// independent of thread scheduling.
//
// Search: uniform grid over the lattice bounding box, points counting-sorted
// into cells with their coordinates (16 bytes each), then for each point the
// block of cells at Chebyshev distance <= 1 and after it rings r = 2, 3, ... are
// scanned.  Any point outside the scanned block differs along some axis by at
// least the distance from the point to that face of the block, so the search
// stops once k candidates are nearer than the nearest face that has cells
// behind it.
//
// The whole build runs on the stream with one host wait at its end: the grid
// is laid out on the device from the bounding box, and the rows are emitted
// only if they fit the caller's capacity, which the host reports afterwards.
// A coordinate off the lattice ends the work at once all the same: it sets a
// flag of the call (bbox[6]), and every later kernel leaves when it is set, so
// that no time goes into a cloud whose points have fallen together and no
// output array is touched.
#include <math.h>

#include "common.cuh"

namespace xmgn {

namespace {
constexpr int kMaxK = 32;

// bbox: least and greatest lattice coordinate per axis, [6]: a coordinate is off the lattice.
__global__ void quantize_kernel(const float* __restrict__ xyz, int64_t n, float scale,
                                int32_t* __restrict__ q, int32_t* __restrict__ bbox,
                                uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  int lo[3] = {INT32_MAX, INT32_MAX, INT32_MAX}, hi[3] = {INT32_MIN, INT32_MIN, INT32_MIN};
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float v = rintf(xyz[3 * i + a] * scale);  // exact product (power-of-two scale)
      int32_t qi = 0;
      if (!(fabsf(v) < 16777216.0f)) {  // also catches NaN / inf
        dev_flag(err, DEV_ERR_RANGE);
        bbox[6] = 1;
      } else {
        qi = int32_t(v);
      }
      q[3 * i + a] = qi;
      lo[a] = min(lo[a], qi);
      hi[a] = max(hi[a], qi);
    }
  }
  // one update of the box per block: with one per warp the six words took
  // 155 us of serialised atomics at 2M points
  __shared__ int32_t box[6];
  if (threadIdx.x < 6) box[threadIdx.x] = threadIdx.x < 3 ? INT32_MAX : INT32_MIN;
  __syncthreads();
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int32_t l = __reduce_min_sync(0xffffffffu, lo[a]), h = __reduce_max_sync(0xffffffffu, hi[a]);
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&box[a], l);
      atomicMax(&box[3 + a], h);
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) atomicMin(&bbox[threadIdx.x], box[threadIdx.x]);
  else if (threadIdx.x < 6) atomicMax(&bbox[threadIdx.x], box[threadIdx.x]);
}

__global__ void bbox_init_kernel(int32_t* bbox) {
  pdl_wait();
  pdl_trigger();
  if (threadIdx.x < 3) {
    bbox[threadIdx.x] = INT32_MAX;
    bbox[3 + threadIdx.x] = INT32_MIN;
  } else if (threadIdx.x == 3) {
    bbox[6] = 0;
  }
}

// Uniform grid of one reference set.
struct Grid {
  int32_t lo[3];
  int32_t c;     // cell edge in lattice units
  int32_t g[3];  // cells per axis
  int32_t bad;   // bbox[6]
};
constexpr int kMaxLevels = 16;
struct LevelSizes {
  int64_t n[kMaxLevels];
};

// Cells of a grid over n points.  On a surface the points of an occupied cell
// grow as (n / cells)^(2/3) n^(1/3): two cells per point leave 2.5 points in an
// occupied cell at 2k points but 10 at 200k and 18 at 1.25M, so the cells per
// point grow with the square root of n up to six.  (Of the 6 n counters, the
// scan and the clearing cost 20 us at 1.25M points; the search there reads 9
// occupied cells per point.)
__host__ __device__ inline int64_t cell_budget(int64_t n) {
  double per = 2.0 * sqrt(double(n) / 8000.0);
  if (per < 2.0) per = 2.0;
  if (per > 6.0) per = 6.0;
  const int64_t b = int64_t(per * double(n)) + 1024;
  return b < (int64_t(1) << 30) ? b : (int64_t(1) << 30);
}

// The grid of every level (thread l: the first sizes.n[l] points) over the box
// of all points: at most cell_budget cells.
// A range error that the device's error word holds already counts as this
// call's, as the host reports it.
__global__ void grid_layout_kernel(int32_t* bbox, LevelSizes sizes, int levels, const uint32_t* __restrict__ err,
                                   Grid* __restrict__ out) {
  pdl_wait();
  pdl_trigger();
  const int l = threadIdx.x;
  if (l >= levels) return;
  const int32_t bad = (bbox[6] != 0 || (*err & DEV_ERR_RANGE)) ? 1 : 0;
  if (l == 0) bbox[6] = bad;
  const int64_t budget = cell_budget(sizes.n[l]);
  double vol = 1.0;
  Grid G;
  for (int a = 0; a < 3; ++a) {
    G.lo[a] = bbox[a];
    vol *= double(int64_t(bbox[3 + a]) - bbox[a] + 1);
  }
  double c = cbrt(vol / double(budget - 1024));
  if (c < 1) c = 1;
  int64_t e = int64_t(ceil(c));
  for (;;) {
    int64_t tot = 1;
    for (int a = 0; a < 3; ++a) {
      const int64_t g = (int64_t(bbox[3 + a]) - bbox[a]) / e + 1;
      G.g[a] = int32_t(g);
      tot *= g;
    }
    if (tot <= budget) break;
    e = e + e / 4 + 1;
  }
  G.c = int32_t(e);
  G.bad = bad;
  out[l] = G;
}

__device__ __forceinline__ int cell_coord(int32_t q, int32_t lo, int32_t c) {
  return int(uint32_t(q - lo) / uint32_t(c));
}

// Cell of every reference point, and its place among the cell's points.
__global__ void cell_count_kernel(const int32_t* __restrict__ q, int64_t n, const Grid* __restrict__ grid,
                                  int32_t* __restrict__ cell_of, int32_t* __restrict__ at, int32_t* __restrict__ cnt) {
  pdl_wait();
  pdl_trigger();
  const Grid G = *grid;
  if (G.bad) return;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int cx = cell_coord(q[3 * i], G.lo[0], G.c);
    const int cy = cell_coord(q[3 * i + 1], G.lo[1], G.c);
    const int cz = cell_coord(q[3 * i + 2], G.lo[2], G.c);
    const int32_t cell = (cz * G.g[1] + cy) * G.g[0] + cx;
    cell_of[i] = cell;
    at[i] = atomicAdd(&cnt[cell], 1);
  }
}

__global__ void cell_scatter_kernel(const int32_t* __restrict__ q, const int32_t* __restrict__ cell_of,
                                    const int32_t* __restrict__ at, int64_t n, const int32_t* __restrict__ start,
                                    const Grid* __restrict__ grid, int4* __restrict__ pts) {
  pdl_wait();
  pdl_trigger();
  if (grid->bad) return;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x)
    pts[start[cell_of[i]] + at[i]] = make_int4(q[3 * i], q[3 * i + 1], q[3 * i + 2], int32_t(i));
}

__device__ __forceinline__ bool key_less(int64_t d1, int32_t j1, int64_t d2, int32_t j2) {
  return d1 < d2 || (d1 == d2 && j1 < j2);
}

// The KC best candidates of one lane, ascending by (d^2, index), in registers.
template <int KC>
struct Best {
  int64_t d[KC];
  int32_t j[KC];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int a = 0; a < KC; ++a) d[a] = INT64_MAX, j[a] = INT32_MAX;
  }
  __device__ __forceinline__ void insert(int64_t dn, int32_t jn) {
    if (!key_less(dn, jn, d[KC - 1], j[KC - 1])) return;
    bool lt = true;  // new key < slot a
#pragma unroll
    for (int a = KC - 1; a > 0; --a) {
      const bool below = key_less(dn, jn, d[a - 1], j[a - 1]);
      d[a] = below ? d[a - 1] : (lt ? dn : d[a]);
      j[a] = below ? j[a - 1] : (lt ? jn : j[a]);
      lt = below;
    }
    if (lt) d[0] = dn, j[0] = jn;
  }
  __device__ __forceinline__ void pop() {
#pragma unroll
    for (int a = 0; a + 1 < KC; ++a) d[a] = d[a + 1], j[a] = j[a + 1];
    d[KC - 1] = INT64_MAX;
    j[KC - 1] = INT32_MAX;
  }
};

// The (y, z) rows of ring r >= 2 around a cell that lie in the grid and can hold
// cells of it: all rows of the clamped square, or, once both x faces are outside
// the grid, those on its rim only (an inner row has no cell but its two ends).
// So a point looks at no more rows than the grid has cells, also where the grid
// is thin and a far point needs many rings: with all (2r + 1)^2 rows of every
// ring, a point 2700 cells off a flat cloud would step through 2.6e10.
__device__ __forceinline__ int ring_rows(const Grid& g, int cx, int cy, int cz, int r) {
  const int ny = min(cy + r, g.g[1] - 1) - max(cy - r, 0) + 1, nz = min(cz + r, g.g[2] - 1) - max(cz - r, 0) + 1;
  if (cx - r >= 0 || cx + r < g.g[0]) return ny * nz;
  const int fy = (cy - r >= 0) + (cy + r < g.g[1]), fz = (cz - r >= 0) + (cz + r < g.g[2]);  // faces inside the grid
  return fz * ny + fy * (nz - fz);  // the rows of the z faces, then the two ends of the others
}
// Row `id` of them.  Called, not inlined, and with nothing kept between rows: most
// points need no such ring, and the registers would cost the search resident warps
// (three levels up to 1.25M points 1938 us, inlined 1953; 200k points on a
// line 55 -> 2.6 ms against all rows of every ring).
__device__ __noinline__ int2 ring_row(const Grid* grid, int cx, int cy, int cz, int r, int id) {
  const Grid g = *grid;
  int y, z;
  const int ylo = cy - r, yhi = cy + r, zlo = cz - r, zhi = cz + r;
  const int y0 = max(ylo, 0), z0 = max(zlo, 0), ny = min(yhi, g.g[1] - 1) - y0 + 1;
  y = y0 + id % ny;
  z = z0 + id / ny;
  if (cx - r >= 0 || cx + r < g.g[0]) return make_int2(y, z);
  const int fz = (zlo >= 0) + (zhi < g.g[2]);
  const int i = id - fz * ny;
  if (i < 0) {
    z = id < ny && zlo >= 0 ? zlo : zhi;
  } else {
    const int m = min(zhi, g.g[2] - 1) - z0 + 1 - fz;
    y = i < m && ylo >= 0 ? ylo : yhi;
    z = (zlo >= 0 ? z0 + 1 : z0) + i % m;
  }
  return make_int2(y, z);
}

template <int G>
__device__ __forceinline__ int group_get(uint32_t mask, int v, int l) {
  if constexpr (G == 1) return v;
  return __shfl_sync(mask, v, l, G);
}

// kNN among n_ref cell-sorted reference points.  QUERY false: of every
// reference point, in cell order (itself excluded); true: of the points
// q0..q1-1, which are not reference points but lie inside the grid.  A group
// of G lanes serves a point: each lane finds the cell ranges of one (y, z) row of
// the block (the cells of a row are neighbours in memory), then the lanes read
// every range together, each keeping the best of what it read; the lists are
// merged at the end.  Row i of the output is nbr[i*stride + off .. + k), -1 if
// missing.  rcnt[j] counts the rows that list j; rank[slot] is the slot's place
// among them (for the reverse edges).
//
// Bound by the latency of the dependent reads (range, then points).  Against a
// thread per point with its candidate list in local memory, the cell ids read
// first and the coordinates gathered: 114 -> 23 us at 2k points (eight lanes
// per point), 185 -> 86 us at 200k, and 1.43 -> 0.66 ms for the three levels up
// to 1.25M points.  Rows are read from the middle of the block out and left out
// when they are farther away than the k-th best so far (93 -> 85 us, 0.77 -> 0.64 ms).
template <int KC, int G, bool QUERY>
__global__ void __launch_bounds__(128, KC <= 6 ? 8 : KC == 8 ? 6 : 0)
    knn_kernel(const int32_t* __restrict__ q, const int4* __restrict__ pts, const int32_t* __restrict__ start,
               int64_t q0, int64_t q1, int k, const Grid* __restrict__ grid, int32_t* __restrict__ nbr, int64_t stride,
               int off, int32_t* __restrict__ rcnt, int32_t* __restrict__ rank) {
  pdl_wait();
  pdl_trigger();
  const Grid gr = *grid;
  if (gr.bad) return;
  const int lane = threadIdx.x & 31, gl = lane % G;
  const uint32_t mask = G == 1 ? 0u : ((G == 32 ? 0xffffffffu : ((1u << G) - 1u)) << (lane - gl));
  for (int64_t t = q0 + (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) / G; t < q1;
       t += int64_t(gridDim.x) * blockDim.x / G) {
    int4 p;
    if (QUERY)
      p = make_int4(q[3 * t], q[3 * t + 1], q[3 * t + 2], int32_t(t));
    else
      p = pts[t];
    const int cx = cell_coord(p.x, gr.lo[0], gr.c), cy = cell_coord(p.y, gr.lo[1], gr.c),
              cz = cell_coord(p.z, gr.lo[2], gr.c);
    const int64_t ry = int64_t(p.y) - gr.lo[1], rz = int64_t(p.z) - gr.lo[2];
    Best<KC> best;
    best.clear();
    auto scan = [&](int s, int e) {
      for (s += gl; s < e; s += G) {
        const int4 c = pts[s];
        const int32_t dx = c.x - p.x, dy = c.y - p.y, dz = c.z - p.z;
        const int64_t d = int64_t(dx) * dx + int64_t(dy) * dy + int64_t(dz) * dz;
        if (QUERY || c.w != p.w) best.insert(d, c.w);
      }
    };
    for (int r = 1;; ++r) {
      const int x0 = max(cx - r, 0), x1 = min(cx + r, gr.g[0] - 1);
      const int rows = r == 1 ? 9 : ring_rows(gr, cx, cy, cz, r);
      // This lane's row of the G rows from `base` on (the 3 x 3 rows of the first block from the middle out):
      // one range, or the two end cells of an inner row; far2: no point of the row is nearer than its root.
      int64_t far2 = 0;
      auto ranges = [&](int base) {
        int4 v = make_int4(0, 0, 0, 0);
        const int id = base + gl;
        int y, z;
        if (r == 1) {
          y = cy + int((0x22161u >> (2 * id)) & 3u) - 1;
          z = cz + int((0x28215u >> (2 * id)) & 3u) - 1;
        } else {
          const int2 w = ring_row(grid, cx, cy, cz, r, id);
          y = w.x, z = w.y;
        }
        const int dy = y - cy, dz = z - cz;
        if (id < rows && y >= 0 && y < gr.g[1] && z >= 0 && z < gr.g[2]) {
          const int64_t my = dy == 0 ? 0 : dy < 0 ? ry - int64_t(y + 1) * gr.c + 1 : int64_t(y) * gr.c - ry;
          const int64_t mz = dz == 0 ? 0 : dz < 0 ? rz - int64_t(z + 1) * gr.c + 1 : int64_t(z) * gr.c - rz;
          far2 = my * my + mz * mz;
          if (far2 > best.d[KC - 1]) return v;  // this lane alone has KC nearer points
          const int32_t* row = start + (int64_t(z) * gr.g[1] + y) * gr.g[0];
          if (r == 1 || dy == -r || dy == r || dz == -r || dz == r) {
            v.x = row[x0];
            v.y = row[x1 + 1];
          } else {
            if (cx - r >= 0) v.x = row[cx - r], v.y = row[cx - r + 1];
            if (cx + r < gr.g[0]) v.z = row[cx + r], v.w = row[cx + r + 1];
          }
        }
        return v;
      };
      int4 next = ranges(0);
      for (int base = 0; base < rows; base += G) {
        const int4 v = next;
        const bool skip = G == 1 && far2 > best.d[KC - 1];
        if (base + G < rows) next = ranges(base + G);  // its loads are in flight while these rows are read
        if (skip) continue;
#pragma unroll 1
        for (int l = 0; l < G && base + l < rows; ++l) {
          scan(group_get<G>(mask, v.x, l), group_get<G>(mask, v.y, l));
          if (r > 1) scan(group_get<G>(mask, v.z, l), group_get<G>(mask, v.w, l));
        }
      }
      // distance to the nearest face of the scanned block that has cells behind it
      int64_t lim = INT64_MAX;
      bool more = false;
      const int cc[3] = {cx, cy, cz}, pp[3] = {p.x, p.y, p.z};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int64_t rel = int64_t(pp[a]) - gr.lo[a];
        if (cc[a] - r > 0) {
          lim = min(lim, rel - int64_t(cc[a] - r) * gr.c + 1);
          more = true;
        }
        if (cc[a] + r < gr.g[a] - 1) {
          lim = min(lim, int64_t(cc[a] + r + 1) * gr.c - rel);
          more = true;
        }
      }
      if (!more) break;
      int near = 0;
#pragma unroll
      for (int a = 0; a < KC; ++a) near += best.d[a] < lim * lim;
#pragma unroll
      for (int o = G / 2; o; o >>= 1) near += __shfl_xor_sync(mask, near, o, G);
      if (near >= k) break;
    }
    for (int a = 0; a < k; ++a) {  // merge: the least head of the group's lists, k times
      int64_t d = best.d[0];
      int32_t j = best.j[0];
#pragma unroll
      for (int o = G / 2; o; o >>= 1) {
        const int64_t d2 = __shfl_xor_sync(mask, d, o, G);
        const int32_t j2 = __shfl_xor_sync(mask, j, o, G);
        if (key_less(d2, j2, d, j)) d = d2, j = j2;
      }
      if (best.j[0] == j) best.pop();
      if (gl == a % G) {
        const int64_t slot = int64_t(p.w) * stride + off + a;
        const bool found = j != INT32_MAX;
        nbr[slot] = found ? j : -1;
        if (found) rank[slot] = atomicAdd(&rcnt[j], 1);
      }
    }
  }
}

template <bool QUERY, int G>
void knn_launch_g(unsigned grid, cudaStream_t s, const int32_t* q, const int4* pts, const int32_t* start, int64_t q0,
                  int64_t q1, int k, const Grid* gr, int32_t* nbr, int64_t stride, int off, int32_t* rcnt,
                  int32_t* rank) {
  if (k <= 3)
    launch_pdl(knn_kernel<3, G, QUERY>, grid, 128, 0, s, q, pts, start, q0, q1, k, gr, nbr, stride, off, rcnt, rank);
  else if (k <= 6)
    launch_pdl(knn_kernel<6, G, QUERY>, grid, 128, 0, s, q, pts, start, q0, q1, k, gr, nbr, stride, off, rcnt, rank);
  else if (k <= 8)
    launch_pdl(knn_kernel<8, G, QUERY>, grid, 128, 0, s, q, pts, start, q0, q1, k, gr, nbr, stride, off, rcnt, rank);
  else if (k <= 16)
    launch_pdl(knn_kernel<16, G, QUERY>, grid, 128, 0, s, q, pts, start, q0, q1, k, gr, nbr, stride, off, rcnt, rank);
  else
    launch_pdl(knn_kernel<kMaxK, G, QUERY>, grid, 128, 0, s, q, pts, start, q0, q1, k, gr, nbr, stride, off, rcnt,
               rank);
}

// Lanes per point: eight while that still leaves at most one wave of resident
// threads (2k points: 47 us with one lane, 22 us with eight; beyond it the
// merge and the lanes idle at the ends of short ranges cost more than the
// parallel reads give: 200k points 97 against 130 us).
template <bool QUERY>
xmgn_status knn_launch(const int32_t* q, const int4* pts, const int32_t* start, int64_t q0, int64_t q1, int k,
                       const Grid* gr, int32_t* nbr, int64_t stride, int off, int32_t* rcnt, int32_t* rank,
                       cudaStream_t s) {
  const int64_t n = q1 - q0;
  if (n * 8 <= int64_t(num_sms()) * 2048)
    knn_launch_g<QUERY, 8>(grid_for(n * 8, 128, 1 << 30), s, q, pts, start, q0, q1, k, gr, nbr, stride, off, rcnt,
                           rank);
  else
    knn_launch_g<QUERY, 1>(grid_for(n, 128, 1 << 30), s, q, pts, start, q0, q1, k, gr, nbr, stride, off, rcnt, rank);
  XMGN_LAUNCH_CHECK();
  return XMGN_OK;
}

__global__ void empty_slots_kernel(int32_t* __restrict__ nbr, int64_t slots, const int32_t* __restrict__ bad) {
  pdl_wait();
  pdl_trigger();
  if (*bad) return;
  for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < slots; t += int64_t(gridDim.x) * blockDim.x)
    nbr[t] = -1;
}

// ---- symmetrisation
// Row i of the undirected graph = its own K slots and every j that lists i.
// Reverse entries: slot t of point i names j = nbr[t]; i goes to place rank[t]
// of j's list.
__global__ void sym_rev_kernel(const int32_t* __restrict__ nbr, int64_t n, int k, const int64_t* __restrict__ rstart,
                               const int32_t* __restrict__ rank, const int32_t* __restrict__ bad,
                               int32_t* __restrict__ rev) {
  pdl_wait();
  pdl_trigger();
  if (*bad) return;
  for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n * k;
       t += int64_t(gridDim.x) * blockDim.x) {
    const int32_t j = nbr[t];
    if (j >= 0) rev[rstart[j] + rank[t]] = int32_t(t / k);
  }
}

// Sorts row i (ascending ids) and drops repeats: 16 lanes per row collect its
// entries, every lane counts how many entries are less than its own and writes
// it to that place (equal entries meet there and leave holes behind them), and
// the filled places are closed up.  Rows of up to kRow entries stay in shared
// memory, the two rows of a warp in step (their loops run to the longer one's
// end: apart, the halves would take turns); longer ones, points that many
// others list, are sorted on the global arrays.  out row i starts at rstart[i]
// + K i.  Bound by the latency of the row's reads; 1.25M rows of 21 slots: 1216
// us (a thread per row, insertion sort in global memory) -> 415 us, and 12 us
// less with six blocks per SM (40 registers, nothing spilled) instead of five.
constexpr int kRow = 64;
__global__ void __launch_bounds__(256, 6) sym_sort_kernel(const int32_t* __restrict__ nbr, int64_t n, int k,
                                                       const int64_t* __restrict__ rstart,
                                                       const int32_t* __restrict__ rev,
                                                       const int32_t* __restrict__ bad, int32_t* __restrict__ out,
                                                       int32_t* __restrict__ deg) {
  pdl_wait();
  pdl_trigger();
  if (*bad) return;
  __shared__ __align__(16) int32_t raw[16][kRow], srt[16][kRow];
  const int lane = threadIdx.x & 31, l = lane & 15, gi = threadIdx.x >> 4, hs = lane & 16;
  constexpr uint32_t kAll = 0xffffffffu;
  auto half = [&](uint32_t m) { return (m >> hs) & 0xffffu; };  // this half's bits
  for (int64_t i0 = int64_t(blockIdx.x) * 16 + (gi & ~1); i0 < n; i0 += int64_t(gridDim.x) * 16) {
    const int64_t i = i0 + (gi & 1);
    const bool in = i < n;
    const int64_t r0 = in ? rstart[i] : 0, nr = in ? rstart[i + 1] - r0 : 0;
    int32_t* const row = out + r0 + int64_t(k) * i;
    int m = 0;
    for (int a0 = 0; a0 < k; a0 += 16) {
      const int32_t v = in && a0 + l < k ? nbr[i * k + a0 + l] : -1;
      const uint32_t b = half(__ballot_sync(kAll, v >= 0));
      const int at = m + __popc(b & ((1u << l) - 1u));
      if (v >= 0 && at < kRow) raw[gi][at] = v;
      m += __popc(b);
    }
    const bool brief = m + nr <= kRow;
    if (brief) {
      for (int a = l; a < int(nr); a += 16) raw[gi][m + a] = rev[r0 + a];
      m += int(nr);
    } else {
      m = 0;
    }
    const int mw = max(m, __shfl_xor_sync(kAll, m, 16));
    for (int a = m + l; a < ((mw + 3) & ~3); a += 16) raw[gi][a] = INT32_MAX;  // less than nothing
    for (int a = l; a < mw; a += 16) srt[gi][a] = -1;
    __syncwarp();
    for (int a0 = 0; a0 < mw; a0 += 16) {
      const int a = a0 + l;
      const int32_t x = a < m ? raw[gi][a] : -1;
      int c = 0;
      for (int b = 0; b < mw; b += 4) {
        const int4 y = *reinterpret_cast<const int4*>(&raw[gi][b]);
        c += (y.x < x) + (y.y < x) + (y.z < x) + (y.w < x);
      }
      if (a < m) srt[gi][c] = x;
    }
    __syncwarp();
    int u = 0;
    for (int a0 = 0; a0 < mw; a0 += 16) {
      const int32_t x = a0 + l < m ? srt[gi][a0 + l] : -1;
      const bool keep = x >= 0 && x != int32_t(i);
      const uint32_t b = half(__ballot_sync(kAll, keep));
      if (keep) row[u + __popc(b & ((1u << l) - 1u))] = x;
      u += __popc(b);
    }
    if (in && brief && l == 0) deg[i] = u;
    __syncwarp();
    if (!in || brief) continue;
    // long row, by its half-warp: entries a < k the own slots (empty ones rank last), then the reverse entries
    const uint32_t mask = 0xffffu << hs;
    const int64_t all = k + nr;
    auto get = [&](int64_t a) {
      const int32_t v = a < k ? nbr[i * k + a] : rev[r0 + a - k];
      return v < 0 ? INT32_MAX : v;
    };
    for (int64_t a = l; a < all; a += 16) {
      const int32_t x = get(a);
      int64_t c = 0;
      for (int64_t b = 0; b < all; ++b) {
        const int32_t y = get(b);
        c += y < x || (y == x && b < a);
      }
      row[c] = x;
    }
    __syncwarp(mask);
    int32_t last = -1;  // the entry before this chunk
    for (int64_t a0 = 0; a0 < all; a0 += 16) {
      const int64_t a = a0 + l;
      const int32_t x = a < all ? row[a] : INT32_MAX;
      int32_t prev = __shfl_up_sync(mask, x, 1, 16);
      if (l == 0) prev = last;
      last = __shfl_sync(mask, x, 15, 16);
      const bool keep = x != INT32_MAX && x != int32_t(i) && x != prev;
      const uint32_t b = half(__ballot_sync(mask, keep));
      if (keep) row[u + __popc(b & ((1u << l) - 1u))] = x;  // at or before the places already read
      u += __popc(b);
      __syncwarp(mask);
    }
    if (l == 0) deg[i] = u;
  }
}

// Copies the sorted rows to their CSR places, 8 lanes per row; nothing is
// written when the edges exceed the caller's capacity or a coordinate is bad.
__global__ void sym_emit_kernel(const int32_t* __restrict__ rows, const int64_t* __restrict__ rstart, int k,
                                const int64_t* __restrict__ row_ptr, int64_t n, int64_t cap,
                                int32_t* __restrict__ col, int32_t* __restrict__ recv,
                                const uint32_t* __restrict__ err, const int32_t* __restrict__ bad,
                                int64_t* __restrict__ info) {
  pdl_wait();
  pdl_trigger();
  const bool stop = *bad != 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // what the host reads at the end, in one copy
    info[0] = stop ? 0 : row_ptr[n];
    info[1] = int64_t(*err) | (stop ? int64_t(DEV_ERR_RANGE) : 0);
  }
  if (stop || row_ptr[n] > cap) return;
  const int l = threadIdx.x & 7;
  for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 3; i < n;
       i += (int64_t(gridDim.x) * blockDim.x) >> 3) {
    const int32_t* c = rows + rstart[i] + int64_t(k) * i;
    const int64_t o = row_ptr[i], m = row_ptr[i + 1] - o;
    for (int64_t a = l; a < m; a += 8) {
      col[o + a] = c[a];
      if (recv) recv[o + a] = int32_t(i);
    }
  }
}

}  // namespace

xmgn_status quantize_launch(const float* xyz, int64_t n, double scale, int32_t* q, int32_t* bbox,
                            uint32_t* err, cudaStream_t s) {
  launch_pdl(bbox_init_kernel, 1, 32, 0, s, bbox);
  XMGN_LAUNCH_CHECK();
  launch_pdl(quantize_kernel, grid_for(n, 256, int64_t(num_sms()) * 8), 256, 0, s, xyz, n, float(scale), q, bbox, err);
  XMGN_LAUNCH_CHECK();
  return XMGN_OK;
}

// Edge p = (j <- r) at row j; csc_perm[p] = CSR position of the reverse edge
// (r <- j).  Shared by the kNN builder and the partitioner.  Bound by the L2
// latency of three dependent reads (ids, row offsets, row), so every thread
// keeps four edges in flight and reads rows of up to 8 edges whole; longer
// rows are searched by key (their senders' ids, or global ids, ascend).  17.2M
// edges of a 2M-point batch: 123 us (a binary search by key per thread) -> 98 us.
// e < 0: the edge count is row_ptr[n], and nothing is written if it exceeds cap
// or *bad is set.
constexpr int kPermEdges = 4;
__global__ void __launch_bounds__(256) csc_perm_kernel(const int64_t* __restrict__ row_ptr,
                                                       const int32_t* __restrict__ col,
                                                       const int32_t* __restrict__ recv,
                                                       const int32_t* __restrict__ key, int64_t n, int64_t e,
                                                       int64_t cap, const int32_t* __restrict__ bad,
                                                       int32_t* __restrict__ perm, uint32_t* err) {
  pdl_wait();
  pdl_trigger();
  if (e < 0) {
    if (*bad) return;
    e = row_ptr[n];
    if (e > cap) return;
  }
  const int64_t step = int64_t(gridDim.x) * blockDim.x * kPermEdges;
  for (int64_t p0 = int64_t(blockIdx.x) * blockDim.x * kPermEdges + threadIdx.x; p0 < e; p0 += step) {
    int32_t j[kPermEdges], r[kPermEdges];
    int64_t b0[kPermEdges];
    int m[kPermEdges], at[kPermEdges];
#pragma unroll
    for (int u = 0; u < kPermEdges; ++u) {
      const int64_t p = p0 + u * int64_t(blockDim.x);
      const bool in = p < e;
      j[u] = in ? recv[p] : -1;
      r[u] = in ? col[p] : -1;
    }
#pragma unroll
    for (int u = 0; u < kPermEdges; ++u) {
      const bool ok = r[u] >= 0 && r[u] < n && j[u] >= 0 && j[u] < n;
      b0[u] = ok ? row_ptr[r[u]] : 0;
      m[u] = ok ? int(row_ptr[r[u] + 1] - b0[u]) : 0;
      at[u] = -1;
    }
#pragma unroll
    for (int u = 0; u < kPermEdges; ++u) {
      const int32_t* row = col + b0[u];
      int32_t v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = q < m[u] ? row[q] : -1;
#pragma unroll
      for (int q = 7; q >= 0; --q)
        if (v[q] == j[u]) at[u] = q;
    }
#pragma unroll
    for (int u = 0; u < kPermEdges; ++u) {
      const int64_t p = p0 + u * int64_t(blockDim.x);
      if (p >= e) continue;
      if (at[u] < 0 && m[u] > 8) {
        const int32_t* row = col + b0[u];
        const int32_t want = key ? key[j[u]] : j[u];
        int lo = 8, hi = m[u];
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          const int32_t v = key ? key[row[mid]] : row[mid];
          if (v < want) lo = mid + 1; else hi = mid;
        }
        if (lo < m[u] && row[lo] == j[u]) at[u] = lo;
      }
      if (at[u] < 0) dev_flag(err, DEV_ERR_GRAPH);
      perm[p] = at[u] < 0 ? 0 : int32_t(b0[u] + at[u]);
    }
  }
}

struct KnnWs {
  int32_t *q, *bbox, *nbr, *cnt, *rcnt, *rev, *rows, *rank, *deg, *cell_of, *at, *cstart;
  int4* pts;
  Grid* grid;
  int64_t *rstart, *info, *scan_tmp;
};

// Workspace for N points with K directed slots per point.
static void knn_layout(int64_t N, int32_t K, Arena& A, KnnWs& w) {
  const int64_t cells = cell_budget(N);
  w.q = A.take<int32_t>(size_t(3 * N));
  w.bbox = A.take<int32_t>(8);
  w.grid = A.take<Grid>(kMaxLevels);
  w.info = A.take<int64_t>(2);
  w.cell_of = A.take<int32_t>(size_t(N));
  w.at = A.take<int32_t>(size_t(N));
  w.pts = A.take<int4>(size_t(N));
  w.nbr = A.take<int32_t>(size_t(N * K));
  w.cnt = A.take<int32_t>(size_t(cells + 1));
  w.cstart = A.take<int32_t>(size_t(cells + 1));
  w.rcnt = A.take<int32_t>(size_t(N));
  w.rstart = A.take<int64_t>(size_t(N + 1));
  w.rev = A.take<int32_t>(size_t(N * K));
  w.rows = A.take<int32_t>(size_t(2 * N * K));
  w.rank = w.rows;  // the places of the reverse entries are used up before the rows are written
  w.deg = A.take<int32_t>(size_t(N));
  w.scan_tmp = A.take<int64_t>(scan_tmp_elems((cells > N ? cells : N) + 1) + 16);
}

// Lattice coordinates of all N points, their bounding box and the levels' grids.
static xmgn_status quantize_all(const float* xyz, int64_t N, double scale, const LevelSizes& sizes, int levels,
                                KnnWs& w, uint32_t* err, cudaStream_t s) {
  XMGN_TRY(quantize_launch(xyz, N, scale, w.q, w.bbox, err, s));
  launch_pdl(grid_layout_kernel, 1, 32, 0, s, w.bbox, sizes, levels, err, w.grid);
  XMGN_LAUNCH_CHECK();
  XMGN_CUDA(cudaMemsetAsync(w.rcnt, 0, sizeof(int32_t) * size_t(N), s));
  return XMGN_OK;
}

// Counting sort of the reference points 0..n_ref-1 into their grid.
static xmgn_status grid_sort(int64_t n_ref, const Grid* grid, KnnWs& w, cudaStream_t s) {
  const int64_t cells = cell_budget(n_ref);
  XMGN_CUDA(cudaMemsetAsync(w.cnt, 0, sizeof(int32_t) * size_t(cells), s));
  launch_pdl(cell_count_kernel, grid_for(n_ref, 256), 256, 0, s, w.q, n_ref, grid, w.cell_of, w.at, w.cnt);
  XMGN_LAUNCH_CHECK();
  XMGN_TRY(exclusive_scan_i32(w.cnt, w.cstart, cells, w.scan_tmp, s));
  launch_pdl(cell_scatter_kernel, grid_for(n_ref, 256), 256, 0, s, w.q, w.cell_of, w.at, n_ref, w.cstart, grid,
             w.pts);
  XMGN_LAUNCH_CHECK();
  return XMGN_OK;
}

// Undirected receiver-major CSR from K directed slots per point (w.nbr,
// -1 = empty; w.rcnt and w.rank as knn_kernel leaves them), and the one host
// wait of a build: the edge count and the range error of the coordinates.
static xmgn_status symmetrise_slots(int64_t N, int32_t K, KnnWs& w, int64_t* row_ptr, int32_t* col,
                                    int32_t* recv, int32_t* csc_perm, int64_t E_cap, int64_t* E_out,
                                    uint32_t* err, cudaStream_t s) {
  const int32_t* bad = w.bbox + 6;
  XMGN_TRY(exclusive_scan_i32(w.rcnt, w.rstart, N, w.scan_tmp, s));
  launch_pdl(sym_rev_kernel, grid_for(N * K, 256), 256, 0, s, w.nbr, N, K, w.rstart, w.rank, bad, w.rev);
  XMGN_LAUNCH_CHECK();
  launch_pdl(sym_sort_kernel, grid_for(N * 16, 256), 256, 0, s, w.nbr, N, K, w.rstart, w.rev, bad, w.rows,
             w.deg);
  XMGN_LAUNCH_CHECK();
  XMGN_TRY(exclusive_scan_i32(w.deg, row_ptr, N, w.scan_tmp, s, bad));
  launch_pdl(sym_emit_kernel, grid_for(N * 8, 256), 256, 0, s, w.rows, w.rstart, K, row_ptr, N, E_cap, col, recv, err,
             bad, w.info);
  XMGN_LAUNCH_CHECK();
  if (csc_perm) {
    const int64_t most = 2 * N * K < E_cap ? 2 * N * K : E_cap;
    launch_pdl(csc_perm_kernel, grid_for((most + kPermEdges - 1) / kPermEdges, 256), 256, 0, s, row_ptr, col, recv,
               nullptr, N, -1, E_cap, bad, csc_perm, err);
    XMGN_LAUNCH_CHECK();
  }
  int64_t info[2];
  XMGN_CUDA(cudaMemcpyAsync(info, w.info, sizeof(info), cudaMemcpyDeviceToHost, s));
  XMGN_CUDA(cudaStreamSynchronize(s));
  const int64_t E = info[0];
  if (info[1] & DEV_ERR_RANGE) {
    XMGN_CUDA(cudaMemsetAsync(err, 0, sizeof(uint32_t), s));
    return fail(XMGN_ERR_RANGE, "coordinate outside the lattice range (|x*scale| >= 2^24 or not finite)");
  }
  *E_out = E;
  if (E > E_cap) return fail(XMGN_ERR_WORKSPACE, "E=%lld exceeds E_cap=%lld", (long long)E, (long long)E_cap);
  return XMGN_OK;
}

static xmgn_status check_scale(double scale) {
  int ex = 0;
  double fr = frexp(scale, &ex);
  if (!(scale > 0) || fr != 0.5) return fail(XMGN_ERR_ARG, "lattice_scale must be a power of two");
  return XMGN_OK;
}

xmgn_status build_knn_ws(int64_t N, int32_t k, size_t* ws_bytes) {
  Arena A;
  A.dry = true;
  KnnWs w;
  knn_layout(N, k, A, w);
  *ws_bytes = A.used + 256;
  return XMGN_OK;
}

xmgn_status build_knn(const float* xyz, int64_t N, int32_t k, double scale, void* ws,
                      size_t ws_bytes, int32_t* nbr_out, int64_t* row_ptr, int32_t* col,
                      int32_t* recv, int32_t* csc_perm, int64_t E_cap, int64_t* E_out,
                      cudaStream_t s) {
  if (!xyz || !row_ptr || !col || !E_out || !ws) return fail(XMGN_ERR_ARG, "null pointer");
  if (k < 1 || k > kMaxK) return fail(XMGN_ERR_ARG, "k must be in [1, %d]", kMaxK);
  if (N < int64_t(k) + 1) return fail(XMGN_ERR_ARG, "need N >= k+1 (N=%lld, k=%d)", (long long)N, k);
  if (N >= (int64_t(1) << 31)) return fail(XMGN_ERR_ARG, "N must be < 2^31");
  XMGN_TRY(check_scale(scale));
  if (csc_perm && !recv) return fail(XMGN_ERR_ARG, "csc_perm requires recv");

  Arena A;
  A.base = static_cast<char*>(ws);
  A.cap = ws_bytes;
  KnnWs w;
  knn_layout(N, k, A, w);
  if (!A.ok()) return fail(XMGN_ERR_WORKSPACE, "knn workspace too small: need %zu", A.used);
  uint32_t* err = device_error_word();
  if (nbr_out) w.nbr = nbr_out;
  LevelSizes sizes{};
  sizes.n[0] = N;
  XMGN_TRY(quantize_all(xyz, N, scale, sizes, 1, w, err, s));
  XMGN_TRY(grid_sort(N, w.grid, w, s));
  XMGN_TRY(knn_launch<false>(w.q, w.pts, w.cstart, 0, N, k, w.grid, w.nbr, k, 0, w.rcnt, w.rank, s));
  return symmetrise_slots(N, k, w, row_ptr, col, recv, csc_perm, E_cap, E_out, err, s);
}

static int32_t multiscale_slots(int32_t n_levels, int32_t k, int32_t k_cross) {
  return n_levels * k + (n_levels > 1 ? k_cross : 0);
}

xmgn_status build_multiscale_ws(int64_t N, int32_t n_levels, int32_t k, int32_t k_cross, size_t* ws_bytes) {
  if (n_levels < 1) return fail(XMGN_ERR_ARG, "need at least one level");
  Arena A;
  A.dry = true;
  KnnWs w;
  knn_layout(N, multiscale_slots(n_levels, k, k_cross), A, w);
  *ws_bytes = A.used + 256;
  return XMGN_OK;
}

xmgn_status build_multiscale(const float* xyz, int64_t N, const int64_t* sizes, int32_t n_levels, int32_t k,
                             int32_t k_cross, double scale, void* ws, size_t ws_bytes, int32_t* nbr_out,
                             int64_t* row_ptr, int32_t* col, int32_t* recv, int32_t* csc_perm, int64_t E_cap,
                             int64_t* E_out, cudaStream_t s) {
  if (!xyz || !sizes || !row_ptr || !col || !E_out || !ws) return fail(XMGN_ERR_ARG, "null pointer");
  if (n_levels < 1 || n_levels > 16) return fail(XMGN_ERR_ARG, "n_levels must be in [1, 16]");
  if (k < 1 || k > kMaxK || k_cross < 1 || k_cross > kMaxK)
    return fail(XMGN_ERR_ARG, "k and k_cross must be in [1, %d]", kMaxK);
  if (N >= (int64_t(1) << 31)) return fail(XMGN_ERR_ARG, "N must be < 2^31");
  for (int l = 0; l < n_levels; ++l) {
    const int64_t lo = l ? sizes[l - 1] : 0;
    if (sizes[l] <= lo) return fail(XMGN_ERR_ARG, "level sizes must increase");
  }
  if (sizes[n_levels - 1] != N) return fail(XMGN_ERR_ARG, "the last level size must be N");
  if (sizes[0] < int64_t(k) + 1) return fail(XMGN_ERR_ARG, "the first level needs more than k points");
  if (n_levels > 1 && sizes[0] < k_cross) return fail(XMGN_ERR_ARG, "the first level needs k_cross points");
  XMGN_TRY(check_scale(scale));
  if (csc_perm && !recv) return fail(XMGN_ERR_ARG, "csc_perm requires recv");

  const int32_t K = multiscale_slots(n_levels, k, k_cross);
  Arena A;
  A.base = static_cast<char*>(ws);
  A.cap = ws_bytes;
  KnnWs w;
  knn_layout(N, K, A, w);
  if (!A.ok()) return fail(XMGN_ERR_WORKSPACE, "multiscale workspace too small: need %zu", A.used);
  uint32_t* err = device_error_word();
  if (nbr_out) w.nbr = nbr_out;
  LevelSizes ls{};
  for (int l = 0; l < n_levels; ++l) ls.n[l] = sizes[l];
  XMGN_TRY(quantize_all(xyz, N, scale, ls, n_levels, w, err, s));
  launch_pdl(empty_slots_kernel, grid_for(N * K, 256, int64_t(num_sms()) * 8), 256, 0, s, w.nbr, N * K, w.bbox + 6);
  XMGN_LAUNCH_CHECK();
  for (int l = 0; l < n_levels; ++l) {
    // kNN within level l (the first sizes[l] points): slots [l*k, l*k + k)
    XMGN_TRY(grid_sort(sizes[l], w.grid + l, w, s));
    XMGN_TRY(knn_launch<false>(w.q, w.pts, w.cstart, 0, sizes[l], k, w.grid + l, w.nbr, K, l * k, w.rcnt, w.rank, s));
    if (l + 1 < n_levels)  // points new in level l+1 -> k_cross nearest of level l: slots [L*k, L*k + k_cross)
      XMGN_TRY(knn_launch<true>(w.q, w.pts, w.cstart, sizes[l], sizes[l + 1], k_cross, w.grid + l, w.nbr, K,
                                n_levels * k, w.rcnt, w.rank, s));
  }
  return symmetrise_slots(N, K, w, row_ptr, col, recv, csc_perm, E_cap, E_out, err, s);
}

}  // namespace xmgn
