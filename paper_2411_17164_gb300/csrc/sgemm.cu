// FP32 products of the plain path on the CUDA cores (fused multiply-adds in
// fp32 throughout, each output one running sum over the reduction in index
// order):
//
//   NN  C[M, N] = epi(A[M, K] B[K, N] + bias [+ gathered rows])
//   NT  C[M, N] = epi(A[M, K] B[N, K]^T)
//   TN  G[K1, N] = sum over rows m of A[m, :]^T B[m, :]
//
// sgemm_kernel: 128 x BN tiles (BN 128 or 64), 16-deep slices double-buffered
// in shared memory (the next slice travels in registers while this one is
// multiplied: one barrier per slice), 8 x BN/16 outputs per thread held as
// packed pairs so that one fma.rn.f32x2 does two multiply-adds per issue slot.
// The FMA pipe is what bounds it: per slice and thread 16 x 64 multiply-adds
// stand against 64 shared-memory loads of 16 bytes, all free of bank conflicts
// (a warp reads 64 + 128 consecutive bytes per step), and at K = 128 the first
// loads and the epilogue beside it, which nothing hides.  Launch list of a
// 15-layer step, 212k x 128 x 128: NN 160 us (43 TFLOP/s), with the gathered rows
// 203 (34), NT 204 (34), TN 135 (51); over all products of the step 36 TFLOP/s of
// 80.5 at 2070 MHz.  The 64 x 64 scalar tiles before: 142 against 36.5 ms a step,
// the split first edge layer included.
// general_nnt_kernel / general_tn_kernel take what the 16-byte loads cannot:
// widths, leading dimensions or bases that are not multiples of four floats
// (the node encoder's six inputs, parameter vectors at odd addresses).
#include "model.cuh"

namespace xmgn {

namespace {

constexpr int GT = 64;   // output tile edge of the general kernels
constexpr int BK = 16;   // reduction step
constexpr int BM = 128;  // tile rows of sgemm_kernel

__device__ __forceinline__ float src_get(const RowSrc& A, int64_t r, int k) {
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    if (s < A.nseg) {
      const RowSeg& g = A.s[s];
      if (k < g.width) {
        int64_t row = g.idx ? int64_t(g.idx[r]) : r;
        return g.p[row * g.ld + k];
      }
      k -= g.width;
    }
  }
  return 0.f;
}

__device__ __forceinline__ float silu_f(float z) { return z / (1.f + __expf(-z)); }
__device__ __forceinline__ float silu_grad_f(float z) {
  float s = 1.f / (1.f + __expf(-z));
  return s * (1.f + z * (1.f - s));
}

__device__ __forceinline__ float epi_value(int epi, float v, float old_or_aux) {
  switch (epi) {
    case EPI_SILU: return silu_f(v);
    case EPI_ACCUM: return old_or_aux + v;
    case EPI_SILU_GRAD: return v * silu_grad_f(old_or_aux);
    default: return v;
  }
}

// The sums that come out of a product before its epilogue: acc + bias[n] +
// the gathered node-projection rows of output row m.
__device__ __forceinline__ float add_terms(float v, const float* bias, const RowAdd& g, int64_t m, int n) {
  if (bias) v += bias[n];
  if (g.p) v += g.p[int64_t(g.i0[m]) * g.ld + n] + g.p[int64_t(g.i1[m]) * g.ld + g.off1 + n];
  return v;
}

template <bool NT>
__global__ void __launch_bounds__(256) general_nnt_kernel(RowSrc A, int64_t M, const float* __restrict__ B, int N,
                                                          const float* __restrict__ bias, float* __restrict__ C,
                                                          int64_t ldc, int epi, float* __restrict__ pre,
                                                          const float* __restrict__ aux, RowAdd add) {
  pdl_wait();
  pdl_trigger();
  __shared__ float As[BK][GT + 4];
  __shared__ float Bs[BK][GT + 4];
  const int K = A.K;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int64_t m0 = int64_t(blockIdx.x) * GT;
  const int n0 = blockIdx.y * GT;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int idx = t + 256 * i;
      int mm = idx >> 4, kk = idx & 15;
      int64_t m = m0 + mm;
      int k = k0 + kk;
      As[kk][mm] = (m < M && k < K) ? src_get(A, m, k) : 0.f;
      int nn = idx & 63, kb = idx >> 6;
      int n = n0 + nn, kq = k0 + kb;
      float bv = 0.f;
      if (n < N && kq < K) bv = NT ? B[int64_t(n) * K + kq] : B[int64_t(kq) * N + n];
      Bs[kb][nn] = bv;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int64_t m = m0 + ty * 4 + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int n = n0 + tx * 4 + j;
      if (n >= N) continue;
      const float v = add_terms(acc[i][j], bias, add, m, n);
      const int64_t at = m * ldc + n;
      if (pre) pre[at] = v;
      C[at] = epi_value(epi, v, epi == EPI_ACCUM ? C[at] : epi == EPI_SILU_GRAD ? aux[at] : 0.f);
    }
  }
}

__global__ void __launch_bounds__(256) general_tn_kernel(RowSrc A, int64_t M, const float* __restrict__ B,
                                                         int64_t ldb, int N, int64_t rows_per_chunk,
                                                         float* __restrict__ part) {
  pdl_wait();
  pdl_trigger();
  __shared__ float As[BK][GT + 4];
  __shared__ float Bs[BK][GT + 4];
  const int K1 = A.K;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int ntn = (N + GT - 1) / GT;
  const int k10 = (blockIdx.x / ntn) * GT;
  const int n0 = (blockIdx.x % ntn) * GT;
  const int64_t r_begin = int64_t(blockIdx.y) * rows_per_chunk;
  const int64_t r_end = min(M, r_begin + rows_per_chunk);
  float acc[4][4] = {};
  for (int64_t r0 = r_begin; r0 < r_end; r0 += BK) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int idx = t + 256 * i;
      int rr = idx >> 6, cc = idx & 63;
      int64_t r = r0 + rr;
      int k1 = k10 + cc, n = n0 + cc;
      bool rv = r < r_end;
      As[rr][cc] = (rv && k1 < K1) ? src_get(A, r, k1) : 0.f;
      Bs[rr][cc] = (rv && n < N) ? B[r * ldb + n] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < BK; ++rr) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[rr][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[rr][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  float* P = part + int64_t(blockIdx.y) * K1 * N;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int k1 = k10 + ty * 4 + i;
    if (k1 >= K1) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int n = n0 + tx * 4 + j;
      if (n < N) P[int64_t(k1) * N + n] = acc[i][j];
    }
  }
}

__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

enum GemmForm : int { G_NN = 0, G_NT = 1, G_TN = 2 };

// One operand tile's share of a thread: 16-deep slices of R (128 or 64) output
// rows or columns, R/64 float4 per thread and slice.
//  ROWS: the slice runs along the rows of the source (K contiguous): float4
//        of four consecutive k of one row, stored transposed.
//  !ROWS: the slice's 16 rows are rows of the source, R contiguous columns.
template <int R>
struct Slice {
  float4 v[R / 64];
};

template <int R>
__device__ __forceinline__ void put_rows(float (*S)[R + 4], const Slice<R>& f, int t) {
  const int kq = (t & 3) * 4;
#pragma unroll
  for (int i = 0; i < R / 64; ++i) {
    const int r = (t >> 2) + 64 * i;
    S[kq + 0][r] = f.v[i].x;
    S[kq + 1][r] = f.v[i].y;
    S[kq + 2][r] = f.v[i].z;
    S[kq + 3][r] = f.v[i].w;
  }
}
template <int R>
__device__ __forceinline__ void put_cols(float (*S)[R + 4], const Slice<R>& f, int t) {
#pragma unroll
  for (int i = 0; i < R / 64; ++i) {
    const int q = t + 256 * i;
    *reinterpret_cast<float4*>(&S[q / (R / 4)][(q % (R / 4)) * 4]) = f.v[i];
  }
}

struct SgemmArgs {
  RowSrc A;
  int64_t M;  // NN/NT: output rows; TN: reduction rows
  const float* B;
  int64_t ldb;
  int N;
  const float* bias;
  float* C;
  int64_t ldc;
  int epi;
  float* pre;
  const float* aux;
  RowAdd add;
  int64_t rows_per_chunk;  // TN
};

// FORM NN / NT: blockIdx.x = row tile, blockIdx.y = column tile.  TN:
// blockIdx.x = tile of K1 x N (columns fastest), blockIdx.y = row chunk, the
// chunk's partial product written to C + chunk * K1 * N.
// Every width (segments of A, N) and leading dimension is a multiple of 4 and
// every base 16-byte aligned.
template <int FORM, int BN>
__global__ void __launch_bounds__(256, 2) sgemm_kernel(const __grid_constant__ SgemmArgs a) {
  pdl_wait();
  pdl_trigger();
  constexpr int TN = BN / 16;  // output columns per thread
  __shared__ __align__(16) float As[2][BK][BM + 4];
  __shared__ __align__(16) float Bs[2][BK][BN + 4];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  int64_t m0, r_begin = 0, r_end = 0;
  int n0;
  if (FORM == G_TN) {
    const int ntn = (a.N + BN - 1) / BN;
    m0 = int64_t(blockIdx.x / ntn) * BM;
    n0 = int(blockIdx.x % ntn) * BN;
    r_begin = int64_t(blockIdx.y) * a.rows_per_chunk;
    r_end = min(a.M, r_begin + a.rows_per_chunk);
  } else {
    m0 = int64_t(blockIdx.x) * BM;
    n0 = blockIdx.y * BN;
  }
  const int K1 = a.A.K;  // NN/NT: reduction depth; TN: output rows
  const int64_t steps = FORM == G_TN ? (r_end > r_begin ? (r_end - r_begin + BK - 1) / BK : 0) : (K1 + BK - 1) / BK;

  Slice<BM> fa;
  Slice<BN> fb;
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  // NN/NT: the segment this thread's next float4 of A lies in, and its rows there
  int seg = 0, seg_k0 = 0;
  const float* arow[BM / 64];
  auto enter_seg = [&]() {
#pragma unroll
    for (int i = 0; i < BM / 64; ++i) {
      const int64_t m = m0 + (t >> 2) + 64 * i;
      const RowSeg& g = a.A.s[seg];
      arow[i] = m < a.M ? g.p + (g.idx ? int64_t(g.idx[m]) : m) * g.ld : nullptr;
    }
  };
  // TN: segment and column of this thread's columns of A (fixed over the rows)
  const float* acol[BM / 64];
  int64_t ald[BM / 64];
  const int32_t* aidx[BM / 64];
  if (FORM == G_TN) {
#pragma unroll
    for (int i = 0; i < BM / 64; ++i) {
      int k = int(m0) + ((t + 256 * i) % (BM / 4)) * 4;
      acol[i] = nullptr;
      ald[i] = 0;
      aidx[i] = nullptr;
#pragma unroll
      for (int s = 0; s < 3; ++s)
        if (s < a.A.nseg && !acol[i]) {
          if (k < a.A.s[s].width) {
            acol[i] = a.A.s[s].p + k;
            ald[i] = a.A.s[s].ld;
            aidx[i] = a.A.s[s].idx;
          }
          k -= a.A.s[s].width;
        }
    }
  } else {
    enter_seg();
  }
  auto load = [&](int64_t step) {
    if (FORM == G_TN) {
#pragma unroll
      for (int i = 0; i < BM / 64; ++i) {
        const int64_t r = r_begin + step * BK + (t + 256 * i) / (BM / 4);
        fa.v[i] = (r < r_end && acol[i])
                      ? *reinterpret_cast<const float4*>(acol[i] + (aidx[i] ? int64_t(aidx[i][r]) : r) * ald[i])
                      : z4;
      }
#pragma unroll
      for (int i = 0; i < BN / 64; ++i) {
        const int q = t + 256 * i;
        const int64_t r = r_begin + step * BK + q / (BN / 4);
        const int n = n0 + (q % (BN / 4)) * 4;
        fb.v[i] = (r < r_end && n < a.N) ? *reinterpret_cast<const float4*>(a.B + r * a.ldb + n) : z4;
      }
      return;
    }
    const int k = int(step) * BK + (t & 3) * 4;
    while (seg < a.A.nseg && k >= seg_k0 + a.A.s[seg].width) {
      seg_k0 += a.A.s[seg].width;
      if (++seg < a.A.nseg) enter_seg();
    }
#pragma unroll
    for (int i = 0; i < BM / 64; ++i)
      fa.v[i] = (seg < a.A.nseg && arow[i]) ? *reinterpret_cast<const float4*>(arow[i] + (k - seg_k0)) : z4;
    if (FORM == G_NT) {
#pragma unroll
      for (int i = 0; i < BN / 64; ++i) {
        const int n = n0 + (t >> 2) + 64 * i;
        fb.v[i] = (n < a.N && k < K1) ? *reinterpret_cast<const float4*>(a.B + int64_t(n) * a.ldb + k) : z4;
      }
    } else {
#pragma unroll
      for (int i = 0; i < BN / 64; ++i) {
        const int q = t + 256 * i;
        const int kb = int(step) * BK + q / (BN / 4), n = n0 + (q % (BN / 4)) * 4;
        fb.v[i] = (kb < K1 && n < a.N) ? *reinterpret_cast<const float4*>(a.B + int64_t(kb) * a.ldb + n) : z4;
      }
    }
  };
  auto put = [&](int b) {
    if (FORM == G_TN) put_cols<BM>(As[b], fa, t); else put_rows<BM>(As[b], fa, t);
    if (FORM == G_NT) put_rows<BN>(Bs[b], fb, t); else put_cols<BN>(Bs[b], fb, t);
  };

  // Warps 4 (rows) x 2 (columns), warp tile 32 x BN/2, lanes 4 x 8: rows
  // wm + 4 lm + {0..3} and + 16, columns wn + 4 ln + {0..3} (and + 32)
  const int wm = (warp >> 1) * 32 + (lane >> 3) * 4;
  const int wn = (warp & 1) * (BN / 2) + (lane & 7) * 4;
  uint64_t acc[8][TN / 2];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;

  if (steps > 0) {
    load(0);
    put(0);
  }
  __syncthreads();
  for (int64_t st = 0; st < steps; ++st) {
    const int b = int(st & 1);
    if (st + 1 < steps) load(st + 1);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float av[8];
      uint64_t bv[TN / 2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 x = *reinterpret_cast<const float4*>(&As[b][kk][wm + 16 * h]);
        av[4 * h] = x.x, av[4 * h + 1] = x.y, av[4 * h + 2] = x.z, av[4 * h + 3] = x.w;
      }
#pragma unroll
      for (int h = 0; h < TN / 4; ++h) {
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(&Bs[b][kk][wn + 32 * h]);
        bv[2 * h] = x.x, bv[2 * h + 1] = x.y;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint64_t aa = pack2(av[i], av[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], aa, bv[j]);
      }
    }
    if (st + 1 < steps) put(b ^ 1);
    __syncthreads();
  }

#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t m = m0 + wm + (i & 3) + 16 * (i >> 2);
    if (m >= (FORM == G_TN ? int64_t(K1) : a.M)) continue;
    const float *g0 = nullptr, *g1 = nullptr;
    if (FORM == G_NN && a.add.p) {
      g0 = a.add.p + int64_t(a.add.i0[m]) * a.add.ld;
      g1 = a.add.p + int64_t(a.add.i1[m]) * a.add.ld + a.add.off1;
    }
#pragma unroll
    for (int h = 0; h < TN / 4; ++h) {
      const int n = n0 + wn + 32 * h;
      if (n >= a.N) continue;
      const float2 p = unpack2(acc[i][2 * h]), q = unpack2(acc[i][2 * h + 1]);
      float4 v = make_float4(p.x, p.y, q.x, q.y);
      if (FORM == G_TN) {
        *reinterpret_cast<float4*>(a.C + (int64_t(blockIdx.y) * K1 + m) * a.N + n) = v;
        continue;
      }
      if (FORM == G_NN) {
        if (a.bias) {
          const float4 x = *reinterpret_cast<const float4*>(a.bias + n);
          v.x += x.x, v.y += x.y, v.z += x.z, v.w += x.w;
        }
        if (g0) {
          const float4 x = *reinterpret_cast<const float4*>(g0 + n), y = *reinterpret_cast<const float4*>(g1 + n);
          v.x += x.x + y.x, v.y += x.y + y.y, v.z += x.z + y.z, v.w += x.w + y.w;
        }
      }
      const int64_t at = m * a.ldc + n;
      if (a.pre) *reinterpret_cast<float4*>(a.pre + at) = v;
      float4 o = z4;
      if (a.epi == EPI_ACCUM) o = *reinterpret_cast<const float4*>(a.C + at);
      if (a.epi == EPI_SILU_GRAD) o = *reinterpret_cast<const float4*>(a.aux + at);
      v.x = epi_value(a.epi, v.x, o.x);
      v.y = epi_value(a.epi, v.y, o.y);
      v.z = epi_value(a.epi, v.z, o.z);
      v.w = epi_value(a.epi, v.w, o.w);
      *reinterpret_cast<float4*>(a.C + at) = v;
    }
  }
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
// Whether sgemm_kernel's 16-byte accesses apply.
bool rows_ok(const RowSrc& A) {
  for (int s = 0; s < A.nseg; ++s)
    if (A.s[s].width % 4 || A.s[s].ld % 4 || !al16(A.s[s].p)) return false;
  return true;
}
bool fast(const SgemmArgs& a) {
  return rows_ok(a.A) && a.N % 4 == 0 && a.ldb % 4 == 0 && a.ldc % 4 == 0 && al16(a.B) && al16(a.bias) && al16(a.C) &&
         al16(a.pre) && al16(a.aux) && al16(a.add.p) && a.add.ld % 4 == 0 && a.add.off1 % 4 == 0;
}

template <int FORM>
xmgn_status run_fast(const SgemmArgs& a, int64_t rows, int64_t chunks, cudaStream_t s) {
  const int64_t tm = (rows + BM - 1) / BM;
  // 64-wide tiles for narrow outputs, and where 128-wide ones would leave SMs idle
  const bool wide = a.N > 64 && tm * ((a.N + 127) / 128) * chunks >= num_sms();
  const int64_t tn = wide ? (a.N + 127) / 128 : (a.N + 63) / 64;
  const dim3 grid = FORM == G_TN ? dim3(unsigned(tm * tn), unsigned(chunks)) : dim3(unsigned(tm), unsigned(tn));
  if (wide)
    launch_pdl(sgemm_kernel<FORM, 128>, grid, 256, 0, s, a);
  else
    launch_pdl(sgemm_kernel<FORM, 64>, grid, 256, 0, s, a);
  XMGN_LAUNCH_CHECK();
  return XMGN_OK;
}

// The terms that one running fp32 sum of a TN product may span: 4096, or 1/128 of
// all where there are more than 128 such chunks.  The rounding error of a chain
// grows with the root of its length and with its share of the whole sum.
int64_t tn_least_chunks(int64_t terms) {
  const int64_t c = (terms + 4095) / 4096;
  return c < 128 ? c : 128;
}

// Row chunks of a TN product: about two resident blocks per SM in one wave, at
// least 256 rows each; as many whole waves of them as keep every chain within the
// above.  With one wave always, a 512 x 512 gradient over 354k rows summed 18.6k
// rows in a chain (19 chunks, now 95): its relative error went from 8.4e-7 to
// 2.2e-7, a training step of one layer from 61.1 to 60.6 ms.
int tn_chunks(int64_t M, int64_t terms, int K1, int N) {
  const int64_t tiles = int64_t((K1 + BM - 1) / BM) * ((N + 127) / 128);
  int64_t c = 2 * int64_t(num_sms()) / tiles;
  if (c > (M + 255) / 256) c = (M + 255) / 256;
  if (c < 1) c = 1;
  const int64_t least = tn_least_chunks(terms);
  if (c < least) c *= (least + c - 1) / c;  // whole waves
  return int(c);
}

}  // namespace

xmgn_status gemm_nn_f32(const RowSrc& A, int64_t M, const float* B, int N, const float* bias, float* C, int64_t ldc,
                        int epi, float* pre, const float* aux, cudaStream_t s, const RowAdd& add) {
  if (M <= 0) return XMGN_OK;
  const SgemmArgs a{A, M, B, N, N, bias, C, ldc, epi, pre, aux, add, 0};
  if (fast(a)) return run_fast<G_NN>(a, M, 1, s);
  dim3 grid(unsigned((M + GT - 1) / GT), unsigned((N + GT - 1) / GT));
  launch_pdl(general_nnt_kernel<false>, grid, 256, 0, s, A, M, B, N, bias, C, ldc, epi, pre, aux, add);
  XMGN_LAUNCH_CHECK();
  return XMGN_OK;
}

xmgn_status gemm_nt_f32(const RowSrc& A, int64_t M, const float* B, int N, float* C, int64_t ldc, int epi,
                        const float* aux, cudaStream_t s) {
  if (M <= 0) return XMGN_OK;
  const SgemmArgs a{A, M, B, A.K, N, nullptr, C, ldc, epi, nullptr, aux, RowAdd{}, 0};
  if (fast(a)) return run_fast<G_NT>(a, M, 1, s);
  dim3 grid(unsigned((M + GT - 1) / GT), unsigned((N + GT - 1) / GT));
  launch_pdl(general_nnt_kernel<true>, grid, 256, 0, s, A, M, B, N, nullptr, C, ldc, epi, nullptr, aux, RowAdd{});
  XMGN_LAUNCH_CHECK();
  return XMGN_OK;
}

size_t gemm_tn_part_elems(int64_t M, int K1, int N) {
  // one wave: the chunk count falls as tiles are added, so count by tile: chunks * tiles <= max(2 SMs, tiles)
  const int64_t tm = (K1 + BM - 1) / BM, tn = (N + 127) / 128;
  const int64_t blocks = 2 * int64_t(num_sms()) > tm * tn ? 2 * int64_t(num_sms()) : tm * tn;
  // more waves: fewer than one wave's chunks above the least count
  return size_t(blocks) * BM * 128 + size_t(tn_least_chunks(M)) * size_t(K1) * size_t(N);
}

xmgn_status gemm_tn_f32(const RowSrc& A, int64_t M, const float* B, int64_t ldb, int N, float* G, float* part,
                        cudaStream_t s, int64_t terms) {
  const int K1 = A.K;
  const int nc = tn_chunks(M, terms > M ? terms : M, K1, N);
  int64_t rpc = (M + nc - 1) / nc;
  rpc = (rpc + BK - 1) / BK * BK;
  if (rpc < BK) rpc = BK;
  const SgemmArgs a{A, M, B, ldb, N, nullptr, part, N, EPI_STORE, nullptr, nullptr, RowAdd{}, rpc};
  if (fast(a) && K1 % 4 == 0) {
    XMGN_TRY(run_fast<G_TN>(a, K1, nc, s));
  } else {
    const int tiles = ((K1 + GT - 1) / GT) * ((N + GT - 1) / GT);
    launch_pdl(general_tn_kernel, dim3(tiles, nc), 256, 0, s, A, M, B, ldb, N, rpc, part);
    XMGN_LAUNCH_CHECK();
  }
  return sum_parts_f32(part, nc, K1 * N, G, s);
}

}  // namespace xmgn
