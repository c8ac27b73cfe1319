// k_sparse.cu -- sparse A (Sec. 5.2.1: the products cost 4 nnz(A) k flops).
//
//   P_W  = A Ht     : CSR SpMM, one warp per row of A; lane l accumulates the
//                     entries j = l, l+32, ... of the output row while the warp
//                     walks the row's nonzeros and gathers rows of Ht (n x k).
//   P_Ht = A^T W    : the same kernel over the CSC form of A (the CSR form of
//                     A^T), gathering rows of W (m x k).
// The CSC copy is built once per run on the device (k_csc.cu), each nonzero
// as an 8-byte {row, value}.
#include "internal.cuh"

namespace aunmf {
namespace {

constexpr int kSpThreads = 256;
constexpr int kSpWarps = kSpThreads / kWarp;
// Nonzeros per chunk of a long row of `len`: one warp's work.  Longer chunks
// for the longest rows, whose partial sums one block then adds.
__device__ __forceinline__ int64_t chunk_nz(int64_t len) { return len <= 32768 ? 256 : 512; }

// The nonzeros of a matrix: column (or row) indices and values in two arrays
// (CSR as given), or index and value bits side by side (the CSC copy: one
// 8-byte load per nonzero).
struct NzSplit {
  const int32_t *__restrict__ idx;
  const float *__restrict__ val;
  __device__ __forceinline__ void get(int64_t e, int &c, float &v) const {
    c = __ldg(idx + e);
    v = __ldg(val + e);
  }
};
struct NzPacked {
  const uint2 *__restrict__ nz;
  __device__ __forceinline__ void get(int64_t e, int &c, float &v) const {
    const uint2 q = __ldg(nz + e);
    c = (int)q.x;
    v = __uint_as_float(q.y);
  }
};

// acc[t] (lane's entries j = lane + 32 t) += sum over nonzeros e in [e0, e1)
// of val[e] X[idx[e], j]: the warp stages 32 nonzeros in registers, then
// broadcasts them and gathers the k-vectors of X (ncols rows), four at a
// time.  (ncols is read only by the checked build.)
template <int KT, class NZ>
__device__ __forceinline__ void spmm_range(const NZ &nz, const float *__restrict__ X, int64_t ncols,
                                           int k,
                                           int64_t e0, int64_t e1, float (&acc)[KT], int lane) {
  (void)ncols;
  for (int64_t eb = e0; eb < e1; eb += 32) {
    const int64_t e = eb + lane;
    int my_c = 0;
    float my_v = 0.f;
    if (e < e1) nz.get(e, my_c, my_v);
    const int cnt = (int)min((int64_t)32, e1 - eb);
    int j = 0;
    for (; j + 4 <= cnt; j += 4) {
      int c[4];
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        c[u] = __shfl_sync(0xffffffffu, my_c, j + u);
        v[u] = __shfl_sync(0xffffffffu, my_v, j + u);
      }
      float g[4][KT];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int t = 0; t < KT; ++t) {
          const int col = lane + 32 * t;
          g[u][t] = (col < k && AUNMF_BOUND((uint64_t)c[u] < (uint64_t)ncols,
                                            AUNMF_CHECK_SPMM_COLUMN))
                        ? __ldg(&X[(int64_t)c[u] * k + col])
                        : 0.f;
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int t = 0; t < KT; ++t) acc[t] = fmaf(v[u], g[u][t], acc[t]);
    }
    for (; j < cnt; ++j) {
      const int c = __shfl_sync(0xffffffffu, my_c, j);
      const float v = __shfl_sync(0xffffffffu, my_v, j);
#pragma unroll
      for (int t = 0; t < KT; ++t) {
        const int col = lane + 32 * t;
        if (col < k && AUNMF_BOUND((uint64_t)c < (uint64_t)ncols, AUNMF_CHECK_SPMM_COLUMN))
          acc[t] = fmaf(v, __ldg(&X[(int64_t)c * k + col]), acc[t]);
      }
    }
  }
}

// Y (rows x k) = S (rows x ncols, row pointers and nonzeros, nnz of them) * X
// (ncols x k), a warp per row.  Rows longer than kLongRowNz are left to the
// chunked kernels below.
template <int KT, class NZ>
__global__ void __launch_bounds__(kSpThreads)
    k_spmm(const int64_t *__restrict__ ptr, const NZ nz, int64_t rows, int64_t ncols, int64_t nnz,
           const float *__restrict__ X, int k, float *__restrict__ Y) {
  (void)nnz;
  const int lane = threadIdx.x & 31;
  const int64_t w0 = (int64_t)blockIdx.x * kSpWarps + (threadIdx.x >> 5);
  const int64_t ws = (int64_t)gridDim.x * kSpWarps;
  for (int64_t r = w0; r < rows; r += ws) {
    const int64_t e0 = ptr[r], e1 = ptr[r + 1];
    if (e1 - e0 > kLongRowNz) continue;
    if (!AUNMF_BOUND(e0 >= 0 && e0 <= e1 && e1 <= nnz, AUNMF_CHECK_SPMM_RANGE)) continue;
    float acc[KT];
#pragma unroll
    for (int t = 0; t < KT; ++t) acc[t] = 0.f;
    spmm_range<KT>(nz, X, ncols, k, e0, e1, acc, lane);
#pragma unroll
    for (int t = 0; t < KT; ++t) {
      const int col = lane + 32 * t;
      if (col < k) Y[r * k + col] = acc[t];
    }
  }
}

// Long rows (a power-law hub can hold 10^6 nonzeros, which one warp would walk
// alone, ~50 ns a nonzero, while the rest of the GPU idles: 0.9 ms of a 2e7-
// nonzero product with rows of up to 18,000): cut into chunks, a warp per
// chunk writes its partial sums, and a block per long row adds its chunks in
// chunk order (so results do not depend on scheduling).  The list is built on
// the device (k_list_long) in any order, each row's chunks in consecutive
// slots; nothing returns to the host.
template <int KT, class NZ>
__global__ void __launch_bounds__(kSpThreads)
    k_spmm_chunks(const NZ nz, int64_t ncols, int64_t nnz, const float *__restrict__ X, int k,
                  const SpLongRows lr) {
  (void)nnz;
  const int lane = threadIdx.x & 31;
  const int64_t w0 = (int64_t)blockIdx.x * kSpWarps + (threadIdx.x >> 5);
  const int64_t ws = (int64_t)gridDim.x * kSpWarps;
  const int64_t nchunks = min((int64_t)lr.count[1], lr.cap_chunks);
  for (int64_t c = w0; c < nchunks; c += ws) {
    const int64_t e0 = lr.chunk[2 * c], e1 = lr.chunk[2 * c + 1];
    if (!AUNMF_BOUND(e0 >= 0 && e0 <= e1 && e1 <= nnz, AUNMF_CHECK_SPMM_RANGE)) continue;
    float acc[KT];
#pragma unroll
    for (int t = 0; t < KT; ++t) acc[t] = 0.f;
    spmm_range<KT>(nz, X, ncols, k, e0, e1, acc, lane);
#pragma unroll
    for (int t = 0; t < KT; ++t) {
      const int col = lane + 32 * t;
      if (col < k) lr.part[c * k + col] = acc[t];
    }
  }
}

// Y's long rows: warp w of a row's block adds the w-th eighth of its chunks in
// order, eight loads in flight, and the eighths are added in order.
template <int KT>
__global__ void __launch_bounds__(kSpThreads)
    k_spmm_long_sum(const SpLongRows lr, int64_t rows, int k, float *__restrict__ Y) {
  (void)rows;
  __shared__ float sw[kSpWarps][32 * KT];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t nlong = min((int64_t)lr.count[0], lr.cap_rows);
  for (int64_t i = blockIdx.x; i < nlong; i += gridDim.x) {
    const int64_t r = lr.row[3 * i], base = lr.row[3 * i + 1], nc = lr.row[3 * i + 2];
    const int64_t per = (nc + kSpWarps - 1) / kSpWarps;
    const int64_t c0 = base + w * per, c1 = min(base + nc, c0 + per);
    float acc[KT];
#pragma unroll
    for (int t = 0; t < KT; ++t) {
      const int col = lane + 32 * t;
      acc[t] = 0.f;
      if (col >= k) continue;
      int64_t c = c0;
      for (; c + 8 <= c1; c += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = lr.part[(c + u) * k + col];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[t] += v[u];
      }
      for (; c < c1; ++c) acc[t] += lr.part[c * k + col];
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < KT; ++t) sw[w][32 * t + lane] = acc[t];
    __syncthreads();
    if (!AUNMF_BOUND(r >= 0 && r < rows, AUNMF_CHECK_SPMM_RANGE)) continue;
    for (int col = threadIdx.x; col < k; col += kSpThreads) {
      float y = sw[0][col];
#pragma unroll
      for (int q = 1; q < kSpWarps; ++q) y += sw[q][col];
      Y[r * k + col] = y;
    }
  }
}

// The long rows of a row-pointer array: {row, first chunk, chunks} per row and
// {first, end nonzero} per chunk, a warp per 32 rows.
__global__ void k_list_long(const int64_t *__restrict__ ptr, int64_t rows, const SpLongRows lr) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t ws = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r0 = w0 * 32; r0 < rows; r0 += ws * 32) {
    const int64_t r = r0 + lane;
    const int64_t e0 = r < rows ? ptr[r] : 0, e1 = r < rows ? ptr[r + 1] : 0;
    unsigned todo = __ballot_sync(0xffffffffu, e1 - e0 > kLongRowNz);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int64_t a = __shfl_sync(0xffffffffu, e0, src), b = __shfl_sync(0xffffffffu, e1, src);
      const int64_t cz = chunk_nz(b - a), nc = (b - a + cz - 1) / cz;
      long long i = 0, base = 0;
      if (lane == 0) {
        i = (long long)atomicAdd(&lr.count[0], 1ull);
        base = (long long)atomicAdd(&lr.count[1], (unsigned long long)nc);
      }
      i = __shfl_sync(0xffffffffu, i, 0);
      base = __shfl_sync(0xffffffffu, base, 0);
      // (always true for a well-formed row-pointer array of nnz nonzeros)
      if (i >= lr.cap_rows || base + nc > lr.cap_chunks) continue;
      if (lane == 0) {
        lr.row[3 * i] = r0 + src;
        lr.row[3 * i + 1] = base;
        lr.row[3 * i + 2] = nc;
      }
      for (int64_t c = lane; c < nc; c += 32) {
        lr.chunk[2 * (base + c)] = a + c * cz;
        lr.chunk[2 * (base + c) + 1] = min(b, a + (c + 1) * cz);
      }
    }
  }
}

int sp_blocks(int64_t warps) {
  int64_t nb = (warps + kSpWarps - 1) / kSpWarps;
  if (nb > 152 * 16) nb = 152 * 16;
  return nb < 1 ? 1 : (int)nb;
}

#define AUNMF_SP_SWITCH(KTV, CALL) \
  switch (KTV) {                   \
    case 1: CALL(1); break;        \
    case 2: CALL(2); break;        \
    case 3: CALL(3); break;        \
    case 4: CALL(4); break;        \
    case 5: case 6: case 7:        \
    case 8: CALL(8); break;        \
    default: CALL(16); break;      \
  }

template <class NZ>
cudaError_t spmm(const int64_t *ptr, const NZ nz, int64_t rows, int64_t ncols, int64_t nnz,
                 const float *X, int k, float *Y, const SpLongRows &lr, cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  const int kt = (k + 31) / 32;
  const int nb = sp_blocks(rows);
#define AUNMF_SP_MAIN(KT) \
  k_spmm<KT, NZ><<<nb, kSpThreads, 0, s>>>(ptr, nz, rows, ncols, nnz, X, k, Y)
  AUNMF_SP_SWITCH(kt, AUNMF_SP_MAIN)
#undef AUNMF_SP_MAIN
  g_launches += 1;
  if (nnz > kLongRowNz) {
    const int nbc = sp_blocks(lr.cap_chunks);
    const int nbl = (int)(lr.cap_rows < 152 * 4 ? lr.cap_rows : 152 * 4);
#define AUNMF_SP_CH(KT)                                                                        \
  k_spmm_chunks<KT, NZ><<<nbc, kSpThreads, 0, s>>>(nz, ncols, nnz, X, k, lr);                   \
  k_spmm_long_sum<KT><<<nbl, kSpThreads, 0, s>>>(lr, rows, k, Y)
    AUNMF_SP_SWITCH(kt, AUNMF_SP_CH)
#undef AUNMF_SP_CH
    g_launches += 2;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_aht_csr(const int64_t *rowptr, const int32_t *colidx, const float *val,
                           int64_t m, int64_t n, int64_t nnz, const float *Ht, int k, float *P,
                           const SpLongRows &lr, cudaStream_t s) {
  return spmm(rowptr, NzSplit{colidx, val}, m, n, nnz, Ht, k, P, lr, s);
}

cudaError_t launch_wta_csc(const int64_t *colptr, const uint2 *cnz, int64_t n, int64_t m,
                           int64_t nnz, const float *W, int k, float *P, const SpLongRows &lr,
                           cudaStream_t s) {
  return spmm(colptr, NzPacked{cnz}, n, m, nnz, W, k, P, lr, s);
}

size_t long_rows_bytes(int64_t nnz, int k) {
  const int64_t cr = nnz / kLongRowNz + 1, cc = nnz / 256 + cr + 1;
  return sizeof(int64_t) * (size_t)(2 + 3 * cr + 2 * cc) + sizeof(float) * (size_t)cc * k;
}

cudaError_t list_long_rows(const int64_t *ptr, int64_t rows, int64_t nnz, int k, void *mem,
                           SpLongRows *lr, cudaStream_t s) {
  lr->cap_rows = nnz / kLongRowNz + 1;
  lr->cap_chunks = nnz / 256 + lr->cap_rows + 1;
  int64_t *p = static_cast<int64_t *>(mem);
  lr->count = reinterpret_cast<unsigned long long *>(p);
  lr->row = p + 2;
  lr->chunk = lr->row + 3 * lr->cap_rows;
  lr->part = reinterpret_cast<float *>(lr->chunk + 2 * lr->cap_chunks);
  if (rows == 0 || nnz <= kLongRowNz) return cudaSuccess;  // no long row: spmm skips the pass
  cudaError_t e = cudaMemsetAsync(lr->count, 0, 2 * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  int64_t nb = (rows + 255) / 256;
  if (nb > 152 * 16) nb = 152 * 16;
  k_list_long<<<(unsigned)nb, 256, 0, s>>>(ptr, rows, *lr);
  g_launches += 1;
  return cudaGetLastError();
}

}  // namespace aunmf
