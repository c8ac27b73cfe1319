// k_sparse.cu -- sparse A (Sec. 5.2.1: the products cost 4 nnz(A) k flops).
//
//   P_W  = A Ht     : CSR SpMM, one warp per row of A; lane l accumulates the
//                     entries j = l, l+32, ... of the output row while the warp
//                     walks the row's nonzeros and gathers rows of Ht (n x k).
//   P_Ht = A^T W    : the same kernel over the CSC form of A (the CSR form of
//                     A^T), gathering rows of W (m x k).
// The CSC copy is built once per run on the device (k_csc.cu), each nonzero
// as an 8-byte {row, value}.
#include <algorithm>

#include "internal.cuh"

namespace aunmf {
namespace {

constexpr int kSpThreads = 256;
constexpr int kSpWarps = kSpThreads / kWarp;
static_assert(kSpMaxSegs == kSpThreads, "a segment per thread");
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

// Y's long row `i` from its chunks' partial sums, by a whole block: warp w adds the
// w-th eighth of the chunks in order, eight loads in flight, and the eighths are
// added in order.  (The partials were written by other blocks of this launch.)
template <int KT>
__device__ __forceinline__ void long_row_sum(const SpLongRows &lr, int64_t i, int64_t rows, int k,
                                             float *__restrict__ Y, float (&sw)[kSpWarps][32 * KT]) {
  (void)rows;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t r = lr.row[3 * i], base = lr.row[3 * i + 1], nc = lr.row[3 * i + 2];
  const int64_t per = (nc + kSpWarps - 1) / kSpWarps;
  const int64_t c0 = base + w * per, c1 = min(base + nc, c0 + per);
  __syncthreads();
#pragma unroll
  for (int t = 0; t < KT; ++t) {
    const int col = lane + 32 * t;
    float acc = 0.f;
    if (col < k) {
      int64_t c = c0;
      for (; c + 8 <= c1; c += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcg(&lr.part[(c + u) * k + col]);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += v[u];
      }
      for (; c < c1; ++c) acc += __ldcg(&lr.part[c * k + col]);
    }
    sw[w][32 * t + lane] = acc;
  }
  __syncthreads();
  if (!AUNMF_BOUND(r >= 0 && r < rows, AUNMF_CHECK_SPMM_RANGE)) return;
  for (int col = threadIdx.x; col < k; col += kSpThreads) {
    float y = sw[0][col];
#pragma unroll
    for (int q = 1; q < kSpWarps; ++q) y += sw[q][col];
    Y[r * k + col] = y;
  }
}

// Y (rows x k) = S (rows x ncols, row pointers and nonzeros, nnz of them) * X
// (ncols x k), a warp per row; before that, the first lr.blocks blocks (one wave)
// take the long rows' chunks.
//
// Long rows (a power-law hub can hold 10^6 nonzeros, which one warp would walk
// alone, ~50 ns a nonzero, while the rest of the GPU idles: 0.9 ms of a 2e7-
// nonzero product with rows of up to 18,000) are cut into chunks: a warp per
// chunk writes its partial sums, and the block that writes a row's last chunk adds
// all of them in chunk order (so results do not depend on scheduling).  The list
// is built on the device (k_list_long) in any order within a segment of the rows,
// each row's chunks in consecutive slots; nothing returns to the host.  One launch
// does all of it: as three (rows, chunks, sums) a matrix without long rows paid two
// empty ones (A H^T at 2000 x 1500, 20,000 nonzeros, k = 10: 22 us, now 13; at
// 300,001 x 200,003, 2e7 nonzeros with long rows, k = 32, both single products
// together 1788 us, now 1704).
// (Blocks an SM holds by the registers that the rows' part alone takes.)
template <int KT, class NZ>
__global__ void __launch_bounds__(kSpThreads, KT == 2 ? 6 : KT <= 4 ? 5 : KT == 8 ? 4 : 2)
    k_spmm(const int64_t *__restrict__ ptr, const NZ nz, int64_t rows, int64_t ncols, int64_t nnz,
           const float *__restrict__ X, int k, float *__restrict__ Y, const SpLongRows lr) {
  (void)nnz;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __shared__ float sw[kSpWarps][32 * KT];
  __shared__ int first[kSpMaxSegs + 1];  // chunks before each segment
  __shared__ int64_t fin[kSpWarps];      // the rows whose last chunk this block wrote
  const bool chunks = (int)blockIdx.x < lr.blocks;
  const int mine = chunks && (int)threadIdx.x < lr.nseg ? (int)lr.seg[threadIdx.x].chunks : 0;
  if (chunks && __syncthreads_or(mine)) {
    {  // prefix sums over the segments (at most one per thread)
      int v = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
      }
      if (lane == 31) fin[w] = v;
      __syncthreads();
      for (int q = 0; q < w; ++q) v += (int)fin[q];
      first[threadIdx.x + 1] = v;
      if (threadIdx.x == 0) first[0] = 0;
      __syncthreads();
    }
    const int total = first[lr.nseg];
    for (int c0 = blockIdx.x * kSpWarps; c0 < total; c0 += lr.blocks * kSpWarps) {
      const int c = c0 + w;
      int64_t done = -1;
      if (c < total) {
        int b = 0, e = lr.nseg;  // first[b] <= c < first[e]
        while (e - b > 1) {
          const int mid = (b + e) >> 1;
          if (first[mid] <= c) b = mid; else e = mid;
        }
        const int64_t slot = lr.seg[b].base + (c - first[b]);
        const int64_t e0 = lr.chunk[3 * slot], e1 = lr.chunk[3 * slot + 1];
        const int64_t i = lr.chunk[3 * slot + 2];
        if (AUNMF_BOUND(e0 >= 0 && e0 <= e1 && e1 <= nnz, AUNMF_CHECK_SPMM_RANGE)) {
          float acc[KT];
#pragma unroll
          for (int t = 0; t < KT; ++t) acc[t] = 0.f;
          spmm_range<KT>(nz, X, ncols, k, e0, e1, acc, lane);
#pragma unroll
          for (int t = 0; t < KT; ++t) {
            const int col = lane + 32 * t;
            if (col < k) lr.part[slot * k + col] = acc[t];
          }
        }
        __threadfence();
        __syncwarp();
        if (lane == 0) {
          const unsigned nc = (unsigned)lr.row[3 * i + 2];
          if (atomicInc(&lr.left[i], nc - 1) == nc - 1) done = i;  // (wraps to 0)
        }
      }
      if (lane == 0) fin[w] = done;
      __syncthreads();
      for (int q = 0; q < kSpWarps; ++q) {
        if (fin[q] < 0) continue;
        __threadfence();
        long_row_sum<KT>(lr, fin[q], rows, k, Y, sw);
      }
      __syncthreads();  // fin has been read
    }
  }
  const int64_t w0 = (int64_t)blockIdx.x * kSpWarps + w;
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

// The long rows of a row-pointer array, a block per segment of `per` rows: {row,
// first chunk, chunks} per row and {first, end nonzero, row's place} per chunk.  A
// segment's places start where its first nonzero says: a row of more than 512
// takes fewer than 1 / 512 places and 3 / 512 chunks a nonzero (ceil(n / 256) <= (n
// + 255) / 256 < 3 n / 512), so segments cannot meet and no counter is shared.
__device__ __forceinline__ void list_segment(const int64_t *__restrict__ ptr, int64_t rows,
                                             int64_t per, const SpLongRows &lr) {
  __shared__ int nlong, nchunks, bad;
  const int lane = threadIdx.x & 31;
  const int64_t s0 = blockIdx.x * per, s1 = min(rows, s0 + per);
  const int64_t p0 = max(ptr[s0], (int64_t)0);
  const int64_t row0 = p0 / kLongRowNz, chunk0 = 3 * p0 / kLongRowNz;
  if (threadIdx.x == 0) nlong = nchunks = bad = 0;
  __syncthreads();
  for (int64_t r0 = s0 + (threadIdx.x & ~31); r0 < s1; r0 += kSpThreads) {
    const int64_t r = r0 + lane;
    const int64_t e0 = r < s1 ? ptr[r] : 0, e1 = r < s1 ? ptr[r + 1] : 0;
    unsigned todo = __ballot_sync(0xffffffffu, e1 - e0 > kLongRowNz);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int64_t a = __shfl_sync(0xffffffffu, e0, src), b = __shfl_sync(0xffffffffu, e1, src);
      const int64_t cz = chunk_nz(b - a), nc = (b - a + cz - 1) / cz;
      int64_t i = 0, base = 0;
      if (lane == 0) {
        i = row0 + atomicAdd(&nlong, 1);
        base = chunk0 + atomicAdd(&nchunks, (int)nc);
      }
      i = __shfl_sync(0xffffffffu, i, 0);
      base = __shfl_sync(0xffffffffu, base, 0);
      // (always true for a well-formed row-pointer array of nnz nonzeros)
      if (i >= lr.cap_rows || base + nc > lr.cap_chunks) {
        bad = 1;
        continue;
      }
      if (lane == 0) {
        lr.row[3 * i] = r0 + src;
        lr.row[3 * i + 1] = base;
        lr.row[3 * i + 2] = nc;
        lr.left[i] = 0;
      }
      for (int64_t c = lane; c < nc; c += 32) {
        int64_t *d = lr.chunk + 3 * (base + c);
        d[0] = a + c * cz;
        d[1] = min(b, a + (c + 1) * cz);
        d[2] = i;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) lr.seg[blockIdx.x] = {chunk0, bad ? 0 : nchunks};
}

__global__ void __launch_bounds__(kSpThreads)
    k_list_long(const int64_t *__restrict__ ptr, int64_t rows, int64_t per, const SpLongRows lr) {
  list_segment(ptr, rows, per, lr);
}

// The same, and in the blocks after the segments' out (fc x fr) = in (fr x fc)^T: the
// factor that the product reads, in one launch (two took a small A H^T 2.5 us more).
__global__ void __launch_bounds__(kSpThreads)
    k_list_transpose(const int64_t *__restrict__ ptr, int64_t rows, int64_t per, const SpLongRows lr,
                     const float *__restrict__ in, int64_t fr, int64_t fc,
                     float *__restrict__ out) {
  __shared__ float t[32][33];
  if ((int)blockIdx.x < lr.nseg)
    list_segment(ptr, rows, per, lr);
  else
    transpose_tiles(in, fr, fc, out, (int64_t)blockIdx.x - lr.nseg, (int64_t)gridDim.x - lr.nseg, t,
                    threadIdx.x & 31, threadIdx.x >> 5, kSpThreads >> 5);
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
  const int nb = std::max(sp_blocks(rows), lr.blocks);
#define AUNMF_SP_MAIN(KT) \
  k_spmm<KT, NZ><<<nb, kSpThreads, 0, s>>>(ptr, nz, rows, ncols, nnz, X, k, Y, lr)
  AUNMF_SP_SWITCH(kt, AUNMF_SP_MAIN)
#undef AUNMF_SP_MAIN
  g_launches += 1;
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

namespace {
int64_t cap_long_rows(int64_t nnz) { return nnz / kLongRowNz + 1; }
int64_t cap_long_chunks(int64_t nnz) { return 3 * nnz / kLongRowNz + 1; }
}  // namespace

size_t long_rows_bytes(int64_t nnz) {
  const size_t cr = (size_t)cap_long_rows(nnz), cc = (size_t)cap_long_chunks(nnz);
  return sizeof(SpSegment) * kSpMaxSegs + sizeof(int64_t) * (3 * cr + 3 * cc) +
         sizeof(unsigned) * cr;
}

size_t long_part_bytes(int64_t nnz, int k) {
  return nnz <= kLongRowNz ? 0 : sizeof(float) * (size_t)cap_long_chunks(nnz) * k;
}

cudaError_t list_long_rows(const int64_t *ptr, int64_t rows, int64_t nnz, int k, void *mem,
                           float *part, SpLongRows *lr, cudaStream_t s, const float *in,
                           int64_t cols, float *out) {
  lr->cap_rows = cap_long_rows(nnz);
  lr->cap_chunks = cap_long_chunks(nnz);
  lr->seg = static_cast<SpSegment *>(mem);
  lr->row = reinterpret_cast<int64_t *>(lr->seg + kSpMaxSegs);
  lr->chunk = lr->row + 3 * lr->cap_rows;
  lr->left = reinterpret_cast<unsigned *>(lr->chunk + 3 * lr->cap_chunks);
  lr->part = part;
  lr->blocks = lr->nseg = 0;
  if (rows == 0 || nnz <= kLongRowNz)  // no long row
    return in ? launch_transpose(in, k, cols, out, s) : cudaSuccess;
  lr->blocks = (int)std::min<int64_t>((lr->cap_chunks + kSpWarps - 1) / kSpWarps, 152 * 4);
  const int64_t per = std::max<int64_t>(512, (rows + kSpMaxSegs - 1) / kSpMaxSegs);
  lr->nseg = (int)((rows + per - 1) / per);
  if (in) {
    const int64_t tiles = (k + 31) / 32 * ((cols + 31) / 32);
    k_list_transpose<<<(unsigned)(lr->nseg + std::min<int64_t>(tiles, 152 * 16)), kSpThreads, 0, s>>>(
        ptr, rows, per, *lr, in, k, cols, out);
  } else {
    k_list_long<<<(unsigned)lr->nseg, kSpThreads, 0, s>>>(ptr, rows, per, *lr);
  }
  g_launches += 1;
  return cudaGetLastError();
}

}  // namespace aunmf
