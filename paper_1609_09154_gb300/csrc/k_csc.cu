// k_csc.cu -- the CSC form of a sparse A (CSR in, CSC out), built once per
// run for the W^T A product (Sec. 5.2.1).
//
// The nonzeros, each packed as an 8-byte {row, value}, are sorted by column
// with a stable radix sort (CUB); the CSR order is row-major, so the entries
// of every column come out in row order, whatever the column's length.  The
// sorted records are the CSC's nonzeros as the product reads them, and the
// column pointers are read off the sorted keys (the first position of each
// column), so no step uses atomics: a column with a million entries (a
// power-law hub) costs no more than a million columns of one.  Carrying the
// records through the sort's passes costs 24 bytes a nonzero and pass instead
// of 16; sorting positions and then gathering rows and values through them
// read two 32-byte sectors a nonzero (1.88 ms of 2.9 for 5e7 nonzeros).
#include <cub/device/device_radix_sort.cuh>

#include "internal.cuh"

namespace aunmf {
namespace {

constexpr int kCscThreads = 256;

int grid_for(int64_t items, int per_sm) {
  int64_t nb = (items + kCscThreads - 1) / kCscThreads;
  if (nb > 152LL * per_sm) nb = 152LL * per_sm;
  return nb < 1 ? 1 : (int)nb;
}

// nz[e] = {r, value bits} for the nonzeros e of row r (a warp per row).
__global__ void k_pack_nz(const int64_t *__restrict__ rowptr, const float *__restrict__ val,
                          int64_t m, int64_t nnz, uint2 *__restrict__ nz) {
  (void)nnz;
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t ws = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = w0; r < m; r += ws)
    for (int64_t e = rowptr[r] + lane; e < rowptr[r + 1]; e += 32)
      if (AUNMF_BOUND(e >= 0 && e < nnz, AUNMF_CHECK_CSC))
        nz[e] = make_uint2((uint32_t)r, __float_as_uint(val[e]));
}

// colptr[c] = the first q with key[q] >= c (c = 0..n): position q starts the
// columns key[q-1]+1 .. key[q] (from 0 at q = 0), and colptr[c] = nnz for the
// columns after the last key.
__global__ void k_colptr(const int32_t *__restrict__ key, int64_t nnz, int64_t n,
                         int64_t *__restrict__ colptr) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nnz;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c1 = key[q];
    if (!AUNMF_BOUND(c1 >= 0 && c1 < n, AUNMF_CHECK_CSC)) continue;
    const int64_t c0 = q == 0 ? 0 : (int64_t)key[q - 1] + 1;
    for (int64_t c = c0; c <= c1; ++c) colptr[c] = q;
  }
}

__global__ void k_colptr_tail(const int32_t *__restrict__ key, int64_t nnz, int64_t n,
                              int64_t *__restrict__ colptr) {
  const int64_t c0 = nnz > 0 ? (int64_t)key[nnz - 1] + 1 : 0;
  for (int64_t c = c0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c <= n;
       c += (int64_t)gridDim.x * blockDim.x)
    colptr[c] = nnz;
}

int key_bits(int64_t n) {
  int b = 1;
  while (b < 31 && (1LL << b) < n) ++b;
  return b;
}

// (the records are 8-byte values to the sort)
typedef unsigned long long Rec;

size_t sort_temp_bytes(int64_t nnz, int64_t n) {
  size_t t = 0;
  cub::DeviceRadixSort::SortPairs(nullptr, t, static_cast<const int32_t *>(nullptr),
                                  static_cast<int32_t *>(nullptr),
                                  static_cast<const Rec *>(nullptr), static_cast<Rec *>(nullptr),
                                  (int)nnz, 0, key_bits(n));
  return t;
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

// Scratch: sorted keys, the records in row order, and the sort's temporary
// storage (12 bytes a nonzero + the CUB buffer).
size_t csc_scratch_bytes(int64_t n, int64_t nnz) {
  const size_t e = (size_t)(nnz > 0 ? nnz : 1);
  return al256(sizeof(int32_t) * e) + al256(sizeof(Rec) * e) + al256(sort_temp_bytes(nnz, n)) + 256;
}

cudaError_t launch_csr_to_csc(const int64_t *rowptr, const int32_t *colidx, const float *val,
                              int64_t m, int64_t n, int64_t nnz, int64_t *colptr, uint2 *cnz,
                              void *scratch, cudaStream_t s) {
  if (nnz > 0x7fffffffLL || n > 0x7fffffffLL) return cudaErrorInvalidValue;
  char *p = static_cast<char *>(scratch);
  const size_t e = (size_t)(nnz > 0 ? nnz : 1);
  int32_t *key = reinterpret_cast<int32_t *>(p);
  Rec *rec = reinterpret_cast<Rec *>(p + al256(sizeof(int32_t) * e));
  void *temp = p + al256(sizeof(int32_t) * e) + al256(sizeof(Rec) * e);
  size_t temp_bytes = sort_temp_bytes(nnz, n);
  if (nnz > 0) {
    k_pack_nz<<<grid_for(m * 32, 16), kCscThreads, 0, s>>>(rowptr, val, m, nnz,
                                                          reinterpret_cast<uint2 *>(rec));
    cudaError_t err = cub::DeviceRadixSort::SortPairs(temp, temp_bytes, colidx, key, rec,
                                                      reinterpret_cast<Rec *>(cnz), (int)nnz, 0,
                                                      key_bits(n), s);
    if (err != cudaSuccess) return err;
    k_colptr<<<grid_for(nnz, 16), kCscThreads, 0, s>>>(key, nnz, n, colptr);
    g_launches += 2;
  }
  k_colptr_tail<<<grid_for(n + 1, 4), kCscThreads, 0, s>>>(key, nnz, n, colptr);
  g_launches += 1;
  return cudaGetLastError();
}

}  // namespace aunmf
