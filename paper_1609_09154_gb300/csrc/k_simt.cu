// k_simt.cu -- FP32/FP64 CUDA-core kernels of the AU-NMF hot path:
//   * Gram matrices X^T X (Alg. 1 lines 3-4: H H^T, W^T W; the all-reduce of
//     Alg. 3 becomes a fixed-order FP64 reduction of per-block partials)
//   * the two products with A on CUDA cores (Alg. 1: A H^T, W^T A)
//   * transposes, ||A||^2 and the relative residual of Sec. 6.2 from the
//     expansion ||A||^2 - 2 <W^T A, H> + <W^T W, H H^T>.
// Internally H is held transposed (Ht, n x k) so that both factors are
// row-major "rows x k" and share the same update kernels.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "ptx.cuh"

namespace aunmf {

// ------------------------------------------------------------------ Gram
// Block b accumulates X^T X over rows [b*chunk, (b+1)*chunk) into
// partials[b] (k x k).  Each thread owns a 4x4 tile of G's upper triangle;
// rows are staged in shared memory 64 at a time.  There are only
// nt (nt + 1) / 2 tiles (91 at k = 50), so the block's threads form
// ngrp = 256 / tiles groups (2 at k = 50, 7 at k = 32), each covering every
// tile for its share of the staged rows (row g, g + ngrp, ...) with running
// sums of its own; the groups' sums are added in group order at the end, so
// the result does not depend on scheduling.
namespace {
constexpr int kGramRows = 64;
constexpr int kGramThreads = 256;
// rows of a group summed in a fresh register before they join the running
// sum (FP32 path) or the FP64 sum (FP64-accurate path)
constexpr int kGramSlab = 32;

// True in exactly one block of the launch, the last to arrive, whose threads
// then see what every block wrote before.  *ticket wraps back to 0.
__device__ __forceinline__ bool last_block(unsigned *ticket) {
  __shared__ unsigned order;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) order = atomicInc(ticket, gridDim.x - 1);
  __syncthreads();
  if (order != gridDim.x - 1) return false;
  __threadfence();
  return true;
}

__device__ __forceinline__ int gram_groups(int ntiles) {
  return ntiles >= kGramThreads ? 1 : kGramThreads / ntiles;
}

// The per-block partial of G = X^T X over the block's rows.
//   FP64 = false: each group's slab of up to 32 rows is summed in a fresh
//     FP32 register and added to an FP32 running sum with Kahan's
//     compensation (the residual's expansion <W^T W, H H^T> needs the Grams
//     to ~1e-7; FP64 additions, at ~2 per SM per clock on this part, would
//     bound the kernel).
//   FP64 = true: within a slab each product is formed exactly and summed in
//     an FP32 pair (hi, lo) (two_fma_acc), and the slab's pair is added to
//     an FP64 running sum: ~1e-14 relative, so a Gram whose smallest
//     eigenvalues sit below FP32's resolution of its largest (condition
//     beyond ~1e7, which ABPP's factors reach on uniform low-rank data) stays
//     positive definite.
// The next 64-row slab is loaded into registers while the current one is
// consumed from shared memory.  Dynamic shared memory: gram_smem_bytes().
// LAST (FP32): the last block to finish adds all partials in FP64 and writes G;
// *ticket starts at 0 and is 0 again after (see launch_gram on when).
template <bool FP64, bool LAST>
__global__ void __launch_bounds__(kGramThreads, 2)
    k_gram_part(const float *__restrict__ X, int64_t rows, int k, int64_t ldx, int64_t chunk,
                typename std::conditional<FP64, double, float>::type *__restrict__ partials,
                float *__restrict__ G, unsigned *ticket) {
  using T = typename std::conditional<FP64, double, float>::type;
  extern __shared__ __align__(16) float sX[];  // [kGramRows][kp], then the group sums
  constexpr int kPre = (kGramRows * 64 + kGramThreads - 1) / kGramThreads;  // k <= 64 prefetch
  const int kp = (k + 3) & ~3;
  const int nt = kp / 4, ntiles = nt * (nt + 1) / 2;
  const int ngrp = gram_groups(ntiles);
  const int64_t r0 = (int64_t)blockIdx.x * chunk;
  const int64_t r1 = min(rows, r0 + chunk);
  T *out = partials + (int64_t)blockIdx.x * k * k;
  const int slab = kGramRows * kp;
  const bool pre = slab <= kPre * kGramThreads;
  T *gsum = reinterpret_cast<T *>(sX + ((slab + 3) & ~3));  // [ngrp][ntiles][16]
  for (int tb = 0; tb < ntiles; tb += kGramThreads) {
    const int g = ngrp > 1 ? (int)threadIdx.x / ntiles : 0;
    const int t = tb + (ngrp > 1 ? (int)threadIdx.x % ntiles : (int)threadIdx.x);
    const bool act = g < ngrp && t < ntiles;
    // t -> (ti, tj), ti <= tj, row-major over the upper triangle
    int ti = 0, tj = 0;
    if (act) {
      int rem = t;
      while (rem >= nt - ti) { rem -= nt - ti; ++ti; }
      tj = ti + rem;
    }
    T sum[4][4];
    float cmp[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        sum[a][b] = T(0);
        cmp[a][b] = 0.f;
      }
    float nxt[kPre];
    // slab index idx -> (row, column) = (idx / kp, idx % kp) by a float
    // reciprocal: idx < 4096 and kp <= 64 keep (idx + 0.5) / kp at least
    // 1 / 128 away from an integer, far beyond the product's rounding, so the
    // truncation is exact (an integer division costs ~20 instructions, and
    // took most of the kernel's issue slots)
    const float inv_kp = 1.f / (float)kp;
    auto fetch = [&](int64_t c0) {
      const int nr = (int)min((int64_t)kGramRows, r1 - c0);
#pragma unroll
      for (int q = 0; q < kPre; ++q) {
        const int idx = threadIdx.x + q * kGramThreads;
        const int rr = __float2int_rz(((float)idx + 0.5f) * inv_kp), cc = idx - rr * kp;
        nxt[q] = (idx < slab && rr < nr && cc < k) ? X[(c0 + rr) * ldx + cc] : 0.f;
      }
    };
    if (pre && r0 < r1) fetch(r0);
    for (int64_t c0 = r0; c0 < r1; c0 += kGramRows) {
      const int nr = (int)min((int64_t)kGramRows, r1 - c0);
      __syncthreads();
      if (pre) {
#pragma unroll
        for (int q = 0; q < kPre; ++q) {
          const int idx = threadIdx.x + q * kGramThreads;
          if (idx < slab) sX[idx] = nxt[q];
        }
        if (c0 + kGramRows < r1) fetch(c0 + kGramRows);
      } else {
        // (eight loads in flight; left to the compiler, the loop's form depended on
        // code elsewhere in the kernel: 20,000 rows, k = 90: 55 against 49 us)
#pragma unroll 8
        for (int idx = threadIdx.x; idx < slab; idx += kGramThreads) {
          const int rr = __float2int_rz(((float)idx + 0.5f) * inv_kp), cc = idx - rr * kp;
          sX[idx] = (rr < nr && cc < k) ? X[(c0 + rr) * ldx + cc] : 0.f;
        }
      }
      __syncthreads();
      if (act) {
        // the group's rows of this stage, kGramSlab at a time
        for (int s0 = g; s0 < nr; s0 += kGramSlab * ngrp) {
          const int s1 = min(nr, s0 + kGramSlab * ngrp);
          float hi[4][4] = {}, lo[4][4] = {};
          for (int rr = s0; rr < s1; rr += ngrp) {
            const float4 a = *reinterpret_cast<const float4 *>(&sX[rr * kp + 4 * ti]);
            const float4 b = *reinterpret_cast<const float4 *>(&sX[rr * kp + 4 * tj]);
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                if constexpr (FP64)
                  two_fma_acc(av[p], bv[q], hi[p][q], lo[p][q]);
                else
                  hi[p][q] = fmaf(av[p], bv[q], hi[p][q]);
              }
          }
#pragma unroll
          for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if constexpr (FP64) {
                sum[p][q] += (double)hi[p][q] + (double)lo[p][q];
              } else {
                const float y = hi[p][q] - cmp[p][q];
                const float tt = sum[p][q] + y;
                cmp[p][q] = (tt - sum[p][q]) - y;
                sum[p][q] = tt;
              }
            }
        }
      }
    }
    // the groups' sums: every entry of every tile is added over the groups by a
    // thread of its own, in group order (FP64: four interleaved chains; one
    // thread per tile doing its 16 entries took most of a small factor's 11-44
    // us: ngrp is 42 at k = 10)
    __syncthreads();
    if (act && ngrp > 1) {
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          gsum[((size_t)g * ntiles + t) * 16 + 4 * p + q] = FP64 ? sum[p][q] : sum[p][q] - cmp[p][q];
    }
    __syncthreads();
    if (ngrp > 1) {
      const int ne = ntiles * 16;
      for (int e = threadIdx.x; e < ne; e += kGramThreads) {
        constexpr int kChains = FP64 ? 4 : 1;
        T c[kChains] = {};
        int h = 0;
#pragma unroll 4
        for (; h + kChains <= ngrp; h += kChains)
#pragma unroll
          for (int u = 0; u < kChains; ++u) c[u] += gsum[(size_t)(h + u) * ne + e];
        for (; h < ngrp; ++h) c[0] += gsum[(size_t)h * ne + e];
        T v = c[0];
        if constexpr (FP64) v = (c[0] + c[1]) + (c[2] + c[3]);
        int rem = e >> 4, i = 0;
        while (rem >= nt - i) { rem -= nt - i; ++i; }
        const int gi = 4 * i + ((e >> 2) & 3), gj = 4 * (i + rem) + (e & 3);
        if (gi < k && gj < k) {
          out[gi * k + gj] = v;
          out[gj * k + gi] = v;
        }
      }
    } else if (act) {
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const T v = FP64 ? sum[p][q] : sum[p][q] - cmp[p][q];
          const int i = 4 * ti + p, j = 4 * tj + q;
          if (i < k && j < k) {
            out[i * k + j] = v;
            out[j * k + i] = v;
          }
        }
    }
  }
  if constexpr (LAST) {
    if (!last_block(ticket)) return;
    const int kk = k * k, nb = gridDim.x;
    for (int e = threadIdx.x; e < kk; e += kGramThreads) {
      double a[8] = {};
      int b = 0;
      for (; b + 8 <= nb; b += 8)
#pragma unroll
        for (int u = 0; u < 8; ++u) a[u] += (double)__ldcg(&partials[(int64_t)(b + u) * kk + e]);
      for (; b < nb; ++b) a[0] += (double)__ldcg(&partials[(int64_t)b * kk + e]);
      G[e] = (float)(((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7])));
    }
  }
}

// k_gram8: the FP32 Gram of a factor with contiguous rows (ldx == k, k <= 64,
// 16-byte aligned), with 8 x 8 register tiles.  A block (one per SM) walks
// its rows in stages of kG8Rows: each stage is one contiguous span of the
// factor, copied with 16-byte loads at the span's own offsets into shared
// memory (no index arithmetic) while the previous stage is consumed.
// Thread (g, t): tile t = (ti, tj), ti <= tj, of the upper triangle in 8 x 8
// blocks (28 tiles at k = 50, 36 at 64), row group g of ngrp = 256 / tiles
// (rows g, g + ngrp, ... of each stage).  Each row costs a thread 16 values
// (float2 loads for even k) and 64 FFMAs, against 8 values and 16 FFMAs per
// row in k_gram_part's 4 x 4 tiles.  As there, slabs are summed in fresh
// registers and folded into Kahan-compensated running sums (~64 rows a
// slab; the sums in registers, the corrections in shared memory), and the
// groups' sums are added in group order, so the result does not depend on
// scheduling.
constexpr int kG8Threads = 256, kG8Rows = 128, kG8MaxK = 64;
constexpr int kG8Buf = kG8Rows * kG8MaxK + 8;  // floats per stage buffer (+ tail pad)
constexpr int kG8Ldc = 68;                     // floats per thread row of corrections
constexpr int kG8Pre = kG8Rows * kG8MaxK / 4 / kG8Threads;  // float4 prefetch per thread
constexpr size_t kG8Smem = sizeof(float) * (2 * (size_t)kG8Buf + (size_t)kG8Threads * kG8Ldc);

template <bool EVEN>
__global__ void __launch_bounds__(kG8Threads, 1)
    k_gram8(const float *__restrict__ X, int64_t rows, int k, int64_t chunk,
            float *__restrict__ partials) {
  extern __shared__ __align__(16) float sg[];
  float *buf0 = sg, *buf1 = sg + kG8Buf;
  float *corr = sg + 2 * kG8Buf;
  const int tid = threadIdx.x;
  const int nt = (k + 7) >> 3, ntiles = nt * (nt + 1) / 2;
  const int ngrp = kG8Threads / ntiles;
  const int g = tid / ntiles, t = tid - g * ntiles;
  const bool act = g < ngrp;
  int ti = 0, tj = 0;
  if (act) {
    int rem = t;
    while (rem >= nt - ti) { rem -= nt - ti; ++ti; }
    tj = ti + rem;
  }
  // stages per slab: ~64 of the thread's own rows between folds
  const int fold_every = max(1, (64 * ngrp + kG8Rows / 2) / kG8Rows);
  const int64_t r0 = (int64_t)blockIdx.x * chunk, r1 = min(rows, r0 + chunk);
  float *kc = corr + (size_t)tid * kG8Ldc;
#pragma unroll
  for (int e = 0; e < 64; e += 4) *reinterpret_cast<float4 *>(kc + e) = make_float4(0.f, 0.f, 0.f, 0.f);
  float acc[8][8], hi[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = hi[i][j] = 0.f;

  // stage c0: the span X[c0 k, (c0 + nr) k), float4 groups then <= 3 floats
  float4 pre[kG8Pre];
  float tailv = 0.f;
  auto fetch = [&](int64_t c0) {
    const int nr = (int)min((int64_t)kG8Rows, r1 - c0);
    const int len = nr * k, n4 = len >> 2;
    const float4 *src = reinterpret_cast<const float4 *>(X + c0 * k);
#pragma unroll
    for (int q = 0; q < kG8Pre; ++q) {
      const int i4 = tid + q * kG8Threads;
      pre[q] = i4 < n4 ? __ldcs(src + i4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    tailv = tid < (len & 3) ? X[c0 * k + (n4 << 2) + tid] : 0.f;
  };
  auto store = [&](float *b, int64_t c0) {
    const int nr = (int)min((int64_t)kG8Rows, r1 - c0);
    const int len = nr * k, n4 = len >> 2;
#pragma unroll
    for (int q = 0; q < kG8Pre; ++q) {
      const int i4 = tid + q * kG8Threads;
      if (i4 < n4) *reinterpret_cast<float4 *>(b + 4 * i4) = pre[q];
    }
    if (tid < (len & 3)) b[(n4 << 2) + tid] = tailv;
  };
  auto fold = [&]() {
#pragma unroll
    for (int e4 = 0; e4 < 64; e4 += 4) {
      float4 cv = *reinterpret_cast<const float4 *>(kc + e4);
      float *c = &cv.x;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e4 + u, i = e >> 3, j = e & 7;
        const float y = acc[i][j] - c[u];
        const float tt = hi[i][j] + y;
        c[u] = (tt - hi[i][j]) - y;
        hi[i][j] = tt;
        acc[i][j] = 0.f;
      }
      *reinterpret_cast<float4 *>(kc + e4) = cv;
    }
  };
  auto load8 = [&](const float *p, float (&v)[8]) {
    if constexpr (EVEN) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float2 w = *reinterpret_cast<const float2 *>(p + 2 * u);
        v[2 * u] = w.x;
        v[2 * u + 1] = w.y;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p[u];
    }
  };

  if (r0 < r1) {
    fetch(r0);
    store(buf0, r0);
  }
  __syncthreads();
  int stage = 0;
  float *cur = buf0, *nxt = buf1;
  for (int64_t c0 = r0; c0 < r1; c0 += kG8Rows, ++stage) {
    const int nr = (int)min((int64_t)kG8Rows, r1 - c0);
    const bool more = c0 + kG8Rows < r1;
    if (more) fetch(c0 + kG8Rows);
    if (act) {
      for (int rr = g; rr < nr; rr += ngrp) {
        const float *row = cur + rr * k;
        float a[8], b[8];
        load8(row + 8 * ti, a);
        load8(row + 8 * tj, b);
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
      }
      if ((stage + 1) % fold_every == 0 || !more) fold();
    }
    if (more) store(nxt, c0 + kG8Rows);
    __syncthreads();
    float *tmp = cur;
    cur = nxt;
    nxt = tmp;
  }
  // the groups' sums (hi - c), added in group order by group 0
  float *gs = sg;  // ngrp x ntiles x 64 floats, over the stage buffers
  __syncthreads();
  if (act && g > 0) {
#pragma unroll
    for (int e = 0; e < 64; ++e) gs[((size_t)g * ntiles + t) * 64 + e] = hi[e >> 3][e & 7] - kc[e];
  }
  __syncthreads();
  if (act && g == 0) {
    float *out = partials + (int64_t)blockIdx.x * k * k;
#pragma unroll
    for (int e = 0; e < 64; ++e) {
      float v = hi[e >> 3][e & 7] - kc[e];
      for (int h = 1; h < ngrp; ++h) v += gs[((size_t)h * ntiles + t) * 64 + e];
      const int i = 8 * ti + (e >> 3), j = 8 * tj + (e & 7);
      if (i < k && j < k) {
        out[i * k + j] = v;
        out[j * k + i] = v;
      }
    }
  }
}

template <bool FP64>
size_t gram_smem_bytes(int k) {
  const int kp = (k + 3) & ~3, nt = kp / 4, ntiles = nt * (nt + 1) / 2;
  const int ngrp = ntiles >= kGramThreads ? 1 : kGramThreads / ntiles;
  const size_t slab = (size_t)((kGramRows * kp + 3) & ~3) * sizeof(float);
  const size_t grp = ngrp > 1 ? (size_t)ngrp * ntiles * 16 * (FP64 ? sizeof(double) : sizeof(float)) : 0;
  return slab + grp;
}

// G_e = sum_b partials[b]_e in FP64: 32 entries per block; each of the block's
// warps sums its share of the partials in four interleaved chains (b
// ascending within each), and the chains and then the warps' sums are added
// in a fixed order, so the result does not depend on scheduling.  32 warps for
// many partials (with eight, 188 partials at k = 50 took 10 us a call), eight
// for few (a wide Gram's 13-19 partials: 11 us at k = 256, 29 us with 32).
int gram_red_threads(int nb) { return nb >= 64 ? 1024 : 256; }
// chains8 (few values, kChainValues): eight warps sum the partials b = w mod 8 each,
// the last nb mod 8 after warp 0's, and the chains are added pairwise -- an order
// that small ABPP Grams keep, whose last bits (1e-16) decide the fifth digit of a
// residual near 2e-3.
constexpr int64_t kChainValues = 24000;
__global__ void __launch_bounds__(1024)
    k_gram_reduce_d(const double *__restrict__ partials, int nb, int k, bool chains8,
                    double *__restrict__ G64, float *__restrict__ G32) {
  __shared__ double sw[32][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int kk = k * k;
  const int e = blockIdx.x * 32 + lane;
  const int nw = blockDim.x >> 5, per = (nb + nw - 1) / nw;
  const int b0 = w * per, b1 = min(nb, b0 + per);
  // four independent chains (loads in flight, FP64 latency overlapped),
  // combined in a fixed order
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  if (e < kk && chains8) {
    const int nb8 = nb & ~7;
#pragma unroll 4
    for (int b = w; b < nb8; b += 8) a0 += partials[(int64_t)b * kk + e];
    if (w == 0)
      for (int b = nb8; b < nb; ++b) a0 += partials[(int64_t)b * kk + e];
  } else if (e < kk) {
    int b = b0;
    for (; b + 4 <= b1; b += 4) {
      a0 += partials[(int64_t)b * kk + e];
      a1 += partials[(int64_t)(b + 1) * kk + e];
      a2 += partials[(int64_t)(b + 2) * kk + e];
      a3 += partials[(int64_t)(b + 3) * kk + e];
    }
    for (; b < b1; ++b) a0 += partials[(int64_t)b * kk + e];
  }
  sw[w][lane] = (a0 + a1) + (a2 + a3);
  __syncthreads();
  if (w == 0 && e < kk) {
    double s = 0.0;
    if (chains8)
      s = ((sw[0][lane] + sw[1][lane]) + (sw[2][lane] + sw[3][lane])) +
          ((sw[4][lane] + sw[5][lane]) + (sw[6][lane] + sw[7][lane]));
    else
      for (int q = 0; q < nw; ++q) s += sw[q][lane];
    G64[e] = s;
    if (G32) G32[e] = (float)s;
  }
}

__global__ void k_widen(const float *__restrict__ G32, int kk, double *__restrict__ G64) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < kk; e += gridDim.x * blockDim.x)
    G64[e] = (double)G32[e];
}

__global__ void __launch_bounds__(1024)
    k_gram_reduce(const float *__restrict__ partials, int nb, int k, float *__restrict__ G) {
  __shared__ double sw[32][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int kk = k * k;
  const int e = blockIdx.x * 32 + lane;
  const int nw = blockDim.x >> 5, per = (nb + nw - 1) / nw;
  const int b0 = w * per, b1 = min(nb, b0 + per);
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  if (e < kk) {
    int b = b0;
    for (; b + 4 <= b1; b += 4) {
      a0 += (double)partials[(int64_t)b * kk + e];
      a1 += (double)partials[(int64_t)(b + 1) * kk + e];
      a2 += (double)partials[(int64_t)(b + 2) * kk + e];
      a3 += (double)partials[(int64_t)(b + 3) * kk + e];
    }
    for (; b < b1; ++b) a0 += (double)partials[(int64_t)b * kk + e];
  }
  sw[w][lane] = (a0 + a1) + (a2 + a3);
  __syncthreads();
  if (w == 0 && e < kk) {
    double t = 0.0;
    for (int i = 0; i < nw; ++i) t += sw[i][lane];
    G[e] = (float)t;
  }
}
}  // namespace

int gram_partial_blocks(int64_t rows, int max_blocks) {
  int64_t nb = (rows + 127) / 128;  // at least 128 rows per block
  if (nb > max_blocks) nb = max_blocks;
  if (nb < 1) nb = 1;
  return (int)nb;
}

namespace {
bool gram_via_gemm(const float *X, int64_t rows, int k, float *G, float *partials, int max_blocks,
                   int *err, cudaStream_t s, cudaError_t *status);
}  // namespace

cudaError_t launch_gram(const float *X, int64_t rows, int k, int64_t ldx, float *G,
                        float *partials, int max_blocks, cudaStream_t s, int *err,
                        unsigned *ticket) {
  // wide ranks: the TMA-fed FP32 product kernel on X^T X (below)
  if (ldx == k && err) {
    cudaError_t st = cudaSuccess;
    if (gram_via_gemm(X, rows, k, G, partials, max_blocks, err, s, &st)) return st;
  }
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = 148;
  // k_gram8 needs >= 16 stages per block to repay its fixed costs: on the
  // sparse workload's 10^6 / 5 10^5 rows it takes the Grams from 0.320 to
  // 0.242 ms per iteration; on the dense one's 96,000 / 64,000 rows it was
  // slower (0.109 against 0.077 ms), so those keep k_gram_part
  if (ldx == k && k <= kG8MaxK && k >= 8 && (reinterpret_cast<uintptr_t>(X) & 15) == 0 &&
      rows >= 16LL * kG8Rows * sms) {
    // one block per SM (its chunk a whole number of stages, so every span
    // starts on a 16-byte boundary), partials reduced as for k_gram_part
    int64_t nb = (rows + kG8Rows - 1) / kG8Rows;
    const int64_t cap = min((int64_t)max_blocks, (int64_t)sms);
    if (nb > cap) nb = cap;
    const int64_t chunk = ((rows + nb - 1) / nb + kG8Rows - 1) / kG8Rows * kG8Rows;
    nb = (rows + chunk - 1) / chunk;
    auto kern = (k & 1) ? k_gram8<false> : k_gram8<true>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kG8Smem);
    kern<<<(unsigned)nb, kG8Threads, kG8Smem, s>>>(X, rows, k, chunk, partials);
    k_gram_reduce<<<(k * k + 31) / 32, gram_red_threads((int)nb), 0, s>>>(partials, (int)nb, k, G);
    g_launches += 2;
    return cudaGetLastError();
  }
  const int nb = gram_partial_blocks(rows, max_blocks);
  const int64_t chunk = (rows + nb - 1) / nb;
  const size_t smem = gram_smem_bytes<false>(k);
  if (smem > 48 * 1024)
    cudaFuncSetAttribute(k_gram_part<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
  // An entry a thread and at most three rounds of loads: the last block's sum takes
  // no longer than the reduction's launch.  Beyond, one SM reading the partials is
  // slower (2000 rows, both in a graph: 22.7 against 12.4 us at k = 32, 43 against 15
  // at k = 50).
  if (ticket && k <= 16 && nb <= 24) {
    k_gram_part<false, true><<<nb, kGramThreads, smem, s>>>(X, rows, k, ldx, chunk, partials, G,
                                                            ticket);
    g_launches += 1;
    return cudaGetLastError();
  }
  k_gram_part<false, false><<<nb, kGramThreads, smem, s>>>(X, rows, k, ldx, chunk, partials, nullptr,
                                                           nullptr);
  k_gram_reduce<<<(k * k + 31) / 32, gram_red_threads(nb), 0, s>>>(partials, nb, k, G);
  g_launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_gram_d(const float *X, int64_t rows, int k, int64_t ldx, double *G64,
                          float *G32, double *partials, int max_blocks, cudaStream_t s) {
  // 64 rows (one stage) per block while 128 would leave most SMs idle
  int nb = gram_partial_blocks(rows, max_blocks);
  if (nb <= max_blocks / 4) nb = (int)((rows + 63) / 64);
  const int64_t chunk = (rows + nb - 1) / nb;
  const size_t smem = gram_smem_bytes<true>(k);
  if (smem > 48 * 1024)
    cudaFuncSetAttribute(k_gram_part<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
  k_gram_part<true, false><<<nb, kGramThreads, smem, s>>>(X, rows, k, ldx, chunk, partials, nullptr,
                                                          nullptr);
  const bool chains8 = (int64_t)nb * k * k <= kChainValues;
  k_gram_reduce_d<<<(k * k + 31) / 32, chains8 ? 256 : gram_red_threads(nb), 0, s>>>(
      partials, nb, k, chains8, G64, G32);
  g_launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_widen(const float *G32, int k, double *G64, cudaStream_t s) {
  k_widen<<<(k * k + 255) / 256, 256, 0, s>>>(G32, k * k, G64);
  g_launches += 1;
  return cudaGetLastError();
}

// ------------------------------------------------------------------ SIMT GEMM
// C (M x N, ld ldc) = Aop (M x K) * B (K x N, ld ldb), FP32 FMA.
//   AK = true : Aop(mm, kk) = A[mm * lda + kk]   (A H^T: A is K-contiguous)
//   AK = false: Aop(mm, kk) = A[kk * lda + mm]   (W^T A as (A^T W): M-contiguous)
// 256 threads as 16 x 16; thread (ty, tx) owns rows ty*TM .. ty*TM+TM-1 and
// columns tx*TN .. tx*TN+TN-1 of the block tile.  (A layout of 8 threads
// along N with BN = 56 at k = 50, which wastes fewer FMAs on padding columns,
// measured 11 % slower even with its shared-memory reads free of bank
// conflicts: 20.4 against 18.3 ms per product at 96000 x 64000.)  The next K-slab is
// prefetched into registers while the current one is consumed from shared
// memory.  Accumulation is compensated: each 32-long K-slab is summed in a
// fresh FP32 register and added to the running sum with Kahan's correction,
// so the error does not grow with K (the residual expansion of Sec. 6.2
// subtracts nearly equal terms and needs the products close to FP32
// rounding).
namespace {
// two resident blocks per SM (at most 128 registers a thread): measured 8-12 %
// faster than one at 96000 x 64000, k = 50, despite a few spilled registers
#ifndef AUNMF_SIMT_MINB
#define AUNMF_SIMT_MINB 2
#endif
#ifndef AUNMF_SIMT_BM
#define AUNMF_SIMT_BM 128
#endif
template <int BM, int BN, int BK, bool AK>
__global__ void __launch_bounds__(256, AUNMF_SIMT_MINB)
    k_gemm_simt(const float *__restrict__ A, int64_t lda, int64_t M, int64_t K,
                const float *__restrict__ B, int ldb, int N, float *__restrict__ C, int ldc,
                int64_t kchunk, int vec) {
  // blockIdx.z: K split [kz0, kz1) (kchunk a multiple of the slab); its
  // partial C goes to C + z * M * ldc.  vec: A is 16-byte aligned with lda % 4
  // == 0, so its tile is read as float4 groups along A's contiguous axis.
  constexpr int TM = BM / 16, TN = BN / 16;
  constexpr int GA = BM * BK / 4 / 256;  // float4 groups of the A tile per thread
  constexpr int LA = BM * BK / 256, LB = BK * BN / 256;
  constexpr int PADA = 4;  // row pad: spreads the transposed stores over banks
  constexpr int SLAB = 128;  // K elements per compensated partial
  constexpr int LDK = TM * TN + 1;  // odd row stride of the per-thread running sums
  static_assert(GA >= 1 && GA * 4 == LA && LB >= 1 && TM % 4 == 0, "tile too small");
  static_assert(SLAB % BK == 0, "slab must be a multiple of BK");
  __shared__ __align__(16) float sA[2][BK][BM + PADA];
  __shared__ __align__(16) float sB[2][BK][BN];
  // Kahan running sum and correction of each thread's TM x TN outputs, in a
  // row of its own (touched once per slab): keeping them in registers would
  // triple the accumulator registers and halve the resident warps
  extern __shared__ float sKahan[];
  float *kh = sKahan + (size_t)threadIdx.x * LDK * 2, *kc = kh + LDK;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int64_t m0 = (int64_t)blockIdx.x * BM;
  const int n0 = blockIdx.y * BN;
  const int64_t kz0 = (int64_t)blockIdx.z * kchunk, kz1 = min(K, kz0 + kchunk);

  // Per-thread tile coordinates, pointers and edge predicates, fixed for the
  // whole K range (the loads of a full K step do no index arithmetic).
  //   AK:  group q is row am[q] of the tile, K offsets ak[q] .. ak[q] + 3
  //   !AK: group q is K offset ak[q], rows am[q] .. am[q] + 3
  // va: 1 all four elements inside A, 2 some (M edge, !AK), 0 none.
  int am[GA], ak[GA], va[GA];
  const float *pa[GA];
#pragma unroll
  for (int q = 0; q < GA; ++q) {
    const int f = tid + 256 * q;
    if (AK) {
      am[q] = f / (BK / 4);
      ak[q] = 4 * (f % (BK / 4));
      va[q] = m0 + am[q] < M ? 1 : 0;
      pa[q] = A + (va[q] ? (m0 + am[q]) : 0) * lda + kz0 + ak[q];
    } else {
      ak[q] = f / (BM / 4);
      am[q] = 4 * (f % (BM / 4));
      va[q] = m0 + am[q] + 3 < M ? 1 : (m0 + am[q] < M ? 2 : 0);
      pa[q] = A + (kz0 + ak[q]) * lda + (va[q] ? m0 + am[q] : 0);
    }
  }
  int bk[LB], bn[LB];
  bool vb[LB];
  const float *pb[LB];
#pragma unroll
  for (int q = 0; q < LB; ++q) {
    const int idx = tid + 256 * q;
    bn[q] = idx % BN;
    bk[q] = idx / BN;
    vb[q] = n0 + bn[q] < N;
    pb[q] = B + (kz0 + bk[q]) * ldb + (vb[q] ? n0 + bn[q] : 0);
  }

  float4 ra[GA];
  float rb[LB];
  // K step [k0, k0 + BK): a full step inside [kz0, kz1) with vec takes the
  // pointers as they stand; the last, partial step (and !vec) checks each
  // element's K index as well.
  auto load = [&](int64_t k0, bool full) {
#pragma unroll
    for (int q = 0; q < GA; ++q) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (full && vec && va[q] == 1) {
        v = __ldg(reinterpret_cast<const float4 *>(pa[q]));
      } else if (full && va[q] == 1) {  // unaligned rows: no index arithmetic either
        v = make_float4(__ldg(pa[q]), __ldg(pa[q] + 1), __ldg(pa[q] + 2), __ldg(pa[q] + 3));
      } else if (va[q]) {
        float e[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int64_t gm = m0 + am[q] + (AK ? 0 : u), gk = k0 + ak[q] + (AK ? u : 0);
          e[u] = (gm < M && gk < kz1) ? __ldg(&A[AK ? gm * lda + gk : gk * lda + gm]) : 0.f;
        }
        v = make_float4(e[0], e[1], e[2], e[3]);
      }
      ra[q] = v;
    }
#pragma unroll
    for (int q = 0; q < LB; ++q)
      rb[q] = (vb[q] && (full || k0 + bk[q] < kz1)) ? __ldg(pb[q]) : 0.f;
  };
  auto advance = [&]() {
#pragma unroll
    for (int q = 0; q < GA; ++q) pa[q] += AK ? (int64_t)BK : (int64_t)BK * lda;
#pragma unroll
    for (int q = 0; q < LB; ++q) pb[q] += (int64_t)BK * ldb;
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < GA; ++q) {
      if (AK) {
        sA[buf][ak[q] + 0][am[q]] = ra[q].x;
        sA[buf][ak[q] + 1][am[q]] = ra[q].y;
        sA[buf][ak[q] + 2][am[q]] = ra[q].z;
        sA[buf][ak[q] + 3][am[q]] = ra[q].w;
      } else {
        *reinterpret_cast<float4 *>(&sA[buf][ak[q]][am[q]]) = ra[q];
      }
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) sB[buf][bk[q]][bn[q]] = rb[q];
  };

  // packed pairs of rows for the two-wide FMA: output (i, j) is half i & 1 of
  // acc[i / 2][j].  Issue bounds this kernel; with the pairs and the unchecked
  // loads of unaligned rows A H^T at 32,001 x 24,001, k = 50, takes 2825 us (3157
  // before) and W^T A 2444 (2672), the same bits.
  using namespace aunmf::ptx;
  f32x2 acc[TM / 2][TN];
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0;
  for (int e = 0; e < TM * TN; ++e) kh[e] = kc[e] = 0.f;
  auto fold = [&]() {  // hi += acc with Kahan's compensation; acc = 0
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int e = i * TN + j;
        const float hi = kh[e], cor = kc[e];
        const float y = (i & 1 ? hi32(acc[i / 2][j]) : lo32(acc[i / 2][j])) - cor;
        const float t = hi + y;
        kc[e] = (t - hi) - y;
        kh[e] = t;
        if (i & 1) acc[i / 2][j] = 0;
      }
  };

  C += (int64_t)blockIdx.z * M * ldc;
  load(kz0, kz0 + BK <= kz1);
  advance();
  store(0);
  __syncthreads();
  int buf = 0, slab_left = SLAB / BK;
  for (int64_t k0 = kz0; k0 < kz1; k0 += BK) {
    const bool more = k0 + BK < kz1;
    if (more) {
      load(k0 + BK, k0 + 2 * BK <= kz1);
      advance();
    }
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      f32x2 a[TM / 2];
      float b[TN];
#pragma unroll
      for (int i = 0; i < TM / 2; i += 2) {
        const float4 v = *reinterpret_cast<const float4 *>(&sA[buf][kk][ty * TM + 2 * i]);
        a[i] = pack2(v.x, v.y);
        a[i + 1] = pack2(v.z, v.w);
      }
      if constexpr (TN == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(&sB[buf][kk][tx * TN]);
        b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
      } else if constexpr (TN == 2) {
        const float2 v = *reinterpret_cast<const float2 *>(&sB[buf][kk][tx * TN]);
        b[0] = v.x; b[1] = v.y;
      } else {
#pragma unroll
        for (int j = 0; j < TN; ++j) b[j] = sB[buf][kk][tx * TN + j];
      }
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const f32x2 bb = pack2(b[j], b[j]);
#pragma unroll
        for (int i = 0; i < TM / 2; ++i) acc[i][j] = fma2(a[i], bb, acc[i][j]);
      }
    }
    // fold once per slab of K (kz0 is a multiple of the slab) and at the end
    if (--slab_left == 0 || !more) {
      fold();
      slab_left = SLAB / BK;
    }
    if (more) {
      store(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t gm = m0 + ty * TM + i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int gn = n0 + tx * TN + j;
      if (gn < N) C[gm * ldc + gn] = kh[i * TN + j] - kc[i * TN + j];
    }
  }
}

// ---------------------------------------------------------------- TMA-fed form
// k_gemm_simt_tma: the same product and the same compensated summation as
// k_gemm_simt, when A's rows are 16-byte aligned; and, in its short form, for
// few output tiles whatever the alignment.  FP32 issue bounds it (k = 50,
// W^T A at 32,000 x 24,000: 48 TFLOP/s of useful FMAs against the 73 a loop
// of packed FMAs reaches).  A's tiles and the fixed factor's 16 x BN tiles
// arrive by TMA in a seven-stage shared-memory ring with mbarriers (full:
// one arrival + the copies' bytes; empty: all 256 threads).  The factor is
// read from a copy whose rows are padded to a multiple of 4 floats (TMA needs
// 16-byte row strides; N = 50 floats is not one), or in place where they are;
// staging its tiles with 4-byte asynchronous copies instead measured 3x
// slower than the whole product should take (11.5 ms for the copies alone at
// 96,000 x 64,000).  Eight warps compute, 8 x BN / 8 outputs per thread (256
// x BN per block, one block per SM), four 16-byte fragment loads per 32
// two-wide FMAs, with the running sums in registers (two warps per SM
// sub-partition may hold up to 255 registers each; a ninth, producer-only
// warp would cap them at 168).  Thread 0 also fills the ring: steps 0 .. 6
// first, then at the top of step s it waits until every thread has released
// the stage read at step s - 1 (warp 0 trails the others, so the wait is
// short) and issues the two copies of step s + 6 into it.
//   Thread (ty, tx), ty = 0..31, tx = 0..7 (a warp: 4 ty x 8 tx): columns
//   simt_col(tx, j); rows ty + 32 i (AK) or ty*4 + {0..3} and 128 + ty*4 +
//   {0..3} (!AK).
// AK (A K-contiguous): the tile is 256 rows of 16 K (64 bytes), copied with
// the 64-byte swizzle (16-byte chunk c of row r lands at chunk
// c ^ ((r >> 1) & 3)), so the four rows a warp reads at once (ty .. ty+3)
// sit in four different bank groups.  !AK: 16 K-rows of 256 (one kilobyte):
// a warp's four row fragments are consecutive.  Either way a warp's loads of
// the factor tile read consecutive words, with no bank conflict.
// Slab sums are folded every 128 K into the running sums with Kahan's
// corrections, which sit in shared memory (one row per thread).  Every wait
// is bounded; on expiry the kernel raises *err, writes nothing and returns
// (thread 0 first waits, bounded, for the copies it has in flight).  The K
// steps of a split are whole (its length is a multiple of 128); rows and
// columns past either matrix are zero-filled by the copies.
constexpr int kTBK = 16, kTStages = 7;
constexpr int kTThreads = 256;
constexpr int kTSlabSteps = 8;  // K steps per compensated slab (128 K, as k_gemm_simt)
// Shape of one form: RT rows and BN / 8 columns per thread, a tile of 32 RT
// rows by BN columns.
template <int RT, int BN>
struct SimtTile {
  static constexpr int BM = 32 * RT, TN = BN / 8, NE = RT * TN;
  static constexpr int kLdc = NE + 4;  // floats per thread row of corrections (+ pad: no bank conflict)
  static constexpr size_t kA = (size_t)BM * kTBK * 4, kB = (size_t)kTBK * BN * 4;
  // after the corrections: the slab sums of the cluster form (slabs tiles)
  static constexpr size_t smem(int slabs) {
    return 1024 + kTStages * (kA + kB) + (slabs ? 0 : (size_t)kTThreads * kLdc * 4) +
           (size_t)slabs * BM * BN * 4 + 2 * kTStages * 8 + 16;
  }
};

// The runs of slabs of a launch of `blocks` blocks (at most one per slab):
// slab u of the product is slab u % nsl of tile u / nsl, and block b has slabs
// first(b) .. first(b + 1) - 1.  A split into whole tiles and whole K splits
// left part of the last wave idle (125 row tiles on 152 SMs: 18 %).
struct SimtRuns {
  int64_t nsl, per, rem;  // slabs per tile; slabs per block, one more in the first rem
  __host__ __device__ int64_t first(int64_t b) const { return b * per + (b < rem ? b : rem); }
  __host__ __device__ int64_t owner(int64_t u) const {
    return u < rem * (per + 1) ? u / (per + 1) : rem + (u - rem * (per + 1)) / per;
  }
};
__host__ __device__ inline SimtRuns simt_runs(int64_t M, int64_t K, int gy, int64_t blocks) {
  const int64_t nsl = (K + kTBK * kTSlabSteps - 1) / (kTBK * kTSlabSteps);
  const int64_t u = (M + 255) / 256 * gy * nsl;
  return {nsl, u / blocks, u % blocks};
}

// Column j (0 .. TN - 1) of thread column tx within the tile.
template <int TN>
__device__ __forceinline__ int simt_col(int tx, int j) {
  if constexpr (TN >= 4)  // 32 columns by fours, then 32 by fours, 16 by twos, 8 by ones
    return j < 4 ? tx * 4 + j : TN == 8 ? 32 + tx * 4 + j - 4 : j < 6 ? 32 + tx * 2 + j - 4 : 48 + tx;
  else
    return tx * TN + j;
}

template <bool AK, int RT, int BN, bool VEC, bool RUNS>
__global__ void __launch_bounds__(kTThreads, 1)
    k_gemm_simt_tma(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                    const float *__restrict__ A, int64_t lda, const float *__restrict__ B,
                    int64_t M, int64_t K, int N, float *__restrict__ C,
                    int ldc, int64_t kchunk, int clus, int group, float *__restrict__ parts,
                    int *err, long long limit, int inject) {
  // The short form (RT = 4, few tiles) stages the factor's tile with 4-byte
  // asynchronous copies straight from B (K x N, contiguous): it spares the
  // launch that pads B's rows to 16 bytes for TMA (mapB is not used).  VEC
  // false (short form only): A's rows are not 16-byte aligned, and its tile is
  // copied the same way into the same places (mapA is not used).
  static_assert((VEC || RT == 4) && !(RUNS && RT == 4), "unaligned rows: short form");
  // clus > 0: the grid's clus K splits of a tile form one cluster (1, 1, clus):
  // every block keeps its slab sums in shared memory, and the cluster folds all
  // of them, in K order, through distributed shared memory: with Kahan's
  // compensation within each `group` slabs, the groups' sums added plainly --
  // the additions of an unclustered pass over K split every `group` slabs, so
  // both give the same bits.  clus == 0: split z writes its partial at C + z M ldc.
  // RUNS (parts given): the grid is one block per SM and the tiles' slabs, tile
  // after tile, are cut into equal runs, one per block (SimtRuns).  A block
  // writes a tile it has all of to C, another one's part to its first (the
  // run's first tile) or second (its last) slot of parts, for k_simt_join.
  // parts and group > 0: every slab's sums go to parts, slab after slab, for
  // k_simt_fold, which adds them as a cluster does.  (A form of its own: the
  // runs' bookkeeping in the slab loop cost a grid of whole tiles 2-4 %: five HALS
  // iterations at 24,000 x 16,000, k = 50, 10,860 -> 10,480 us without it.)
  // inject (test hook): thread 0 never arrives on the first stage's barrier,
  // so every thread's bounded wait runs out
  using namespace aunmf::ptx;
  using T = SimtTile<RT, BN>;
  constexpr int BM = T::BM, TN = T::TN, NE = T::NE;
  constexpr bool BCP = RT == 4;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((1024 - (su32(smem_raw) & 1023)) & 1023);
  float *sA = reinterpret_cast<float *>(smem);
  float *sB = reinterpret_cast<float *>(smem + kTStages * T::kA);
  float *corr = reinterpret_cast<float *>(smem + kTStages * (T::kA + T::kB));
  const int nslab = clus > 0 ? (int)(kchunk / (kTBK * kTSlabSteps)) : 0;
  uint64_t *full =
      reinterpret_cast<uint64_t *>(corr + (clus > 0 ? nslab * BM * BN : kTThreads * T::kLdc));
  uint64_t *empty = full + kTStages;
  int *flag = reinterpret_cast<int *>(empty + kTStages);  // 1: this block finished its K range
  const int tid = threadIdx.x;
  const int64_t m0 = (int64_t)blockIdx.x * BM;
  const int n0 = blockIdx.y * BN;
  const int64_t kz0 = (int64_t)blockIdx.z * kchunk, kz1 = min(K, kz0 + kchunk);
  int nsteps = kz1 > kz0 ? (int)((kz1 - kz0 + kTBK - 1) / kTBK) : 0;
  // RUNS: the tile (row tile * gy + column tile) and the K step within it that
  // the copies and the sums have reached; a tile ends after nst steps
  const int nst = (int)((K + kTBK - 1) / kTBK);
  const int gy = (N + BN - 1) / BN;
  int64_t tile0 = 0;
  int step0 = 0;
  int64_t u0 = 0;
  if (RUNS) {
    const SimtRuns r = simt_runs(M, K, gy, gridDim.x);
    const int64_t u1 = r.first(blockIdx.x + 1);
    u0 = r.first(blockIdx.x);
    tile0 = u0 / r.nsl;
    step0 = (int)(u0 % r.nsl) * kTSlabSteps;
    nsteps = (int)((u1 / r.nsl - tile0) * nst + u1 % r.nsl * kTSlabSteps - step0);
  }
  const bool producer = tid < 32;
  if (tid == 0) {
    for (int st = 0; st < kTStages; ++st) {
      mbar_init(&full[st], BCP ? 1 + kTThreads : 1);
      mbar_init(&empty[st], kTThreads);
    }
    *flag = 1;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // thread 0: fill stage st with step s
  const uint64_t pol_a = policy_evict_first(), pol_b = policy_evict_last();  // A streams once
  int issued = 0;
  int64_t ft = tile0;
  int fk = step0;
  auto fill = [&](int s) {
    const int st = s % kTStages;
    int k0 = (int)(kz0 + (int64_t)s * kTBK);
    int64_t fm = m0;
    int fn = n0;
    if constexpr (RUNS) {
      k0 = fk * kTBK;
      fm = ft / gy * BM;
      fn = (int)(ft % gy) * BN;
      if (++fk == nst) {
        fk = 0;
        ++ft;
      }
    }
    const uint32_t bytes = (uint32_t)(!VEC ? 0 : BCP ? T::kA : T::kA + T::kB);
    if (!VEC) {
      if (!(inject && s == 0)) mbar_arrive(&full[st]);
      return;
    }
    if (inject && s == 0)
      mbar_expect_tx_only(&full[st], bytes);
    else
      mbar_expect_tx(&full[st], bytes);
    // x coordinates (k0 for AK and the factor, m0 otherwise) are multiples
    // of 16 floats; the checked build tests it and skips bad copies
    if (!AUNMF_BOUND(k0 >= 0 && (k0 & 3) == 0 && (fm & 3) == 0 && (fn & 3) == 0,
                     AUNMF_CHECK_TMA_COORD))
      return;
    if (AK)
      tma_load_2d(sA + (size_t)st * BM * kTBK, &mapA, &full[st], k0, (int)fm, pol_a);
    else
      tma_load_2d(sA + (size_t)st * BM * kTBK, &mapA, &full[st], (int)fm, k0, pol_a);
    if (!BCP) tma_load_2d(sB + (size_t)st * kTBK * BN, &mapB, &full[st], fn, k0, pol_b);
    ++issued;
  };
  auto fill_b = [&](int s) {  // every thread's share of the factor's tile
    const int st = s % kTStages;
    const int64_t k0 = kz0 + (int64_t)s * kTBK;
#pragma unroll
    for (int q = 0; q < kTBK * BN / kTThreads; ++q) {
      const int e = tid + q * kTThreads, kk = e / BN, nn = e % BN;
      const bool in = k0 + kk < kz1 && n0 + nn < N;
      cp_async4(sB + (size_t)st * kTBK * BN + e, in ? B + (k0 + kk) * N + n0 + nn : B, in);
    }
    if constexpr (!VEC) {
#pragma unroll
      for (int q = 0; q < kTBK * BM / kTThreads; ++q) {
        const int e = tid + q * kTThreads;
        const int kk = AK ? e % kTBK : e / BM, mm = AK ? e / kTBK : e % BM;
        const bool in = k0 + kk < kz1 && m0 + mm < M;
        const float *src = AK ? A + (m0 + mm) * lda + k0 + kk : A + (k0 + kk) * lda + m0 + mm;
        float *dst = sA + (size_t)st * BM * kTBK +
                     (AK ? mm * kTBK + (((kk >> 2) ^ ((mm >> 1) & 3)) << 2) + (kk & 3) : e);
        cp_async4(dst, in ? src : A, in);
      }
    }
    cp_async_arrive(&full[st]);
  };
  // every stage starts empty: steps 0 .. kTStages - 1
  for (int s = 0; s < kTStages && s < nsteps; ++s) {
    if (tid == 0) fill(s);
    if (BCP) fill_b(s);
  }

  const int w = tid >> 5, l = tid & 31, tx = l & 7, ty = w * 4 + (l >> 3);
  float *kc = corr + (size_t)tid * T::kLdc;  // Kahan corrections of the sums
  if (clus == 0) {
#pragma unroll
    for (int e = 0; e < NE; e += 4) *reinterpret_cast<float4 *>(kc + e) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // slab sums as packed pairs for the two-wide FMA (the same FMAs in half the
  // issue slots): output (i, j) is half i & 1 of acc[i / 2][j] (!AK: a pair of
  // rows arrives as one aligned 8-byte half of a fragment) or half j & 1 of
  // acc[i][j / 2] (AK: TN is even)
  f32x2 acc[NE / 2];
  float hi[NE];
#pragma unroll
  for (int e = 0; e < NE / 2; ++e) acc[e] = 0;
#pragma unroll
  for (int e = 0; e < NE; ++e) hi[e] = 0.f;
  auto fold = [&]() {  // hi += acc with Kahan's compensation; acc = 0
#pragma unroll
    for (int e4 = 0; e4 < NE; e4 += 4) {
      float4 cv = *reinterpret_cast<const float4 *>(kc + e4);
      float *c = &cv.x;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e4 + u, i = e / TN, j = e % TN;
        const f32x2 pr = AK ? acc[i * (TN / 2) + j / 2] : acc[(i / 2) * TN + j];
        const float a = (AK ? (j & 1) : (i & 1)) ? hi32(pr) : lo32(pr);
        const float y = a - c[u];
        const float t = hi[e] + y;
        c[u] = (t - hi[e]) - y;
        hi[e] = t;
      }
      *reinterpret_cast<float4 *>(kc + e4) = cv;
    }
#pragma unroll
    for (int e = 0; e < NE / 2; ++e) acc[e] = 0;
  };
  // row i (0 .. RT - 1) of the thread within the tile
  auto row_of = [&](int i) { return AK ? ty + 32 * i : (i < 4 ? ty * 4 + i : 128 + ty * 4 + i - 4); };
  auto keep_at = [&](float *p) {  // the slab's sums into a tile at p; acc = 0
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      const int i = e / TN, j = e % TN;
      const f32x2 pr = AK ? acc[i * (TN / 2) + j / 2] : acc[(i / 2) * TN + j];
      p[row_of(i) * BN + simt_col<TN>(tx, j)] =
          (AK ? (j & 1) : (i & 1)) ? hi32(pr) : lo32(pr);
    }
#pragma unroll
    for (int e = 0; e < NE / 2; ++e) acc[e] = 0;
  };
  auto keep = [&](int sl) { keep_at(corr + sl * BM * BN); };
  // the thread's TN columns (simt_col) of factor row br
  auto load_b = [&](const float *br, float (&b)[TN]) {
    if constexpr (TN == 2) {
      const float2 v = *reinterpret_cast<const float2 *>(br + tx * 2);
      b[0] = v.x;
      b[1] = v.y;
    } else {
#pragma unroll
      for (int q = 0; q < TN / 4; ++q) {
        const float4 v = *reinterpret_cast<const float4 *>(br + 32 * q + tx * 4);
        b[4 * q] = v.x;
        b[4 * q + 1] = v.y;
        b[4 * q + 2] = v.z;
        b[4 * q + 3] = v.w;
      }
      if constexpr (TN == 6 || TN == 7) {
        const float2 v = *reinterpret_cast<const float2 *>(br + 32 + tx * 2);
        b[4] = v.x;
        b[5] = v.y;
      }
      if constexpr (TN == 7) b[6] = br[48 + tx];
    }
  };
  // AK: rows ty + 32 i share their swizzle (r >> 1) & 3 (32 i leaves those bits alone)
  const int sw = (ty >> 1) & 3;

  bool ok = true;
  int slab = 0, kept = 0, ck = step0;
  bool from0 = step0 == 0;  // the sums began with the tile's first K step
  int64_t ct = tile0;
  for (int s = 0; s < nsteps; ++s) {
    const int st = s % kTStages;
    if (BCP && s >= 1 && s - 1 + kTStages < nsteps) {
      // refill the stage read at step s - 1: every thread waits and copies
      const int sp = s - 1;
      if (!mbar_wait(&empty[sp % kTStages], (uint32_t)(sp / kTStages) & 1u, err, limit)) {
        ok = false;
        break;
      }
      if (tid == 0) fill(sp + kTStages);
      fill_b(sp + kTStages);
    }
    if (!BCP && producer && s >= 1 && s - 1 + kTStages < nsteps) {
      // refill the stage read at step s - 1 (use (s - 1) / kTStages of it)
      const int sp = s - 1;
      int okp = 1;
      if (tid == 0)
        okp = mbar_wait(&empty[sp % kTStages], (uint32_t)(sp / kTStages) & 1u, err, limit) ? 1 : 0;
      if (!__shfl_sync(0xffffffffu, okp, 0)) {
        ok = false;
        break;
      }
      if (tid == 0) fill(sp + kTStages);
    }
    if (!mbar_wait(&full[st], (uint32_t)(s / kTStages) & 1u, err, limit)) {
      ok = false;
      break;
    }
    const float *a = sA + (size_t)st * BM * kTBK;
    const float *b = sB + (size_t)st * kTBK * BN;
    if constexpr (AK) {  // a: [BM rows][16 K], 64-byte swizzle
#pragma unroll
      for (int kq = 0; kq < kTBK / 4; ++kq) {
        float4 av[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i)
          av[i] = *reinterpret_cast<const float4 *>(a + (ty + 32 * i) * kTBK + ((kq ^ sw) << 2));
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float bf[TN];
          load_b(b + (kq * 4 + u) * BN, bf);
          f32x2 bp[TN / 2];
#pragma unroll
          for (int j = 0; j < TN / 2; ++j) bp[j] = pack2(bf[2 * j], bf[2 * j + 1]);
#pragma unroll
          for (int i = 0; i < RT; ++i) {
            const float x = (&av[i].x)[u];
            const f32x2 xx = pack2(x, x);
#pragma unroll
            for (int j = 0; j < TN / 2; ++j)
              acc[i * (TN / 2) + j] = fma2(xx, bp[j], acc[i * (TN / 2) + j]);
          }
        }
      }
    } else {  // a: [16 K][BM rows]
#pragma unroll
      for (int kk = 0; kk < kTBK; ++kk) {
        f32x2 ap[RT / 2];
#pragma unroll
        for (int q = 0; q < RT / 4; ++q) {
          const float4 v = *reinterpret_cast<const float4 *>(a + kk * BM + 128 * q + ty * 4);
          ap[2 * q] = pack2(v.x, v.y);
          ap[2 * q + 1] = pack2(v.z, v.w);
        }
        float bf[TN];
        load_b(b + kk * BN, bf);
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const f32x2 bb = pack2(bf[j], bf[j]);
#pragma unroll
          for (int i = 0; i < RT / 2; ++i) acc[i * TN + j] = fma2(ap[i], bb, acc[i * TN + j]);
        }
      }
    }
    // (cp.async, which fills unaligned rows' stages, is of the same proxy as the loads)
    if constexpr (VEC) fence_async();
    mbar_arrive(&empty[st]);
    const bool last = s + 1 == nsteps || (RUNS && ck + 1 == nst);
    if (++slab == kTSlabSteps || last) {
      if (clus > 0) {
        keep(s / kTSlabSteps);
      } else if (RUNS && group > 0) {
        keep_at(parts + (u0 + kept++) * BM * BN);
      } else {
        fold();
      }
      slab = 0;
    }
    if constexpr (RUNS) {
      ++ck;
      if (last && group > 0) {
        ck = 0;
      } else if (last) {
        const int64_t tm = ct / gy * BM;
        const int tn = (int)(ct % gy) * BN;
        float *slot = parts + (2 * (int64_t)blockIdx.x + (ct != tile0)) * 2 * BM * BN;
        const bool whole = from0 && ck == nst;
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const int64_t gm = tm + row_of(i);
#pragma unroll
          for (int j = 0; j < TN; ++j) {
            const int e = i * TN + j, c = simt_col<TN>(tx, j);
            const float v = hi[e] - kc[e];
            if (!whole) {
              slot[row_of(i) * BN + c] = v;
              slot[(BM + row_of(i)) * BN + c] = (hi[e] - v) - kc[e];  // what v rounded off
            } else if (gm < M && tn + c < N) {
              C[gm * ldc + tn + c] = v;
            }
            hi[e] = 0.f;
          }
        }
#pragma unroll
        for (int e = 0; e < NE; e += 4) *reinterpret_cast<float4 *>(kc + e) = make_float4(0.f, 0.f, 0.f, 0.f);
        ck = 0;
        from0 = true;
        ++ct;
      }
    }
  }
  if (BCP) cp_async_wait_all();
  if (tid == 0) {
    // the copies thread 0 has put in flight land before the block exits
    for (int st = 0; st < kTStages && st < issued; ++st) {
      const int cnt = (issued - st + kTStages - 1) / kTStages;
      mbar_wait_drain(&full[st], (uint32_t)(cnt - 1) & 1u, limit);
    }
  }
  if (clus > 0) {
    // every block of the cluster takes part in both cluster barriers, also
    // after a wait ran out; the tile is written only if all of them finished
    if (!ok) *flag = 0;
    cluster_sync();
    bool all = true;
    for (int z = 0; z < clus; ++z) all = all && ld_cluster_u32(su32(flag), z) == 1u;
    if (all) {
      const int per = (BM + clus - 1) / clus;
      const int ra = (int)blockIdx.z * per, rb = min(BM, ra + per);
      const int total = (int)((K + kTBK * kTSlabSteps - 1) / (kTBK * kTSlabSteps));
      for (int e = ra * BN + tid; e < rb * BN; e += kTThreads) {
        const int64_t gm = m0 + e / BN;
        const int gn = n0 + e % BN;
        if (gm >= M || gn >= N) continue;
        float out = 0.f, h = 0.f, c = 0.f;
        int in_group = 0;
        for (int g0 = 0; g0 < total; g0 += 8) {  // eight remote loads in flight
          float v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int g = g0 + u < total ? g0 + u : total - 1, z = g / nslab;
            v[u] = __uint_as_float(ld_cluster_u32(su32(corr + (g - z * nslab) * BM * BN + e), z));
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            if (g0 + u >= total) break;
            const float y = v[u] - c, t = h + y;
            c = (t - h) - y;
            h = t;
            if (++in_group == group || g0 + u + 1 == total) {
              out = group < total ? out + (h - c) : h - c;
              h = c = 0.f;
              in_group = 0;
            }
          }
        }
        C[gm * ldc + gn] = out;
      }
    }
    cluster_sync();  // no block's shared memory goes away while a peer reads it
    return;
  }
  if (!ok || RUNS) return;
  C += (int64_t)blockIdx.z * M * ldc;
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int64_t gm = m0 + row_of(i);
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int gn = n0 + simt_col<TN>(tx, j);
      if (gn < N) C[gm * ldc + gn] = hi[i * TN + j] - kc[i * TN + j];
    }
  }
}

// Tensor map of the factor's tiles for k_gemm_simt_tma: bn columns x 16 K rows over
// the factor or its padded copy (K x N, ld ldp), no swizzle, zero fill past N and K.
bool simt_factor_map(CUtensorMap *map, const float *Bp, int64_t K, int N, int ldp, int bn) {
  ptx::EncodeTiledFn fn = ptx::encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)N, (cuuint64_t)K};
  cuuint64_t strides[1] = {(cuuint64_t)ldp * 4};
  cuuint32_t box[2] = {(cuuint32_t)bn, (cuuint32_t)kTBK};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(Bp), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor map of A's tiles: AK, a box of 16 K x bm rows over A (M x K, ld lda),
// 64-byte swizzle; !AK, bm rows x 16 K over A stored K x M, no swizzle.  FP32, zero
// fill outside the matrix.
bool simt_map(CUtensorMap *map, const float *A, int64_t lda, int64_t M, int64_t K, bool AK,
              int bm) {
  ptx::EncodeTiledFn fn = ptx::encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)(AK ? K : M), (cuuint64_t)(AK ? M : K)};
  cuuint64_t strides[1] = {(cuuint64_t)(lda * 4)};
  cuuint32_t box[2] = {(cuuint32_t)(AK ? kTBK : bm), (cuuint32_t)(AK ? bm : kTBK)};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(A), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            AK ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BM, int BN>
constexpr size_t simt_kahan_bytes() {
  return sizeof(float) * 256 * 2 * ((BM / 16) * (BN / 16) + 1);
}

int simt_sms() {
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 148;
}

// K splits: the smallest S in 1..4 whose block count fills the resident
// slots most evenly, each split at least 8 slabs long.
int simt_wave_splits(int64_t tiles, int64_t K, int64_t slots) {
  int best = 1;
  double best_eff = 0.0;
  for (int S = 1; S <= 4; ++S) {
    if (S > 1 && K / S < 8 * 128) break;
    const int64_t u = tiles * S;
    const double eff = ((double)u / slots) / (double)((u + slots - 1) / slots);
    if (eff > best_eff + 0.02) { best_eff = eff; best = S; }
  }
  return best;
}

__global__ void k_sum_parts(const float *__restrict__ parts, int S, int64_t len,
                            float *__restrict__ C) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < len;
       e += (int64_t)gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int z = 0; z < S; ++z) s += parts[z * len + e];
    C[e] = s;
  }
}

// The tiles that runs of k_gemm_simt_tma cut: block x takes the tile that the
// boundary of runs x and x + 1 cuts, unless an earlier boundary cuts it too,
// and adds its parts (a sum and what it rounded off) in K order, with the
// additions' errors carried along.
template <int BN>
__global__ void k_simt_join(const float *__restrict__ parts, int64_t M, int64_t K, int N,
                            float *__restrict__ C, int ldc) {
  constexpr int BM = 256;
  const int gy = (N + BN - 1) / BN;
  const SimtRuns r = simt_runs(M, K, gy, gridDim.x + 1);
  const int64_t cut = r.first(blockIdx.x + 1), t = cut / r.nsl;
  const int64_t b0 = r.owner(t * r.nsl), b1 = r.owner((t + 1) * r.nsl - 1);
  if (cut == t * r.nsl || b0 != blockIdx.x) return;
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < BM * BN; e += gridDim.y * blockDim.x) {
    const int64_t gm = t / gy * BM + e / BN;
    const int gn = (int)(t % gy) * BN + e % BN;
    if (gm >= M || gn >= N) continue;
    // tile t is the last of run b0 (its first slot if also the first) and the
    // first of the others
    const float *p = parts + (2 * b0 + (r.first(b0) / r.nsl != t)) * 2 * BM * BN + e;
    float s = p[0], c = p[BM * BN];
#pragma unroll 4
    for (int64_t b = b0 + 1; b <= b1; ++b) {
      const float *q = parts + 4 * b * BM * BN + e;
      const float v = q[0], u = __fadd_rn(s, v), d = __fsub_rn(u, s);
      c += __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(u, d)), __fsub_rn(v, d)), q[BM * BN]);
      s = u;
    }
    C[gm * ldc + gn] = s + c;
  }
}

// The slab sums that k_gemm_simt_tma left for every tile, folded in K order:
// Kahan's compensation within each `group` slabs (a thread each, at most four),
// the groups' sums added plainly.
template <int BN>
__global__ void k_simt_fold(const float *__restrict__ parts, int64_t M, int64_t K, int N, int group,
                            float *__restrict__ C, int ldc) {
  constexpr int BM = 256;
  __shared__ float part[4][64];
  const int gy = (N + BN - 1) / BN;
  const int64_t nsl = simt_runs(M, K, gy, 1).nsl;
  const int64_t x = (int64_t)blockIdx.x * 64 + threadIdx.x, t = x / (BM * BN);
  const int e = (int)(x % (BM * BN));
  const int64_t gm = t / gy * BM + e / BN, a = (int64_t)threadIdx.y * group;
  const int gn = (int)(t % gy) * BN + e % BN;
  const bool in = gm < M && gn < N;
  const int64_t len = in ? min((int64_t)group, nsl - a) : 0;
  const float *p = parts + (t * nsl + a) * BM * BN + e;
  float h = 0.f, c = 0.f;
  for (int64_t g0 = 0; g0 < len; g0 += 16) {  // sixteen loads in flight
    float v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = p[min(g0 + u, len - 1) * BM * BN];
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      if (g0 + u >= len) break;
      const float y = v[u] - c, w = h + y;
      c = (w - h) - y;
      h = w;
    }
  }
  part[threadIdx.y][threadIdx.x] = h - c;
  __syncthreads();
  if (!in || threadIdx.y) return;
  float out = h - c;
  for (int z = 1; z < (int)blockDim.y; ++z) out += part[z][threadIdx.x];
  C[gm * ldc + gn] = out;
}

// One launch of a k_gemm_simt_tma form: grid (gx, gy, S), a cluster per tile
// when group > 0, S blocks with equal runs when parts is given (see the
// kernel), and then the launch that joins the cut tiles or folds the slabs.
template <bool AK, int RT, int BN, bool VEC>
cudaError_t launch_simt_tma(const CUtensorMap &mapA, const CUtensorMap &mapB, const float *A,
                            int64_t lda, const float *B, int64_t M, int64_t K, int N, float *C, int ldc, int64_t kchunk, int S,
                            int group, float *parts, int *err, cudaStream_t s) {
  using T = SimtTile<RT, BN>;
  auto kern = k_gemm_simt_tma<AK, RT, BN, VEC, false>;
  if constexpr (RT == 8)
    if (parts) kern = k_gemm_simt_tma<AK, RT, BN, VEC, true>;
  const bool clus = group > 0 && !parts;
  const size_t smem = T::smem(clus ? (int)(kchunk / (kTBK * kTSlabSteps)) : 0);
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaLaunchConfig_t cfg{};
  const unsigned gx = (unsigned)((M + T::BM - 1) / T::BM), gy = (unsigned)((N + BN - 1) / BN);
  cfg.gridDim = parts ? dim3((unsigned)S) : dim3(gx, gy, (unsigned)S);
  cfg.blockDim = dim3(kTThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = (unsigned)S;
  cfg.attrs = at;
  cfg.numAttrs = clus ? 1 : 0;
  g_launches += 1;
  const cudaError_t e =
      cudaLaunchKernelEx(&cfg, kern, mapA, mapB, A, lda, B, M, K, N, C, ldc, kchunk, clus ? S : 0, group, parts, err,
                         fault::wait_cycles(), fault::site() == AUNMF_INJECT_SIMT_WAIT ? 1 : 0);
  if (e != cudaSuccess || !parts) return e;
  if (group > 0) {
    const int64_t nsl = simt_runs(M, K, gy, 1).nsl;
    k_simt_fold<BN><<<gx * gy * (T::BM * BN / 64), dim3(64, (unsigned)((nsl + group - 1) / group)), 0, s>>>(
        parts, M, K, N, group, C, ldc);
  } else {
    if ((int64_t)gx * gy % S == 0) return e;  // no tile is cut
    k_simt_join<BN><<<dim3((unsigned)S - 1, 16), 256, 0, s>>>(parts, M, K, N, C, ldc);
  }
  g_launches += 1;
  return cudaGetLastError();
}

template <bool AK, int RT, bool VEC>
cudaError_t launch_simt_tma_n(int BN, const CUtensorMap &mapA, const CUtensorMap &mapB,
                              const float *A, int64_t lda, const float *B, int64_t M, int64_t K,
                              int N, float *C, int64_t kchunk, int S, int group, float *parts,
                              int *err, cudaStream_t s) {
  if (BN == 16)
    return launch_simt_tma<AK, RT, 16, VEC>(mapA, mapB, A, lda, B, M, K, N, C, N, kchunk, S, group, parts, err, s);
  if (BN == 32)
    return launch_simt_tma<AK, RT, 32, VEC>(mapA, mapB, A, lda, B, M, K, N, C, N, kchunk, S, group, parts, err, s);
  if constexpr (RT == 8) {
    if (BN == 48)
      return launch_simt_tma<AK, RT, 48, VEC>(mapA, mapB, A, lda, B, M, K, N, C, N, kchunk, S, group, parts, err, s);
    if constexpr (!AK)
      if (BN == 56)
        return launch_simt_tma<AK, RT, 56, VEC>(mapA, mapB, A, lda, B, M, K, N, C, N, kchunk, S, group, parts, err, s);
  }
  return launch_simt_tma<AK, RT, 64, VEC>(mapA, mapB, A, lda, B, M, K, N, C, N, kchunk, S, group, parts, err, s);
}

cudaError_t sum_parts(const float *parts, int S, int64_t len, float *C, cudaStream_t s) {
  int64_t nb = (len + 255) / 256;
  if (nb > 152 * 16) nb = 152 * 16;
  k_sum_parts<<<(unsigned)nb, 256, 0, s>>>(parts, S, len, C);
  g_launches += 1;
  return cudaGetLastError();
}

// The form of a product C (M x N) over K and what it takes from its workspace.
struct SimtPlan {
  enum Form {
    kGeneric,  // k_gemm_simt: the whole K splits S0
    kCluster,  // few output tiles: 128-row tiles, K cut over a cluster of S blocks
    kRuns,     // equal runs of slabs, joined
    kSlabs,    // equal runs whose slab sums are kept and folded as S0 splits would be
    kSplits    // 256-row tiles, the whole K splits S0
  } form;
  int BN, gy, S0;
  int64_t S, kchunk;
  int64_t parts;  // floats before the factor's copy: partial sums or slab sums
};

// aligned: A's rows start on 16-byte boundaries; even: as for launch_aht_simt.
SimtPlan simt_plan(int64_t M, int64_t K, int N, bool aligned, bool even) {
  constexpr int BM = AUNMF_SIMT_BM, SLAB = 128;
  SimtPlan p{};
  p.BN = N <= 16 ? 16 : (N <= 32 ? 32 : 64);
  p.gy = (N + p.BN - 1) / p.BN;
  const int64_t sms = simt_sms(), tiles = (M + 255) / 256 * p.gy, nsl = (K + SLAB - 1) / SLAB;
  // K splits: of 256-row tiles on the SMs where N > 32, else of BM-row tiles,
  // two to an SM.  Each form sums the same splits, so a call's bits do not
  // depend on which one it takes; `even` alone cuts K elsewhere.
  p.S0 = aligned && N > 32 ? simt_wave_splits(tiles, K, sms)
                           : simt_wave_splits((M + BM - 1) / BM * p.gy, K, 2 * sms);
  p.S = p.S0;
  p.kchunk = ((K + p.S0 - 1) / p.S0 + SLAB - 1) / SLAB * SLAB;
  p.parts = 4 * M * N;
  p.form = SimtPlan::kGeneric;
  // TMA-fed forms: coordinates within int32
  if (M >= (1LL << 31) || K >= (1LL << 31)) return p;
  const int64_t tiles4 = (M + 127) / 128 * p.gy;
  if (tiles4 * 2 <= sms) {
    // few output tiles (one block per tile walked all of K, at 77-87 us for 2000 x
    // 1500, k = 10, on 12-16 of the SMs; the cluster takes 13-15).  The line on K: a
    // block's slab sums fit beside its ring in shared memory.
    int64_t S = std::min<int64_t>(sms / tiles4, 8);
    const int64_t kchunk = ((K + S - 1) / S + SLAB - 1) / SLAB * SLAB;
    if (kchunk / SLAB * 128 * p.BN * 4 <= 128 * 1024) {
      p.form = SimtPlan::kCluster;
      p.S = (K + kchunk - 1) / kchunk;
      p.kchunk = kchunk;
      return p;
    }
  }
  if (!aligned) return p;
  // Equal runs of slabs, one block per SM, for single products and losses
  // (whole tiles left up to half of the last wave idle: W^T A 32,000 x 24,000,
  // k = 50, 1659 -> 1594 us; A H^T at k = 64 2263 -> 1898; loss and gradients
  // 20,000 x 10,000, k = 100, 2753 -> 2377).  Whole K splits (S0) in a
  // factorisation: its sweeps amplify the sums' last bits (1e-5 in a trace-form
  // residual after eight sweeps).  Where those splits leave a quarter of the SMs
  // without a block, and the slab sums take at most a quarter gigabyte, equal runs
  // whose slab sums are folded as the splits would be (8 HALS iterations, 15,000 x
  // 1200, k = 20: 3100 -> 1543 us; at 12,000 x 8000, k = 64, 128 blocks, the kept
  // slabs cost 4 %).
  p.form = even                                                        ? SimtPlan::kRuns
           : tiles * 4 <= sms && tiles * p.S0 * 4 <= sms * 3 &&
                     tiles * nsl * 256 * p.BN <= (1LL << 26) ? SimtPlan::kSlabs
                                                             : SimtPlan::kSplits;
  if (p.form == SimtPlan::kSplits) return p;
  p.S = std::min<int64_t>(sms, tiles * nsl);
  p.kchunk = ((K + p.S - 1) / p.S + SLAB - 1) / SLAB * SLAB;
  // (at most the sum and the remainder of two tiles a block, or every slab's sum)
  p.parts = std::max<int64_t>(p.parts, (even ? 4 * p.S : tiles * nsl) * 256 * p.BN);
  return p;
}

template <bool AK>
cudaError_t gemm_simt(const float *A, int64_t lda, int64_t M, int64_t K, const float *B, int N,
                      float *C, float *parts, bool even, int *err, cudaStream_t s) {
  constexpr int BM = AUNMF_SIMT_BM, BK = 16, SLAB = 128;
  const int vec = simt_aligned(A, lda);
  const SimtPlan p = simt_plan(M, K, N, vec, even);
  const int BN = p.BN, S0 = parts ? p.S0 : 1;
  const unsigned gy = (unsigned)p.gy;
  const bool tma = err && parts;
  const int group = (int)(((K + S0 - 1) / S0 + SLAB - 1) / SLAB);  // slabs per K split
  CUtensorMap mapA, mapB;
  if (tma && p.form == SimtPlan::kCluster) {
    if (vec && simt_map(&mapA, A, lda, M, K, AK, 128))
      return launch_simt_tma_n<AK, 4, true>(BN, mapA, mapA, A, lda, B, M, K, N, C, p.kchunk, (int)p.S,
                                            group, nullptr, err, s);
    memset(&mapA, 0, sizeof(mapA));
    return launch_simt_tma_n<AK, 4, false>(BN, mapA, mapA, A, lda, B, M, K, N, C, p.kchunk, (int)p.S,
                                           group, nullptr, err, s);
  }
  if (tma && p.form != SimtPlan::kGeneric && simt_map(&mapA, A, lda, M, K, AK, 256)) {
    const int ldp = (N + 3) & ~3;
    const bool direct = ldp == N && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
    const bool runs = p.form == SimtPlan::kRuns || p.form == SimtPlan::kSlabs;
    // Column tiles of 48 or 56 where these take no more of them: padding columns
    // cost FMAs like any other.  W^T A at k = 50 (56 for 64), 32,000 x 24,000:
    // 1775 -> 1657 us.  AK keeps 64 for 56: its row fragments hold four K of one
    // row, so the odd column would be packed from two rows with moves (A H^T and
    // W^T A at k = 100, 20,000 x 10,000, both with 56: 2983 us, so 2753).
    const int bn = BN < 64                           ? BN
                   : (N + 47) / 48 == (int)gy        ? 48
                   : !AK && (N + 55) / 56 == (int)gy ? 56
                                                     : 64;
    // (parts holds the parts, then the factor's padded copy)
    float *Bp = parts + ((p.parts + 63) & ~63LL);
    const float *Bs = direct ? B : Bp;
    if (simt_factor_map(&mapB, Bs, K, N, ldp, bn)) {
      cudaError_t e = direct ? cudaSuccess : launch_copy2d(B, N, Bp, ldp, K, N, s);
      if (e == cudaSuccess)
        e = launch_simt_tma_n<AK, 8, true>(bn, mapA, mapB, A, lda, B, M, K, N,
                                           !runs && p.S > 1 ? parts : C, p.kchunk, (int)p.S,
                                           p.form == SimtPlan::kSlabs ? group : 0,
                                           runs ? parts : nullptr, err, s);
      if (e != cudaSuccess || runs || p.S == 1) return e;
      return sum_parts(parts, (int)p.S, M * (int64_t)N, C, s);
    }
  }
  const unsigned gx = (unsigned)((M + BM - 1) / BM);
  const int S = S0;
  const int64_t kchunk = ((K + S - 1) / S + SLAB - 1) / SLAB * SLAB;
  float *out = S > 1 ? parts : C;
  const dim3 grid(gx, gy, (unsigned)S);
  auto go = [&](auto kern, size_t sm) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    kern<<<grid, 256, sm, s>>>(A, lda, M, K, B, N, N, out, N, kchunk, vec);
  };
  switch (BN) {
    case 16: go(k_gemm_simt<BM, 16, BK, AK>, simt_kahan_bytes<BM, 16>()); break;
    case 32: go(k_gemm_simt<BM, 32, BK, AK>, simt_kahan_bytes<BM, 32>()); break;
    default: go(k_gemm_simt<BM, 64, BK, AK>, simt_kahan_bytes<BM, 64>()); break;
  }
  g_launches += 1;
  if (S > 1) return sum_parts(parts, S, M * (int64_t)N, C, s);
  return cudaGetLastError();
}
// G = X^T X for X (rows x k, contiguous rows, k >= 96 and a multiple of 4,
// 16-byte aligned) with the TMA-fed FP32 product kernel: C (k x k) = Aop
// (k x rows) B (rows x k) with Aop(i, r) = X[r][i] (A stored K x M) and B =
// X.  The whole square is formed (twice the flops of the upper triangle), in
// Kahan-compensated slabs like every product, over S K splits chosen to fill
// the SMs, whose partials (S x k x k in `partials`) are added in FP64 in
// split order.  At k = 512 on 96,000 / 64,000 rows this replaces k_gram_part,
// whose 4 x 4 tiles need 8,256 tiles per row and so re-stage every row 33
// times.  Returns false (nothing launched) when the shape does not qualify.
bool gram_via_gemm(const float *X, int64_t rows, int k, float *G, float *partials, int max_blocks,
                   int *err, cudaStream_t s, cudaError_t *status) {
  if (k < 96 || (k & 3) || (reinterpret_cast<uintptr_t>(X) & 15) || rows < 1024 ||
      rows >= (1LL << 31))
    return false;
  CUtensorMap mapA, mapB;
  using T = SimtTile<8, 64>;
  if (!simt_map(&mapA, X, k, k, rows, false, T::BM) || !simt_factor_map(&mapB, X, rows, k, k, 64))
    return false;
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = 148;
  const unsigned gx = (unsigned)((k + T::BM - 1) / T::BM), gy = (unsigned)((k + 63) / 64);
  int64_t S = (sms + (int64_t)gx * gy - 1) / ((int64_t)gx * gy);
  S = min(S, (int64_t)max_blocks);
  S = min(S, rows / 512);
  if (S < 1) S = 1;
  const int64_t kchunk = ((rows + S - 1) / S + 127) / 128 * 128;
  S = (rows + kchunk - 1) / kchunk;
  *status = launch_simt_tma<false, 8, 64, true>(mapA, mapB, X, k, X, k, rows, k, partials, k, kchunk, (int)S, 0, nullptr, err, s);
  if (*status != cudaSuccess) return true;
  k_gram_reduce<<<(k * k + 31) / 32, gram_red_threads((int)S), 0, s>>>(partials, (int)S, k, G);
  g_launches += 1;
  *status = cudaGetLastError();
  return true;
}
}  // namespace

cudaError_t launch_aht_simt(const float *A, int64_t m, int64_t n, int64_t lda, const float *Ht,
                            int k, float *P, float *parts, bool even, int *err, cudaStream_t s) {
  return gemm_simt<true>(A, lda, m, n, Ht, k, P, parts, even, err, s);
}

cudaError_t launch_wta_simt(const float *A, int64_t m, int64_t n, int64_t lda, const float *W,
                            int k, float *P, float *parts, bool even, int *err, cudaStream_t s) {
  return gemm_simt<false>(A, lda, n, m, W, k, P, parts, even, err, s);
}

bool simt_aligned(const float *A, int64_t lda) {
  return reinterpret_cast<uintptr_t>(A) % 16 == 0 && lda % 4 == 0;
}

size_t simt_parts_bytes(int64_t m, int64_t n, int k, bool aligned, bool even) {
  const int64_t parts =
      std::max(simt_plan(m, n, k, aligned, even).parts, simt_plan(n, m, k, aligned, even).parts);
  return sizeof(float) * (size_t)(((parts + 63) & ~63LL) + std::max(m, n) * ((k + 3) & ~3));
}

// ------------------------------------------------------------------ transpose
namespace {
__global__ void k_transpose(const float *__restrict__ in, int64_t rows, int64_t cols,
                            float *__restrict__ out) {
  __shared__ float t[32][33];
  transpose_tiles(in, rows, cols, out, blockIdx.x, gridDim.x, t, threadIdx.x, threadIdx.y,
                  blockDim.y);
}

__global__ void k_copy2d(const float *__restrict__ in, int64_t ld_in, float *__restrict__ out,
                         int64_t ld_out, int64_t rows, int64_t cols) {
  const int64_t total = rows * cols;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / cols, c = e % cols;
    out[r * ld_out + c] = in[r * ld_in + c];
  }
}
}  // namespace

cudaError_t launch_transpose(const float *in, int64_t rows, int64_t cols, float *out,
                             cudaStream_t s) {
  if (rows == 0 || cols == 0) return cudaSuccess;
  int64_t tiles = ((rows + 31) / 32) * ((cols + 31) / 32);
  if (tiles > 152 * 64) tiles = 152 * 64;
  k_transpose<<<(unsigned)tiles, dim3(32, 8), 0, s>>>(in, rows, cols, out);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_copy2d(const float *in, int64_t ld_in, float *out, int64_t ld_out,
                          int64_t rows, int64_t cols, cudaStream_t s) {
  if (rows * cols == 0) return cudaSuccess;
  int64_t nb = (rows * cols + 255) / 256;
  if (nb > 152 * 32) nb = 152 * 32;
  k_copy2d<<<(unsigned)nb, 256, 0, s>>>(in, ld_in, out, ld_out, rows, cols);
  g_launches += 1;
  return cudaGetLastError();
}

// ------------------------------------------------------------------ reductions
namespace {
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide FP64 sum in a fixed tree order; result valid in thread 0.
__device__ double block_sum_d(double v) {
  __shared__ double sw[32];
  v = warp_sum_d(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sw[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    r = (lane < (int)(blockDim.x >> 5)) ? sw[lane] : 0.0;
    r = warp_sum_d(r);
  }
  return r;
}

// Two such sums at once (256 threads).
__device__ void block_sum_d2(double &a, double &b) {
  __shared__ double sw[2][8];
  a = warp_sum_d(a);
  b = warp_sum_d(b);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) {
    sw[0][w] = a;
    sw[1][w] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = b = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      a += sw[0][i];
      b += sw[1][i];
    }
  }
}

// out[0] = ||A||^2 (m x n, lda) from per-block FP64 partials, out[1] = 0 for
// products that read A itself; the last block adds the partials.  Rows without
// padding are one vector of m n entries.  Each thread squares 16 entries at a
// time (four 16-byte loads in flight) in FP32 and adds the 16-term sums in
// FP64 (an FP64 add per entry would bound the pass).  EXACT (sparse A, far fewer
// entries): every square in FP64, which no finite entry overflows or loses; in FP32
// pairs an entry above 1.8e19 makes the sum a NaN and one below 1e-23 nothing.
// Bound by HBM at large sizes (a block per row with one FP32 chain per thread left
// 4.6 TB/s), EXACT by the FP64 rate (5e7 entries: 162 us more than the pairs).
template <bool EXACT>
__global__ void __launch_bounds__(256)
    k_norm2(const float *__restrict__ A, int64_t m, int64_t n, int64_t lda,
            double *__restrict__ partials, double *__restrict__ out, unsigned *ticket) {
  double s = 0.0;
  const bool flat = lda == n || m == 1;
  const int64_t rows = flat ? 1 : m, len = flat ? m * n : n;
  // units of 1024 float4 groups (4096 entries) of a row, block-strided
  const int64_t per_row = (len + 4095) / 4096, units = rows * per_row;
  for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
    const int64_t r = flat ? 0 : u / per_row, c0 = (flat ? u : u % per_row) * 4096;
    const float *p = A + r * lda + c0;
    const int64_t left = len - c0;
    float v[16];
    if ((reinterpret_cast<uintptr_t>(p) & 15) == 0 && left >= 4096) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 x = __ldcs(reinterpret_cast<const float4 *>(p) + threadIdx.x + 256 * q);
        v[4 * q] = x.x;
        v[4 * q + 1] = x.y;
        v[4 * q + 2] = x.z;
        v[4 * q + 3] = x.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int c = threadIdx.x + 256 * q;
        v[q] = c < left ? p[c] : 0.f;
      }
    }
    if constexpr (EXACT) {
      double d[4] = {};
#pragma unroll
      for (int q = 0; q < 16; ++q) d[q & 3] = fma((double)v[q], (double)v[q], d[q & 3]);
      s += (d[0] + d[1]) + (d[2] + d[3]);
    } else {
      float a = 0.f, b = 0.f;
#pragma unroll
      for (int q = 0; q < 16; q += 2) {
        a = fmaf(v[q], v[q], a);
        b = fmaf(v[q + 1], v[q + 1], b);
      }
      s += (double)(a + b);
    }
  }
  s = block_sum_d(s);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
  if (!last_block(ticket)) return;
  double t = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) t += __ldcg(&partials[b]);
  t = block_sum_d(t);
  if (threadIdx.x == 0) {
    out[0] = t;
    out[1] = 0.0;
  }
}

// relres = sqrt(max(0, ||A||^2 + d - 2 <P, Ht> + <GW, GH>) / ||A||^2), FP64
// (Sec. 5, relative error; trace form).  When P was formed from a rounded
// copy A~ of A (TF32 / BF16 products), <P, Ht> = <A~, W H> and
//   ||A - WH||^2 = ||A||^2 - 2 <A~, WH> + ||WH||^2 + 2 <A~ - A, WH>;
// the last term is taken as d = n2a[1] = 2 <A~ - A, A> (WH ~ A), which is
// off by 2 <A~ - A, A - WH>, a sum of rounding errors that do not correlate
// with the fit residual.  Without d, the mean of the rounding errors (not
// zero on real value distributions: -8e-6 relative for BF16 on uniform
// low-rank data) would bias the reported residual by ~1e-3 at relres ~1e-2.
// One launch forms both inner products, <P, Ht> over len entries and <GW, GH>
// over k^2, as per-block FP64 partials, and its last block adds them in block
// order and writes the result (a separate one-block kernel took 8-61 us, most
// of it the k^2 FP64 products on one SM).  <P, Ht>: with 16-byte aligned
// arrays, four products at a time are formed and summed in FP32
// (round-to-nearest: unbiased, ~1e-7 relative per group, averaging out over
// the groups) and the group joins an FP64 sum; an FP64 FMA per element bound
// the pass by the FP64 rate.
// LOSS: *loss = 0.5 (||A||^2 + d - 2 <P, Ht> + <GW, GH>), not clamped.
template <bool LOSS>
__global__ void __launch_bounds__(256)
    k_residual(const float *__restrict__ P, const float *__restrict__ Q, int64_t len,
               const float *__restrict__ GW, const float *__restrict__ GH, int kk,
               const double *__restrict__ n2a, double *__restrict__ partials, unsigned *ticket,
               double *__restrict__ relres, DevCounters *ctr, double *__restrict__ last) {
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nt = (int64_t)gridDim.x * blockDim.x;
  double s = 0.0, q = 0.0;
  int64_t tail = 0;
  if (((reinterpret_cast<uintptr_t>(P) | reinterpret_cast<uintptr_t>(Q)) & 15) == 0) {
    const float4 *P4 = reinterpret_cast<const float4 *>(P), *Q4 = reinterpret_cast<const float4 *>(Q);
    const int64_t n4 = len >> 2;
#pragma unroll 4
    for (int64_t g = t0; g < n4; g += nt) {
      const float4 x = P4[g], y = Q4[g];
      s += (double)fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, x.x * y.x)));
    }
    tail = n4 << 2;
  }
  for (int64_t e = tail + t0; e < len; e += nt) s = fma((double)P[e], (double)Q[e], s);
  for (int64_t e = t0; e < kk; e += nt) q = fma((double)GW[e], (double)GH[e], q);
  block_sum_d2(s, q);
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x] = s;
    partials[2 * blockIdx.x + 1] = q;
  }
  if (!last_block(ticket)) return;
  double cross = 0.0, quad = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
    cross += __ldcg(&partials[2 * b]);
    quad += __ldcg(&partials[2 * b + 1]);
  }
  block_sum_d2(cross, quad);
  if (threadIdx.x != 0) return;
  const double a2 = n2a[0];
  const double f = (a2 + n2a[1]) - 2.0 * cross + quad;
  if constexpr (LOSS) {
    *last = 0.5 * f;
  } else {
    const double r2 = f < 0.0 ? 0.0 : f;
    // (a NaN in ||A||^2 has to reach nonfinite: 0 only for A = 0)
    const double rr = a2 == 0.0 ? 0.0 : sqrt(r2 / a2);
    if (!isfinite(rr)) ctr->nonfinite += 1;
    if (relres) relres[ctr->iter] = rr;
    ctr->iter += 1;
    if (last) *last = rr;
  }
}

// Blocks of a residual pass: one per 4096 entries, at most nparts.
int residual_blocks(int64_t len, int nparts) {
  const int64_t nb = (len + 4095) / 4096;
  return (int)(nb < 1 ? 1 : (nb > nparts ? nparts : nb));
}
}  // namespace

cudaError_t launch_loss(const float *P, const float *Ht, int64_t len, const float *GW,
                        const float *GH, int k, const double *n2a, double *partials, int nparts,
                        double *loss, unsigned *ticket, cudaStream_t s) {
  k_residual<true><<<residual_blocks(len, nparts), 256, 0, s>>>(P, Ht, len, GW, GH, k * k, n2a,
                                                               partials, ticket, nullptr, nullptr,
                                                               loss);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_norm2(const float *A, int64_t m, int64_t n, int64_t lda, double *partials,
                         int nparts, double *out, unsigned *ticket, cudaStream_t s) {
  k_norm2<false><<<residual_blocks(m * n, nparts), 256, 0, s>>>(A, m, n, lda, partials, out, ticket);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_norm2_vec(const float *v, int64_t len, double *partials, int nparts,
                             double *out, unsigned *ticket, cudaStream_t s) {
  k_norm2<true><<<residual_blocks(len, nparts), 256, 0, s>>>(v, 1, len, len, partials, out, ticket);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_relres(const float *P, const float *Ht, int64_t len, const float *GW,
                          const float *GH, int k, const double *n2a, double *partials,
                          int nparts, double *relres_dev, DevCounters *ctr, double *last,
                          unsigned *ticket, cudaStream_t s) {
  k_residual<false><<<residual_blocks(len, nparts), 256, 0, s>>>(P, Ht, len, GW, GH, k * k, n2a,
                                                                partials, ticket, relres_dev, ctr,
                                                                last);
  g_launches += 1;
  return cudaGetLastError();
}

}  // namespace aunmf
