// k_wide.cu -- local updates (LUC) and gradient rows for ranks above 64.
//
// Every one of them needs X G (rows x k times k x k, 2 k^2 flops a row): MU and
// the gradient with the old X, the HALS sweep with the entries before a
// coordinate already updated.  Both are run as products blocked over 16
// coordinates, whose operands are reused from shared memory by 8 x 4 register
// tiles; a warp per row, which walks all of G for every one or two rows, was
// bound by reading G and by a shuffle reduction per coordinate (HALS at k = 256,
// 12,001 rows: 327 us; the gradient at k = 100, 20,000 rows: 58 us).
#include <math.h>

#include "internal.cuh"
#include "ptx.cuh"

namespace aunmf {
namespace {

using namespace aunmf::ptx;

constexpr int kWThreads = 256, kNB = 16;  // coordinates per block
// 16-byte group of rows r4 = r / 4 of column j of the X tile: permuted within
// aligned eights so that a warp's eight row groups of one j (r4 = 0, 2, ..) and a
// warp storing one r of 8 consecutive j fall into different banks.
__device__ __forceinline__ int perm4(int r4, int j) { return r4 ^ ((r4 >> 3) & 1) ^ (j & 7); }

// acc[a][c] += rows (4 r4 + 2 a, + 1) of column j times g[c] (four coordinates):
// pairs of rows arrive packed.
template <int R>
__device__ __forceinline__ void tile_fma(const float *sX, int j, int r4, const float *g,
                                         f32x2 (&acc)[4][4]) {
  const float *col = sX + (size_t)j * R;
  const ulonglong2 xa = *reinterpret_cast<const ulonglong2 *>(col + 4 * perm4(r4, j));
  const ulonglong2 xb = *reinterpret_cast<const ulonglong2 *>(col + 4 * perm4(r4 + 1, j));
  const float4 gv = *reinterpret_cast<const float4 *>(g);
  const f32x2 x[4] = {xa.x, xa.y, xb.x, xb.y};
  const float gc[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const f32x2 gg = pack2(gc[c], gc[c]);
#pragma unroll
    for (int a = 0; a < 4; ++a) acc[a][c] = fma2(x[a], gg, acc[a][c]);
  }
}
// the thread's 8 x 4 sums into e[c][R] (perm4 of column 0)
template <int R>
__device__ __forceinline__ void tile_out(float *e, int r4, const f32x2 (&acc)[4][4]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    *reinterpret_cast<ulonglong2 *>(e + c * R + 4 * perm4(r4, 0)) =
        make_ulonglong2(acc[0][c], acc[1][c]);
    *reinterpret_cast<ulonglong2 *>(e + c * R + 4 * perm4(r4 + 1, 0)) =
        make_ulonglong2(acc[2][c], acc[3][c]);
  }
}

// ---------------------------------------------------------------- MU, gradient
// MU: X <- X P / (X G + eps), every entry from the old X; gradient: out = g (X G -
// P).  A block of 256 threads holds R = 512 / JS rows of X (64, 128 or 256) in
// shared memory as [k][R] and goes through the columns 16 at a time: warp w takes
// rows 64 (w / JS) .. + 63 and the j-th of JS shares of the sum over the k
// entries, a thread 8 rows x 4 columns (packed FMAs); then every thread adds the
// shares of R / 16 entries pairwise and finishes them.  P's entries of a block are
// loaded into registers before its sums, and the next block's columns of G are
// copied in meanwhile.  Bound by FMA issue and shared-memory reads.
template <int JS>
struct WideTile {
  static constexpr int R = 512 / JS;
  static constexpr size_t smem(int k) {
    return sizeof(float) * ((size_t)k * R + 2 * (size_t)k * kNB + (size_t)JS * kNB * R);
  }
};

template <int JS, bool MU>
__global__ void __launch_bounds__(kWThreads, 1)
    k_wide_xg(float *__restrict__ X, const float *__restrict__ P, const float *__restrict__ G,
              int64_t rows, int k, float eps, const float *__restrict__ gscale,
              float *__restrict__ out, int vec) {
  constexpr int R = WideTile<JS>::R, NP = R / 16;
  extern __shared__ __align__(16) float sm[];
  float *sX = sm;                                // [k][R], perm4 within a column
  float *sG = sX + (size_t)k * R;                // [2][k][16]
  float *sE = sG + 2 * (size_t)k * kNB;          // [JS][16][R]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int js = w % JS, rb = w / JS, rg = lane & 7, cg = lane >> 3;
  const int nblk = (k + kNB - 1) / kNB;
  const int jper = (k + JS - 1) / JS;
  const float gs = !MU && gscale ? *gscale : 1.f;

  // columns [16 b, 16 b + 16) of G into buffer `buf`
  auto stage_g = [&](int b, int buf) {
    const int i0 = b * kNB;
    float *dst = sG + (size_t)buf * k * kNB;
    if (vec) {
      for (int e = tid; e < k * 4; e += kWThreads) {
        const int j = e >> 2, c = i0 + 4 * (e & 3);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(su32(dst + 4 * e)),
                     "l"(c < k ? G + (size_t)j * k + c : G), "r"(c < k ? 16 : 0)
                     : "memory");
      }
    } else {
      for (int e = tid; e < k * kNB; e += kWThreads) {
        const int j = e >> 4, c = i0 + (e & 15);
        cp_async4(dst + e, c < k ? G + (size_t)j * k + c : G, c < k);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  const int64_t tiles = (rows + R - 1) / R;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t r0 = tile * R;
    const int nr = (int)min((int64_t)R, rows - r0);
    __syncthreads();  // the previous tile is done with every buffer
    for (int r = w; r < R; r += 8)  // a warp per row, lanes along k
      for (int j = lane; j < k; j += 32)
        cp_async4(sX + (size_t)j * R + 4 * perm4(r >> 2, j) + (r & 3),
                  r < nr ? X + (r0 + r) * k + j : X, r < nr);
    stage_g(0, 0);
    for (int b = 0; b < nblk; ++b) {
      const int buf = b & 1, i0 = b * kNB;
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();  // G's block and X are there; the other buffer has been read
      if (b + 1 < nblk) stage_g(b + 1, buf ^ 1);
      float p[NP];
#pragma unroll
      for (int u = 0; u < NP; ++u) {
        const int r = (tid >> 4) + 16 * u, c = tid & 15;
        p[u] = r < nr && i0 + c < k ? __ldg(P + (r0 + r) * k + i0 + c) : 0.f;
      }
      f32x2 acc[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[q][c] = 0;
      const float *g = sG + (size_t)buf * k * kNB + 4 * cg;
      const int j0 = js * jper, j1 = min(k, j0 + jper);
#pragma unroll 4
      for (int j = j0; j < j1; ++j) tile_fma<R>(sX, j, 16 * rb + 2 * rg, g + j * kNB, acc);
      tile_out<R>(sE + (size_t)(js * kNB + 4 * cg) * R, 16 * rb + 2 * rg, acc);
      __syncthreads();
      // 16 lanes along a row's 16 columns
#pragma unroll
      for (int u = 0; u < NP; ++u) {
        const int r = (tid >> 4) + 16 * u, c = tid & 15;
        if (r >= nr || i0 + c >= k) continue;
        float v[JS];
#pragma unroll
        for (int s = 0; s < JS; ++s)
          v[s] = sE[(size_t)(s * kNB + c) * R + 4 * perm4(r >> 2, 0) + (r & 3)];
#pragma unroll
        for (int h = JS / 2; h > 0; h >>= 1)
#pragma unroll
          for (int s = 0; s < h; ++s) v[s] += v[s + h];
        if constexpr (MU) {
          const float x = sX[(size_t)(i0 + c) * R + 4 * perm4(r >> 2, i0 + c) + (r & 3)];
          X[(r0 + r) * k + i0 + c] = x * p[u] / (v[0] + eps);
        } else {
          out[(r0 + r) * k + i0 + c] = gs * (v[0] - p[u]);
        }
      }
    }
  }
}

// ---------------------------------------------------------------- HALS
// The sweep x_i <- max(0, x_i + (p_i - (x G)_i) / G_ii), i ascending, for k % 4
// == 0 and 16-byte aligned rows.  A block holds 64 rows of X as [k][64] and takes
// the coordinates 16 at a time.  (x G)_i is summed as 32 chains and a binary tree:
// chain l over the entries j = 128 t + 4 l + u (t, then u ascending), the chains
// added pairwise over l ^ 16, 8, 4, 2, 1 -- the order of a warp that holds a row
// in 32 lanes, whose results are kept to the bit (FP32 sweeps of wide ranks
// amplify a last bit to 1e-2 within a few iterations).  A block of 16 coordinates
// changes the entries of 4 of the 32 chains only (4 consecutive l, one in each
// class l % 4 = q).  So
//   1. eight warps form the tree's sums over the other 28 chains, for all 64 x 16
//      (row, coordinate) pairs: for class q, with m the index of the changed chain
//      among its eight (l = q + 4 m), s1 = c(m ^ 4), s2 = c(m ^ 2) + c(m ^ 6), s3 =
//      (c(m ^ 1) + c(m ^ 5)) + (c(m ^ 3) + c(m ^ 7)); a thread 8 rows x 4 coordinates;
//   2. four threads per row sweep the 16 coordinates: thread q holds its changed
//      chain's entries, forms T_q = ((chain + s1) + s2) + s3, two shuffles give (x
//      G)_i = (T_0 + T_2) + (T_1 + T_3), and the thread whose chain holds x_i
//      updates it.  Meanwhile the next block's rows of G are copied in.
// Bound by latency, step 2's dependent chain and step 1's loads at two warps a
// scheduler (k = 256, 7,999 rows, one tile an SM: 870 clocks a coordinate, 28 %
// issue).  HALS at k = 256, 7,999 rows: 115 us, 12,001 rows: 193 us (two rounds of
// tiles on 152 SMs); a warp per two rows 321 and 327 us.
constexpr int kHR = 64;
constexpr int kHQ = 3 * kNB * kHR + 8;  // floats of one class in sS (+ 8: classes in other banks)

template <int KT4>
constexpr size_t hals_smem(int k) {
  return sizeof(float) * ((size_t)k * kHR + (size_t)k * kNB + 4 * (size_t)kHQ +
                          2 * (size_t)kNB * KT4 * 16);
}

template <int KT4, bool UNIT>
__global__ void __launch_bounds__(kWThreads, 1)
    k_wide_hals(float *__restrict__ X, const float *__restrict__ P, const float *__restrict__ G,
                int64_t rows, int k) {
  extern __shared__ __align__(16) float sm[];
  float *sX = sm;                        // [k][64], perm4 within a column
  float *sG = sX + (size_t)k * kHR;      // [k][16]: G(j, i0 + c)
  float *sS = sG + (size_t)k * kNB;      // [4 q](kHQ)[3][16][64]
  float *sC = sS + 4 * kHQ;              // [2][16][KT4][16]: G(i0 + c, 128 t + 16 m + e)
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int q = w & 3, part = w >> 2, rg = lane & 7, cg = lane >> 3;
  const int nblk = (k + kNB - 1) / kNB;

  // (G is symmetric: its columns of the block stand for its rows)
  auto copy16 = [](float *dst, const float *src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(su32(dst)), "l"(src),
                 "r"(in ? 16 : 0)
                 : "memory");
  };
  auto stage_g = [&](int b) {
    const int i0 = b * kNB, m = (i0 & 127) >> 4;
    for (int e = tid; e < k * 4; e += kWThreads) {
      const int j = e >> 2, c = i0 + 4 * (e & 3);
      copy16(sG + 4 * e, c < k ? G + (size_t)j * k + c : G, c < k);
    }
    float *d = sC + (b & 1) * kNB * KT4 * 16;
    for (int e = tid; e < kNB * KT4 * 4; e += kWThreads) {
      const int c = e / (KT4 * 4), j = 128 * ((e >> 2) % KT4) + 16 * m + 4 * (e & 3);
      const bool in = i0 + c < k && j < k;
      copy16(d + 4 * e, in ? G + (size_t)(i0 + c) * k + j : G, in);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  const int64_t tiles = (rows + kHR - 1) / kHR;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t r0 = tile * kHR;
    const int nr = (int)min((int64_t)kHR, rows - r0);
    __syncthreads();
    for (int r = w; r < kHR; r += 8)
      for (int j = lane; j < k; j += 32)
        cp_async4(sX + (size_t)j * kHR + 4 * perm4(r >> 2, j) + (r & 3),
                  r < nr ? X + (r0 + r) * k + j : X, r < nr);
    stage_g(0);
    for (int b = 0; b < nblk; ++b) {
      const int i0 = b * kNB, m = (i0 & 127) >> 4, tb = i0 >> 7;
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      // this thread's P (step 2: row tid / 4, class tid % 4), in flight during step 1
      const int r2 = tid >> 2, q2 = tid & 3;
      const float4 p4 = r2 < nr && i0 + 4 * q2 < k
                            ? __ldg(reinterpret_cast<const float4 *>(P + (r0 + r2) * k + i0) + q2)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
      // ---- 1
      {
        auto chain = [&](int x, f32x2 (&acc)[4][4]) {  // chain l = q + 4 (m ^ x)
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][c] = 0;
          const int l4 = 4 * (q + 4 * (m ^ x));
#pragma unroll
          for (int t = 0; t < KT4; ++t) {
            if (128 * t + l4 >= k) break;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int j = 128 * t + l4 + u;
              tile_fma<kHR>(sX, j, 2 * rg, sG + j * kNB + 4 * cg, acc);
            }
          }
        };
        auto add = [](f32x2 (&a)[4][4], const f32x2 (&c)[4][4]) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) a[i][e] = add2(a[i][e], c[i][e]);
        };
        auto put = [&](int s, const f32x2 (&a)[4][4]) {
          tile_out<kHR>(sS + q * kHQ + (s * kNB + 4 * cg) * kHR, 2 * rg, a);
        };
        f32x2 a[4][4], c[4][4];
        if (part == 0) {
          chain(4, a);
          put(0, a);
          chain(2, a);
          chain(6, c);
          add(a, c);
          put(1, a);
        } else {
          f32x2 d[4][4];
          chain(1, a);
          chain(5, c);
          add(a, c);
          chain(3, c);
          chain(7, d);
          add(c, d);
          add(a, c);
          put(2, a);
        }
      }
      __syncthreads();
      if (b + 1 < nblk) stage_g(b + 1);  // G's rows of this block have been read
      // ---- 2
      {
        const float *gc = sC + (b & 1) * kNB * KT4 * 16;
        const int rp = 4 * perm4(r2 >> 2, 0) + (r2 & 3);
        // the changed chain of this class: x[t][u] = x_{128 t + 16 m + 4 q + u}; the
        // block's own entries x[tb] are updated one by one
        float x[KT4][4];
#pragma unroll
        for (int t = 0; t < KT4; ++t)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = 128 * t + 16 * m + 4 * q2 + u;
            x[t][u] = j < k ? sX[(size_t)j * kHR + 4 * perm4(r2 >> 2, j) + (r2 & 3)] : 0.f;
          }
        const float pp[4] = {p4.x, p4.y, p4.z, p4.w};
        const float *ss = sS + q2 * kHQ + rp;
#pragma unroll
        for (int i = 0; i < kNB; ++i) {
          if (i0 + i >= k) break;
          const float4 *gi = reinterpret_cast<const float4 *>(gc + i * KT4 * 16) + q2;
          float v = 0.f;
#pragma unroll
          for (int t = 0; t < KT4; ++t) {
            const float4 g = gi[4 * t];
            v = fmaf(x[t][0], g.x, v);
            v = fmaf(x[t][1], g.y, v);
            v = fmaf(x[t][2], g.z, v);
            v = fmaf(x[t][3], g.w, v);
          }
          v += ss[i * kHR];
          v += ss[(kNB + i) * kHR];
          v += ss[(2 * kNB + i) * kHR];
          v += __shfl_xor_sync(0xffffffffu, v, 2);
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          const float gii = gc[(i * KT4 + tb) * 16 + i];
          if (q2 == (i >> 2) && (UNIT || gii > 0.f)) {
            // UNIT: Eq. halsupdate as printed, no division by G_ii
            float xi = x[0][i & 3];
#pragma unroll
            for (int t = 1; t < KT4; ++t) xi = t == tb ? x[t][i & 3] : xi;
            const float c = pp[i & 3] - v, z = xi + (UNIT ? c : c / gii);
            xi = z > 0.f ? z : 0.f;
#pragma unroll
            for (int t = 0; t < KT4; ++t) x[t][i & 3] = t == tb ? xi : x[t][i & 3];
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = i0 + 4 * q2 + u;
          float xi = x[0][u];
#pragma unroll
          for (int t = 1; t < KT4; ++t) xi = t == tb ? x[t][u] : xi;
          if (j < k) sX[(size_t)j * kHR + 4 * perm4(r2 >> 2, j) + (r2 & 3)] = xi;
        }
      }
    }
    __syncthreads();
    for (int r = w; r < nr; r += 8)
      for (int j = lane; j < k; j += 32)
        X[(r0 + r) * k + j] = sX[(size_t)j * kHR + 4 * perm4(r >> 2, j) + (r & 3)];
  }
}

int wide_sms() {
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 152;
}

template <int JS, bool MU>
cudaError_t launch_xg(float *X, const float *P, const float *G, int64_t rows, int k, float eps,
                      const float *gscale, float *out, int sms, cudaStream_t s) {
  const size_t smem = WideTile<JS>::smem(k);
  cudaFuncSetAttribute(k_wide_xg<JS, MU>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int64_t tiles = (rows + WideTile<JS>::R - 1) / WideTile<JS>::R;
  const int vec = (k & 3) == 0 && (reinterpret_cast<uintptr_t>(G) & 15) == 0;
  k_wide_xg<JS, MU><<<(unsigned)(tiles < sms ? tiles : sms), kWThreads, smem, s>>>(
      X, P, G, rows, k, eps, gscale, out, vec);
  g_launches += 1;
  return cudaGetLastError();
}

template <bool MU>
cudaError_t wide_xg(float *X, const float *P, const float *G, int64_t rows, int k, float eps,
                    const float *gscale, float *out, cudaStream_t s) {
  // R = 512 / JS rows per tile, as many as fit (k R floats in 128 KB), at the
  // fewest row-steps: rounds x (R + 64), 64 rows' worth for a round's serial part
  const int sms = wide_sms();
  int best = 8;
  int64_t cost = 0;
  for (int js = 8; js >= 2; js >>= 1) {
    const int R = 512 / js;
    if ((int64_t)k * R > 32768) break;
    const int64_t tiles = (rows + R - 1) / R, c = (tiles + sms - 1) / sms * (R + 64);
    if (js == 8 || c < cost) {
      best = js;
      cost = c;
    }
  }
  if (best == 2) return launch_xg<2, MU>(X, P, G, rows, k, eps, gscale, out, sms, s);
  if (best == 4) return launch_xg<4, MU>(X, P, G, rows, k, eps, gscale, out, sms, s);
  return launch_xg<8, MU>(X, P, G, rows, k, eps, gscale, out, sms, s);
}

template <int KT4, bool UNIT>
cudaError_t launch_sweep(float *X, const float *P, const float *G, int64_t rows, int k,
                         cudaStream_t s) {
  const size_t smem = hals_smem<KT4>(k);
  cudaFuncSetAttribute(k_wide_hals<KT4, UNIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)smem);
  const int64_t tiles = (rows + kHR - 1) / kHR;
  const int sms = wide_sms();
  k_wide_hals<KT4, UNIT><<<(unsigned)(tiles < sms ? tiles : sms), kWThreads, smem, s>>>(X, P, G,
                                                                                       rows, k);
  g_launches += 1;
  return cudaGetLastError();
}

template <bool UNIT>
cudaError_t wide_sweep(float *X, const float *P, const float *G, int64_t rows, int k,
                       cudaStream_t s) {
  switch ((k + 127) / 128) {
    case 1: return launch_sweep<1, UNIT>(X, P, G, rows, k, s);
    case 2: return launch_sweep<2, UNIT>(X, P, G, rows, k, s);
    case 3: return launch_sweep<3, UNIT>(X, P, G, rows, k, s);
    default: return launch_sweep<4, UNIT>(X, P, G, rows, k, s);
  }
}

}  // namespace

cudaError_t launch_mu_wide(float *X, const float *P, const float *G, int64_t rows, int k, float eps,
                           cudaStream_t s) {
  return wide_xg<true>(X, P, G, rows, k, eps, nullptr, nullptr, s);
}

cudaError_t launch_grad_wide(const float *X, const float *P, const float *G, int64_t rows, int k,
                             const float *gscale, float *out, cudaStream_t s) {
  return wide_xg<false>(const_cast<float *>(X), P, G, rows, k, 0.f, gscale, out, s);
}

cudaError_t launch_hals_wide(float *X, const float *P, const float *G, int64_t rows, int k,
                             bool unit, cudaStream_t s) {
  return unit ? wide_sweep<true>(X, P, G, rows, k, s) : wide_sweep<false>(X, P, G, rows, k, s);
}

}  // namespace aunmf
