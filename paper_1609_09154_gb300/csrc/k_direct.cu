// k_direct.cu -- the tensor-core products straight from the caller's FP32 A
// (Alg. 1 lines 3-4: A H^T and W^T A) for ranks up to 64, sm_103a.
//
// k_gemm_tc (k_tc.cu) streams rounded, K-major copies of A and of A^T that a
// layout pass writes first: 12 m n bytes of traffic for TF32 (read A, write
// both copies) before the first product has read its 4 m n.  Here every
// work unit rounds (and for W^T A transposes) its own tiles on the way from
// shared memory to shared memory, so a product moves A once and nothing else:
//   C (M x k) = X (M x K) Y^T, X(i, t) = A[i][t] (AHT) or A[t][i] (!AHT),
// Y = the factor's hi/lo split (2k rows, launch_split_transpose), as there.
//
// One CTA per SM, 18 warps, persistent over (256-row tile, K split) units:
//   warp 0       fills the raw ring by TMA: 256 rows x 32 K of FP32 A (AHT,
//                128-byte swizzle) or 32 K-rows x 256 columns (!AHT)
//   warp 1       TMEM, tcgen05.mma (two M = 128 MMAs share the Y tile)
//   warps 2-9    epilogue: one row of C per thread, <= 64 sums in registers,
//                TMEM chains restarted every 4 MMAs (see k_tc.cu on why)
//   warps 10-17  converters, two groups of four warps that take operand stages
//                in turn: read a raw tile, round to nearest TF32 / BF16 and write
//                the K-major 128-byte-swizzled operand tile; a group's first
//                thread also issues the copy of the stage's Y tile
// A raw tile is 32 KB; an operand stage is 32 (TF32) or 64 (BF16) K.
// When A's rows are not 16-byte aligned (lda % 4 != 0) no tensor map describes A,
// but the rows r = c (mod 4) are 16 lda bytes apart: four maps, each based on the
// 16-byte boundary at or before row c, whose rows start sh_c = 0 to 3 floats later.
// A tile is then four boxes 36 floats wide (AHT), or eight of 132 (!AHT), and the
// converters read each row at its class's shift.  (Row by row with untiled bulk
// copies it ran at 0.62 TB/s (AHT, 144-byte copies) and 2.6 TB/s (1,040 bytes);
// with 4-byte asynchronous copies at 1.6 TB/s; this way at 3.0 (TF32, the converters'
// scalar reads) and 4.2 (BF16) against 5.5 for aligned rows, whole calls at 38912 x
// 8192, k = 50.)
// The operands, MMA order and chain lengths are those of k_gemm_tc, so the
// products are the same to the bit.
//
// What bounds it: HBM, and close behind it each tile's way through a CTA (TF32,
// k = 50: the copy in, the converters' read and write, the MMAs' operand reads
// and the Y copy move ~174 KB through shared memory per 32 KB tile, by count; the
// loads and stores among them, 81 KB, by measurement).  A H^T at 96,000 x 64,000,
// k = 50: the call takes 4.04 ms, 90 % of the measured copy rate, against 14.4 +
// 3.65 ms for the layout pass and the product.  Measured on the way: all
// eight converter warps on one stage at a time 4.25 ms (each stage's latency
// chain in series); X through TMEM instead of shared memory 4.55 ms (room for
// one operand stage only beside the accumulators: conversion waits for the
// MMAs).
//
// Every mbarrier wait is bounded; on expiry the kernel raises the device error
// flag, drains the copies and MMAs it has in flight, frees TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "tc.cuh"
#include "tcgen.cuh"

namespace aunmf {
namespace tc {
namespace {

using namespace aunmf::ptx;

constexpr int kDThreads = 576;       // 18 warps
constexpr int kDGroup = 128;         // threads of one of the two converter groups
constexpr int kOp = 2;               // operand slots (group g writes slot g)
// Raw ring: four tiles of 32 KB; unaligned rows: three of 256 rows of 36 floats
// (AHT; class c's 64 rows together) or of 4 classes x 2 halves x 8 K-rows x 132.
template <bool VEC>
struct Raw {
  static constexpr int N = VEC ? 4 : 3;
  static constexpr uint32_t kBytes = VEC ? 32768 : 256 * 36 * 4;
};
constexpr int kWAht = 36, kWWta = 132;  // box widths of the unaligned form (floats)
static_assert(64 * kWWta <= 256 * kWAht, "one slot size for both directions");
struct MapsA {
  CUtensorMap m[4];  // VEC: m[0]
};
constexpr int kDTileM = 256;
constexpr uint32_t kXBytes = 32768;  // operand tile of X: 256 rows x 128 bytes

struct DirectArgs {
  const float *A;      // m x n, lda (for the shifts of unaligned rows)
  int64_t lda;
  int64_t M, K;        // C's rows, the contraction
  int64_t units;       // (tiles of 256 rows) x S
  int64_t stages;      // operand stages of the whole K
  int64_t per_split;   // operand stages per split
  int S;
  int k;               // columns of C (and its row stride)
  int BN;              // MMA N: 2k rounded up to 16
  uint32_t tmem_cols;
  float *P;            // S x M x k partials (S == 1: C)
  double *norm;        // NORM: per-CTA {sum a^2, sum a (round(a) - a)}
  int *err;
  long long wait_cycles;
  int inject;
};

// all converters
__device__ __forceinline__ void conv_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// (h, l) += x, exact to ~2^-48 (FP32 pair)
__device__ __forceinline__ void pair_acc(float x, float &h, float &l) {
  const float s = __fadd_rn(h, x), z = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(x, z)));
  h = s;
}

template <bool AHT, bool BF16, bool VEC, bool NORM>
__global__ void __launch_bounds__(kDThreads, 1)
    k_gemm_direct(const __grid_constant__ MapsA mapA, const __grid_constant__ CUtensorMap mapY,
                  const DirectArgs L) {
  constexpr int RPS = BF16 ? 2 : 1;   // raw tiles per operand stage
  constexpr int KS = 32 * RPS;        // K per operand stage (128 bytes)
  constexpr int KPM = BF16 ? 16 : 8;  // K per MMA (32 bytes)
  constexpr int kRaw = Raw<VEC>::N;
  constexpr uint32_t kRawBytes = Raw<VEC>::kBytes;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((1024 - (su32(smem_raw) & 1023)) & 1023);
  const uint32_t ybytes = (uint32_t)L.BN * 128, opbytes = kXBytes + ybytes;
  uint8_t *raw = smem, *op = smem + (size_t)kRaw * kRawBytes;
  uint64_t *rfull = reinterpret_cast<uint64_t *>(op + (size_t)kOp * opbytes);
  uint64_t *rempty = rfull + kRaw;
  uint64_t *ofull = rempty + kRaw;
  uint64_t *oempty = ofull + kOp;
  uint64_t *yfull = oempty + kOp;
  uint64_t *tfull = yfull + kOp;
  uint64_t *tempty = tfull + 2;
  uint64_t *drain = tempty + 2;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(drain + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kRaw; ++s) {
      mbar_init(&rfull[s], 1);
      mbar_init(&rempty[s], kDGroup);
    }
    for (int s = 0; s < kOp; ++s) {
      mbar_init(&ofull[s], kDGroup);
      mbar_init(&oempty[s], 1);
      mbar_init(&yfull[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 256);
    }
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async();
    for (int c = 0; c < (VEC ? 1 : 4); ++c)
      asm volatile("prefetch.tensormap [%0];" ::"l"(&mapA.m[c]) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&mapY) : "memory");
  }
  if (warp == 1) tmem_alloc(tslot, L.tmem_cols);
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *tslot;

  // operand stages [s0, s1) of unit u
  auto range = [&](int64_t u, int64_t &tile, int64_t &s0, int64_t &s1) {
    tile = u / L.S;
    const int64_t sp = u - tile * L.S;
    s0 = sp * L.per_split;
    s1 = min(L.stages, s0 + L.per_split);
  };

  if (warp == 0) {
    if (lane == 0) {
      const uint64_t pol = policy_evict_first();  // A streams through once
      constexpr uint32_t kTx = VEC ? 32768 : 4u * (AHT ? 256 * kWAht : 64 * kWWta);
      int r = 0;
      uint32_t ph = 0;
      bool ok = true;
      int64_t issued = 0;
      for (int64_t u = blockIdx.x; u < L.units && ok; u += gridDim.x) {
        int64_t tile, s0, s1;
        range(u, tile, s0, s1);
        for (int64_t t = s0 * RPS; t < s1 * RPS; ++t) {
          if (!mbar_wait(&rempty[r], ph ^ 1u, L.err, L.wait_cycles)) { ok = false; break; }
          mbar_expect_tx(&rfull[r], kTx);
          uint8_t *dst = raw + (size_t)r * kRawBytes;
          const int kc = (int)(t * 32), mc = (int)(tile * kDTileM);
          // (checked build: a bad coordinate skips the copies; the stage then
          // never fills and the bounded waits end the launch)
          if (AUNMF_BOUND(kc >= 0 && mc >= 0 && t * 32 <= 0x7fffffffLL, AUNMF_CHECK_TMA_COORD)) {
            if constexpr (VEC) {
              if (AHT)
                tma_load_2d(dst, &mapA.m[0], &rfull[r], kc, mc, pol);
              else
                tma_load_2d(dst, &mapA.m[0], &rfull[r], mc, kc, pol);
            } else {
              for (int c = 0; c < 4; ++c) {  // (tiles start at multiples of 4 rows)
                if (AHT) {
                  tma_load_2d(dst + c * 64 * kWAht * 4, &mapA.m[c], &rfull[r], kc, mc >> 2, pol);
                } else {
                  uint8_t *d = dst + c * 16 * kWWta * 4;
                  tma_load_2d(d, &mapA.m[c], &rfull[r], mc, kc >> 2, pol);
                  tma_load_2d(d + 8 * kWWta * 4, &mapA.m[c], &rfull[r], mc + kWWta, kc >> 2, pol);
                }
              }
            }
          }
          ++issued;
          if (++r == kRaw) { r = 0; ph ^= 1u; }
        }
      }
      // every copy issued lands before the CTA exits
      for (int s = 0; s < kRaw; ++s) {
        const int64_t cnt = issued / kRaw + (s < issued % kRaw ? 1 : 0);
        if (cnt > 0) mbar_wait_drain(&rfull[s], (uint32_t)((cnt - 1) & 1), L.wait_cycles);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int st = 0, buf = 0;
      uint32_t ph = 0, tph = 0;
      bool ok = true, withheld = false;
      const uint32_t id = idesc(BF16, 128, L.BN);
      for (int64_t u = blockIdx.x; u < L.units && ok; u += gridDim.x) {
        int64_t tile, s0, s1;
        range(u, tile, s0, s1);
        for (int64_t s = s0; s < s1; ++s) {
          if (!mbar_wait(&tempty[buf], tph ^ 1u, L.err, L.wait_cycles) ||
              !mbar_wait(&yfull[st], ph, L.err, L.wait_cycles) ||
              !mbar_wait(&ofull[st], ph, L.err, L.wait_cycles)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d0 = tbase + (uint32_t)(buf * 2 * L.BN), d1 = d0 + (uint32_t)L.BN;
          const uint32_t xs = su32(op + (size_t)st * opbytes), ys = xs + kXBytes;
#pragma unroll
          for (int kk = 0; kk < KS / KPM; ++kk) {
            const uint32_t off = (uint32_t)(kk * 32);
            const uint64_t bd = sdesc(ys + off);
            mma<BF16>(d0, sdesc(xs + off), bd, id, kk > 0);
            mma<BF16>(d1, sdesc(xs + kXBytes / 2 + off), bd, id, kk > 0);
          }
          mma_commit(&oempty[st]);
          if (++st == kOp) { st = 0; ph ^= 1u; }
          if (L.inject && !withheld)
            withheld = true;  // test hook: the epilogue's wait for this chunk runs out
          else
            mma_commit(&tfull[buf]);
          if (++buf == 2) { buf = 0; tph ^= 1u; }
        }
      }
    }
  } else if (warp < 10) {
    // epilogue: warp w drains TMEM lane quarter w % 4 of accumulator half
    // (w - 2) / 4; C_i = acc_2i + acc_2i+1 for i < BN / 2
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int rl = half * 128 + q * 32 + lane;
    int buf = 0;
    uint32_t tph = 0;
    bool ok = true;
    for (int64_t u = blockIdx.x; u < L.units && ok; u += gridDim.x) {
      int64_t tile, s0, s1;
      range(u, tile, s0, s1);
      float acc[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) acc[j] = 0.f;
      for (int64_t s = s0; s < s1; ++s) {
        if (!mbar_wait(&tfull[buf], tph, L.err, L.wait_cycles)) { ok = false; break; }
        tc_fence_after();
        const uint32_t taddr =
            tbase + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 2 * L.BN + half * L.BN);
#pragma unroll
        for (int g = 0; g < 8; ++g) {  // 16 columns at a time: BN is a multiple of 16
          if (16 * g >= L.BN) break;
          uint32_t r[16];
          tmem_ld16_async(taddr + (uint32_t)(16 * g), r);
          tmem_wait_ld(r);
#pragma unroll
          for (int j = 0; j < 8; ++j)
            acc[8 * g + j] += __uint_as_float(r[2 * j]) + __uint_as_float(r[2 * j + 1]);
        }
        tc_fence_before();
        mbar_arrive(&tempty[buf]);
        if (++buf == 2) { buf = 0; tph ^= 1u; }
      }
      if (!ok) break;
      const int64_t row = tile * kDTileM + rl;
      if (row < L.M) {
        float *dg = L.P + ((u - tile * L.S) * L.M + row) * L.k;
#pragma unroll
        for (int o = 0; o < 64; ++o)
          if (o < L.k) dg[o] = acc[o];
      }
    }
  } else {
    // converters
    const int grp = (warp - 10) >> 2, t = (threadIdx.x - 320) & 127;
    const uint64_t pol_y = policy_evict_last();
    int64_t yissued = 0;
    bool ok = true;
    // NORM: chains of 16 terms, as launch_prepare sums them, joined in FP32 pairs
    // (a chain over the thread's whole 64 terms of a tile errs four times as much on
    // entries of few values; every chain into FP64, as there, took 524 us for the
    // loss of 20,000 x 24,000, k = 50, TF32, and 500 BF16, this way 495 and 416, the
    // chain of 64 480 and 409).  The pairs hold a quarter of the sums, so that a
    // tile's four chains fit wherever one does, and go to FP64 before they are large.
    float nh = 0.f, nl = 0.f, dh = 0.f, dl = 0.f;
    double na = 0.0, nd = 0.0;
    float sq = 0.f, sd = 0.f;
    auto join = [&]() {
      if constexpr (NORM) {
        pair_acc(0.25f * sq, nh, nl);
        pair_acc(0.25f * sd, dh, dl);
        sq = sd = 0.f;
      }
    };
    auto use = [&](float a) {  // rounded value, and the two sums of it
      float v;
      if constexpr (BF16)
        v = __bfloat162float(__float2bfloat16_rn(a));
      else
        v = round_tf32(a);
      if constexpr (NORM) {
        sq = fmaf(a, a, sq);
        sd = fmaf(a, v - a, sd);  // difference exact
      }
      return v;
    };
    auto pack_bf = [&](float a, float b) {  // (values already BF16-valued) -> bf16x2
      return (__float_as_uint(a) >> 16) | (__float_as_uint(b) & 0xffff0000u);
    };
    // The CTA's operand stages are numbered q = 0, 1, ... over its units; group
    // g takes q = g, g + 2, ...  Walks them: unit u, stage s of it.
    struct Walk {
      int64_t u, tile, s, s1, q;
    };
    auto enter = [&](Walk &w) {  // first stage of unit w.u, if there is one
      if (w.u < L.units) range(w.u, w.tile, w.s, w.s1);
    };
    auto step = [&](Walk &w, int64_t by) {
      w.q += by;
      while (by > 0 && w.u < L.units) {
        if (w.s + by < w.s1) { w.s += by; return; }
        by -= w.s1 - w.s;
        w.u += gridDim.x;
        enter(w);
      }
    };
    Walk w{(int64_t)blockIdx.x, 0, 0, 0, 0};
    enter(w);
    step(w, grp);
    // unaligned form: the shift of class c, and (!AHT) the place of this thread's
    // rows t and t + 128 in class c's first K-row
    int sh[4], o0[4], o1[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      sh[c] = VEC ? 0 : (int)(((reinterpret_cast<uintptr_t>(L.A) >> 2) + c * (L.lda & 3)) & 3);
      const int f0 = sh[c] + t, f1 = f0 + 128;
      o0[c] = c * 16 * kWWta + f0 + (f0 < kWWta ? 0 : 7 * kWWta);
      o1[c] = c * 16 * kWWta + f1 + (f1 < kWWta ? 0 : 7 * kWWta);
    }
    for (; w.u < L.units && ok; step(w, 2)) {
      const uint32_t use_no = (uint32_t)(w.q >> 1);  // uses of operand slot grp so far
      if (!mbar_wait(&oempty[grp], (use_no & 1u) ^ 1u, L.err, L.wait_cycles)) break;
      uint8_t *xo = op + (size_t)grp * opbytes;
      if (t == 0) {
        mbar_expect_tx(&yfull[grp], ybytes);
        tma_load_2d(xo + kXBytes, &mapY, &yfull[grp], (int)(w.s * KS), 0, pol_y);
        ++yissued;
      }
#pragma unroll
      for (int h = 0; h < RPS; ++h) {
        const int64_t tr = w.q * RPS + h;  // raw tile number
        const int r = (int)(tr % kRaw);
        if (!mbar_wait(&rfull[r], (uint32_t)(tr / kRaw) & 1u, L.err, L.wait_cycles)) {
          ok = false;
          break;
        }
        const float *rw = reinterpret_cast<const float *>(raw + (size_t)r * kRawBytes);
        // (unaligned form: K past the end, which a class without rows does not
        // zero-fill)
        const int kv = VEC ? 32 : (int)min((int64_t)32, L.K - (w.s * RPS + h) * 32);
        auto at = [&](int kk, int i) {  // !AHT: entry (kk, t + 128 i) of the raw tile
          if constexpr (VEC) return rw[kk * 256 + t + 128 * i];
          return kk < kv ? rw[(i ? o1 : o0)[kk & 3] + (kk >> 2) * kWWta] : 0.f;
        };
        if constexpr (AHT && !VEC) {
          // a warp per row (TF32) or two (BF16), lanes along K
          constexpr int LPR = BF16 ? 16 : 32;
          const int l = lane & (LPR - 1);
#pragma unroll 8
          for (int row = (t >> 5) * (32 / LPR) + lane / LPR; row < 256; row += 4 * (32 / LPR)) {
            const float *src = rw + ((row & 3) * 64 + (row >> 2)) * kWAht + sh[row & 3];
            const int x = row & 7;
            if constexpr (BF16) {
              const float a = 2 * l < kv ? src[2 * l] : 0.f, b = 2 * l + 1 < kv ? src[2 * l + 1] : 0.f;
              reinterpret_cast<uint32_t *>(xo)[row * 32 + (((4 * h + (l >> 2)) ^ x) << 2) + (l & 3)] =
                  pack_bf(use(a), use(b));
            } else {
              reinterpret_cast<float *>(xo)[row * 32 + (((l >> 2) ^ x) << 2) + (l & 3)] =
                  use(l < kv ? src[l] : 0.f);
            }
          }
        } else if constexpr (AHT && !BF16) {
          // same swizzled place in the operand tile
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float4 v = reinterpret_cast<const float4 *>(rw)[t + 128 * i];
            reinterpret_cast<float4 *>(xo)[t + 128 * i] =
                make_float4(use(v.x), use(v.y), use(v.z), use(v.w));
          }
        } else if constexpr (AHT) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int row = (t >> 2) + 32 * i, j = t & 3, x = row & 7;
            const float4 a = reinterpret_cast<const float4 *>(rw)[row * 8 + ((2 * j) ^ x)];
            const float4 b = reinterpret_cast<const float4 *>(rw)[row * 8 + ((2 * j + 1) ^ x)];
            uint4 o;
            o.x = pack_bf(use(a.x), use(a.y));
            o.y = pack_bf(use(a.z), use(a.w));
            o.z = pack_bf(use(b.x), use(b.y));
            o.w = pack_bf(use(b.z), use(b.w));
            reinterpret_cast<uint4 *>(xo)[row * 8 + ((4 * h + j) ^ x)] = o;
          }
        } else if constexpr (!BF16) {
          // thread t owns rows t and t + 128 of the operand tile
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int c = i >> 1, row = t + 128 * (i & 1);
            const float a0 = at(4 * c, i & 1), a1 = at(4 * c + 1, i & 1);
            const float a2 = at(4 * c + 2, i & 1), a3 = at(4 * c + 3, i & 1);
            reinterpret_cast<float4 *>(xo)[row * 8 + (c ^ (row & 7))] =
                make_float4(use(a0), use(a1), use(a2), use(a3));
            if ((i & 3) == 3) join();
          }
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int c = i >> 1, row = t + 128 * (i & 1);
            float a[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) a[e] = at(8 * c + e, i & 1);
            uint4 o;
            o.x = pack_bf(use(a[0]), use(a[1]));
            o.y = pack_bf(use(a[2]), use(a[3]));
            o.z = pack_bf(use(a[4]), use(a[5]));
            o.w = pack_bf(use(a[6]), use(a[7]));
            reinterpret_cast<uint4 *>(xo)[row * 8 + ((4 * h + c) ^ (row & 7))] = o;
            if (i & 1) join();
          }
        }
        if constexpr (NORM)
          if (nh > 1e30f) {  // (|dh| is smaller)
            na += (double)nh;
            nd += (double)dh;
            if (isinf(nh)) nl = 0.f;  // (inf - inf in the pair's sum)
            nh = dh = 0.f;
          }
        // Both proxies meet here: the raw tile has been read and the next copy
        // overwrites it, the operand tile has been written and the MMAs read it.
        // (An arrival right behind the loads, without the fence, was seen to let a
        // tile that hits L2 overwrite the slot under them: values of the tile after
        // next.)
        fence_async();
        mbar_arrive(&rempty[r]);
      }
      if (!ok) break;
      mbar_arrive(&ofull[grp]);
    }
    if (t == 0 && yissued > 0)  // the Y copies issued land before the CTA exits
      mbar_wait_drain(&yfull[grp], (uint32_t)((yissued - 1) & 1), L.wait_cycles);
    if constexpr (NORM) {
      // fixed order: lanes by butterfly, then the eight warps
      double a = 4.0 * (na + ((double)nh + (double)nl)), d = 4.0 * (nd + ((double)dh + (double)dl));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        d += __shfl_xor_sync(0xffffffffu, d, o);
      }
      __shared__ double ws[2][8];
      if (lane == 0) {
        ws[0][warp - 10] = a;
        ws[1][warp - 10] = d;
      }
      conv_bar();
      if (grp == 0 && t == 0) {
        a = d = 0.0;
        for (int w = 0; w < 8; ++w) {
          a += ws[0][w];
          d += ws[1][w];
        }
        L.norm[2 * blockIdx.x] = a;
        L.norm[2 * blockIdx.x + 1] = d;
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    if (lane == 0) {
      mma_commit(drain);
      mbar_wait_drain(drain, 0u, L.wait_cycles);
    }
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tbase, L.tmem_cols);
  }
}

// 2-D map over row-major FP32 rows x cols (leading dimension ld) with a box of
// box_cols x box_rows; zero fill outside.
bool map_f32(CUtensorMap *map, const float *base, int64_t rows, int64_t cols, int64_t ld,
             int box_cols, int box_rows, bool swizzle) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * 4)};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

cudaError_t launch_gemm_direct(bool aht, const float *A, int64_t m, int64_t n, int64_t lda,
                               const void *Y, int k, int64_t ldy, bool bf16, float *parts, int S,
                               double *part, double *norm2, int *err, cudaStream_t s) {
  const int64_t M = aht ? m : n, K = aht ? n : m;
  const int ks = bf16 ? 64 : 32;
  DirectArgs L{};
  L.BN = (2 * k + 15) / 16 * 16;
  if (L.BN > 128 || (aht && norm2)) return cudaErrorInvalidValue;
  L.A = A;
  L.lda = lda;
  L.M = M;
  L.K = K;
  L.S = S;
  L.stages = (K + ks - 1) / ks;
  L.per_split = (L.stages + S - 1) / S;
  L.units = (M + kDTileM - 1) / kDTileM * S;
  L.k = k;
  L.tmem_cols = 32;
  while (L.tmem_cols < (uint32_t)(4 * L.BN)) L.tmem_cols <<= 1;
  L.P = parts;
  L.norm = part;
  L.err = err;
  L.wait_cycles = fault::wait_cycles();
  L.inject = fault::site() == AUNMF_INJECT_TC_WAIT ? 1 : 0;
  MapsA mapA;
  CUtensorMap mapY;
  if (!factor_map(&mapY, Y, bf16, 2 * k, K, ldy, L.BN)) return cudaErrorInvalidValue;
  const bool vec = (reinterpret_cast<uintptr_t>(A) & 15) == 0 && (lda & 3) == 0;
  for (int c = 0; c < 4; ++c) {
    bool ok;
    if (vec) {
      ok = aht ? map_f32(&mapA.m[c], A, m, n, lda, 32, 256, true)
               : map_f32(&mapA.m[c], A, m, n, lda, 256, 32, false);
    } else {
      // rows c, c + 4, ...; a class without rows is never used unmasked: class 0's
      const int cc = c < m ? c : 0;
      const uintptr_t a = reinterpret_cast<uintptr_t>(A + cc * lda), b = a & ~(uintptr_t)15;
      ok = map_f32(&mapA.m[c], reinterpret_cast<const float *>(b), (m - cc + 3) / 4,
                   n + (int64_t)((a - b) >> 2), 4 * lda, aht ? kWAht : kWWta, aht ? 64 : 8, false);
    }
    if (!ok) return cudaErrorInvalidValue;
  }
  const size_t raw = vec ? (size_t)Raw<true>::N * Raw<true>::kBytes
                         : (size_t)Raw<false>::N * Raw<false>::kBytes;
  const size_t smem = 1024 + raw +
                      (size_t)kOp * (kXBytes + (size_t)L.BN * 128) + 256;
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = (int)std::min<int64_t>(L.units, sms > 0 ? sms : 148);
  auto go = [&](auto kern) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<grid, kDThreads, smem, s>>>(mapA, mapY, L);
  };
  auto pick = [&](auto a, auto b, auto t, auto nm) {
    go(k_gemm_direct<decltype(a)::value, decltype(b)::value, decltype(t)::value, decltype(nm)::value>);
  };
  using Y1 = std::true_type;
  using N0 = std::false_type;
  auto by_vec = [&](auto a, auto b, auto nm) {
    if (vec) pick(a, b, Y1{}, nm); else pick(a, b, N0{}, nm);
  };
  auto by_prec = [&](auto a, auto nm) {
    if (bf16) by_vec(a, Y1{}, nm); else by_vec(a, N0{}, nm);
  };
  if (aht) by_prec(Y1{}, N0{});
  else if (norm2) by_prec(N0{}, Y1{});
  else by_prec(N0{}, N0{});
  g_launches += 1;
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess || !norm2 ? e : launch_sum_norm(part, grid, norm2, s);
}

}  // namespace tc
}  // namespace aunmf
