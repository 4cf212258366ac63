// Differentiable form with eta kept on the chip (Section 2.9; p <= 256
// covariates): the products X B and X^T G run on the tensor cores as in
// nll_tc.cu, but the risk-set scan is the epilogue of the forward product and
// G is formed between the two products of the backward pass.  X is read once
// in each direction and nothing of size n x C is written: at n = 2^22,
// p = 256, C = 64 that is 2 x 2.15 GB of traffic instead of 9.3 GB (eta
// written, read by the scan and by the gradient kernel; G written and read),
// k_nll_fwd takes 403 us (316 at 6.8 TB/s) where the product and the scan took
// 742, and k_nll_bwd 459 where the gradient rows and the product took 843.
//
// Both kernels form eta transposed: D (128 x rows) = Bcat^T X^T, so a TMEM
// lane is a column of B and a TMEM column is a subject, and a thread walks
// subjects in time order.  Bcat^T holds, for each group of 16 columns, the 16
// high parts in lanes 0..15 of a warp's quadrant and the 16 low parts in
// lanes 16..31; one exchange between lanes l and l + 16 adds them, after
// which lane l owns the column for the first half of the rows and lane l + 16
// for the second half.
//
//   k_nll_fwd  a CTA owns four units of consecutive rows (two sets of
//              epilogue warps x two halves of a quadrant); a tile is 64 rows
//              of two units.  The epilogue takes e = exp(eta), running sums
//              in float-float (8 rows in FP32 at a time, as k_nll_scan), the
//              prefix at the group ends, and sum delta eta.
//   k_nll_bwd  a CTA owns a range of rows; a tile of 128 rows of X stays in
//              shared memory for both products: eta (as above), G = g (e
//              Lambda - delta) as bf16 high and low parts written back to
//              shared memory in the K-major layout of a tensor-core operand,
//              then D2 (128 x p) += G_tile^T X_tile, X read as the MN-major
//              operand.  The partial sums of the CTAs go to k_xtg_reduce.
//              The tensor pipe bounds it, so both products are issued as few
//              wide instructions: X always the wide operand, Bcat^T kept in
//              tensor memory, tiles of 128 rows (cycles per 64 rows: 3,570 with
//              X as the first operand of the second product and 64-row tiles,
//              2,780 with X as its second, 1,980 with 128-row tiles).
//
// Warp roles: warp 0 TMA, warp 1 MMA and TMEM allocation, then the epilogue
// sets of four warps (one per TMEM quadrant): two in the forward kernel, four
// in the backward kernel.  Every wait is bounded; a wait
// that expires sets *err and the CTA unwinds.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "internal.h"
#include "tc.cuh"
#include "workspace.h"

namespace survgpu {
namespace {

using tc::mbar_wait;

constexpr int kFuThreads = 320;      // forward: two epilogue sets of four warps
constexpr int kFuBwdThreads = 576;   // backward: four
constexpr int kFuBoxK = 64;
constexpr int kFuMaxStages = 12;
constexpr int kFuMaxKb = 4;          // p <= 256
constexpr uint64_t kFuWaitNs = 2000000000ull;
constexpr uint32_t kFuBoxBytes = 64 * 128;   // 64 rows x 64 bf16

struct alignas(8) FuBars {
  uint64_t full[kFuMaxStages];
  uint64_t empty[kFuMaxStages];
  uint64_t bfull;
  uint64_t tfull[2];
  uint64_t tempty[2];
  uint64_t gfull[2];
  uint64_t gempty[2];
  uint64_t done;
  uint32_t tmem_base;
  int32_t abort;
};

__device__ __forceinline__ void raise_abort(FuBars* b, unsigned* err) {
  atomicOr(err, 1u);
  *reinterpret_cast<volatile int32_t*>(&b->abort) = 1;
}
__device__ __forceinline__ bool aborted(FuBars* b) { return *reinterpret_cast<volatile int32_t*>(&b->abort) != 0; }

__device__ __forceinline__ unsigned char* align1k(unsigned char* p) {
  return reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// eta of the thread's rows from the two halves of its TMEM lane: v0 the rows
// of the first half, v1 of the second (see above)
template <int N>
__device__ __forceinline__ void combine(const float (&v0)[N], const float (&v1)[N], bool upper, float (&eta)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float got = __shfl_xor_sync(0xffffffffu, upper ? v0[i] : v1[i], 16);
    eta[i] = (upper ? v1[i] : v0[i]) + got;
  }
}

// ----------------------------------------------------------------- forward
__global__ void __launch_bounds__(kFuThreads, 1)
    k_nll_fwd(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapB, int64_t n, int nkb,
              int C, int ns, int64_t ru, const uint32_t* __restrict__ endw, const uint32_t* __restrict__ evw,
              const int32_t* __restrict__ wordk, float2* __restrict__ rec, float2* __restrict__ wt,
              float2* __restrict__ wd, unsigned* err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sB = align1k(smem_raw);                       // nkb boxes of 128 rows
  unsigned char* sX = sB + (size_t)nkb * 2 * kFuBoxBytes;      // ns stages of 2 boxes (one per half)
  FuBars* bars = reinterpret_cast<FuBars*>(sX + (size_t)ns * 2 * kFuBoxBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // unit u = 4 cta + 2 set + half holds rows [u ru, (u + 1) ru); tiles of set
  // s: 64 rows of each half, while the first half has rows
  int64_t u0[2], nt[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    u0[s] = (int64_t)blockIdx.x * 4 + 2 * s;
    const int64_t left = n - u0[s] * ru;
    nt[s] = left <= 0 ? 0 : min(ru, (left + 63) / 64 * 64) / 64;
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < kFuMaxStages; ++s) {
      tc::mbar_init(&bars->full[s], 1);
      tc::mbar_init(&bars->empty[s], 1);
    }
    tc::mbar_init(&bars->bfull, 1);
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(&bars->tfull[a], 1);
      tc::mbar_init(&bars->tempty[a], 128);
    }
    tc::mbar_init(&bars->done, 1);
    bars->abort = 0;
    tc::mbar_fence_init();
  }
  if (warp == 1) tc::tmem_alloc(&bars->tmem_base, 256);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = bars->tmem_base;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    tc::tma_prefetch_map(&mapX);
    tc::tma_prefetch_map(&mapB);
    tc::mbar_arrive_expect_tx(&bars->bfull, (uint32_t)nkb * 2 * kFuBoxBytes);
    for (int kb = 0; kb < nkb; ++kb)
      tc::tma_load_2d(sB + (size_t)kb * 2 * kFuBoxBytes, &mapB, &bars->bfull, kb * kFuBoxK, 0);
    int64_t it = 0;
    int s = 0;
    uint32_t round = 0;
    for (int64_t t = 0; t < nt[0] && !aborted(bars); ++t)
      for (int a = 0; a < 2; ++a) {
        if (t >= nt[a]) continue;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          if (round > 0 && !mbar_wait(&bars->empty[s], (round - 1) & 1, kFuWaitNs)) {
            raise_abort(bars, err);
            break;
          }
          unsigned char* st = sX + (size_t)s * 2 * kFuBoxBytes;
          tc::mbar_arrive_expect_tx(&bars->full[s], 2 * kFuBoxBytes);
          tc::tma_load_2d(st, &mapX, &bars->full[s], kb * kFuBoxK, (int)(u0[a] * ru + 64 * t));
          tc::tma_load_2d(st + kFuBoxBytes, &mapX, &bars->full[s], kb * kFuBoxK, (int)((u0[a] + 1) * ru + 64 * t));
          if (++s == ns) {
            s = 0;
            ++round;
          }
        }
      }
    // every issued copy has landed before the CTA may exit: the last use of
    // each slot (slots before s in this round, the others in the previous)
    if (!mbar_wait(&bars->bfull, 0, kFuWaitNs)) raise_abort(bars, err);
    for (int q = 0; q < ns; ++q) {
      const int64_t last = q < s ? (int64_t)round : (int64_t)round - 1;
      if (last >= 0 && !mbar_wait(&bars->full[q], (uint32_t)(last & 1), kFuWaitNs)) raise_abort(bars, err);
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer
    const uint32_t idesc = tc::idesc_bf16_f32(128, 128, false, false);
    bool ok = mbar_wait(&bars->bfull, 0, kFuWaitNs);
    if (!ok) raise_abort(bars, err);
    int s = 0;
    uint32_t round = 0;
    for (int64_t t = 0; ok && t < nt[0]; ++t)
      for (int a = 0; ok && a < 2; ++a) {
        if (t >= nt[a]) continue;
        if (t > 0 && !mbar_wait(&bars->tempty[a], (uint32_t)((t - 1) & 1), kFuWaitNs)) {
          raise_abort(bars, err);
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const uint32_t d = tmem + (uint32_t)(a * 128);
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait(&bars->full[s], round & 1, kFuWaitNs) || aborted(bars)) {
            raise_abort(bars, err);
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint32_t b_addr = tc::smem_u32(sB + (size_t)kb * 2 * kFuBoxBytes);
          const uint32_t x_addr = tc::smem_u32(sX + (size_t)s * 2 * kFuBoxBytes);
#pragma unroll
          for (int k = 0; k < kFuBoxK / 16; ++k)
            tc::mma_bf16(d, tc::sdesc_sw128(b_addr + 32u * k, 16u, 1024u), tc::sdesc_sw128(x_addr + 32u * k, 16u, 1024u),
                         idesc, (kb | k) != 0 ? 1u : 0u);
          tc::mma_commit(&bars->empty[s]);
          if (++s == ns) {
            s = 0;
            ++round;
          }
        }
        if (ok) tc::mma_commit(&bars->tfull[a]);
      }
    tc::mma_commit(&bars->done);
    if (!mbar_wait(&bars->done, 0, kFuWaitNs)) raise_abort(bars, err);
  } else if (warp >= 2) {
    // ---------------- epilogue: the risk-set scan
    const int a = (warp - 2) >> 2, q = warp & 3;
    const bool upper = lane >= 16;
    const int c = 16 * q + (lane & 15);
    const bool has = c < C;
    const bool busy = 16 * q < C;           // the warp's quadrant holds columns
    const int64_t unit = u0[a] + (upper ? 1 : 0);
    const int64_t row0 = unit * ru;
    const int64_t nwords = (n + 31) >> 5;
    const uint32_t tq = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(a * 128);
    ff acc = ff_zero(), dl = ff_zero();
    // end and event masks of a tile's 64 rows and the group of its first end,
    // loaded one tile ahead
    uint32_t en1[2], ev1[2];
    int k1;
    auto load_masks = [&](int64_t t) {
      const int64_t w = (row0 >> 5) + 2 * t;
      const bool in = t < nt[a] && w < nwords, two = in && w + 1 < nwords;
      en1[0] = in ? endw[w] : 0u;
      ev1[0] = in ? evw[w] : 0u;
      k1 = in ? wordk[w] : 0;
      en1[1] = two ? endw[w + 1] : 0u;
      ev1[1] = two ? evw[w + 1] : 0u;
    };
    load_masks(0);
    for (int64_t t = 0; t < nt[a]; ++t) {
      const uint32_t en[2] = {en1[0], en1[1]}, ev[2] = {ev1[0], ev1[1]};
      int k = k1;
      load_masks(t + 1);
      const bool good = mbar_wait(&bars->tfull[a], (uint32_t)(t & 1), kFuWaitNs) && !aborted(bars);
      if (!__all_sync(0xffffffffu, good)) {   // the whole warp leaves together
        raise_abort(bars, err);
        break;
      }
      tc::fence_after_sync();
      if (busy) {
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          float v0[16], v1[16], eta[16];
          tc::tmem_ld16x2(tq + (uint32_t)(16 * ch), tq + (uint32_t)(64 + 16 * ch), v0, v1);
          combine(v0, v1, upper, eta);
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const uint32_t e8 = en[ch >> 1] >> (16 * (ch & 1) + 8 * g) & 255u;
            const uint32_t d8 = ev[ch >> 1] >> (16 * (ch & 1) + 8 * g) & 255u;
            float e[8], p = 0.f, s = 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) e[u] = expf(eta[8 * g + u]);
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (d8 >> u & 1u) s += eta[8 * g + u];
            if (e8 == 0u) {
#pragma unroll
              for (int u = 0; u < 8; ++u) p += e[u];
            } else {
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                p += e[u];
                if (e8 >> u & 1u) {   // a group end: the running prefix of the unit
                  const ff r = ff_add_f(acc, p);
                  if (has) rec[(size_t)k * C + c] = make_float2(r.hi, r.lo);
                  ++k;
                }
              }
            }
            acc = ff_add_f(acc, p);
            dl = ff_add_f(dl, s);
          }
        }
      }
      tc::fence_before_sync();
      tc::mbar_arrive(&bars->tempty[a]);
    }
    if (has) {
      wt[(size_t)unit * C + c] = make_float2(acc.hi, acc.lo);
      wd[(size_t)unit * C + c] = make_float2(dl.hi, dl.lo);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, 256);
  }
}

// ---------------------------------------------------------------- backward
__global__ void __launch_bounds__(kFuBwdThreads, 1)
    k_nll_bwd(const __grid_constant__ CUtensorMap mapX, const uint32_t* __restrict__ bcat, int ldw, int64_t n, int p,
              int nkb, int C, int Cp, int K, int ns, int64_t rows_per_cta, const uint32_t* __restrict__ endw,
              const uint32_t* __restrict__ evw, const int32_t* __restrict__ wordk, const float* __restrict__ lam,
              const double* __restrict__ gout, float* __restrict__ part, unsigned* err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t xbytes = (uint32_t)nkb * 2 * kFuBoxBytes;      // one tile of X: nkb boxes of 128 rows
  unsigned char* sX = align1k(smem_raw);                        // ns tiles
  unsigned char* sG = sX + (size_t)ns * xbytes;                 // G: 2 boxes of 128 rows (parts) x 64 subjects
  constexpr uint32_t gbytes = 128u * 128u;                      // one box
  FuBars* bars = reinterpret_cast<FuBars*>(sG + 2 * (size_t)gbytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int NB = 2 * Cp;
  const int64_t r_lo = min((int64_t)blockIdx.x * rows_per_cta, n);
  const int64_t r_hi = min(r_lo + rows_per_cta, n);
  const int64_t nt = (r_hi - r_lo + 127) / 128;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kFuMaxStages; ++s) {
      tc::mbar_init(&bars->full[s], 1);
      tc::mbar_init(&bars->empty[s], 1);
    }
    tc::mbar_init(&bars->tfull[0], 1);
    tc::mbar_init(&bars->tempty[0], 16);   // one arrival per epilogue warp
    tc::mbar_init(&bars->gfull[0], 16);
    tc::mbar_init(&bars->gempty[0], 1);
    tc::mbar_init(&bars->done, 1);
    bars->abort = 0;
    tc::mbar_fence_init();
  }
  if (warp == 1) tc::tmem_alloc(&bars->tmem_base, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = bars->tmem_base;
  const uint32_t a1 = tmem + 384u;          // Bcat^T: 32 columns (64 covariates) per box
  if (warp >= 2 && warp < 6) {
    // Bcat^T into tensor memory, a row a lane: as an operand in shared memory
    // it was fetched again for every tile (two thirds of the first product's
    // shared-memory traffic)
    const uint32_t* src = bcat + (size_t)(32 * (warp & 3) + lane) * ldw;
    for (int w0 = 0; w0 < nkb * 32; w0 += 8) {
      uint32_t v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = w0 + i < ldw ? src[w0 + i] : 0u;
      tc::tmem_st8(a1 + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)w0, v);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t d2 = tmem + 128u;          // D1: 128 columns (the subjects of a tile); D2: nkb x 64 columns

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    tc::tma_prefetch_map(&mapX);
    int s = 0;
    uint32_t round = 0;
    for (int64_t t = 0; t < nt && !aborted(bars); ++t) {
      if (round > 0 && !mbar_wait(&bars->empty[s], (round - 1) & 1, kFuWaitNs)) {
        raise_abort(bars, err);
        break;
      }
      unsigned char* st = sX + (size_t)s * xbytes;
      tc::mbar_arrive_expect_tx(&bars->full[s], xbytes);
      for (int kb = 0; kb < nkb; ++kb)
        tc::tma_load_2d(st + (size_t)kb * 2 * kFuBoxBytes, &mapX, &bars->full[s], kb * kFuBoxK, (int)(r_lo + 128 * t));
      if (++s == ns) {
        s = 0;
        ++round;
      }
    }
    for (int q = 0; q < ns; ++q) {
      const int64_t last = q < s ? (int64_t)round : (int64_t)round - 1;
      if (last >= 0 && !mbar_wait(&bars->full[q], (uint32_t)(last & 1), kFuWaitNs)) raise_abort(bars, err);
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer: eta of tile t + 1 before X^T G of tile t
    const uint32_t id1 = tc::idesc_bf16_f32(128, 128, false, false);
    const uint32_t id2 = tc::idesc_bf16_f32(128, nkb * kFuBoxK, false, true);
    bool ok = true;
    int s1 = 0, s2 = 0;
    uint32_t round1 = 0;
    auto first = [&](int64_t t) -> bool {   // D1 = Bcat^T X_tile^T
      if (t >= 1 && !mbar_wait(&bars->tempty[0], (uint32_t)((t - 1) & 1), kFuWaitNs)) return false;
      if (!mbar_wait(&bars->full[s1], round1 & 1, kFuWaitNs) || aborted(bars)) return false;
      tc::fence_after_sync();
      const uint32_t x = tc::smem_u32(sX + (size_t)s1 * xbytes);
      for (int kb = 0; kb < nkb; ++kb) {
        const uint32_t x_addr = x + (uint32_t)kb * 2 * kFuBoxBytes;
#pragma unroll
        for (int k = 0; k < kFuBoxK / 16; ++k)
          tc::mma_bf16_ts(tmem, a1 + (uint32_t)(32 * kb + 8 * k),
                          tc::sdesc_sw128(x_addr + 32u * k, 16u, 1024u), id1, (kb | k) != 0 ? 1u : 0u);
      }
      tc::mma_commit(&bars->tfull[0]);
      if (++s1 == ns) {
        s1 = 0;
        ++round1;
      }
      return true;
    };
    if (ok && nt > 0 && !first(0)) {
      raise_abort(bars, err);
      ok = false;
    }
    for (int64_t t = 0; ok && t < nt; ++t) {
      if (t + 1 < nt && !first(t + 1)) {
        raise_abort(bars, err);
        ok = false;
        break;
      }
      if (!mbar_wait(&bars->gfull[0], (uint32_t)(t & 1), kFuWaitNs) || aborted(bars)) {
        raise_abort(bars, err);
        ok = false;
        break;
      }
      tc::fence_after_sync();
      const uint32_t x = tc::smem_u32(sX + (size_t)s2 * xbytes), gb = tc::smem_u32(sG);
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        tc::mma_bf16(d2, tc::sdesc_sw128(gb + (uint32_t)(ks >> 2) * gbytes + 32u * (ks & 3), 16u, 1024u),
                     tc::sdesc_sw128(x + 2048u * ks, 2 * kFuBoxBytes, 1024u), id2, (t | ks) != 0 ? 1u : 0u);
      tc::mma_commit(&bars->empty[s2]);
      tc::mma_commit(&bars->gempty[0]);
      if (++s2 == ns) s2 = 0;
    }
    tc::mma_commit(&bars->done);
    if (!mbar_wait(&bars->done, 0, kFuWaitNs)) raise_abort(bars, err);
  } else if (warp >= 2) {
    // ---------------- epilogue: 32 rows of each tile per set
    const int a = (warp - 2) >> 2, q = warp & 3;
    const bool upper = lane >= 16;
    const int c = 16 * q + (lane & 15);
    const bool has = c < C, busy = 16 * q < Cp;
    const float g = has ? (float)gout[c] : 0.f;
    const int64_t nwords = (n + 31) >> 5;
    const uint32_t tq = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(32 * a);
    const int sh = upper ? 16 : 0;
    bool ok = true;
    // The masks of the thread's 16 rows of a tile (half a word of the set's 32)
    // are loaded two tiles ahead, and Lambda of its first group, which needs
    // them, one ahead: two dependent loads a tile stood in every
    // epilogue's way otherwise.
    struct Rows {
      uint32_t en, ev;
      int k;
    };
    auto load_rows = [&](int64_t t) {
      Rows r = {0u, 0u, K};
      const int64_t w = (r_lo + 128 * t + 32 * a) >> 5;
      if (t < nt && w < nwords) {
        const uint32_t word = endw[w];
        r.en = word >> sh & 0xffffu;
        r.ev = evw[w] >> sh & 0xffffu;
        r.k = wordk[w] + __popc(word & ((1u << sh) - 1u));
      }
      return r;
    };
    auto load_lam = [&](int k) { return has && k < K ? lam[(size_t)k * C + c] : 0.f; };
    Rows cur = load_rows(0), nxt = load_rows(1);
    float l = load_lam(cur.k);
    for (int64_t t = 0; t < nt; ++t) {
      const int64_t row = r_lo + 128 * t + 32 * a;
      const uint32_t en = cur.en, ev = cur.ev;
      int k = cur.k;
      const float l_next = load_lam(nxt.k);
      cur = nxt;
      nxt = load_rows(t + 2);
      const int left = (int)max((int64_t)0, min((int64_t)16, r_hi - (row + sh)));   // the thread's rows of this CTA
      const bool good = mbar_wait(&bars->tfull[0], (uint32_t)(t & 1), kFuWaitNs) && !aborted(bars);
      if (!__all_sync(0xffffffffu, good)) {   // the whole warp leaves together
        raise_abort(bars, err);
        ok = false;
        break;
      }
      tc::fence_after_sync();
      float eta[16];
      if (busy) {
        float v0[16], v1[16];
        tc::tmem_ld16x2(tq, tq + 16u, v0, v1);
        combine(v0, v1, upper, eta);
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->tempty[0]);
      uint32_t hi[8], lo[8];
      if (busy) {
        float x[16];
        if (__all_sync(0xffffffffu, en == 0u && left == 16)) {   // every thread's rows in one group
#pragma unroll
          for (int u = 0; u < 16; ++u) x[u] = g * (expf(eta[u]) * l - (ev >> u & 1u ? 1.f : 0.f));
        } else {
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const float d = ev >> u & 1u ? 1.f : 0.f;
            x[u] = (has && u < left) ? g * (expf(eta[u]) * l - d) : 0.f;
            if (en >> u & 1u) l = load_lam(++k);   // the next row lies in the next group
          }
        }
#pragma unroll
        for (int u = 0; u < 16; u += 2) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(x[u], x[u + 1]);
          const uint32_t hb = *reinterpret_cast<const uint32_t*>(&h);
          const __nv_bfloat162 m = __floats2bfloat162_rn(x[u] - __uint_as_float(hb << 16),
                                                         x[u + 1] - __uint_as_float(hb & 0xffff0000u));
          hi[u >> 1] = hb;
          lo[u >> 1] = *reinterpret_cast<const uint32_t*>(&m);
        }
      }
      // the previous tile's G has been read (every warp waits: an arrival for
      // this tile must not fall into the previous tile's phase)
      if (t >= 1 && !mbar_wait(&bars->gempty[0], (uint32_t)((t - 1) & 1), kFuWaitNs)) ok = false;
      if (busy) {
        // rows c (high) and 64 + c (low) of the operand tile, 128 bytes = 64
        // subjects each, 16-byte chunks permuted by the row within 8 rows
        unsigned char* gt = sG + (size_t)(a >> 1) * gbytes;
        const int ch = 4 * (a & 1) + (upper ? 2 : 0);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const int rl = 64 + c;
          *reinterpret_cast<uint4*>(gt + c * 128 + (((ch + v) ^ (c & 7)) << 4)) =
              make_uint4(hi[4 * v], hi[4 * v + 1], hi[4 * v + 2], hi[4 * v + 3]);
          *reinterpret_cast<uint4*>(gt + rl * 128 + (((ch + v) ^ (rl & 7)) << 4)) =
              make_uint4(lo[4 * v], lo[4 * v + 1], lo[4 * v + 2], lo[4 * v + 3]);
        }
      }
      if (!__all_sync(0xffffffffu, ok)) {
        raise_abort(bars, err);
        ok = false;
        break;
      }
      tc::fence_proxy_async();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bars->gfull[0]);
      l = l_next;
    }
    // ---------------- the CTA's partial sums: 16 columns in turn for each set
    bool have = ok && nt > 0;
    if (!mbar_wait(&bars->done, 0, 2 * kFuWaitNs) || aborted(bars)) {
      raise_abort(bars, err);
      have = false;
    }
    tc::fence_after_sync();
    // TMEM lane 32 q + lane: part `row` of G; lanes write consecutive columns
    const int row = 32 * q + lane, pc = row & 63;
    const int col = row < 64 ? pc : Cp + pc;
    for (int p0 = 16 * a; p0 < p; p0 += 64) {
      float v[16];
      if (have) {
        tc::tmem_ld16(d2 + ((uint32_t)(32 * q) << 16) + (uint32_t)p0, v);
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = 0.f;
      }
      if (pc < Cp)
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (p0 + i < p) part[((size_t)blockIdx.x * p + p0 + i) * NB + col] = v[i];
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, 512);
  }
}

// B (p x C, row-major FP32) -> the 128 rows of Bcat^T in the order above, ld
// bf16 a row; zeros in the padding rows and columns.
__global__ void k_split_bt16(const float* B, int64_t p, int C, int64_t ld, __nv_bfloat16* BcatT) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 128 * ld) return;
  const int r = (int)(i / ld);
  const int64_t j = i - (int64_t)r * ld;
  const int c = 16 * (r >> 5) + (r & 15);
  __nv_bfloat16 v = __float2bfloat16_rn(0.f);
  if (c < C && j < p) {
    const float b = B[j * C + c];
    const __nv_bfloat16 hi = __float2bfloat16_rn(b);
    v = (r & 16) ? __float2bfloat16_rn(b - __bfloat162float(hi)) : hi;
  }
  BcatT[i] = v;
}

int optin_smem() {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return v;
}

size_t fwd_smem(int nkb, int ns) { return 1024 + (size_t)(nkb + ns) * 2 * kFuBoxBytes + sizeof(FuBars); }
// (at least half of an SM's shared memory: one CTA per SM, since a CTA takes all
// of its tensor memory and a second one would wait for it)
size_t bwd_smem(int nkb, int ns) {
  const size_t b = 1024 + (size_t)ns * nkb * 2 * kFuBoxBytes + 2 * (size_t)128 * 128 + sizeof(FuBars);
  return std::max(b, (size_t)118 * 1024);
}

}  // namespace

bool nll_fused_fits(int64_t n, int p, int C) {
  const int nkb = (p + kFuBoxK - 1) / kFuBoxK;
  const size_t most = (size_t)optin_smem();
  return n <= (int64_t(1) << 30) && nkb <= kFuMaxKb && C <= 64 && fwd_smem(nkb, 4) <= most &&
         bwd_smem(nkb, 3) <= most;
}

int64_t nll_fused_unit_rows(int64_t n, int units) {
  const int64_t per = (n + units - 1) / units;
  return (per + 63) / 64 * 64;
}

cudaError_t nll_fused_split(const float* B, int64_t p, int C, int64_t ld, void* BcatT, cudaStream_t s) {
  k_split_bt16<<<(unsigned)((128 * ld + 255) / 256), 256, 0, s>>>(B, p, C, ld, static_cast<__nv_bfloat16*>(BcatT));
  return cudaGetLastError();
}

cudaError_t nll_fused_forward(const void* X, int64_t n, int p, int64_t ldx, const void* BcatT, int C, int ctas,
                              int64_t ru, const RowMasks& m, const uint32_t* event, float2* rec, float2* wt, float2* wd, unsigned* err,
                              cudaStream_t s) {
  const int nkb = (p + kFuBoxK - 1) / kFuBoxK;
  CUtensorMap mx, mb;
  cudaError_t st = nll_make_map(&mx, X, n, p, ldx, 64);
  if (st == cudaSuccess) st = nll_make_map(&mb, BcatT, 128, p, ldx, 128);
  if (st != cudaSuccess) return st;
  int ns = kFuMaxStages;
  while (ns > 4 && fwd_smem(nkb, ns) > (size_t)optin_smem()) --ns;
  const size_t smem = fwd_smem(nkb, ns);
  st = cudaFuncSetAttribute(k_nll_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (st != cudaSuccess) return st;
  k_nll_fwd<<<ctas, kFuThreads, smem, s>>>(mx, mb, n, nkb, C, ns, ru, m.end, event, m.first, rec, wt, wd, err);
  return cudaGetLastError();
}

cudaError_t nll_fused_backward(const void* X, int64_t n, int p, int64_t ldx, const void* BcatT, int C, int Cp, int K,
                               const RowMasks& m, const uint32_t* event, const float* lam,
                               const double* gout, float* part, int nx,
                               float* grad_B, unsigned* err, cudaStream_t s) {
  const int nkb = (p + kFuBoxK - 1) / kFuBoxK;
  CUtensorMap mx;
  cudaError_t st = nll_make_map(&mx, X, n, p, ldx, 128);
  if (st != cudaSuccess) return st;
  int ns = 6;
  while (ns > 3 && bwd_smem(nkb, ns) > (size_t)optin_smem()) --ns;
  const size_t smem = bwd_smem(nkb, ns);
  st = cudaFuncSetAttribute(k_nll_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (st != cudaSuccess) return st;
  const int64_t per = (n + nx - 1) / nx;
  const int64_t rows_per_cta = (per + 63) / 64 * 64;
  k_nll_bwd<<<nx, kFuBwdThreads, smem, s>>>(mx, static_cast<const uint32_t*>(BcatT), (int)(ldx / 2), n, p, nkb, C, Cp, K, ns, rows_per_cta, m.end, event, m.first, lam,
                                         gout, part, err);
  st = cudaGetLastError();
  return st == cudaSuccess ? nll_xtg_reduce(part, nx, p, 2 * Cp, C, Cp, grad_B, s) : st;
}

}  // namespace survgpu
