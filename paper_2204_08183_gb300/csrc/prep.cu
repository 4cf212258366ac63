// Once-per-fit preparation kernels (the "precomputed" parts of Section 2.7):
// input validation, the Breslow tie-group table (group ends e_k and event
// counts d_k), the Kaplan-Meier censoring survival G(t_k) and the competing
// weights W_r = I(status_r = 2) / G(y_r) (Section 2.2), delta^T X_j (the
// constant first term of Eq. cox_g), the warp/row partition tables of the
// persistent kernel, and eta = X beta for a warm start.
//
// Integer work (ends, counts) is exact; G(t_k) is a sequential FP64 product
// from the smallest time upward in a single thread, so its rounding follows
// one fixed order.
#include <algorithm>
#include <climits>
#include <cuda_bf16.h>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace survgpu {
namespace {

constexpr int kPrepThreads = 256;

inline unsigned grid_for(int64_t count, int threads, unsigned cap = 65535u * 32u) {
  int64_t g = (count + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > (int64_t)cap) g = cap;
  return (unsigned)g;
}

// Blocks of a column of `len` stored values: contiguous chunks of at least
// kColChunk, at most kMaxColBlocks (a partial sum each).
constexpr int kColThreads = 256;
constexpr int kColChunk = 4096;
constexpr int kMaxColBlocks = 512;

// Partial sum of one block in a fixed order (thread 0 stores it).
template <typename A>
__device__ __forceinline__ void block_partial(A v, A* dst) {
  __shared__ A s_w[kColThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) s_w[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    A a = s_w[0];
    for (int q = 1; q < kColThreads / 32; ++q) a = acc_add(a, s_w[q]);
    *dst = a;
  }
}

// One pass over the stored entries of CSC column blockIdx.y: row indices in
// range and increasing, values finite and (flag) all 1.  With FULL it also
// leaves the block's share of delta^T X_j in part[j][blockIdx.x] and the
// column's offsets at the warps' first rows in woff[j][.]: entry i is the
// first at or after the first row of every warp after its predecessor's
// warp, up to its own.  A thread takes 4 consecutive entries (16-byte loads of
// the indices and values), so neighbours are compared in registers, and looks
// for a warp boundary once per 4: rows increase, so without one between the
// entry before and the last there is none inside.  Values of 1 are counted
// instead of added.  Whether a row is an event comes from a bit per subject: a
// column at 5 % touches most sectors of the status bytes, 0.8 GB through L2
// for 100 columns of 10^7 subjects (197 us with them; one entry at a time
// 222; three separate passes before that 248).  Four whole entries of 1, nearly all
// of an indicator column, are checked together (a lambda_max call at 10^6 x 500:
// 166 us with every entry checked by itself, 159).
template <typename T, bool FULL>
__global__ void __launch_bounds__(kColThreads) k_check_csc(const int64_t* col_ptr, const int32_t* row_idx,
                                                           const T* values, int64_t p, int64_t n,
                                                           const uint32_t* event, int32_t nwarps, uint32_t wpw,
                                                           typename AccOf<T>::type* part, int32_t* woff,
                                                           unsigned* perr) {
  using A = typename AccOf<T>::type;
  constexpr int U = 2;
  const int lane = threadIdx.x & 31;
  const float inv_wpw = 1.f / (float)wpw;
  const bool vec = (((uintptr_t)row_idx | (uintptr_t)values) & 15) == 0;
  unsigned bits = 0;
  for (int64_t j = blockIdx.y; j < p; j += gridDim.y) {
    const int64_t a = col_ptr[j], b = col_ptr[j + 1];
    A acc;
    acc_zero(acc);
    int ones = 0;
    // the warp that holds row r: r / 32 / wpw by a float quotient, corrected
    auto warp_of = [&](int32_t r) {
      const uint32_t x = (uint32_t)r >> 5;
      uint32_t q = (uint32_t)((float)x * inv_wpw);
      const int32_t rem = (int32_t)(x - q * wpw);
      if (rem < 0) --q;
      else if (rem >= (int32_t)wpw) ++q;
      return (int32_t)q;
    };
    int32_t* wo = FULL ? woff + j * (nwarps + 1) : nullptr;
    if (FULL && blockIdx.x == 0 && a == b)
      for (int g = threadIdx.x; g <= nwarps; g += kColThreads) wo[g] = 0;
    // entries 4 q .. 4 q + 3 of the array per thread, those inside [a, b)
    const int64_t qa = a >> 2, qb = a < b ? (b + 3) >> 2 : qa;
    // whole rounds of U x kColThreads quads per block (every lane takes part)
    for (int64_t q0 = qa + (int64_t)blockIdx.x * (U * kColThreads); q0 < qb; q0 += (int64_t)gridDim.x * (U * kColThreads)) {
      int32_t r[U][4], rp[U];
      T v[U][4];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t i = (q0 + u * kColThreads + threadIdx.x) * 4;
        if (vec && i >= a && i + 4 <= b) {
          const int4 t = __ldcs(reinterpret_cast<const int4*>(row_idx + i));
          r[u][0] = t.x, r[u][1] = t.y, r[u][2] = t.z, r[u][3] = t.w;
          if (values) {
            if constexpr (sizeof(T) == 4) {
              const float4 f = __ldcs(reinterpret_cast<const float4*>(values + i));
              v[u][0] = f.x, v[u][1] = f.y, v[u][2] = f.z, v[u][3] = f.w;
            } else {
              const double2 f = __ldcs(reinterpret_cast<const double2*>(values + i));
              const double2 g = __ldcs(reinterpret_cast<const double2*>(values + i + 2));
              v[u][0] = f.x, v[u][1] = f.y, v[u][2] = g.x, v[u][3] = g.y;
            }
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[u][e] = T(1);
          }
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const bool in = i + e >= a && i + e < b;
            r[u][e] = in ? row_idx[i + e] : -1;
            v[u][e] = (values && in) ? values[i + e] : T(1);
          }
        }
        rp[u] = (lane == 0 && i > a && i < b) ? row_idx[i - 1] : -1;
      }
      uint32_t st[U][4];
      if (FULL) {
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int e = 0; e < 4; ++e) st[u][e] = (uint32_t)r[u][e] < (uint32_t)n ? event[r[u][e] >> 5] : 0u;   // n < 2^31
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t i = (q0 + u * kColThreads + threadIdx.x) * 4;
        const int32_t up = __shfl_up_sync(0xffffffffu, r[u][3], 1);
        const int32_t before = lane == 0 ? rp[u] : up;   // entry i - 1 (if it is one of the column's)
        bool good = true;
        int32_t prev = before, last = -1;
        const bool whole = i >= a && i + 4 <= b;
        bool one = whole;
        if (values)
#pragma unroll
          for (int e = 0; e < 4; ++e) one = one && v[u][e] == T(1);
        if (one) {
          // four of the column's entries, all 1: rising from row 0 or later to
          // a row before n is all there is to check
          last = r[u][3];
          good = r[u][0] >= 0 && last < (int32_t)n && r[u][0] < r[u][1] && r[u][1] < r[u][2] && r[u][2] < last &&
                 (i == a || before < r[u][0]);
          if (FULL)
#pragma unroll
            for (int e = 0; e < 4; ++e) ones += (int)(st[u][e] >> (r[u][e] & 31) & 1u);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (one || i + e < a || i + e >= b) continue;
          if (r[u][e] < 0 || r[u][e] >= n || (i + e > a && prev >= r[u][e])) good = false;
          prev = last = r[u][e];
          if (values) {
            if (!isfinite(v[u][e])) bits |= PREP_NONFINITE;
            if (v[u][e] != T(1)) bits |= PREP_VALUES_NOT_ONE;
          }
          if (FULL && (st[u][e] >> (r[u][e] & 31) & 1u)) {
            if (v[u][e] == T(1)) ++ones;
            else acc = acc_add_v(acc, v[u][e]);
          }
        }
        if (!good) bits |= PREP_INDEX;
        if (FULL && good && last >= 0 && (i <= a || before >= 0)) {
          int32_t g0 = i > a ? warp_of(before) + 1 : 0;   // the first warp without its offset
          const int32_t g1 = warp_of(last);
          if (g0 <= g1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              if (i + e < a || i + e >= b) continue;
              const int32_t ge = warp_of(r[u][e]);
              for (; g0 <= ge; ++g0) wo[g0] = (int32_t)(i + e - a);
            }
          }
          if (i + 4 >= b)   // the column's last entry
            for (int32_t g = g1 + 1; g <= nwarps; ++g) wo[g] = (int32_t)(b - a);
        }
      }
    }
    if (FULL) {
      __syncthreads();   // the previous column's partial has been read
      block_partial<A>(acc_add_v(acc, (T)ones), part + j * gridDim.x + blockIdx.x);
    }
  }
  if (bits) atomicOr(perr, bits);
}

// Dense column blockIdx.y: finite values and, with part, the block's share of
// delta^T X_j.  Four rows a load (16 bytes of FP32) where base and pitch
// allow it.  Bound by the bytes of X; one block per column left two thirds
// of the chip idle (1.2 ms for 1 GB of 50 columns, after a check pass of
// 0.45 ms with a 64-bit division per element).
template <typename T>
__global__ void __launch_bounds__(kColThreads) k_check_dense(const T* X, int64_t ld, int64_t n, int64_t p,
                                                             const int8_t* status, typename AccOf<T>::type* part,
                                                             unsigned* perr) {
  using A = typename AccOf<T>::type;
  constexpr int U = 4;
  unsigned bits = 0;
  const bool vec = (((uintptr_t)X & 15) | ((uintptr_t)(ld * sizeof(T)) & 15) | ((uintptr_t)status & 3)) == 0;
  const int64_t quads = (n + 3) >> 2;
  for (int64_t j = blockIdx.y; j < p; j += gridDim.y) {
    const T* x = X + j * ld;
    A acc;
    acc_zero(acc);
    for (int64_t q0 = (int64_t)blockIdx.x * (U * kColThreads) + threadIdx.x; q0 < quads;
         q0 += (int64_t)gridDim.x * (U * kColThreads)) {
      T v[U][4];
      uint32_t st[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t i = (q0 + u * kColThreads) * 4;
        st[u] = 0;
        if (vec && i + 4 <= n) {
          if constexpr (sizeof(T) == 4) {
            const float4 f = __ldcs(reinterpret_cast<const float4*>(x + i));
            v[u][0] = f.x, v[u][1] = f.y, v[u][2] = f.z, v[u][3] = f.w;
          } else {
            const double2 f = __ldcs(reinterpret_cast<const double2*>(x + i));
            const double2 g = __ldcs(reinterpret_cast<const double2*>(x + i + 2));
            v[u][0] = f.x, v[u][1] = f.y, v[u][2] = g.x, v[u][3] = g.y;
          }
          if (part) st[u] = *reinterpret_cast<const uint32_t*>(status + i);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            v[u][e] = i + e < n ? x[i + e] : T(0);
            if (part && i + e < n) st[u] |= (uint32_t)(uint8_t)status[i + e] << (8 * e);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (!isfinite(v[u][e])) bits |= PREP_NONFINITE;
          if ((st[u] >> (8 * e) & 255u) == 1u) acc = acc_add_v(acc, v[u][e]);
        }
    }
    if (part) {
      __syncthreads();
      block_partial<A>(acc, part + j * gridDim.x + blockIdx.x);
    }
  }
  if (bits) atomicOr(perr, bits);
}

// delta^T X_j from its nb partial sums (one warp a column, fixed order), and
// the initial trust-region width.
template <typename A>
__global__ void __launch_bounds__(kColThreads) k_coord_init(const A* part, int nb, int64_t p, double* dTx,
                                                            double* width) {
  const int lane = threadIdx.x & 31;
  const int64_t j = ((int64_t)blockIdx.x * kColThreads + threadIdx.x) >> 5;
  if (j >= p) return;   // the whole warp
  A a;
  acc_zero(a);
  for (int q = lane; q < nb; q += 32) a = acc_add(a, part[j * nb + q]);
  a = warp_sum(a);
  if (lane == 0) {
    dTx[j] = acc_to_d(a);
    width[j] = 1.0;
  }
}

__global__ void k_check_finite(const double* v, int64_t count, unsigned* perr) {
  unsigned bits = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    if (!isfinite(v[i])) bits |= PREP_NONFINITE;
  if (bits) atomicOr(perr, bits);
}

// --- tie groups: i is a group end iff i == n-1 or time[i] != time[i+1].
//
// Two streaming passes over the times and status codes (5 bytes a subject),
// bound by memory at large n and by their launch at small n.  k_group_count
// checks both arrays and counts, per block of kGrpRows subjects, the group
// ends, events (status 1) and censored (status 0); its last block (ticket)
// scans the block counts.  k_group_write takes each row's prefix from them
// and writes the table.  A lane owns 4 consecutive rows (one 16-byte and one
// 4-byte load), a warp 4 rounds of 128 rows; the three counts of a warp
// (at most 512 each) travel in one word of three 10-bit fields, so one
// shuffle scan serves all of them.
//
// Counts per group come from the prefix counts at the group ends: end k adds
// its prefix to d_k and takes it from d_{k+1} (integer atomics, exact in any
// order), so the work does not depend on how the subjects are spread over the
// groups.  (One warp per 2048 subjects walking its group segments one after
// another took 728 us for 333,331 subjects with hardly any ties and 107 us
// for 100,003, where few warps ran; without it a fit of the former takes
// 21.82 instead of 22.54 ms and one evaluation of the latter 249 instead of
// 380 us.)
constexpr int kGrpThreads = 256;
constexpr int kGrpRounds = 4;
constexpr int kGrpRows = kGrpThreads * 4 * kGrpRounds;
static_assert(kGrpRows == kGroupRows, "rows of a block");

struct RowQuad {
  unsigned end, ev, ce, bad;   // 4-bit masks of the quad's rows; prep error bits
};

// Times and status codes of rows i .. i + 3 (those below n), and for lane 31
// the time after them.
struct RawQuad {
  int32_t t[5];
  uint32_t st;
};
__device__ __forceinline__ RawQuad load_raw(const int32_t* time, const int8_t* status, int64_t n, int64_t i, bool vec) {
  RawQuad q = {{0, 0, 0, 0, 0}, 0u};
  if (vec && i + 4 <= n) {
    const int4 v = *reinterpret_cast<const int4*>(time + i);
    q.t[0] = v.x, q.t[1] = v.y, q.t[2] = v.z, q.t[3] = v.w;
    q.st = *reinterpret_cast<const uint32_t*>(status + i);
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u < n) {
        q.t[u] = time[i + u];
        q.st |= (uint32_t)(uint8_t)status[i + u] << (8 * u);
      }
  }
  if ((threadIdx.x & 31) == 31 && i + 4 < n) q.t[4] = time[i + 4];
  return q;
}
// Their flags.  Every lane of the warp takes part.
__device__ __forceinline__ RowQuad quad_flags(const RawQuad& q, int64_t n, int64_t i, int max_status) {
  const int lane = threadIdx.x & 31;
  int32_t t[5] = {q.t[0], q.t[1], q.t[2], q.t[3], 0};
  const uint32_t st = q.st;
  t[4] = __shfl_down_sync(0xffffffffu, t[0], 1);
  if (lane == 31) t[4] = q.t[4];
  RowQuad r = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (i + u >= n) continue;
    const bool last = i + u == n - 1;
    if (last || t[u] != t[u + 1]) r.end |= 1u << u;
    if (!last && t[u] < t[u + 1]) r.bad |= PREP_UNSORTED;
    const int sv = (int)(int8_t)(st >> (8 * u));
    if (sv == 1) r.ev |= 1u << u;
    if (sv == 0) r.ce |= 1u << u;
    if (sv < 0 || sv > max_status) r.bad |= PREP_STATUS;
  }
  return r;
}
__device__ __forceinline__ unsigned quad_counts(const RowQuad& r) {
  return (unsigned)__popc(r.end) | (unsigned)__popc(r.ev) << 10 | (unsigned)__popc(r.ce) << 20;
}
// The masks of 8 lanes as one word of 32 rows (in each of them).
__device__ __forceinline__ uint32_t word_of(unsigned nibble) {
  uint32_t w = nibble << (4 * (threadIdx.x & 7));
#pragma unroll
  for (int d = 1; d < 8; d <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, d);
  return w;
}
// 16-byte loads of the times and 4-byte loads of the status codes
__device__ __forceinline__ bool quad_aligned(const int32_t* time, const int8_t* status) {
  return (((uintptr_t)time & 15) | ((uintptr_t)status & 3)) == 0;
}

// cnt [3][nb]: exclusive prefixes over the blocks of ends, events and
// censored on exit.  *ticket is zero on entry and on exit.  crowd (if given):
// the most ends among 32 and among kGrpRows rows.
__global__ void __launch_bounds__(kGrpThreads) k_group_count(const int32_t* time, const int8_t* status, int64_t n,
                                                             int model, int64_t nb, int32_t* cnt, unsigned* perr,
                                                             int32_t* K, int32_t* total_events, unsigned* ticket,
                                                             uint32_t* event, int32_t* crowd) {
  __shared__ unsigned s_w[kGrpThreads / 32];
  __shared__ int32_t s_p[3][kGrpThreads / 32];
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool vec = quad_aligned(time, status);
  const int64_t r0 = (int64_t)blockIdx.x * kGrpRows + w * (128 * kGrpRounds) + lane * 4;
  unsigned c = 0, bad = 0, most = 0;
  RawQuad raw[kGrpRounds];
#pragma unroll
  for (int it = 0; it < kGrpRounds; ++it) raw[it] = load_raw(time, status, n, r0 + 128 * it, vec);
#pragma unroll
  for (int it = 0; it < kGrpRounds; ++it) {
    const RowQuad q = quad_flags(raw[it], n, r0 + 128 * it, model == 1 ? 2 : 1);
    c += quad_counts(q);
    bad |= q.bad;
    if (event) {
      const uint32_t ev = word_of(q.ev);
      if ((lane & 7) == 0 && r0 + 128 * it < n) event[(r0 + 128 * it) >> 5] = ev;
    }
    if (crowd) most = max(most, (unsigned)__popc(word_of(q.end)));
  }
  if (bad) atomicOr(perr, bad);
  c = __reduce_add_sync(0xffffffffu, c);
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 0) {
    s_w[w] = c;
    s_p[0][w] = (int32_t)most;
  }
  __syncthreads();
  if (crowd && tid == 32) {
    for (int q = 0; q < kGrpThreads / 32; ++q) most = max(most, (unsigned)s_p[0][q]);
    atomicMax(crowd, (int32_t)most);
  }
  if (tid < 3) {
    int32_t v = 0;
    for (int q = 0; q < kGrpThreads / 32; ++q) v += (int32_t)(s_w[q] >> (10 * tid) & 1023u);
    cnt[tid * nb + blockIdx.x] = v;
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) {
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  // last block: contiguous chunks of block counts per thread, chunk sums
  // scanned over the block, the chunks walked again
  const int64_t per = (nb + kGrpThreads - 1) / kGrpThreads;
  const int64_t lo = min((int64_t)tid * per, nb), hi = min(lo + per, nb);
  constexpr int kKeep = 12;   // counts kept in registers (12.6 million subjects)
  int32_t keep[3][kKeep], sum[3] = {0, 0, 0};
#pragma unroll
  for (int q = 0; q < kKeep; ++q)
#pragma unroll
    for (int m = 0; m < 3; ++m) keep[m][q] = lo + q < hi ? __ldcg(cnt + m * nb + lo + q) : 0;
#pragma unroll
  for (int q = 0; q < kKeep; ++q)
#pragma unroll
    for (int m = 0; m < 3; ++m) sum[m] += keep[m][q];
  for (int64_t b = lo + kKeep; b < hi; ++b)
#pragma unroll
    for (int m = 0; m < 3; ++m) sum[m] += __ldcg(cnt + m * nb + b);
  if (crowd) {   // the most ends of a block
    int32_t top = 0;
#pragma unroll
    for (int q = 0; q < kKeep; ++q) top = max(top, keep[0][q]);
    for (int64_t b = lo + kKeep; b < hi; ++b) top = max(top, __ldcg(cnt + b));
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) atomicMax(crowd + 1, top);
  }
  int32_t inc[3] = {sum[0], sum[1], sum[2]};
#pragma unroll
  for (int d = 1; d < 32; d <<= 1)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int32_t v = __shfl_up_sync(0xffffffffu, inc[m], d);
      if (lane >= d) inc[m] += v;
    }
  if (lane == 31)
#pragma unroll
    for (int m = 0; m < 3; ++m) s_p[m][w] = inc[m];
  __syncthreads();
  int32_t run[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    run[m] = inc[m] - sum[m];
    for (int q = 0; q < w; ++q) run[m] += s_p[m][q];
  }
#pragma unroll
  for (int q = 0; q < kKeep; ++q)
    if (lo + q < hi)
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        cnt[m * nb + lo + q] = run[m];
        run[m] += keep[m][q];
      }
  for (int64_t b = lo + kKeep; b < hi; ++b)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int32_t v = __ldcg(cnt + m * nb + b);
      cnt[m * nb + b] = run[m];
      run[m] += v;
    }
  if (tid == kGrpThreads - 1) {   // its chunk ends at nb (or is empty): the totals
    *K = run[0];
    *total_events = run[1];
    *ticket = 0u;
  }
}

// gend, and dk and ck (zeroed before; ck may be null); with wk0, also the
// first group whose end is at or after each warp's first row (warp g starts
// at row g * rpw, rpw a multiple of 32): the number of ends before that row.
__global__ void __launch_bounds__(kGrpThreads) k_group_write(const int32_t* time, const int8_t* status, int64_t n,
                                                             int64_t nb, const int32_t* cnt, int32_t K, int32_t* gend,
                                                             int32_t* dk, int32_t* ck, int32_t nwarps, int64_t rpw,
                                                             int32_t* wk0, RowMasks masks) {
  __shared__ unsigned s_w[kGrpThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool vec = quad_aligned(time, status);
  const int64_t r0 = (int64_t)blockIdx.x * kGrpRows + w * (128 * kGrpRounds) + lane * 4;
  RawQuad raw[kGrpRounds];
  RowQuad q[kGrpRounds];
  unsigned c = 0;
#pragma unroll
  for (int it = 0; it < kGrpRounds; ++it) raw[it] = load_raw(time, status, n, r0 + 128 * it, vec);
#pragma unroll
  for (int it = 0; it < kGrpRounds; ++it) {
    q[it] = quad_flags(raw[it], n, r0 + 128 * it, 2);
    c += quad_counts(q[it]);
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) s_w[w] = c;
  __syncthreads();
  int32_t base[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    base[m] = cnt[m * nb + blockIdx.x];
    for (int v = 0; v < w; ++v) base[m] += (int32_t)(s_w[v] >> (10 * m) & 1023u);
  }
  unsigned before = 0;  // counts of the warp's earlier rounds
#pragma unroll
  for (int it = 0; it < kGrpRounds; ++it) {
    const unsigned mine = quad_counts(q[it]);
    unsigned incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned v = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += v;
    }
    const unsigned ex = before + incl - mine;
    before += __shfl_sync(0xffffffffu, incl, 31);
    const int64_t i0 = r0 + 128 * it;
    int32_t k = base[0] + (int32_t)(ex & 1023u);
    const int32_t e0 = base[1] + (int32_t)(ex >> 10 & 1023u), c0 = base[2] + (int32_t)(ex >> 20);
    if (wk0 && (lane & 7) == 0 && i0 < n && (uint32_t)i0 % (uint32_t)rpw == 0)
      wk0[(uint32_t)i0 / (uint32_t)rpw] = k;
    if (masks.end) {
      const uint32_t en = word_of(q[it].end);
      if ((lane & 7) == 0 && i0 < n) {
        masks.end[i0 >> 5] = en;
        masks.first[i0 >> 5] = k;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (q[it].end >> u & 1u) {
        const unsigned upto = (2u << u) - 1u;
        gend[k] = (int32_t)(i0 + u);
        const int32_t e = e0 + __popc(q[it].ev & upto), cc = c0 + __popc(q[it].ce & upto);
        if (e) {
          atomicAdd(dk + k, e);
          if (k + 1 < K) atomicSub(dk + k + 1, e);
        }
        if (ck && cc) {
          atomicAdd(ck + k, cc);
          if (k + 1 < K) atomicSub(ck + k + 1, cc);
        }
        ++k;
      }
  }
  if (wk0 && blockIdx.x == 0)   // warps that start at or after row n
    for (int64_t g = (n + rpw - 1) / rpw + tid; g <= nwarps; g += kGrpThreads) wk0[g] = K;
}

// Kaplan-Meier censoring survival (Section 2.2):
//   G(t_k) = prod_{k' >= k} f_k',  f_k' = 1 - c_k' / n_k',  n_k' = e_k' + 1
// (groups k' >= k have t_k' <= t_k).  The factors are independent: one
// thread each (k_km_factor writes them into Gk).  The product is ordered:
// up to kKmSerial groups one thread multiplies them in the order of the
// definition, k = K - 1 down to 0, exactly as a sequential loop does; above
// that the groups are cut into 1024 contiguous chunks, each thread forms
// its chunk's product, a fixed-shape suffix scan over the chunks gives each
// chunk the product of the chunks after it, and each thread walks its chunk
// downward from there.  That order is fixed (the result does not depend on
// timing) and keeps the relative error below (2 L + 12) u, L = ceil(K /
// 1024), against (K - 1) u for the sequential product.
constexpr int kKmSerial = 4096;
constexpr int kKmThreads = 1024;

__global__ void k_km_factor(const int32_t* gend, const int32_t* ck, int32_t K, double* f) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < K; k += (int64_t)gridDim.x * blockDim.x)
    f[k] = 1.0 - (double)ck[k] / (double)((int64_t)gend[k] + 1);
}

// Gk holds the factors on entry and G(t_k) on exit (one block).  The ordered
// product is a chain of dependent FP64 multiplications by one thread, so its
// operands come from shared memory, eight ahead of their use, and nothing
// else stands in the chain (out of global memory, with the float-float copies
// written on the way, 1000 groups took 225 us and 3,650 groups 318).
__global__ void __launch_bounds__(kKmThreads) k_km_product(int32_t K, double* Gk) {
  if (K <= kKmSerial) {
    __shared__ double s_f[kKmSerial];
    for (int k = threadIdx.x; k < K; k += kKmThreads) s_f[k] = Gk[k];
    __syncthreads();
    if (threadIdx.x == 0) {
      double acc = 1.0;
      int k = K - 1;
      double f[8];
      if (k >= 7) {
#pragma unroll
        for (int u = 0; u < 8; ++u) f[u] = s_f[k - u];
      }
      for (; k >= 7; k -= 8) {
        double nx[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) nx[u] = k - 8 - u >= 0 ? s_f[k - 8 - u] : 1.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          acc = acc * f[u];
          s_f[k - u] = acc;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) f[u] = nx[u];
      }
      for (; k >= 0; --k) {
        acc = acc * s_f[k];
        s_f[k] = acc;
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += kKmThreads) Gk[k] = s_f[k];
    return;
  }
  __shared__ double s_w[32];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int64_t L = ((int64_t)K + kKmThreads - 1) / kKmThreads;
  const int64_t a = min((int64_t)t * L, (int64_t)K), b = min(a + L, (int64_t)K);
  double v = 1.0;
  for (int64_t k = b - 1; k >= a; --k) v = v * Gk[k];
  // inclusive suffix products over the lanes, then over the warps
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double u = __shfl_down_sync(0xffffffffu, v, d);
    if (lane + d < 32) v = v * u;
  }
  if (lane == 0) s_w[w] = v;
  __syncthreads();
  if (w == 0) {
    double q = s_w[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const double u = __shfl_down_sync(0xffffffffu, q, d);
      if (lane + d < 32) q = q * u;
    }
    __syncwarp();
    s_w[lane] = q;
  }
  __syncthreads();
  double in_warp = __shfl_down_sync(0xffffffffu, v, 1);
  if (lane == 31) in_warp = 1.0;
  const double later_warps = w < 31 ? s_w[w + 1] : 1.0;
  double acc = later_warps * in_warp;   // product of the chunks after this one
  for (int64_t k = b - 1; k >= a; --k) {
    acc = acc * Gk[k];
    Gk[k] = acc;
  }
}

// G(t_k) as float-float and 1 / G(t_k) in the working precision.
template <typename T>
__global__ void k_km_finish(int32_t K, const double* Gk, float2* Gkff, T* inv) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < K; k += (int64_t)gridDim.x * blockDim.x) {
    const ff q = d_to_ff(Gk[k]);
    Gkff[k] = make_float2(q.hi, q.lo);
    inv[k] = (T)(1.0 / Gk[k]);
  }
}

// W_r = I(status_r = 2) / G(y_r), rows in the blocks of k_group_count (a
// row's group is the number of group ends before it): 5 bytes read and one
// value written a subject, whatever the group sizes.  (A warp per group left
// the largest of 1000 groups to one warp: 384 us for 5 x 10^6 subjects.)
template <typename T>
__global__ void __launch_bounds__(kGrpThreads) k_w2(const int32_t* time, const int8_t* status, int64_t n, int64_t nb,
                                                    const int32_t* cnt, const T* inv, T* w2) {
  __shared__ unsigned s_w[kGrpThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool vec = quad_aligned(time, status);
  const int64_t r0 = (int64_t)blockIdx.x * kGrpRows + w * (128 * kGrpRounds) + lane * 4;
  RawQuad raw[kGrpRounds];
  RowQuad q[kGrpRounds];
  unsigned c = 0;
#pragma unroll
  for (int it = 0; it < kGrpRounds; ++it) raw[it] = load_raw(time, status, n, r0 + 128 * it, vec);
#pragma unroll
  for (int it = 0; it < kGrpRounds; ++it) {
    q[it] = quad_flags(raw[it], n, r0 + 128 * it, 2);
    c += (unsigned)__popc(q[it].end);
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) s_w[w] = c;
  __syncthreads();
  int32_t k0 = cnt[blockIdx.x];
  for (int v = 0; v < w; ++v) k0 += (int32_t)s_w[v];
#pragma unroll
  for (int it = 0; it < kGrpRounds; ++it) {
    const int mine = __popc(q[it].end);
    int incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += v;
    }
    int32_t k = k0 + incl - mine;
    k0 += __shfl_sync(0xffffffffu, incl, 31);
    const int64_t i0 = r0 + 128 * it;
    T v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool comp = i0 + u < n && !((q[it].ev | q[it].ce) >> u & 1u);   // status 2 (0 and 1 are the others)
      v[u] = comp ? inv[k] : T(0);
      k += (int)(q[it].end >> u & 1u);
    }
    if (i0 + 4 <= n) {   // w2 is the library's own, 256-byte aligned
      if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4*>(w2 + i0) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
        *reinterpret_cast<double2*>(w2 + i0) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2*>(w2 + i0 + 2) = make_double2(v[2], v[3]);
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < n) w2[i0 + u] = v[u];
    }
  }
}

// first group whose end is at or after the warp's first row
__global__ void k_warp_groups(const int32_t* gend, int32_t K, int64_t n, int32_t nwarps, int64_t rows_per_warp,
                              int32_t* wk0) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g > nwarps) return;
  int64_t R = g * rows_per_warp;
  if (R > n) R = n;
  int64_t lo = 0, hi = K;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)gend[mid] < R) lo = mid + 1; else hi = mid;
  }
  wk0[g] = (int32_t)lo;
}

// entry offset (relative to col_ptr[j]) of the first nonzero at or after
// each warp's first row
__global__ void k_warp_offsets(const int64_t* col_ptr, const int32_t* row_idx, int64_t p, int64_t n,
                               int32_t nwarps, int64_t rows_per_warp, int32_t* woff) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t nw1 = (int64_t)nwarps + 1;
  if (t >= p * nw1) return;
  const int64_t j = t / nw1, g = t - j * nw1;
  int64_t R = g * rows_per_warp;
  if (R > n) R = n;
  const int64_t a = col_ptr[j], b = col_ptr[j + 1];
  int64_t lo = 0, hi = b - a;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)row_idx[a + mid] < R) lo = mid + 1; else hi = mid;
  }
  woff[t] = (int32_t)lo;
}

// eta (float-float or double) and e = exp(eta)
__device__ __forceinline__ void eta_store(float2* eta, float* e, int64_t i, ff v) {
  eta[i] = make_float2(v.hi, v.lo);
  const float ev = expf(v.hi);
  e[i] = fmaf(ev, v.lo, ev);
}
__device__ __forceinline__ void eta_store(double* eta, double* e, int64_t i, double v) {
  eta[i] = v;
  e[i] = exp(v);
}

template <typename T>
__global__ void k_eta_dense(const T* X, int64_t ld, int64_t n, int64_t p, const double* beta, void* eta, T* e) {
  using A = typename AccOf<T>::type;
  using E = typename std::conditional<sizeof(T) == 4, float2, double>::type;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    A v;
    acc_zero(v);
    for (int64_t j = 0; j < p; ++j) {
      const double b = beta[j];
      if (b == 0.0) continue;
      if constexpr (sizeof(T) == 4) v = ff_add(v, ff_mul_f(d_to_ff(b), X[j * ld + i]));
      else v = v + X[j * ld + i] * b;
    }
    eta_store(reinterpret_cast<E*>(eta), e, i, v);
  }
}

template <typename T>
__global__ void k_eta_zero(int64_t n, void* eta, T* e) {
  using E = typename std::conditional<sizeof(T) == 4, float2, double>::type;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if constexpr (sizeof(T) == 4) reinterpret_cast<E*>(eta)[i] = make_float2(0.f, 0.f);
    else reinterpret_cast<E*>(eta)[i] = 0.0;
    e[i] = T(1);
  }
}

template <typename T>
__global__ void k_eta_axpy_csc(const int32_t* rows, const T* vals, int64_t nnz, double delta, void* eta) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nnz; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = rows[i];
    const T x = vals ? vals[i] : T(1);
    if constexpr (sizeof(T) == 4) {
      float2* et = reinterpret_cast<float2*>(eta);
      const float2 q = et[r];
      const ff v = ff_add({q.x, q.y}, ff_mul_f(d_to_ff(delta), x));
      et[r] = make_float2(v.hi, v.lo);
    } else {
      double* et = reinterpret_cast<double*>(eta);
      et[r] = et[r] + x * delta;
    }
  }
}

template <typename T>
__global__ void k_eta_exp(int64_t n, const void* eta, T* e) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if constexpr (sizeof(T) == 4) {
      const float2 q = reinterpret_cast<const float2*>(eta)[i];
      const float ev = expf(q.x);
      e[i] = fmaf(ev, q.y, ev);
    } else {
      e[i] = exp(reinterpret_cast<const double*>(eta)[i]);
    }
  }
}

__global__ void k_fill_f64(double* v, double value, int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    v[i] = value;
}

template <typename D, typename S>
__device__ __forceinline__ D to_wide(S v) { return (D)v; }
template <>
__device__ __forceinline__ float to_wide<float, __nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ double to_wide<double, __nv_bfloat16>(__nv_bfloat16 v) { return (double)__bfloat162float(v); }

// column blockIdx.y of a dense matrix, widened to the working precision and
// padded to the pitch ld with zeros
template <typename S, typename D>
__global__ void k_convert_dense(const S* src, int64_t n, int64_t p, D* dst, int64_t ld) {
  constexpr int U = 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = blockIdx.y; j < p; j += gridDim.y) {
    const S* x = src + j * n;
    D* y = dst + j * ld;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < ld; i0 += U * stride) {
      D v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t i = i0 + u * stride;
        v[u] = i < n ? to_wide<D>(x[i]) : D(0);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * stride < ld) y[i0 + u * stride] = v[u];
    }
  }
}

template <typename S, typename D>
__global__ void k_convert_vec(const S* src, int64_t count, D* dst) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x)
    dst[t] = (D)src[t];
}

}  // namespace

int prep_col_blocks(int64_t longest, int64_t p) {
  const int64_t most = std::max<int64_t>(1, std::min<int64_t>(kMaxColBlocks, 65536 / std::max<int64_t>(1, p)));
  return (int)std::max<int64_t>(1, std::min<int64_t>(most, (longest + kColChunk - 1) / kColChunk));
}

cudaError_t prep_check_csc(const int64_t* col_ptr, const int32_t* row_idx, const void* values, int prec, int64_t p,
                           int64_t n, int nb, const PrepColumns* out, unsigned* perr, cudaStream_t s) {
  if (p <= 0) return cudaSuccess;
  const dim3 grid((unsigned)nb, (unsigned)(p < 65535 ? p : 65535));
  const PrepColumns o = out ? *out : PrepColumns{};
  const uint32_t wpw = (uint32_t)std::max<int64_t>(1, o.rows_per_warp / 32);
  if (prec == 0) {
    auto k = out ? k_check_csc<float, true> : k_check_csc<float, false>;
    k<<<grid, kColThreads, 0, s>>>(col_ptr, row_idx, (const float*)values, p, n, o.event, o.nwarps, wpw, (ff*)o.part,
                                   o.woff, perr);
  } else {
    auto k = out ? k_check_csc<double, true> : k_check_csc<double, false>;
    k<<<grid, kColThreads, 0, s>>>(col_ptr, row_idx, (const double*)values, p, n, o.event, o.nwarps, wpw,
                                   (double*)o.part, o.woff, perr);
  }
  return cudaGetLastError();
}

cudaError_t prep_check_dense(const void* X, int prec, int64_t ld, int64_t n, int64_t p, int nb,
                             const PrepColumns* out, unsigned* perr, cudaStream_t s) {
  if (n <= 0 || p <= 0) return cudaSuccess;
  const dim3 grid((unsigned)nb, (unsigned)(p < 65535 ? p : 65535));
  const int8_t* status = out ? out->status : nullptr;
  void* part = out ? out->part : nullptr;
  if (prec == 0) k_check_dense<float><<<grid, kColThreads, 0, s>>>((const float*)X, ld, n, p, status, (ff*)part, perr);
  else k_check_dense<double><<<grid, kColThreads, 0, s>>>((const double*)X, ld, n, p, status, (double*)part, perr);
  return cudaGetLastError();
}

cudaError_t prep_coord_init(const void* part, int prec, int nb, int64_t p, double* dTx, double* width,
                            cudaStream_t s) {
  if (p <= 0) return cudaSuccess;
  const unsigned g = (unsigned)((p * 32 + kColThreads - 1) / kColThreads);
  if (prec == 0) k_coord_init<ff><<<g, kColThreads, 0, s>>>((const ff*)part, nb, p, dTx, width);
  else k_coord_init<double><<<g, kColThreads, 0, s>>>((const double*)part, nb, p, dTx, width);
  return cudaGetLastError();
}

cudaError_t prep_check_finite_f64(const double* v, int64_t count, unsigned* perr, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_check_finite<<<grid_for(count, kPrepThreads, 1024), kPrepThreads, 0, s>>>(v, count, perr);
  return cudaGetLastError();
}

size_t prep_count_bytes(int64_t n) { return 3 * sizeof(int32_t) * (size_t)((n + kGrpRows - 1) / kGrpRows); }

cudaError_t prep_group_count(const int32_t* time, const int8_t* status, int64_t n, int model, void* cnt,
                             unsigned* perr, int32_t* K, int32_t* total_events, unsigned* ticket, cudaStream_t s,
                             uint32_t* event, int32_t* crowd) {
  if (n <= 0) return cudaSuccess;
  const int64_t nb = (n + kGrpRows - 1) / kGrpRows;
  k_group_count<<<(unsigned)nb, kGrpThreads, 0, s>>>(time, status, n, model, nb, static_cast<int32_t*>(cnt), perr, K,
                                                     total_events, ticket, event, crowd);
  return cudaGetLastError();
}

cudaError_t prep_group_write(const int32_t* time, const int8_t* status, int64_t n, const void* cnt, int32_t K,
                             int32_t* gend, int32_t* dk, int32_t* ck, int32_t nwarps, int64_t rows_per_warp,
                             int32_t* wk0, cudaStream_t s, const RowMasks* masks) {
  if (K <= 0 || n <= 0) return cudaSuccess;
  cudaError_t st = cudaMemsetAsync(dk, 0, sizeof(int32_t) * (size_t)K, s);
  if (st == cudaSuccess && ck) st = cudaMemsetAsync(ck, 0, sizeof(int32_t) * (size_t)K, s);
  if (st != cudaSuccess) return st;
  const int64_t nb = (n + kGrpRows - 1) / kGrpRows;
  k_group_write<<<(unsigned)nb, kGrpThreads, 0, s>>>(time, status, n, nb, static_cast<const int32_t*>(cnt), K, gend,
                                                     dk, ck, nwarps, rows_per_warp, wk0, masks ? *masks : RowMasks{});
  return cudaGetLastError();
}

cudaError_t prep_km(const int32_t* gend, const int32_t* ck, int32_t K, double* Gk, cudaStream_t s) {
  if (K <= 0) return cudaSuccess;
  k_km_factor<<<grid_for(K, kPrepThreads, 16384), kPrepThreads, 0, s>>>(gend, ck, K, Gk);
  cudaError_t st = cudaGetLastError();
  if (st != cudaSuccess) return st;
  k_km_product<<<1, kKmThreads, 0, s>>>(K, Gk);
  return cudaGetLastError();
}

cudaError_t prep_weights(const int32_t* time, const int8_t* status, int64_t n, const void* cnt, int32_t K,
                         const double* Gk, float2* Gkff, void* inv, void* w2, int prec, cudaStream_t s) {
  if (K <= 0 || n <= 0) return cudaSuccess;
  const int64_t nb = (n + kGrpRows - 1) / kGrpRows;
  const unsigned g = grid_for(K, kPrepThreads, 16384);
  const int32_t* c = static_cast<const int32_t*>(cnt);
  if (prec == 0) {
    k_km_finish<float><<<g, kPrepThreads, 0, s>>>(K, Gk, Gkff, (float*)inv);
    k_w2<float><<<(unsigned)nb, kGrpThreads, 0, s>>>(time, status, n, nb, c, (const float*)inv, (float*)w2);
  } else {
    k_km_finish<double><<<g, kPrepThreads, 0, s>>>(K, Gk, Gkff, (double*)inv);
    k_w2<double><<<(unsigned)nb, kGrpThreads, 0, s>>>(time, status, n, nb, c, (const double*)inv, (double*)w2);
  }
  return cudaGetLastError();
}

cudaError_t prep_warp_groups(const int32_t* gend, int32_t K, int64_t n, int32_t nwarps, int64_t rows_per_warp,
                             int32_t* wk0, cudaStream_t s) {
  k_warp_groups<<<grid_for((int64_t)nwarps + 1, kPrepThreads), kPrepThreads, 0, s>>>(gend, K, n, nwarps,
                                                                                       rows_per_warp, wk0);
  return cudaGetLastError();
}

cudaError_t prep_warp_offsets(const int64_t* col_ptr, const int32_t* row_idx, int64_t p, int64_t n, int32_t nwarps,
                              int64_t rows_per_warp, int32_t* woff, cudaStream_t s) {
  const int64_t total = p * ((int64_t)nwarps + 1);
  if (total <= 0) return cudaSuccess;
  k_warp_offsets<<<grid_for(total, kPrepThreads, 1u << 30), kPrepThreads, 0, s>>>(col_ptr, row_idx, p, n, nwarps,
                                                                                   rows_per_warp, woff);
  return cudaGetLastError();
}

cudaError_t prep_eta_dense(const void* X, int prec, int64_t ld, int64_t n, int64_t p, const double* beta, void* eta,
                           void* e, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const unsigned g = grid_for(n, kPrepThreads, 8192);
  if (prec == 0) k_eta_dense<float><<<g, kPrepThreads, 0, s>>>((const float*)X, ld, n, p, beta, eta, (float*)e);
  else k_eta_dense<double><<<g, kPrepThreads, 0, s>>>((const double*)X, ld, n, p, beta, eta, (double*)e);
  return cudaGetLastError();
}

cudaError_t prep_eta_zero(int prec, int64_t n, void* eta, void* e, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const unsigned g = grid_for(n, kPrepThreads, 8192);
  if (prec == 0) k_eta_zero<float><<<g, kPrepThreads, 0, s>>>(n, eta, (float*)e);
  else k_eta_zero<double><<<g, kPrepThreads, 0, s>>>(n, eta, (double*)e);
  return cudaGetLastError();
}

cudaError_t prep_eta_axpy_csc(const int64_t* col_ptr, const int32_t* row_idx, const void* values, int prec,
                              int64_t j, int64_t nnz_j, double delta, void* eta, cudaStream_t s) {
  (void)col_ptr;
  if (nnz_j <= 0) return cudaSuccess;
  (void)j;
  const unsigned g = grid_for(nnz_j, kPrepThreads, 8192);
  if (prec == 0) k_eta_axpy_csc<float><<<g, kPrepThreads, 0, s>>>(row_idx, (const float*)values, nnz_j, delta, eta);
  else k_eta_axpy_csc<double><<<g, kPrepThreads, 0, s>>>(row_idx, (const double*)values, nnz_j, delta, eta);
  return cudaGetLastError();
}

cudaError_t prep_eta_exp(int prec, int64_t n, const void* eta, void* e, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const unsigned g = grid_for(n, kPrepThreads, 8192);
  if (prec == 0) k_eta_exp<float><<<g, kPrepThreads, 0, s>>>(n, eta, (float*)e);
  else k_eta_exp<double><<<g, kPrepThreads, 0, s>>>(n, eta, (double*)e);
  return cudaGetLastError();
}

cudaError_t prep_fill_f64(double* v, double value, int64_t count, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_fill_f64<<<grid_for(count, kPrepThreads, 1024), kPrepThreads, 0, s>>>(v, value, count);
  return cudaGetLastError();
}

cudaError_t prep_convert_dense(const void* src, int src_dtype, int64_t n, int64_t p, void* dst, int prec, int64_t ld,
                               cudaStream_t s) {
  if (ld * p <= 0) return cudaSuccess;
  const dim3 g(grid_for((ld + 3) / 4, kPrepThreads, 1024), (unsigned)std::min<int64_t>(p, 65535));
  if (src_dtype == 0 && prec == 0) k_convert_dense<float, float><<<g, kPrepThreads, 0, s>>>((const float*)src, n, p, (float*)dst, ld);
  else if (src_dtype == 0) k_convert_dense<float, double><<<g, kPrepThreads, 0, s>>>((const float*)src, n, p, (double*)dst, ld);
  else if (src_dtype == 2 && prec == 0)
    k_convert_dense<__nv_bfloat16, float><<<g, kPrepThreads, 0, s>>>((const __nv_bfloat16*)src, n, p, (float*)dst, ld);
  else if (src_dtype == 2)
    k_convert_dense<__nv_bfloat16, double><<<g, kPrepThreads, 0, s>>>((const __nv_bfloat16*)src, n, p, (double*)dst, ld);
  else if (prec == 0) k_convert_dense<double, float><<<g, kPrepThreads, 0, s>>>((const double*)src, n, p, (float*)dst, ld);
  else k_convert_dense<double, double><<<g, kPrepThreads, 0, s>>>((const double*)src, n, p, (double*)dst, ld);
  return cudaGetLastError();
}

cudaError_t prep_convert_vec(const void* src, int src_dtype, int64_t count, void* dst, int prec, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  const unsigned g = grid_for(count, kPrepThreads, 16384);
  if (src_dtype == 0 && prec == 0) k_convert_vec<float, float><<<g, kPrepThreads, 0, s>>>((const float*)src, count, (float*)dst);
  else if (src_dtype == 0) k_convert_vec<float, double><<<g, kPrepThreads, 0, s>>>((const float*)src, count, (double*)dst);
  else if (prec == 0) k_convert_vec<double, float><<<g, kPrepThreads, 0, s>>>((const double*)src, count, (float*)dst);
  else k_convert_vec<double, double><<<g, kPrepThreads, 0, s>>>((const double*)src, count, (double*)dst);
  return cudaGetLastError();
}

}  // namespace survgpu
