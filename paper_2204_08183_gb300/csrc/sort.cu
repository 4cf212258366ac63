// Stable order of decreasing time (Section 2.7 arranges the subjects by
// decreasing observed time; ties keep their input order).  Least-significant
// digit radix sort over the key ~(t ^ 0x80000000), which orders signed times
// descending; every pass is stable, so equal times keep the input order and
// the permutation is unique.
//
// The times of a cohort span far fewer values than 2^32 (a day grid of ten
// years needs 12 bits), so k_range finds the key range first and only the
// bits of key - smallest key are sorted, in the fewest passes of at most 8
// bits and digits of equal width: 2 passes of 6 bits instead of 4 of 8.
// Narrow digits also give longer runs per digit in the scatter.  The bytes
// bound a pass: the first reads the times themselves, the last writes no keys.
//
// Per pass, tiles of 4096 elements:
//   k_hist     digit counts of each tile (digit-major table);
//   k_scan     one block per digit: exclusive prefix of its tile counts, and
//              the digit's total;
//   k_scatter  ranks within the tile (warp ballots over the digit's bits, one
//              counter per warp and digit), the tile put in order in shared
//              memory, and each digit's run written out contiguously.
// Four passes of 8 bits, with one block scanning the whole count table (8.6
// ms of it) and scatters straight from registers, took 9.3 ms of device time
// at n = 10^7 and days 1..3650; ordering and grouping such records takes
// 0.88 instead of 10.35 ms in all (with the tie-group table in two passes and the
// scratch pool).
#include <algorithm>
#include <cstdint>

#include "internal.h"

namespace survgpu {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 16;                   // elements per thread
constexpr int kTile = kThreads * kItems;
constexpr int kMaxBits = 8;
constexpr int kMaxBins = 1 << kMaxBits;

inline size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

__device__ __forceinline__ uint32_t key_of(int32_t t) { return ~((uint32_t)t ^ 0x80000000u); }

// range[0] = max key, range[1] = max ~key (both zeroed before)
__global__ void __launch_bounds__(kThreads) k_range(const int32_t* time, int64_t n, uint32_t* range) {
  uint32_t hi = 0, lo = 0;
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  for (; i + 3 * stride < n; i += 4 * stride) {
    uint32_t k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) k[u] = key_of(time[i + u * stride]);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      hi = max(hi, k[u]);
      lo = max(lo, ~k[u]);
    }
  }
  for (; i < n; i += stride) {
    const uint32_t k = key_of(time[i]);
    hi = max(hi, k);
    lo = max(lo, ~k);
  }
  hi = __reduce_max_sync(0xffffffffu, hi);
  lo = __reduce_max_sync(0xffffffffu, lo);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(range, hi);
    atomicMax(range + 1, lo);
  }
}

__global__ void k_iota(int32_t* perm, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    perm[i] = (int32_t)i;
}

// Sort key of element i: from the times (first pass) or the keys of the
// previous pass, both relative to the smallest key.
struct Source {
  const int32_t* time;    // first pass, else null
  const uint32_t* keys;
  const int32_t* vals;    // later passes
  uint32_t kmin;
  __device__ __forceinline__ uint32_t key(int64_t i) const { return time ? key_of(time[i]) - kmin : keys[i]; }
  __device__ __forceinline__ int32_t val(int64_t i) const { return time ? (int32_t)i : vals[i]; }
};

__global__ void __launch_bounds__(kThreads) k_hist(Source src, int64_t n, int shift, int bits, int64_t ntiles,
                                                   uint32_t* counts) {
  __shared__ uint32_t s[kWarps][kMaxBins];
  const int bins = 1 << bits, w = threadIdx.x >> 5;
  for (int d = threadIdx.x; d < kWarps * kMaxBins; d += kThreads) (&s[0][0])[d] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kTile;
  uint32_t k[kItems];
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int64_t i = base + u * kThreads + threadIdx.x;
    k[u] = i < n ? src.key(i) : 0u;
  }
#pragma unroll
  for (int u = 0; u < kItems; ++u)
    if (base + u * kThreads + threadIdx.x < n) atomicAdd(&s[w][(k[u] >> shift) & (bins - 1)], 1u);
  __syncthreads();
  for (int d = threadIdx.x; d < bins; d += kThreads) {
    uint32_t c = 0;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) c += s[q][d];
    counts[(int64_t)d * ntiles + blockIdx.x] = c;
  }
}

// Digit d = blockIdx.x: exclusive prefix of its tile counts in place, total[d].
__global__ void __launch_bounds__(kThreads) k_scan(uint32_t* counts, int64_t ntiles, uint32_t* total) {
  __shared__ uint32_t s_w[kWarps];
  uint32_t* a = counts + (int64_t)blockIdx.x * ntiles;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t per = (ntiles + kThreads - 1) / kThreads;
  const int64_t lo = min((int64_t)tid * per, ntiles), hi = min(lo + per, ntiles);
  uint32_t sum = 0;
  for (int64_t q = lo; q < hi; ++q) sum += a[q];
  uint32_t inc = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= d) inc += v;
  }
  if (lane == 31) s_w[w] = inc;
  __syncthreads();
  uint32_t run = inc - sum;
  for (int q = 0; q < w; ++q) run += s_w[q];
  if (tid == kThreads - 1) total[blockIdx.x] = run + sum;
  for (int64_t q = lo; q < hi; ++q) {
    const uint32_t v = a[q];
    a[q] = run;
    run += v;
  }
}

// kout null: the last pass (only the permutation is written)
__global__ void __launch_bounds__(kThreads) k_scatter(Source src, int64_t n, int shift, int bits, int64_t ntiles,
                                                      const uint32_t* counts, const uint32_t* total, uint32_t* kout,
                                                      int32_t* vout) {
  __shared__ uint32_t s_cnt[kWarps][kMaxBins];
  __shared__ uint32_t s_first[kMaxBins];   // first place of each digit in the tile
  __shared__ uint32_t s_out[kMaxBins];     // place in the output of a digit's first element, minus s_first
  __shared__ uint32_t s_w[2][kWarps];
  __shared__ uint32_t s_key[kTile];
  __shared__ int32_t s_val[kTile];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int bins = 1 << bits;
  const int64_t base = (int64_t)blockIdx.x * kTile;
  const int m = (int)min((int64_t)kTile, n - base);
  for (int d = tid; d < kWarps * kMaxBins; d += kThreads) (&s_cnt[0][0])[d] = 0;
  // a warp holds 512 consecutive elements, 32 a round: rounds and lanes in order
  uint32_t k[kItems];
  int32_t v[kItems];
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int i = w * (32 * kItems) + u * 32 + lane;
    k[u] = i < m ? src.key(base + i) : 0u;
    v[u] = i < m ? src.val(base + i) : 0;
  }
  __syncthreads();
  uint32_t rank[kItems];
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const bool in = w * (32 * kItems) + u * 32 + lane < m;
    const uint32_t d = (k[u] >> shift) & (bins - 1);
    unsigned peers = __ballot_sync(0xffffffffu, in);
#pragma unroll
    for (int b = 0; b < kMaxBits; ++b) {
      if (b >= bits) break;
      const bool set = (d >> b) & 1u;
      const unsigned bal = __ballot_sync(0xffffffffu, set);
      peers &= set ? bal : ~bal;
    }
    uint32_t before = 0;
    if (in) before = s_cnt[w][d];
    __syncwarp();
    const unsigned lower = peers & ((1u << lane) - 1u);
    rank[u] = before + __popc(lower);
    if (in && lower == 0u) s_cnt[w][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // digit d = thread d: counts of the earlier warps, the tile's first place of
  // the digit, and the digit's place in the output (scans over the digits)
  uint32_t tile_d = 0, tot_d = 0;
  if (tid < bins) {
#pragma unroll
    for (int q = 0; q < kWarps; ++q) {
      const uint32_t c = s_cnt[q][tid];
      s_cnt[q][tid] = tile_d;
      tile_d += c;
    }
    tot_d = total[tid];
  }
  uint32_t it = tile_d, io = tot_d;
#pragma unroll
  for (int dd = 1; dd < 32; dd <<= 1) {
    const uint32_t a = __shfl_up_sync(0xffffffffu, it, dd), b = __shfl_up_sync(0xffffffffu, io, dd);
    if (lane >= dd) {
      it += a;
      io += b;
    }
  }
  if (lane == 31) {
    s_w[0][w] = it;
    s_w[1][w] = io;
  }
  __syncthreads();
  if (tid < bins) {
    uint32_t first = it - tile_d, out = io - tot_d;
    for (int q = 0; q < w; ++q) {
      first += s_w[0][q];
      out += s_w[1][q];
    }
    s_first[tid] = first;
    s_out[tid] = out + counts[(int64_t)tid * ntiles + blockIdx.x] - first;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    if (w * (32 * kItems) + u * 32 + lane < m) {
      const uint32_t d = (k[u] >> shift) & (bins - 1);
      const uint32_t at = s_first[d] + s_cnt[w][d] + rank[u];
      s_key[at] = k[u];
      s_val[at] = v[u];
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int i = u * kThreads + tid;
    if (i < m) {
      const uint32_t key = s_key[i];
      const uint32_t pos = s_out[(key >> shift) & (bins - 1)] + (uint32_t)i;
      if (kout) kout[pos] = key;
      vout[pos] = s_val[i];
    }
  }
}

}  // namespace

size_t radix_sort_workspace(int64_t n) {
  const int64_t ntiles = (n + kTile - 1) / kTile;
  return align256(4 * (size_t)n) * 3 + align256(4 * (size_t)kMaxBins * (size_t)ntiles) + align256(4 * kMaxBins) +
         256;
}

cudaError_t radix_sort_desc(const int32_t* time, int64_t n, int32_t* perm, void* work, cudaStream_t s,
                            int* launches) {
  if (n <= 0) return cudaSuccess;
  const int64_t ntiles = (n + kTile - 1) / kTile;
  char* wp = static_cast<char*>(work);
  const size_t nb = align256(4 * (size_t)n);
  uint32_t* kbuf[2] = {reinterpret_cast<uint32_t*>(wp), reinterpret_cast<uint32_t*>(wp + nb)};
  int32_t* vbuf = reinterpret_cast<int32_t*>(wp + 2 * nb);
  uint32_t* counts = reinterpret_cast<uint32_t*>(wp + 3 * nb);
  uint32_t* total = reinterpret_cast<uint32_t*>(wp + 3 * nb + align256(4 * (size_t)kMaxBins * (size_t)ntiles));
  uint32_t* range = total + kMaxBins;
  cudaError_t st;
  if ((st = cudaMemsetAsync(range, 0, 8, s)) != cudaSuccess) return st;
  const unsigned gr = (unsigned)std::min<int64_t>((n + 4 * kThreads - 1) / (4 * kThreads), 152 * 8);
  k_range<<<gr, kThreads, 0, s>>>(time, n, range);
  int nl = 1;
  uint32_t r[2];
  if ((st = cudaGetLastError()) != cudaSuccess) return st;
  if ((st = cudaMemcpyAsync(r, range, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return st;
  if ((st = cudaStreamSynchronize(s)) != cudaSuccess) return st;
  const uint32_t kmin = ~r[1], span = r[0] - kmin;
  int nbits = 0;
  while (nbits < 32 && (span >> nbits) != 0u) ++nbits;
  if (nbits == 0) {   // one distinct time: the input order
    k_iota<<<(unsigned)std::min<int64_t>((n + kThreads - 1) / kThreads, 65535), kThreads, 0, s>>>(perm, n);
    ++nl;
  }
  // a permutation written over its own times: keep a copy of them
  const char *t0 = reinterpret_cast<const char*>(time), *p0 = reinterpret_cast<const char*>(perm);
  if (nbits && t0 < p0 + 4 * n && p0 < t0 + 4 * n) {
    if ((st = cudaMemcpyAsync(kbuf[1], time, 4 * (size_t)n, cudaMemcpyDeviceToDevice, s)) != cudaSuccess) return st;
    time = reinterpret_cast<const int32_t*>(kbuf[1]);
  }
  const int passes = (nbits + kMaxBits - 1) / kMaxBits;
  const int width = passes ? (nbits + passes - 1) / passes : 0;
  const uint32_t* kin = nullptr;
  const int32_t* vin = nullptr;
  for (int i = 0; i < passes; ++i) {
    const int shift = i * width, bits = std::min(width, nbits - shift);
    const bool last = i == passes - 1;
    uint32_t* kout = last ? nullptr : kbuf[i & 1];
    int32_t* vout = ((passes - 1 - i) & 1) ? vbuf : perm;
    const Source src{i == 0 ? time : nullptr, kin, vin, kmin};
    k_hist<<<(unsigned)ntiles, kThreads, 0, s>>>(src, n, shift, bits, ntiles, counts);
    k_scan<<<1 << bits, kThreads, 0, s>>>(counts, ntiles, total);
    k_scatter<<<(unsigned)ntiles, kThreads, 0, s>>>(src, n, shift, bits, ntiles, counts, total, kout, vout);
    nl += 3;
    kin = kout;
    vin = vout;
  }
  if (launches) *launches += nl;
  return cudaGetLastError();
}

}  // namespace survgpu
