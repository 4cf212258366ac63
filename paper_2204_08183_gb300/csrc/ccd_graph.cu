// Per-coordinate CCD schedule (Sections 2.4 and 2.7): two kernels per
// coordinate, one sweep of them captured once as a CUDA graph and replayed
// until the device reports that the fit has stopped.
//
//   k_pass(j)   CTA c reads the step of coordinate q = j - 1 (line c % kRep),
//               each warp applies eta += x_q * step and e = exp(eta) to its
//               own rows, then runs the row pass (step 2) of coordinate j
//               over those rows and the CTA publishes its warp totals and its
//               aggregate.
//   k_btrans(j) every CTA scans the aggregates in a fixed order, transforms its
//               share of the group ends (steps 3-4) and publishes three
//               partial sums.  The last CTA to finish (atomic ticket; nobody
//               waits for it) sums the partials in a fixed order, takes the
//               FP64 Newton step of Section 2.4, stores beta_j and its
//               trust-region width, on j = 0 evaluates the objective and the
//               stopping rule, and publishes the step for k_pass(j + 1).
//
// Kernel boundaries order every producer before its consumers: no kernel
// waits on another CTA.  A warp only reads and writes eta / e on its own
// rows, so the update of q needs no barrier before the pass.  Launches use
// programmatic dependent launch: loads of static tables are issued before
// griddepcontrol.wait, which hides most of the launch gap.
//
// Batched fits (cross-validation x lambda path, Section 2.8): the same two
// kernels run every fit at once, fit f on blockIdx.y with its own
// parameters (CcdParams::fits[f], copied to shared memory at the start of
// each CTA).  Fits stop independently; each one counts itself into a device
// counter when it stops, and the host replays the sweep until all have.
#include <algorithm>
#include <cstdlib>
#include <cstring>

#include "graph_common.cuh"

namespace survgpu {
namespace {

using namespace ccdk;

// Pass kernel shape: 512 threads, two CTAs per SM (64 registers a thread):
// tiles of 4 16-byte loads per array per lane (2 for Fine-Gray, whose six
// running sums take the registers), 4 rounds of the column's nonzeros
// prefetched.  Measured at N = 10^7 against one CTA of 16 warps per
// SM, and against staging e in shared memory with bulk copies (whole SM or
// per warp), this shape was the fastest.
template <int MODEL, int LAYOUT>
struct GCfg {
  static constexpr int NT = 512;
  static constexpr int MINB = 2;
  static constexpr int U = (MODEL == 1 && LAYOUT == 1) ? 1 : (MODEL == 1 || LAYOUT == 1 ? 2 : 4);
  static constexpr int SR = 4;
};

// Fill every control line for the first coordinate of a fit (of fit
// blockIdx.y in a batched launch).
__global__ void k_graph_init(const __grid_constant__ CcdParams P0) {
  const CcdParams& P = P0.fits ? P0.fits[blockIdx.y] : P0;
  const int r = threadIdx.x;
  if (r >= kRep) return;
  CtlLine* L = &P.gctl->line[r];
  L->stop = 0;
  L->nevals = 0;
  L->applied = 0.0;
  L->delta_hi = 0.f;
  L->delta_lo = 0.f;
  L->beta = P.beta[0];
  L->width = P.width[0];
  L->pen = P.pen[0];
  L->dtx = P.dTx[0];
  L->f_prev = 0.0;
  L->passes = 0;
  L->eta_updates = 0;
  L->dirty = 1;
  L->j0 = 0;
  L->q = -1;
  L->batches = 0;
}

// MULTI selects the group-end handling for warps that hold many ends (see
// warp_pass); the host picks it when the tie groups outnumber the warps.
// TW picks the tile shape: 0 the configured one, 1 half the 16-byte loads of
// e per lane a tile, 2 half the rounds of nonzeros loaded together (twice
// the loads spilled at the 64-register cap).
template <int MODEL, int LAYOUT, typename T, bool BATCH, bool MULTI, int TW = 0>
__global__ void __launch_bounds__(GCfg<MODEL, LAYOUT>::NT, GCfg<MODEL, LAYOUT>::MINB)
    k_pass(const __grid_constant__ CcdParams P0, int j) {
  using A = typename AccOf<T>::type;
  using C = Cfg<MODEL, LAYOUT, T>;
  constexpr int M = C::M;
  __shared__ A s_wtot[kMaxWarpsPerCta][M];
  __shared__ int s_stop, s_dirty;
  __shared__ double s_applied;
  __shared__ float s_delta[2];
  __shared__ CcdParams s_fit;
  if (BATCH) load_fit(s_fit, P0);
  const CcdParams& P = BATCH ? s_fit : P0;

  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int w = tid >> 5;
  const int WPC = P.wpc;
  const int c = blockIdx.x;
  const int G = P.G;
  const int64_t n = P.n;
  const int64_t nwords = (n + 31) >> 5;
  const int gw = c * WPC + w;
  const int64_t word_lo = min((int64_t)gw * P.wpw, nwords);
  const int64_t word_hi = min(word_lo + P.wpw, nwords);
  const int64_t row_lo = word_lo * 32;
  const int64_t row_hi = min(word_hi * 32, n);
  const int q = j == 0 ? P.p - 1 : j - 1;  // coordinate whose step is applied here

  // column j's first nonzeros and the warp's group ends do not depend on
  // earlier kernels: load them before waiting for the previous kernel
  using GC = GCfg<MODEL, LAYOUT>;
  constexpr int U = TW == 1 ? (GC::U > 1 ? GC::U / 2 : 1) : GC::U;
  constexpr int SR = TW == 2 ? GC::SR / 2 : GC::SR;
  PassPrefetch<T, SR> pf;
  pass_prefetch<LAYOUT, T, SR>(P, j, gw, pf);
  pdl_wait();

  // the step of q (zero before the first coordinate of a fit), read once
  if (tid == 0) {
    const CtlLine* L = &P.gctl->line[c % kRep];
    s_stop = __ldcg(&L->stop);
    s_applied = __ldcg(&L->applied);
    s_delta[0] = __ldcg(&L->delta_hi);
    s_delta[1] = __ldcg(&L->delta_lo);
    s_dirty = __ldcg(&L->dirty);
  }
  __syncthreads();
  if (s_stop) return;  // the same value in every CTA
  const double applied = s_applied;
  // dense X in the FP32 mode: the update rides along the row pass (one sweep
  // over the warp's rows); otherwise it runs first
  constexpr bool kFuse = LAYOUT == 1 && sizeof(T) == 4;
  if (applied != 0.0 && !kFuse) warp_update<LAYOUT, T>(P, q, gw, row_lo, row_hi, applied, ff{s_delta[0], s_delta[1]});
  // CSC: with a zero pending step e is the e of the previous coordinate's
  // pass (after the fit's first pass), and so are the sums of its dense
  // components, stored by that pass; they are reused bit for bit
  const bool dense = LAYOUT == 1 || applied != 0.0 || s_dirty != 0;
  const T* xq = (kFuse && applied != 0.0) ? reinterpret_cast<const T*>(P.X) + (size_t)q * P.ld : nullptr;

  // ------------------------------------------- step 2 for coordinate j
  A* rec = reinterpret_cast<A*>(P.rec);
  A tot[M];
  warp_pass<MODEL, LAYOUT, T, U, SR, MULTI>(P, j, row_lo, row_hi, rec, tot, pf, dense, xq, ff{s_delta[0], s_delta[1]});
  pdl_launch_dependents();
  if (lane == 0)
#pragma unroll
    for (int m = 0; m < M; ++m) s_wtot[w][m] = tot[m];
  __syncthreads();
  if (w == 0) {
    // warp offsets inside the CTA (exclusive scan of the warp totals) and
    // the CTA aggregate (their total), every lane in the same order
    A v[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
      acc_zero(v[m]);
      if (lane < WPC) v[m] = s_wtot[lane][m];
    }
    warp_scan_n<M>(v, lane);
#pragma unroll
    for (int m = 0; m < M; ++m) {
      // the stored values of the dense CSC components stay when they were reused
      const bool keep = LAYOUT == 0 && !dense && (m == 0 || m == 3);
      A ex = shfl_up(v[m], 1);
      if (lane == 0) acc_zero(ex);
      if (lane < WPC && !keep) P.wt[(size_t)m * P.nwarps + c * WPC + lane] = pack8(ex);
      v[m] = shfl_idx(v[m], WPC - 1);
    }
    if (lane == 0)
#pragma unroll
      for (int m = 0; m < M; ++m)
        if (!(LAYOUT == 0 && !dense && (m == 0 || m == 3))) P.agg[(size_t)m * G + c] = pack8(v[m]);
  }
}

// The transform, its work spread evenly: every CTA scans the
// pass CTAs' aggregates (one per thread, two-level warp scans in shared
// memory; Fine-Gray also takes the grand totals of the suffix components)
// and takes an even share of the group ends, about one a thread (batched fits:
// about four).  A split by pass CTA gave the CTAs holding the first rows (many
// small tie groups) most of the work; and with a CTA per pass CTA and one end
// a thread, the reductions of 200 batched fits cost more than their ends (50
// us of a coordinate's 280 at n = 10^6).  It reads the control line and its
// first end's group table entries before the wait: the line was written by
// the previous coordinate's transform, which finished before this
// coordinate's pass kernel passed its own wait.
//
// Threads: it is a chain of float-float scans and reductions, and several
// warps on a scheduler lengthen every one of them, so the block has one warp
// per scheduler and the ends more CTAs, as long as a thread then gets one end
// (us a coordinate, 512 and 128 threads: 27.1 and 24.8 for 1000 ends of
// Fine-Gray, 20.5 and 18.5 for 3650 of Cox; 28.6 and 39.0 for 310,400, where
// 128 threads on every SM walk 16 ends each).
constexpr int kBtSmall = 128, kBtLarge = 512;
constexpr int kBtMaxG = 384;   // pass CTAs

// Up to 4096 ends a single fit's transform is one cluster of at most 16 CTAs
// (two ends a thread), whose partial sums meet in the first CTA's shared
// memory at a cluster barrier: the fence, the ticket and the way through L2
// that other transforms end with take 1 us longer (ms a fit with the ticket
// and the cluster: 10.02 and 9.76 for Fine-Gray at 5 x 10^6 x 50,
// 1000 ends; 2.32 and 2.25 for dense Cox at 500,009 x 24, 3650 ends).
constexpr int kBtCluster = 16;
inline bool btrans_one_cluster(int K) { return K <= 2 * kBtSmall * kBtCluster; }
constexpr int kBtMaxCtas = kMaxTransCtas;
// Sparse Cox data in FP32, whose pass is the shortest, wants the larger blocks
// from 8192 ends on: at 10,000 to 19,000 of them 79 to 148 small blocks start
// later behind the pass than 20 to 38 large ones (us a coordinate at 3 x 10^6
// rows, 128 and 512 threads: 26.4 and 24.1; 6 % on average over even, 2 % over
// exponential times; other data between 1 % this and 6 % the other way).
template <int MODEL, int LAYOUT, typename T>
inline int btrans_threads(int K) {
  constexpr int most = MODEL == 0 && LAYOUT == 0 && sizeof(T) == 4 ? 8192 : kBtSmall * kBtMaxCtas;
  return K <= most ? kBtSmall : kBtLarge;
}

template <int MODEL, int LAYOUT, typename T, int kBtNT, bool BATCH = false, bool CLUSTER = false>
__global__ void __launch_bounds__(kBtNT, 1) k_btrans(const __grid_constant__ CcdParams P0, int j) {
  using A = typename AccOf<T>::type;
  constexpr int M = MODEL == 0 ? 3 : 6;
  constexpr int kBtWarps = kBtNT / 32, kAgg = kBtNT == kBtSmall ? 3 : 1;
  __shared__ A s_T[kBtNT * kAgg][M];
  __shared__ A s_w[kBtWarps][M];
  __shared__ A s_all[M];   // grand totals (Fine-Gray: the suffix components)
  __shared__ A s_red[kBtWarps][3];
  __shared__ int s_last, s_stop;
  __shared__ double s_lin[2];
  __shared__ double s_next[4];
  __shared__ uint64_t s_part[CLUSTER ? 3 * kBtCluster : 1];   // the CTAs' partials (in the first CTA)
  __shared__ CcdParams s_fit;
  if (CLUSTER) cluster_arrive();   // this CTA has started
  if (BATCH) load_fit(s_fit, P0);
  const CcdParams& P = BATCH ? s_fit : P0;
  GraphCtl* ctl = P.gctl;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int WPC = P.wpc, G = P.G, G2 = gridDim.x, c2 = blockIdx.x;
  const bool eval = j == 0;
  LineView lv;
  if (tid == 0) {
    lv = load_line(ctl, c2);
    s_stop = lv.stop;
  }
  // the next coordinate's scalars for the control line (warp 3; last written a
  // sweep ago, or, for two coordinates, two transforms ago)
  static_assert(kBtWarps >= 4 && kBtNT * kAgg >= kBtMaxG, "three warps sum the partials, the fourth does the rest");
  double nx[4] = {0.0, 0.0, 0.0, 0.0};
  if (w == 3 && lane == 0) {
    const int jn = j + 1 < P.p ? j + 1 : 0;
    nx[0] = __ldcg(P.beta + jn);
    nx[1] = __ldcg(P.width + jn);
    nx[2] = P.pen[jn];
    nx[3] = P.dTx[jn];
  }
  const int stride = G2 * kBtNT;
  const int k0 = c2 * kBtNT + tid;
  int d1 = 0, gw1 = 0;
  double g1 = 0.0;
  float2 gf1 = make_float2(0.f, 0.f);
  if (k0 < P.K) {
    d1 = P.dk[k0];
    gw1 = (int)((P.gend[k0] >> 5) / P.wpw);
    if (MODEL == 1) {
      g1 = P.Gk[k0];
      gf1 = P.Gkff[k0];
    }
  }
  __syncthreads();
  if (CLUSTER) cluster_wait();
  if (s_stop) {  // the same value in every CTA of the fit
    pdl_wait();
    return;
  }
  pdl_wait();

  // prefixes of the pass CTAs' aggregates
  scan_aggregates<kBtNT, kAgg, M, A>(P.agg, G, s_T, s_w, MODEL == 1 ? s_all : nullptr);
  __syncthreads();

  // steps 3-4 at the group ends
  A fg1, fg2;
  acc_zero(fg1);
  acc_zero(fg2);
  double pl = 0.0;
  A tot3[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    acc_zero(tot3[i]);
    if (MODEL == 1) tot3[i] = s_all[(3 + i) % M];
  }
  const A* rec = reinterpret_cast<const A*>(P.rec);
  for (int k = k0; k < P.K; k += stride) {
    int d, gwk;
    double g;
    float2 gf;
    if (k == k0) {
      d = d1, gwk = gw1, g = g1, gf = gf1;
    } else {
      d = P.dk[k];
      gwk = (int)((P.gend[k] >> 5) / P.wpw);
      g = MODEL == 1 ? P.Gk[k] : 0.0;
      gf = MODEL == 1 ? P.Gkff[k] : make_float2(0.f, 0.f);
    }
    if (d == 0) continue;
    const int f = gwk / WPC;
    A Pm[M];
#pragma unroll
    for (int m = 0; m < M; ++m)
      Pm[m] = acc_add(acc_add(s_T[f][m], unpack8<A>(__ldcg(P.wt + (size_t)m * P.nwarps + gwk))),
                      rec[(size_t)k * M + m]);
    A den = Pm[0], num1 = Pm[1], num2 = Pm[2];
    if (MODEL == 1) {
      // the competing-event suffix strictly after the end, weighted by G(t_k)
      const A gg = acc_base<A>(g, ff{gf.x, gf.y});
      den = acc_add(den, acc_mul(gg, acc_add(tot3[0], acc_neg(Pm[3 % M]))));
      num1 = acc_add(num1, acc_mul(gg, acc_add(tot3[1], acc_neg(Pm[4 % M]))));
      num2 = acc_add(num2, acc_mul(gg, acc_add(tot3[2], acc_neg(Pm[5 % M]))));
    }
    const A inv = acc_recip(den);
    const A Gr = acc_mul(num1, inv);
    const A H = acc_mul(num2, inv);
    fg1 = acc_add(fg1, acc_scale(Gr, d));
    fg2 = acc_add(fg2, acc_scale(acc_add(H, acc_neg(acc_mul(Gr, Gr))), d));
    if (eval) pl += (double)d * log(acc_to_d(den));
  }

  // CTA partials, fixed order
  {
    A r[3] = {fg1, fg2, eval ? acc_from_d(pl, (A*)nullptr) : A{}};
    warp_sum_n<3>(r);
    if (lane == 0)
#pragma unroll
      for (int i = 0; i < 3; ++i) s_red[w][i] = r[i];
  }
  __syncthreads();
  uint64_t* part = reinterpret_cast<uint64_t*>(P.slot_part);
  if (tid < 3) {
    A a = s_red[0][tid];
#pragma unroll 1
    for (int qw = 1; qw < kBtWarps; ++qw) a = acc_add(a, s_red[qw][tid]);
    if (CLUSTER) store_remote(&s_part[tid * kBtCluster + c2], 0, pack8(a));
    else part[(size_t)tid * G2 + c2] = pack8(a);
  }
  if (CLUSTER) {
    cluster_arrive();
    pdl_launch_dependents();
    cluster_wait();
    if (c2 != 0) return;
  } else {
    __syncthreads();
    if (tid == 0) {
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      unsigned prev;
      asm volatile("atom.add.release.gpu.u32 %0, [%1], 1;" : "=r"(prev) : "l"(&ctl->ticket) : "memory");
      s_last = prev == (unsigned)(G2 - 1);
    }
    pdl_launch_dependents();
    __syncthreads();
    if (!s_last) return;
  }

  // ------------------------------- last CTA: the step of coordinate j
  if (w < 3) {
    A acc;
    acc_zero(acc);
    if (CLUSTER) {
      if (lane < G2) acc = acc_add(acc, unpack8<A>(s_part[w * kBtCluster + lane]));
    } else {
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      for (int qc = lane; qc < G2; qc += 32) acc = acc_add(acc, unpack8<A>(__ldcg(part + (size_t)w * G2 + qc)));
    }
    A r[1] = {acc};
    warp_sum_n<1>(r);
    if (lane == 0) s_red[0][w] = r[0];
  } else if (w == 3) {
    if (eval) {
      double lin, pen;
      warp_lin_pen(P, -1, 0.0, lin, pen);
      if (lane == 0) {
        s_lin[0] = lin;
        s_lin[1] = pen;
      }
    }
    if (lane == 0)
#pragma unroll
      for (int i = 0; i < 4; ++i) s_next[i] = nx[i];
  }
  __syncthreads();
  if (w == 0)
    publish_step(P, j, lv, lv.dtx - acc_to_d(s_red[0][0]), -acc_to_d(s_red[0][1]), eval, s_lin[0], s_lin[1],
                 acc_to_d(s_red[0][2]), s_next);
}

// CTAs of the balanced transform: about one group end a thread.
inline int btrans_ctas(int K, int nt) {
  return std::max(4, std::min(kBtMaxCtas, (K + nt - 1) / nt));
}
// Per fit of a batch: about four ends a thread (kBtSmall threads).
inline int btrans_ctas_batch(int K) {
  return std::max(1, std::min(kBtMaxCtas, (K + 4 * kBtSmall - 1) / (4 * kBtSmall)));
}

// Grid of the pass kernel: as many CTAs per SM (up to MINB) as fit.
template <int MODEL, int LAYOUT, typename T>
cudaError_t grid_graph(int* G, int* wpc) {
  using GC = GCfg<MODEL, LAYOUT>;
  int dev = 0, sms = 0, occ = 0;
  cudaError_t st = cudaGetDevice(&dev);
  if (st != cudaSuccess) return st;
  if ((st = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return st;
  if ((st = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_pass<MODEL, LAYOUT, T, false, false>, GC::NT, 0)) !=
      cudaSuccess)
    return st;
  if (occ < 1) return cudaErrorLaunchOutOfResources;
  *G = sms * std::min(occ, GC::MINB);
  *wpc = GC::NT / 32;
  return cudaSuccess;
}

template <int MODEL, int LAYOUT, typename T>
cudaError_t capture_sweep(const CcdParams& P, bool pdl, cudaStream_t cs, cudaGraph_t* g) {
  using GC = GCfg<MODEL, LAYOUT>;
  if (P.G > kBtMaxG) return cudaErrorInvalidValue;   // the transform scans three aggregates a thread at most
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  const int bt = btrans_threads<MODEL, LAYOUT, T>(P.K);
  const unsigned cl = (unsigned)std::min(kBtCluster, btrans_ctas(P.K, bt));
  cudaLaunchAttribute attr_cl[2];
  const bool cluster = P.nfit == 0 && btrans_one_cluster(P.K) &&
                       cluster_launch(k_btrans<MODEL, LAYOUT, T, kBtSmall, false, true>, cl, kBtSmall, attr[0], attr_cl);
  cudaError_t st = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (st != cudaSuccess) return st;
  cudaLaunchConfig_t cp = {};
  cp.gridDim = dim3(P.G, P.nfit > 0 ? P.nfit : 1);
  cp.blockDim = dim3(GC::NT);
  cp.stream = cs;
  cp.attrs = attr;
  cp.numAttrs = 1;
  cudaLaunchConfig_t ct = cp;
  // batched fits: Cox only (the censoring weights of Fine-Gray would have
  // to be re-estimated on each training set)
  // The many-ends form of the row pass where warps hold two group ends or
  // more on average, and, with more than one dense component, where they hold
  // few rows: the ends are then few on average but crowd into the warps of the
  // latest times, whose way through them one after another is the pass (us a
  // coordinate, the plain and the many-ends form: 20.9 and 18.2 at 500,009 x
  // 24 dense Cox, 31.8 and 26.7 at 200,003 x 40 sparse Fine-Gray; at 5 x 10^6
  // x 50 dense Fine-Gray the plain form, 49.0 against 52.4).
  // Not for Fine-Gray in FP32 where the ends are spread evenly, two to four a
  // warp: its six (dense) or two components pay for the scan of each tile (us a
  // coordinate at 3 x 10^6 rows with 10,000 even ends, the many-ends and the
  // plain form: 54.3 and 44.1 dense, 44.4 and 39.0 at 10 % density; 57.6 and 63.1
  // dense with 30,000).
  constexpr int kEven = MODEL == 1 && sizeof(T) == 4 ? (LAYOUT == 1 ? 5 : 4) : 0;
  const bool many = (int64_t)P.K >= 2 * (int64_t)P.nwarps && (P.nfit > 0 || P.warp_ends >= kEven);
  const bool few_rows = P.nfit == 0 && P.wpw <= 16 && (Cfg<MODEL, LAYOUT, T>::ND > 1 || sizeof(T) == 8);
  auto kp = k_pass<MODEL, LAYOUT, T, false, false>;
  auto kt = bt == kBtSmall ? k_btrans<MODEL, LAYOUT, T, kBtSmall> : k_btrans<MODEL, LAYOUT, T, kBtLarge>;
  ct.gridDim = dim3(btrans_ctas(P.K, bt));
  ct.blockDim = dim3(bt);
  if (cluster) {
    kt = k_btrans<MODEL, LAYOUT, T, kBtSmall, false, true>;
    ct.gridDim = dim3(cl);
    ct.attrs = attr_cl;
    ct.numAttrs = 2;
  }
  if constexpr (MODEL == 0) {
    const bool multi = P.pass_form == 2 || (P.pass_form == 0 && (many || few_rows));
    if (P.nfit > 0) {
      kp = multi ? k_pass<MODEL, LAYOUT, T, true, true> : k_pass<MODEL, LAYOUT, T, true, false>;
      if constexpr (LAYOUT == 0 && sizeof(T) == 4) {
        // tile shapes the cross-validation tuner may pick
        if (P.tile_form == 1)
          kp = multi ? k_pass<MODEL, LAYOUT, T, true, true, 1> : k_pass<MODEL, LAYOUT, T, true, false, 1>;
        if (P.tile_form == 2)
          kp = multi ? k_pass<MODEL, LAYOUT, T, true, true, 2> : k_pass<MODEL, LAYOUT, T, true, false, 2>;
      }
      kt = k_btrans<MODEL, LAYOUT, T, kBtSmall, true>;
      ct.gridDim = dim3(btrans_ctas_batch(P.K), P.nfit);
      ct.blockDim = dim3(kBtSmall);
    } else if (multi) {
      kp = k_pass<MODEL, LAYOUT, T, false, true>;
    }
  } else {
    if (many || few_rows) kp = k_pass<MODEL, LAYOUT, T, false, true>;
    if (P.nfit > 0) {
      cudaGraph_t junk = nullptr;
      cudaStreamEndCapture(cs, &junk);
      if (junk) cudaGraphDestroy(junk);
      return cudaErrorInvalidValue;
    }
  }
  cudaError_t lst = cudaSuccess;
  for (int j = 0; j < P.p && lst == cudaSuccess; ++j) {
    lst = cudaLaunchKernelEx(&cp, kp, P, j);
    if (lst == cudaSuccess) lst = cudaLaunchKernelEx(&ct, kt, P, j);
  }
  st = cudaStreamEndCapture(cs, g);
  return lst != cudaSuccess ? lst : st;
}

}  // namespace

#define SURV_DISPATCH_G(FN, ...)                                             \
  do {                                                                       \
    if (model == 0 && layout == 0 && prec == 0) return FN<0, 0, float>(__VA_ARGS__);  \
    if (model == 0 && layout == 0 && prec == 1) return FN<0, 0, double>(__VA_ARGS__); \
    if (model == 0 && layout == 1 && prec == 0) return FN<0, 1, float>(__VA_ARGS__);  \
    if (model == 0 && layout == 1 && prec == 1) return FN<0, 1, double>(__VA_ARGS__); \
    if (model == 1 && layout == 0 && prec == 0) return FN<1, 0, float>(__VA_ARGS__);  \
    if (model == 1 && layout == 0 && prec == 1) return FN<1, 0, double>(__VA_ARGS__); \
    if (model == 1 && layout == 1 && prec == 0) return FN<1, 1, float>(__VA_ARGS__);  \
    if (model == 1 && layout == 1 && prec == 1) return FN<1, 1, double>(__VA_ARGS__); \
    return cudaErrorInvalidValue;                                            \
  } while (0)

namespace {
cudaError_t capture_any(int model, int layout, int prec, const CcdParams& P, bool pdl, cudaStream_t cs,
                        cudaGraph_t* g) {
  SURV_DISPATCH_G(capture_sweep, P, pdl, cs, g);
}
}  // namespace

cudaError_t graph_grid_size(int model, int layout, int prec, int* G, int* wpc) {
  SURV_DISPATCH_G(grid_graph, G, wpc);
}

cudaError_t graph_init(const CcdParams& P, cudaStream_t s) {
  k_graph_init<<<dim3(1, P.nfit > 0 ? P.nfit : 1), 32, 0, s>>>(P);
  return cudaGetLastError();
}

void graph_cache_free(GraphCache* gc) {
  if (!gc) return;
  if (gc->exec) cudaGraphExecDestroy(gc->exec);
  for (auto& e : gc->ev)
    if (e) cudaEventDestroy(e);
  if (gc->flag) cudaFreeHost(gc->flag);
  if (gc->cs) cudaStreamDestroy(gc->cs);
  *gc = GraphCache();
}

cudaError_t time_one_sweep(int model, int layout, int prec, const CcdParams& P, cudaStream_t s, float* ms) {
  *ms = 0.f;
  GraphCache gc;
  struct Guard {
    GraphCache* g;
    cudaGraph_t graph = nullptr;
    cudaEvent_t a = nullptr, b = nullptr;
    ~Guard() {
      if (graph) cudaGraphDestroy(graph);
      if (a) cudaEventDestroy(a);
      if (b) cudaEventDestroy(b);
      graph_cache_free(g);
    }
  } guard{&gc};
  cudaError_t st;
  if ((st = cudaStreamCreateWithFlags(&gc.cs, cudaStreamNonBlocking)) != cudaSuccess) return st;
  const bool pdl = !P.no_pdl;
  if ((st = capture_any(model, layout, prec, P, pdl, gc.cs, &guard.graph)) != cudaSuccess) return st;
  if ((st = cudaGraphInstantiate(&gc.exec, guard.graph, 0)) != cudaSuccess) return st;
  if ((st = cudaEventCreate(&guard.a)) != cudaSuccess) return st;
  if ((st = cudaEventCreate(&guard.b)) != cudaSuccess) return st;
  if ((st = cudaEventRecord(guard.a, s)) != cudaSuccess) return st;
  if ((st = cudaGraphLaunch(gc.exec, s)) != cudaSuccess) return st;
  if ((st = cudaEventRecord(guard.b, s)) != cudaSuccess) return st;
  if ((st = cudaEventSynchronize(guard.b)) != cudaSuccess) return st;
  return cudaEventElapsedTime(ms, guard.a, guard.b);
}

cudaError_t graph_cache_prepare(GraphCache* gc) {
  if (gc->cs) return cudaSuccess;
  cudaError_t st;
  if ((st = cudaStreamCreateWithFlags(&gc->cs, cudaStreamNonBlocking)) != cudaSuccess) return st;
  for (auto& e : gc->ev)
    if ((st = cudaEventCreateWithFlags(&e, cudaEventDisableTiming)) != cudaSuccess) return st;
  return cudaMallocHost(&gc->flag, 2 * sizeof(int));
}

cudaError_t replay_until_stop(const CcdParams& P, cudaStream_t s, GraphCache* gc, cudaEvent_t t0,
                              int launches_per_replay, int* replays, int* launches, int max_replays_in) {
  cudaError_t st;
  gc->flag[0] = gc->flag[1] = 0;
  if (t0 && (st = cudaEventRecord(t0, s)) != cudaSuccess) return st;
  // One replay per sweep.  The stop flag of replay i is read while replay
  // i + 1 runs; kernels of a replay after the stop return at once.  The
  // device stops at the evaluation of sweep max_sweeps at the latest, which
  // falls in replay max_sweeps.  A batched launch ends when every fit has
  // counted itself as stopped.
  const int max_replays = max_replays_in > 0 ? max_replays_in : P.max_sweeps + 2;
  const int target = P.nfit > 0 ? P.nfit : 1;
  const void* stop_src =
      P.nfit > 0 ? static_cast<const void*>(P.done_count) : static_cast<const void*>(&P.gctl->done);
  int i = 0;
  for (; i < max_replays; ++i) {
    if ((st = cudaGraphLaunch(gc->exec, s)) != cudaSuccess) return st;
    *launches += launches_per_replay;
    if ((st = cudaMemcpyAsync(gc->flag + (i & 1), stop_src, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
      return st;
    if ((st = cudaEventRecord(gc->ev[i & 1], s)) != cudaSuccess) return st;
    if (i >= 1) {
      if ((st = cudaEventSynchronize(gc->ev[(i - 1) & 1])) != cudaSuccess) return st;
      if (gc->flag[(i - 1) & 1] >= target) {
        ++i;
        break;
      }
    }
  }
  *replays = i;
  // the last replay's flag copy must land before the host buffer is reused
  return cudaEventSynchronize(gc->ev[(i - 1) & 1]);
}

cudaError_t run_ccd_graph(int model, int layout, int prec, const CcdParams& P, cudaStream_t s, GraphCache* gc,
                          cudaEvent_t t0, int* replays, int* launches) {
  *replays = 0;
  *launches = 0;
  GraphCache local;
  struct LocalGuard {
    GraphCache* g;
    ~LocalGuard() { graph_cache_free(g); }
  } guard{gc ? nullptr : &local};
  if (!gc) gc = &local;
  cudaError_t st;
  if ((st = graph_cache_prepare(gc)) != cudaSuccess) return st;
  // programmatic dependent launch between the kernels; SURV_FLAG_NO_PDL
  // turns it off (plain stream order), for comparison
  const bool pdl = !P.no_pdl;
  const int mlp = (model * 4 + layout * 2 + prec) * 2 + (pdl ? 1 : 0);
  if (!gc->exec || gc->mlp != mlp || std::memcmp(&gc->key, &P, sizeof(P)) != 0) {
    if (gc->exec) {
      cudaGraphExecDestroy(gc->exec);
      gc->exec = nullptr;
    }
    // capture on a private stream (the caller's may be the legacy stream)
    cudaGraph_t g = nullptr;
    st = capture_any(model, layout, prec, P, pdl, gc->cs, &g);
    if (st == cudaSuccess) st = cudaGraphInstantiate(&gc->exec, g, 0);
    if (g) cudaGraphDestroy(g);
    if (st != cudaSuccess) {
      gc->exec = nullptr;
      return st;
    }
    gc->key = P;
    gc->mlp = mlp;
  }
  return replay_until_stop(P, s, gc, t0, 2 * P.p, replays, launches);
}

}  // namespace survgpu
