// CCD for cohorts that a few SMs hold (Sections 2.4 and 2.7): one kernel on
// one thread-block cluster runs whole sweeps.
//
// At these sizes the kernel pair of ccd_graph.cu is bound by its dependent
// steps, not by bytes: two launches a coordinate, an aggregate and a partial
// exchange through L2, a ticket, and replays that run empty after the stop
// (17 to 30 us a coordinate whatever the size).  Here the CTAs of one cluster
// exchange through distributed shared memory and the hardware's cluster
// barrier, and every CTA takes the Newton step itself from the same numbers in
// the same order, so a coordinate needs two cluster barriers and nothing else
// (8 to 25 us, in FP64 11 to 45; its row pass, on 16 SMs instead of 152, is the longest part,
// the two barriers take 1 us):
//
//   rows     each warp updates and passes over its own rows (warp_pass, the
//            same code as the kernel pair); warp totals -> the CTA's aggregate,
//            stored into every CTA of the cluster; barrier
//   ends     prefix of the CTAs before, steps 3-4 at the CTA's group ends,
//            the CTA's three partial sums stored into every CTA; barrier
//   step     the partials summed in rank order, trust-region Newton step
//
// The barrier is hardware and the CTAs of a cluster run together, so there
// is no wait that could fail to end.  A launch runs a bounded number of
// sweeps; the state goes back to the control line, and the host launches
// again until the fit reports its stop.
#include <algorithm>
#include <cmath>

#include "graph_common.cuh"

namespace survgpu {
namespace {

using namespace ccdk;

constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClMax = 16;    // CTAs of the cluster (8 where 16 cannot be placed)
constexpr int kClMaxP = 1024; // coordinate scalars in shared memory: 32 bytes each

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// 16-byte loads per lane a tile: a warp holds few rows, and rows that a tile
// has beyond them are worked on all the same, which costs most in FP64
// (sparse Cox, ms a fit with 1, 2 and 4 loads: 4.83, 4.91, 5.16 at 20,000 x
// 100; 5.42, 4.94, 4.75 at 200,000)
template <typename T>
struct ClCfg {
  static constexpr int U = sizeof(T) == 8 ? 1 : 2;
  static constexpr int SR = 4;
};

// ONE: a single evaluation, which takes its group ends in FP64 (FP32 mode), as
// the persistent kernel does: H - G^2 cancels where a covariate varies little
// against its mean, and float-float has 9 bits fewer for it.  (A kernel of its
// own: as a branch it cost fits of dense Fine-Gray 5 %.)
template <int MODEL, int LAYOUT, typename T, bool MULTI, bool ONE>
__global__ void __launch_bounds__(kClThreads, 1) k_cluster(const __grid_constant__ CcdParams P, int sweeps) {
  using A = typename AccOf<T>::type;
  using C = Cfg<MODEL, LAYOUT, T>;
  constexpr int M = C::M;
  constexpr int U = ClCfg<T>::U, SR = ClCfg<T>::SR;
  extern __shared__ double s_coord[];   // beta, width, lambda * penalty factor, delta^T X of each coordinate
  __shared__ A s_wtot[kClWarps][M];     // warp totals (components of an unchanged e stay)
  __shared__ A s_base[kClWarps][M];     // sums of the rows before each warp
  __shared__ A s_tot[3];                // Fine-Gray: grand totals of the weighted components
  __shared__ A s_agg[kClMax][M];        // every CTA's totals (written by the CTAs)
  __shared__ A s_part[kClMax][3];       // every CTA's partial sums (written by the CTAs)
  __shared__ A s_red[kClWarps][3];
  __shared__ double s_lin[2], s_applied;
  __shared__ float s_delta[2];
  __shared__ int s_stop;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int rank = (int)cluster_rank(), CL = P.G, WPC = P.wpc, p = P.p;
  const int64_t n = P.n, nwords = (n + 31) >> 5;
  const bool rows = w < WPC;            // warps that hold rows
  const int gw = rank * WPC + (rows ? w : 0);
  const int64_t word_lo = min((int64_t)gw * P.wpw, nwords), word_hi = min(word_lo + P.wpw, nwords);
  const int64_t row_lo = word_lo * 32, row_hi = min(word_hi * 32, n);
  const int kc_lo = P.wk0[rank * WPC], kc_hi = P.wk0[(rank + 1) * WPC];
  double *s_beta = s_coord, *s_width = s_coord + p, *s_pen = s_coord + 2 * p, *s_dtx = s_coord + 3 * p;
  for (int i = tid; i < p; i += kClThreads) {
    s_beta[i] = P.beta[i];
    s_width[i] = P.width[i];
    s_pen[i] = P.pen[i];
    s_dtx[i] = P.dTx[i];
  }
  const CtlLine* L = &P.gctl->line[0];
  double applied = L->applied;
  ff delta = {L->delta_hi, L->delta_lo};
  int nevals = L->nevals, stop = L->stop;
  double f_prev = L->f_prev;
  long long passes = L->passes, eta_updates = L->eta_updates;
  // The first pass of a launch forms every component: the warp totals of an
  // unchanged e are kept in shared memory, which a launch finds undefined.
  bool fresh = true;
  if (stop) return;   // the same in every CTA
  // the group end that thread tid takes first
  int d1 = 0, wl1 = 0;
  double g1 = 0.0;
  float2 gf1 = make_float2(0.f, 0.f);
  if (kc_lo + tid < kc_hi) {
    const int k = kc_lo + tid;
    d1 = P.dk[k];
    wl1 = (int)((P.gend[k] >> 5) / P.wpw) - rank * WPC;
    if (MODEL == 1) {
      g1 = P.Gk[k];
      gf1 = P.Gkff[k];
    }
  }
  constexpr bool kFuse = LAYOUT == 1 && sizeof(T) == 4;
  A* rec = reinterpret_cast<A*>(P.rec);
  const bool single = P.single_j >= 0;
  int j = single ? P.single_j : 0;
  PassPrefetch<T, SR> pf;
  if (rows) pass_prefetch<LAYOUT, T, SR>(P, j, gw, pf);
  __syncthreads();
  cluster_arrive();   // every CTA of the cluster has started: its shared memory may be written
  cluster_wait();
  if (passes == 0 && rows) {
    // a fit's first launch: eta = X beta and e on the warp's own rows, a column at a time (a launch
    // per nonzero coefficient outside cost more than the evaluation it prepared)
    using E = typename std::conditional<sizeof(T) == 4, float2, double>::type;
    for (int64_t r = row_lo + lane; r < row_hi; r += 32) {
      reinterpret_cast<E*>(P.eta)[r] = E{};
      reinterpret_cast<T*>(P.e)[r] = T(1);
    }
    __syncwarp();
    for (int i = 0; i < p; ++i) {
      const double b = s_beta[i];
      if (b != 0.0) warp_update<LAYOUT, T>(P, i, gw, row_lo, row_hi, b, d_to_ff(b));
    }
  }

  for (int sw = 0; sw < sweeps && !stop;) {
    const int q = j == 0 ? p - 1 : j - 1;
    const bool eval = j == 0 || single;
    const bool dense = LAYOUT == 1 || applied != 0.0 || fresh;
    // ------------------------------------------------ steps 1-2, own rows
    if (rows) {
      if (applied != 0.0 && !kFuse) warp_update<LAYOUT, T>(P, q, gw, row_lo, row_hi, applied, delta);
      const T* xq = (kFuse && applied != 0.0) ? reinterpret_cast<const T*>(P.X) + (size_t)q * P.ld : nullptr;
      A tot[M];
      warp_pass<MODEL, LAYOUT, T, U, SR, MULTI, true>(P, j, row_lo, row_hi, rec, tot, pf, dense, xq, delta);
      if (lane == 0)
#pragma unroll
        for (int m = 0; m < M; ++m)
          if (dense || !(m == 0 || m == 3)) s_wtot[w][m] = tot[m];
    }
    __syncthreads();
    A wex[M];
    if (w == 0) {
      A v[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        acc_zero(v[m]);
        if (lane < WPC) v[m] = s_wtot[lane][m];
      }
      warp_scan_n<M>(v, lane);
#pragma unroll
      for (int m = 0; m < M; ++m) {
        wex[m] = shfl_up(v[m], 1);
        if (lane == 0) acc_zero(wex[m]);
        const A t = shfl_idx(v[m], WPC - 1);
        if (lane < CL) store_remote(&s_agg[rank][m], lane, pack8(t));
      }
    }
    cluster_arrive();
    cluster_wait();
    if (w == 0) {
      A v[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        acc_zero(v[m]);
        if (lane < CL) v[m] = s_agg[lane][m];
      }
      warp_scan_n<M>(v, lane);
#pragma unroll
      for (int m = 0; m < M; ++m) {
        A before = shfl_idx(v[m], rank > 0 ? rank - 1 : 0);
        if (rank == 0) acc_zero(before);
        const A all = shfl_idx(v[m], CL - 1);
        if (lane < WPC) s_base[lane][m] = acc_add(before, wex[m]);
        if (MODEL == 1 && m >= 3 && lane == 0) s_tot[m % 3] = all;
      }
    }
    __syncthreads();
    // ------------------------------------------------ steps 3-4, own ends
    A fg1, fg2;
    acc_zero(fg1);
    acc_zero(fg2);
    double pg1 = 0.0, pg2 = 0.0, pl = 0.0;
    for (int k = kc_lo + tid; k < kc_hi; k += kClThreads) {
      int d = d1, wl = wl1;
      double g = g1;
      float2 gf = gf1;
      if (k != kc_lo + tid) {
        d = P.dk[k];
        wl = (int)((P.gend[k] >> 5) / P.wpw) - rank * WPC;
        if (MODEL == 1) {
          g = P.Gk[k];
          gf = P.Gkff[k];
        }
      }
      if (d == 0) continue;
      A Pm[M];
#pragma unroll
      for (int m = 0; m < M; ++m) Pm[m] = acc_add(s_base[wl][m], rec[(size_t)k * M + m]);
      if constexpr (ONE) {
        double den = acc_to_d(Pm[0]), num1 = acc_to_d(Pm[1]), num2 = acc_to_d(Pm[2]);
        if (MODEL == 1) {
          den += g * (acc_to_d(s_tot[0]) - acc_to_d(Pm[3 % M]));
          num1 += g * (acc_to_d(s_tot[1]) - acc_to_d(Pm[4 % M]));
          num2 += g * (acc_to_d(s_tot[2]) - acc_to_d(Pm[5 % M]));
        }
        const double inv = 1.0 / den;
        const double Gr = num1 * inv, H = num2 * inv;
        pg1 += d * Gr;
        pg2 += d * (H - Gr * Gr);
        pl += d * log(den);
        continue;
      }
      A den = Pm[0], num1 = Pm[1], num2 = Pm[2];
      if (MODEL == 1) {
        const A gg = acc_base<A>(g, ff{gf.x, gf.y});
        den = acc_add(den, acc_mul(gg, acc_add(s_tot[0], acc_neg(Pm[3 % M]))));
        num1 = acc_add(num1, acc_mul(gg, acc_add(s_tot[1], acc_neg(Pm[4 % M]))));
        num2 = acc_add(num2, acc_mul(gg, acc_add(s_tot[2], acc_neg(Pm[5 % M]))));
      }
      const A inv = acc_recip(den);
      const A Gr = acc_mul(num1, inv);
      const A H = acc_mul(num2, inv);
      fg1 = acc_add(fg1, acc_scale(Gr, d));
      fg2 = acc_add(fg2, acc_scale(acc_add(H, acc_neg(acc_mul(Gr, Gr))), d));
      if (eval) pl += (double)d * log(acc_to_d(den));
    }
    if constexpr (ONE) {
      fg1 = acc_from_d(pg1, (A*)nullptr);
      fg2 = acc_from_d(pg2, (A*)nullptr);
    }
    const int nred = min((kc_hi - kc_lo + 31) >> 5, kClWarps);   // warps that had ends
    if (w < nred) {
      A r[3] = {fg1, fg2, eval ? acc_from_d(pl, (A*)nullptr) : A{}};
      warp_sum_n<3>(r);
      if (lane == 0)
#pragma unroll
        for (int i = 0; i < 3; ++i) s_red[w][i] = r[i];
    }
    __syncthreads();
    if (w == 0) {
      A r[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        acc_zero(r[i]);
        if (lane < nred) r[i] = s_red[lane][i];
      }
      warp_sum_n<3>(r);
      if (lane < CL)
#pragma unroll
        for (int i = 0; i < 3; ++i) store_remote(&s_part[rank][i], lane, pack8(r[i]));
    } else if (w == 1 && eval) {
      // pieces of the objective at the current beta, in the order of warp_lin_pen
      double lin = 0.0, pen = 0.0;
      for (int i = lane; i < p; i += 32) {
        const double b = s_beta[i];
        lin += b * s_dtx[i];
        if (P.penalty == 1) pen -= s_pen[i] * fabs(b);
        else if (P.penalty == 2) pen -= s_pen[i] * b * b * 0.5;
      }
      lin = warp_sum(lin);
      pen = warp_sum(pen);
      if (lane == 0) {
        s_lin[0] = lin;
        s_lin[1] = pen;
      }
    }
    cluster_arrive();
    // the next coordinate's column entries do not depend on this step
    const int jn = j + 1 < p ? j + 1 : 0;
    if (rows && !single) pass_prefetch<LAYOUT, T, SR>(P, jn, gw, pf);
    cluster_wait();
    // ------------------------------------------------ the step (every CTA)
    if (w == 0) {
      A r[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        acc_zero(r[i]);
        if (lane < CL) r[i] = s_part[lane][i];
      }
      warp_sum_n<3>(r);
      if (lane == 0) {
        const double grad = s_dtx[j] - acc_to_d(r[0]), hess = -acc_to_d(r[1]);
        int st = 0;
        double ap = 0.0;
        if (eval) {
          const double ll = s_lin[0] - acc_to_d(r[2]);
          const double f = ll + s_lin[1];
          const double fp = nevals >= 1 ? f_prev : 0.0;
          const bool conv = nevals >= 1 && fabs(f - fp) / fabs(f) < P.tol;
          st = (single || conv || nevals >= P.max_sweeps) ? 1 : 0;
          if (st && rank == 0) {
            P.out[OUT_LOGLIK] = ll;
            P.out[OUT_OBJECTIVE] = f;
            P.out[OUT_OBJECTIVE_PREV] = fp;
            P.out[OUT_SWEEPS] = (double)nevals;
            P.out[OUT_CONVERGED] = conv ? 1.0 : 0.0;
            P.out[OUT_ETA_UPDATES] = (double)eta_updates;
            P.out[OUT_PASSES] = (double)(passes + 1);
            P.out[OUT_GRAD] = grad;
            P.out[OUT_HESS] = hess;
            P.gctl->done = 1;
          }
          ++nevals;
          f_prev = f;
        }
        ++passes;
        if (!st) {
          const double b = s_beta[j], wd = s_width[j];
          const double step = newton_step(b, grad, hess, P.penalty, s_pen[j]);
          if (step != 0.0) ap = copysign(fmin(fabs(step), wd), step);
          s_beta[j] = b + ap;
          s_width[j] = fmax(2.0 * fabs(ap), wd / 2.0);
          if (ap != 0.0) ++eta_updates;
        }
        const ff df = d_to_ff(ap);
        s_applied = ap;
        s_delta[0] = df.hi;
        s_delta[1] = df.lo;
        s_stop = st;
      }
    }
    __syncthreads();
    applied = s_applied;
    delta = {s_delta[0], s_delta[1]};
    stop = s_stop;
    fresh = false;
    if (!stop && jn == 0) ++sw;
    if (!stop) j = jn;
  }
  // the state for the next launch
  if (rank == 0) {
    for (int i = tid; i < p; i += kClThreads) {
      P.beta[i] = s_beta[i];
      P.width[i] = s_width[i];
    }
    if (tid == 0) {
      CtlLine* W = &P.gctl->line[0];
      W->stop = stop;
      W->nevals = nevals;
      W->applied = applied;
      W->delta_hi = delta.hi;
      W->delta_lo = delta.lo;
      W->f_prev = f_prev;
      W->passes = passes;
      W->eta_updates = eta_updates;
      W->dirty = 0;
    }
  }
}

// Form of the row pass: the many-ends form where warps hold two group ends or
// more on average, and where fewer crowd into the warps of the latest times,
// whose way through them one after another is then the pass: always in FP64,
// and in FP32 from 96 ends if a warp has a whole tile of rows (with fewer rows a
// lane's FP32 sums would be longer than the 4 rows of the other form).  us a
// coordinate, ends one after another and the many-ends form: FP64 dense
// Cox 22.9 and 20.3 for 60 ends of 16,384 rows, 55.9 and 21.1 for 359
// (Fine-Gray 97.5 and 32.2); FP32 dense Fine-Gray 17.9 and 18.4 for 60 ends of
// 70,000 rows, 21.2 and 20.4 for 100, 40.2 and 22.6 for 365; sparse Cox 12.9
// and 13.7 for 60 ends of 300,000 rows, 15.0 and 14.7 for 100, 26.2 and 15.9
// for 365.
bool many_ends(int prec, int64_t K, int64_t nwarps, int64_t wpw) {
  return prec == 1 || K >= 2 * nwarps || (K >= 96 && wpw >= 8);
}

template <int MODEL, int LAYOUT, typename T>
cudaError_t cluster_size_of(int* G) {
  static_assert(kClWarps <= 32 && kClMax <= 32, "one lane per warp and per CTA");
  auto k = k_cluster<MODEL, LAYOUT, T, true, false>;
  *G = 0;
  cudaError_t st = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (st != cudaSuccess) return st;
  for (int cl : {kClMax, 8}) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)cl, 1, 1};
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(cl);
    c.blockDim = dim3(kClThreads);
    c.dynamicSmemBytes = 4 * sizeof(double) * kClMaxP;
    c.attrs = at;
    c.numAttrs = 1;
    int num = 0;
    if (cudaOccupancyMaxActiveClusters(&num, k, &c) == cudaSuccess && num >= 1) {
      *G = cl;
      return cudaSuccess;
    }
    cudaGetLastError();
  }
  return cudaSuccess;
}

template <int MODEL, int LAYOUT, typename T>
cudaError_t launch_cluster(const CcdParams& P, int sweeps, cudaStream_t s) {
  auto k = k_cluster<MODEL, LAYOUT, T, true, false>;
  if constexpr (sizeof(T) == 4) {
    const bool many = many_ends(0, P.K, P.nwarps, P.wpw);
    if (P.single_j >= 0) k = many ? k_cluster<MODEL, LAYOUT, T, true, true> : k_cluster<MODEL, LAYOUT, T, false, true>;
    else if (!many) k = k_cluster<MODEL, LAYOUT, T, false, false>;
  }
  cudaError_t st = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (st != cudaSuccess) return st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)P.G, 1, 1};
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(P.G);
  c.blockDim = dim3(kClThreads);
  c.dynamicSmemBytes = 4 * sizeof(double) * (size_t)P.p;
  c.stream = s;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, k, P, sweeps);
}

#define SURV_DISPATCH_CL(FN, ...)                                                          \
  do {                                                                                     \
    if (model == 0 && layout == 0 && prec == 0) return FN<0, 0, float>(__VA_ARGS__);       \
    if (model == 0 && layout == 0 && prec == 1) return FN<0, 0, double>(__VA_ARGS__);      \
    if (model == 0 && layout == 1 && prec == 0) return FN<0, 1, float>(__VA_ARGS__);       \
    if (model == 0 && layout == 1 && prec == 1) return FN<0, 1, double>(__VA_ARGS__);      \
    if (model == 1 && layout == 0 && prec == 0) return FN<1, 0, float>(__VA_ARGS__);       \
    if (model == 1 && layout == 0 && prec == 1) return FN<1, 0, double>(__VA_ARGS__);      \
    if (model == 1 && layout == 1 && prec == 0) return FN<1, 1, float>(__VA_ARGS__);       \
    if (model == 1 && layout == 1 && prec == 1) return FN<1, 1, double>(__VA_ARGS__);      \
    return cudaErrorInvalidValue;                                                          \
  } while (0)

// us a coordinate of a fit in one cluster,
//   fixed + row n/10^5 + many n/10^5 + end E/1000          (the many-ends form)
//         + serial max(0, W - 5)/10                         (the other form)
//         + (entry + entry_end f) nnz/10^4,                 (CSC)
// E the group ends of its busiest CTA and W of its busiest warp, both bounded by
// the rows, by K (0.4 and 0.12 of it for exponential times) and by `crowd`, the
// most ends among 32 rows; f = min(1, K/300) min(1, (crowd + 1)/3) the share of
// entry rounds with an end.  Of the kernel pair on the whole chip:
// other + other_log log2 K, where n hardly counts.  Least squares over 5,100
// fits of 300 to 300,000 rows with exponential, censored and uniform times, 40 to
// 39,000 ends and 0.5 to 50 % density: 4 to 9 % rms (the cluster on sparse data in
// FP32 14 to 15, the pair on sparse Fine-Gray 11).  The choice between the two
// costs 0 to 1.1 % on average against the faster one (up to 56 % for single fits
// next to the line), and at most 12 % more than the schedule that stood before
// the cluster (20 fits more than 5 %).  Limits on n and on K alone lost
// where both were near them or columns dense (ms a fit, cluster and pair: 7.6
// and 1.6 for sparse Cox at 300,000 x 60 with half of the entries stored, 9.8
// and 8.7 at 5 % with 27,000 ends; 7.5 and 4.3 for sparse Fine-Gray at 262,000 x
// 40 with half of the entries).
struct FitCost {
  double fixed, row, many, end, serial, entry, entry_end, other, other_log;
};
constexpr FitCost kFitCost[2][2][2] = {   // model, layout, precision
    {{{9.6, 0.8, 0.4, 2.4, 5.0, 0.3, 1.75, 4.0, 1.16}, {12.3, 19.0, 0.0, 6.0, 0.0, 3.0, 2.0, 21.5, 0.65}},
     {{9.7, 0.8, 3.6, 3.0, 5.0, 0.0, 0.0, 11.0, 0.64}, {10.7, 60.0, 0.0, 5.9, 0.0, 0.0, 0.0, 22.8, 0.62}}},
    {{{14.0, 0.3, 1.8, 4.4, 8.2, 0.3, 2.8, 14.6, 0.94}, {16.8, 38.0, 0.0, 8.5, 0.0, 4.5, 5.0, 33.0, 0.95}},
     {{13.7, 0.5, 6.8, 5.1, 9.0, 0.0, 0.0, 12.8, 0.95}, {15.1, 98.0, 0.0, 8.9, 0.0, 0.0, 0.0, 33.3, 0.9}}}};

// The same in batches of four coordinates (sparse Cox, FP32).  A row pass (6 %
// rms, real values 8 %): its busiest warp walks its ends one after another, and
// streams e only after a step.  It serves the coordinates up to the first that
// steps, so with a share `moving` of them 1 / moving (1 - (1 - moving)^4), four
// where none does.
double batch_us(const FitShape& f, double moving) {
  const int64_t nwords = (f.n + 31) / 32, wpw = (nwords + f.batch_warps - 1) / f.batch_warps;
  const double dens = std::min(0.5, std::sqrt(f.nnz / (double)f.n));
  const double walk = 0.1 * (double)(f.crowd * wpw) * (0.5 + 0.5 * std::min(1.0, 3.0 * moving));
  const double pass = f.values ? 29.0 + walk * (13.0 + 26.0 * dens) : 17.6 + walk * (5.3 + 14.5 * dens);
  return pass * (moving > 0.0 ? moving / (1.0 - std::pow(1.0 - moving, 4)) : 0.25);
}

// Rows up to which the figures above hold.
int64_t cluster_rows(int prec) { return prec == 1 ? 40000 : 300000; }

// Row words a warp and row warps of a cluster of G CTAs: no more warps than the
// words need, so that the rows are spread evenly over the CTAs.
void cluster_partition(int64_t n, int G, int64_t* wpw, int* wpc) {
  const int64_t nwords = (n + 31) / 32, most = (int64_t)G * kClWarps;
  *wpw = (nwords + most - 1) / most;
  *wpc = (int)(((nwords + *wpw - 1) / *wpw + G - 1) / G);
}

}  // namespace

cudaError_t cluster_grid_size(int model, int layout, int prec, int64_t n, int64_t p, int* G, int* wpc) {
  *G = 0;
  *wpc = 0;
  if (n > cluster_rows(prec) || p > kClMaxP) return cudaSuccess;
  cudaError_t st = [&] { SURV_DISPATCH_CL(cluster_size_of, G); }();
  if (st != cudaSuccess || *G == 0) return st;
  int64_t wpw = 0;
  cluster_partition(n, *G, &wpw, wpc);
  return cudaSuccess;
}

bool cluster_is_faster(int model, int layout, int prec, const FitShape& f, double moving) {
  const FitCost& c = kFitCost[model][layout][prec];
  int64_t wpw = 0;
  int wpc = 0;
  cluster_partition(f.n, kClMax, &wpw, &wpc);
  const double rows = (double)f.n * 1e-5, K = f.K, crowd = f.crowd;
  double us = c.fixed + c.row * rows +
              (c.entry + c.entry_end * std::min(1.0, K / 300.0) * std::min(1.0, (crowd + 1.0) / 3.0)) * f.nnz * 1e-4;
  if (many_ends(prec, f.K, (int64_t)kClMax * wpc, wpw))
    us += c.many * rows + c.end * 1e-3 * std::min(std::min(0.4 * K, (double)f.n / 16.0), crowd * (double)f.n / 512.0);
  else
    us += c.serial * 0.1 * std::max(0.0, std::min(crowd * (double)wpw, 0.12 * K) - 5.0);
  if (f.batch_warps == 0) return us < c.other + c.other_log * std::log2(std::max(2.0, K));
  return us - 1.8 * (1.0 - moving) < batch_us(f, moving);   // (a zero step: no update, no walk of e)
}

cudaError_t run_cluster(int model, int layout, int prec, const CcdParams& P, int sweeps, cudaStream_t s) {
  SURV_DISPATCH_CL(launch_cluster, P, sweeps, s);
}

}  // namespace survgpu
