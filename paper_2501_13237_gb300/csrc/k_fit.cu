// a8 -- noise-strength extrapolation to lambda* in float64 (Sec. 2.2.3 (B);
// App. B.2): one thread per observable for POLY and EXP_LOGLIN (fit_kernel),
// clusters that take the observables that need EXP3 (exp3_kernel).
//   POLY(m):     least squares in t = (lambda - lambda*)/max|lambda - lambda*| by
//                Householder QR; estimate = constant coefficient.
//   EXP_LOGLIN:  criterion 2 (|y| >= 1e-10), criterion 3 (sign of the
//                lambda = 0 value, else of the smallest-lambda value); weights
//                w = F^2 exp(-20 |lambda* - lambda| / d), d = smallest lambda > 0
//                with F > 0.99 (else the lambda span); weighted line through
//                (lambda, log|y|) in the pairwise closed form (no underflow when
//                F^2 underflows); estimate = sign * exp(alpha - b lambda*).
//                Fewer than two surviving points -> EXP3 on all points.
//   EXP3:        a e^{-b lambda} + c by variable projection: (a, c) linear in b;
//                b on a 4001-point grid of [-B, B], B = 50/span, then golden
//                section on the best bracket to 1e-12 B.
// NOFIT: value at lambda* when lambda* was emulated, else NaN.
//
// Fidelity extrapolation (A) over a bond-dimension ladder D_1 < ... < D_k
// (Sec. 2.2.3 (A); App. B.1), ladder_kernel, one thread per (lambda, obs):
//   obar = least-squares line of <O>^{(D_j)} against F^{(D_j)}, at F = 1
//   (one rung: the value; equal fidelities: the mean);
//   criterion 1: |(O_k - O_{k-1}) / (F_k - F_{k-1})| (1 - F_k) < |O_k| / 2
//   (F_k = 1: left side 0; F_k = F_{k-1}: 0 if O_k = O_{k-1}, else infinite).
// The fit then sees only the levels passing criterion 1 (mask), keeps the dip
// size of all levels, and falls back to the D_k emulation at lambda*.
#include <cooperative_groups.h>

#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace nne {

constexpr int FIT_MAXL = 64;
constexpr int FIT_NEEDS_EXP3 = 1 << 20;   // status between fit_kernel and exp3_kernel
constexpr double DELTA_F = 2.0, DELTA_D = 20.0, SMALL = 1e-10, DIP_FID = 0.99;

__device__ void nofit(int nl, const double* lam, const double* y, double ls, double* est, int* st) {
  double v = nan("");
  for (int j = 0; j < nl; ++j)
    if (lam[j] == ls) { v = y[j]; break; }
  *est = v;
  *st = NNE_ERR_NOFIT;
}

__device__ void poly_fit(int nl, const double* lam, const double* y, double ls, int deg, double* est, int* st) {
  const int nc = deg + 1;
  if (nl < nc || nc > 16) { nofit(nl, lam, y, ls, est, st); return; }
  double V[FIT_MAXL][16];
  double b[FIT_MAXL];
  double scale = 0;
  for (int j = 0; j < nl; ++j) scale = fmax(scale, fabs(lam[j] - ls));
  if (scale == 0) scale = 1;
  for (int j = 0; j < nl; ++j) {
    const double t = (lam[j] - ls) / scale;
    double p = 1;
    for (int k = 0; k < nc; ++k) { V[j][k] = p; p *= t; }
    b[j] = y[j];
  }
  for (int k = 0; k < nc; ++k) {
    double xn = 0;
    for (int j = k; j < nl; ++j) xn += V[j][k] * V[j][k];
    xn = sqrt(xn);
    if (xn == 0) continue;
    const double alpha = V[k][k] >= 0 ? -xn : xn;
    double v[FIT_MAXL];
    for (int j = k; j < nl; ++j) v[j] = V[j][k];
    v[k] -= alpha;
    double vn = 0;
    for (int j = k; j < nl; ++j) vn += v[j] * v[j];
    if (vn == 0) continue;
    for (int c = k; c < nc; ++c) {
      double s = 0;
      for (int j = k; j < nl; ++j) s += v[j] * V[j][c];
      s = 2 * s / vn;
      for (int j = k; j < nl; ++j) V[j][c] -= s * v[j];
    }
    double s = 0;
    for (int j = k; j < nl; ++j) s += v[j] * b[j];
    s = 2 * s / vn;
    for (int j = k; j < nl; ++j) b[j] -= s * v[j];
  }
  double c[16];
  for (int k = nc - 1; k >= 0; --k) {
    double s = b[k];
    for (int q = k + 1; q < nc; ++q) s -= V[k][q] * c[q];
    if (V[k][k] == 0) { nofit(nl, lam, y, ls, est, st); return; }
    c[k] = s / V[k][k];
  }
  *est = c[0];
  *st = NNE_OK;
}

__device__ double exp3_profile(double b, int nl, const double* lam, const double* y, double* a_out, double* c_out) {
  double e[FIT_MAXL];
  double em = 0, ym = 0;
  for (int j = 0; j < nl; ++j) { e[j] = exp(-b * lam[j]); em += e[j]; ym += y[j]; }
  em /= nl;
  ym /= nl;
  double see = 0, sey = 0;
  for (int j = 0; j < nl; ++j) { see += (e[j] - em) * (e[j] - em); sey += (e[j] - em) * (y[j] - ym); }
  double a = see > 0 ? sey / see : 0.0;
  double c = ym - a * em;
  double loss = 0;
  for (int j = 0; j < nl; ++j) { const double r = a * e[j] + c - y[j]; loss += r * r; }
  *a_out = a;
  *c_out = c;
  return loss;
}

// EXP3 needs at least three levels that are not all equal; 50 / span otherwise.
__device__ bool exp3_range(int nl, const double* lam, double* B) {
  double lmin = 1e300, lmax = -1e300;
  for (int j = 0; j < nl; ++j) { lmin = fmin(lmin, lam[j]); lmax = fmax(lmax, lam[j]); }
  const double span = nl > 0 ? lmax - lmin : 0;
  if (nl < 3 || !(span > 0)) return false;
  *B = 50.0 / span;
  return true;
}

__device__ void loglin_fit(int nl, const double* lam, const double* y, const double* logf, double ls,
                           const double* yzero, int o, double dgiven, double* est, int* st) {
  // (*st = FIT_NEEDS_EXP3: fewer than two levels survive, or all survivors share one lambda)
  int jmin = 0;
  for (int j = 1; j < nl; ++j)
    if (lam[j] < lam[jmin]) jmin = j;
  const double ref = yzero ? (yzero[o] >= 0 ? 1.0 : -1.0) : (y[jmin] >= 0 ? 1.0 : -1.0);
  bool keep[FIT_MAXL];
  int nk = 0;
  for (int j = 0; j < nl; ++j) {
    const double sg = y[j] > 0 ? 1.0 : (y[j] < 0 ? -1.0 : 0.0);
    keep[j] = fabs(y[j]) >= SMALL && sg == ref;
    nk += keep[j];
  }
  if (nk < 2) { *st = FIT_NEEDS_EXP3; return; }
  // dip size over all supplied levels (given by the caller when the fit sees a subset)
  double d = dgiven > 0 ? dgiven : 1e300;
  bool found = dgiven > 0;
  for (int j = 0; j < nl && dgiven <= 0; ++j) {
    const double F = exp(logf ? logf[j] : 0.0);
    if (lam[j] > 0 && F > DIP_FID && lam[j] < d) { d = lam[j]; found = true; }
  }
  if (!found) {
    double lmin = 1e300, lmax = -1e300;
    for (int j = 0; j < nl; ++j) { lmin = fmin(lmin, lam[j]); lmax = fmax(lmax, lam[j]); }
    d = lmax - lmin > 0 ? lmax - lmin : 1.0;
  }
  double lw2[FIT_MAXL], x[FIT_MAXL], zz[FIT_MAXL];
  int m = 0;
  for (int j = 0; j < nl; ++j) {
    if (!keep[j]) continue;
    const double lf = logf ? logf[j] : 0.0;
    lw2[m] = 2.0 * (DELTA_F * lf - DELTA_D * fabs(ls - lam[j]) / d);
    x[m] = lam[j];
    zz[m] = log(fabs(y[j]));
    ++m;
  }
  double lpmax = -1e308;
  bool any = false;
  for (int i = 0; i < m; ++i)
    for (int j = i + 1; j < m; ++j)
      if (x[i] != x[j]) { lpmax = fmax(lpmax, lw2[i] + lw2[j] + 2.0 * log(fabs(x[i] - x[j]))); any = true; }
  if (!any) { *st = FIT_NEEDS_EXP3; return; }
  double num = 0, den = 0;
  for (int i = 0; i < m; ++i)
    for (int j = i + 1; j < m; ++j)
      if (x[i] != x[j]) {
        const double c = exp(lw2[i] + lw2[j] + 2.0 * log(fabs(x[i] - x[j])) - lpmax);
        num += c * (zz[i] - zz[j]) / (x[i] - x[j]);
        den += c;
      }
  const double slope = num / den;
  double lwmax = -1e308;
  for (int i = 0; i < m; ++i) lwmax = fmax(lwmax, lw2[i]);
  double sw = 0, swz = 0;
  for (int i = 0; i < m; ++i) {
    const double W = exp(lw2[i] - lwmax);
    sw += W;
    swz += W * (zz[i] - slope * x[i]);
  }
  const double alpha = swz / sw;
  *est = ref * exp(alpha + slope * ls);
  *st = NNE_OK;
}

__device__ double dip_all(int nl, const double* lam, const double* logf) {
  double d = 1e300;
  bool found = false;
  for (int j = 0; j < nl; ++j) {
    const double F = exp(logf ? logf[j] : 0.0);
    if (lam[j] > 0 && F > DIP_FID && lam[j] < d) { d = lam[j]; found = true; }
  }
  if (found) return d;
  double lmin = 1e300, lmax = -1e300;
  for (int j = 0; j < nl; ++j) { lmin = fmin(lmin, lam[j]); lmax = fmax(lmax, lam[j]); }
  return lmax - lmin > 0 ? lmax - lmin : 1.0;
}

// The levels of observable o that the fit may use (mask null: all): count.
__device__ int gather_levels(int nl, const double* lam, const double* vals, const double* logf, int n_obs, int o,
                             const uint8_t* mask, double* y, double* lc, double* fc) {
  int m = 0;
  for (int j = 0; j < nl; ++j) {
    if (mask && !mask[(long long)j * n_obs + o]) continue;
    y[m] = vals[(long long)j * n_obs + o];
    lc[m] = lam[j];
    if (fc) fc[m] = logf ? logf[j] : 0.0;
    ++m;
  }
  return m;
}

// NOFIT of a masked fit: the value at lambda* over all levels.
__device__ void store_fit(int nl, const double* lam, const double* vals, int n_obs, int o, double ls,
                          const uint8_t* mask, const double* fb, double est, int st, double* out, int* status) {
  if (st == NNE_ERR_NOFIT && (fb || mask)) {
    const double* src = fb ? fb : vals;
    est = nan("");
    for (int j = 0; j < nl; ++j)
      if (lam[j] == ls) { est = src[(long long)j * n_obs + o]; break; }
  }
  out[o] = est;
  status[o] = st;
}

// mask (nl x n_obs, lambda-major; null: every level): levels the fit may use;
// fb (nl x n_obs; null: the fitted values): where the NOFIT fallback reads the
// value at lambda*.  Observables that need EXP3 get status FIT_NEEDS_EXP3.
__global__ void fit_kernel(int nl, const double* lam, const double* vals, const double* logf, int n_obs, int method,
                           int degree, double ls, const double* yzero, const uint8_t* mask, const double* fb,
                           double* out, int* status) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= n_obs) return;
  double y[FIT_MAXL], lc[FIT_MAXL], fc[FIT_MAXL];
  const int m = gather_levels(nl, lam, vals, logf, n_obs, o, mask, y, lc, fc);
  const double dgiven = mask ? dip_all(nl, lam, logf) : -1.0;
  double est = nan("");
  int st = NNE_ERR_NOFIT;
  if (m == 0) {
    st = NNE_ERR_NOFIT;
  } else if (method == NNE_FIT_POLY) {
    poly_fit(m, lc, y, ls, degree, &est, &st);
  } else if (method == NNE_FIT_EXP_LOGLIN) {
    loglin_fit(m, lc, y, logf ? fc : nullptr, ls, yzero, o, dgiven, &est, &st);
  } else {
    st = FIT_NEEDS_EXP3;
  }
  if (st == FIT_NEEDS_EXP3) {
    status[o] = st;
    return;
  }
  store_fit(nl, lam, vals, n_obs, o, ls, mask, fb, est, st, out, status);
}

// EXP3 of the observables fit_kernel marked.  Clusters of EXP3_CS CTAs each take `per`
// neighbouring observables at a time, EXP3_CLUSTERS of them at most.
//
// Bound by float64 arithmetic, which runs at 1/64 of the float32 rate: a
// profile at one b costs about 40 operations per level (the exponential most
// of all), and the grid has 4001 points.  One thread per observable took the
// 4061 profiles one after the other: 22.7 ms for 199 observables at 5 levels
// of which a handful need EXP3.  The grid's points are independent, so they
// are dealt to the EXP3_CS x 128 threads (the best is the smallest loss, the
// lowest index among equal ones, as a scan in order finds it); the golden
// section that follows is a serial chain of about 60 profiles, each formed by
// one warp with a level per lane and the sums in level order (whole call of
// that table: 22.8 ms -> 0.3 ms).  The warp's lanes repeat each other's sums, a
// third of the work on top of the grid's: where a cluster has more than EXP3_WARP
// observables that need it (a large table), its CTAs take a grid each and a thread
// a golden section, with the same operations in the same order.  Whole calls, ms, one
// thread per observable throughout, a cluster each throughout, now: EXP3 of 50000
// observables at 5 levels 68.2, 91.2, 68.6; of 200000 250, 364, 261; a fit of 100000
// observables of which 1 % fall back 57.3, 2.6, 2.4; none of 10^6 3.3, 9.0, 3.3.
constexpr int EXP3_CS = 8, EXP3_THREADS = 128, EXP3_GRID = 4001;
constexpr int EXP3_CLUSTERS = 4 * 152, EXP3_MOST = 128, EXP3_WARP = 8;

__device__ __forceinline__ double exp3_step(double B) { return (2 * B) / (EXP3_GRID - 1); }
__device__ __forceinline__ double exp3_gridb(int i, double B, double step) {
  return (i == EXP3_GRID - 1) ? B : i * step - B;
}

// Golden section around grid point bi: the estimate at ls.  profile(b, &a, &c) is the loss.
template <typename F>
__device__ __forceinline__ double exp3_golden(int bi, double B, double step, double ls, F profile) {
  double a, c;
  double lo = exp3_gridb(max(bi - 1, 0), B, step), hi = exp3_gridb(min(bi + 1, EXP3_GRID - 1), B, step);
  const double g = (sqrt(5.0) - 1.0) / 2.0;
  double x1 = hi - g * (hi - lo), x2 = lo + g * (hi - lo);
  auto f = [&](double b) { return b == 0.0 ? 1e300 : profile(b, &a, &c); };
  double f1 = f(x1), f2 = f(x2);
  const double tol = 1e-12 * B;
  for (int it = 0; it < 200 && hi - lo > tol; ++it) {
    if (f1 <= f2) {
      hi = x2; x2 = x1; f2 = f1;
      x1 = hi - g * (hi - lo);
      f1 = f(x1);
    } else {
      lo = x1; x1 = x2; f1 = f2;
      x2 = lo + g * (hi - lo);
      f2 = f(x2);
    }
  }
  double b = 0.5 * (lo + hi);
  if (b == 0.0) b = lo;
  profile(b, &a, &c);
  return a * exp(-b * ls) + c;
}

// The golden section and the result of observable o by one thread.
__device__ __noinline__ void exp3_finish_thread(int bi, int nl, const double* lam, const double* vals, int n_obs, int o,
                                                double ls, const uint8_t* mask, const double* fb, double* out,
                                                int* status) {
  double y[FIT_MAXL], lc[FIT_MAXL], B = 0, est = 0;
  const int m = gather_levels(nl, lam, vals, nullptr, n_obs, o, mask, y, lc, nullptr);
  int st = NNE_OK;
  if (exp3_range(m, lc, &B))
    est = exp3_golden(bi, B, exp3_step(B), ls,
                      [&](double b, double* a, double* c) { return exp3_profile(b, m, lc, y, a, c); });
  else
    nofit(m, lc, y, ls, &est, &st);
  store_fit(nl, lam, vals, n_obs, o, ls, mask, fb, est, st, out, status);
}

struct Exp3Best {
  double loss;
  int at;
  __device__ __forceinline__ void take(double l, int i) {
    if (l < loss || (l == loss && i < at)) { loss = l; at = i; }
  }
};

// ONE: one observable per cluster, whose levels are gathered before the first exchange.
template <bool ONE>
__global__ void __cluster_dims__(EXP3_CS, 1, 1) __launch_bounds__(EXP3_THREADS, 8)
    exp3_kernel(int nl, const double* lam, const double* vals, int n_obs, double ls, const uint8_t* mask,
                const double* fb, double* out, int* status, int per) {
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int cl = (int)(blockIdx.x / EXP3_CS), ncl = (int)(gridDim.x / EXP3_CS);
  constexpr int NW = EXP3_THREADS / 32;
  __shared__ double ys[NW + 1][FIT_MAXL], lams[NW + 1][FIT_MAXL];   // of each warp's golden section, of the grid's observable
  __shared__ int list[EXP3_MOST], count[NW];
  __shared__ double wbest[NW];
  __shared__ int widx[NW];
  __shared__ Exp3Best best_s[EXP3_MOST / EXP3_CS][EXP3_CS];   // by observable of this CTA and CTA of the cluster
  __shared__ int m_s, ok_s;
  __shared__ double B_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double *y = ys[NW], *lc = lams[NW];
  auto levels = [&](int q) {   // of observable q of the list, by one thread
    m_s = gather_levels(nl, lam, vals, nullptr, n_obs, list[q], mask, y, lc, nullptr);
    double B = 0;
    ok_s = exp3_range(m_s, lc, &B) ? 1 : 0;
    B_s = B;
  };
  for (long long o0 = (long long)cl * per; o0 < n_obs; o0 += (long long)ncl * per) {
    int n_fit = 1;
    if (ONE) {
      if (status[o0] != FIT_NEEDS_EXP3) return;
      if (tid == 0) {
        list[0] = (int)o0;
        levels(0);
      }
    } else {
      // the marked observables, the same list in every CTA
      const bool mine = tid < per && o0 + tid < n_obs && status[o0 + tid] == FIT_NEEDS_EXP3;
      if (!__syncthreads_or(mine)) continue;
      const unsigned votes = __ballot_sync(0xffffffffu, mine);
      if (lane == 0) count[warp] = __popc(votes);
      __syncthreads();
      n_fit = 0;
      int before = 0;
      for (int w = 0; w < NW; ++w) {
        if (w < warp) before += count[w];
        n_fit += count[w];
      }
      if (mine) list[before + __popc(votes & ((1u << lane) - 1))] = (int)(o0 + tid);
    }
    // also: every CTA runs, has read its statuses and is done with best_s
    cluster.sync();
    const bool many = !ONE && n_fit > EXP3_WARP;   // then a CTA for a grid
    double step = 0;                               // of the last observable
    for (int q = many ? rank : 0; q < n_fit; q += many ? EXP3_CS : 1) {
      if (!ONE) {
        if (tid == 0) levels(q);
        __syncthreads();
      }
      const int m = m_s;
      const double B = B_s;
      if (ok_s) {
        Exp3Best best{1e300, 0};
        step = exp3_step(B);
        for (int i = (many ? 0 : rank * EXP3_THREADS) + tid; i < EXP3_GRID; i += (many ? 1 : EXP3_CS) * EXP3_THREADS) {
          const double b = exp3_gridb(i, B, step);
          double a, c;
          const double l = (b == 0.0) ? 1e300 : exp3_profile(b, m, lc, y, &a, &c);
          if (l < best.loss) { best.loss = l; best.at = i; }
        }
        for (int d = 16; d > 0; d >>= 1)
          best.take(__shfl_xor_sync(0xffffffffu, best.loss, d), __shfl_xor_sync(0xffffffffu, best.at, d));
        if (lane == 0) {
          wbest[warp] = best.loss;
          widx[warp] = best.at;
        }
        __syncthreads();
        if (tid == 0) {
          for (int w = 1; w < NW; ++w) best.take(wbest[w], widx[w]);
          if (many) best_s[q / EXP3_CS][0] = best;
          else *cluster.map_shared_rank(&best_s[q / EXP3_CS][rank], q % EXP3_CS) = best;
        }
      }
      if (!ONE) __syncthreads();   // y, lc, m_s are free
    }
    cluster.sync();
    // observable q by CTA q % EXP3_CS
    auto best_of = [&](int q) {
      Exp3Best best = best_s[q / EXP3_CS][0];
      for (int r = 1; r < (many ? 1 : EXP3_CS); ++r) best.take(best_s[q / EXP3_CS][r].loss, best_s[q / EXP3_CS][r].at);
      return best.at;
    };
    if (many) {   // a thread each
      const int q = tid * EXP3_CS + rank;
      if (q < n_fit) exp3_finish_thread(best_of(q), nl, lam, vals, n_obs, list[q], ls, mask, fb, out, status);
    } else if (warp * EXP3_CS + rank < n_fit) {   // a warp each
      const int q = warp * EXP3_CS + rank, o = list[q];
      const bool last = q == n_fit - 1;   // whose levels are still at hand
      double *yt = ys[last ? NW : warp], *lt = lams[last ? NW : warp];
      int m = m_s, st = NNE_OK;
      bool ok = ok_s;
      double B = B_s, est = 0;
      if (!last) {
        if (lane == 0) m = gather_levels(nl, lam, vals, nullptr, n_obs, o, mask, yt, lt, nullptr);
        m = __shfl_sync(0xffffffffu, m, 0);
        ok = exp3_range(m, lt, &B);
        step = exp3_step(B);
      }
      if (ok) {
        // lane j forms the exponentials of levels j and j + 32
        est = exp3_golden(best_of(q), B, step, ls, [&](double b, double* a, double* c) {
          const double e0 = lane < m ? exp(-b * lt[lane]) : 0.0, e1 = lane + 32 < m ? exp(-b * lt[lane + 32]) : 0.0;
          auto e = [&](int j) { return __shfl_sync(0xffffffffu, j < 32 ? e0 : e1, j & 31); };
          double em = 0, ym = 0;
          for (int j = 0; j < m; ++j) { em += e(j); ym += yt[j]; }
          em /= m;
          ym /= m;
          double see = 0, sey = 0;
          for (int j = 0; j < m; ++j) { const double ej = e(j); see += (ej - em) * (ej - em); sey += (ej - em) * (yt[j] - ym); }
          *a = see > 0 ? sey / see : 0.0;
          *c = ym - *a * em;
          double loss = 0;
          for (int j = 0; j < m; ++j) { const double r = *a * e(j) + *c - yt[j]; loss += r * r; }
          return loss;
        });
      } else {
        nofit(m, lt, yt, ls, &est, &st);
      }
      if (lane == 0) store_fit(nl, lam, vals, n_obs, o, ls, mask, fb, est, st, out, status);
      __syncwarp();
    }
    __syncthreads();   // list is free
  }
}

// Both kernels; the EXP3 pass only where the method can reach it.
static cudaError_t launch_fit(cudaStream_t st, int nl, const double* lam, const double* vals, const double* logf,
                              int n_obs, int method, int degree, double ls, const double* yzero, const uint8_t* mask,
                              const double* fb, double* out, int* status) {
  fit_kernel<<<(n_obs + 63) / 64, 64, 0, st>>>(nl, lam, vals, logf, n_obs, method, degree, ls, yzero, mask, fb, out,
                                              status);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || method == NNE_FIT_POLY) return e;
  // equal shares in as few passes as EXP3_MOST allows
  const long long passes = (n_obs - 1) / ((long long)EXP3_CLUSTERS * EXP3_MOST) + 1;
  const int per = (int)((n_obs - 1) / (passes * EXP3_CLUSTERS) + 1);
  const int clusters = std::min(EXP3_CLUSTERS, (n_obs - 1) / per + 1);
  (per == 1 ? exp3_kernel<true> : exp3_kernel<false>)<<<clusters * EXP3_CS, EXP3_THREADS, 0, st>>>(
      nl, lam, vals, n_obs, ls, mask, fb, out, status, per);
  return cudaGetLastError();
}

// (A) over k rungs: vals (k x nl x n_obs), logf (k x nl) -> obar (nl x n_obs), conv (nl x n_obs).
__global__ void ladder_kernel(int k, int nl, int n_obs, const double* vals, const double* logf, double* obar,
                              uint8_t* conv) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)nl * n_obs) return;
  const int i = (int)(idx / n_obs), o = (int)(idx % n_obs);
  auto O = [&](int j) { return vals[((long long)j * nl + i) * n_obs + o]; };
  auto F = [&](int j) { return exp(logf[(long long)j * nl + i]); };
  double ob;
  if (k == 1) {
    ob = O(0);
  } else {
    double fm = 0, om = 0;
    for (int j = 0; j < k; ++j) { fm += F(j); om += O(j); }
    fm /= k;
    om /= k;
    double sff = 0, sfo = 0;
    for (int j = 0; j < k; ++j) {
      const double df = F(j) - fm;
      sff += df * df;
      sfo += df * (O(j) - om);
    }
    ob = sff == 0.0 ? om : om + (sfo / sff) * (1.0 - fm);
  }
  bool c = true;
  if (k >= 2) {
    const double ok = O(k - 1), ok1 = O(k - 2), fk = F(k - 1), fk1 = F(k - 2);
    double lhs;
    if (fk == 1.0) lhs = 0.0;
    else if (fk == fk1) lhs = ok == ok1 ? 0.0 : INFINITY;
    else lhs = fabs((ok - ok1) / (fk - fk1)) * (1.0 - fk);
    c = lhs < fabs(ok) / 2.0;
  }
  obar[idx] = ob;
  conv[idx] = c ? 1 : 0;
}

cudaError_t extrapolate_fit(cudaStream_t st, int n_lambda, const double* d_lam, const double* d_vals,
                            const double* d_logfid, int n_obs, int method, int degree, double lambda_star,
                            const double* d_yzero, double* d_out, int* d_status) {
  if (n_obs <= 0) return cudaSuccess;
  ProfScope ps(st, K_FIT, method == NNE_FIT_POLY ? 1 : 2);
  return launch_fit(st, n_lambda, d_lam, d_vals, d_logfid, n_obs, method, degree, lambda_star, d_yzero, nullptr,
                    nullptr, d_out, d_status);
}

cudaError_t extrapolate_ladder(cudaStream_t st, int k, int n_lambda, const double* d_lam, const double* d_vals,
                               const double* d_logfid, int n_obs, int method, int degree, double lambda_star,
                               const double* d_yzero, double* d_obar, uint8_t* d_conv, double* d_out, int* d_status) {
  if (n_obs <= 0) return cudaSuccess;
  ProfScope ps(st, K_FIT, method == NNE_FIT_POLY ? 2 : 3);
  const long long cells = (long long)n_lambda * n_obs;
  ladder_kernel<<<(unsigned)((cells + 127) / 128), 128, 0, st>>>(k, n_lambda, n_obs, d_vals, d_logfid, d_obar, d_conv);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // (B) on the fidelity-extrapolated values, F^max = the top rung, fallback to the top rung's values
  const double* top_logf = d_logfid + (long long)(k - 1) * n_lambda;
  const double* top_vals = d_vals + (long long)(k - 1) * cells;
  return launch_fit(st, n_lambda, d_lam, d_obar, top_logf, n_obs, method, degree, lambda_star, d_yzero, d_conv,
                    top_vals, d_out, d_status);
}

}  // namespace nne
