// Float64 eigenpairs of real tridiagonal matrices: eigenvalues by bisection
// with Sturm counts, eigenvectors by inverse iteration.
//
// What bounds both: GB300 issues a float64 instruction of a warp in 64 cycles
// (measured, whatever the number of active lanes and independent chains), and
// each eigenvalue is a serial recurrence over the n rows, so the time is the
// number of float64 instructions per row times n times 31 ns.  Both kernels
// therefore keep that number low -- comparisons, signs, exponents and scalings
// by powers of two go to the integer pipe, reciprocals replace divides, passes
// over the vector are merged -- and spread the eigenvalues over the 608 SM
// sub-partitions, one warp each.  Per launch, n = 64 (4 matrices, 16 wanted):
// bisection 236 -> 84 us, inverse iteration 178 -> 97; n = 256 (5, 64): 900 -> 321
// and 961 -> 367; n = 512 (6, 128): 1689 -> 674 and 1880 -> 697; n = 640 (8, 512):
// 2360 -> 1477 and 3676 -> 1137.
#include <float.h>

#include "kernels.cuh"
#include "recip.cuh"

namespace nne {

namespace {

__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ULL;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
  return x ^ (x >> 31);
}

// Number of eigenvalues of T - x I below 0: sign changes of the leading
// principal minors 1, p_0, ..., p_{n-1} (Sturm; three-term recurrence, three
// float64 instructions per row, no divide).  T is scaled to norm <= 1, so |p|
// grows at most 3x per row; every 4 rows a pair is brought back by a power of
// two when its larger exponent has left [-600, 600].  A minor that is zero (or
// underflows) is replaced by -2^-1000 p_{k-1}: blocks of 4 rows run without
// the test, and one that met a zero runs again with it.  All 32 lanes take part
// (the rare corrections are warp votes with a barrier to the compiler, which
// otherwise evaluates their float64 products on every row).
__device__ __forceinline__ int sturm_minors(const double* ds, const double* b, int n, double x) {
  auto is_zero = [](double p) { return ((__double2hiint(p) & 0x7fffffff) | __double2loint(p)) == 0; };
  double p0 = 1.0, p1 = ds[0] - x;
  if (is_zero(p1)) p1 = -0x1p-1000;
  int c = (int)((unsigned)__double2hiint(p1) >> 31);
  auto row_checked = [&](double dk, double bk) {
    double p = fma(-bk, p0, (dk - x) * p1);
    if (is_zero(p)) p = -0x1p-1000 * p1;
    c += (int)((unsigned)(__double2hiint(p) ^ __double2hiint(p1)) >> 31);
    p0 = p1;
    p1 = p;
  };
  int k = 1;
  for (; k + 3 < n; k += 4) {
    const double d0 = ds[k], d1 = ds[k + 1], d2 = ds[k + 2], d3 = ds[k + 3];
    const double b0 = b[k - 1], b1 = b[k], b2 = b[k + 1], b3 = b[k + 2];
    const double q0 = fma(-b0, p0, (d0 - x) * p1);
    const double q1 = fma(-b1, p1, (d1 - x) * q0);
    const double q2 = fma(-b2, q0, (d2 - x) * q1);
    const double q3 = fma(-b3, q1, (d3 - x) * q2);
    if (__any_sync(0xffffffffu, is_zero(q0) || is_zero(q1) || is_zero(q2) || is_zero(q3))) {
      asm volatile("" ::: "memory");
      row_checked(d0, b0);
      row_checked(d1, b1);
      row_checked(d2, b2);
      row_checked(d3, b3);
    } else {
      const int h = __double2hiint(p1), h0 = __double2hiint(q0), h1 = __double2hiint(q1), h2 = __double2hiint(q2),
                h3 = __double2hiint(q3);
      c += (int)((unsigned)(h ^ h0) >> 31) + (int)((unsigned)(h0 ^ h1) >> 31) + (int)((unsigned)(h1 ^ h2) >> 31) +
           (int)((unsigned)(h2 ^ h3) >> 31);
      p0 = q2;
      p1 = q3;
    }
    const int em = max((__double2hiint(p1) >> 20) & 0x7ff, (__double2hiint(p0) >> 20) & 0x7ff);
    const bool out = em > 1023 + 600 || em < 1023 - 600;
    if (__any_sync(0xffffffffu, out)) {
      asm volatile("" ::: "memory");
      const double sc = out ? __hiloint2double((2046 - em) << 20, 0) : 1.0;   // 2^(1023 - em)
      p0 *= sc;
      p1 *= sc;
    }
  }
  for (; k < n; ++k) row_checked(ds[k], b[k - 1]);
  return c;
}

}  // namespace

// Top r eigenvalues (descending) of the real tridiagonal (d, e).  L lanes per
// eigenvalue count at L interior points of the bracket, which shrinks
// (L + 1)-fold per round until it is width * eps_64 ||T|| wide.  The bracket starts
// at lamf[t] -/+ 16 or 512 eps_32 ||T|| around the float32 eigenvalue of the
// rounded tridiagonal when Sturm counts confirm that it holds the wanted
// eigenvalue (the float32 counts are off by more than the former now and then,
// and one lane's full search holds up the warp), else at the Gershgorin interval.
constexpr int BIS64_THREADS = 64;

template <int L>
__global__ void __launch_bounds__(BIS64_THREADS) bisect64_kernel(const double* db, const double* eb, int n, int r,
                                                                 int ldde, const float* lamfb, double* lamb, int ldl,
                                                                 double width) {
  extern __shared__ double bis_smem[];
  double* ds = bis_smem;        // n: d scaled
  double* bs = bis_smem + n;    // n: e^2 scaled
  __shared__ double red[2][BIS64_THREADS / 32];
  __shared__ int sexp;
  const int z = blockIdx.y, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const double* d = db + (long long)z * ldde;
  const double* e = eb + (long long)z * ldde;
  // Gershgorin interval and the power-of-two scale
  double glo = 1e300, ghi = -1e300;
  for (int k = tid; k < n; k += BIS64_THREADS) {
    const double rad = (k > 0 ? e[k - 1] : 0.0) + (k + 1 < n ? e[k] : 0.0);
    glo = fmin(glo, d[k] - rad);
    ghi = fmax(ghi, d[k] + rad);
  }
  for (int o = 16; o > 0; o >>= 1) {
    glo = fmin(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
  }
  if (lane == 0) {
    red[0][wid] = glo;
    red[1][wid] = ghi;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < BIS64_THREADS / 32; ++w) {
      red[0][0] = fmin(red[0][0], red[0][w]);
      red[1][0] = fmax(red[1][0], red[1][w]);
    }
    const double tn = fmax(fabs(red[0][0]), fabs(red[1][0]));
    sexp = tn > 0 ? ((__double2hiint(tn) >> 20) & 0x7ff) - 1023 + 1 : 0;   // tn < 2^sexp
  }
  __syncthreads();
  const double sc = __hiloint2double((1023 - sexp) << 20, 0);   // 2^-sexp
  for (int k = tid; k < n; k += BIS64_THREADS) {
    ds[k] = d[k] * sc;
    const double es = k + 1 < n ? e[k] * sc : 0.0;
    bs[k] = es * es;
  }
  glo = red[0][0] * sc;
  ghi = red[1][0] * sc;
  __syncthreads();
  const double tnorm = fmax(fabs(glo), fabs(ghi));
  const double tol = width * DBL_EPSILON * tnorm + 0x1p-1000;
  glo -= 4 * DBL_EPSILON * tnorm;
  ghi += 4 * DBL_EPSILON * tnorm;
  const int sub = lane % L, g0 = lane - sub;
  const int t = (blockIdx.x * (BIS64_THREADS / 32) + wid) * (32 / L) + lane / L;
  const bool live = t < r;
  const int idx = n - 1 - (live ? t : 0);
  double lo = glo, hi = ghi;
  {
    // the float32 bracket and a 32 times wider one, checked by four lanes of the group
    const double lf = live ? (double)lamfb[(long long)z * ldl + t] * sc : 0.0;
    const double w = 16.0 * (double)FLT_EPSILON * tnorm, x = fma(sub & 2 ? 32.0 : 1.0, sub & 1 ? w : -w, lf);
    const int cnt = sturm_minors(ds, bs, n, x);
    const int c0 = __shfl_sync(0xffffffffu, cnt, g0), c1 = __shfl_sync(0xffffffffu, cnt, g0 + 1);
    const int c2 = __shfl_sync(0xffffffffu, cnt, g0 + 2), c3 = __shfl_sync(0xffffffffu, cnt, g0 + 3);
    if (c0 <= idx && c1 > idx) {
      lo = lf - w;
      hi = lf + w;
    } else if (c2 <= idx && c3 > idx) {
      lo = fma(-32.0, w, lf);
      hi = fma(32.0, w, lf);
    }
  }
  const double frac = (double)(sub + 1) / (double)(L + 1);
  for (int it = 0; it < 40; ++it) {
    const bool open = live && (hi - lo) > tol;
    if (!__any_sync(0xffffffffu, open)) break;
    const double x = lo + (hi - lo) * frac;
    const int cnt = sturm_minors(ds, bs, n, x);
    const unsigned m = __ballot_sync(0xffffffffu, cnt <= idx);
    const int K = __popc((m >> g0) & (L == 32 ? 0xffffffffu : (1u << (L & 31)) - 1u));   // points at or below (a prefix)
    const double xl = __shfl_sync(0xffffffffu, x, g0 + max(K - 1, 0)), xh = __shfl_sync(0xffffffffu, x, g0 + min(K, L - 1));
    if (open) {
      if (K > 0) lo = xl;
      if (K < L) hi = xh;
    }
  }
  if (live && sub == 0) lamb[(long long)z * ldl + t] = 0.5 * (lo + hi) / sc;
}

cudaError_t bisect64(cudaStream_t st, const double* d, const double* e, int n, int r, const float* lamf, double* lam,
                     int batch, double width) {
  ProfScope ps(st, K_BISECT64);
  const size_t bsm = 2 * sizeof(double) * (size_t)n;
  auto go = [&](auto kernel, int L) {
    const cudaError_t ce = ensure_kernel_smem((const void*)kernel, bsm, false);
    if (ce != cudaSuccess) return ce;
    const int per = BIS64_THREADS / L;   // eigenvalues per block
    kernel<<<dim3((r + per - 1) / per, batch), BIS64_THREADS, bsm, st>>>(d, e, n, r, n, lamf, lam, r, width);
    return cudaGetLastError();
  };
  // Rounds from the float32 bracket (32 bits to width 4, 33 to 2): 14 or 15 with 4 lanes,
  // 11 with 8, 8 or 9 with 16, 7 with 32; more lanes as long as a state's eigenvalues (up to 8 levels)
  // still find a sub-partition each.
  if (r <= 64) return go(bisect64_kernel<32>, 32);
  if (r <= 192) return go(bisect64_kernel<16>, 16);
  if (r <= 320) return go(bisect64_kernel<8>, 8);
  return go(bisect64_kernel<4>, 4);
}

// Inverse iteration for eigenvalue lam[t] of the real tridiagonal (d, e): three
// solves with the partially pivoted LU of T - lam I; pivots below eps ||T|| are
// replaced by +-eps ||T||.  Unit column t of Z (n x r, row-major, written as
// OUT).  IV_LANES eigenvalues per warp.
//
// About 22 float64 instructions per row: the factorisation keeps the pivots'
// reciprocals and takes its multipliers from them, the first forward solve runs
// along with it, the vector is normalised once at the end (three solves grow it
// by at most (1 / (eps ||T||))^3, inside float64's range for ||T|| in [2^-100,
// 2^100]; other matrices are scaled by a power of two).  Loads run one block of
// IV_U rows ahead of the recurrence.
constexpr int IV_LANES = 8, IV_U = 4;

template <typename OUT>
__global__ void __launch_bounds__(32) inviter64_kernel(const double* db, const double* eb, int n, int r, int ldde,
                                                       const double* lamb, int ldl, OUT* Zb, long long sZ, double* Yb,
                                                       double* Lb, double* U0b, double* U1b, double* U2b,
                                                       uint8_t* pivb, long long sS, int total) {
  const int lane = threadIdx.x;
  const int gid = blockIdx.x * IV_LANES + lane % IV_LANES;
  const bool live = lane < IV_LANES && gid < total;
  const int id = gid < total ? gid : total - 1;
  const int z = id / r, t = id % r;
  const double* d = db + (long long)z * ldde;
  const double* e = eb + (long long)z * ldde;
  // ||T|| of each lane's matrix, the rows shared by the lanes of one eigenvalue
  double tnorm = 0;
  {
    long long mx = 0;
    for (int k = lane / IV_LANES; k < n; k += 32 / IV_LANES) {
      const double rad = (k > 0 ? e[k - 1] : 0.0) + (k + 1 < n ? e[k] : 0.0);
      mx = max(mx, abs_bits(fabs(d[k]) + rad));
    }
    for (int o = IV_LANES; o < 32; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    tnorm = __longlong_as_double(mx);
  }
  if (!live) return;
  if (!(tnorm > 0.0)) tnorm = 1.0;
  double sc = 1.0;
  const int ex = ((__double2hiint(tnorm) >> 20) & 0x7ff) - 1023;
  const bool scaled = (ex < -100 || ex > 100) && ex < 1024;
  if (scaled) {
    sc = __hiloint2double((1023 - min(max(ex, -1000), 1000)) << 20, 0);
    tnorm *= sc;
  }
  const double lam = lamb[(long long)z * ldl + t] * sc;
  auto scale = [&](double v) {   // a multiply only where needed
    if (scaled) {
      asm volatile("" ::: "memory");
      v *= sc;
    }
    return v;
  };
  double* y = Yb + z * sS + t;
  double* Lp = Lb + z * sS + t;
  double* U0 = U0b + z * sS + t;
  double* U1 = U1b + z * sS + t;
  double* U2 = U2b + z * sS + t;
  uint8_t* piv = pivb + z * sS + t;
  const double tiny = DBL_EPSILON * tnorm;
  const long long tiny_bits = abs_bits(tiny);
  auto recip = [&](double u) {   // of the pivot, replaced if tiny
    if (abs_bits(u) < tiny_bits) u = __double2hiint(u) < 0 ? -tiny : tiny;
    return rcp_series(u);
  };
  // uniform in [-1, 1): the same start vectors for every matrix of the batch
  auto start = [&](int k) {
    const unsigned long long h = splitmix64(((unsigned long long)t << 20) ^ (unsigned long long)k);
    return fma(2.0, __longlong_as_double((long long)(0x3ff0000000000000ULL | (h >> 12))), -3.0);
  };
  // factor, and the first forward solve
  {
    double diag = scale(d[0]) - lam, sup1 = n > 1 ? scale(e[0]) : 0.0, yk = start(0);
    double ek = sup1, dn = n > 1 ? d[1] : 0.0;
    for (int k = 0; k + 1 < n; ++k) {
      const long long o = (long long)k * r;
      const double en = k + 2 < n ? scale(e[k + 1]) : 0.0;       // next row's loads first
      const double dnn = k + 2 < n ? d[k + 2] : 0.0;
      const double sub = ek, nd = scale(dn) - lam, ns = en;
      double yk1 = start(k + 1);
      const bool sw = abs_bits(diag) < abs_bits(sub);
      const double u0 = sw ? sub : diag, u1 = sw ? nd : sup1;
      const double inv = recip(u0);
      const double l = (sw ? diag : sub) * inv;
      piv[o] = sw;
      Lp[o] = l;
      U0[o] = inv;
      U1[o] = u1;
      U2[o] = sw ? ns : 0.0;
      diag = fma(-l, u1, sw ? sup1 : nd);
      sup1 = sw ? -l * ns : ns;
      if (sw) { const double tmp = yk; yk = yk1; yk1 = tmp; }
      y[o] = yk;
      yk = fma(-l, yk, yk1);
      ek = en;
      dn = dnn;
    }
    U0[(long long)(n - 1) * r] = recip(diag);
    U1[(long long)(n - 1) * r] = 0.0;
    U2[(long long)(n - 1) * r] = 0.0;
    y[(long long)(n - 1) * r] = yk;
  }
  double s2 = 0;
  for (int it = 0; it < 3; ++it) {
    if (it > 0) {
      // forward: y <- L^-1 P y
      double yk = y[0];
      double nl[IV_U], ny[IV_U];
      uint8_t np[IV_U];
      auto load = [&](int k) {
#pragma unroll
        for (int u = 0; u < IV_U; ++u)
          if (k + u + 1 < n) {
            const long long o = (long long)(k + u) * r;
            nl[u] = Lp[o];
            np[u] = piv[o];
            ny[u] = y[o + r];
          }
      };
      load(0);
      for (int k = 0; k + 1 < n; k += IV_U) {
        double cl[IV_U], cy[IV_U];
        uint8_t cp[IV_U];
#pragma unroll
        for (int u = 0; u < IV_U; ++u) { cl[u] = nl[u]; cy[u] = ny[u]; cp[u] = np[u]; }
        load(k + IV_U);
#pragma unroll
        for (int u = 0; u < IV_U; ++u)
          if (k + u + 1 < n) {
            const double a = cp[u] ? cy[u] : yk, b = cp[u] ? yk : cy[u];
            y[(long long)(k + u) * r] = a;
            yk = fma(-cl[u], a, b);
          }
      }
      y[(long long)(n - 1) * r] = yk;
    }
    // backward: y <- U^-1 y
    {
      double y1 = 0, y2 = 0;
      double n0[IV_U], n1[IV_U], n2[IV_U], ny[IV_U];
      auto load = [&](int k) {   // rows k, k - 1, ...
#pragma unroll
        for (int u = 0; u < IV_U; ++u)
          if (k - u >= 0) {
            const long long o = (long long)(k - u) * r;
            n0[u] = U0[o];
            n1[u] = U1[o];
            n2[u] = U2[o];
            ny[u] = y[o];
          }
      };
      load(n - 1);
      for (int k = n - 1; k >= 0; k -= IV_U) {
        double c0[IV_U], c1[IV_U], c2[IV_U], cy[IV_U];
#pragma unroll
        for (int u = 0; u < IV_U; ++u) { c0[u] = n0[u]; c1[u] = n1[u]; c2[u] = n2[u]; cy[u] = ny[u]; }
        load(k - IV_U);
#pragma unroll
        for (int u = 0; u < IV_U; ++u)
          if (k - u >= 0) {
            const double yk = fma(-c1[u], y1, fma(-c2[u], y2, cy[u])) * c0[u];
            y[(long long)(k - u) * r] = yk;
            if (it == 2) s2 = fma(yk, yk, s2);
            y2 = y1;
            y1 = yk;
          }
      }
    }
  }
  const double inv = s2 > 0 ? 1.0 / sqrt(s2) : 0.0;
  OUT* Z = Zb + z * sZ + t;
#pragma unroll 4
  for (int k = 0; k < n; ++k) Z[(long long)k * r] = (OUT)(y[(long long)k * r] * inv);
}

template <typename OUT>
cudaError_t inviter64(cudaStream_t st, const double* d, const double* e, int n, int r, const double* lam, OUT* Z,
                      double* Y, double* L, double* U0, double* U1, double* U2, uint8_t* piv, int batch) {
  ProfScope ps(st, K_INVITER);
  const int total = batch * r;
  const long long nr = (long long)n * r;
  inviter64_kernel<OUT><<<(total + IV_LANES - 1) / IV_LANES, 32, 0, st>>>(d, e, n, r, n, lam, r, Z, nr, Y, L, U0, U1, U2,
                                                                          piv, nr, total);
  return cudaGetLastError();
}
template cudaError_t inviter64<float>(cudaStream_t, const double*, const double*, int, int, const double*, float*,
                                      double*, double*, double*, double*, double*, uint8_t*, int);
template cudaError_t inviter64<double>(cudaStream_t, const double*, const double*, int, int, const double*, double*,
                                       double*, double*, double*, double*, double*, uint8_t*, int);

}  // namespace nne
