// The Hermitian eigensolver of the truncation step and the entropy, written for GB300:
//   * Householder reduction to real tridiagonal form, one thread-block cluster
//     per matrix: in the cluster's shared memory (k_eig_small.cu), double-float
//     (k_tridiag_df.cu), or here, on the matrix in L2 with two cluster barriers per
//     column;
//   * eigenvalues of the tridiagonal by 32-way multisection with Sturm
//     counts (one warp per wanted eigenvalue; float64: k_tri64.cu narrows the
//     float32 brackets);
//   * eigenvectors by inverse iteration with a partially pivoted tridiagonal
//     LU (float32 here, one thread each; float64 in k_tri64.cu), back-transformed
//     through the phase scaling and the Householder reflectors (k_eig_small.cu) and
//     orthonormalised by the QR (k_qr.cu).
// Precision follows the state: float for complex64 states (by default with the
// reduction, eigenvalues and tridiagonal eigenvectors in float64 or double-float),
// double for complex128.  The reductions are written in a fixed order, so results are
// bitwise reproducible run to run.  The double-float and the L2-resident reductions do not
// depend on what else is batched either; those in one cluster's shared memory (tridiag_smem,
// _keep) sum K over as many CTAs as the batch lets run at once.
#include <map>
#include <mutex>

#include "kernels.cuh"
#include <float.h>

namespace cg = cooperative_groups;

namespace nne {

template <typename R> struct Lim;
template <> struct Lim<float> {
  static __device__ __forceinline__ float eps() { return FLT_EPSILON; }
  static __device__ __forceinline__ float tiny() { return FLT_MIN; }
  static __device__ __forceinline__ float big() { return 1e30f; }
};
template <> struct Lim<double> {
  static __device__ __forceinline__ double eps() { return DBL_EPSILON; }
  static __device__ __forceinline__ double tiny() { return DBL_MIN; }
  static __device__ __forceinline__ double big() { return 1e250; }
};

// Sum over the block in a fixed order; every thread gets the total.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* red) {
  v = warp_sum_r(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  T t = 0;
  const int nw = blockDim.x >> 5;
  for (int i = 0; i < nw; ++i) t += red[i];
  return t;
}

// Householder vector of x (length m, in smem v, overwritten): P = I - 2 v v^H,
// P x = alpha e_1.  Returns alpha.  Whole block participates.
template <typename R>
__device__ cx<R> householder(cx<R>* v, int m, double* red) {
  double s = 0;
  for (int t = threadIdx.x; t < m; t += blockDim.x) s += norm2d(v[t]);
  const double xn2 = block_sum(s, red);
  const cx<R> x0 = v[0];
  double pr, pi, ax0;
  unit_phase_of(x0, &pr, &pi, &ax0);
  const double xn = sqrt(xn2);
  cx<R> alpha = mk<R>(0, 0);
  double un = 0;
  if (xn > 0) {
    alpha = mk<R>((R)(-xn * pr), (R)(-xn * pi));
    un = sqrt(2.0 * xn2 + 2.0 * xn * ax0);
  }
  __syncthreads();
  const R inv = un > 0 ? (R)(1.0 / un) : R(0);
  for (int t = threadIdx.x; t < m; t += blockDim.x) {
    cx<R> u = v[t];
    if (t == 0) u = u - alpha;
    v[t] = inv * u;
  }
  __syncthreads();
  return alpha;
}

// ---------------------------------------------------------------- tridiagonal
// H (n x n) -> real tridiagonal d, complex subdiagonal e (e[k] = T[k+1][k]);
// reflector j (length n-j-1) is stored conjugated in row j of Vh, columns j+1..n-1.
// LOWER: only the lower triangle of H is read and updated (the rank-2 update
// touches half the entries; the product A v reads each row's lower part and,
// strided, its upper part as the conjugated column), 2 m^2 instead of 3 m^2
// complex multiply-adds per column: the float64 instantiation, whose rate on
// GB300 is 1/64 of float32, takes it.
template <typename R, bool LOWER>
__global__ void __launch_bounds__(256) tridiag_kernel(cx<R>* Hb, long long sH, int n, R* db, cx<R>* eb, int ldde,
                                                       cx<R>* Pb, double* Kb, cx<R>* Vhb, long long sVh) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int z = blockIdx.y;
  cx<R>* H = Hb + z * sH;
  R* d = db + (long long)z * ldde;
  cx<R>* e = eb + (long long)z * ldde;
  cx<R>* P = Pb + (long long)z * ldde;
  double* Kp = Kb + z * 32;
  extern __shared__ unsigned char smem_raw[];
  cx<R>* v = reinterpret_cast<cx<R>*>(smem_raw);
  cx<R>* w = v + n;
  __shared__ double red[32];
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
  const int gw = rank * nw + warp, GW = CS * nw;

  for (int j = 0; j + 2 < n; ++j) {
    const int m = n - j - 1;
    if (LOWER) {
      const cx<R>* colj = H + (long long)(j + 1) * n + j;
      for (int t = tid; t < m; t += nth) v[t] = colj[(long long)t * n];   // column j below the diagonal
    } else {
      const cx<R>* rowj = H + (long long)j * n + (j + 1);
      for (int t = tid; t < m; t += nth) v[t] = conj(rowj[t]);   // column j below the diagonal
    }
    __syncthreads();
    const R djj = H[(long long)j * n + j].re;
    const cx<R> alpha = householder(v, m, red);
    if (rank == 0 && tid == 0) {
      d[j] = djj;
      e[j] = alpha;
    }
    // p = A v on own rows; partial of K = v^H p
    double kp = 0;
    for (int t = gw; t < m; t += GW) {
      const cx<R>* row = H + (long long)(j + 1 + t) * n + (j + 1);
      cx<R> acc = mk<R>(0, 0);
      if (LOWER) {
        for (int k = lane; k <= t; k += 32) fma_(acc, row[k], v[k]);
        // upper part of row t: conj(A[k][t]) for k > t, read down column t
        const cx<R>* colt = H + (long long)(j + 1) * n + (j + 1 + t);
        for (int k = t + 1 + lane; k < m; k += 32) fma_(acc, conj(colt[(long long)k * n]), v[k]);
      } else {
        for (int k = lane; k < m; k += 32) fma_(acc, row[k], v[k]);
      }
      acc = warp_sum(acc);
      if (lane == 0) {
        P[t] = acc;
        kp += (double)v[t].re * acc.re + (double)v[t].im * acc.im;
      }
    }
    kp = block_sum(kp, red);
    if (tid == 0) Kp[rank] = kp;
    __threadfence();
    cluster.sync();
    double K = 0;
    for (int c = 0; c < CS; ++c) K += Kp[c];
    const R twoK = (R)(2.0 * K);
    for (int t = tid; t < m; t += nth) {
      const cx<R> p = P[t];
      w[t] = mk<R>(2 * p.re - twoK * v[t].re, 2 * p.im - twoK * v[t].im);
    }
    if (rank == 0) {
      cx<R>* rj = Vhb + z * sVh + (long long)j * n + (j + 1);
      for (int t = tid; t < m; t += nth) rj[t] = conj(v[t]);   // reflector j, conjugated, for the back-transform
    }
    __syncthreads();
    for (int t = gw; t < m; t += GW) {
      cx<R>* row = H + (long long)(j + 1 + t) * n + (j + 1);
      const cx<R> vt = v[t], wt = w[t];
      const int kend = LOWER ? t + 1 : m;
      for (int k = lane; k < kend; k += 32) {
        cx<R> a = row[k];
        const cx<R> wk = w[k], vk = v[k];
        // a -= vt conj(wk) + wt conj(vk)
        a.re -= vt.re * wk.re + vt.im * wk.im + wt.re * vk.re + wt.im * vk.im;
        a.im -= vt.im * wk.re - vt.re * wk.im + wt.im * vk.re - wt.re * vk.im;
        row[k] = a;
      }
    }
    __threadfence();
    cluster.sync();
  }
  if (rank == 0 && tid == 0) {
    if (n >= 2) {
      d[n - 2] = H[(long long)(n - 2) * n + (n - 2)].re;
      d[n - 1] = H[(long long)(n - 1) * n + (n - 1)].re;
      e[n - 2] = H[(long long)(n - 1) * n + (n - 2)];
    } else {
      d[0] = H[0].re;
    }
  }
}

// |e_k| and the phases phi (phi_0 = 1, phi_{k+1} = phi_k e_k/|e_k|) that make
// the tridiagonal real: T = D T' D^H with T'_{k+1,k} = |e_k|.  One CTA per
// matrix: each thread multiplies the unit phases of a contiguous chunk, a
// block-wide scan (FP64, fixed order) gives every chunk its prefix.
__device__ __forceinline__ cx<double> shfl_up_cd(cx<double> v, int d) {
  return mk<double>(__shfl_up_sync(0xffffffffu, v.re, d), __shfl_up_sync(0xffffffffu, v.im, d));
}
__device__ __forceinline__ cx<double> unit_phase(double er, double ei, double* a) {
  const double a2 = er * er + ei * ei;
  *a = sqrt(a2);
  if (!(a2 > 0)) return mk<double>(1.0, 0.0);
  const double inv = 1.0 / *a;
  return mk<double>(er * inv, ei * inv);
}
template <typename R>
__global__ void __launch_bounds__(256) tridiag_phases_kernel(const cx<R>* eb, int n, int ldde, R* eabs,
                                                             cx<R>* phib) {
  __shared__ cx<double> wtot[8];
  const int z = blockIdx.x;
  const cx<R>* e = eb + (long long)z * ldde;
  R* ea = eabs + (long long)z * ldde;
  cx<R>* phi = phib + (long long)z * ldde;
  const int m = n - 1, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int chunk = m > 0 ? (m + 255) / 256 : 0;
  const int k0 = min(m, tid * chunk), k1 = min(m, k0 + chunk);
  cx<double> p = mk<double>(1.0, 0.0);
  for (int k = k0; k < k1; ++k) {
    double a;
    p = p * unit_phase((double)e[k].re, (double)e[k].im, &a);
    ea[k] = (R)a;
  }
  // inclusive scan within the warp, then over the warp totals
  for (int d = 1; d < 32; d <<= 1) {
    const cx<double> t = shfl_up_cd(p, d);
    if (lane >= d) p = t * p;
  }
  if (lane == 31) wtot[wid] = p;
  __syncthreads();
  cx<double> pre = mk<double>(1.0, 0.0);
  for (int w = 0; w < wid; ++w) pre = pre * wtot[w];
  cx<double> excl = shfl_up_cd(p, 1);
  if (lane == 0) excl = mk<double>(1.0, 0.0);
  cx<double> q = pre * excl;
  const double qa = sqrt(q.re * q.re + q.im * q.im);
  q = mk<double>(q.re / qa, q.im / qa);
  if (tid == 0) phi[0] = mk<R>(1, 0);
  for (int k = k0; k < k1; ++k) {
    double a;
    q = q * unit_phase((double)e[k].re, (double)e[k].im, &a);
    phi[k + 1] = mk<R>((R)q.re, (R)q.im);
  }
}

template <typename R>
__device__ __forceinline__ int sturm_count(const R* d, const R* e, int n, R x, R pivmin) {
  R q = d[0] - x;
  if (fabs(q) < pivmin) q = -pivmin;
  int c = q < R(0);
  for (int k = 1; k < n; ++k) {
    q = (d[k] - x) - (e[k - 1] * e[k - 1]) / q;
    if (fabs(q) < pivmin) q = -pivmin;
    c += q < R(0);
  }
  return c;
}

// Top r eigenvalues (descending) of the real tridiagonal (d, e): one warp each.
template <typename R>
__global__ void bisect_kernel(const R* db, const R* eb, int n, int r, int ldde, R* lamb, int ldl, int total) {
  const int gw = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (gw >= total) return;
  const int z = gw / r, t = gw % r;
  const R* d = db + (long long)z * ldde;
  const R* e = eb + (long long)z * ldde;
  R lo = Lim<R>::big(), hi = -Lim<R>::big(), emax = 0;
  for (int k = lane; k < n; k += 32) {
    const R rad = (k > 0 ? e[k - 1] : R(0)) + (k + 1 < n ? e[k] : R(0));
    lo = fmin(lo, d[k] - rad);
    hi = fmax(hi, d[k] + rad);
    if (k + 1 < n) emax = fmax(emax, e[k]);
  }
  for (int m = 16; m > 0; m >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, m));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, m));
    emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, m));
  }
  const R tnorm = fmax(fabs(lo), fabs(hi));
  const R pivmin = Lim<R>::tiny() * fmax(R(1), emax * emax);
  const R eps = Lim<R>::eps();
  lo -= 4 * eps * tnorm + pivmin;
  hi += 4 * eps * tnorm + pivmin;
  const int idx = n - 1 - t;     // ascending index of the wanted eigenvalue
  const R tol = 2 * eps * tnorm + 2 * pivmin;
  for (int it = 0; it < 64 && (hi - lo) > tol; ++it) {
    const R x = lo + (hi - lo) * (R)(lane + 1) / R(33);
    const int cnt = sturm_count(d, e, n, x, pivmin);
    const unsigned mask = __ballot_sync(0xffffffffu, cnt <= idx);
    R nlo = lo, nhi = hi;
    if (mask) {
      const int l = 31 - __clz(mask);
      nlo = __shfl_sync(0xffffffffu, x, l);
      const R xn = __shfl_sync(0xffffffffu, x, (l + 1) & 31);
      if (l < 31) nhi = xn;
    } else {
      nhi = __shfl_sync(0xffffffffu, x, 0);
    }
    lo = nlo;
    hi = nhi;
  }
  if (lane == 0) lamb[(long long)z * ldl + t] = R(0.5) * (lo + hi);
}

__device__ __forceinline__ unsigned long long splitmix(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ULL;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
  return x ^ (x >> 31);
}

// Inverse iteration for eigenvalue lam[t] of the real tridiagonal (d, e):
// 3 solves with the partially pivoted LU of (T - lam I); tiny pivots are
// replaced by eps*||T||.  Output column t of Z (n x r, row-major).  The
// factorisation keeps the pivots' reciprocals, so the solves multiply.  One
// thread per eigenvector (float32; float64 has its own, k_tri64.cu).
template <typename R>
__global__ void inviter_kernel(const R* db, const R* eb, int n, int r, int ldde, const R* lamb, int ldl, R* Zb,
                               long long sZ, R* Lb, R* U0b, R* U1b, R* U2b, uint8_t* pivb, long long sS, int total) {
  const int gid = (int)(blockIdx.x * (long long)blockDim.x + threadIdx.x);
  if (gid >= total) return;
  const int z = gid / r, t = gid % r;
  const R* d = db + (long long)z * ldde;
  const R* e = eb + (long long)z * ldde;
  const R lam = lamb[(long long)z * ldl + t];
  R* y = Zb + z * sZ;
  R* L = Lb + z * sS;
  R* U0 = U0b + z * sS;
  R* U1 = U1b + z * sS;
  R* U2 = U2b + z * sS;
  uint8_t* piv = pivb + z * sS;
  R tnorm = 0;
  for (int k = 0; k < n; ++k) {
    const R rad = (k > 0 ? e[k - 1] : R(0)) + (k + 1 < n ? e[k] : R(0));
    tnorm = fmax(tnorm, fabs(d[k]) + rad);
  }
  if (tnorm == R(0)) tnorm = R(1);
  const R tiny = Lim<R>::eps() * tnorm;
  // factor
  R diag = d[0] - lam, sup1 = n > 1 ? e[0] : R(0);
  for (int k = 0; k + 1 < n; ++k) {
    const R sub = e[k], nd = d[k + 1] - lam, ns = (k + 2 < n) ? e[k + 1] : R(0);
    const long long o = (long long)k * r + t;
    if (fabs(diag) >= fabs(sub)) {
      const R l = diag != R(0) ? sub / diag : R(0);
      piv[o] = 0; L[o] = l; U0[o] = diag; U1[o] = sup1; U2[o] = 0;
      diag = nd - l * sup1;
      sup1 = ns;
    } else {
      const R l = diag / sub;
      piv[o] = 1; L[o] = l; U0[o] = sub; U1[o] = nd; U2[o] = ns;
      diag = sup1 - l * nd;
      sup1 = -l * ns;
    }
  }
  U0[(long long)(n - 1) * r + t] = diag;
  // pivots -> their reciprocals (tiny pivots replaced first)
  for (int k = 0; k < n; ++k) {
    const long long o = (long long)k * r + t;
    R u0 = U0[o];
    if (fabs(u0) < tiny) u0 = u0 < R(0) ? -tiny : tiny;
    U0[o] = R(1) / u0;
  }
  // start vector
  for (int k = 0; k < n; ++k) {
    // the same start vectors for every batch entry: identical inputs give bitwise identical outputs
    const unsigned long long h = splitmix(((unsigned long long)t << 20) ^ (unsigned long long)k);
    y[(long long)k * r + t] = (R)((double)(h >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0);
  }
  const R big = Lim<R>::big();
  for (int it = 0; it < 3; ++it) {
    for (int k = 0; k + 1 < n; ++k) {
      const long long o = (long long)k * r + t, o1 = o + r;
      R yk = y[o], yk1 = y[o1];
      if (piv[o]) { const R tmp = yk; yk = yk1; yk1 = tmp; y[o] = yk; }
      y[o1] = yk1 - L[o] * yk;
    }
    for (int k = n - 1; k >= 0; --k) {
      const long long o = (long long)k * r + t;
      R acc = y[o];
      if (k + 1 < n) acc -= U1[o] * y[o + r];
      if (k + 2 < n) acc -= U2[o] * y[o + 2 * r];
      R yk = acc * U0[o];
      if (!(fabs(yk) < big)) {
        // rescale everything computed so far and the untouched right-hand side
        const R s = isfinite(yk) ? R(1) / fabs(yk) : R(0);
        for (int i = 0; i < n; ++i) y[(long long)i * r + t] *= s;
        yk = isfinite(yk) ? yk * s : R(1);
      }
      y[o] = yk;
    }
    R mx = 0;
    for (int k = 0; k < n; ++k) mx = fmax(mx, fabs(y[(long long)k * r + t]));
    if (!(mx > R(0))) mx = R(1);
    const R imx = R(1) / mx;
    double s2 = 0;
    for (int k = 0; k < n; ++k) {
      const R v = y[(long long)k * r + t] * imx;
      s2 += (double)v * v;
    }
    const R inv = (R)(1.0 / (sqrt(s2) * (double)mx));
    for (int k = 0; k < n; ++k) y[(long long)k * r + t] *= inv;
  }
}

// S[z] = -sum_i p_i ln p_i, p_i = max(lam_i, 0) / sum_j max(lam_j, 0), over the
// n eigenvalues of a Gram matrix (the squared Schmidt values of a bond,
// App. A.1).  One block per matrix, FP64 sums in a fixed order; rounding can
// leave tiny negative eigenvalues, which count as zero.
template <typename R>
__global__ void __launch_bounds__(256) entropy_kernel(const R* lamb, int n, int ldl, double* S, long long sS) {
  __shared__ double red[8];
  const R* lam = lamb + (long long)blockIdx.x * ldl;
  double t = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) t += fmax((double)lam[i], 0.0);
  const double tot = block_sum(t, red);
  double h = 0;
  if (tot > 0)
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const double p = fmax((double)lam[i], 0.0) / tot;
      if (p > 0) h -= p * log(p);
    }
  h = block_sum(h, red);
  if (threadIdx.x == 0) S[(long long)blockIdx.x * sS] = h;
}

// ---------------------------------------------------------------- launchers
template <typename K, typename... Args>
static cudaError_t launch_cluster_t(K kernel, int cs, int batch, int threads, size_t smem, cudaStream_t st,
                                    Args... args) {
  cudaError_t e = ensure_kernel_smem((const void*)kernel, smem, cs > 8);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs, batch, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename K, typename... Args>
static cudaError_t launch_cluster(K kernel, int cs, int batch, size_t smem, cudaStream_t st, Args... args) {
  return launch_cluster_t(kernel, cs, batch, 256, smem, st, args...);
}

static int cluster_size_for(int n) { return n >= 512 ? 8 : (n >= 128 ? 4 : (n >= 32 ? 2 : 1)); }

// Float64 reductions are bounded by their arithmetic (1/64 of the float32
// rate): each CTA gets an SM of its own (its shared-memory request is raised
// to TRIDIAG64_SMEM, so no two share a float64 pipe) and a matrix takes as
// many CTAs as let eight such clusters (a state's noise levels, over its
// sub-batch streams) run at once: the largest size whose occupancy query
// gives at least 8 active clusters (GB300's GPCs hold only 7 clusters of
// 13-16 single-SM CTAs).  The size depends on nothing but the kernel, so
// results do not depend on how instances are batched.
int tridiag64_cluster_size(const void* kernel) {
  static std::mutex mu;
  static std::map<const void*, int> memo;
  std::lock_guard<std::mutex> lk(mu);
  auto it = memo.find(kernel);
  if (it != memo.end()) return it->second;
  int cs = 8;
  for (int c = 16; c > 8; --c) {
    if (ensure_kernel_smem(kernel, TRIDIAG64_SMEM, true) != cudaSuccess) break;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c, 8, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = TRIDIAG64_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int active = 0;
    if (cudaOccupancyMaxActiveClusters(&active, kernel, &cfg) == cudaSuccess && active >= 8) {
      cs = c;
      break;
    }
    (void)cudaGetLastError();
  }
  memo[kernel] = cs;
  return cs;
}

// The L2-resident reduction, one cluster per matrix; float64 reads and
// updates the lower triangle only.
template <typename R>
static cudaError_t tridiag_global(cudaStream_t st, cx<R>* H, long long sH, int n, R* d, cx<R>* e, int ldde, cx<R>* P,
                                  double* Kp, cx<R>* Vh, long long sVh, int batch) {
  constexpr bool lower = std::is_same<R, double>::value;
  const bool wide = lower && n >= 512;
  const int cs = wide ? tridiag64_cluster_size((const void*)tridiag_kernel<R, lower>) : cluster_size_for(n);
  size_t smem = 2 * sizeof(cx<R>) * (size_t)n;
  if (wide) smem = std::max(smem, TRIDIAG64_SMEM);
  ProfScope ps(st, K_TRIDIAG, 1, 16.0 / 3.0 * (double)n * n * n * batch);
  return launch_cluster(tridiag_kernel<R, lower>, cs, batch, smem, st, H, sH, n, d, e, ldde, P, Kp, Vh, sVh);
}

__global__ void re_d2f_pair_kernel(const double* a, const double* b, float* fa, float* fb, long long count) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    fa[i] = (float)a[i];
    fb[i] = (float)b[i];
  }
}

// Top r eigenvalues of batch tridiagonals in float64: a float32 multisection of
// the rounded tridiagonal brackets every eigenvalue to about eps_32 ||T||,
// float64 bisection narrows the brackets.  scratch: batch x (2 n + r) floats.
static cudaError_t bisect_f64(cudaStream_t st, const double* d, const double* e, int n, int r, float* scratch,
                              double* lam, int batch, double width) {
  float* df = scratch;
  float* ef = df + (size_t)n * batch;
  float* lamf = ef + (size_t)n * batch;
  const int total = batch * r;
  cudaError_t ce;
  {
    ProfScope ps(st, K_BISECT);
    re_d2f_pair_kernel<<<64, 256, 0, st>>>(d, e, df, ef, (long long)n * batch);
    bisect_kernel<float><<<(total * 32 + 255) / 256, 256, 0, st>>>(df, ef, n, r, n, lamf, r, total);
  }
  if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  return bisect64(st, d, e, n, r, lamf, lam, batch, width);
}

EighWork eigh_workspace(int n, int r) {
  EighWork w;
  const long long qn = std::max(n, r);
  // cx: e, phi, P (n each), Vh (n x n), WY factors (ceil(n/32) x 32 x 32), WY application workspace
  //     (for r columns), QR workspace of an n x r matrix
  w.cx_elems = 3LL * n + (long long)n * n + ((n + 31) / 32) * 1024LL + wy_workspace(n, r) + qr_workspace(n, r).cx_elems +
               32;
  // re: d, eabs (n each), lam (r), Z (n r), L/U0/U1/U2 (4 n r), Kpart (32 doubles = 64 floats)
  w.re_elems = 2LL * n + r + 5LL * n * r + 64 + qn;
  w.u8_elems = (long long)n * r;
  return w;
}

template <typename R>
cudaError_t eigh_top(cudaStream_t st, cx<R>* H, long long sH, int n, int r, cx<R>* U, long long sU, void* cx_ws,
                     void* re_ws, void* u8_ws, int batch, int* err) {
  (void)err;
  if (batch <= 0) return cudaSuccess;
  const EighWork w = eigh_workspace(n, r);
  cx<R>* cxb = reinterpret_cast<cx<R>*>(cx_ws);
  R* reb = reinterpret_cast<R*>(re_ws);
  uint8_t* u8b = reinterpret_cast<uint8_t*>(u8_ws);
  // per-batch-entry layouts are interleaved by "ld" strides below
  const int ldde = n;
  cx<R>* e = cxb;                                   // batch x n
  cx<R>* phi = e + (long long)batch * n;            // batch x n
  cx<R>* P = phi + (long long)batch * n;            // batch x n
  cx<R>* Vh = P + (long long)batch * n;             // batch x n x n
  cx<R>* Tw = Vh + (long long)batch * n * n;        // batch x nb x 1024
  const int nbw = (n + 31) / 32;
  cx<R>* wyws = Tw + (long long)batch * nbw * 1024;          // batch x wy_workspace(n, r)
  cx<R>* qrws = wyws + (long long)batch * wy_workspace(n, r);   // QR workspace for batch n x r matrices
  R* d = reb;                                       // batch x n
  R* eabs = d + (long long)batch * n;               // batch x n
  R* lam = eabs + (long long)batch * n;             // batch x r
  R* Z = lam + (long long)batch * r;                // batch x n r
  R* Ls = Z + (long long)batch * n * r;             // 4 arrays of batch x n r
  R* U0 = Ls + (long long)batch * n * r;
  R* U1 = U0 + (long long)batch * n * r;
  R* U2 = U1 + (long long)batch * n * r;
  double* Kp = reinterpret_cast<double*>(U2 + (long long)batch * n * r + 1);
  Kp = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(Kp) + 15) & ~uintptr_t(15));
  (void)w;
  cudaError_t ce;
  if (smem_cluster_size<R>(n) > 0) {
    ce = tridiag_smem<R>(st, H, sH, n, d, e, ldde, Vh, (long long)n * n, batch);
  } else {
    if ((ce = cudaMemsetAsync(Vh, 0, sizeof(cx<R>) * (size_t)batch * n * n, st)) != cudaSuccess) return ce;
    ce = tridiag_global<R>(st, H, sH, n, d, e, ldde, P, Kp, Vh, (long long)n * n, batch);
  }
  if (ce != cudaSuccess) return ce;
  {
    ProfScope ps(st, K_ELEMWISE);
    tridiag_phases_kernel<R><<<batch, 256, 0, st>>>(e, n, ldde, eabs, phi);
  }
  if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  const int total = batch * r;
  if constexpr (std::is_same<R, double>::value) {
    // the division-free float64 bisection (the inverse iteration's scratch is still free)
    if ((ce = bisect_f64(st, d, eabs, n, r, reinterpret_cast<float*>(Ls), lam, batch, BISECT_C128)) != cudaSuccess) return ce;
  } else {
    ProfScope ps(st, K_BISECT);
    bisect_kernel<R><<<(total * 32 + 255) / 256, 256, 0, st>>>(d, eabs, n, r, ldde, lam, r, total);
  }
  if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  const long long sS = (long long)n * r;
  if constexpr (std::is_same<R, double>::value) {
    if ((ce = inviter64<double>(st, d, eabs, n, r, lam, Z, Z, Ls, U0, U1, U2, u8b, batch)) != cudaSuccess) return ce;
  } else {
    ProfScope ps(st, K_INVITER);
    inviter_kernel<R><<<(total + 127) / 128, 128, 0, st>>>(d, eabs, n, r, ldde, lam, r, Z, sS, Ls, U0, U1, U2, u8b,
                                                           sS, total);
  }
  if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  ce = backtransform_wy<R>(st, Vh, (long long)n * n, n, Z, sS, phi, ldde, r, U, sU, Tw, wyws, batch);
  if (ce != cudaSuccess) return ce;
  // orthonormalise the eigenvector block (QR; Q written over U)
  return qr<R>(st, U, sU, n, r, U, sU, nullptr, 0, qrws, batch);
}

// ---------------------------------------------------------------- mixed precision
__global__ void cx_f2d_kernel(const cx<float>* X, long long sX, int rows, int cols, int ldx, cx<double>* Y,
                              long long sY) {
  const long long count = (long long)rows * cols;
  const int z = blockIdx.y;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    const cx<float> v = X[z * sX + (i / cols) * ldx + i % cols];
    Y[z * sY + i] = mk<double>(v.re, v.im);
  }
}

__global__ void cx_d2f_kernel(const cx<double>* X, cx<float>* Y, long long count) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x)
    Y[i] = mk<float>((float)X[i].re, (float)X[i].im);
}

static inline size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

// Complex64 eigenproblems up to this size keep the float64 reduction, larger
// ones take the double-float one (k_tridiag_df.cu).  The double-float kernel is
// the faster at every size (n = 64: 174 against 514 us, 128: 431 against 1300),
// but small bonds cut shallow circuits between near-degenerate pairs, where the
// kept vector follows the last bits of the reduction: <P> of 5 in 45 bursts of
// jobs with bonds of 12-40 moved by more than 2e-5 of their norm (up to 7.6e-5,
// as far as the complex64 result itself is from an exact one), against 1 in 200
// circuits with bonds of 41-72.  Up to bonds of 40 results stay as they were.
constexpr int EIGH_F64_MAX = 160;

MixedEighWork eigh_mixed_workspace(int n, int r) {
  // per matrix; every array is batch-major, so a batch of b matrices needs b times these bytes
  MixedEighWork w;
  const size_t nn = (size_t)n * n, nr = (size_t)n * r;
  const int nbw = (n + 31) / 32;
  const size_t nf = (size_t)std::min(n, EIGH_F64_MAX);   // a state's smaller problems take the float64 path
  w.cx_bytes = al256(std::max(16 * nn, 32 * nf * nf)) + al256(16 * (size_t)n) * 3 + al256(8 * nn) + al256(8 * (size_t)n) +
               al256(8 * (size_t)nbw * 1024) + al256(8 * (size_t)wy_workspace(n, r)) +
               al256(8 * (size_t)qr_workspace(n, r).cx_elems) + 1024;
  w.re_bytes = al256(8 * (size_t)n) * 2 + al256(8 * (size_t)r) + al256(8 * nr) * 5 + al256(4 * nr) + 512 +
               al256(4 * (size_t)n) * 2 + al256(4 * (size_t)r) + 1024;
  w.u8_bytes = al256(nr) + 256;
  return w;
}

// Top-r eigenvectors of the complex64 Hermitian H[z] (n x n, ld n), written to
// U[z] (n x r, ld r, columns by decreasing eigenvalue, orthonormal).  The
// Householder reduction runs in float64 (n <= EIGH_F64_MAX) or double-float, the eigenvalues
// (bisection) and the eigenvectors of the tridiagonal (inverse iteration) in
// float64; the back-transformation
// through the reflectors and the final orthonormalisation run in float32.  A
// float32 reduction has a backward error of eps_32 ||H||, which turns the
// eigenvectors next to the truncation cut by eps_32 ||H|| / gap there (about
// 0.1 on saturated chi = 512 states); in float64 that error is below the
// rounding of the input, and the float32 back-transformation only adds
// eps_32-sized, gap-independent errors.
cudaError_t eigh_top_mixed(cudaStream_t st, cx<float>* H, long long sH, int n, int r, cx<float>* U, long long sU,
                           void* cx_ws, void* re_ws, void* u8_ws, int batch, int* err) {
  (void)err;
  if (batch <= 0) return cudaSuccess;
  const size_t nn = (size_t)n * n, nr = (size_t)n * r;
  const int nbw = (n + 31) / 32;
  const size_t B = (size_t)batch;
  unsigned char* c = reinterpret_cast<unsigned char*>(cx_ws);
  auto take = [&](unsigned char*& base, size_t bytes) {
    unsigned char* p = base;
    base += al256(bytes);
    return p;
  };
  cx<double>* Hd = reinterpret_cast<cx<double>*>(take(c, 16 * nn * B * (n <= EIGH_F64_MAX ? 2 : 1)));
  cx<double>* ed = reinterpret_cast<cx<double>*>(take(c, 16 * (size_t)n * B));
  cx<double>* phid = reinterpret_cast<cx<double>*>(take(c, 16 * (size_t)n * B));
  float4* P = reinterpret_cast<float4*>(take(c, 16 * (size_t)n * B));
  cx<float>* Vhf = reinterpret_cast<cx<float>*>(take(c, 8 * nn * B));
  cx<float>* phif = reinterpret_cast<cx<float>*>(take(c, 8 * (size_t)n * B));
  cx<float>* Tw = reinterpret_cast<cx<float>*>(take(c, 8 * (size_t)nbw * 1024 * B));
  cx<float>* wyws = reinterpret_cast<cx<float>*>(take(c, 8 * (size_t)wy_workspace(n, r) * B));
  cx<float>* qrws = reinterpret_cast<cx<float>*>(take(c, 8 * (size_t)qr_workspace(n, r).cx_elems * B));
  unsigned char* q = reinterpret_cast<unsigned char*>(re_ws);
  double* dd = reinterpret_cast<double*>(take(q, 8 * (size_t)n * B));
  double* eabs = reinterpret_cast<double*>(take(q, 8 * (size_t)n * B));
  double* lam = reinterpret_cast<double*>(take(q, 8 * (size_t)r * B));
  double* Z = reinterpret_cast<double*>(take(q, 8 * nr * B));
  double* Ls = reinterpret_cast<double*>(take(q, 8 * nr * B));
  double* U0 = reinterpret_cast<double*>(take(q, 8 * nr * B));
  double* U1 = reinterpret_cast<double*>(take(q, 8 * nr * B));
  double* U2 = reinterpret_cast<double*>(take(q, 8 * nr * B));
  float* Zf = reinterpret_cast<float*>(take(q, 4 * nr * B));
  float2* Kp = reinterpret_cast<float2*>(take(q, 8 * 32 * B));
  float* df = reinterpret_cast<float*>(take(q, 4 * (2 * (size_t)n + r) * B));
  uint8_t* piv = reinterpret_cast<uint8_t*>(u8_ws);
  cudaError_t ce;
  if (n <= EIGH_F64_MAX) {
    cx<double>* Vhd = Hd + nn * B;
    {
      ProfScope ps(st, K_ELEMWISE);
      const dim3 grid((unsigned)std::min<size_t>((nn + 255) / 256, 1024), batch);
      cx_f2d_kernel<<<grid, 256, 0, st>>>(H, sH, n, n, n, Hd, (long long)nn);
    }
    if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
    if ((ce = cudaMemsetAsync(Vhd, 0, 16 * nn * B, st)) != cudaSuccess) return ce;
    if ((ce = tridiag_smem_keep(st, Hd, (long long)nn, n, dd, ed, n, Vhd, (long long)nn, batch)) != cudaSuccess)
      return ce;
    ProfScope ps(st, K_ELEMWISE);
    cx_d2f_kernel<<<1024, 256, 0, st>>>(Vhd, Vhf, (long long)(nn * B));
    if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  } else {
    if ((ce = cudaMemsetAsync(Vhf, 0, 8 * nn * B, st)) != cudaSuccess) return ce;
    if ((ce = tridiag_df(st, H, sH, n, reinterpret_cast<float4*>(Hd), P, Kp, dd, ed, Vhf, batch)) != cudaSuccess)
      return ce;
  }
  {
    ProfScope ps(st, K_ELEMWISE);
    tridiag_phases_kernel<double><<<batch, 256, 0, st>>>(ed, n, n, eabs, phid);
  }
  if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  if ((ce = bisect_f64(st, dd, eabs, n, r, df, lam, batch, BISECT_C64)) != cudaSuccess) return ce;
  if ((ce = inviter64<float>(st, dd, eabs, n, r, lam, Zf, Z, Ls, U0, U1, U2, piv, batch)) != cudaSuccess) return ce;
  {
    ProfScope ps(st, K_ELEMWISE);
    cx_d2f_kernel<<<64, 256, 0, st>>>(phid, phif, (long long)(n * B));
  }
  if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  ce = backtransform_wy<float>(st, Vhf, (long long)nn, n, Zf, (long long)nr, phif, n, r, U, sU, Tw, wyws, batch);
  if (ce != cudaSuccess) return ce;
  return qr<float>(st, U, sU, n, r, U, sU, nullptr, 0, qrws, batch);
}

template <typename R>
cudaError_t gram_entropy(cudaStream_t st, cx<R>* H, long long sH, int n, void* cx_ws, void* re_ws, int batch,
                         double* S, long long sS) {
  if (batch <= 0) return cudaSuccess;
  if (n <= 1) return cudaMemset2DAsync(S, sizeof(double) * sS, 0, sizeof(double), batch, st);
  cx<R>* e = reinterpret_cast<cx<R>*>(cx_ws);       // batch x n
  cx<R>* phi = e + (long long)batch * n;            // batch x n
  cx<R>* P = phi + (long long)batch * n;            // batch x n
  cx<R>* Vh = P + (long long)batch * n;             // batch x n x n
  R* d = reinterpret_cast<R*>(re_ws);               // batch x n
  R* eabs = d + (long long)batch * n;               // batch x n
  R* lam = eabs + (long long)batch * n;             // batch x n
  double* Kp = reinterpret_cast<double*>(lam + (long long)batch * n + 1);
  Kp = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(Kp) + 15) & ~uintptr_t(15));
  cudaError_t ce;
  if (smem_cluster_size<R>(n) > 0) {
    ce = tridiag_smem<R>(st, H, sH, n, d, e, n, Vh, (long long)n * n, batch);
  } else {
    if ((ce = cudaMemsetAsync(Vh, 0, sizeof(cx<R>) * (size_t)batch * n * n, st)) != cudaSuccess) return ce;
    ce = tridiag_global<R>(st, H, sH, n, d, e, n, P, Kp, Vh, (long long)n * n, batch);
  }
  if (ce != cudaSuccess) return ce;
  {
    ProfScope ps(st, K_ELEMWISE);
    tridiag_phases_kernel<R><<<batch, 256, 0, st>>>(e, n, n, eabs, phi);
  }
  if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  const int total = batch * n;
  {
    ProfScope ps(st, K_BISECT);
    bisect_kernel<R><<<(total * 32 + 255) / 256, 256, 0, st>>>(d, eabs, n, n, n, lam, n, total);
  }
  if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  {
    ProfScope ps(st, K_ELEMWISE);
    entropy_kernel<R><<<batch, 256, 0, st>>>(lam, n, n, S, sS);
  }
  return cudaGetLastError();
}

#define NNE_INST_LINALG(R)                                                                                       \
  template cudaError_t eigh_top<R>(cudaStream_t, cx<R>*, long long, int, int, cx<R>*, long long, void*, void*, \
                                   void*, int, int*);                                                       \
  template cudaError_t gram_entropy<R>(cudaStream_t, cx<R>*, long long, int, void*, void*, int, double*, long long);
NNE_INST_LINALG(float)
NNE_INST_LINALG(double)

}  // namespace nne
