// Hermitian eigensolver pieces for matrices that fit in one cluster's shared
// memory (n <= 640 complex64 / 448 complex128 with 16 CTAs), plus the
// blocked (compact-WY) back-transformation shared by both reduction paths.
#include <map>
#include <mutex>
#include <tuple>

#include "kernels.cuh"
#include "recip.cuh"

namespace cg = cooperative_groups;

namespace nne {

constexpr int KEEP_THREADS = 256;
struct PublishShared {
  double red[KEEP_THREADS / 32];
  double ax0, ph[2], xn, inv;
};
// Named barriers of a part of the block's warps.
__device__ __forceinline__ void barrier_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void barrier_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The reflector of row r (x0 = conj of its first entry) by the 256 threads of the
// owning CTA: v goes to vd of every CTA of the cluster, conj(v) to row r of Vh, and
// d[r], e[r] = alpha.  The last warp forms |x0| and its phase, a divide per lane, while the
// others sum the norm: as one thread's chain the three square roots and five
// divides (some 650 cycles each) were 40 % of a column.
__device__ __forceinline__ void tridiag_publish(cg::cluster_group& cluster, const cx<double>* Hl_row, int n, int r,
                                                cx<double>* vd, cx<double>* Vh, double* d, cx<double>* e,
                                                PublishShared& sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, last = KEEP_THREADS / 32 - 1;
  const int m = n - r - 1;
  if (warp == last) {
    const cx<double> x0 = conj(Hl_row[r + 1]);
    const double s = fmax(fabs(x0.re), fabs(x0.im)), mine = lane & 1 ? x0.im : x0.re;
    const bool nz = s > 0.0;
    const double q = mine / (nz ? s : 1.0);
    const double a = __shfl_sync(0xffffffffu, q, 0), b = __shfl_sync(0xffffffffu, q, 1);
    const double rr = sqrt(a * a + b * b);
    if (lane == 0) sh.ax0 = nz ? s * rr : 0.0;
    __syncwarp();
    barrier_arrive(2, 64);
    const double ph = q / (nz ? rr : 1.0);
    if (lane < 2) sh.ph[lane] = nz ? ph : (lane ? 0.0 : 1.0);
  } else {
    double sp = 0;
    if (tid < m) sp += norm2(Hl_row[r + 1 + tid]);
    sp = warp_sum_r(sp);
    if (lane == 0) sh.red[warp] = sp;
    __syncwarp();
    barrier_sync(1, KEEP_THREADS - 32);
    if (warp == 0) {
      double xn2 = 0;
      for (int w2 = 0; 32 * w2 < m; ++w2) xn2 += sh.red[w2];
      const double xn = sqrt(xn2);
      barrier_sync(2, 64);
      double un = 0;
      if (xn > 0.0) un = sqrt(2.0 * xn2 + 2.0 * xn * sh.ax0);
      if (lane == 0) {
        sh.xn = xn;
        sh.inv = un > 0.0 ? 1.0 / un : 0.0;
      }
    }
  }
  __syncthreads();
  const double xn = sh.xn, inv = sh.inv;
  const cx<double> alpha = xn > 0.0 ? mk<double>(-xn * sh.ph[0], -xn * sh.ph[1]) : mk<double>(0, 0);
  if (tid == KEEP_THREADS - 1) {
    d[r] = Hl_row[r].re;
    e[r] = alpha;
  }
  if (tid < m) {
    cx<double> u = conj(Hl_row[r + 1 + tid]);
    if (tid == 0) u = u - alpha;
    const cx<double> v = inv * u;
    for (int c = 0; c < (int)cluster.num_blocks(); ++c) cluster.map_shared_rank(vd, c)[tid] = v;
    Vh[(long long)r * n + (r + 1) + tid] = conj(v);
  }
}

// Householder tridiagonalisation of the Hermitian H[z] (n x n, n <= 224) by one
// cluster.  Rows are dealt to the CTAs cyclically and stay in shared memory.
// Column j: every CTA forms p = A v on its rows and stores p and its warps' shares of
// K = v^H p into every CTA; after a cluster barrier each applies
// A <- A - v w^H - w v^H with w = 2p - 2Kv to its rows, and the owner of row j+1 forms
// v_{j+1} and stores it into every CTA; a second barrier closes the column.  Sums run in
// a fixed order: the results, to the last bit, are those that small jobs follow.
// Bound by its chain of float64 instructions (64 cycles each).  Stores into the other CTAs
// in place of loads from them, no add of a zero share and the reflector's chain over
// two warps: 1 to 5 matrices of 64 rows 532 -> 378 us, of 160 rows 1904 -> 1490; 40 of
// 64 rows 732 -> 585.
__global__ void __launch_bounds__(KEEP_THREADS) tridiag_smem_kernel(const cx<double>* Hb, long long sH, int n, double* db,
                                                                    cx<double>* eb, int ldde, cx<double>* Vhb,
                                                                    long long sVh, int maxloc) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int z = blockIdx.y;
  const cx<double>* H = Hb + z * sH;
  double* d = db + (long long)z * ldde;
  cx<double>* e = eb + (long long)z * ldde;
  cx<double>* Vh = Vhb + z * sVh;
  extern __shared__ unsigned char smem_raw[];
  cx<double>* Hl = reinterpret_cast<cx<double>*>(smem_raw);     // [maxloc][n] own rows
  cx<double>* vbuf = Hl + (long long)maxloc * n;                // 2 x n: v of even and of odd columns
  cx<double>* p = vbuf + 2 * n;                                 // n
  cx<double>* w = p + n;                                        // n: w = 2p - 2Kv
  constexpr int NW = KEEP_THREADS / 32;
  __shared__ double kpart[16][NW];                              // all warps' shares of K
  __shared__ PublishShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nloc = n > rank ? (n - rank + CS - 1) / CS : 0;
  for (long long e2 = tid; e2 < (long long)nloc * n; e2 += KEEP_THREADS) {
    const int li = (int)(e2 / n), c = (int)(e2 % n);
    Hl[e2] = H[(long long)(rank + li * CS) * n + c];
  }
  // every CTA of the cluster is running before anyone writes into its shared memory
  cluster.sync();
  if (n > 2 && rank == 0) tridiag_publish(cluster, Hl, n, 0, vbuf, Vh, d, e, sh);
  cluster.sync();
  for (int j = 0; j + 2 < n; ++j) {
    const int m = n - j - 1;
    const cx<double>* v = vbuf + (j & 1) * n;
    // p = A v on own rows i > j; K share = sum Re(conj(v_t) p_t)
    const int lstart = (j + 1 - rank + CS - 1) / CS;
    double kp = 0;
    for (int li = lstart + warp; li < nloc; li += NW) {
      const int i = rank + li * CS, t = i - j - 1;
      const cx<double>* row = Hl + (long long)li * n + (j + 1);
      cx<double> a0 = mk<double>(0, 0), a1 = a0, a2 = a0, a3 = a0;
      int k = lane;
      for (; k + 96 < m; k += 128) {
        fma_(a0, row[k], v[k]);
        fma_(a1, row[k + 32], v[k + 32]);
        fma_(a2, row[k + 64], v[k + 64]);
        fma_(a3, row[k + 96], v[k + 96]);
      }
      for (; k < m; k += 32) fma_(a0, row[k], v[k]);
      if (m > 96) a0 = (a0 + a1) + (a2 + a3);
      // lanes 0-15 sum the real parts, 16-31 the imaginary
      const bool im = lane >= 16;
      double s = (im ? a0.im : a0.re) + __shfl_xor_sync(0xffffffffu, im ? a0.re : a0.im, 16);
      for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const cx<double> acc = mk<double>(__shfl_sync(0xffffffffu, s, 0), __shfl_sync(0xffffffffu, s, 16));
      if (lane < CS) cluster.map_shared_rank(p, lane)[t] = acc;
      kp += v[t].re * acc.re + v[t].im * acc.im;
    }
    if (lane < CS) *cluster.map_shared_rank(&kpart[rank][warp], lane) = kp;
    const int nact = min(NW, (m + CS - 1) / CS);   // warps with rows, at most, in any CTA
    cluster.sync();
    if (32 * warp < m) {
      double kk = 0;
      if (lane < CS)
        for (int w2 = 0; w2 < nact; ++w2) kk += kpart[lane][w2];
      for (int o = 1; o < 32; o <<= 1) {
        const double other = __shfl_down_sync(0xffffffffu, kk, o);
        kk += (lane + o < 32) ? other : 0.0;
      }
      const double twoK = 2.0 * __shfl_sync(0xffffffffu, kk, 0);
      if (tid < m) {
        const cx<double> pt = p[tid], vt = v[tid];
        w[tid] = mk<double>(2 * pt.re - twoK * vt.re, 2 * pt.im - twoK * vt.im);
      }
    }
    __syncthreads();
    for (int li = lstart + warp; li < nloc; li += NW) {
      const int i = rank + li * CS, t = i - j - 1;
      cx<double>* row = Hl + (long long)li * n + (j + 1);
      const cx<double> vt = v[t], wt = w[t];
#pragma unroll 4
      for (int k = lane; k < m; k += 32) {
        cx<double> a = row[k];
        const cx<double> wk = w[k], vk = v[k];
        a.re -= vt.re * wk.re + vt.im * wk.im + wt.re * vk.re + wt.im * vk.im;
        a.im -= vt.im * wk.re - vt.re * wk.im + wt.im * vk.re - wt.re * vk.im;
        row[k] = a;
      }
    }
    // the owner of row j+1 forms the next reflector
    if (j + 3 < n && rank == (j + 1) % CS) {
      __syncthreads();
      tridiag_publish(cluster, Hl + (long long)((j + 1) / CS) * n, n, j + 1, vbuf + ((j + 1) & 1) * n, Vh, d, e, sh);
    }
    cluster.sync();
  }
  if (tid == 0) {
    if (n >= 2) {
      if ((n - 2) % CS == rank) d[n - 2] = Hl[(long long)((n - 2) / CS) * n + (n - 2)].re;
      if ((n - 1) % CS == rank) {
        d[n - 1] = Hl[(long long)((n - 1) / CS) * n + (n - 1)].re;
        e[n - 2] = Hl[(long long)((n - 1) / CS) * n + (n - 2)];
      }
    } else if (rank == 0) {
      d[0] = Hl[0].re;
    }
  }
}

// Householder tridiagonalisation of the Hermitian H[z] (n x n) by one
// cluster, the rows dealt to the CTAs cyclically and in shared memory.
//
// One exchange per column, as the double-float kernel (k_tridiag_df.cu): the
// rank-2 update of column j shares a pass with the product p = A v_{j+1}; the
// CTAs push their part of p to all others before the column's only cluster
// barrier, and after it every CTA forms K = v^H p, w = 2p - 2Kv, the next column
// (row j+1 of its owner, less its part of the update) and its reflector itself.
//
// In float64 the time is the number of float64 instructions on a column's chain
// times 64 cycles (an SM issues one per 19 cycles, a warp one per 64, whatever
// the lanes): two rows share a warp's reduction, single values (K, norm, pivot)
// are formed by one warp, the pivot's parts on lanes of one instruction stream
// and from reciprocal square roots by series instead of divides.  us per launch
// (the earlier two-barrier kernel in brackets), float64: n = 64:
// 387 (515), 256: 3129 (4163); float32, n = 128: 234 (328).
// Sums run in a fixed order.
// Pivots smaller than SMALL are scaled by UP before they are squared (their squares
// would be denormal and |x0| inaccurate, and the reflector not unitary).
template <typename R> struct PivotScale;
template <> struct PivotScale<float> {
  static __device__ __forceinline__ float small() { return 0x1p-50f; }
  static __device__ __forceinline__ float up() { return 0x1p70f; }
  static __device__ __forceinline__ float dn() { return 0x1p-70f; }
  static __device__ __forceinline__ float floor2() { return 0.f; }         // squared norms at or below count as null
};
template <> struct PivotScale<double> {
  static __device__ __forceinline__ double small() { return 0x1p-400; }
  static __device__ __forceinline__ double up() { return 0x1p500; }
  static __device__ __forceinline__ double dn() { return 0x1p-500; }
  static __device__ __forceinline__ double floor2() { return 0x1p-1000; }  // the estimate flushes denormals
};

constexpr int TRI_THREADS = 256, TRI_NW = TRI_THREADS / 32;

template <typename R, int EPT>
__global__ void __launch_bounds__(TRI_THREADS) tridiag_fused_kernel(const cx<R>* Hb, long long sH, int n, R* db,
                                                                     cx<R>* eb, int ldde, cx<R>* Vhb, long long sVh,
                                                                     int maxloc) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int z = blockIdx.y;
  const cx<R>* H = Hb + z * sH;
  R* d = db + (long long)z * ldde;
  cx<R>* e = eb + (long long)z * ldde;
  cx<R>* Vh = Vhb + z * sVh;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<R>* Hl = reinterpret_cast<cx<R>*>(smem_raw);     // [maxloc][n] own rows
  cx<R>* vb = Hl + (long long)maxloc * n;             // [2][n] reflectors of this and the last column
  cx<R>* pb = vb + 2 * n;                             // [2][n] p of all rows, then w in its place
  R* kbuf = reinterpret_cast<R*>(pb + 2 * n);         // [2][CS][NW] shares of K, pushed by their warps
  __shared__ R redN[TRI_NW];
  __shared__ cx<R> x0_s, alpha_s;
  __shared__ R inv_s, K_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nloc = n > rank ? (n - rank + CS - 1) / CS : 0;
  auto in = [&](int i, int c) { return H[(long long)i * n + c]; };
  for (long long q = tid; q < (long long)nloc * n; q += TRI_THREADS) {
    const int li = (int)(q / n), c = (int)(q % n), i = rank + li * CS;
    Hl[q] = in(i, c);
  }
  auto warp_real = [&](R v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  cx<R> x[EPT];   // the current column below its diagonal, entries tid, tid + 256, ...
#pragma unroll
  for (int q = 0; q < EPT; ++q) x[q] = tid + q * TRI_THREADS < n - 1 ? conj(in(0, tid + q * TRI_THREADS + 1)) : mk<R>(0, 0);
  // reflector r from the column x (m entries) -> vout, Vh row r, e[r]
  auto reflector = [&](int r, int m, cx<R>* vout) {
    if (32 * warp < m) {
      R s = 0;
#pragma unroll
      for (int q = 0; q < EPT; ++q)
        if (tid + q * TRI_THREADS < m) s += norm2(x[q]);
      s = warp_real(s);
      if (lane == 0) redN[warp] = s;
    } else if (lane == 0) {
      redN[warp] = R(0);
    }
    if (tid == 0) x0_s = x[0];
    __syncthreads();
    if (warp == 0) {
      R xn2 = lane < TRI_NW ? redN[lane] : R(0);
      for (int o = TRI_NW / 2; o > 0; o >>= 1) xn2 += __shfl_xor_sync(0xffffffffu, xn2, o);
      xn2 = __shfl_sync(0xffffffffu, xn2, 0);
      using PS = PivotScale<R>;
      cx<R> x0 = x0_s;
      const bool tiny = fmax(fabs(x0.re), fabs(x0.im)) < PS::small();
      if (tiny) x0 = PS::up() * x0;
      const R q2 = norm2(x0);
      // lane 0: 1 / |x0|, lane 1: 1 / ||x||, in one evaluation
      const R arg = lane == 0 ? q2 : xn2;
      const R is = arg > PS::floor2() ? rsqrt_series(arg) : R(0);
      const R root = arg * is;   // |x0|, ||x||
      const R qi = __shfl_sync(0xffffffffu, is, 0), ax0s = __shfl_sync(0xffffffffu, root, 0),
              xn = __shfl_sync(0xffffffffu, root, 1);
      // alpha = -e^{i arg x0} ||x||: real part on lane 0, imaginary on lane 1
      const R ph = ((lane == 0 ? x0.re : x0.im) * qi);
      const R al = -(qi > R(0) ? ph : (lane == 0 ? R(1) : R(0))) * xn;
      const R ax0 = tiny ? ax0s * PS::dn() : ax0s;
      const R un2 = R(2) * fma(xn, ax0, xn2);
      const R inv = xn > R(0) ? rsqrt_series(un2) : R(0);
      const R al_im = __shfl_sync(0xffffffffu, al, 1);
      if (lane == 0) {
        alpha_s = mk<R>(al, al_im);
        inv_s = inv;
        if (rank == 0) e[r] = mk<R>(al, al_im);
      }
    }
    __syncthreads();
    const R inv = inv_s;
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      const int t = tid + q * TRI_THREADS;
      if (t < m) {
        cx<R> u = x[q];
        if (t == 0) u = u - alpha_s;
        const cx<R> v = inv * u;
        vout[t] = v;
        if (rank == r % CS) {
          Vh[(long long)r * n + r + 1 + t] = conj(v);   // conjugated, for the back-transformation
        }
      }
    }
    // left of the reflector: zeros
    if (rank == r % CS)
      for (int t = tid; t <= r; t += TRI_THREADS) Vh[(long long)r * n + t] = mk<R>(0, 0);
  };
  // a -= v conj(wk) + w conj(vk)
  auto rank2 = [](cx<R>& a, cx<R> vt, cx<R> wt, cx<R> vk, cx<R> wk) {
    a.re -= vt.re * wk.re + vt.im * wk.im + wt.re * vk.re + wt.im * vk.im;
    a.im -= vt.im * wk.re - vt.re * wk.im + wt.im * vk.re - wt.re * vk.im;
  };
  if (n > 2) reflector(0, n - 1, vb);
  if (rank == 0 && tid == 0) d[0] = in(0, 0).re;
  int oc = 1 % CS, ol = 1 / CS;   // row j + 1: its CTA and place there
  cluster.sync();   // every CTA of the cluster runs before anyone writes into its shared memory
  for (int j = 0; j + 2 < n; ++j) {
    const int m = n - j - 1, buf = j & 1;
    const cx<R>* v = vb + buf * n;               // v_j: entry t is row j + 1 + t
    const cx<R>* vo = vb + (buf ^ 1) * n + 1;    // v_{j-1}, w_{j-1} at row j + 1
    const cx<R>* wo = pb + (buf ^ 1) * n + 1;
    cx<R>* p = pb + buf * n;
    // own rows i > j, two per warp at a time: update with column j - 1, product with v_j
    const int l0 = ol + (oc > rank ? 1 : 0);
    R ks = 0;
    for (int li = l0 + warp; li < nloc; li += 2 * TRI_NW) {
      const bool two = li + TRI_NW < nloc;
      const int t = rank + li * CS - j - 1, t2 = t + TRI_NW * CS;
      cx<R>* row = Hl + (long long)li * n + (j + 1);
      cx<R>* row2 = Hl + (long long)(two ? li + TRI_NW : li) * n + (j + 1);
      cx<R> a0 = mk<R>(0, 0), a1 = a0, b0 = a0, b1 = a0;
      if (j == 0) {
        for (int k = lane; k < m; k += 32) {
          fma_(a0, row[k], v[k]);
          if (two) fma_(b0, row2[k], v[k]);
        }
      } else {
        const cx<R> vt = vo[t], wt = wo[t], vt2 = two ? vo[t2] : vt, wt2 = two ? wo[t2] : wt;
        int k = lane;
        for (; k + 32 < m; k += 64) {
          cx<R> r0 = row[k], r1 = row[k + 32];
          const cx<R> wk0 = wo[k], vk0 = vo[k], wk1 = wo[k + 32], vk1 = vo[k + 32];
          const cx<R> v0 = v[k], v1 = v[k + 32];
          rank2(r0, vt, wt, vk0, wk0);
          rank2(r1, vt, wt, vk1, wk1);
          row[k] = r0;
          row[k + 32] = r1;
          fma_(a0, r0, v0);
          fma_(a1, r1, v1);
          if (two) {
            r0 = row2[k];
            r1 = row2[k + 32];
            rank2(r0, vt2, wt2, vk0, wk0);
            rank2(r1, vt2, wt2, vk1, wk1);
            row2[k] = r0;
            row2[k + 32] = r1;
            fma_(b0, r0, v0);
            fma_(b1, r1, v1);
          }
        }
        for (; k < m; k += 32) {
          cx<R> r0 = row[k];
          rank2(r0, vt, wt, vo[k], wo[k]);
          row[k] = r0;
          fma_(a0, r0, v[k]);
          if (two) {
            r0 = row2[k];
            rank2(r0, vt2, wt2, vo[k], wo[k]);
            row2[k] = r0;
            fma_(b0, r0, v[k]);
          }
        }
        a0 = a0 + a1;
        b0 = b0 + b1;
      }
      // both rows' sums in five steps: lanes 0-15 end with the first row's, 16-31 with the second's
      const bool up = lane & 16;
      cx<R> s = (up ? b0 : a0) + shfl_xor(up ? a0 : b0, 16);
      for (int o = 8; o > 0; o >>= 1) s = s + shfl_xor(s, o);
      if (!up || two) {
        const int tr = up ? t2 : t;
        const cx<R> vt = v[tr];
        ks += vt.re * s.re + vt.im * s.im;   // the same on 16 lanes
        if ((lane & 15) < CS) *cluster.map_shared_rank(p + tr, lane & 15) = s;
      }
    }
    {
      const R kw = ks + __shfl_xor_sync(0xffffffffu, ks, 16);
      if (lane < CS) cluster.map_shared_rank(kbuf + (buf * CS + rank) * TRI_NW, lane)[warp] = kw;
    }
    cluster.sync();
    // row j + 1 (its owner's last word on it)
    cx<R> a[EPT];
    const cx<R>* rj1 = cluster.map_shared_rank(Hl + (long long)ol * n + (j + 1), oc);
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      const int t = tid + q * TRI_THREADS;
      a[q] = t + 1 < m ? conj(rj1[t + 1]) : mk<R>(0, 0);   // entry (j + 2 + t, j + 1) by symmetry
    }
    if (warp == 0) {
      R K = 0;
      for (int q = lane; q < CS * TRI_NW; q += 32) K += kbuf[buf * CS * TRI_NW + q];
      K = warp_real(K);
      if (lane == 0) K_s = R(2) * K;
    }
    __syncthreads();
    const R twoK = K_s;
    auto wof = [&](cx<R> vt, cx<R> pt) { return mk<R>(pt.re + pt.re - twoK * vt.re, pt.im + pt.im - twoK * vt.im); };
    if (32 * warp + 1 < m) {
      const cx<R> v0 = v[0], w0 = wof(v0, p[0]);
#pragma unroll
      for (int q = 0; q < EPT; ++q) {
        const int t = tid + q * TRI_THREADS;
        if (t + 1 < m) {
          const cx<R> vt = v[t + 1], wt = wof(vt, p[t + 1]);
          p[t + 1] = wt;   // (entry 0 stays p: no row needs w_0 again)
          rank2(a[q], vt, wt, v0, w0);
        }
        x[q] = a[q];
      }
      if (rank == oc && tid == 0) {
        // d[j + 1] = A[j+1][j+1] - 2 Re(v_0 conj(w_0))
        d[j + 1] = Hl[(long long)ol * n + (j + 1)].re - R(2) * (v0.re * w0.re + v0.im * w0.im);
      }
    }
    if (++oc == CS) {   // to row j + 2
      oc = 0;
      ++ol;
    }
    if (j + 3 < n) {
      reflector(j + 1, m - 1, vb + (buf ^ 1) * n);
    } else if (tid == 0) {
      // the last 2 x 2 block: subdiagonal, and the corner by its owner
      if (rank == (n - 1) % CS) {
        const cx<R> v0 = v[0], w0 = wof(v0, p[0]), v1 = v[1], w1 = p[1];
        cx<R> sub = Hl[(long long)((n - 1) / CS) * n + (n - 2)];
        rank2(sub, v1, w1, v0, w0);
        e[n - 2] = sub;
        d[n - 1] = Hl[(long long)((n - 1) / CS) * n + (n - 1)].re - R(2) * (v1.re * w1.re + v1.im * w1.im);
      }
    }
    __syncthreads();
  }
  if (n == 2 && rank == 0 && tid == 0) {
    d[1] = in(1, 1).re;
    e[0] = in(1, 0);
  }
  cluster.sync();   // rows of this CTA may still be read by others
}

// U[k][c] = phi_k Z[k][c] (complex from the real tridiagonal eigenvectors).
template <typename R>
__global__ void phase_scale_kernel(const R* Zb, long long sZ, const cx<R>* phib, int ldde, int n, int r, cx<R>* Ub,
                                   long long sU) {
  const int z = blockIdx.y;
  const R* Z = Zb + z * sZ;
  const cx<R>* phi = phib + (long long)z * ldde;
  cx<R>* U = Ub + z * sU;
  const long long count = (long long)n * r;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(i / r);
    U[i] = Z[i] * phi[k];
  }
}

// Compact-WY factors of blocks of 32 consecutive tridiagonal reflectors:
// block b (reflectors 32b .. 32b+bw-1) gives T_b with
// P_{32b} ... P_{32b+bw-1} = I - V_b T_b V_b^H, V_b^H = Vh rows 32b...
// The Gram matrix by 2 x 2 entries per thread (upper triangle only) over WT_C staged
// columns, then T with one row per lane: column l, once known, goes into the sums of
// all columns right of it.  Both sum in ascending order.  One CTA per block of
// reflectors, bound by the Gram's chains (64 rows 56 -> 14 us; the complex64 eigenproblems of
// chi 64, 256 rows, 160 -> 25 us: each entry used to walk two rows in global memory).
constexpr int WT_C = 32;
template <typename R>
__global__ void __launch_bounds__(256) wy_t_kernel(const cx<R>* Vhb, long long sVh, int n, int nref, cx<R>* Tb,
                                                    long long sT) {
  __shared__ cx<R> G[32][33];
  __shared__ cx<R> Vs[32][WT_C + 1];
  const int b = blockIdx.x, z = blockIdx.y;
  const cx<R>* Vh = Vhb + z * sVh;
  cx<R>* T = Tb + z * sT + (long long)b * 1024;
  const int j0 = 32 * b, bw = min(32, nref - j0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // thread q of the first 136 forms entries (a, c), (a, c + 16), (a + 16, c), (a + 16, c + 16), a <= c < 16
  int a = 0, c = 0;
  if (tid < 136) {
    int q = tid;
    while (q >= 16 - a) q -= 16 - a++;
    c = a + q;
  }
  cx<R> g00 = mk<R>(0, 0), g01 = g00, g11 = g00, g10 = g00;
  for (int c0 = j0 + 1; c0 < n; c0 += WT_C) {
    for (int r = warp; r < 32; r += 8)
      Vs[r][lane] = r < bw && c0 + lane < n ? Vh[(long long)(j0 + r) * n + c0 + lane] : mk<R>(0, 0);
    __syncthreads();
    if (tid < 136) {
      const int m = min(WT_C, n - c0);
#pragma unroll 4
      for (int i = 0; i < m; ++i) {
        // rows hold conj(v): G[a][c] = v_a^H v_c = sum conj(Vh_c) Vh_a
        const cx<R> a0 = Vs[a][i], a1 = Vs[a + 16][i], b0 = Vs[c][i], b1 = Vs[c + 16][i];
        fmac_(g00, b0, a0);
        fmac_(g01, b1, a0);
        fmac_(g10, a1, b0);   // (c, a + 16), the mirror of (a + 16, c), which lies below the diagonal
        fmac_(g11, b1, a1);
      }
    }
    __syncthreads();
  }
  if (tid < 136) {
    G[a][c] = g00;
    G[a][c + 16] = g01;
    G[c][a + 16] = g10;
    G[a + 16][c + 16] = g11;
  }
  __syncthreads();
  if (warp == 0) {
    cx<R> acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = mk<R>(0, 0);
#pragma unroll
    for (int l = 0; l < 32; ++l) {
      cx<R> t = mk<R>(0, 0);
      if (l < bw) {
        const R tau = G[l][l].re > R(0.5) ? R(2) : R(0);
        if (lane < l) t = mk<R>(-tau * acc[l].re, -tau * acc[l].im);
        if (lane == l) t = mk<R>(tau, 0);
      }
      T[lane * 32 + l] = t;
      if (lane <= l && l < bw) {
#pragma unroll
        for (int i = l + 1; i < 32; ++i) fma_(acc[i], t, G[l][i]);
      }
    }
  }
}

template <typename K, typename... Args>
static cudaError_t launch_cl(K kernel, int cs, int batch, size_t smem, cudaStream_t st, Args... args) {
  cudaError_t e = ensure_kernel_smem((const void*)kernel, smem, cs > 8);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs, batch, 1);
  cfg.blockDim = dim3(256, 1, 1);
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

constexpr size_t SMEM_LIMIT = 226 * 1024;   // dynamic shared memory per CTA (227 KB less the static part)

template <typename R>
static size_t tridiag_smem_bytes(int n, int cs) {
  const size_t maxloc = (n + cs - 1) / cs;
  return sizeof(cx<R>) * (maxloc * n + 4 * (size_t)n) + sizeof(R) * 2 * 16 * TRI_NW;
}

// Smallest power-of-two cluster whose shared memory holds the matrix (0: none does).
template <typename R>
int smem_cluster_size(int n) {
  for (int cs = 1; cs <= 16; cs *= 2) {
    const size_t maxloc = (n + cs - 1) / cs;
    if (tridiag_smem_bytes<R>(n, cs) <= SMEM_LIMIT && (cs >= 16 || maxloc <= 64)) return cs;
  }
  return 0;
}

// Cluster size for `batch` matrices: among the sizes from smem_cluster_size(n)
// up to `most` that hold the matrix, the largest whose clusters all fit on the GPU
// at once (cudaOccupancyMaxActiveClusters); a cluster of 16 does not fit on
// every GPC, so for a batch of 8 a size of 13 or 14 can finish in one wave
// where 16 needs two.  Cached per kernel, (n, batch) and device.
template <typename R>
static int tridiag_cluster_size(const void* kernel, int n, int batch, int most) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, int, int, int>, int> cache;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  auto key = std::make_tuple(kernel, n, batch, dev);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  const int cs0 = smem_cluster_size<R>(n);
  int best = cs0, best_waves = 1 << 30;
  for (int cs = std::max(cs0, 2); cs <= std::max(cs0, std::min(16, most)) && cs0 > 0; ++cs) {
    const size_t smem = tridiag_smem_bytes<R>(n, cs);
    if (smem > SMEM_LIMIT) continue;
    if (ensure_kernel_smem(kernel, smem, cs > 8) != cudaSuccess) continue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs, batch, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int active = 0;
    if (cudaOccupancyMaxActiveClusters(&active, kernel, &cfg) != cudaSuccess ||
        active < 1) {
      cudaGetLastError();
      continue;
    }
    const int waves = (batch + active - 1) / active;
    if (waves < best_waves || (waves == best_waves && cs > best)) {
      best_waves = waves;
      best = cs;
    }
  }
  cache[key] = best;
  return best;
}

template <typename R>
cudaError_t tridiag_smem(cudaStream_t st, const cx<R>* H, long long sH, int n, R* d, cx<R>* e, int ldde, cx<R>* Vh,
                         long long sVh, int batch) {
  if (smem_cluster_size<R>(n) == 0 || n > 3 * TRI_THREADS) return cudaErrorInvalidValue;
  auto kernel = n <= TRI_THREADS ? tridiag_fused_kernel<R, 1> : tridiag_fused_kernel<R, 3>;
  const int cs = tridiag_cluster_size<R>((const void*)kernel, n, batch, (n + 7) / 8);
  const size_t smem = tridiag_smem_bytes<R>(n, cs);
  ProfScope ps(st, K_TRIDIAG, 1, 16.0 / 3.0 * (double)n * n * n * batch);   // Hermitian tridiagonalisation flops
  return launch_cl(kernel, cs, batch, smem, st, H, sH, n, d, e, ldde, Vh, sVh, (n + cs - 1) / cs);
}

// The two-barrier kernel, for the float64 reduction of complex64 states' small
// eigenproblems (n <= EIGH_F64_MAX), whose last bits small jobs' results follow.
cudaError_t tridiag_smem_keep(cudaStream_t st, const cx<double>* H, long long sH, int n, double* d, cx<double>* e,
                              int ldde, cx<double>* Vh, long long sVh, int batch) {
  if (smem_cluster_size<double>(n) == 0 || n > KEEP_THREADS - 32) return cudaErrorInvalidValue;
  const int cs = tridiag_cluster_size<double>((const void*)tridiag_smem_kernel, n, batch, 16);
  const size_t smem = tridiag_smem_bytes<double>(n, cs);
  ProfScope ps(st, K_TRIDIAG, 1, 16.0 / 3.0 * (double)n * n * n * batch);
  return launch_cl(tridiag_smem_kernel, cs, batch, smem, st, H, sH, n, d, e, ldde, Vh, sVh, (n + cs - 1) / cs);
}

template <typename R>
cudaError_t backtransform_wy(cudaStream_t st, const cx<R>* Vh, long long sVh, int n, const R* Z, long long sZ,
                             const cx<R>* phi, int ldde, int r, cx<R>* U, long long sU, cx<R>* Tw, cx<R>* wy_ws,
                             int batch) {
  cudaError_t e;
  {
    ProfScope ps(st, K_BACKTRANSFORM);
    const long long count = (long long)n * r;
    int blocks = (int)std::min<long long>((count + 255) / 256, 1024);
    phase_scale_kernel<R><<<dim3(std::max(blocks, 1), batch), 256, 0, st>>>(Z, sZ, phi, ldde, n, r, U, sU);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const int nref = n - 2;
  if (nref <= 0) return cudaSuccess;
  const int nb = (nref + 31) / 32;
  const long long sT = (long long)nb * 1024;
  {
    ProfScope ps(st, K_BACKTRANSFORM);
    wy_t_kernel<R><<<dim3(nb, batch), 256, 0, st>>>(Vh, sVh, n, nref, Tw, sT);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  for (int b = nb - 1; b >= 0; --b) {
    const int j0 = 32 * b, bw = std::min(32, nref - j0);
    const int r0 = j0 + 1, mb = n - r0;
    const cx<R>* Vb = Vh + (long long)j0 * n + r0;    // bw x mb, rows = conj(v)
    cx<R>* Ub = U + (long long)r0 * r;
    // U_b <- (I - V T V^H) U_b
    if ((e = wy_apply<R>(st, true, Vb, sVh, n, Tw + (long long)b * 1024, sT, 32, false, bw, mb, r, Ub, sU, r, wy_ws,
                         batch)) != cudaSuccess)
      return e;
  }
  return cudaSuccess;
}

#define NNE_INST_EIGS(R)                                                                                        \
  template int smem_cluster_size<R>(int);                                                                       \
  template cudaError_t tridiag_smem<R>(cudaStream_t, const cx<R>*, long long, int, R*, cx<R>*, int, cx<R>*,    \
                                       long long, int);                                                         \
  template cudaError_t backtransform_wy<R>(cudaStream_t, const cx<R>*, long long, int, const R*, long long,    \
                                           const cx<R>*, int, int, cx<R>*, long long, cx<R>*, cx<R>*, int);
NNE_INST_EIGS(float)
NNE_INST_EIGS(double)

}  // namespace nne
