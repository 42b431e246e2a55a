// Householder reduction of complex Hermitian matrices to real tridiagonal form
// in double-float arithmetic (complex64 states' eigenproblems): float64
// quality on the float32 pipes.
//
// tridiag_df_kernel   the matrix in L2, lower triangle only: the first jend
//                     columns of matrices of more than 1024 rows;
// tridiag_dfs_kernel  one exchange per column, the rows in the shared memory of
//                     one cluster (sizes that fit, and the rest of larger
//                     ones) or in L2 (up to 1024 rows).
#include <map>
#include <mutex>
#include <tuple>

#include "df.cuh"
#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace nne {

// Double-float copy of a Hermitian complex64 matrix, both triangles from the lower one.
__global__ void cx_f2df_kernel(const cx<float>* X, long long sX, int n, float4* Y, long long sY) {
  const long long count = (long long)n * n;
  const int z = blockIdx.y;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / n), c = (int)(i % n);
    const cx<float> v = X[z * sX + (c <= r ? i : (long long)c * n + r)];
    Y[z * sY + i] = make_float4(v.re, 0.f, c < r ? v.im : (c > r ? -v.im : 0.f), 0.f);
  }
}

// Upper triangle of the trailing block from row and column `off` on <- conjugate of the lower.
__global__ void df_mirror_kernel(float4* Y, long long sY, int n0, int off) {
  const int n = n0 - off, z = blockIdx.y;
  const long long count = (long long)n * n;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / n), c = (int)(i % n);
    if (c <= r) continue;
    const float4 a = Y[z * sY + (long long)(off + c) * n0 + off + r];
    Y[z * sY + (long long)(off + r) * n0 + off + c] = make_float4(a.x, a.y, -a.z, -a.w);
  }
}

// Every O(m) step of a column is double-float as well (norms, the reflector,
// K, w), so the float64 pipe only sees one thread's pivot per column; the
// reflectors go out rounded to float32 for the float32 back-transformation,
// d and e in float64.
template <int U>
__global__ void __launch_bounds__(512) tridiag_df_kernel(float4* Hb, long long sH, int n, double* db, cx<double>* eb,
                                                          int ldde, float4* Pb, float2* Kb, cx<float>* Vhb,
                                                          long long sVh, int jend) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int z = blockIdx.y;
  float4* H = Hb + z * sH;
  double* d = db + (long long)z * ldde;
  cx<double>* e = eb + (long long)z * ldde;
  float4* P = Pb + (long long)z * ldde;
  float2* Kp = Kb + z * 32;
  extern __shared__ __align__(16) unsigned char df_smem[];
  float4* vdf = reinterpret_cast<float4*>(df_smem);   // n: the Householder vector
  float4* wdf = vdf + n;                              // n: w = 2p - 2Kv
  __shared__ float red[64];
  __shared__ float4 alpha_s;
  __shared__ float2 inv_s;
  const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
  const int gw = rank * nw + warp, GW = CS * nw;

  for (int j = 0; j < jend; ++j) {
    const int m = n - j - 1;
    // column j below the diagonal, and its squared norm
    float nh = 0.f, nl = 0.f;
    {
      const float4* colj = H + (long long)(j + 1) * n + j;
      for (int t = tid; t < m; t += nth) {
        const float4 a = colj[(long long)t * n];
        vdf[t] = a;
        df_mac(nh, nl, a.x, a.y, a.x, a.y);
        df_mac(nh, nl, a.z, a.w, a.z, a.w);
      }
    }
    const float2 xn2f = df_block_sum(nh, nl, red);
    if (tid == 0) {
      // pivot in float64 on one thread: alpha = -e^{i arg x0} ||x||, un = ||x - alpha e0||
      const float4 x0 = vdf[0];
      const cx<double> x0d = mk<double>(df_to_d(x0.x, x0.y), df_to_d(x0.z, x0.w));
      double pr, pi, ax0;
      unit_phase_of(x0d, &pr, &pi, &ax0);
      const double xn2 = df_to_d(xn2f.x, xn2f.y), xn = sqrt(xn2);
      cx<double> alpha = mk<double>(0, 0);
      double un = 0;
      if (xn > 0) {
        alpha = mk<double>(-xn * pr, -xn * pi);
        un = sqrt(2.0 * xn2 + 2.0 * xn * ax0);
      }
      const double inv = un > 0 ? 1.0 / un : 0.0;
      alpha_s = df_from_cd(alpha);
      const float ih = (float)inv;
      inv_s = make_float2(ih, (float)(inv - (double)ih));
      if (rank == 0) {
        const float4 hjj = H[(long long)j * n + j];
        d[j] = df_to_d(hjj.x, hjj.y);
        e[j] = alpha;
      }
    }
    __syncthreads();
    {
      const float4 al = alpha_s;
      const float2 iv = inv_s;
      cx<float>* rj = Vhb + z * sVh + (long long)j * n + (j + 1);
      for (int t = tid; t < m; t += nth) {
        float4 u = vdf[t];
        if (t == 0) {
          df_add(u.x, u.y, -al.x, -al.y);
          df_add(u.z, u.w, -al.z, -al.w);
        }
        const float2 vr = df_mul(u.x, u.y, iv.x, iv.y), vi = df_mul(u.z, u.w, iv.x, iv.y);
        vdf[t] = make_float4(vr.x, vr.y, vi.x, vi.y);
        if (rank == 0) rj[t] = mk<float>(vr.x, -vi.x);   // reflector j, conjugated, for the back-transform
      }
    }
    __syncthreads();
    // p = A v on own rows (lower part of row t, then its upper part read down column t); K = v^H p
    float kh = 0.f, kl = 0.f;
    for (int t = gw; t < m; t += GW) {
      const float4* row = H + (long long)(j + 1 + t) * n + (j + 1);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), acc2 = acc;
      int k = lane;
      for (; k + 32 * (U - 1) <= t; k += 32 * U) {
        float4 a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = row[k + 32 * u];
#pragma unroll
        for (int u = 0; u < U; ++u) df_cmac<false>((u & 1) ? acc2 : acc, a[u], vdf[k + 32 * u]);
      }
      for (; k <= t; k += 32) df_cmac<false>(acc, row[k], vdf[k]);
      const float4* colt = H + (long long)(j + 1) * n + (j + 1 + t);
      k = t + 1 + lane;
      for (; k + 32 * (U - 1) < m; k += 32 * U) {
        float4 a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = colt[(long long)(k + 32 * u) * n];
#pragma unroll
        for (int u = 0; u < U; ++u) df_cmac<true>((u & 1) ? acc2 : acc, a[u], vdf[k + 32 * u]);
      }
      for (; k < m; k += 32) df_cmac<true>(acc, colt[(long long)k * n], vdf[k]);
      df_add(acc.x, acc.y, acc2.x, acc2.y);
      df_add(acc.z, acc.w, acc2.z, acc2.w);
      acc = df_warp_sum(acc);
      if (lane == 0) {
        P[t] = acc;
        const float4 vt = vdf[t];
        df_mac(kh, kl, vt.x, vt.y, acc.x, acc.y);
        df_mac(kh, kl, vt.z, vt.w, acc.z, acc.w);
      }
    }
    {
      const float2 kp = df_block_sum(kh, kl, red);
      if (tid == 0) Kp[rank] = kp;
    }
    __threadfence();
    cluster.sync();
    float Kh = 0.f, Kl = 0.f;
    for (int c = 0; c < CS; ++c) df_add(Kh, Kl, Kp[c].x, Kp[c].y);
    // w = 2p - 2 K v  (2K exact in double-float)
    const float K2h = 2.f * Kh, K2l = 2.f * Kl;
    for (int t = tid; t < m; t += nth) {
      const float4 p = P[t], vt = vdf[t];
      float rh = 2.f * p.x, rl = 2.f * p.y, ih = 2.f * p.z, il = 2.f * p.w;
      df_mac(rh, rl, -K2h, -K2l, vt.x, vt.y);
      df_mac(ih, il, -K2h, -K2l, vt.z, vt.w);
      df_norm(rh, rl);
      df_norm(ih, il);
      wdf[t] = make_float4(rh, rl, ih, il);
    }
    __syncthreads();
    // A <- A - v w^H - w v^H on the lower triangle of own rows (U entries in flight per lane)
    for (int t = gw; t < m; t += GW) {
      float4* row = H + (long long)(j + 1 + t) * n + (j + 1);
      const float4 vt = vdf[t], wt = wdf[t];
      for (int k0 = lane; k0 <= t; k0 += 32 * U) {
        float4 a[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (k0 + 32 * u <= t) a[u] = row[k0 + 32 * u];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = k0 + 32 * u;
          if (k > t) break;
          const float4 wk = wdf[k], vk = vdf[k];
          float4 b = a[u];
          // re: - (vt.re wk.re + vt.im wk.im + wt.re vk.re + wt.im vk.im)
          df_mac(b.x, b.y, -vt.x, -vt.y, wk.x, wk.y);
          df_mac(b.x, b.y, -vt.z, -vt.w, wk.z, wk.w);
          df_mac(b.x, b.y, -wt.x, -wt.y, vk.x, vk.y);
          df_mac(b.x, b.y, -wt.z, -wt.w, vk.z, vk.w);
          // im: - (vt.im wk.re - vt.re wk.im + wt.im vk.re - wt.re vk.im)
          df_mac(b.z, b.w, -vt.z, -vt.w, wk.x, wk.y);
          df_mac(b.z, b.w, vt.x, vt.y, wk.z, wk.w);
          df_mac(b.z, b.w, -wt.z, -wt.w, vk.x, vk.y);
          df_mac(b.z, b.w, wt.x, wt.y, vk.z, vk.w);
          df_norm(b.x, b.y);
          df_norm(b.z, b.w);
          row[k] = b;
        }
      }
    }
    __threadfence();
    cluster.sync();
  }
}

// ---------------------------------------------------------------- one exchange per column
// One cluster per matrix; the rows, both triangles, are dealt cyclically to
// its CTAs.  Thread t of every CTA owns entries t, t + NT, ... (EPT of them) of
// the current column.
//
// What bounds it: per column a chain of one exchange and two sums, and 3
// complex multiply-adds per entry of the trailing matrix on the float32 pipes.
// Hence
//   * one cluster barrier per column: the CTAs push their part of p = A v to
//     all others before it; after it every CTA forms K = v^H p, w, the next
//     column (the stored row j+1 of its owner, minus its part of the rank-2
//     update) and the next reflector itself, with the same operations in the
//     same order, so no second exchange is needed;
//   * one pass over the matrix per column: the rank-2 update of column j and
//     the product with v_{j+1} read and write each entry once;
//   * the pivot is formed by one warp (all warps doing so cost more issue slots
//     than the broadcast; for K of up to 380 rows, and for gathering p to push it in one
//     piece, the extra block barrier cost more than it saved);
//   * no float64: GB300 has two float64 lanes per SM.
// The matrix is scaled by a power of two to a largest diagonal entry in
// [1, 2); columns below norm 2^-50 then count as null (their squares would
// leave float32's range, and an inaccurate norm makes a reflector that is not
// unitary), a backward error of 2^-50 of that entry, below the arithmetic's 2^-46.
//
// ROWS_C64   rows in shared memory, from the complex64 matrix (lower triangle read);
// ROWS_DF    rows in shared memory, from the double-float trailing block at
//            `off` that ROWS_GLOBAL left (lower triangle read), scaled by *pre already;
// ROWS_GLOBAL  rows in place in a double-float matrix (both triangles), columns
//            off .. jend - 1 only, the trailing block then up to date; *pre is set.
// The block starts at row and column `off` and has n = n0 - off rows.
enum DfRows { ROWS_C64, ROWS_DF, ROWS_GLOBAL };

struct DfsLayout {   // shared memory, in float4 from the base
  int n, maxloc;
  bool global;
  __host__ __device__ size_t v() const { return global ? 0 : (size_t)maxloc * n; }   // [2][n] reflectors of this and the last column
  __host__ __device__ size_t w() const { return v() + 2 * (size_t)n; }               // n: w of the last column
  __host__ __device__ size_t p() const { return w() + n; }                           // [2][n] p of all rows, pushed by their owners
  __host__ __device__ size_t k() const { return p() + 2 * (size_t)n; }               // [2][n] float2: the rows' terms of K, pushed with p
  __host__ __device__ size_t bytes() const { return 16 * k() + 2 * sizeof(float2) * (size_t)n; }
};

template <int NT, int EPT, int ROWS>
__global__ void __launch_bounds__(NT) tridiag_dfs_kernel(void* Hsrc, long long sH, int n0, int off, int jend,
                                                         double* db, cx<double>* eb, int ldde, cx<float>* Vhb,
                                                         long long sVh, float* pre, int maxloc) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int z = blockIdx.y, n = n0 - off;
  double* d = db + (long long)z * ldde + off;
  cx<double>* e = eb + (long long)z * ldde + off;
  cx<float>* Vh = Vhb + z * sVh + (long long)off * n0 + off;
  extern __shared__ __align__(16) float4 dfs_smem[];
  constexpr int NW = NT / 32;
  const DfsLayout lay{n, maxloc, ROWS == ROWS_GLOBAL};
  float4* vb = dfs_smem + lay.v();
  float4* wb = dfs_smem + lay.w();
  float4* pb = dfs_smem + lay.p();
  float2* kbuf = reinterpret_cast<float2*>(dfs_smem + lay.k());
  __shared__ float2 redN[NW], redK[NW];
  __shared__ float redM[NW];
  __shared__ float4 x0_s, alpha_s;
  __shared__ float2 inv_s, K_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nloc = n > rank ? (n - rank + CS - 1) / CS : 0;
  auto source = [&](int i, int c) {   // entry (i, c), c <= i
    const long long at = z * sH + (long long)(off + i) * n0 + off + c;
    if (ROWS != ROWS_C64) return reinterpret_cast<const float4*>(Hsrc)[at];
    const cx<float> a = reinterpret_cast<const cx<float>*>(Hsrc)[at];
    return make_float4(a.re, 0.f, a.im, 0.f);
  };
  auto row_of = [&](int li) -> float4* {   // own row li
    if (ROWS == ROWS_GLOBAL)
      return reinterpret_cast<float4*>(Hsrc) + z * sH + (long long)(off + rank + li * CS) * n0 + off;
    return dfs_smem + (long long)li * n;
  };
  // power-of-two scale from the largest diagonal entry
  float mx = 0.f;
  for (int t = tid; t < n; t += NT) mx = fmaxf(mx, fabsf(source(t, t).x));
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) redM[warp] = mx;
  __syncthreads();
  for (int w2 = 0; w2 < NW; ++w2) mx = fmaxf(mx, redM[w2]);
  int ex = 0;
  if (mx > 0.f && mx < INFINITY) ex = min(max(ilogbf(mx), -120), 120);
  const float sc = ldexpf(1.f, -ex);
  const double back = ROWS == ROWS_DF ? ldexp((double)pre[z], ex) : ldexp(1.0, ex);
  float4 x[EPT];   // the current column below its diagonal
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    const int t = tid + q * NT;
    x[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t < n - 1) {
      const float4 a = source(t + 1, 0);
      x[q] = make_float4(a.x * sc, a.y * sc, a.z * sc, a.w * sc);
    }
  }
  const float4 a00 = source(0, 0);
  if (ROWS == ROWS_GLOBAL) {
    cluster.sync();   // the unscaled entries have been read
    if (rank == 0 && tid == 0) pre[z] = ldexpf(1.f, ex);
    for (long long q = tid; q < (long long)nloc * n; q += NT) {
      float4* a = row_of((int)(q / n)) + q % n;
      *a = make_float4(a->x * sc, a->y * sc, a->z * sc, a->w * sc);
    }
  } else {
    for (long long q = tid; q < (long long)nloc * n; q += NT) {
      const int li = (int)(q / n), c = (int)(q % n), i = rank + li * CS;
      float4 a;
      if (c <= i) {
        a = source(i, c);
      } else {
        a = source(c, i);
        a.z = -a.z;
        a.w = -a.w;
      }
      if (c == i) a.z = a.w = 0.f;
      dfs_smem[q] = make_float4(a.x * sc, a.y * sc, a.z * sc, a.w * sc);
    }
  }
  // warp sum of a double-float, the same bits on every lane
  auto warp_df = [&](float hi, float lo) {
    for (int o = 16; o > 0; o >>= 1) {
      const float bh = __shfl_xor_sync(0xffffffffu, hi, o), bl = __shfl_xor_sync(0xffffffffu, lo, o);
      df_add_sym(hi, lo, bh, bl);
    }
    return make_float2(hi, lo);
  };
  // b -= v conj(wk) + w conj(vk)
  auto rank2 = [](float4& b, float4 vt, float4 wt, float4 vk, float4 wk) {
    df_mac(b.x, b.y, -vt.x, -vt.y, wk.x, wk.y);
    df_mac(b.z, b.w, -vt.z, -vt.w, wk.x, wk.y);
    df_mac(b.x, b.y, -vt.z, -vt.w, wk.z, wk.w);
    df_mac(b.z, b.w, vt.x, vt.y, wk.z, wk.w);
    df_mac(b.x, b.y, -wt.x, -wt.y, vk.x, vk.y);
    df_mac(b.z, b.w, -wt.z, -wt.w, vk.x, vk.y);
    df_mac(b.x, b.y, -wt.z, -wt.w, vk.z, vk.w);
    df_mac(b.z, b.w, wt.x, wt.y, vk.z, vk.w);
    df_norm(b.x, b.y);
    df_norm(b.z, b.w);
  };
  // reflector r (column r below the diagonal: m entries x) -> vout, Vh row r, e[r]
  auto reflector = [&](int r, int m, float4* vout) {
    float nh = 0.f, nl = 0.f;
#pragma unroll
    for (int q = 0; q < EPT; ++q)
      if (tid + q * NT < m) {
        df_mac(nh, nl, x[q].x, x[q].y, x[q].x, x[q].y);
        df_mac(nh, nl, x[q].z, x[q].w, x[q].z, x[q].w);
      }
    if (tid == 0) x0_s = x[0];
    const float2 part = warp_df(nh, nl);
    if (lane == 0) redN[warp] = part;
    __syncthreads();
    float2 inv;
    if (warp == 0) {
      float2 ar = make_float2(0.f, 0.f), ai = ar;   // alpha; inv = 1 / ||x - alpha e_0||
      inv = ar;
      const float2 mine = lane < NW ? redN[lane] : make_float2(0.f, 0.f);
      float2 xn2 = warp_df(mine.x, mine.y);
      df_norm(xn2.x, xn2.y);
      const float4 x0 = x0_s;
      if (xn2.x >= 0x1p-100f) {
        // alpha = -e^{i arg x_0} ||x||, the phase from x_0 scaled away from float32's denormal squares
        const bool small = fmaxf(fabsf(x0.x), fabsf(x0.z)) < 0x1p-30f;
        const float up = small ? 0x1p60f : 1.f, dn = small ? 0x1p-60f : 1.f;
        const float2 a = make_float2(x0.x * up, x0.y * up), b = make_float2(x0.z * up, x0.w * up);
        const float2 q2 = df_add2(df_mul2(a, a), df_mul2(b, b));
        const float2 xn = df_mul2(xn2, df_rsqrt(xn2));
        float2 pr = make_float2(1.f, 0.f), pi = make_float2(0.f, 0.f), ax0 = pi;
        if (q2.x > 0x1p-100f) {
          const float2 qi = df_rsqrt(q2);
          pr = df_mul2(a, qi);
          pi = df_mul2(b, qi);
          ax0 = df_mul2(q2, qi);
          ax0 = make_float2(ax0.x * dn, ax0.y * dn);
        }
        ar = df_mul(-pr.x, -pr.y, xn.x, xn.y);
        ai = df_mul(-pi.x, -pi.y, xn.x, xn.y);
        const float2 u2 = df_add2(xn2, df_mul2(xn, ax0));
        inv = df_rsqrt(make_float2(2.f * u2.x, 2.f * u2.y));
      }
      if (lane == 0) {
        alpha_s = make_float4(ar.x, ar.y, ai.x, ai.y);
        inv_s = inv;
        if (rank == 0) e[r] = mk<double>(df_to_d(ar.x, ar.y) * back, df_to_d(ai.x, ai.y) * back);
      }
    }
    __syncthreads();
    inv = inv_s;
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      const int t = tid + q * NT;
      if (t < m) {
        float4 u = x[q];
        if (t == 0) {
          const float4 al = alpha_s;
          df_add(u.x, u.y, -al.x, -al.y);
          df_add(u.z, u.w, -al.z, -al.w);
        }
        const float2 vr = df_mul(u.x, u.y, inv.x, inv.y), vi = df_mul(u.z, u.w, inv.x, inv.y);
        vout[t] = make_float4(vr.x, vr.y, vi.x, vi.y);
        if (rank == 0) Vh[(long long)r * n0 + r + 1 + t] = mk<float>(vr.x, -vi.x);
      }
    }
  };
  reflector(0, n - 1, vb);
  if (rank == 0 && tid == 0) d[0] = df_to_d(a00.x, a00.y) * (ROWS == ROWS_DF ? (double)pre[z] : 1.0);
  int oc = 1 % CS, ol = 1 / CS;   // row j + 1: its CTA and place there
  cluster.sync();   // every CTA of the cluster runs before anyone writes into its shared memory
  const int jlast = ROWS == ROWS_GLOBAL ? jend - off : n - 2;   // columns 0 .. jlast - 1
  for (int j = 0; j < jlast; ++j) {
    const int m = n - j - 1, buf = j & 1;
    const float4* v = vb + buf * n;              // v_j: entry t is row j + 1 + t
    const float4* vo = vb + (buf ^ 1) * n + 1;   // v_{j-1} at row j + 1
    const float4* wo = wb + 1;                   // w_{j-1} at row j + 1
    float4* p = pb + buf * n;
    float2* kb = kbuf + buf * n;
    // own rows i > j, two per warp at a time: A <- A - v_{j-1} w^H - w v_{j-1}^H
    // on columns > j, p_i = row . v_j, and its term of K = v_j^H p
    const int l0 = ol + (oc > rank ? 1 : 0);   // first own row > j
    for (int li = l0 + warp; li < nloc; li += 2 * NW) {
      const bool two = li + NW < nloc;
      const int t = rank + li * CS - j - 1, t2 = t + NW * CS;
      float4* row = row_of(li) + (j + 1);
      float4* row2 = row_of(two ? li + NW : li) + (j + 1);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), acc2 = acc;
      if (j == 0) {
        for (int k = lane; k < m; k += 32) {
          const float4 vn = v[k];
          df_cmac<false>(acc, row[k], vn);
          if (two) df_cmac<false>(acc2, row2[k], vn);
        }
      } else if (two) {
        const float4 vt = vo[t], wt = wo[t], vt2 = vo[t2], wt2 = wo[t2];
        float4 b = row[min(lane, m - 1)], b2 = row2[min(lane, m - 1)];
        for (int k = lane; k < m; k += 32) {
          const int kn = min(k + 32, m - 1);
          float4 nb, nb2;
          if (ROWS == ROWS_GLOBAL) {   // the next entries' loads ahead of this one's arithmetic
            nb = row[kn];
            nb2 = row2[kn];
          }
          const float4 wk = wo[k], vk = vo[k], vn = v[k];
          rank2(b, vt, wt, vk, wk);
          rank2(b2, vt2, wt2, vk, wk);
          row[k] = b;
          row2[k] = b2;
          df_cmac<false>(acc, b, vn);
          df_cmac<false>(acc2, b2, vn);
          b = ROWS == ROWS_GLOBAL ? nb : row[kn];
          b2 = ROWS == ROWS_GLOBAL ? nb2 : row2[kn];
        }
      } else {
        const float4 vt = vo[t], wt = wo[t];
        for (int k = lane; k < m; k += 32) {
          float4 b = row[k];
          rank2(b, vt, wt, vo[k], wo[k]);
          row[k] = b;
          df_cmac<false>(acc, b, v[k]);
        }
      }
      // both rows' sums in five steps: lanes 0-15 end with the first row's, 16-31 with the second's, the
      // same bits on each (every CTA gets them) and whichever place a row has
      const bool up = lane & 16;
      {
        const float4 give = up ? acc : acc2;
        acc = up ? acc2 : acc;
        const float bh = __shfl_xor_sync(0xffffffffu, give.x, 16), bl = __shfl_xor_sync(0xffffffffu, give.y, 16);
        const float ch = __shfl_xor_sync(0xffffffffu, give.z, 16), cl = __shfl_xor_sync(0xffffffffu, give.w, 16);
        df_add_sym(acc.x, acc.y, bh, bl);
        df_add_sym(acc.z, acc.w, ch, cl);
      }
      for (int o = 8; o > 0; o >>= 1) {
        const float bh = __shfl_xor_sync(0xffffffffu, acc.x, o), bl = __shfl_xor_sync(0xffffffffu, acc.y, o);
        const float ch = __shfl_xor_sync(0xffffffffu, acc.z, o), cl = __shfl_xor_sync(0xffffffffu, acc.w, o);
        df_add_sym(acc.x, acc.y, bh, bl);
        df_add_sym(acc.z, acc.w, ch, cl);
      }
      if ((!up || two) && (lane & 15) < CS) {
        const int tr = up ? t2 : t;
        *cluster.map_shared_rank(p + tr, lane & 15) = acc;
        const float4 vt = v[tr];
        float kh = 0.f, kl = 0.f;
        df_mac(kh, kl, vt.x, vt.y, acc.x, acc.y);
        df_mac(kh, kl, vt.z, vt.w, acc.z, acc.w);
        *cluster.map_shared_rank(kb + tr, lane & 15) = make_float2(kh, kl);
      }
    }
    cluster.sync();
    // row j + 1 (its owner's last word on it), and K = v^H p by every warp
    float4 a[EPT];
    {
      const float4* rj1 =
          ROWS == ROWS_GLOBAL
              ? reinterpret_cast<const float4*>(Hsrc) + z * sH + (long long)(off + j + 1) * n0 + off + (j + 1)
              : cluster.map_shared_rank(dfs_smem + (long long)ol * n + (j + 1), oc);
#pragma unroll
      for (int q = 0; q < EPT; ++q) {
        const int t = tid + q * NT;
        a[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t + 1 < m) {
          a[q] = ROWS == ROWS_GLOBAL ? __ldcg(rj1 + t + 1) : rj1[t + 1];
          a[q].z = -a[q].z;   // entry (j + 2 + t, j + 1) by symmetry
          a[q].w = -a[q].w;
        }
      }
    }
    // (its terms in the order of the rows, not of their CTAs, whose number follows the batch)
    float2 K;
    if (ROWS == ROWS_GLOBAL) {
      // up to 1023 terms: summed by every warp they took some 1000 cycles of issue slots, more than a barrier
      K = tid < m ? kb[tid] : make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 1; q < EPT; ++q)
        if (tid + q * NT < m) df_add(K.x, K.y, kb[tid + q * NT].x, kb[tid + q * NT].y);
      K = warp_df(K.x, K.y);
      if (lane == 0) redK[warp] = K;
      __syncthreads();
      K = warp_df(lane < NW ? redK[lane].x : 0.f, lane < NW ? redK[lane].y : 0.f);
      if (tid == 0) K_s = K;   // for the last column's update
    } else {
      float2 part[4];   // four chains: the sum stands between the barrier and the next reflector
#pragma unroll
      for (int u = 0; u < 4; ++u) part[u] = lane + 32 * u < m ? kb[lane + 32 * u] : make_float2(0.f, 0.f);
      for (int q = lane + 128; q < m; q += 128) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (q + 32 * u < m) df_add(part[u].x, part[u].y, kb[q + 32 * u].x, kb[q + 32 * u].y);
      }
      df_add(part[0].x, part[0].y, part[1].x, part[1].y);
      df_add(part[2].x, part[2].y, part[3].x, part[3].y);
      df_add(part[0].x, part[0].y, part[2].x, part[2].y);
      K = warp_df(part[0].x, part[0].y);
    }
    const float k2h = -2.f * K.x, k2l = -2.f * K.y;
    auto wof = [&](float4 vt, float4 pt) {   // w = 2 p - 2 K v
      float4 w = make_float4(2.f * pt.x, 2.f * pt.y, 2.f * pt.z, 2.f * pt.w);
      df_mac(w.x, w.y, k2h, k2l, vt.x, vt.y);
      df_mac(w.z, w.w, k2h, k2l, vt.z, vt.w);
      df_norm(w.x, w.y);
      df_norm(w.z, w.w);
      return w;
    };
    const float4 v0 = v[0], w0 = wof(v0, p[0]);
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      const int t = tid + q * NT;
      if (t + 1 < m) {
        const float4 vt = v[t + 1], wt = wof(vt, p[t + 1]);
        wb[t + 1] = wt;
        rank2(a[q], vt, wt, v0, w0);
      }
      x[q] = a[q];
    }
    if (rank == oc && tid == 0) {
      // d[j + 1] = A[j+1][j+1] - 2 Re(v_0 conj(w_0))
      const float4 g = row_of(ol)[j + 1];
      float gh = g.x, gl = g.y;
      df_mac(gh, gl, -2.f * v0.x, -2.f * v0.y, w0.x, w0.y);
      df_mac(gh, gl, -2.f * v0.z, -2.f * v0.w, w0.z, w0.w);
      d[j + 1] = df_to_d(gh, gl) * back;
    }
    if (++oc == CS) {   // to row j + 2
      oc = 0;
      ++ol;
    }
    if (ROWS == ROWS_GLOBAL ? j + 1 < jlast : j + 3 < n) {
      reflector(j + 1, m - 1, vb + (buf ^ 1) * n);
    } else if (ROWS != ROWS_GLOBAL && tid == 0) {
      // the last 2 x 2 block: subdiagonal, and the corner by its owner
      if (rank == 0) e[n - 2] = mk<double>(df_to_d(x[0].x, x[0].y) * back, df_to_d(x[0].z, x[0].w) * back);
      if (rank == (n - 1) % CS) {
        const float4 g = dfs_smem[(long long)((n - 1) / CS) * n + (n - 1)], v1 = v[1], w1 = wb[1];
        float gh = g.x, gl = g.y;
        df_mac(gh, gl, -2.f * v1.x, -2.f * v1.y, w1.x, w1.y);
        df_mac(gh, gl, -2.f * v1.z, -2.f * v1.w, w1.z, w1.w);
        d[n - 1] = df_to_d(gh, gl) * back;
      }
    }
    __syncthreads();
  }
  if (ROWS == ROWS_GLOBAL) {
    // the last column's rank-2 update of the trailing block (rows and columns jlast and on; v_{jlast-1}
    // and w at row jlast are entries 0, which wb does not hold: w_0 is not needed beyond row jlast)
    const int j = jlast - 1, m = n - j - 1;
    const float4* v = vb + (j & 1) * n;
    const float k2h = -2.f * K_s.x, k2l = -2.f * K_s.y;
    if (tid == 0) {
      const float4 pt = pb[(j & 1) * n], vt = v[0];
      float4 w = make_float4(2.f * pt.x, 2.f * pt.y, 2.f * pt.z, 2.f * pt.w);
      df_mac(w.x, w.y, k2h, k2l, vt.x, vt.y);
      df_mac(w.z, w.w, k2h, k2l, vt.z, vt.w);
      df_norm(w.x, w.y);
      df_norm(w.z, w.w);
      wb[0] = w;
    }
    __syncthreads();
    for (int li = warp; li < nloc; li += NW) {
      const int t = rank + li * CS - j - 1;
      if (t < 0) continue;
      float4* row = row_of(li) + (j + 1);
      const float4 vt = v[t], wt = wb[t];
      for (int k = lane; k < m; k += 32) {
        float4 b = row[k];
        rank2(b, vt, wt, v[k], wb[k]);
        row[k] = b;
      }
    }
  }
  cluster.sync();   // rows of this CTA may still be read by others
}

// ---------------------------------------------------------------- launchers
namespace {

// double-float reduction launch: 256 threads, TRIDIAG_DF_UNROLL loads in flight per lane in the
// product A v and the rank-2 update (its loads wait on L2: ncu shows long-scoreboard stalls and
// 1.6 % L2 throughput with one load per lane)
constexpr int TRIDIAG_DF_THREADS = 256;
constexpr int TRIDIAG_DF_UNROLL = 4;

template <typename... KArgs, typename... Args>
cudaError_t launch_df(void (*kernel)(KArgs...), int cs, int batch, int threads, size_t smem, cudaStream_t st, Args... args) {
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

constexpr size_t DFS_SMEM = 226 * 1024;   // dynamic shared memory per CTA (227 KB less the static part)

// CTAs per matrix: more of them shorten a column's pass over the matrix.  Sixteen is
// the most a cluster holds, but only seven such clusters run at once on the GPU's GPCs
// (one CTA per SM), of twelve eight: sixteen where the launch's batch takes no more waves of
// them (launches on other streams are not counted).  The result does not depend on the
// number.  380 rows of 12 CTAs fill their shared memory.  Measured, us, five or six
// matrices on 16 CTAs and eight on 12: 180 rows 625 and 629, 256 rows 1102 and 1203, 380 rows
// 2349 and 2554, 512 rows 4224 and 5286; 640 rows, two and eight, 7561 and 9116.  The kernels
// before: 256 rows, five matrices, 4.17 ms (float64); 512 rows, eight, 9.9 and 640 rows 17.0
// (lower triangle in L2, two barriers a column).
constexpr int DFS_CS = 12, DFS_CS_FEW = 16, DFS_MAX = 380, DFS_GLOBAL_MAX = 1024;

// Clusters of `cs` CTAs that run at once, a CTA to an SM; cached per kernel, size and device.
int dfs_active(const void* kernel, int cs, int threads) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, int, int>, int> cache;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  auto key = std::make_tuple(kernel, cs, dev);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  int active = 0;
  if (ensure_kernel_smem(kernel, DFS_SMEM, cs > 8) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = DFS_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&active, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      active = 0;
    }
  }
  cache[key] = active;
  return active;
}

template <int NT, int EPT, int ROWS>
cudaError_t dfs_launch(cudaStream_t st, void* H, long long sH, int n0, int off, int jend, double* d, cx<double>* e,
                       int ldde, cx<float>* Vh, long long sVh, float* pre, int batch) {
  auto kernel = tridiag_dfs_kernel<NT, EPT, ROWS>;
  const int few = dfs_active((const void*)kernel, DFS_CS_FEW, NT), many = dfs_active((const void*)kernel, DFS_CS, NT);
  const int cs = few > 0 && (many < 1 || (batch + few - 1) / few <= (batch + many - 1) / many) ? DFS_CS_FEW : DFS_CS;
  const int n = n0 - off, maxloc = (n + cs - 1) / cs;
  const size_t smem = DfsLayout{n, maxloc, ROWS == ROWS_GLOBAL}.bytes();
  if (n < 3 || n > NT * EPT || smem > DFS_SMEM) return cudaErrorInvalidValue;
  return launch_df(kernel, cs, batch, NT, smem, st, H, sH, n0, off, jend, d, e, ldde, Vh, sVh, pre, maxloc);
}

}  // namespace

// d, e (T[k+1][k] = e[k]) and the float32 reflectors (row j of Vh, conjugated,
// columns j + 1 on; the rest of Vh untouched) of the Hermitian H[z] (n x n,
// lower triangle read).  Up to DFS_MAX rows the whole reduction runs in shared
// memory; above, on rows in L2 until the trailing block fits (beyond
// DFS_GLOBAL_MAX rows with the two-barrier kernel first, whose vectors are not
// tied to a thread each).  work: batch x n x n float4 (n > DFS_MAX only), P:
// batch x n float4, Kp: batch x 32 float2.
cudaError_t tridiag_df(cudaStream_t st, const cx<float>* H, long long sH, int n, float4* work, float4* P, float2* Kp,
                       double* d, cx<double>* e, cx<float>* Vh, int batch) {
  const long long nn = (long long)n * n;
  cudaError_t ce;
  if (n <= DFS_MAX) {
    ProfScope ps(st, K_TRIDIAG, 1, 16.0 / 3.0 * (double)n * n * n * batch);
    void* h = const_cast<cx<float>*>(H);
    if (n <= 256) return dfs_launch<256, 1, ROWS_C64>(st, h, sH, n, 0, 0, d, e, n, Vh, nn, nullptr, batch);
    return dfs_launch<512, 1, ROWS_C64>(st, h, sH, n, 0, 0, d, e, n, Vh, nn, nullptr, batch);
  }
  {
    ProfScope ps(st, K_ELEMWISE);
    const dim3 grid((unsigned)std::min<long long>((nn + 255) / 256, 1024), batch);
    cx_f2df_kernel<<<grid, 256, 0, st>>>(H, sH, n, work, nn);
    if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  }
  ProfScope ps(st, K_TRIDIAG, n > DFS_GLOBAL_MAX ? 4 : 2, 16.0 / 3.0 * (double)n * n * n * batch);
  int off = 0;
  if (n > DFS_GLOBAL_MAX) {
    const int cs = tridiag64_cluster_size((const void*)tridiag_df_kernel<TRIDIAG_DF_UNROLL>);
    const size_t smem = std::max<size_t>(32 * (size_t)n, TRIDIAG64_SMEM);
    off = n - DFS_GLOBAL_MAX;
    if ((ce = launch_df(tridiag_df_kernel<TRIDIAG_DF_UNROLL>, cs, batch, TRIDIAG_DF_THREADS, smem, st, work, nn, n, d,
                        e, n, P, Kp, Vh, nn, off)) != cudaSuccess)
      return ce;
    df_mirror_kernel<<<dim3(1024, batch), 256, 0, st>>>(work, nn, n, off);
    if ((ce = cudaGetLastError()) != cudaSuccess) return ce;
  }
  float* pre = reinterpret_cast<float*>(Kp);
  if ((ce = dfs_launch<512, 2, ROWS_GLOBAL>(st, work, nn, n, off, n - DFS_MAX, d, e, n, Vh, nn, pre, batch)) !=
      cudaSuccess)
    return ce;
  return dfs_launch<512, 1, ROWS_DF>(st, work, nn, n, n - DFS_MAX, 0, d, e, n, Vh, nn, pre, batch);
}

}  // namespace nne
