// Blocked Householder QR for tall complex matrices (m x n, row-major).
//
// Panels of 32 columns are factored by one thread-block cluster per matrix:
// the panel rows are spread over the cluster's CTAs (cyclically) and kept in
// registers (shared memory where they do not fit); per column the cluster exchanges
// one round of partial sums through distributed shared memory.  Each panel also yields the compact-WY
// factor T (P_0 ... P_{b-1} = I - V T V^H).  Trailing updates and the explicit Q then apply each panel's
// block reflector (wy_apply).  All reductions are in a fixed order (deterministic).
#include <type_traits>

#include "kernels.cuh"
#include "recip.cuh"

namespace cg = cooperative_groups;

namespace nne {

constexpr int QB = 32;   // panel width
constexpr int PS = QB + 1;   // padded row stride of the shared-memory panel (avoids bank conflicts)

constexpr int QR_THREADS = 512;
constexpr int QR_WARPS = QR_THREADS / 32;
constexpr int QR_CS_MAX = 16;

// a - v * w, evaluated the same way wherever it is used (the owner of a row
// and every CTA predicting that row's next pivot must agree bit for bit)
template <typename R>
__device__ __forceinline__ cx<R> hh_upd(cx<R> a, cx<R> v, cx<R> w) {
  return mk<R>(fma(-v.re, w.re, fma(v.im, w.im, a.re)), fma(-v.re, w.im, fma(-v.im, w.re, a.im)));
}

// One round's contribution of a CTA to the cluster-wide sums.
template <typename R>
struct QrMsg {
  cx<R> w[QB];   // c < j: v_c^H v_j ; c > j: v_j^H a_c (partials over own rows)
  cx<R> ex[3];   // a_j[j+1] (owner of row j), v_{j+1} and a_{j+1}[j+1] (owner of row j+1); 0 elsewhere
  double nrm;    // partial squared norm of the next pivot column
};

// Factor the panel A[pb:m, pb:pb+bw] (bw <= 32) of matrix z = blockIdx.y.
// Column j takes one cluster barrier: every CTA pushes its partial sums into
// every CTA's shared memory, then all sum them in rank order.  The squared
// norm of column j+1 below row j is downdated from the same round (the
// reflector is unitary on rows >= j: ||a'_{j+1}||^2 over rows > j equals the
// pre-update norm over rows >= j minus |a'_j[j+1]|^2); when that cancels
// more than half of it, an extra round recomputes it.  The compact-WY factor
// T is built column by column from the v_c^H v_j of the same rounds.
template <typename R>
__global__ void __launch_bounds__(QR_THREADS) qr_panel_kernel(cx<R>* Ab, long long sA, int lda, int m, int pb, int bw,
                                                               cx<R>* Vb, long long sV, int ldv, cx<R>* Tb,
                                                               long long sT, int maxloc, int zr) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int z = blockIdx.y;
  cx<R>* A = Ab + z * sA;
  cx<R>* V = Vb + z * sV;
  cx<R>* T = Tb + z * sT;
  extern __shared__ unsigned char smem_raw[];
  cx<R>* P = reinterpret_cast<cx<R>*>(smem_raw);       // [maxloc][PS]
  __shared__ QrMsg<R> msg[2][QR_CS_MAX];
  __shared__ cx<R> red[QR_WARPS][QB];
  __shared__ double redn[QR_WARPS];
  __shared__ cx<R> wfull[QB];
  __shared__ cx<R> gcol[QB];
  __shared__ cx<R> alphas[QB];
  __shared__ cx<R> Ts[QB][QB + 1];
  __shared__ cx<R> ex_s[3];
  __shared__ double nrm_s;
  __shared__ cx<R> x0_s;
  __shared__ double xn2_s;
  __shared__ int recompute_s;
  __shared__ cx<R> alpha_s;
  __shared__ R inv_s, tau_s;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int mp = m - pb;                                   // panel rows
  const int nloc = mp > rank ? (mp - rank + CS - 1) / CS : 0;
  for (int e = tid; e < nloc * QB; e += QR_THREADS) {
    const int li = e / QB, c = e % QB;
    const long long gi = pb + rank + (long long)li * CS;
    P[li * PS + c] = c < bw ? A[gi * lda + pb + c] : mk<R>(0, 0);
  }
  for (int e = tid; e < QB * QB; e += QR_THREADS) Ts[e / QB][e % QB] = mk<R>(0, 0);
  // every CTA of the cluster is running before anyone writes into its shared memory
  cluster.sync();
  int round = 0;
  // first local row whose panel row index is >= p
  auto first_local = [&](int p) { return p > rank ? (p - rank + CS - 1) / CS : 0; };
  // reflector of the next column from x0_s, xn2_s (one thread; FP64 is slow on this part)
  auto pivot = [&]() {
    const double xn2 = xn2_s;
    const cx<R> x0 = x0_s;
    double pr, pi, ax0;
    unit_phase_of(x0, &pr, &pi, &ax0);
    const double xn = sqrt(xn2);
    cx<R> alpha = mk<R>(0, 0);
    double un = 0;
    if (xn > 0) {
      alpha = mk<R>((R)(-xn * pr), (R)(-xn * pi));
      un = sqrt(2.0 * xn2 + 2.0 * xn * ax0);
    }
    alpha_s = alpha;
    inv_s = un > 0 ? (R)(1.0 / un) : R(0);
    tau_s = un > 0 ? R(2) : R(0);
  };
  // cluster-wide squared norm of column c over panel rows >= p (one round)
  auto norm_round = [&](int c, int p, bool with_x0) {
    const int l0 = first_local(p);
    R sacc = 0;
    for (int li = l0 + tid; li < nloc; li += QR_THREADS) sacc += norm2(P[li * PS + c]);
    sacc = warp_sum_r(sacc);
    if (lane == 0) redn[wid] = (double)sacc;
    __syncthreads();
    const int buf = round & 1;
    if (tid < CS) {
      double t = 0;
      for (int w = 0; w < QR_WARPS; ++w) t += redn[w];
      QrMsg<R>* dst = cluster.map_shared_rank(&msg[buf][rank], tid);
      dst->nrm = t;
      cx<R> x0 = mk<R>(0, 0);
      if (with_x0 && c < mp && rank == c % CS) x0 = P[(c / CS) * PS + c];
      dst->ex[2] = x0;
    }
    cluster.sync();
    if (tid == 0) {
      double t = 0;
      cx<R> x0 = mk<R>(0, 0);
      for (int src = 0; src < CS; ++src) {
        t += msg[buf][src].nrm;
        x0 = x0 + msg[buf][src].ex[2];
      }
      xn2_s = t;
      if (with_x0) x0_s = x0;
      pivot();
    }
    ++round;
    __syncthreads();
  };
  norm_round(0, 0, true);
  for (int j = 0; j < bw; ++j) {
    const int lstart = first_local(j);
    const cx<R> x0 = x0_s;
    const cx<R> alpha = alpha_s;
    const R inv = inv_s, tau = tau_s;
    if (tid == 0) alphas[j] = alpha;
    const int owner = j % CS, ljo = j / CS;
    // v = (x - alpha e_j) / un on own rows
    for (int li = lstart + tid; li < nloc; li += QR_THREADS) {
      cx<R> u = P[li * PS + j];
      if (rank == owner && li == ljo) u = u - alpha;
      P[li * PS + j] = inv * u;
    }
    __syncthreads();
    const bool has_next = j + 1 < bw;
    // partials: lane c holds v_c^H v_j (c < j) or v_j^H a_c (c > j); lane j+1 also |a_{j+1}|^2
    {
      const int c = lane;
      cx<R> acc = mk<R>(0, 0);
      R nacc = 0;
      if (c < j) {
        for (int li = lstart + wid; li < nloc; li += QR_WARPS) fmac_(acc, P[li * PS + c], P[li * PS + j]);
      } else if (c > j && c < bw) {
        for (int li = lstart + wid; li < nloc; li += QR_WARPS) {
          const cx<R> a = P[li * PS + c];
          fmac_(acc, P[li * PS + j], a);
          if (c == j + 1) nacc += norm2(a);
        }
      }
      red[wid][c] = acc;
      if (c == j + 1) redn[wid] = (double)nacc;
    }
    __syncthreads();
    const int buf = round & 1;
    if (tid < QB) {
      cx<R> t = mk<R>(0, 0);
      for (int w = 0; w < QR_WARPS; ++w) t = t + red[w][tid];
      for (int d = 0; d < CS; ++d) cluster.map_shared_rank(&msg[buf][rank], d)->w[tid] = t;
    } else if (tid == QB) {
      double nt = 0;
      if (has_next)
        for (int w = 0; w < QR_WARPS; ++w) nt += redn[w];
      cx<R> e0 = mk<R>(0, 0), e1 = mk<R>(0, 0), e2 = mk<R>(0, 0);
      if (has_next) {
        if (rank == owner) e0 = P[ljo * PS + j + 1];
        if (j + 1 < mp && rank == (j + 1) % CS) {
          const int l1 = (j + 1) / CS;
          e1 = P[l1 * PS + j];
          e2 = P[l1 * PS + j + 1];
        }
      }
      for (int d = 0; d < CS; ++d) {
        QrMsg<R>* dst = cluster.map_shared_rank(&msg[buf][rank], d);
        dst->ex[0] = e0;
        dst->ex[1] = e1;
        dst->ex[2] = e2;
        dst->nrm = nt;
      }
    }
    cluster.sync();
    ++round;
    if (tid < QB) {
      cx<R> t = mk<R>(0, 0);
      for (int src = 0; src < CS; ++src) t = t + msg[buf][src].w[tid];
      if (tid > j) wfull[tid] = mk<R>(2 * t.re, 2 * t.im);
      else wfull[tid] = mk<R>(0, 0);
      gcol[tid] = tid < j ? t : mk<R>(0, 0);
    } else if (tid == QB) {
      double nt = 0;
      cx<R> e0 = mk<R>(0, 0), e1 = mk<R>(0, 0), e2 = mk<R>(0, 0);
      for (int src = 0; src < CS; ++src) {
        nt += msg[buf][src].nrm;
        e0 = e0 + msg[buf][src].ex[0];
        e1 = e1 + msg[buf][src].ex[1];
        e2 = e2 + msg[buf][src].ex[2];
      }
      nrm_s = nt;
      ex_s[0] = e0;
      ex_s[1] = e1;
      ex_s[2] = e2;
    }
    __syncthreads();
    // T[0:j, j] = -tau_j T[0:j, 0:j] (V^H v_j), T[j][j] = tau_j (rank 0, last warp)
    if (rank == 0 && wid == QR_WARPS - 1) {
      cx<R> acc = mk<R>(0, 0);
      if (lane < j)
        for (int l = lane; l < j; ++l) fma_(acc, Ts[lane][l], gcol[l]);
      if (lane < j) Ts[lane][j] = mk<R>(-tau * acc.re, -tau * acc.im);
      if (lane == j) Ts[j][j] = mk<R>(tau, 0);
    }
    // a_c <- a_c - v (2 v^H a_c), c in (j, bw), own rows >= j
    if (has_next)
      for (int e = tid; e < (nloc - lstart) * QB; e += QR_THREADS) {
        const int li = lstart + e / QB, c = e % QB;
        if (c > j && c < bw) P[li * PS + c] = hh_upd(P[li * PS + c], P[li * PS + j], wfull[c]);
      }
    if (tid == 0 && has_next) {
      const cx<R> vj = inv * (x0 - alpha);                      // the owner's v_j, same operations
      const cx<R> ajn = hh_upd(ex_s[0], vj, wfull[j + 1]);      // a'_j[j+1]
      const cx<R> x0n = j + 1 < mp ? hh_upd(ex_s[2], ex_s[1], wfull[j + 1]) : mk<R>(0, 0);
      const double nA = nrm_s;
      const double xn2n = nA - (double)norm2(ajn);
      x0_s = x0n;
      xn2_s = xn2n > 0 ? xn2n : 0.0;
      recompute_s = !(xn2n > 0.5 * nA);
      if (!recompute_s) pivot();
    }
    __syncthreads();
    if (has_next && recompute_s) norm_round(j + 1, j + 1, false);
  }
  // write back V and the R part of A
  for (int e = tid; e < nloc * QB; e += QR_THREADS) {
    const int li = e / QB, c = e % QB;
    if (c >= bw) continue;
    const int pi = rank + li * CS;
    const long long gi = pb + pi;
    const cx<R> val = P[li * PS + c];
    V[gi * ldv + pb + c] = pi >= c ? val : mk<R>(0, 0);
    A[gi * lda + pb + c] = pi < c ? val : (pi == c ? alphas[c] : mk<R>(0, 0));
  }
  if (rank == 0) {
    for (int e = tid; e < QB * QB; e += QR_THREADS) T[e] = Ts[e / QB][e % QB];
    // rows of the outer block above this panel: zero in its reflector columns
    for (int e = tid; e < zr * QB; e += QR_THREADS)
      if (e % QB < bw) V[(long long)(pb - zr + e / QB) * ldv + pb + e % QB] = mk<R>(0, 0);
  }
}

// Shared-memory state of one register-resident panel factorisation.  Norm
// sums are kept in the state's precision R: the downdate below cancels at
// most half of a norm before an exact recompute, which bounds its relative
// error at a few units of R.
template <typename R>
struct PanelMsg {
  cx<R> w[QB];   // c < j: v_c^H v_j ; c > j: v_j^H a_c (partials over own rows)
  cx<R> ex[3];   // a_j[j+1] (owner of row j), v_{j+1} and a_{j+1}[j+1] (owner of row j+1); 0 elsewhere
  R nrm;         // partial squared norm of the next pivot column
};
template <typename R>
struct PanelShared {
  PanelMsg<R> msg[2][QR_CS_MAX];
  cx<R> red[QR_WARPS][QB];
  R redn[QR_WARPS];
  cx<R> wfull[QB];
  cx<R> gcol[QB];
  cx<R> alphas[QB];
  cx<R> Ts[QB][QB + 1];
  cx<R> ex_loc[3];
  cx<R> ex_s[3];
  R nrm_s;
  cx<R> x0_s;
  R xn2_s;
  int recompute_s;
  cx<R> alpha_s;
  R inv_s, tau_s;
};

// Reflector pivot from the squared norm xn2 of the column at and below the
// diagonal and its diagonal entry x0: alpha = -e^{i arg x0} ||x||,
// un = ||x - alpha e_0||, tau = 2 (0 for a zero column).  Evaluated in R,
// the phase of x0 by unit_phase_of.
template <typename R>
__device__ __forceinline__ void hh_pivot(R xn2, cx<R> x0, cx<R>* alpha, R* inv, R* tau) {
  R pr, pi, ax0;
  unit_phase_of(x0, &pr, &pi, &ax0);
  const R xn = sqrt(xn2);
  cx<R> a = mk<R>(0, 0);
  R un = 0;
  if (xn > R(0)) {
    a = mk<R>(-xn * pr, -xn * pi);
    un = sqrt(R(2) * xn2 + R(2) * xn * ax0);
  }
  *alpha = a;
  *inv = un > R(0) ? R(1) / un : R(0);
  *tau = un > R(0) ? R(2) : R(0);
}

// One cluster round: the squared norm of a column over the panel rows from
// a given row down (sacc: this thread's partial, meaningful on lane c), and
// with with_x0 the column's diagonal entry (x0_mine, held by the thread
// holds_x0); tid 0 then forms the reflector pivot.
template <typename R>
__device__ __forceinline__ void panel_norm_round(R sacc, cx<R> x0_mine, bool holds_x0, PanelShared<R>& sh,
                                                 cg::cluster_group& cluster, int CS, int rank, int c, bool with_x0,
                                                 bool x0_here, int& round) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (lane == c) sh.redn[wid] = sacc;
  if (with_x0 && holds_x0) sh.ex_loc[2] = x0_mine;
  __syncthreads();
  const int buf = round & 1;
  if (tid < CS) {
    R t0 = 0, t1 = 0;
    for (int w = 0; w < QR_WARPS; w += 2) {
      t0 += sh.redn[w];
      t1 += sh.redn[w + 1];
    }
    PanelMsg<R>* dst = cluster.map_shared_rank(&sh.msg[buf][rank], tid);
    dst->nrm = t0 + t1;
    dst->ex[2] = (with_x0 && x0_here) ? sh.ex_loc[2] : mk<R>(0, 0);
  }
  cluster.sync();
  if (tid == 0) {
    R t = 0;
    cx<R> x0 = mk<R>(0, 0);
    for (int src = 0; src < CS; ++src) {
      t += sh.msg[buf][src].nrm;
      x0 = x0 + sh.msg[buf][src].ex[2];
    }
    sh.xn2_s = t;
    if (with_x0) sh.x0_s = x0;
    cx<R> al;
    R iv, ta;
    hh_pivot<R>(sh.xn2_s, sh.x0_s, &al, &iv, &ta);
    sh.alpha_s = al;
    sh.inv_s = iv;
    sh.tau_s = ta;
  }
  ++round;
  __syncthreads();
}

// Register-resident panel factorisation (same arithmetic per column as a
// plain Householder QR): warp w of a CTA holds its local rows w, w + 16, ...
// (at most RPW of them), lane c holds column c, so the reflector entry of a
// row is a shuffle from lane j and no shared-memory traffic touches the
// panel.  Rows are dealt to the CTAs of the cluster cyclically.  Column j
// takes one cluster round: every CTA pushes its partial sums into every
// CTA's shared memory, then all sum them in rank order.  The squared norm of
// column j+1 below row j is downdated in the same round (the reflector is
// unitary on rows >= j); when that cancels more than half of it an extra
// round recomputes it.  T is built column by column from the v_c^H v_j of
// the same rounds.
template <typename R, int RPW>
__global__ void __launch_bounds__(QR_THREADS) qr_panel_reg_kernel(cx<R>* Ab, long long sA, int lda, int m, int pb,
                                                                   int bw, cx<R>* Vb, long long sV, int ldv,
                                                                   cx<R>* Tb, long long sT, int zr) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int z = blockIdx.y;
  cx<R>* A = Ab + z * sA;
  cx<R>* V = Vb + z * sV;
  cx<R>* T = Tb + z * sT;
  __shared__ PanelShared<R> sh;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int mp = m - pb;
  const int nloc = mp > rank ? (mp - rank + CS - 1) / CS : 0;
  // this warp's live registers: k < kmax (local row wid + 16 k < nloc)
  const int kmax = nloc > wid ? (nloc - wid + QR_WARPS - 1) / QR_WARPS : 0;
  cx<R> a[RPW];
#pragma unroll
  for (int k = 0; k < RPW; ++k) {
    const int li = wid + QR_WARPS * k;
    a[k] = mk<R>(0, 0);
    if (li < nloc && lane < bw) a[k] = A[(long long)(pb + rank + li * CS) * lda + pb + lane];
  }
  for (int e = tid; e < QB * QB; e += QR_THREADS) sh.Ts[e / QB][e % QB] = mk<R>(0, 0);
  // every CTA of the cluster is running before anyone writes into its shared memory
  cluster.sync();
  int round = 0;
  {
    // column 0 over all rows, and its entry in row 0 (rank 0, warp 0, register 0, lane 0)
    R sacc = 0;
#pragma unroll
    for (int k = 0; k < RPW; ++k)
      if (k < kmax) sacc += norm2(a[k]);
    panel_norm_round<R>(sacc, a[0], rank == 0 && wid == 0 && lane == 0, sh, cluster, CS, rank, 0, true, rank == 0,
                        round);
  }
  for (int j = 0; j < bw; ++j) {
    const cx<R> x0 = sh.x0_s;
    const cx<R> alpha = sh.alpha_s;
    const R inv = sh.inv_s, tau = sh.tau_s;
    if (tid == 0) sh.alphas[j] = alpha;
    const int owner = j % CS;
    const bool has_next = j + 1 < bw;
    // registers k >= kmin of this warp hold rows >= j: local row li >= first local row >= j
    const int l0 = j > rank ? (j - rank + CS - 1) / CS : 0;
    const int kmin = l0 > wid ? (l0 - wid + QR_WARPS - 1) / QR_WARPS : 0;
    // row of register k: rank + (wid + 16 k) CS; rows j and j+1, if here, sit at these registers
    const int dj = j - rank - wid * CS, dj1 = j + 1 - rank - wid * CS;
    const int kj = (dj >= 0 && dj % (QR_WARPS * CS) == 0) ? dj / (QR_WARPS * CS) : -1;
    const int kj1 = (dj1 >= 0 && dj1 % (QR_WARPS * CS) == 0 && j + 1 < mp) ? dj1 / (QR_WARPS * CS) : -1;
    // v = (x - alpha e_j) / un (every lane forms it from lane j's entry; lane j keeps it);
    // partials: lane c < j: v_c^H v_j; lane c > j: v_j^H a_c; lane j+1 also |a_{j+1}|^2;
    // and the pre-update entries every CTA needs for the next pivot
    // branch-free: every lane accumulates conj(x) v; lanes c > j want v^H a_c = conj of that
    cx<R> acc0 = mk<R>(0, 0), acc1 = mk<R>(0, 0);
    R nacc = 0;
    cx<R> e_a = mk<R>(0, 0), e_b = mk<R>(0, 0);
#pragma unroll
    for (int k = 0; k < RPW; ++k) {
      if (k >= kmin && k < kmax) {
        cx<R> u = shfl_idx(a[k], j);
        if (k == kj) u = u - alpha;
        const cx<R> v = inv * u;
        if (lane == j) a[k] = v;
        const cx<R> x = a[k];
        if (k & 1) fmac_(acc1, x, v); else fmac_(acc0, x, v);
        nacc += norm2(x);
        if (k == kj) e_a = x;                       // row j: lane j+1 holds a_j[j+1]
        if (k == kj1) e_b = lane == j ? v : x;      // row j+1: lane j -> v_{j+1}, lane j+1 -> a_{j+1}[j+1]
      }
    }
    {
      const cx<R> acc = acc0 + acc1;
      sh.red[wid][lane] = lane > j ? conj(acc) : acc;
    }
    if (lane == j + 1) sh.redn[wid] = nacc;
    if (has_next) {
      if (kj >= 0 && lane == j + 1) sh.ex_loc[0] = e_a;
      if (kj1 >= 0 && lane == j) sh.ex_loc[1] = e_b;
      if (kj1 >= 0 && lane == j + 1) sh.ex_loc[2] = e_b;
    }
    __syncthreads();
    const int buf = round & 1;
    if (tid < QB) {
      cx<R> t0 = mk<R>(0, 0), t1 = t0, t2 = t0, t3 = t0;
      for (int w = 0; w < QR_WARPS; w += 4) {
        t0 = t0 + sh.red[w][tid];
        t1 = t1 + sh.red[w + 1][tid];
        t2 = t2 + sh.red[w + 2][tid];
        t3 = t3 + sh.red[w + 3][tid];
      }
      const cx<R> t = (t0 + t1) + (t2 + t3);
      for (int d = 0; d < CS; ++d) cluster.map_shared_rank(&sh.msg[buf][rank], d)->w[tid] = t;
    } else if (tid == QB) {
      R nt = 0;
      cx<R> e0 = mk<R>(0, 0), e1 = mk<R>(0, 0), e2 = mk<R>(0, 0);
      if (has_next) {
        R n0 = 0, n1 = 0;
        for (int w = 0; w < QR_WARPS; w += 2) {
          n0 += sh.redn[w];
          n1 += sh.redn[w + 1];
        }
        nt = n0 + n1;
        if (rank == owner) e0 = sh.ex_loc[0];
        if (j + 1 < mp && rank == (j + 1) % CS) {
          e1 = sh.ex_loc[1];
          e2 = sh.ex_loc[2];
        }
      }
      for (int d = 0; d < CS; ++d) {
        PanelMsg<R>* dst = cluster.map_shared_rank(&sh.msg[buf][rank], d);
        dst->ex[0] = e0;
        dst->ex[1] = e1;
        dst->ex[2] = e2;
        dst->nrm = nt;
      }
    }
    cluster.sync();
    ++round;
    if (tid < QB) {
      cx<R> t0 = mk<R>(0, 0), t1 = t0;
      int src = 0;
      for (; src + 1 < CS; src += 2) {
        t0 = t0 + sh.msg[buf][src].w[tid];
        t1 = t1 + sh.msg[buf][src + 1].w[tid];
      }
      if (src < CS) t0 = t0 + sh.msg[buf][src].w[tid];
      const cx<R> t = t0 + t1;
      sh.wfull[tid] = tid > j ? mk<R>(2 * t.re, 2 * t.im) : mk<R>(0, 0);
      sh.gcol[tid] = tid < j ? t : mk<R>(0, 0);
    } else if (tid == QB) {
      R nt = 0;
      cx<R> e0 = mk<R>(0, 0), e1 = mk<R>(0, 0), e2 = mk<R>(0, 0);
      for (int src = 0; src < CS; ++src) {
        nt += sh.msg[buf][src].nrm;
        e0 = e0 + sh.msg[buf][src].ex[0];
        e1 = e1 + sh.msg[buf][src].ex[1];
        e2 = e2 + sh.msg[buf][src].ex[2];
      }
      sh.nrm_s = nt;
      sh.ex_s[0] = e0;
      sh.ex_s[1] = e1;
      sh.ex_s[2] = e2;
    }
    __syncthreads();
    // T[0:j, j] = -tau_j T[0:j, 0:j] (V^H v_j), T[j][j] = tau_j (rank 0, last warp)
    if (rank == 0 && wid == QR_WARPS - 1) {
      cx<R> ta0 = mk<R>(0, 0), ta1 = ta0;
      if (lane < j) {
        int l = lane;
        for (; l + 1 < j; l += 2) {
          fma_(ta0, sh.Ts[lane][l], sh.gcol[l]);
          fma_(ta1, sh.Ts[lane][l + 1], sh.gcol[l + 1]);
        }
        if (l < j) fma_(ta0, sh.Ts[lane][l], sh.gcol[l]);
        const cx<R> ta = ta0 + ta1;
        sh.Ts[lane][j] = mk<R>(-tau * ta.re, -tau * ta.im);
      }
      if (lane == j) sh.Ts[j][j] = mk<R>(tau, 0);
    }
    // a_c <- a_c - v (2 v^H a_c), c in (j, bw), own rows >= j
    if (has_next) {
      const cx<R> wf = sh.wfull[lane];
      const bool upd = lane > j && lane < bw;
#pragma unroll
      for (int k = 0; k < RPW; ++k)
        if (k >= kmin && k < kmax) {
          const cx<R> v = shfl_idx(a[k], j);
          if (upd) a[k] = hh_upd(a[k], v, wf);
        }
    }
    if (tid == 0 && has_next) {
      const cx<R> vj = inv * (x0 - alpha);                      // the owner's v_j, same operations
      const cx<R> ajn = hh_upd(sh.ex_s[0], vj, sh.wfull[j + 1]);      // a'_j[j+1]
      const cx<R> x0n = j + 1 < mp ? hh_upd(sh.ex_s[2], sh.ex_s[1], sh.wfull[j + 1]) : mk<R>(0, 0);
      const R nA = sh.nrm_s;
      const R xn2n = nA - norm2(ajn);
      sh.x0_s = x0n;
      sh.xn2_s = xn2n > R(0) ? xn2n : R(0);
      sh.recompute_s = !(xn2n > R(0.5) * nA);
      if (!sh.recompute_s) {
        cx<R> al;
        R iv, ta;
        hh_pivot<R>(sh.xn2_s, x0n, &al, &iv, &ta);
        sh.alpha_s = al;
        sh.inv_s = iv;
        sh.tau_s = ta;
      }
    }
    __syncthreads();
    if (has_next && sh.recompute_s) {
      // column j+1 over rows >= j+1
      const int l1 = j + 1 > rank ? (j + 1 - rank + CS - 1) / CS : 0;
      const int kmin1 = l1 > wid ? (l1 - wid + QR_WARPS - 1) / QR_WARPS : 0;
      R sacc = 0;
#pragma unroll
      for (int k = 0; k < RPW; ++k)
        if (k >= kmin1 && k < kmax) sacc += norm2(a[k]);
      panel_norm_round<R>(sacc, mk<R>(0, 0), false, sh, cluster, CS, rank, j + 1, false, false, round);
    }
  }
  // write back V and the R part of A
#pragma unroll
  for (int k = 0; k < RPW; ++k) {
    const int li = wid + QR_WARPS * k;
    if (li < nloc && lane < bw) {
      const int pi = rank + li * CS;
      const long long gi = pb + pi;
      V[gi * ldv + pb + lane] = pi >= lane ? a[k] : mk<R>(0, 0);
      A[gi * lda + pb + lane] = pi < lane ? a[k] : (pi == lane ? sh.alphas[lane] : mk<R>(0, 0));
    }
  }
  if (rank == 0) {
    for (int e = tid; e < QB * QB; e += QR_THREADS) T[e] = sh.Ts[e / QB][e % QB];
    // rows of the outer block above this panel: zero in its reflector columns
    for (int e = tid; e < zr * QB; e += QR_THREADS)
      if (e % QB < bw) V[(long long)(pb - zr + e / QB) * ldv + pb + e % QB] = mk<R>(0, 0);
  }
}

// Register-resident panel factorisation with one pass over the panel and one
// cluster exchange per column.
//
// Layout as above: warp w of a CTA holds its local rows w, w + 16, ... (RPW of
// them), lane c holds column c; rows are dealt to the CTAs cyclically.  What
// bounds a column is the chain pass - block sum - exchange - pivot, so
//   * the update with reflector j and the products with the raw next column x
//     (S_c = sum conj(a_c) x over rows > j) share one pass; with h_c = (S_c -
//     alpha conj(row[c])) / un, row = row j+1 of the panel, both v^H a_c (c to the
//     right) and the v_c^H v of T (c to the left) follow after the exchange, and
//     S of the column itself is its exact squared norm: nothing is downdated
//     and no column needs a second round;
//   * after the exchange one warp of each CTA sums the shares and forms the
//     pivot (all 16 doing so cost more issue slots than the broadcast, and in
//     float64 queue for the SM's two lanes); a 17th warp without rows extends T.
// A 32-column panel of 8 matrices, complex64 (us, the kernel above in brackets):
// 2048 rows 90 (138), 512 rows 58 (91), 256 rows 55 (64); complex128, 256 rows of
// 4 matrices, 267 (332).
__device__ __forceinline__ void fused_pivot(double xn2, cx<double> x0, cx<double>* alpha, double* inv, double* tau) {
  hh_pivot<double>(xn2, x0, alpha, inv, tau);
}
// hh_pivot without divides and square roots on the column's chain (440 -> about
// 150 cycles); |x0| below 2^-50 is scaled away from denormal squares.
__device__ __forceinline__ void fused_pivot(float xn2, cx<float> x0, cx<float>* alpha, float* inv, float* tau) {
  const float s = fmaxf(fabsf(x0.re), fabsf(x0.im));
  const float up = s < 0x1p-50f ? 0x1p70f : 1.f, dn = s < 0x1p-50f ? 0x1p-70f : 1.f;
  const float a = x0.re * up, b = x0.im * up, q2 = fmaf(a, a, b * b);
  const bool nz = q2 > 0.f;
  const float qi = nz ? rsqrt_series(q2) : 0.f;
  const float pr = nz ? a * qi : 1.f, pi = b * qi, ax0 = q2 * qi * dn;
  const bool live = xn2 > 0.f;
  const float xn = live ? xn2 * rsqrt_series(xn2) : 0.f;
  *alpha = mk<float>(-xn * pr, -xn * pi);
  const float un2 = 2.f * fmaf(xn, ax0, xn2);
  *inv = live ? rsqrt_series(un2) : 0.f;
  *tau = live ? 2.f : 0.f;
}
template <typename R>
struct __align__(4 * sizeof(R)) VX {
  cx<R> v, x;
};
template <typename R>
struct FusedMsg {
  cx<R> s[QB];     // this CTA's S_c
  cx<R> row[QB];   // row j of the panel (from its owner only)
};
template <typename R, int RPW>
struct FusedShared {
  FusedMsg<R> msg[2][QR_CS_MAX];
  cx<R> row[QB];                 // row j of the panel (its owner)
  cx<R> g[QB];                   // the T warp's copy of h
  cx<R> sum[QB];                 // complex128: the block sums
  cx<R> raw[QR_WARPS][RPW][2];   // a warp's rows: entries of the last and of this column,
  VX<R> vx[QR_WARPS][RPW];       // and what becomes of them
  cx<R> red[QR_WARPS][QB + 1];
  cx<R> alphas[QB];
  cx<R> h[QB];                   // of the column: h_c, 1 / un
  R inv;
  cx<R> Ts[QB][QB + 1];
};

constexpr int FUSED_THREADS = QR_THREADS + 32;   // and the T warp

template <typename R, int RPW>
__global__ void __launch_bounds__(FUSED_THREADS) qr_panel_fused_kernel(cx<R>* Ab, long long sA, int lda, int m, int pb,
                                                                     int bw, cx<R>* Vb, long long sV, int ldv,
                                                                     cx<R>* Tb, long long sT, int zr) {
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks(), lcs = __ffs(CS) - 1;   // a power of two (integer divides cost more than the pass)
  const int rank = (int)cluster.block_rank();
  const int z = blockIdx.y;
  cx<R>* A = Ab + z * sA;
  cx<R>* V = Vb + z * sV;
  cx<R>* T = Tb + z * sT;
  constexpr bool F64 = std::is_same<R, double>::value;
  __shared__ FusedShared<R, RPW> sh;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int mp = m - pb;
  const int nloc = mp > rank ? (mp - rank + CS - 1) >> lcs : 0;
  const bool t_warp = wid == QR_WARPS;   // holds no rows
  const int kmax = !t_warp && nloc > wid ? (nloc - wid + QR_WARPS - 1) / QR_WARPS : 0;   // this warp's live registers
  cx<R> a[RPW];
#pragma unroll
  for (int k = 0; k < RPW; ++k) {
    const int li = wid + QR_WARPS * k;
    a[k] = mk<R>(0, 0);
    if (!t_warp && li < nloc && lane < bw) a[k] = A[(long long)(pb + rank + li * CS) * lda + pb + lane];
  }
  for (int e = tid; e < QB * QB; e += FUSED_THREADS) sh.Ts[e / QB][e % QB] = mk<R>(0, 0);
  // every CTA of the cluster is running before anyone writes into its shared memory
  cluster.sync();
  cx<R> alpha = mk<R>(0, 0), wf = mk<R>(0, 0);   // of the last column; wf: this lane's 2 v^H a_c
  R inv = 0;
  for (int j = 0; j < bw; ++j) {
    const int buf = j & 1;
    // register of row j - 1 (the last pivot row) and of row j, -1 if not in this warp
    const int lstep = lcs + 4, mask = (QR_WARPS << lcs) - 1, d1 = j - 1 - rank - (wid << lcs), d0 = d1 + 1;
    const int k1 = (j > 0 && d1 >= 0 && (d1 & mask) == 0) ? d1 >> lstep : -1;
    const int k0 = (d0 >= 0 && (d0 & mask) == 0 && j < mp) ? d0 >> lstep : -1;
    // first register with a row >= j - 1
    const int jr = j > 0 ? j - 1 : 0;
    const int l1 = jr > rank ? (jr - rank + CS - 1) >> lcs : 0;
    const int kmin = l1 > wid ? (l1 - wid + QR_WARPS - 1) / QR_WARPS : 0;
    cx<R> acc0 = mk<R>(0, 0), acc1 = mk<R>(0, 0);
    if (t_warp) {
    } else if (j == 0) {
#pragma unroll
      for (int k = 0; k < RPW; ++k)
        if (k < kmax) {
          const cx<R> x = shfl_idx(a[k], 0);
          if (k & 1) fmac_(acc1, a[k], x); else fmac_(acc0, a[k], x);
        }
    } else {
      // the last column's and this column's raw entries to shared memory; lane k
      // turns row k's into v and the updated x (0 where the row takes no part);
      // every lane then reads (v, x) of a row with one broadcast load
      const cx<R> wj = shfl_idx(wf, j);
      if (lane == j - 1 || lane == j) {
#pragma unroll
        for (int k = 0; k < RPW; ++k) sh.raw[wid][k][lane - (j - 1)] = a[k];
      }
      if (!F64) __syncwarp();
      if (!F64 && lane < RPW) {
        cx<R> u = sh.raw[wid][lane][0], x = sh.raw[wid][lane][1];
        const bool live = lane >= kmin && lane < kmax;
        if (lane == k1) u = u - alpha;
        const cx<R> v = live ? inv * u : mk<R>(0, 0);
        x = hh_upd(x, v, wj);
        if (!live || lane == k1) x = mk<R>(0, 0);
        sh.vx[wid][lane] = VX<R>{v, x};
      }
      if (!F64) __syncwarp();
    }
    if (F64 && j > 0) {
      // float64 instructions cost the SM 19 cycles each however few lanes they use:
      // lane = row for the CTA's rows, 32 at a time, by as few warps as that takes
      __syncthreads();
      const cx<R> wj = shfl_idx(wf, j);
      for (int q = wid; 32 * q < QR_WARPS * RPW; q += QR_WARPS) {
        const int w = lane & (QR_WARPS - 1), k = 2 * q + (lane >> 4);
        const int pi = rank + ((w + QR_WARPS * k) << lcs);
        if (k < RPW) {
          cx<R> u = sh.raw[w][k][0], x = sh.raw[w][k][1];
          const bool live = pi >= j - 1 && pi < mp;
          if (pi == j - 1) u = u - alpha;
          const cx<R> v = live ? inv * u : mk<R>(0, 0);
          x = hh_upd(x, v, wj);
          if (!live || pi == j - 1) x = mk<R>(0, 0);
          sh.vx[w][k] = VX<R>{v, x};
        }
      }
      __syncthreads();
    }
    if (!t_warp && j > 0) {
#pragma unroll
      for (int k = 0; k < RPW; ++k) {
        const VX<R> q = sh.vx[wid][k];
        if (lane != j - 1) a[k] = hh_upd(a[k], q.v, wf);   // wf = 0 left of the column
        else if (k >= kmin) a[k] = q.v;
        if (k & 1) fmac_(acc1, a[k], q.x); else fmac_(acc0, a[k], q.x);
      }
    }
    if (!t_warp) sh.red[wid][lane] = acc0 + acc1;
    if (!t_warp && k0 >= 0) {
      cx<R> r = mk<R>(0, 0);
#pragma unroll
      for (int k = 0; k < RPW; ++k)
        if (k == k0) r = a[k];
      sh.row[lane] = r;
    }
    __syncthreads();
    // warp d forms the block sums (lane = column) and stores them to CTA d in one piece:
    // stores that scatter over the CTAs cost their number of pieces (a shared-memory
    // pipe 92 % busy, and about 680 cycles more per column).  In float64 two warps
    // form the real and the imaginary sums once.
    if (F64) {
      if (wid < 2) {
        R t = 0;
#pragma unroll
        for (int w = 0; w < QR_WARPS; ++w) t += wid ? sh.red[w][lane].im : sh.red[w][lane].re;
        (wid ? sh.sum[lane].im : sh.sum[lane].re) = t;
      }
      __syncthreads();
    }
    if (wid < CS) {
      cx<R> t0 = mk<R>(0, 0), t1 = t0, t2 = t0, t3 = t0;
      if (F64) {
        t0 = sh.sum[lane];
      } else {
#pragma unroll
        for (int w = 0; w < QR_WARPS; w += 4) {
          t0 = t0 + sh.red[w][lane];
          t1 = t1 + sh.red[w + 1][lane];
          t2 = t2 + sh.red[w + 2][lane];
          t3 = t3 + sh.red[w + 3][lane];
        }
        t0 = (t0 + t1) + (t2 + t3);
      }
      FusedMsg<R>* dst = cluster.map_shared_rank(&sh.msg[buf][rank], wid);
      dst->s[lane] = t0;
      if (rank == (j & (CS - 1))) dst->row[lane] = sh.row[lane];
    }
    cluster.sync();
    if (wid == 0) {   // one warp: lane c forms h_c of the column, and all its pivot
      cx<R> s0 = mk<R>(0, 0), s1 = s0;
#pragma unroll
      for (int src = 0; src < QR_CS_MAX; src += 2) {   // independent loads
        if (src < CS) s0 = s0 + sh.msg[buf][src].s[lane];
        if (src + 1 < CS) s1 = s1 + sh.msg[buf][src + 1].s[lane];
      }
      const cx<R> S = s0 + s1;
      const R xn2 = __shfl_sync(0xffffffffu, S.re, j);
      const cx<R> rc = j < mp ? sh.msg[buf][j & (CS - 1)].row[lane] : mk<R>(0, 0);
      R tau;
      fused_pivot(xn2, shfl_idx(rc, j), &alpha, &inv, &tau);
      sh.h[lane] = inv * (S - alpha * conj(rc));
      if (lane == 0) {
        sh.alphas[j] = alpha;
        sh.inv = inv;
      }
    }
    __syncthreads();
    const cx<R> h = sh.h[lane];
    alpha = sh.alphas[j];
    inv = sh.inv;
    wf = (lane > j && lane < bw) ? mk<R>(R(2) * h.re, -R(2) * h.im) : mk<R>(0, 0);
    // T[0:j, j] = -tau T[0:j, 0:j] (V^H v_j), T[j][j] = tau, by a warp that has no rows, while
    // the others are at the next column.  A row of T depends on itself only: CTA r keeps
    // rows r, r + CS, ..., CS lanes to a row (with all rows in one CTA the up to 31
    // dependent float64 steps held up the next column's barrier:
    // complex128 emulation at chi 256 35.3 -> 33.2 ms, the entropy profile 32.7 -> 31.2 ms).
    if (t_warp) {
      const R tau = inv > R(0) ? R(2) : R(0);
      const int sub = lane & (CS - 1), row = rank + lane - sub;
      sh.g[lane] = h;
      __syncwarp();
      cx<R> ta = mk<R>(0, 0);
      for (int l = sub; l < j; l += CS) fma_(ta, sh.Ts[row][l], sh.g[l]);
      for (int o = 1; o < CS; o <<= 1) ta = ta + shfl_xor(ta, o);
      if (sub == 0 && row < j) sh.Ts[row][j] = mk<R>(-tau * ta.re, -tau * ta.im);
      if (sub == 0 && row == j) sh.Ts[j][j] = mk<R>(tau, 0);
      __syncwarp();
    }
  }
  // the last column's reflector
  {
    const int j = bw - 1, d1 = j - rank - (wid << lcs);
    const int k1 = (d1 >= 0 && (d1 & ((QR_WARPS << lcs) - 1)) == 0) ? d1 >> (lcs + 4) : -1;
    const int l1 = j > rank ? (j - rank + CS - 1) >> lcs : 0;
    const int kmin = l1 > wid ? (l1 - wid + QR_WARPS - 1) / QR_WARPS : 0;
#pragma unroll
    for (int k = 0; k < RPW; ++k)
      if (k >= kmin && k < kmax && lane == j) {
        cx<R> u = a[k];
        if (k == k1) u = u - alpha;
        a[k] = inv * u;
      }
  }
  __syncthreads();
  // write back V and the R part of A
#pragma unroll
  for (int k = 0; k < RPW; ++k) {
    const int li = wid + QR_WARPS * k;
    if (!t_warp && li < nloc && lane < bw) {
      const int pi = rank + li * CS;
      const long long gi = pb + pi;
      V[gi * ldv + pb + lane] = pi >= lane ? a[k] : mk<R>(0, 0);
      A[gi * lda + pb + lane] = pi < lane ? a[k] : (pi == lane ? sh.alphas[lane] : mk<R>(0, 0));
    }
  }
  for (int e = tid; e < QB * QB; e += FUSED_THREADS)
    if (((e / QB) & (CS - 1)) == rank) T[e] = sh.Ts[e / QB][e % QB];
  if (rank == 0) {
    // rows of the outer block above this panel: zero in its reflector columns
    for (int e = tid; e < zr * QB; e += FUSED_THREADS)
      if (e % QB < bw) V[(long long)(pb - zr + e / QB) * ldv + pb + e % QB] = mk<R>(0, 0);
  }
}

constexpr int QR_KEEP_MAX = 160;
constexpr int QNB = 128;   // outer block: 4 panels applied to the trailing matrix together

// Compact-WY factor of an outer block of np_in <= 4 panels from the panels'
// factors T_a (32 x 32, upper) and the Gram G = V^H V of the block's
// reflectors (nbw x nbw): the product of the panels' block reflectors is
// I - V T V^H with T upper triangular, T_aa = T_a and, block column by block
// column, T[0:a, a] = -T[0:a, 0:a] G[0:a, a] T_a.  One CTA per matrix;
// writes T (QNB x QNB, zero outside nbw x nbw).
// G's block column and T_a are staged; a thread's rows (warp + 8 q, one column) run
// through the sums together, each in ascending order,
// without a load from L2 per step (64 columns 11 -> 6 us, 128 columns about 40 -> 20 us).
template <typename R>
__global__ void __launch_bounds__(256) wy_merge_t_kernel(const cx<R>* Tpb, long long sTp, const cx<R>* Gb, long long sG,
                                                         int nbw, cx<R>* Tob, long long sTo) {
  extern __shared__ unsigned char smem_raw[];
  cx<R>* X = reinterpret_cast<cx<R>*>(smem_raw);   // [QNB - QB][QB + 1]
  cx<R>* Gs = X + (QNB - QB) * (QB + 1);           // [QNB - QB][QB + 1]
  cx<R>* Ts = Gs + (QNB - QB) * (QB + 1);          // [QB][QB + 1]
  const int z = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const cx<R>* Tp = Tpb + z * sTp;
  const cx<R>* G = Gb + z * sG;
  cx<R>* T = Tob + z * sTo;
  const int np_in = (nbw + QB - 1) / QB;
  for (int e = tid; e < QNB * QNB; e += 256) {
    const int a = e / QNB / QB, b = e % QNB / QB;
    if (a != b || a >= np_in) T[e] = mk<R>(0, 0);
  }
#pragma unroll
  for (int q = 0; q < QNB / 8; ++q) {
    const int r = warp + 8 * q;   // every thread's loads in flight together
    if (r / QB < np_in) T[(long long)r * QNB + r / QB * QB + lane] = Tp[(long long)r * QB + lane];
  }
  constexpr int RQ = 4;   // rows of a thread in flight
  for (int b = 1; b < np_in; ++b) {
    const int rows = b * QB, c0 = b * QB;
    for (int r = warp; r < rows; r += 8)
      Gs[r * (QB + 1) + lane] = c0 + lane < nbw ? G[(long long)r * nbw + c0 + lane] : mk<R>(0, 0);
    for (int r = warp; r < QB; r += 8) Ts[r * (QB + 1) + lane] = Tp[(long long)b * QB * QB + r * QB + lane];
    __syncthreads();
    for (int r0 = warp; r0 < rows; r0 += 8 * RQ) {
      // X = T[0:rows, 0:rows] G[0:rows, c0:c0+32]   (T upper triangular)
      cx<R> acc[RQ];
#pragma unroll
      for (int q = 0; q < RQ; ++q) acc[q] = mk<R>(0, 0);
      const cx<R>* Tr = T + (long long)r0 * QNB;
      const int full = r0 + 8 * (RQ - 1);
      for (int l = r0; l < full; ++l) {
        const cx<R> g = Gs[l * (QB + 1) + lane];
#pragma unroll
        for (int q = 0; q < RQ - 1; ++q)
          if (r0 + 8 * q <= l) fma_(acc[q], Tr[q * 8 * QNB + l], g);
      }
#pragma unroll 4
      for (int l = full; l < rows; ++l) {
        const cx<R> g = Gs[l * (QB + 1) + lane];
#pragma unroll
        for (int q = 0; q < RQ; ++q) fma_(acc[q], Tr[q * 8 * QNB + l], g);
      }
#pragma unroll
      for (int q = 0; q < RQ; ++q) X[(r0 + 8 * q) * (QB + 1) + lane] = c0 + lane < nbw ? acc[q] : mk<R>(0, 0);
      __syncwarp();   // a warp reads back its own rows
      // T[0:rows, c0:c0+32] = -X T_b   (T_b upper triangular)
#pragma unroll
      for (int q = 0; q < RQ; ++q) acc[q] = mk<R>(0, 0);
#pragma unroll 4
      for (int l = 0; l < QB; ++l) {
        if (l > lane) continue;
        const cx<R> t = Ts[l * (QB + 1) + lane];
#pragma unroll
        for (int q = 0; q < RQ; ++q) fma_(acc[q], X[(r0 + 8 * q) * (QB + 1) + l], t);
      }
#pragma unroll
      for (int q = 0; q < RQ; ++q)
        T[(long long)(r0 + 8 * q) * QNB + c0 + lane] = mk<R>(-acc[q].re, -acc[q].im);
    }
    __syncthreads();
  }
}

template <typename R>
__global__ void qr_extract_r2_kernel(const cx<R>* Ab, long long sA, int lda, int k, int n, cx<R>* Rb, long long sR) {
  const int z = blockIdx.y;
  const cx<R>* A = Ab + z * sA;
  cx<R>* Rm = Rb + z * sR;
  const long long count = (long long)k * n;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    const int row = (int)(i / n), col = (int)(i % n);
    Rm[i] = col >= row ? A[(long long)row * lda + col] : mk<R>(0, 0);
  }
}

template <typename K, typename... Args>
static cudaError_t launch_cluster_qr(K kernel, int cs, int batch, int threads, size_t smem, cudaStream_t st,
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

QrWork qr_workspace(int m, int n) {
  QrWork w;
  const int k = std::min(m, n);
  const int np = (k + QB - 1) / QB;
  const int nblk = (k + QNB - 1) / QNB;
  // V (m x n) + panel T (np x 32 x 32) + WY application workspace (a block's own columns)
  // + block T (nblk x 128 x 128) + Gram (128 x 128) + W1, W2 (128 x n each)
  w.cx_elems = (long long)m * n + (long long)np * QB * QB + wy_workspace(m, std::min(n, QNB - QB)) + (long long)nblk * QNB * QNB +
               (long long)QNB * QNB + 2LL * QNB * n + 64;
  return w;
}

// Factor the panel A[pb:m, pb:pb+bw] of every matrix (V, its T at Tp); zr rows
// above pb belong to the same outer block and get zeros in V's panel columns.
template <typename R>
static cudaError_t panel_factor(cudaStream_t st, cx<R>* A, long long sA, int m, int n, int pb, int bw, cx<R>* V,
                                long long sV, cx<R>* Tp, long long sT, int zr, int batch) {
  const int mp = m - pb;
  // panel flops: per column j, reflector products and update of the bw-1-j columns to its right
  // and the v_c^H v_j of the j columns to its left, over mp - j rows (8 real flops per complex MAC)
  double work = 0;
  for (int j = 0; j < bw; ++j) work += 8.0 * (double)(mp - j) * (2.0 * (bw - 1 - j) + j + 1);
  ProfScope ps(st, K_QR_FACTOR, 1, work * batch);
  // register-resident panel when every CTA's rows fit 16 warps x 16 registers
  int csr = mp >= 512 ? 8 : (mp >= 128 ? 4 : (mp >= 32 ? 2 : 1));
  // float64 runs at two lanes per SM and bounds the panel: more CTAs per matrix
  if (std::is_same<R, double>::value && mp >= 64) csr = 8;
  if ((mp + csr - 1) / csr > 16 * QR_WARPS) csr = 16;
  const int nl = (mp + csr - 1) / csr;
  // The fused kernel is the faster at every size; complex64 matrices of up to
  // QR_KEEP_MAX rows (at most 64 to a CTA) keep the other one so that small jobs'
  // results stay as they were (see EIGH_F64_MAX).
  const bool fused = std::is_same<R, double>::value || m > QR_KEEP_MAX;
  auto go = [&](auto kernel) {
    return launch_cluster_qr(kernel, csr, batch, fused ? FUSED_THREADS : QR_THREADS, 0, st, A, sA, n, m, pb, bw, V, sV, n, Tp, sT, zr);
  };
#define NNE_PANEL(RPW)                                                                       \
  if (nl <= RPW * QR_WARPS) {                                                                \
    if (fused) return go(qr_panel_fused_kernel<R, RPW>);                                     \
    if constexpr (std::is_same<R, float>::value && RPW <= 4) return go(qr_panel_reg_kernel<R, RPW>); \
  }
  NNE_PANEL(1)
  NNE_PANEL(2)
  NNE_PANEL(4)
  NNE_PANEL(8)
  NNE_PANEL(16)
#undef NNE_PANEL
  int cs = mp >= 512 ? 8 : (mp >= 128 ? 4 : (mp >= 32 ? 2 : 1));
  int maxloc = (mp + cs - 1) / cs;
  size_t smem = sizeof(cx<R>) * (size_t)maxloc * PS;
  if (smem > 160 * 1024) {
    cs = 16;
    maxloc = (mp + cs - 1) / cs;
    smem = sizeof(cx<R>) * (size_t)maxloc * PS;
  }
  return launch_cluster_qr(qr_panel_kernel<R>, cs, batch, QR_THREADS, smem, st, A, sA, n, m, pb, bw, V, sV, n, Tp, sT,
                           maxloc, zr);
}

// Blocked Householder QR.  Outer blocks of 128 columns: their four 32-column
// panels are factored and applied to the rest of the block one at a time
// (wy_apply); the block's reflectors are then merged into one compact-WY
// factor (Gram V^H V and wy_merge_t) and applied to the trailing columns, and
// later to Q, with three GEMMs each (tensor cores for complex64).
template <typename R>
cudaError_t qr(cudaStream_t st, cx<R>* A, long long sA, int m, int n, cx<R>* Q, long long sQ, cx<R>* Rout,
               long long sR, void* cx_ws, int batch) {
  const int k = std::min(m, n);
  if (k <= 0 || batch <= 0) return cudaSuccess;
  const int np = (k + QB - 1) / QB, nblk = (k + QNB - 1) / QNB;
  cx<R>* V = reinterpret_cast<cx<R>*>(cx_ws);
  const long long sV = (long long)m * n;
  cx<R>* T = V + sV * batch;
  const long long sT = (long long)np * QB * QB;
  cx<R>* wyws = T + sT * batch;
  cx<R>* Tb = wyws + wy_workspace(m, std::min(n, QNB - QB)) * batch;   // a block's own columns
  const long long sTb = (long long)nblk * QNB * QNB;
  cx<R>* G = Tb + sTb * batch;
  const long long sG = (long long)QNB * QNB;
  cx<R>* W1 = G + sG * batch;
  const long long sW = (long long)QNB * n;
  cx<R>* W2 = W1 + sW * batch;
  const cx<R> one = mk<R>(1, 0), zero = mk<R>(0, 0), mone = mk<R>(-1, 0);
  const size_t merge_smem = sizeof(cx<R>) * (2 * (QNB - QB) + QB) * (QB + 1);
  cudaError_t e;
  if ((e = ensure_kernel_smem((const void*)wy_merge_t_kernel<R>, merge_smem, false)) != cudaSuccess) return e;
  for (int b = 0; b < nblk; ++b) {
    const int b0 = b * QNB, bend = std::min(k, b0 + QNB), nbw = bend - b0, mpb = m - b0;
    for (int pb = b0; pb < bend; pb += QB) {
      const int bw = std::min(QB, bend - pb), mp = m - pb, p = pb / QB;
      if ((e = panel_factor<R>(st, A, sA, m, n, pb, bw, V, sV, T + p * QB * QB, sT, pb - b0, batch)) != cudaSuccess)
        return e;
      const int nt_in = bend - pb - bw;
      if (nt_in > 0) {
        // rest of the block: A_t <- (I - V T V^H)^H A_t
        cx<R>* Vp = V + (long long)pb * n + pb;
        cx<R>* At = A + (long long)pb * n + pb + bw;
        if ((e = wy_apply<R>(st, false, Vp, sV, n, T + p * QB * QB, sT, QB, true, bw, mp, nt_in, At, sA, n, wyws,
                             batch)) != cudaSuccess)
          return e;
      }
    }
    // block factor: G = V_b^H V_b, then T_b
    cx<R>* Vb = V + (long long)b0 * n + b0;
    if ((e = cgemm<R>(st, OP_C, OP_N, nbw, nbw, mpb, one, Vb, sV, n, Vb, sV, n, zero, G, sG, nbw, batch)) !=
        cudaSuccess)
      return e;
    {
      ProfScope ps(st, K_WY);
      wy_merge_t_kernel<R><<<batch, 256, merge_smem, st>>>(T + (b0 / QB) * QB * QB, sT, G, sG, nbw,
                                                           Tb + (long long)b * QNB * QNB, sTb);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const int ntr = n - bend;
    if (ntr > 0) {
      // trailing columns: C <- (I - V_b T_b V_b^H)^H C
      cx<R>* Ct = A + (long long)b0 * n + bend;
      cx<R>* Tbb = Tb + (long long)b * QNB * QNB;
      if ((e = cgemm<R>(st, OP_C, OP_N, nbw, ntr, mpb, one, Vb, sV, n, Ct, sA, n, zero, W1, sW, ntr, batch)) !=
          cudaSuccess)
        return e;
      if ((e = cgemm<R>(st, OP_C, OP_N, nbw, ntr, nbw, one, Tbb, sTb, QNB, W1, sW, ntr, zero, W2, sW, ntr, batch)) !=
          cudaSuccess)
        return e;
      if ((e = cgemm<R>(st, OP_N, OP_N, mpb, ntr, nbw, mone, Vb, sV, n, W2, sW, ntr, one, Ct, sA, n, batch)) !=
          cudaSuccess)
        return e;
    }
  }
  if (Rout) {
    ProfScope ps(st, K_ELEMWISE);
    qr_extract_r2_kernel<R><<<dim3(64, batch), 256, 0, st>>>(A, sA, n, k, n, Rout, sR);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if ((e = identity<R>(st, Q, sQ, m, k, batch)) != cudaSuccess) return e;
  for (int b = nblk - 1; b >= 0; --b) {
    const int b0 = b * QNB, nbw = std::min(k, b0 + QNB) - b0, mpb = m - b0, kc = k - b0;
    cx<R>* Vb = V + (long long)b0 * n + b0;
    cx<R>* Qb = Q + (long long)b0 * k + b0;
    cx<R>* Tbb = Tb + (long long)b * QNB * QNB;
    // Q_b <- (I - V_b T_b V_b^H) Q_b
    if ((e = cgemm<R>(st, OP_C, OP_N, nbw, kc, mpb, one, Vb, sV, n, Qb, sQ, k, zero, W1, sW, kc, batch)) !=
        cudaSuccess)
      return e;
    if ((e = cgemm<R>(st, OP_N, OP_N, nbw, kc, nbw, one, Tbb, sTb, QNB, W1, sW, kc, zero, W2, sW, kc, batch)) !=
        cudaSuccess)
      return e;
    if ((e = cgemm<R>(st, OP_N, OP_N, mpb, kc, nbw, mone, Vb, sV, n, W2, sW, kc, one, Qb, sQ, k, batch)) !=
        cudaSuccess)
      return e;
  }
  return cudaSuccess;
}

template cudaError_t qr<float>(cudaStream_t, cx<float>*, long long, int, int, cx<float>*, long long, cx<float>*,
                               long long, void*, int);
template cudaError_t qr<double>(cudaStream_t, cx<double>*, long long, int, int, cx<double>*, long long, cx<double>*,
                                long long, void*, int);

}  // namespace nne
