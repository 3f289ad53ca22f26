// Blocked Householder QR with panel-wise pivoting for the UDV stack of
// Eq. (3) (Sec. 2: the O(Lambda N^3) stabilised matrix work behind
// G_ij(tau_l)).
//
// Input and output as the column-pivoted QR of k_cluster.cu: X^T stored
// row-major (row c = column c of X) in; Q^T, D = |diag R| and
// Rtil = D^{-1} R P^T with X = Q diag(D) Rtil out.  Pivoting works on blocks
// of kNB columns: at the start of each panel the columns not yet factorised
// are sorted by the norm of their remaining part (rows c0 .. n - 1, after all
// earlier reflectors), the kNB largest form the panel, and within the panel
// each step takes the column of largest remaining norm (downdated as in
// LAPACK's xGEQP3).  For the graded products B_l ... B_1 U D of the stack
// this keeps |R_ij| close to |R_ii| as column pivoting does, so that
// T = D^{-1} R P^T stays well conditioned, while the trailing updates run as
// matrix products:
//
//   for each panel of w <= kNB columns (rows c0 .. n - 1):
//     k_qrb_panel  sort the remaining columns, FP64 Householder QR of the
//                  panel in registers with local pivoting, the compact-WY
//                  factor T of its reflectors (H_0 ... H_{w-1} = I - V T V^T)
//                  and Y = T^T V^T;
//     trailing columns A <- (I - V T^T V^T) A = A - V (Y A), written in the
//     transposed storage (rows of A_rows = columns of A) as two tensor-core
//     products:
//       W^T = A_rows Y^T          (M = trailing columns, N = w, K = m)
//       A_rows -= W^T V^T         (M = trailing columns, N = m, K = w)
//   Q^T accumulated backwards from I, Q^T <- Q^T (I - V T^T V^T):
//       W^T = Qt_rows V           (M = m, N = w, K = m)
//       Qt_rows -= W^T Y          (M = m, N = m, K = w)
//
// The products run on the digit-sliced tcgen05 path (k_ozaki.cu), which keeps
// FP64-level accuracy relative to the size of each row and column; only the
// panels use the FP64 pipe.
//
// Storage per matrix: two buffers that the panels alternate between (the
// rows of panel p, R on and above the diagonal, stay in the buffer that
// panel wrote), the Householder vectors V^T in the Rtil buffer and
// Y = T^T V^T in the X buffer (each consumed before it is overwritten).
#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>

#include "common.cuh"
#include "kernels.h"
#include "qr_scalars.cuh"

namespace dqmc {
namespace {

namespace cg = cooperative_groups;

constexpr int kNB = kQrbNB;

constexpr int kPCS = 4;             // CTAs per matrix (one cluster)
constexpr int kPCW = kNB / kPCS;    // column warps per CTA
constexpr int kPW = 16;             // warps per CTA: columns, scalars, copies
constexpr int kPT = 32 * kPW;

// x 2^-e on the exponent field; what would leave the range of normal numbers
// becomes zero.  Inf and NaN stay.
__device__ __forceinline__ double qb_shift(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = static_cast<int>((b >> 52) & 0x7FF), f = ex - e;
  if (ex == 0x7FF || f >= 0x7FF) return x;
  if (ex == 0 || f <= 0) return 0.0;
  return __longlong_as_double(b - (static_cast<long long>(e) << 52));
}

__device__ __forceinline__ int qb_exp(double x) {  // floor(log2 |x|), 0 for x = 0
  const int ex = (__double2hiint(x) >> 20) & 0x7FF;
  return ex ? ex - 1023 : 0;
}

// A CTA's best column for a step: sigma, the pivot key (0: no live column) and
// the column.
struct QbCand {
  double sigma;
  unsigned key;
  int col;
};

__device__ __forceinline__ void qb_bar(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// One panel, one cluster of four CTAs per matrix; rows of the transposed
// storage are columns of X; `src` holds the matrix after the previous panel
// (the input X^T for the first), `dst` receives the rows c0 .. n - 1.
//
// What bounds it: the chain of w Householder steps.  The work of a step is
// small (an FP64 warp instruction takes its SM quarter 64 to 76 clocks, and a
// step has a few per warp), so the kernel is laid out for a short chain: a
// warp per panel column, the column in registers (row c0 + lane + 32 t in
// x[t]), eight columns per CTA; sums over the lanes in integer arithmetic; the
// scalars of the reflector in one warp beside the dot products, without
// sqrt() and division; and one cluster barrier per step, which carries each
// CTA's candidate for the next pivot column with its sigma, prepared before
// the other columns' norms are touched again.
//
//  1. Sort: the rows c >= c0 of src by the norm of their entries c0 .. n - 1
//     (each CTA finds the keys of a quarter of them and writes them to all).
//     The w largest are the panel, column i with warp i / 4 of CTA i mod 4.
//     Ranks w .. m - 1 go to dst rows c0 + w .. n - 1 (whole rows, copied by
//     spare warps beside step 2), perm follows.
//  2. Step j (as k_qr_smem): x_p the pivot, s = |x_p[j..)|, v = x_p[j..) with
//     v[j] = sign(x_p[j]) (|x_p[j]| + s), H = I - kap v v^T.  Every column's
//     warp forms g = v . x_s: for a column not yet chosen the factor
//     c = kap g, R_js and the downdated norm (summed afresh as in k_qr_smem),
//     then x_s -= c v; for a finished column, whose registers hold v_s, the
//     entry v_s . v_j of the Gram matrix.
//  3. H_0 ... H_{w-1} = I - V T V^T with T[0:q, q] = -kap_q T[0:q, 0:q] (V^T
//     v_q)[0:q], T[q][q] = kap_q, a column of T per step by the warp of the
//     scalars.  V leaves scaled by powers of two to 1 <= |v_q[q]| < 2 (the
//     digit-sliced products that follow add over q), T with it.  Then
//     Y = T^T V^T, 32 rows at a time spread over the CTAs.
//  4. Panel rows to dst rows c0 .. c0 + w - 1 (entries below c0 moved with
//     their column, R on and above the diagonal), v_q to row c0 + q of Vt, Y
//     to rows c0 .. of Yt (entries c0 ..), D[c0 + q] = |beta_q|, perm.
//
// A whole factorisation at n = 256 (with its 30 products, about 1.4 ms of it):
// 4 matrices 2.98 -> 1.89 ms, 64: 3.49 -> 2.71 ms, 128: 6.51 -> 4.86 ms; n =
// 160, 16 matrices: 1.69 -> 1.08 ms.  Before: a pair of CTAs with the rows
// split, columns in shared memory, two exchanges per step and sqrt() and a
// division in the chain.
__global__ void __launch_bounds__(kPT, 2) k_qrb_panel(const double* Wsall, long long sWs, double* Wdall,
                                                     long long sWd, int* permall, double* Vall,
                                                     long long sV, double* Yall, long long sY,
                                                     double* Dall, long long sD, int n, int c0, int w,
                                                     int* status) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = static_cast<int>(cl.block_rank());
  const int b = blockIdx.x / kPCS;
  const int m = n - c0, nt = (m + 31) / 32, mp = 32 * nt;
  const double* Ws = Wsall + b * sWs;
  double* Wd = Wdall + b * sWd;
  int* perm = permall + static_cast<long long>(b) * n;
  double* Vt = Vall + b * sV;
  double* Yt = Yall + b * sY;
  double* D = Dall + b * sD;
  extern __shared__ __align__(16) double qb_sm[];
  double* Vb = qb_sm;            // [w][mp] reflectors
  double* buf = qb_sm + w * mp;  // [2][kPCS][mp] candidates by step parity and CTA
  __shared__ float key[kMaxN];
  __shared__ short src_of[kMaxN];  // rank -> source row - c0
  __shared__ int pold[kMaxN];      // perm[c0 ..] on entry
  __shared__ double T[kNB][kNB + 1];
  __shared__ double G[kNB][kNB + 1];  // v_s . v_q, s < q
  __shared__ double kaps[kNB], betas[kNB], vjs[kNB];
  __shared__ QbCand cand[2][kPCS];
  __shared__ unsigned keys[2][kPCW];
  __shared__ unsigned char wait_sum[kPCW];
  __shared__ double kap_sh, vj_sh;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  constexpr int kR = kMaxN / 32;

  // 1. sort the remaining columns
  cl.sync();  // the peers run: their shared memory may be written
  for (int c = rank + kPCS * wp; c < m; c += kPCS * kPW) {
    const float k = qb_norm_key(Ws + static_cast<size_t>(c0 + c) * n + c0, m, lane);
    if (lane < kPCS) *cl.map_shared_rank(key + c, lane) = k;
  }
  for (int i = threadIdx.x; i < m; i += kPT) pold[i] = (c0 == 0) ? i : perm[c0 + i];
  cl.sync();
  for (int i = threadIdx.x; i < m; i += kPT) {
    const float ki = key[i];
    int rk = 0;
    for (int i2 = 0; i2 < m; ++i2) {
      const float k2 = key[i2];
      rk += (k2 > ki || (k2 == ki && i2 < i)) ? 1 : 0;
    }
    src_of[rk] = static_cast<short>(i);
  }
  __syncthreads();
  // columns too large for the sums to come: see kQsBig (keys: log2 of the squared
  // norms, 3e38 for one that is not finite)
  const float kmax = key[src_of[0]];
  const bool big = kmax >= 1020.0f && kmax < 1.0e38f;

  // 2. the panel
  double x[kR];
  int step = -1;                     // of this warp's column
  const int cid = rank + kPCS * wp;  // the column (column warps)
  if (wp < kPCW) {
    const bool exists = cid < w;
    bool live = exists;
    int es = 0;
#pragma unroll
    for (int t = 0; t < kR; ++t) {
      const int r = lane + 32 * t;
      x[t] = (exists && r < m) ? Ws[static_cast<size_t>(c0 + src_of[cid]) * n + c0 + r] : 0.0;
      if (big) x[t] *= kQsDown;
    }
    auto sumsq = [&](int j) {  // rows > j
      double a = (lane > j) ? x[0] * x[0] : 0.0;
#pragma unroll
      for (int t = 1; t < kR; ++t)
        if (t < nt) a = fma(x[t], x[t], a);
      return a;
    };
    auto pick = [&](const unsigned* ks) {  // warp of the largest key, -1: none
      const unsigned k = (lane < kPCW) ? ks[lane] : 0u;
      const unsigned km = __reduce_max_sync(0xFFFFFFFFu, k);
      return km ? __ffs(__ballot_sync(0xFFFFFFFFu, k == km)) - 1 : -1;
    };
    auto key_of = [](double v) { return (static_cast<unsigned>(__double2hiint(v)) & 0x7FFFFFFFu) + 1u; };
    // this warp's column as the CTA's candidate for step j (has: false: no
    // live column left)
    auto send = [&](int j, bool has, unsigned k) {
      QbCand cd{0.0, 0u, kNB};
      if (has) {
#pragma unroll
        for (int t = 0; t < kR; ++t)
          if (t < nt)
#pragma unroll
            for (int q = 0; q < kPCS; ++q)
              *cl.map_shared_rank(buf + ((j & 1) * kPCS + rank) * mp + lane + 32 * t, q) = x[t];
        cd.sigma = qs_warp_sum_pos(sumsq(j));
        cd.key = k;
        cd.col = cid;
      }
      if (lane < kPCS) *cl.map_shared_rank(&cand[j & 1][rank], lane) = cd;
    };
    double n1 = qs_warp_sum_pos(sumsq(-1)), n2 = n1;
    if (lane == 0) keys[0][wp] = live ? key_of(n1) : 0u;
    qb_bar(2, 32 * kPCW);
    {
      const int np = pick(keys[0]);
      if (np == wp || (np < 0 && wp == 0)) send(0, np >= 0, key_of(n1));
    }
    for (int j = 0; j < w; ++j) {
      cl.sync();
      int win = 0;
      QbCand best = cand[j & 1][0];
#pragma unroll
      for (int q = 1; q < kPCS; ++q) {
        const QbCand y = cand[j & 1][q];
        if (y.key > best.key || (y.key == best.key && y.col < best.col)) {
          best = y;
          win = q;
        }
      }
      const bool own = best.col == cid;
      const double* xp = buf + ((j & 1) * kPCS + win) * mp + lane;
      double v[kR];
#pragma unroll
      for (int t = 0; t < kR; ++t) v[t] = (t < nt) ? xp[32 * t] : 0.0;
      if (lane <= j) v[0] = 0.0;
      double a = 0.0;
      if (exists && !own) {
        a = x[0] * v[0];
#pragma unroll
        for (int t = 1; t < kR; ++t)
          if (t < nt) a = fma(x[t], v[t], a);
        a = qs_warp_sum(a);
      }
      const double xj = __shfl_sync(0xFFFFFFFFu, x[0], j);
      qb_bar(1, 32 * (kPCW + 1));
      const double vj = vj_sh;
      double c = 0.0;
      int rc = 0;
      unsigned k = 0u;
      if (own) {
        step = j;
        es = qb_exp(vj);
        live = false;
        if (lane == j) x[0] = vj;
      } else if (exists) {
        const double g = fma(vj, xj, a);
        if (live) {
          c = kap_sh * g;
          const double rj = fma(-c, vj, xj);
          if (lane == j) x[0] = rj;
          n1 = fma(-rj, rj, n1);
          if (__double2hiint(n1) < 0) n1 = 0.0;
          const int hn = __double2hiint(n1), hr = __double2hiint(n2);
          rc = (hn > hr - (26 << 20)) ? 0 : (hn > hr - (40 << 20)) ? 1 : 2;
          k = key_of(n1);
        } else if (lane < kPCS) {
          *cl.map_shared_rank(&G[step][j], lane) = qb_shift(g, es + qb_exp(vj));
        }
      }
      if (j + 1 == w) break;
      if (lane == 0) {
        keys[0][wp] = k;
        wait_sum[wp] = rc == 2;
      }
      qb_bar(2, 32 * kPCW);
      int np = pick(keys[0]);
      const bool ahead = !__any_sync(0xFFFFFFFFu, lane < kPCW && wait_sum[lane]);
      if (live) {
#pragma unroll
        for (int t = 0; t < kR; ++t)
          if (t < nt) x[t] = fma(-c, v[t], x[t]);
      }
      if (!ahead) {
        if (rc == 2) {
          n1 = n2 = qs_warp_sum_pos(sumsq(j));
          k = key_of(n1);
        }
        if (lane == 0) keys[1][wp] = k;
        qb_bar(2, 32 * kPCW);
        np = pick(keys[1]);
      }
      if (np == wp || (np < 0 && wp == 0))
        send(j + 1, np >= 0, k);
      else if (rc == 1)
        n1 = n2 = qs_warp_sum_pos(sumsq(j));
    }
    cl.sync();  // the Gram matrix is complete; no shared memory of a peer is touched any more
  } else if (wp == kPCW) {
    // column q of T from the Gram matrix; lanes over its rows, four partial
    // sums shorten the chain
    auto t_column = [&](int q) {
      double ti = 0.0;
      if (lane < q) {
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        for (int i = lane; i < q; i += 4)
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (i + u < q) a[u] = fma(T[lane][i + u], G[i + u][q], a[u]);
        ti = -kaps[q] * ((a[0] + a[1]) + (a[2] + a[3]));
      }
      __syncwarp();
      T[lane][q] = (lane == q) ? kaps[q] : ti;
      __syncwarp();
    };
    for (int j = 0; j < w; ++j) {
      cl.sync();
      int win = 0;
      QbCand best = cand[j & 1][0];
#pragma unroll
      for (int q = 1; q < kPCS; ++q) {
        const QbCand y = cand[j & 1][q];
        if (y.key > best.key || (y.key == best.key && y.col < best.col)) {
          best = y;
          win = q;
        }
      }
      double beta, kap, vj;
      qs_reflector(buf[((j & 1) * kPCS + win) * mp + j], best.sigma, beta, kap, vj);
      if (lane == 0) {
        kap_sh = kap;
        vj_sh = vj;
        betas[j] = beta;
        vjs[j] = vj;
        kaps[j] = qb_shift(kap, -2 * qb_exp(vj));
      }
      qb_bar(1, 32 * (kPCW + 1));
      if (j > 0) t_column(j - 1);
    }
    cl.sync();
    t_column(w - 1);
  } else if (wp == kPCW + 1) {  // keeps the reflectors
    if (rank == 0)
      for (int pos = w + lane; pos < m; pos += 32) perm[c0 + pos] = pold[src_of[pos]];
    for (int j = 0; j < w; ++j) {
      cl.sync();
      int win = 0;
      QbCand best = cand[j & 1][0];
#pragma unroll
      for (int q = 1; q < kPCS; ++q) {
        const QbCand y = cand[j & 1][q];
        if (y.key > best.key || (y.key == best.key && y.col < best.col)) {
          best = y;
          win = q;
        }
      }
      const double* xp = buf + ((j & 1) * kPCS + win) * mp + lane;
      for (int t = 0; t < nt; ++t) Vb[j * mp + lane + 32 * t] = xp[32 * t];
    }
    cl.sync();
  } else {
    // whole rows of the trailing columns, one per warp and two steps; nothing
    // here is shared, so the arrivals need not order it
    constexpr int kSpare = kPW - kPCW - 2;
    int pos = w + rank + kPCS * (wp - kPCW - 2);
    double t[kR];
    auto load = [&] {
      const double* s = Ws + static_cast<size_t>(c0 + src_of[pos]) * n;
#pragma unroll
      for (int u = 0; u < kR; ++u) t[u] = (lane + 32 * u < n) ? s[lane + 32 * u] : 0.0;
    };
    auto store = [&] {
      double* d = Wd + static_cast<size_t>(c0 + pos) * n;
#pragma unroll
      for (int u = 0; u < kR; ++u)
        if (lane + 32 * u < n) d[lane + 32 * u] = t[u];
      pos += kPCS * kSpare;
    };
    for (int j = 0; j <= w; ++j) {  // the w steps and the last barrier
      if (pos < m) {
        if (j & 1)
          store();
        else if (j < w)
          load();
      }
      asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    while (pos < m) {
      load();
      store();
    }
  }
  __syncthreads();
  // 3. V scaled; Y = T^T V^T
  for (int q = wp; q < w; q += kPW) {
    const double vj = vjs[q];
    const int e = qb_exp(vj);
    for (int r = lane; r < mp; r += 32)
      Vb[q * mp + r] = (r < q) ? 0.0 : qb_shift(r == q ? vj : Vb[q * mp + r], e);
  }
  __syncthreads();
  for (int g = rank; g < nt; g += kPCS) {
    // a warp takes the columns i and 31 - i: 33 terms each
    const int r = 32 * g + lane;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = h ? kNB - 1 - wp : wp;
      if (q < w) {
        double y0 = 0.0, y1 = 0.0;
        int s = 0;
        for (; s + 1 <= q; s += 2) {
          y0 = fma(T[s][q], Vb[s * mp + r], y0);
          y1 = fma(T[s + 1][q], Vb[(s + 1) * mp + r], y1);
        }
        if (s == q) y0 = fma(T[s][q], Vb[s * mp + r], y0);
        if (r < m) {
          Yt[static_cast<size_t>(c0 + q) * n + c0 + r] = y0 + y1;
          Vt[static_cast<size_t>(c0 + q) * n + c0 + r] = Vb[q * mp + r];
        }
      }
    }
  }
  // 4. panel rows of this CTA's columns
  if (wp < kPCW && cid < w) {
    const int q = step;
    double* d = Wd + static_cast<size_t>(c0 + q) * n;
    const double* s = Ws + static_cast<size_t>(c0 + src_of[cid]) * n;
    const double up = big ? kQsUp : 1.0;
    if (lane <= q) d[c0 + lane] = ((lane == q) ? betas[q] : x[0]) * up;
    for (int r = lane; r < c0; r += 32) d[r] = s[r];  // entries above the panel
    if (lane == 0) {
      perm[c0 + q] = pold[src_of[cid]];
      double dd = absd(betas[q]) * up;
      if (!(dd > 0.0) || !isfinite(dd)) {
        atomicExch(status, dd > 0.0 ? kDevNonFinite : kDevSingular);
        if (!(dd > 0.0)) dd = DBL_MIN;
      }
      D[c0 + q] = dd;
    }
  }
}

// Rtil[i][perm[c']] = R[i][c'] / D[i]: R[i][c'] = W[c'][i] for c' >= i (the
// diagonal holding beta_i), 0 below the diagonal, with W the buffer the panel
// of c' wrote (WA for even panels, WB for odd ones).
__global__ void __launch_bounds__(256) k_qrb_finalize(const double* WAall, const double* WBall,
                                                     long long sW, const int* permall,
                                                     const double* Dall, long long sD,
                                                     double* Rall, long long sR, int n) {
  const int b = blockIdx.y;
  const double* WA = WAall + b * sW;
  const double* WB = WBall + b * sW;
  const int* perm = permall + static_cast<long long>(b) * n;
  const double* D = Dall + b * sD;
  double* Rt = Rall + b * sR;
  __shared__ double tile[32][33];
  const int tiles = (n + 31) / 32;
  const int ti = blockIdx.x / tiles, tc = blockIdx.x - ti * tiles;  // rows i, columns c'
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;           // 32 x 8
  for (int k = ty; k < 32; k += 8) {  // read W[c'][i], i fastest
    const int cp = tc * 32 + k, i = ti * 32 + tx;
    const double* W = ((cp / kNB) & 1) ? WB : WA;
    tile[k][tx] = (cp < n && i < n) ? W[static_cast<size_t>(cp) * n + i] : 0.0;
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    const int i = ti * 32 + k, cp = tc * 32 + tx;
    if (i < n && cp < n) {
      const double v = (cp >= i) ? tile[tx][k] / D[i] : 0.0;
      Rt[static_cast<size_t>(i) * n + perm[cp]] = v;
    }
  }
}

// One tensor-core product of the blocked QR (no scales).
OzProduct qb_prod(int M, int Nc, int K, const double* A, long long sA, long long a_sv,
                  long long a_sk, const double* B, long long sB, long long b_sv, long long b_sk,
                  double* C, long long sC, int ldc, double alpha, double beta) {
  OzProduct p{};
  p.M = M; p.Nc = Nc; p.K = K;
  p.A = A; p.sA = sA; p.a_sv = a_sv; p.a_sk = a_sk;
  p.B = B; p.sB = sB; p.b_sv = b_sv; p.b_sk = b_sk;
  p.C = C; p.sC = sC; p.ldc = ldc;
  p.alpha = alpha; p.beta = beta;
  return p;
}

}  // namespace

int qr_blocked_launches(int n, int batch, int oz_batch) {
  int sum = 2;  // identity and finalize
  for (int c0 = 0; c0 < n; c0 += kNB) {
    const int w = std::min(kNB, n - c0), m = n - c0, nt = m - w;
    auto products = [&](int M, int Nc, int K) {
      return ozaki_product_launches(M, Nc, K, false, batch, oz_batch);
    };
    // the panel; its trailing columns, of which the last one has none; Q
    sum += 1 + (nt > 0 ? products(nt, w, m) + products(nt, m, w) : 0) + products(m, w, m) + products(m, m, w);
  }
  return sum;
}

// Dynamic shared memory of a panel of w columns, m rows.
static size_t qb_panel_smem(int w, int m) {
  return static_cast<size_t>(w + 2 * kPCS) * ((m + 31) / 32 * 32) * sizeof(double);
}

cudaError_t launch_qr_blocked(double* Xt, long long sX, double* Qt, long long sQ, double* D,
                              long long sD, double* Rtil, long long sR, const QrbWork& wk, int n,
                              int batch, void* oz, int oz_batch, int* status, cudaStream_t st,
                              bool split_rows) {
  if (n <= 0 || batch <= 0 || n > kMaxN) return n > kMaxN ? cudaErrorInvalidValue : cudaSuccess;
  double* WA = wk.W0;
  double* WB = wk.W1;
  const long long sW = wk.sW;
  double* Vt = Rtil;  // Householder vectors, row c0 + q = v_q
  double* Yt = Xt;    // Y = T^T V^T of every panel
  double* Wt = wk.Wt;
  const long long sWt = wk.sWt;
  const int smem = static_cast<int>(qb_panel_smem(kNB, n));
  cudaError_t e = cudaFuncSetAttribute(k_qrb_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  for (int c0 = 0, p = 0; c0 < n; c0 += kNB, ++p) {
    const int w = std::min(kNB, n - c0), m = n - c0, nt = n - c0 - w;
    const double* src = (p == 0) ? Xt : ((p & 1) ? WA : WB);
    const long long sSrc = (p == 0) ? sX : sW;
    double* dst = (p & 1) ? WB : WA;
    if (split_rows) {
      e = launch_qr_panel2(src, sSrc, dst, sW, wk.perm, Vt, sR, Yt, sX, D, sD, n, c0, w, batch,
                           status, st);
    } else {  // one cluster per matrix
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(kPCS * batch, 1, 1);
      cfg.blockDim = dim3(kPT, 1, 1);
      cfg.dynamicSmemBytes = qb_panel_smem(w, m);
      cfg.stream = st;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = kPCS;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      e = cudaLaunchKernelEx(&cfg, k_qrb_panel, src, sSrc, dst, sW, wk.perm, Vt, sR, Yt, sX, D, sD,
                             n, c0, w, status);
    }
    if (e != cudaSuccess) return e;
    if (nt == 0) continue;
    const long long off_trail = static_cast<long long>(c0 + w) * n + c0;
    const long long off_p = static_cast<long long>(c0) * n + c0;
    // W^T = A_rows Y^T: A_rows = trailing rows of dst from column c0
    OzProduct p1 = qb_prod(nt, w, m, dst + off_trail, sW, n, 1, Yt + off_p, sX, n, 1, Wt, sWt, w,
                           1.0, 0.0);
    e = launch_ozaki_product(p1, batch, oz, oz_batch, status, st);
    if (e != cudaSuccess) return e;
    // A_rows -= W^T V^T
    OzProduct p2 = qb_prod(nt, m, w, Wt, sWt, w, 1, Vt + off_p, sR, 1, n, dst + off_trail, sW, n,
                           -1.0, 1.0);
    e = launch_ozaki_product(p2, batch, oz, oz_batch, status, st);
    if (e != cudaSuccess) return e;
  }
  e = launch_set_identity(Qt, sQ, nullptr, 0, n, batch, st);
  if (e != cudaSuccess) return e;
  const int last = ((n - 1) / kNB) * kNB;
  for (int c0 = last; c0 >= 0; c0 -= kNB) {
    const int w = std::min(kNB, n - c0), m = n - c0;
    const long long off_p = static_cast<long long>(c0) * n + c0;
    // W^T = Qt_rows V (rows c0.. of Q^T, columns c0..)
    OzProduct p3 = qb_prod(m, w, m, Qt + off_p, sQ, n, 1, Vt + off_p, sR, n, 1, Wt, sWt, w, 1.0,
                           0.0);
    e = launch_ozaki_product(p3, batch, oz, oz_batch, status, st);
    if (e != cudaSuccess) return e;
    // Qt_rows -= W^T Y
    OzProduct p4 = qb_prod(m, m, w, Wt, sWt, w, 1, Yt + off_p, sX, 1, n, Qt + off_p, sQ, n, -1.0,
                           1.0);
    e = launch_ozaki_product(p4, batch, oz, oz_batch, status, st);
    if (e != cudaSuccess) return e;
  }
  const int tiles = (n + 31) / 32;
  k_qrb_finalize<<<dim3(tiles * tiles, batch), 256, 0, st>>>(WA, WB, sW, wk.perm, D, sD, Rtil, sR,
                                                             n);
  return cudaGetLastError();
}

}  // namespace dqmc
