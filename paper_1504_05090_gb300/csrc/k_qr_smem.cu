// Householder QR with column pivoting for the UDV stack of Eq. (3) (Sec. 2),
// the matrix kept in shared memory from the first step to the last.
//
// Input and output as k_qrp_cluster (k_cluster.cu): X^T stored row-major
// (row c = column c of X) in; Q^T, D = |diag R| and Rtil = D^{-1} R P^T out.
// One cluster of CS CTAs per matrix (CS = 1: no cluster), CTA `rank` owning
// the columns c = rank + CS i.
//
// What bounds it: the FP64 pipe.  On GB300 one FP64 warp instruction occupies
// its SM quarter for 64 to 76 clocks, whatever its latency would be, so the
// kernel is laid out for the fewest FP64 instructions: four lanes per column,
// rows interleaved over them, so that a warp works on eight columns at once, a
// dot product ends with two additions and finished rows drop out four at a
// time; reflectors are left unscaled; and everything that is not a
// multiply-add of the factorisation runs beside it, the pivot search on
// integer keys and the reflector's scalars in one warp that has an SM quarter
// to itself meanwhile (a second warp there would double its serial chain).
//
// Reflector of x_p at step j: s = |x_p[j..)|, v = x_p[j..) with v[j] =
// sign(x_p[j]) u, u = |x_p[j]| + s; H = I - kap v v^T, kap = 1 / (s u); beta =
// -sign(x_p[j]) s.
//
// One step j, its pivot column x_p and sigma = sum_{r>j} x_p[r]^2 at hand:
//   1. d_s = sum_{r>j} x_p[r] x_s[r] of the live columns, eight per warp; one
//      warp forms the reflector's scalars beside it.
//   2. c_s = kap (v[j] x_s[j] + d_s), R_js = x_s[j] - c_s v[j], and the
//      squared norm downdated by R_js^2.
//   3. x_s[r] -= c_s x_p[r], r > j.  Beside it one warp already prepares step
//      j + 1: it takes the column of the largest norm (high word of the FP64
//      number as an integer key), updates it and forms its sigma.
//      CS > 1: every CTA does so for the best of its own columns and sends the
//      result to all CTAs (distributed shared memory, buffered by step
//      parity); after the step's one cluster barrier all take the same winner.
//      A norm that lost half of its digits since it was last summed (LAPACK's
//      xLAQP2 criterion, squared norm below 2^-26 of then) is summed afresh in
//      the update, for the step after the next; below 2^-40 the downdated
//      value would be too rough to choose by, and the next pivot waits.
// Q = H_0 ... H_{n-1} is accumulated backwards, the columns in registers, a
// group of them per warp, without a barrier.
#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>

#include "common.cuh"
#include "kernels.h"
#include "qr_scalars.cuh"

namespace cg = cooperative_groups;

namespace dqmc {
namespace {

constexpr int kQT = 256;  // threads per CTA

// Row length of a column in shared memory: a multiple of 4, odd in units of
// four doubles, so that the four columns a half warp reads lie in different
// banks.
__host__ __device__ __forceinline__ int qs_ld(int n) {
  const int p = (n + 3) & ~3;
  return (p & 4) ? p : p + 4;
}
__host__ __device__ __forceinline__ int qs_cols(int n, int cs) { return (n + cs - 1) / cs; }

size_t qs_smem(int n, int cs) {
  const size_t ld = qs_ld(n);
  return (qs_cols(n, cs) * ld + (cs > 1 ? 2 * cs * ld : 0)) * sizeof(double);
}

// Sum over the kL lanes of a column.
template <int kL>
__device__ __forceinline__ double qs_lsum(double a) {
#pragma unroll
  for (int o = kL / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
  return a;
}

// A CTA's best column for a step: sigma, the high word of its squared norm (the
// pivot key) and the column (kMaxN: no live column).
struct Cand {
  double sigma;
  unsigned key;
  int col;
};

// n <= kL kSlots: lanes per column and rows per lane in the accumulation of Q.
template <int CS, int kL, int kSlots>
__global__ void __launch_bounds__(kQT, 2) k_qr_smem(double* Xall, long long sX, double* Qall,
                                                long long sQ, double* Dall, long long sD,
                                                double* Rall, long long sR, int n, int* status) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (CS > 1) ? static_cast<int>(cl.block_rank()) : 0;
  const int b = blockIdx.x / CS;
  double* Xg = Xall + b * sX;
  double* Qt = Qall + b * sQ;
  double* D = Dall + b * sD;
  double* Rt = Rall + b * sR;
  const int ld = qs_ld(n), npad = (n + 3) & ~3, nslots = npad >> 2;  // slots of four rows
  const int ncol = (n - rank + CS - 1) / CS;  // own columns rank + CS i
  extern __shared__ __align__(16) double qs_sm[];
  double* Xs = qs_sm;                           // [ncol][ld]
  double* buf = Xs + qs_cols(n, CS) * ld;       // [2][CS][ld] candidates (CS > 1)
  __shared__ double kaps[kMaxN], betas[kMaxN];
  __shared__ double dsum[kMaxN / CS], cvec[kMaxN / CS], n1[kMaxN / CS], n2[kMaxN / CS];
  __shared__ unsigned key[kMaxN / CS];
  __shared__ unsigned char live[2][kMaxN / CS], rec[kMaxN / CS], colof[kMaxN / CS == kMaxN ? kMaxN : 1];
  __shared__ short stepof[kMaxN / CS];
  __shared__ Cand cand[2][CS];  // by step parity and CTA
  __shared__ int wait_sum[2], stale[2], big_sh;
  __shared__ double kap_sh, vj_sh;
  __shared__ double vjs[CS == 1 ? kMaxN : 1];  // v_j[j]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int nw = kQT / 32;
  const int l4 = lane & 3, lg = lane >> 2;
  // the warp of the scalars: a different SM quarter for neighbouring CTAs;
  // the other warps of its quarter stand back meanwhile
  const int ws = blockIdx.x & 3, wv = (ws + 1) & 3;
  const bool helper = ((w - ws) & 3) != 0;               // of another quarter,
  const int wu = (w >> 2) * 3 + ((w - ws + 3) & 3);      // its rank among them
  constexpr int nu = nw / 4 * 3;                         // and their number

  for (int e = tid; e < ncol * ld; e += kQT) {
    const int c = e / ld, r = e - c * ld;
    Xs[e] = (r < n) ? Xg[static_cast<size_t>(rank + CS * c) * n + r] : 0.0;
  }
  for (int i = tid; i < ncol; i += kQT) {
    live[0][i] = static_cast<unsigned char>(i);
    stepof[i] = static_cast<short>(n);
  }
  if (tid < 2) {
    wait_sum[tid] = 0;
    stale[tid] = -1;
    big_sh = 0;
  }
  __syncthreads();
  for (int g = w; 8 * g < ncol; g += nw) {
    const int c = 8 * g + lg;
    const double* x = Xs + min(c, ncol - 1) * ld + l4;
    double a = 0.0;
    for (int t = 0; t < nslots; ++t) a = fma(x[4 * t], x[4 * t], a);
    a = qs_lsum<4>(a);
    if (l4 == 0 && c < ncol) {
      n1[c] = n2[c] = a;
      key[c] = static_cast<unsigned>(__double2hiint(a));
    }
  }
  __syncthreads();
  if constexpr (CS > 1) cl.sync();  // the peers run: their shared memory may be written
  {  // columns too large for the sums to come: see kQsBig
    int big = 0;
    for (int i = tid; i < ncol; i += kQT) big |= key[i] >= kQsBig && key[i] < kQsNonFinite;
    big = __syncthreads_or(big);
    if (CS == 1) {
      if (tid == 0) big_sh = big;
    } else {
      if (big && tid < CS) *cl.map_shared_rank(&big_sh, tid) = 1;
      cl.sync();
      big = big_sh;
    }
    if (big) {
      for (int e = tid; e < ncol * ld; e += kQT) Xs[e] *= kQsDown;
      for (int i = tid; i < ncol; i += kQT) {
        n1[i] = n2[i] = n1[i] * (kQsDown * kQsDown);
        key[i] = static_cast<unsigned>(__double2hiint(n1[i]));
      }
      __syncthreads();
    }
  }

  // Warp ws: own column lp (-1: none) brought to step j (upd: with the factor
  // of step j - 1 and its column xq), its sigma and, for CS > 1, both to every
  // CTA.
  auto prepare = [&](int j, int lp, const double* xq, bool upd) {
    Cand cd{0.0, 0u, kMaxN};
    if (lp >= 0) {
      double* x = Xs + lp * ld;
      const double f = upd ? -cvec[lp] : 0.0;
      double sg = 0.0, xr[kMaxN / 32];
#pragma unroll
      for (int t = 0; t < kMaxN / 32; ++t) {
        const int r = lane + 32 * t;
        xr[t] = 0.0;
        if (r >= j && r < n) {
          xr[t] = x[r];
          if (upd) x[r] = xr[t] = fma(f, xq[r], xr[t]);
          if (r > j) sg = fma(xr[t], xr[t], sg);
        }
      }
      if constexpr (CS > 1) {
#pragma unroll
        for (int t = 0; t < kMaxN / 32; ++t) {
          const int r = lane + 32 * t;
          if (r >= j && r < npad)
#pragma unroll
            for (int q = 0; q < CS; ++q)
              *cl.map_shared_rank(buf + ((j & 1) * CS + rank) * ld + r, q) = xr[t];
        }
      }
      cd.sigma = qs_warp_sum_pos(sg);
      cd.key = key[lp];
      cd.col = rank + CS * lp;
    }
    if (lane < CS) {
      Cand* dst = &cand[j & 1][rank];
      if constexpr (CS > 1) dst = cl.map_shared_rank(dst, lane);
      *dst = cd;
    }
  };
  // The live column of largest key, the first one among equals (so that the
  // choice does not depend on CS); -1 if there is none.
  auto best = [&](const unsigned char* lv, int m, int skip) {
    unsigned kb = 0, cb = kMaxN;
    for (int i = lane; i < m; i += 32) {
      const int c = lv[i];
      if (c != skip) {
        const unsigned k = key[c];
        if (cb == kMaxN || k > kb || (k == kb && c < static_cast<int>(cb))) {
          kb = k;
          cb = c;
        }
      }
    }
    const unsigned km = __reduce_max_sync(0xFFFFFFFFu, kb);
    const unsigned cm = __reduce_min_sync(0xFFFFFFFFu, kb == km ? cb : static_cast<unsigned>(kMaxN));
    return cm < kMaxN ? static_cast<int>(cm) : -1;
  };

  int m = ncol;      // live columns
  if (w == ws) prepare(0, best(live[0], m, -1), nullptr, false);
  for (int j = 0; j < n; ++j) {
    if constexpr (CS > 1)
      cl.sync();
    else
      __syncthreads();
    const unsigned char* lv = live[j & 1];
    int win = 0;
#pragma unroll
    for (int q = 1; q < CS; ++q) {
      const Cand& x = cand[j & 1][q];
      const Cand& y = cand[j & 1][win];
      if (x.col < kMaxN && (y.col == kMaxN || x.key > y.key || (x.key == y.key && x.col < y.col))) win = q;
    }
    const int pcol = cand[j & 1][win].col;                    // the pivot column
    const int lp = (win == rank) ? (pcol - rank) / CS : -1;  // its local index, if own
    const double* xp = (CS > 1) ? buf + ((j & 1) * CS + win) * ld : Xs + pcol * ld;
    const int t0 = (j + 1) >> 2;
    // 1. scalars beside the dot products
    if (w == ws) {
      double beta, kap, vj;
      qs_reflector(xp[j], cand[j & 1][win].sigma, beta, kap, vj);
      if (lane == 0) {
        kap_sh = kaps[j] = kap;
        vj_sh = vj;
        betas[j] = beta;
        if constexpr (CS == 1) vjs[j] = vj;
        wait_sum[(j + 1) & 1] = 0;
        if ((cand[j & 1][win].key & 0x7FFFFFFFu) >= 0x7FF00000u) atomicExch(status, kDevNonFinite);
      }
    } else if (helper) {
      for (int g = wu; 8 * g < m; g += nu) {
        const int i = 8 * g + lg, c = lv[min(i, m - 1)];
        const double* x = Xs + c * ld + l4;
        const double* v = xp + l4;
        double a = 0.0;
        if (t0 < nslots) a = (4 * t0 + l4 > j) ? x[4 * t0] * v[4 * t0] : 0.0;
#pragma unroll 4
        for (int t = t0 + 1; t < nslots; ++t) a = fma(x[4 * t], v[4 * t], a);
        a = qs_lsum<4>(a);
        if (l4 == 0 && i < m) dsum[c] = a;
      }
      if constexpr (CS > 1) {
        // the sum that the own candidate missed (below), if it lost
        const int c = stale[j & 1];
        if (c >= 0 && c != lp && wu == ((m + 7) >> 3) % nu) {
          const double* x = Xs + c * ld + l4;
          const int t1 = j >> 2;
          double a = (4 * t1 + l4 >= j) ? x[4 * t1] * x[4 * t1] : 0.0;
#pragma unroll 4
          for (int t = t1 + 1; t < nslots; ++t) a = fma(x[4 * t], x[4 * t], a);
          a = qs_lsum<4>(a);
          if (lane == 0) n1[c] = n2[c] = a;
        }
      }
    }
    __syncthreads();
    // 2. factors of the live columns
    const double kap = kap_sh, vj = vj_sh;
    for (int i = tid; i < m; i += kQT) {
      const int c = lv[i];
      if (c == lp) continue;
      const double xj = Xs[c * ld + j];
      const double cs = kap * fma(vj, xj, dsum[c]);
      const double rj = fma(-cs, vj, xj);
      Xs[c * ld + j] = rj;
      cvec[c] = cs;
      double nn = fma(-rj, rj, n1[c]);
      if (__double2hiint(nn) < 0) nn = 0.0;
      n1[c] = nn;
      // 2^-26 = sqrt(DBL_EPSILON); compared on the high words
      const int hn = __double2hiint(nn), hr = __double2hiint(n2[c]);
      const int rc = (hn > hr - (26 << 20)) ? 0 : (hn > hr - (40 << 20)) ? 1 : 2;
      rec[c] = static_cast<unsigned char>(rc);
      if (rc == 2) wait_sum[j & 1] = 1;
      key[c] = static_cast<unsigned>(__double2hiint(nn));
    }
    __syncthreads();
    // 3. update and, unless a norm has to be summed first, the next pivot
    const bool ahead = wait_sum[j & 1] == 0;
    const int ml = (lp >= 0) ? m - 1 : m;  // own live columns after this step
    const int np = ahead ? best(lv, m, lp) : -1;
    if (ahead && w == ws) {
      if (j + 1 < n) prepare(j + 1, np, xp, true);
      // a candidate that loses to another CTA's stays live and needs its norm
      // summed afresh like the other columns (as with CS = 1); the next step
      // does so beside its dot products
      if (CS > 1 && lane == 0) stale[(j + 1) & 1] = (np >= 0 && rec[np]) ? np : -1;
    } else if (!ahead || helper) {
      const int wi = ahead ? wu : w, wn = ahead ? nu : nw;
      for (int g = wi; 8 * g < m; g += wn) {
        const int i = 8 * g + lg, c = lv[min(i, m - 1)];
        const bool ok = i < m && c != lp && c != np;
        double* x = Xs + c * ld + l4;
        const double* v = xp + l4;
        if (ok) {
          const double f = -cvec[c];
          if (t0 < nslots && 4 * t0 + l4 > j) x[4 * t0] = fma(f, v[4 * t0], x[4 * t0]);
          int t = t0 + 1;
          for (; t + 4 <= nslots; t += 4) {
            double a[4], u[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              a[q] = x[4 * (t + q)];
              u[q] = v[4 * (t + q)];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) x[4 * (t + q)] = fma(f, u[q], a[q]);
          }
          for (; t < nslots; ++t) x[4 * t] = fma(f, v[4 * t], x[4 * t]);
        }
        const bool rs = ok && rec[c];
        if (__any_sync(0xFFFFFFFFu, rs)) {
          double a = 0.0;
          for (int t = t0; t < nslots; ++t)
            if (4 * t + l4 > j) a = fma(x[4 * t], x[4 * t], a);
          a = qs_lsum<4>(a);
          if (rs && l4 == 0) {
            n1[c] = n2[c] = a;
            // a key that is still good enough stays until the next step: the
            // choice is then the same whether or not this CTA waits
            if (rec[c] == 2) key[c] = static_cast<unsigned>(__double2hiint(a));
          }
        }
      }
    }
    if (w == wv) {  // the live list without the pivot
      int at = m;
      for (int i = lane; i < m; i += 32)
        if (lv[i] == lp) at = i;
      at = static_cast<int>(__reduce_min_sync(0xFFFFFFFFu, static_cast<unsigned>(at)));
      for (int i = lane; i < ml; i += 32) live[(j + 1) & 1][i] = (i == at) ? lv[m - 1] : lv[i];
      if (lp >= 0) {
        if (lane == 0) {
          stepof[lp] = static_cast<short>(j);
          if constexpr (CS == 1) colof[j] = static_cast<unsigned char>(lp);
        }
        if (CS > 1)  // v_j to global memory (the input X is on chip)
          for (int r = j + lane; r < n; r += 32)
            __stcg(Xg + static_cast<size_t>(j) * n + r, (r == j) ? vj : xp[r]);
      }
    }
    if (!ahead) {
      __syncthreads();
      if (w == ws && j + 1 < n) {
        prepare(j + 1, best(lv, m, lp), nullptr, false);
        if (CS > 1 && lane == 0) stale[(j + 1) & 1] = -1;
      }
    }
    m = ml;
  }
  __syncthreads();
  if constexpr (CS > 1) cl.sync();  // every v_j is in global memory

  // Q: 32 / kL columns per warp; column c takes the reflectors j <= c, so the
  // work of a group grows with its columns: pairs of warps that share an SM
  // quarter (w, w + 4) take groups from both ends.
  constexpr int kG = 32 / kL;
  const int lq = lane & (kL - 1), lc0 = lane / kL;
  const int ngrp = (n + kG - 1) / kG, nwt = CS * nw;
  for (int base = 0; base < ngrp; base += nwt) {
    const int span = min(nwt, ngrp - base), half = (span + 1) >> 1;
    // position of this warp: quarter-major over the CTAs, first halves first
    const int a0 = (w >> 2) * (nwt >> 1) + (w & 3) * CS + rank;
    int g = -1;
    if (w < 4) {
      if (a0 < half) g = base + a0;
    } else {
      const int k = a0 - (nwt >> 1);
      if (k < span - half) g = base + span - 1 - k;
    }
    if (g < 0) continue;
    const int c = kG * g + lc0;
    double q[kSlots];
#pragma unroll
    for (int t = 0; t < kSlots; ++t) q[t] = (kL * t + lq == c) ? 1.0 : 0.0;
    // reflectors in blocks of kL, so that the rows a block leaves out are
    // known at compile time; CS > 1 loads the next one from L2 ahead
    const int jtop = min(kG * g + kG - 1, n - 1);
    double vn[CS > 1 ? kSlots : 1];
    if constexpr (CS > 1) {
#pragma unroll
      for (int t = 0; t < kSlots; ++t) {
        const int r = kL * t + lq;
        vn[t] = (r < n && r >= jtop) ? __ldcg(Xg + static_cast<size_t>(jtop) * n + r) : 0.0;
      }
    }
#pragma unroll
    for (int tj = kSlots - 1; tj >= 0; --tj) {
      for (int j = min(jtop, kL * tj + kL - 1); j >= kL * tj; --j) {
        const double kap = kaps[j];
        double v[kSlots], a = 0.0;
        if constexpr (CS > 1) {
          const int jn = max(j - 1, 0);
          const double* vg = Xg + static_cast<size_t>(jn) * n;
#pragma unroll
          for (int t = tj; t < kSlots; ++t) v[t] = vn[t];
#pragma unroll
          for (int t = (tj > 0 ? tj - 1 : 0); t < kSlots; ++t) {
            const int r = kL * t + lq;
            vn[t] = (r < n && (t > tj || r >= jn)) ? __ldcg(vg + r) : 0.0;
          }
        } else {
          const double* vg = Xs + colof[CS == 1 ? j : 0] * ld;
#pragma unroll
          for (int t = tj; t < kSlots; ++t) {
            const int r = kL * t + lq;
            double x = (r < n) ? vg[r] : 0.0;
            if (t == tj && r <= j) x = (r == j) ? vjs[CS == 1 ? j : 0] : 0.0;
            v[t] = x;
          }
        }
#pragma unroll
        for (int t = tj; t < kSlots; ++t) a = fma(v[t], q[t], a);
        a = -kap * qs_lsum<kL>(a);
#pragma unroll
        for (int t = tj; t < kSlots; ++t) q[t] = fma(a, v[t], q[t]);
      }
    }
#pragma unroll
    for (int t = 0; t < kSlots; ++t) {
      const int r = kL * t + lq;
      if (c < n && r < n) Qt[static_cast<size_t>(c) * n + r] = q[t];
    }
  }
  // D = |beta| and Rtil[i][c] = R[i][s] / D[i] with s the step of column c
  double* rd = kaps;
  __syncthreads();  // the last use of kaps
  for (int i = tid; i < n; i += kQT) {
    double d = absd(betas[i]);
    if (!(d > 0.0)) {
      atomicExch(status, kDevSingular);
      d = DBL_MIN;
    }
    if (rank == 0) D[i] = big_sh ? d * kQsUp : d;
    rd[i] = 1.0 / d;
  }
  __syncthreads();
  for (int e = tid; e < n * ncol; e += kQT) {
    const int i = e / ncol, lc = e - i * ncol, s = stepof[lc];
    double v = 0.0;
    if (s > i)
      v = Xs[lc * ld + i] * rd[i];
    else if (s == i)
      v = betas[i] * rd[i];
    Rt[static_cast<size_t>(i) * n + rank + CS * lc] = v;
  }
}

template <int CS, int kL, int kSlots>
cudaError_t qs_launch(double* Xt, long long sX, double* Qt, long long sQ, double* D, long long sD,
                      double* Rt, long long sR, int n, int batch, int* status, cudaStream_t st) {
  const size_t sm = qs_smem(n, CS);
  cudaError_t e = cudaFuncSetAttribute(k_qr_smem<CS, kL, kSlots>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CS * batch, 1, 1);
  cfg.blockDim = dim3(kQT, 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CS > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_qr_smem<CS, kL, kSlots>, Xt, sX, Qt, sQ, D, sD, Rt, sR, n, status);
}

}  // namespace

// CTAs per matrix of k_qr_smem, or 0 where another kernel takes the matrix.
// The choice of kernel depends on n and the group's interval alone (qr_ctas in
// dqmc.cu), so that a chain's numbers do not depend on how many chains share its
// context (the result does not depend on the CTAs either).  Measured (us for the
// batch, GB300): this kernel against the blocked QR (the default mode's
// alternative from n = 64 on) and the column-pivoted QR on global memory
// (k_qrp_cluster):
//   n = 16:  32 matrices 45 / - / 124; 256: 46 / - / 463
//   n = 36:  32: 106 / - / 278;       256: 127 / - / 1083
//   n = 64:  32: 258 / 580 / 531;     256: 353 / 1987 / 2076; 1024: 1257 / 6884 / 7369
//   n = 100: 32: 446 (4 CTAs; 707 with one) / 1093; 64: 530 (707) / 1101; 256: 1067 (1) / 3743
//   n = 144: 8: 773 (8 CTAs; 906 with 4, 1677 with one) / 1557; 32: 905 (4) / 1596;
//            64: 1128 (4) / 1647; 256: 3347 (1) / 5743
// From n = 145 on the matrix no longer fits one CTA's shared memory, and with
// four CTAs per matrix a batch that fills the chip was slower than the blocked
// QR, whose trailing updates run on the tensor cores (n = 196, 64 matrices:
// 3184 / 2652; n = 256: 6287 / 3494).
// One CTA per matrix keeps the most matrices in flight and is always right up
// to n = 64, where the FP64 work of a step does not outweigh a cluster
// barrier; above, a matrix is spread over 4 or 8 CTAs while all the chains of
// the context (`chains`, their groups run side by side) leave SMs idle: the
// chip holds 72 clusters of four CTAs (two per SM) and 15 of eight with an SM
// per CTA.
int qr_smem_ctas(int n, int chains, int nsm) {
  if (n <= 64) return 1;
  if (n > 144) return 0;
  return (n > 128 && chains <= nsm / 10) ? 8 : (chains <= nsm * 9 / 19 ? 4 : 1);
}

cudaError_t launch_qr_smem(int cs, double* Xt, long long sX, double* Qt, long long sQ, double* D,
                           long long sD, double* Rt, long long sR, int n, int batch, int* status,
                           cudaStream_t st) {
#define QS_CASE(CS, kL, kSlots) \
  return qs_launch<CS, kL, kSlots>(Xt, sX, Qt, sQ, D, sD, Rt, sR, n, batch, status, st)
  if (n <= 0 || batch <= 0) return cudaSuccess;
  if (cs == 1) {
    if (n <= 16) QS_CASE(1, 4, 4);
    if (n <= 36) QS_CASE(1, 4, 9);
    if (n <= 64) QS_CASE(1, 4, 16);
    if (n <= 104) QS_CASE(1, 8, 13);
    if (n <= 144) QS_CASE(1, 8, 18);
  } else if (cs == 4) {
    if (n <= 104) QS_CASE(4, 8, 13);
    if (n <= 144) QS_CASE(4, 8, 18);
  } else if (cs == 8) {
    if (n <= 144) QS_CASE(8, 8, 18);
  }
#undef QS_CASE
  return cudaErrorInvalidValue;
}

}  // namespace dqmc
