// Gauss-Jordan inverse with the matrix in shared memory (the stabilised Green
// functions behind Eq. (3) and G_ij(tau_l), Sec. 2).
//
// As k_gj_cluster (k_cluster.cu): partial pivoting over the rows not yet used,
// no row is moved; with pr[k] the pivot row of step k and ip its inverse
// permutation, the in-place result Z gives A^{-1}[k][j] = Z[pr[k]][ip[j]].
// One cluster of CS CTAs per matrix (CS = 1: no cluster), rows i = rank + CS li
// owned by CTA `rank`.  T = double, or df32 (float pairs; A stays FP64 in
// memory and is split on load).
//
// What bounds it: the FP64 pipe (one warp instruction per 64 to 76 clocks and
// SM quarter), or for float pairs the FP32 pipe and shared-memory bandwidth
// about equally.  A warp works on eight rows at a time, four lanes per row and
// columns interleaved over them, so that a ragged size wastes at most three
// columns and seven rows.
//
// Step k, the pivot row p, 1 / A[p][k] and column k (fcol) at hand:
//   1. prow = A[p][.] / A[p][k] (1 / A[p][k] at k), also into row p itself.
//   2. rows i != p: A[i][j] -= fcol[i] prow[j]; column k, zeroed when it was
//      copied to fcol, becomes -fcol[i] / A[p][k].  Column k + 1 is left out:
//      beside the update one warp forms its new values into the next fcol,
//      takes the largest of the unused rows as the next pivot (integer keys)
//      and its reciprocal.
//   CS > 1: every CTA then sends its candidate row to all CTAs (distributed
//   shared memory, buffered by step parity); one cluster barrier per step.
#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>

#include "common.cuh"
#include "gj_key.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace dqmc {
namespace {

constexpr int kGT = 256;  // threads per CTA

// Row length in shared memory: a multiple of 4, odd in units of four elements
// (the four rows that a half warp reads lie in different banks).
__host__ __device__ __forceinline__ int gs_ld(int n) {
  const int p = (n + 3) & ~3;
  return (p & 4) ? p : p + 4;
}

size_t gs_smem(int n, int cs) {
  const size_t ld = gs_ld(n);
  return (static_cast<size_t>((n + cs - 1) / cs) * ld + ld + (cs > 1 ? 2 * cs * ld : 0)) * 8;
}

// Pivot keys: the bits of |x| (rounded to FP32 for FP64, as k_gj_cluster
// compares it) order as the numbers.
__device__ __forceinline__ unsigned gs_key(double x) {
  bool ok;
  const unsigned k = gj_key_bits(static_cast<uint64_t>(__double_as_longlong(x)), ok);
  return ok ? k : static_cast<unsigned>(__float_as_int(static_cast<float>(absd(x))));
}
__device__ __forceinline__ unsigned gs_key(df32 x) {
  return static_cast<unsigned>(__float_as_int(x.hi)) & 0x7FFFFFFFu;
}
// Inf or NaN as the pivot (FP64: finite numbers beyond FP32's range are not)
__device__ __forceinline__ bool gs_bad(double piv, unsigned) {
  return (static_cast<unsigned>(__double2hiint(piv)) & 0x7FFFFFFFu) >= 0x7FF00000u;
}
__device__ __forceinline__ bool gs_bad(df32, unsigned key) { return key >= 0x7F800000u; }
__device__ __forceinline__ double gs_d(double x) { return x; }
__device__ __forceinline__ double gs_d(df32 x) { return static_cast<double>(x); }
__device__ __forceinline__ double gs_neg(double x) { return -x; }
__device__ __forceinline__ df32 gs_neg(df32 x) { return -x; }
// a b + c: for float pairs the product's error terms and one TwoSum with c.hi,
// rounded once (relative error about 2^-48).
__device__ __forceinline__ double gs_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ df32 gs_fma(df32 a, df32 b, df32 c) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  const df32 s = df_two_sum(c.hi, p);
  return df_fast_two_sum(s.hi, s.lo + (c.lo + e));
}

// A CTA's best row for the next step: pivot key, row (kMaxN: none), the pivot
// and its reciprocal.
template <typename T>
struct GsCand {
  double piv;
  T inv;
  unsigned key;
  int row;
};

template <int CS, typename T>
__global__ void __launch_bounds__(kGT) k_gj_smem(const double* Aall, long long sA, double* Iall,
                                                long long sI, int n, double* logabs, int* status) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (CS > 1) ? static_cast<int>(cl.block_rank()) : 0;
  const int b = blockIdx.x / CS;
  const double* A = Aall + b * sA;
  double* Ainv = Iall + b * sI;
  const int ld = gs_ld(n), nslots = (n + 3) >> 2;
  const int nrow = (n - rank + CS - 1) / CS;
  extern __shared__ __align__(16) unsigned char gs_sm[];
  T* As = reinterpret_cast<T*>(gs_sm);              // [nrow][ld]
  T* prow = As + ((n + CS - 1) / CS) * ld;          // [ld]
  T* buf = prow + ld;                               // [2][CS][ld] candidate rows (CS > 1)
  __shared__ T fcol[2][kMaxN / CS];                 // column k of the own rows, by parity
  __shared__ unsigned char used[kMaxN / CS];
  __shared__ short ip[kMaxN];                       // step of every row
  __shared__ double pivs[kMaxN];
  __shared__ GsCand<T> cand[2][CS];                 // by step parity and CTA
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int nw = kGT / 32;
  const int l4 = lane & 3, lg = lane >> 2;
  // the warp of the next pivot: a different SM quarter for neighbouring CTAs
  const int ws = blockIdx.x & 3;
  const int wu = (w > ws) ? w - 1 : w;  // rank among the updating warps

  for (int e = tid; e < nrow * ld; e += kGT) {
    const int i = e / ld, j = e - i * ld;
    As[e] = (j < n) ? T(A[static_cast<size_t>(rank + CS * i) * n + j]) : T(0.0);
  }
  for (int i = tid; i < nrow; i += kGT) used[i] = 0;
  __syncthreads();
  if constexpr (CS > 1) cl.sync();  // the peers run: their shared memory may be written

  // Warp ws: column kn with the update of the step before (pivot row p if own,
  // else -1; first: none) into fcol, and the best unused row.
  auto next_pivot = [&](int kn, int p, bool first) {
    T* fc = fcol[kn & 1];
    const T pk = first ? T(0.0) : prow[kn];
    unsigned kb = 0, rb = kMaxN;
    for (int i = lane; i < nrow; i += 32) {
      T x = As[i * ld + kn];
      if (!first) x = (i == p) ? pk : gs_fma(gs_neg(fcol[(kn + 1) & 1][i]), pk, x);
      fc[i] = x;
      As[i * ld + kn] = T(0.0);
      if (!used[i]) {
        const unsigned k = gs_key(x);
        if (rb == kMaxN || k > kb) {
          kb = k;
          rb = i;
        }
      }
    }
    const unsigned km = __reduce_max_sync(0xFFFFFFFFu, rb < kMaxN ? kb : 0u);
    const unsigned rm = __reduce_min_sync(0xFFFFFFFFu, (rb < kMaxN && kb == km) ? rb : static_cast<unsigned>(kMaxN));
    __syncwarp();
    GsCand<T> c;
    c.key = km;
    c.row = kMaxN;
    c.piv = 1.0;
    c.inv = T(1.0);
    if (rm < kMaxN) {
      c.row = rank + CS * static_cast<int>(rm);
      c.piv = gs_d(fc[rm]);
      double piv = c.piv;
      if ((__double_as_longlong(piv) << 1) == 0LL) piv = DBL_MIN;
      c.inv = T(1.0 / piv);
    }
    if (lane < CS) {
      GsCand<T>* dst = &cand[kn & 1][rank];
      if constexpr (CS > 1) dst = cl.map_shared_rank(dst, lane);
      *dst = c;
    }
  };

  if (w == ws) next_pivot(0, -1, true);
  const int nchunk = (nslots + 15) >> 4, csz = (nslots + nchunk - 1) / nchunk;
  const int ngrp = (nrow + 7) >> 3;
  for (int k = 0; k < n; ++k) {
    __syncthreads();
    int win = 0;
    if constexpr (CS > 1) {
      // the own candidate row to every CTA
      const int row = cand[k & 1][rank].row;
      if (row < kMaxN) {
        const T* x = As + (row - rank) / CS * ld;
        for (int j = tid; j < n; j += kGT) {
          const T v = x[j];
#pragma unroll
          for (int q = 0; q < CS; ++q) *cl.map_shared_rank(buf + ((k & 1) * CS + rank) * ld + j, q) = v;
        }
      }
      cl.sync();
#pragma unroll
      for (int q = 1; q < CS; ++q) {
        const GsCand<T>& x = cand[k & 1][q];
        const GsCand<T>& y = cand[k & 1][win];
        if (x.row < kMaxN && (y.row == kMaxN || x.key > y.key || (x.key == y.key && x.row < y.row))) win = q;
      }
    }
    // 1. the scaled pivot row
    const GsCand<T>& c = cand[k & 1][win];
    const T inv = c.inv;
    const int pg = c.row;
    const int p = (win == rank) ? (pg - rank) / CS : -1;  // own row index, or -1
    {
      const T* x = (CS > 1) ? buf + ((k & 1) * CS + win) * ld : As + p * ld;
      for (int j = tid; j < n; j += kGT) {
        const T v = (j == k) ? inv : x[j] * inv;
        prow[j] = v;
        if (p >= 0 && j != k + 1) As[p * ld + j] = v;
      }
    }
    if (tid == 0) {
      ip[pg] = static_cast<short>(k);
      pivs[k] = c.piv;
      if (p >= 0) used[p] = 1;
      if (gs_bad(T(c.piv), c.key)) atomicExch(status, kDevNonFinite);
      if (c.key == 0u && (__double_as_longlong(c.piv) << 1) == 0LL) atomicExch(status, kDevSingular);
    }
    __syncthreads();
    // 2. update and the next pivot
    if (w == ws) {
      if (k + 1 < n) next_pivot(k + 1, p, false);
    } else {
      for (int u = wu; u < ngrp * nchunk; u += nw - 1) {
        const int g = u / nchunk, ch = u - g * nchunk;
        const int i = 8 * g + lg;
        if (i < nrow && i != p) {
          const T f = gs_neg(fcol[k & 1][i]);
          T* x = As + i * ld + l4;
          const T* v = prow + l4;
          const int ta = ch * csz, tb = min(ta + csz, nslots);
          int t = ta;
          for (; t + 4 <= tb; t += 4) {
            T a[4], r[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              a[q] = x[4 * (t + q)];
              r[q] = v[4 * (t + q)];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const T y = gs_fma(f, r[q], a[q]);
              if (4 * (t + q) + l4 != k + 1) x[4 * (t + q)] = y;
            }
          }
          for (; t < tb; ++t) {
            const T y = gs_fma(f, v[4 * t], x[4 * t]);
            if (4 * t + l4 != k + 1) x[4 * t] = y;
          }
        }
      }
    }
  }
  __syncthreads();
  // A^{-1}: row i of Z is row ip[i] of the inverse, its columns permuted
  for (int i = w; i < nrow; i += nw) {
    const T* z = As + i * ld;
    double* out = Ainv + static_cast<size_t>(ip[rank + CS * i]) * n;
    for (int j = lane; j < n; j += 32) out[j] = gs_d(z[ip[j]]);
  }
  if (logabs && rank == 0) {  // log|det| = sum_k log|pivot_k|
    double la = 0.0;
    for (int k = tid; k < n; k += kGT) la += log(absd(pivs[k]));
    for (int o = 16; o > 0; o >>= 1) la += __shfl_xor_sync(0xFFFFFFFFu, la, o);
    __shared__ double lsum[nw];
    if (lane == 0) lsum[w] = la;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int q = 0; q < nw; ++q) t += lsum[q];
      logabs[b] = t;
    }
  }
  if constexpr (CS > 1) cl.sync();
}

template <int CS, typename T>
cudaError_t gs_launch(const double* A, long long sA, double* Ainv, long long sI, int n, int batch,
                      double* logabs, int* status, cudaStream_t st) {
  const size_t sm = gs_smem(n, CS);
  cudaError_t e = cudaFuncSetAttribute(k_gj_smem<CS, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CS * batch, 1, 1);
  cfg.blockDim = dim3(kGT, 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CS > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_gj_smem<CS, T>, A, sA, Ainv, sI, n, logabs, status);
}

}  // namespace

// CTAs per matrix of k_gj_smem for `conc` matrices in flight, or 0 where
// k_gj_cluster (the matrix in global memory, 2 or 4 CTAs) is the better one.
// All of them give the same numbers bit for bit.  Measured (us for the batch,
// GB300; FP64 then float pairs), this kernel against k_gj_cluster:
//   n = 16:  32 matrices 21 / 47;               1024: 49 / 391, 57 / 375
//   n = 64:  32: 129 (4 CTAs; 161 with one) / 227, 116 (4) / 199;
//            1024: 719 (1) / 2840, 367 (1) / 1868
//   n = 100: 32: 281 (4) / 426, 217 (4) / 365;  1024: 2450 (1) / 6230, 1512 (1) / 4428
//   n = 144: 1: 454 (8) / 780; 32: 523 (4) / 788; 1024: 7171 (1) / 12657, 4418 (4) / 8200
//   n = 196: 1: 804 (8) / 1270; 32: 942 (4) / 1288; 256: 5703 (4) / 6480, 3260 (4) / 4667
//   n = 256: 1: 1240 (8) / 1928; 32: 1662 (4) / 1942, 1128 (4) / 1664;
//            64: 3313 (4) / 3037, 2246 (4) / 2248; 256: 13243 (4) / 10917, 8967 (4) / 7537
// A matrix is spread over more SMs while the batch leaves them idle (72
// clusters of four CTAs or 15 of eight fit with two CTAs, one CTA per SM); a
// batch that fills the chip takes the fewest CTAs per matrix that its shared
// memory allows, except for float pairs above n = 112, whose single CTAs run
// out of warps.  Above n = 200 a CTA of four fills an SM's shared memory, and
// k_gj_cluster's 16 warps per CTA win once the chip is full.
int gj_smem_ctas(int n, long long conc, int nsm, bool pair) {
  if (n <= 48) return 1;
  const bool few = conc <= nsm / 10;
  if (n <= 144) {
    if (n > 128 && few) return 8;
    return (conc <= nsm * 9 / 19 || (pair && n > 112)) ? 4 : 1;
  }
  if (few) return 8;
  return (n <= 200 || conc <= nsm * 9 / 38) ? 4 : 0;
}

cudaError_t launch_gj_smem(int cs, const double* A, long long sA, double* Ainv, long long sI, int n,
                           int batch, double* logabs, int* status, cudaStream_t st, bool pair) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
#define GS_CASE(CS) \
  return pair ? gs_launch<CS, df32>(A, sA, Ainv, sI, n, batch, logabs, status, st) \
              : gs_launch<CS, double>(A, sA, Ainv, sI, n, batch, logabs, status, st)
  if (cs == 1 && n <= 144) GS_CASE(1);
  if (cs == 4) GS_CASE(4);
  if (cs == 8) GS_CASE(8);
#undef GS_CASE
  return cudaErrorInvalidValue;
}

}  // namespace dqmc
