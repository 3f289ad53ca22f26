// Sweep kernels of libdqmc: HS-field initialisation, the Metropolis pass of
// one time slice with delayed rank-k Sherman-Morrison updates, Kronecker
// multiplication by B_l = exp(-dtau K) exp(V_l) (slice wrap and UDV stack
// products), drift check and equal-time observables.
//
// Paper: Rost & Bluemer, arXiv:1504.05090, Sec. 2, Eqs. (1)-(3).  The
// Metropolis ratio and the Sherman-Morrison update follow from Eq. (3) for a
// single flip s -> -s of the Ising field (e^{V'} = e^{V}(I + Delta e_i e_i^T)):
//   R_sigma = 1 + Delta_sigma (1 - G_ii),  Delta_sigma = e^{-2 sigma lambda s} - 1,
//   G' = G - (Delta/R) (I - G) e_i e_i^T G.
// Only spin up is evolved: on the bipartite half-filled lattice
// G_dn = I - P G_up^T P (P = diag((-1)^{x+y})), so G_dn,ii = 1 - G_up,ii.
#include <cooperative_groups.h>

#include <math_constants.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace dqmc {
namespace cg = cooperative_groups;

// ---------------------------------------------------------------------------
// Initial Ising field: s = +1 iff word 0 of Philox(i + N*l, ~0, chain, 1) is odd.
// ---------------------------------------------------------------------------
__global__ void k_init_field(int8_t* field, int C, int L, int N, int chain0, uint32_t k0,
                             uint32_t k1) {
  const long long total = static_cast<long long>(C) * L * N;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < total;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(e / (static_cast<long long>(L) * N));
    const int rem = static_cast<int>(e - static_cast<long long>(c) * L * N);  // l*N + i
    const uint4 r = philox4x32_10(make_uint4(static_cast<uint32_t>(rem), 0xFFFFFFFFu,
                                             static_cast<uint32_t>(chain0 + c), kTagInitField),
                                  k0, k1);
    field[e] = (r.x & 1u) ? int8_t(1) : int8_t(-1);
  }
}

// ---------------------------------------------------------------------------
// Metropolis pass over the N sites of one slice, one cluster of cs CTAs per
// chain.  G (row-major, working precision) stays in global memory
// (L2-resident); accepted flips are buffered as column vectors U[m] and row
// vectors V[m] in shared memory, G_cur = G + sum_m U[m] V[m]^T, and folded into
// G every k accepts (delayed rank-k update).  The diagonal of G_cur is tracked
// in shared memory so that a rejected proposal costs O(1).  Between two accepted
// flips the diagonal does not change, so the 32 lanes of every warp decide 32
// sites at once and take the first accepted one; all warps agree without a
// barrier.
// ---------------------------------------------------------------------------
// Working-precision helpers.
__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(double x) { return static_cast<float>(x); }
__device__ __forceinline__ float to_f32(df32 x) { return x.hi + x.lo; }

// Sherman-Morrison coefficient -Delta_up / R_up in the working precision:
// FP32 for float, FP64 for double, and a float reciprocal refined by one
// Newton step in df32 arithmetic for df32 (no FP64 instruction).
__device__ __forceinline__ float sm_coef(const MetroArgs& a, int s, float g) {
  const float du = s > 0 ? a.em2h : a.ep2h;
  return -du / fmaf(du, 1.0f - g, 1.0f);
}
__device__ __forceinline__ double sm_coef(const MetroArgs& a, int s, double g) {
  const double du = s > 0 ? a.em2 : a.ep2;
  return -du / fma(du, 1.0 - g, 1.0);
}
__device__ __forceinline__ df32 sm_coef(const MetroArgs& a, int s, df32 g) {
  const df32 du = s > 0 ? df32(a.em2h, a.em2l) : df32(a.ep2h, a.ep2l);
  const df32 one(1.0f, 0.0f);
  const df32 ru = one + du * (one - g);
  const df32 y0(1.0f / ru.hi, 0.0f);
  const df32 y = y0 + y0 * (one - ru * y0);
  return -(du * y);
}

// Float pairs, two at a time: a 64-bit register pair holds the high (or low)
// words of two neighbouring rows, and one packed FP32 instruction works on
// both.  The packed forms run at the lane rate of the scalar ones (measured
// 117 against 108 lanes per clock and SM) with half the instructions to issue;
// every lane rounds as the scalar instruction does, so the sums are the same
// bit for bit.
__device__ __forceinline__ uint64_t pk_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void pk_unpack(uint64_t x, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x));
}
__device__ __forceinline__ uint64_t pk_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t pk_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t pk_sub(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t pk_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Two ProdSum<df32> side by side: the same twelve operations per term; the
// high product is formed negated (-uh vh), which is exact.
struct ProdSum2 {
  uint64_t hi, lo;
  __device__ __forceinline__ ProdSum2() : hi(0ull), lo(0ull) {}
  // vh, vl: splats of the second factor's words, nvh: of its negated high word;
  // kSwap: the second factor comes first in the product's error terms
  template <bool kSwap = false>
  __device__ __forceinline__ void add(uint64_t uh, uint64_t ul, uint64_t vh, uint64_t vl, uint64_t nvh) {
    const uint64_t np = pk_mul(uh, nvh);
    uint64_t e = pk_fma(uh, vh, np);
    e = kSwap ? pk_fma(ul, vh, e) : pk_fma(uh, vl, e);
    e = kSwap ? pk_fma(uh, vl, e) : pk_fma(ul, vh, e);
    const uint64_t t = pk_sub(hi, np);
    const uint64_t bb = pk_sub(t, hi);
    const uint64_t x = pk_sub(hi, pk_sub(t, bb));
    const uint64_t y = pk_add(np, bb);  // -(p - bb)
    lo = pk_add(lo, pk_add(pk_sub(x, y), e));
    hi = t;
  }
  __device__ __forceinline__ void get(df32& a, df32& b) const {
    float h0, h1, l0, l1;
    pk_unpack(hi, h0, h1);
    pk_unpack(lo, l0, l1);
    a = df_fast_two_sum(h0, l0);
    b = df_fast_two_sum(h1, l1);
  }
};

// U (or V) of the pending updates: [k][NP] numbers, or for float pairs [k][NP]
// high words followed by [k][NP] low words, so that neighbouring entries load
// as one packed operand.
template <typename T>
struct UStore {
  T* u;
  int NP;
  __device__ __forceinline__ UStore(T* base, int, int np) : u(base), NP(np) {}
  __device__ __forceinline__ T get(int m, int j) const { return u[m * NP + j]; }
  __device__ __forceinline__ void set(int m, int j, T x) const { u[m * NP + j] = x; }
};
template <>
struct UStore<df32> {
  float *h, *l;
  int NP;
  __device__ __forceinline__ UStore(df32* base, int k, int np)
      : h(reinterpret_cast<float*>(base)), l(h + k * np), NP(np) {}
  __device__ __forceinline__ df32 get(int m, int j) const { return df32(h[m * NP + j], l[m * NP + j]); }
  __device__ __forceinline__ void set(int m, int j, df32 x) const {
    h[m * NP + j] = x.hi;
    l[m * NP + j] = x.lo;
  }
};

// Column j of G, rows ra .. rb-1 (both multiples of 4): G += U V^T over the cnt
// pending updates, eight rows at a time, the next eight loaded while the
// current ones are computed.  Column j of V is read in chunks of MC updates
// per row batch (the same additions in the same order for any MC).
template <typename T, int MC>
__device__ __forceinline__ void delayed_flush(T* G, const UStore<T>& U, const UStore<T>& V, int cnt, int N,
                                              int NP, int j, int ra, int rb) {
  constexpr int RB = 8;
  if (j >= N) return;
  T cur[RB], nxt[RB];
#pragma unroll
  for (int q = 0; q < RB; ++q) cur[q] = (ra + q < rb) ? G[static_cast<size_t>(ra + q) * N + j] : T(0);
  for (int r0 = ra; r0 < rb; r0 += RB) {
    const int r1 = r0 + RB;
#pragma unroll
    for (int q = 0; q < RB; ++q)
      nxt[q] = (r1 + q < rb) ? G[static_cast<size_t>(r1 + q) * N + j] : T(0);
    if constexpr (std::is_same<T, df32>::value) {
      // 2 x 16-byte loads of U and twelve packed instructions per update and
      // four rows; bound by the FP32 pipe (64 packed lanes per clock and SM)
      ProdSum2 acc[RB / 2];
      // a chunk of MC updates without a branch inside, so that its loads are
      // issued ahead of its arithmetic; then the rest one by one
      auto chunk = [&](auto width, int m0) {
        constexpr int W = decltype(width)::value;
        uint64_t vh[W], vl[W], nvh[W];
#pragma unroll
        for (int mm = 0; mm < W; ++mm) {
          const df32 v = V.get(m0 + mm, j);
          vh[mm] = pk_pack(v.hi, v.hi);
          vl[mm] = pk_pack(v.lo, v.lo);
          nvh[mm] = pk_pack(-v.hi, -v.hi);
        }
#pragma unroll
        for (int q = 0; q < RB; q += 4) {
          ulonglong2 uh[W], ul[W];
#pragma unroll
          for (int mm = 0; mm < W; ++mm) {
            uh[mm] = *reinterpret_cast<const ulonglong2*>(U.h + (m0 + mm) * NP + r0 + q);
            ul[mm] = *reinterpret_cast<const ulonglong2*>(U.l + (m0 + mm) * NP + r0 + q);
          }
#pragma unroll
          for (int mm = 0; mm < W; ++mm) {
            acc[q / 2].add(uh[mm].x, ul[mm].x, vh[mm], vl[mm], nvh[mm]);
            acc[q / 2 + 1].add(uh[mm].y, ul[mm].y, vh[mm], vl[mm], nvh[mm]);
          }
        }
      };
      int m0 = 0;
      for (; m0 + MC <= cnt; m0 += MC) chunk(std::integral_constant<int, MC>(), m0);
      for (; m0 < cnt; ++m0) chunk(std::integral_constant<int, 1>(), m0);
#pragma unroll
      for (int q = 0; q < RB; q += 2) {
        df32 s0, s1;
        acc[q / 2].get(s0, s1);
        if (r0 + q < rb) G[static_cast<size_t>(r0 + q) * N + j] = cur[q] + s0;
        if (r0 + q + 1 < rb) G[static_cast<size_t>(r0 + q + 1) * N + j] = cur[q + 1] + s1;
      }
    } else {
      ProdSum<T> acc[RB];
      auto chunk = [&](auto width, int m0) {
        constexpr int W = decltype(width)::value;
        T v[W];
#pragma unroll
        for (int mm = 0; mm < W; ++mm) v[mm] = V.get(m0 + mm, j);
        if constexpr (std::is_same<T, float>::value) {  // four rows of U per 16-byte load
#pragma unroll
          for (int q = 0; q < RB; q += 4) {
#pragma unroll
            for (int mm = 0; mm < W; ++mm) {
              const float4 u = *reinterpret_cast<const float4*>(U.u + (m0 + mm) * NP + r0 + q);
              acc[q].add(u.x, v[mm]);
              acc[q + 1].add(u.y, v[mm]);
              acc[q + 2].add(u.z, v[mm]);
              acc[q + 3].add(u.w, v[mm]);
            }
          }
        } else {
#pragma unroll
          for (int q = 0; q < RB; ++q) {
#pragma unroll
            for (int mm = 0; mm < W; ++mm) acc[q].add(U.u[(m0 + mm) * NP + r0 + q], v[mm]);
          }
        }
      };
      int m0 = 0;
      for (; m0 + MC <= cnt; m0 += MC) chunk(std::integral_constant<int, MC>(), m0);
      for (; m0 < cnt; ++m0) chunk(std::integral_constant<int, 1>(), m0);
#pragma unroll
      for (int q = 0; q < RB; ++q)
        if (r0 + q < rb) G[static_cast<size_t>(r0 + q) * N + j] = cur[q] + acc[q].get();
    }
#pragma unroll
    for (int q = 0; q < RB; ++q) cur[q] = nxt[q];
  }
}

// Barrier between the cs CTAs of one chain's cluster around the flushes of G
// (global memory).  Thread 0 arrives on every peer's mbarrier (release at
// cluster scope) and waits for its own for at most 0.2 s; a wait that gives up
// sets kDevTimeout and lets the CTA go on, so the kernel always ends.  The __threadfence pair makes the CTA's global writes visible before
// the arrival and the peers' writes after the wait.  Barrier phases alternate
// between two mbarriers: a peer can be at most one phase ahead (it cannot pass
// phase f + 1 before this CTA arrived for it), so an arrival for phase f + 1
// never lands on the mbarrier that still collects phase f.
constexpr unsigned long long kPeerWaitNs = 200000000ull;  // 0.2 s of %globaltimer
constexpr long long kPeerWaitPolls = 1LL << 24;             // and at most this many polls

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// `broken` (shared) is set once a wait gave up; later barriers of the launch
// then only synchronise the CTA.
// kGlobal: G in global memory is ordered too (a flush); otherwise only the
// shared memory written to the peers.
template <bool kGlobal>
__device__ __forceinline__ void peer_barrier(uint64_t* bars, int cs, int rank, int& phase,
                                             int* status, int* broken) {
  __syncthreads();
  // thread r arrives at peer r (one after the other they would wait for each
  // other's release)
  const bool ok = !*broken;
  const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(bars + (phase & 1)));
  if (static_cast<int>(threadIdx.x) < cs && static_cast<int>(threadIdx.x) != rank && ok) {
    if (kGlobal) __threadfence();
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(threadIdx.x));
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote)
                 : "memory");
  }
  if (threadIdx.x == 0 && ok) {
    uint32_t done = 0;
    unsigned long long t0 = 0;  // read only once a wait gets long (the timer is slow)
    for (long long it = 0; it < kPeerWaitPolls && !done; ++it) {
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
          " selp.u32 %0, 1, 0, p;\n}"
          : "=r"(done)
          : "r"(local), "r"((phase >> 1) & 1)
          : "memory");
      if (!done && (it & 255) == 255) {
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > kPeerWaitNs) break;
      }
    }
    if (!done) {
      atomicExch(status, kDevTimeout);
      *broken = 1;
    }
    if (kGlobal) __threadfence();
  }
  ++phase;
  __syncthreads();
}

// Columns of G staged in shared memory per window of sites (k_metropolis).
constexpr int kWin = 32;
constexpr int kRing = 8;  // rows of G asked for ahead

// Pending updates per register chunk of the flush: as many as 128 registers
// per thread (512 threads) allow beside the eight rows in flight.
template <typename T>
constexpr int kFlushMC() {
  return std::is_same<T, float>::value ? 16 : std::is_same<T, df32>::value ? 4 : 8;
}

constexpr int kHalves = 2;
constexpr int kMetroThreads = kHalves * kMaxN;  // most threads per CTA besides the scalar warp

// H = 2 threads per column (4 and 8 were measured: never faster, and up to
// twice slower with many small chains); both share the rows of a flush.  Of an
// accepted flip, half of the working threads (role 0) correct the column G e_i
// for the pending updates, the other half (role 1) the row e_i^T G, one column
// each; float pairs take two columns per thread with packed instructions, so
// that half of the warps have no part in a flip: they wait at the CTA's
// barrier for the next flush, and the flips synchronise the others only.  In
// FP32, where a flip is little more than its barriers, one thread does both for
// its column and the flip needs one barrier instead of two.  One warp forms the
// Sherman-Morrison coefficient of the flip: a chain of dependent operations
// that, repeated by every warp, took more of the FP64 pipe than the
// corrections.  In FP64 it is a warp of its own (kScalarWarp); for float pairs,
// whose flush needs the registers that a 17th warp would cost, one of the idle
// warps (if there is one).
//
// Thread-block cluster of cs CTAs per chain (cs = 1: one CTA).  Every CTA
// takes the same site decisions from the same data (identical instruction
// streams, so identical results); in a flush each CTA adds U V^T to its own
// block of rows of G.  Two peer barriers bracket every flush: no CTA
// overwrites rows that a peer may still read for the sites before the flush,
// and every CTA reads the new rows after it.  U and V are formed by every CTA
// for itself, or, in FP64 from N = 128 on (kSplitN), each CTA corrects only its
// share of the columns and sends the entries to its peers: the corrections are
// then a quarter of the FP64 work of a pass instead of a copy of it on every
// SM, for one more peer barrier per accepted flip.
constexpr int kSplitN = 128;

template <typename T>
constexpr bool kScalarWarp() {
  return std::is_same<T, double>::value;
}

template <typename T>
__global__ void __launch_bounds__(kMetroThreads + (kScalarWarp<T>() ? 32 : 0)) k_metropolis(T* Gall, int8_t* fieldall, MetroArgs a) {
  const int cs = a.cs;
  const int c = blockIdx.x / cs;
  const int rank = blockIdx.x - c * cs;  // cluster rank (the cluster spans blockIdx.x)
  const int N = a.N;
  constexpr int H = kHalves;
  const int NP = (blockDim.x - (kScalarWarp<T>() ? 32 : 0)) / H;  // columns (N rounded up to a warp)
  const int h = threadIdx.x / NP;        // H: the scalar warp
  // rows of G this thread folds the delayed updates into, in units of four:
  // the CTA's block, split between its H thread groups
  const int n4 = N >> 2, part = rank * H + h, parts = cs * H;
  const int ra = 4 * ((part * n4) / parts), rb = (h < H) ? 4 * (((part + 1) * n4) / parts) : 0;
  __shared__ T coef_sh;
  __shared__ uint64_t xbar[2];
  __shared__ int xbroken;
  int xphase = 0;
  if (cs > 1) {
    if (threadIdx.x == 0) {
      // a peer wait of an earlier launch gave up: results are void already,
      // so this launch does not wait again
      xbroken = (*reinterpret_cast<volatile int*>(a.status) == kDevTimeout);
      for (int b = 0; b < 2; ++b)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(
                         static_cast<uint32_t>(__cvta_generic_to_shared(xbar + b))),
                     "r"(cs - 1));
      asm volatile("fence.mbarrier_init.release.cluster;");
    }
    cooperative_groups::this_cluster().sync();
  }
  const int j = threadIdx.x - h * NP;  // column of this thread
  const int lane = threadIdx.x & 31;
  const bool act = h < H && j < N;
  T* G = Gall + static_cast<size_t>(c) * N * N;
  int8_t* s_l = fieldall + (static_cast<size_t>(c) * a.L + a.l0) * N;

  extern __shared__ __align__(16) unsigned char sm_raw[];
  double* uu = reinterpret_cast<double*>(sm_raw);  // [NP] proposal uniforms
  float* uuf = reinterpret_cast<float*>(uu + NP);   // [NP] the same, rounded to float
  T* Ubase = reinterpret_cast<T*>(uuf + NP);        // [k][NP], see UStore
  const UStore<T> U(Ubase, a.k, NP);
  T* Vbase = Ubase + a.k * NP;                      // [k][NP]
  const UStore<T> V(Vbase, a.k, NP);
  T* d = Vbase + a.k * NP;                          // [NP] diag of G_cur
  float* df = reinterpret_cast<float*>(d + NP);     // [NP] diag of G_cur, rounded to float
  int* ss = reinterpret_cast<int*>(df + NP);        // [NP] field of the slice
  T* ring = reinterpret_cast<T*>(ss + NP);          // [kRing][NP] rows of G to come (FP32)
  T* cw = ring + (std::is_same<T, float>::value ? kRing * NP : 0);  // [kWin][NP + 1] window of columns of G

  const uint32_t sweep = *a.sweep_ctr;
  if (act && h == 0) {
    const T gjj = G[static_cast<size_t>(j) * N + j];
    d[j] = gjj;
    df[j] = to_f32(gjj);
    ss[j] = s_l[j];
    const uint4 r = philox4x32_10(make_uint4(static_cast<uint32_t>(j + N * a.l0), sweep,
                                             static_cast<uint32_t>(a.chain0 + c), kTagProposal),
                                  a.key0, a.key1);
    const double u = uniform53(r.x, r.y);
    uu[j] = u;
    uuf[j] = static_cast<float>(u);
  }
  __syncthreads();

  // Columns wb .. wb + kWin - 1 of G in shared memory, cw[c][j] = G[j][wb + c]:
  // loaded with whole-row segments (a column of the row-major G would take one
  // memory transaction per row), reloaded every kWin sites and after a flush.
  const int ldw = NP + 1;  // odd stride in 8-byte words: conflict-free transposed stores
  auto load_window = [&](int wb, int nthr) {
    constexpr int kU = 8;
    const int tot = N * kWin;
    for (int e0 = threadIdx.x; e0 < tot; e0 += kU * nthr) {
      T t[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int e = e0 + u * nthr, r = e / kWin, c = e - r * kWin;
        t[u] = (e < tot && wb + c < N) ? G[static_cast<size_t>(r) * N + wb + c] : T(0);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int e = e0 + u * nthr, r = e / kWin, c = e - r * kWin;
        if (e < tot) cw[c * ldw + r] = t[u];
      }
    }
  };
  int wb = 0;
  load_window(0, blockDim.x);
  __syncthreads();
  // The entry of U (role 0) or V (role 1) that this thread forms of an accepted
  // flip: its own column cj, or with a split correction one of the CTA's share
  // (the first 2 ns threads); float pairs: two neighbouring columns cj, cj + 1
  // with packed instructions.  role < 0: none.
  constexpr bool kPair = std::is_same<T, df32>::value;
  constexpr bool kBoth = std::is_same<T, float>::value;  // role 2: column and row
  const bool split = std::is_same<T, double>::value && cs > 1 && N >= kSplitN;
  int role = (h < 2 && act) ? h : -1, cj = j;
  // kPair: warps 0 .. pw-1 role 0, pw .. 2 pw-1 role 1, the next (if there is
  // one) the coefficient; all others only flush
  const int warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5, pw = (NP / 2 + 31) >> 5;
  const int nact = kPair ? 32 * min(nwarp, 2 * pw + 1) : kBoth ? NP : static_cast<int>(blockDim.x);
  if (kBoth) role = (h == 0 && act) ? 2 : -1;
  if (kPair) {
    role = warp < pw ? 0 : warp < 2 * pw ? 1 : -1;
    cj = 2 * (static_cast<int>(threadIdx.x) - 32 * pw * max(role, 0));
    if (cj >= N) role = -1;
  }
  const int coef_thread = kScalarWarp<T>() ? H * NP : (nwarp > 2 * pw ? 64 * pw : 32 * pw);
  if (split) {
    const int s0 = (rank * N) / cs, ns = ((rank + 1) * N) / cs - s0;
    role = static_cast<int>(threadIdx.x) / ns;
    cj = s0 + static_cast<int>(threadIdx.x) - role * ns;
    if (role > 1) role = -1;
  }
  // Rows of G of the sites to come, asked for ahead by the threads of role 1
  // (or 2), each for its own columns.  Float pairs and FP64 keep the kPre rows
  // after the last accepted site in registers; in FP32, where an L2 access takes
  // about as long as a flip, cp.async brings rows kRing sites ahead into a ring
  // in shared memory (for the other types the ring's bookkeeping cost more than
  // the wait: 686 against 663 us per slice, 16 x 16 in float pairs; FP32 8 x 8
  // with it 48 instead of 52 us).  A flush rewrites G, after which the rows are
  // asked for again.
  struct Entry {
    T x[kPair ? 2 : 1];
  };
  auto ld_row = [&](int q) -> Entry {
    Entry e;
    const T* src = G + static_cast<size_t>(q) * N + cj;
    if constexpr (kPair) {
      const float4 f = *reinterpret_cast<const float4*>(src);
      e.x[0] = df32(f.x, f.y);
      e.x[1] = df32(f.z, f.w);
    } else {
      e.x[0] = *src;
    }
    return e;
  };
  constexpr int kPre = 2;
  Entry pr[kPre];
  // first row in pr; for the ring: the last group of copies holds rows pbase ..
  // rq-1
  int pbase = 0, rq = 0;
  auto prefetch = [&](int q0) {
    if (role < 1) return;
    if constexpr (kBoth) {
      pbase = max(rq, q0);
      const int qe = min(q0 + kRing, N);
      for (rq = pbase; rq < qe; ++rq)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(static_cast<uint32_t>(
                         __cvta_generic_to_shared(ring + (rq % kRing) * NP + cj))),
                     "l"(G + static_cast<size_t>(rq) * N + cj)
                     : "memory");
      asm volatile("cp.async.commit_group;" ::: "memory");
    } else {
      pbase = q0;
#pragma unroll
      for (int q = 0; q < kPre; ++q)
        if (q0 + q < N) pr[q] = ld_row(q0 + q);
    }
  };
  auto row_entry = [&](int i) -> Entry {  // the own entries of row i
    if constexpr (kBoth) {
      // a slot is asked for again only once its copy has landed (groups are not
      // ordered against each other): the rows up to i are those of the groups
      // waited for here
      if (i >= pbase)
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      else
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      if (i >= rq) return ld_row(i);  // further ahead than the ring
      Entry e;
      e.x[0] = ring[(i % kRing) * NP + cj];
      return e;
    } else {
      return i == pbase ? pr[0] : i == pbase + 1 ? pr[1] : ld_row(i);
    }
  };
  prefetch(0);
  int cnt = 0;
  unsigned naccept = 0;
  // pending updates of a flush and the first site of the next window (-1: the
  // slice ends), for the warps that take no part in the flips
  __shared__ int flush_sh[2];
  // barrier of the warps that work on the flips
  auto sync_act = [&]() {
    if constexpr (kPair || kBoth)
      asm volatile("bar.sync 1, %0;" ::"r"(nact) : "memory");
    else
      __syncthreads();
  };
  int i = 0;
  do {
    if (static_cast<int>(threadIdx.x) < nact) {
      while (i < N && cnt < a.k) {
        // Decision u < R_up R_dn with R_up = 1 + D_up (1 - G_ii), R_dn = 1 + D_dn G_ii
        // (G_dn,ii = 1 - G_up,ii) of sites i .. i + 31, one per lane: in FP32 unless
        // u lies within 1e-4 of R, where it is retaken in FP64.
        bool acc = false;
        if (i + lane < N) {
          const int q = i + lane, s = ss[q];
          const float gf = df[q];
          const float duf = s > 0 ? a.em2h : a.ep2h, ddf = s > 0 ? a.ep2h : a.em2h;
          const float Rf = fmaf(duf, 1.0f - gf, 1.0f) * fmaf(ddf, gf, 1.0f);
          const float uf = uuf[q];
          if (uf < Rf * 0.9999f) {
            acc = true;
          } else if (!(uf > Rf * 1.0001f)) {
            const double g = static_cast<double>(d[q]);
            const double du = s > 0 ? a.em2 : a.ep2, dd = s > 0 ? a.ep2 : a.em2;
            acc = uu[q] < fma(du, 1.0 - g, 1.0) * fma(dd, g, 1.0);
          }
        }
        const unsigned hits = __ballot_sync(0xFFFFFFFFu, acc);
        if (hits == 0u) {
          i += 32;
          continue;
        }
        i += __ffs(hits) - 1;  // the next accepted site
        if (i >= wb + kWin) {  // nobody reads the window between two accepted sites
          wb = i;
          load_window(wb, nact);
          sync_act();
        }
        ++naccept;
        if constexpr (kBoth) {
          T coef = T(0);
          if (lane == 0) coef = sm_coef(a, ss[i], d[i]);
          coef = __shfl_sync(0xFFFFFFFFu, coef, 0);
          if (role == 2) {
            ProdSum<T> sc, sr;
#pragma unroll 4
            for (int m = 0; m < cnt; ++m) {
              sc.add(U.get(m, j), V.get(m, i));
              sr.add(U.get(m, i), V.get(m, j));
            }
            const T row = row_entry(i).x[0];
            const T uj = coef * ((j == i ? T(1) : T(0)) - (cw[(i - wb) * ldw + j] + sc.get()));
            const T vj = row + sr.get();
            U.set(cnt, j, uj);
            V.set(cnt, j, vj);
            // a slower warp may still be deciding: what it reads of the sites
            // up to i is left alone, and what it makes of later ones, beyond
            // the first accepted site i, it does not use
            if (j > i) {
              const T dj = d[j] + uj * vj;
              d[j] = dj;
              df[j] = to_f32(dj);
            }
          }
          prefetch(i + 1);
          sync_act();
          if (threadIdx.x == 0) ss[i] = -ss[i];  // site i is not read again
          ++cnt;
          ++i;
          continue;
        }
        if (static_cast<int>(threadIdx.x) == coef_thread) coef_sh = sm_coef(a, ss[i], d[i]);
        // column (role 0: e_i - G e_i, scaled below) or row (role 1: e_i^T G)
        // entry of G_cur, four updates' loads at a time ahead of their serial sums
        Entry w0;  // role 0 of float pairs: the unscaled entries of U
        if (role >= 0) {
          // the entry of G, read after the sums
          auto g_entry = [&]() -> Entry {
            Entry e;
            if (role == 0) {
              e.x[0] = cw[(i - wb) * ldw + cj];
              if constexpr (kPair) e.x[1] = cw[(i - wb) * ldw + cj + 1];
            } else {
              e = row_entry(i);
            }
            return e;
          };
          int m = 0;
          if constexpr (kPair) {
            const UStore<df32>& P = role == 0 ? U : V;  // two entries of the own columns
            const UStore<df32>& S = role == 0 ? V : U;  // the entry of site i
            ProdSum2 sa;
            auto terms = [&](auto width, auto swap) {
              constexpr int W = decltype(width)::value;
              uint64_t ph[W], pl[W];
              df32 sp[W];
#pragma unroll
              for (int q = 0; q < W; ++q) {
                ph[q] = *reinterpret_cast<const uint64_t*>(P.h + (m + q) * NP + cj);
                pl[q] = *reinterpret_cast<const uint64_t*>(P.l + (m + q) * NP + cj);
                sp[q] = S.get(m + q, i);
              }
#pragma unroll
              for (int q = 0; q < W; ++q)
                sa.template add<decltype(swap)::value>(ph[q], pl[q], pk_pack(sp[q].hi, sp[q].hi),
                                                       pk_pack(sp[q].lo, sp[q].lo), pk_pack(-sp[q].hi, -sp[q].hi));
            };
            if (role == 0) {
              for (; m + 4 <= cnt; m += 4) terms(std::integral_constant<int, 4>(), std::false_type());
              for (; m < cnt; ++m) terms(std::integral_constant<int, 1>(), std::false_type());
            } else {
              for (; m + 4 <= cnt; m += 4) terms(std::integral_constant<int, 4>(), std::true_type());
              for (; m < cnt; ++m) terms(std::integral_constant<int, 1>(), std::true_type());
            }
            df32 s0, s1;
            sa.get(s0, s1);
            const Entry g0 = g_entry();
            if (role == 0) {
              s0 = (cj == i ? T(1) : T(0)) - (g0.x[0] + s0);
              s1 = (cj + 1 == i ? T(1) : T(0)) - (g0.x[1] + s1);
            } else {
              s0 = g0.x[0] + s0;
              s1 = g0.x[1] + s1;
            }
            if (role == 1) {
              *reinterpret_cast<uint64_t*>(V.h + cnt * NP + cj) = pk_pack(s0.hi, s1.hi);
              *reinterpret_cast<uint64_t*>(V.l + cnt * NP + cj) = pk_pack(s0.lo, s1.lo);
            }
            w0.x[0] = s0;
            w0.x[1] = s1;
          } else {
            ProdSum<T> sa;
            const int ju = (role == 0) ? cj : i, jv = (role == 0) ? i : cj;
            for (; m + 4 <= cnt; m += 4) {
              T u[4], v[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                u[q] = U.get(m + q, ju);
                v[q] = V.get(m + q, jv);
              }
#pragma unroll
              for (int q = 0; q < 4; ++q) sa.add(u[q], v[q]);
            }
            for (; m < cnt; ++m) sa.add(U.get(m, ju), V.get(m, jv));
            const T gs = g_entry().x[0] + sa.get();
            const T x = (role == 0) ? (cj == i ? T(1) : T(0)) - gs : gs;
            if (!split) {
              (role == 0 ? U : V).set(cnt, cj, x);
            } else {
              if constexpr (std::is_same<T, double>::value) {
                double* dst = (role == 0 ? U.u : V.u) + cnt * NP + cj;
                cg::cluster_group cl = cg::this_cluster();
                for (int r = 0; r < cs; ++r) *cl.map_shared_rank(dst, r) = x;
              }
            }
          }
        }
        prefetch(i + 1);
        if (split)
          peer_barrier<false>(xbar, cs, rank, xphase, a.status, &xbroken);
        else
          sync_act();
        // every warp is at site i here, so the diagonal of the sites to come is
        // updated before anyone decides the next site (barrier below)
        if constexpr (kPair) {
          if (role == 0) {
            const df32 cf = coef_sh;
            df32 uj[2], dj[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              uj[q] = cf * w0.x[q];
              dj[q] = d[cj + q] + uj[q] * V.get(cnt, cj + q);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
              if (cj + q > i) {
                d[cj + q] = dj[q];
                df[cj + q] = to_f32(dj[q]);
              }
            *reinterpret_cast<uint64_t*>(U.h + cnt * NP + cj) = pk_pack(uj[0].hi, uj[1].hi);
            *reinterpret_cast<uint64_t*>(U.l + cnt * NP + cj) = pk_pack(uj[0].lo, uj[1].lo);
          }
        } else if (act && h == 0) {
          const T uj = coef_sh * U.get(cnt, j);
          U.set(cnt, j, uj);
          if (j > i) {
            const T dj = d[j] + uj * V.get(cnt, j);
            d[j] = dj;
            df[j] = to_f32(dj);
          }
        }
        if (threadIdx.x == 0) ss[i] = -ss[i];  // site i is not read again
        ++cnt;
        ++i;
        sync_act();
      }
      if (threadIdx.x == 0) {
        flush_sh[0] = cnt;
        flush_sh[1] = (i < N) ? i : -1;
      }
    }
    // flush, by all warps; no copy of a row may be under way while G is rewritten
    if constexpr (kBoth) asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (cs > 1)
      peer_barrier<true>(xbar, cs, rank, xphase, a.status, &xbroken);
    else
      __syncthreads();
    cnt = flush_sh[0];
    wb = flush_sh[1];
    if (cnt > 0) delayed_flush<T, kFlushMC<T>()>(G, U, V, cnt, N, NP, j, ra, rb);
    cnt = 0;
    if (wb >= 0) {
      if (cs > 1)
        peer_barrier<true>(xbar, cs, rank, xphase, a.status, &xbroken);
      else
        __syncthreads();
      load_window(wb, blockDim.x);
      __syncthreads();
      rq = wb;
      prefetch(wb);
    }
  } while (wb >= 0);
  // No CTA leaves while a peer may still arrive on its barrier or read the
  // slice's field.
  if (cs > 1) cooperative_groups::this_cluster().sync();
  // The field is written back after the slice: a peer CTA of the cluster may
  // still be reading the slice's initial field when this one accepts a flip.
  if (rank == 0) {
    if (act && h == 0) s_l[j] = static_cast<int8_t>(ss[j]);
    if (threadIdx.x == 0) a.accepted[c] += naccept;
  }
}

// ---------------------------------------------------------------------------
// Kronecker transform of nv vectors held in shared memory (row stride ld):
// v <- Ey (x) Ex applied to (pre o v), then multiplied by post.
// ---------------------------------------------------------------------------
// Two taps read with one load (16 bytes for 8-byte types).
template <typename T>
struct alignas(2 * sizeof(T)) KronPair {
  T a, b;
};

// Tap t of a table (below).  Float pairs: taps 2i, 2i + 1 as (hi, hi, lo, lo), so
// that one 16-byte load gives both packed operands.
template <typename T>
__device__ __forceinline__ void kron_put_tap(T* tab, int t, double x) {
  if constexpr (std::is_same<T, df32>::value) {
    const df32 d(x);
    float* f = reinterpret_cast<float*>(tab) + 4 * (t >> 1) + (t & 1);
    f[0] = d.hi;
    f[2] = d.lo;
  } else {
    tab[t] = static_cast<T>(x);
  }
}

// One side of the transform in float pairs: two neighbouring
// outputs along the side are the two lanes of packed sums, and a thread takes
// them for V vectors (vi, vi + nv / V), which share the tap load.  The same
// operations in the same order per output as with scalar sums.
// What bounds it: no one thing at 16 x 16 (issue slots 57 % busy; the waits are
// shared by the FP32 pipe, dependent sums, loads of the tile and barriers).  A
// term's twelve packed operations stand for 24 scalar ones and leave slots for
// the loads.
// Two vectors per thread where that still gives every thread of the CTA work
// (nv N >= 4 threads: 4 vectors at 16 x 16, all of 8 x 8 in one CTA), else one.
// Sweeps with scalar sums, then packed: 16 x 16, 64 chains 379.4 -> 375.7 ms
// (320 passes, 11 us each); 8 x 8, 3 x 256 chains 117.4 -> 115.7; two chains of
// 16 x 16 unchanged at 80.1.
template <int V, bool kY>
__device__ __forceinline__ void kron_side_df32(const df32* in, df32* out, int nv, int ld, int Lx,
                                               int Ly, const df32* t0, const df32* t1,
                                               const df32* post) {
  const int h = nv / V, per = (Lx * Ly) >> 1, n = kY ? Ly : Lx, w = kY ? Lx : Lx >> 1;
  const int str = kY ? Lx : 1;
  for (int e = threadIdx.x; e < h * per; e += blockDim.x) {
    const int vi = e / per, rr = e - vi * per, q = rr / w, r = rr - q * w;
    const int o = 2 * (kY ? q : r);  // the first output along the side
    const int base = vi * ld + (kY ? r : Lx * q);
    const df32* p = in + base;
    ProdSum2 a[V];
#pragma unroll 2
    for (int k = 0; k < n; ++k) {
      const int b = o + n - k;  // tap index of output o; b + 1 that of o + 1
      const ulonglong2 t = *reinterpret_cast<const ulonglong2*>((b & 1) ? t1 + b - 1 : t0 + b);
#pragma unroll
      for (int u = 0; u < V; ++u) {
        const df32 x = p[u * h * ld + str * k];
        a[u].add(t.x, t.y, pk_pack(x.hi, x.hi), pk_pack(x.lo, x.lo), pk_pack(-x.hi, -x.hi));
      }
    }
#pragma unroll
    for (int u = 0; u < V; ++u) {
      df32 y0, y1;
      a[u].get(y0, y1);
      const int i0 = (kY ? r : Lx * q) + str * o, i1 = i0 + str;
      df32* d = out + (vi + u * h) * ld;
      d[i0] = post ? y0 * post[i0] : y0;
      d[i1] = post ? y1 * post[i1] : y1;
    }
  }
}

template <typename T>
__device__ __forceinline__ void kron_transform(T* v, T* tmp, int nv, int ld, int Lx, int Ly, int N,
                                               const T* tx, const T* ty, const T* txs,
                                               const T* tys, const T* pre, const T* post) {
  const int tot = nv * N;
  if (pre) {  // diagonal factor applied once per element, not once per tap
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
      const int vi = e / N, i = e - vi * N;
      v[vi * ld + i] *= pre[i];
    }
    __syncthreads();
  }
  // Both sides are even: a thread takes two neighbouring outputs (x, x + 1) of one
  // row (then (y, y + 1) of one column).  Both sums read the same input
  // entry (one load), and their taps E[x - x'], E[x + 1 - x'] are adjacent:
  // one 16-byte load from tx (tap index even) or from txs, the same taps
  // shifted by one (odd).  Same additions in the same order per output.
  if constexpr (std::is_same<T, df32>::value) {
    if ((nv & 1) == 0 && nv * N >= 4 * static_cast<int>(blockDim.x)) {
      kron_side_df32<2, false>(v, tmp, nv, ld, Lx, Ly, tx, txs, nullptr);
      __syncthreads();
      kron_side_df32<2, true>(tmp, v, nv, ld, Lx, Ly, ty, tys, post);
    } else {
      kron_side_df32<1, false>(v, tmp, nv, ld, Lx, Ly, tx, txs, nullptr);
      __syncthreads();
      kron_side_df32<1, true>(tmp, v, nv, ld, Lx, Ly, ty, tys, post);
    }
    __syncthreads();
    return;
  }
  const int hx = Lx >> 1, hy = Ly >> 1;
  const int ptx = nv * Ly * hx;
  for (int e = threadIdx.x; e < ptx; e += blockDim.x) {
    const int vi = e / (Ly * hx), rr = e - vi * (Ly * hx), y = rr / hx, x = 2 * (rr - y * hx);
    const T* row = v + vi * ld + Lx * y;
    ProdSum<T> a0, a1;
    for (int xp = 0; xp < Lx; ++xp) {
      const int b = x + Lx - xp;  // tap index of output x; b + 1 that of x + 1
      const KronPair<T> t2 = (b & 1) ? *reinterpret_cast<const KronPair<T>*>(txs + b - 1)
                                     : *reinterpret_cast<const KronPair<T>*>(tx + b);
      const T r = row[xp];
      a0.add(t2.a, r);
      a1.add(t2.b, r);
    }
    tmp[vi * ld + Lx * y + x] = a0.get();
    tmp[vi * ld + Lx * y + x + 1] = a1.get();
  }
  __syncthreads();
  const int pty = nv * hy * Lx;
  for (int e = threadIdx.x; e < pty; e += blockDim.x) {
    const int vi = e / (hy * Lx), rr = e - vi * (hy * Lx), yp2 = rr / Lx, x = rr - yp2 * Lx;
    const int y = 2 * yp2;
    const T* col = tmp + vi * ld + x;
    ProdSum<T> a0, a1;
    for (int yp = 0; yp < Ly; ++yp) {
      const int b = y + Ly - yp;
      const KronPair<T> t2 = (b & 1) ? *reinterpret_cast<const KronPair<T>*>(tys + b - 1)
                                     : *reinterpret_cast<const KronPair<T>*>(ty + b);
      const T c = col[Lx * yp];
      a0.add(t2.a, c);
      a1.add(t2.b, c);
    }
    const int i0 = x + Lx * y, i1 = i0 + Lx;
    v[vi * ld + i0] = post ? a0.get() * post[i0] : a0.get();
    v[vi * ld + i1] = post ? a1.get() * post[i1] : a1.get();
  }
  __syncthreads();
}

// Shared-memory staging common to both Kronecker kernels.
template <typename T>
struct KronStage {
  T* v;
  T* tmp;
  T* tx;   // active taps x
  T* ty;   // active taps y
  T* txs;  // the same taps shifted by one, txs[k] = tx[k + 1] (paired loads)
  T* tys;
  T* sc;   // diag scale of the current slice
};

template <typename T>
__device__ __forceinline__ KronStage<T> kron_stage(unsigned char* raw, int nv, int ld) {
  KronStage<T> s;
  s.v = reinterpret_cast<T*>(raw);
  s.tmp = s.v + nv * ld;
  s.tx = s.tmp + nv * ld;
  s.ty = s.tx + 2 * kMaxSide;
  s.txs = s.ty + 2 * kMaxSide;
  s.tys = s.txs + 2 * kMaxSide;
  s.sc = s.tys + 2 * kMaxSide;
  return s;
}

// Resolve the slice range of batch entry b (one chain, or one chain x block).
__device__ __forceinline__ bool kron_entry_range(const KronArgs& a, int b, int* chain, int* first,
                                                 int* count) {
  *chain = b / a.per_chain;
  if (a.cp) {
    const int blk = b - *chain * a.per_chain;
    const int lo = a.cp[blk] + a.step, hi = a.cp[blk + 1];
    *first = lo;
    *count = (lo < hi) ? 1 : 0;
    return lo < hi;
  }
  *first = a.l0_first;
  *count = a.n_slices;
  return a.n_slices > 0;
}

template <typename T>
__device__ __forceinline__ void kron_load_taps(const KronArgs& a, KronStage<T> s) {
  if (threadIdx.x < 2 * kMaxSide) {  // each circulant row twice over (kron_transform)
    const int t = threadIdx.x, tx = t % a.Lx, ty = t % a.Ly;
    const bool inv = (a.kind == kBIT);
    const int tx1 = (t + 1) % a.Lx, ty1 = (t + 1) % a.Ly;
    kron_put_tap(s.tx, t, inv ? a.taps.exi[tx] : a.taps.ex[tx]);
    kron_put_tap(s.ty, t, inv ? a.taps.eyi[ty] : a.taps.ey[ty]);
    kron_put_tap(s.txs, t, inv ? a.taps.exi[tx1] : a.taps.ex[tx1]);
    kron_put_tap(s.tys, t, inv ? a.taps.eyi[ty1] : a.taps.ey[ty1]);
  }
}

template <typename T>
__device__ __forceinline__ void kron_load_scale(const KronArgs& a, KronStage<T> s,
                                                const int8_t* f_l, int N) {
  // e^{+-c}, precomputed on the host: FP64 exp is dozens of FP64-pipe passes.
  const T up = static_cast<T>((a.kind == kBIT) ? a.emc : a.ec);
  const T dn = static_cast<T>((a.kind == kBIT) ? a.ec : a.emc);
  for (int i = threadIdx.x; i < N; i += blockDim.x) s.sc[i] = f_l[i] > 0 ? up : dn;
}

// Vectors are contiguous rows of each N x N matrix.  Each CTA owns nv rows of
// one batch entry and applies `count` successive slice factors to them.
template <typename T>
__global__ void __launch_bounds__(256) k_kron_rows(const T* in, T* out, KronArgs a) {
  const int b = blockIdx.y;
  int chain, first, count;
  if (!kron_entry_range(a, b, &chain, &first, &count)) return;
  const int N = a.N, nv = a.nv, ld = N + 1;
  const int r0 = blockIdx.x * nv;
  const int nrows = min(nv, N - r0);
  extern __shared__ __align__(16) unsigned char sm_raw[];
  KronStage<T> s = kron_stage<T>(sm_raw, nv, ld);
  kron_load_taps(a, s);
  const T* src = in + static_cast<size_t>(b) * a.mat_stride;
  T* dst = out + static_cast<size_t>(b) * a.out_stride;
  for (int e = threadIdx.x; e < nrows * N; e += blockDim.x) {
    const int vi = e / N, i = e - vi * N;
    T val = src[static_cast<size_t>(r0 + vi) * N + i];
    if (a.vscale) val *= static_cast<T>(a.vscale[static_cast<size_t>(b) * a.vscale_stride + r0 + vi]);
    s.v[vi * ld + i] = val;
  }
  const int8_t* f = a.field + static_cast<size_t>(chain) * a.L * N;
  for (int st = 0; st < count; ++st) {
    const int l0 = first + st * a.dir;
    __syncthreads();
    kron_load_scale(a, s, f + static_cast<size_t>(l0) * N, N);
    __syncthreads();
    if (a.kind == kBT)
      kron_transform(s.v, s.tmp, nrows, ld, a.Lx, a.Ly, N, s.tx, s.ty, s.txs, s.tys, (const T*)nullptr,
                     (const T*)s.sc);
    else
      kron_transform(s.v, s.tmp, nrows, ld, a.Lx, a.Ly, N, s.tx, s.ty, s.txs, s.tys, (const T*)s.sc,
                     (const T*)nullptr);
  }
  for (int e = threadIdx.x; e < nrows * N; e += blockDim.x) {
    const int vi = e / N, i = e - vi * N;
    dst[static_cast<size_t>(r0 + vi) * N + i] = s.v[vi * ld + i];
  }
}

// Vectors are the columns of each row-major N x N matrix (in place).
template <typename T>
__global__ void __launch_bounds__(256) k_kron_cols(T* X, KronArgs a) {
  const int b = blockIdx.y;
  int chain, first, count;
  if (!kron_entry_range(a, b, &chain, &first, &count)) return;
  const int N = a.N, nv = a.nv, ld = N + 1;
  const int c0 = blockIdx.x * nv;
  const int ncols = min(nv, N - c0);
  extern __shared__ __align__(16) unsigned char sm_raw[];
  KronStage<T> s = kron_stage<T>(sm_raw, nv, ld);
  kron_load_taps(a, s);
  T* M = X + static_cast<size_t>(b) * a.mat_stride;
  for (int e = threadIdx.x; e < ncols * N; e += blockDim.x) {
    const int i = e / ncols, jj = e - i * ncols;
    s.v[jj * ld + i] = M[static_cast<size_t>(i) * N + c0 + jj];
  }
  const int8_t* f = a.field + static_cast<size_t>(chain) * a.L * N;
  for (int st = 0; st < count; ++st) {
    const int l0 = first + st * a.dir;
    __syncthreads();
    kron_load_scale(a, s, f + static_cast<size_t>(l0) * N, N);
    __syncthreads();
    if (a.kind == kBT)
      kron_transform(s.v, s.tmp, ncols, ld, a.Lx, a.Ly, N, s.tx, s.ty, s.txs, s.tys, (const T*)nullptr,
                     (const T*)s.sc);
    else
      kron_transform(s.v, s.tmp, ncols, ld, a.Lx, a.Ly, N, s.tx, s.ty, s.txs, s.tys, (const T*)s.sc,
                     (const T*)nullptr);
  }
  for (int e = threadIdx.x; e < ncols * N; e += blockDim.x) {
    const int i = e / ncols, jj = e - i * ncols;
    M[static_cast<size_t>(i) * N + c0 + jj] = s.v[jj * ld + i];
  }
}

// ---------------------------------------------------------------------------
// Slice wrap G <- B_l G B_l^-1 of a small lattice with G in shared memory, one
// CTA per matrix: the columns and the rows in one launch and one trip through
// memory.  The operations of k_kron_cols and k_kron_rows in the same order.
//
// What bounds it: the two passes were mostly launch, latency and barriers (a
// CTA had four vectors, seven barriers and three dependent trips to memory for
// 256 elements); here a thread has all its elements in flight at once, and the
// arithmetic fills the rest.  8 x 8 float pairs, 256 chains beside two other
// such groups: 37.7 + 37.7 us before, 38.5 now.
// ---------------------------------------------------------------------------
constexpr int kWT = 512;
template <typename T>
__global__ void __launch_bounds__(kWT, 2) k_wrap_smem(T* X, KronArgs a) {
  const int b = blockIdx.x, N = a.N, ld = N + 1, tot = N * N;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  KronStage<T> s = kron_stage<T>(sm_raw, N, ld);
  T* sc2 = s.sc + N;           // scale of the rows' pass
  T* taps2 = sc2 + N;          // its taps, as s.tx ...
  T* M = X + static_cast<size_t>(b) * a.mat_stride;
  constexpr int kU = 8;  // elements in flight per thread: all of them at N = 64
  T r[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const int e = threadIdx.x + u * kWT;
    r[u] = (e < tot) ? M[e] : T(0);
  }
  if (threadIdx.x < 2 * kMaxSide) {  // each circulant row twice over (kron_transform)
    const int t = threadIdx.x, tx = t % a.Lx, ty = t % a.Ly, tx1 = (t + 1) % a.Lx, ty1 = (t + 1) % a.Ly;
    kron_put_tap(s.tx, t, a.taps.ex[tx]);
    kron_put_tap(s.ty, t, a.taps.ey[ty]);
    kron_put_tap(s.txs, t, a.taps.ex[tx1]);
    kron_put_tap(s.tys, t, a.taps.ey[ty1]);
    kron_put_tap(taps2, t, a.taps.exi[tx]);
    kron_put_tap(taps2 + 2 * kMaxSide, t, a.taps.eyi[ty]);
    kron_put_tap(taps2 + 4 * kMaxSide, t, a.taps.exi[tx1]);
    kron_put_tap(taps2 + 6 * kMaxSide, t, a.taps.eyi[ty1]);
  }
  const T up = static_cast<T>(a.ec), dn = static_cast<T>(a.emc);
  const int8_t* f = a.field + (static_cast<size_t>(b) * a.L + a.l0_first) * N;
  for (int i = threadIdx.x; i < N; i += kWT) {
    const bool plus = f[i] > 0;
    s.sc[i] = plus ? up : dn;
    sc2[i] = plus ? dn : up;
  }
  __syncthreads();
  for (int e0 = threadIdx.x; e0 < tot; e0 += kU * kWT) {
    if (e0 >= kU * kWT)
#pragma unroll
      for (int u = 0; u < kU; ++u) r[u] = (e0 + u * kWT < tot) ? M[e0 + u * kWT] : T(0);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = e0 + u * kWT;
      if (e < tot) {
        const int i = e / N, j = e - i * N;
        T val = r[u];
        val *= s.sc[i];
        s.v[j * ld + i] = val;
      }
    }
  }
  __syncthreads();
  kron_transform(s.v, s.tmp, N, ld, a.Lx, a.Ly, N, s.tx, s.ty, s.txs, s.tys, (const T*)nullptr,
                 (const T*)nullptr);
  for (int e = threadIdx.x; e < tot; e += kWT) {
    const int i = e / N, j = e - i * N;
    T val = s.v[j * ld + i];
    val *= sc2[j];
    s.tmp[i * ld + j] = val;
  }
  __syncthreads();
  kron_transform(s.tmp, s.v, N, ld, a.Lx, a.Ly, N, taps2, taps2 + 2 * kMaxSide, taps2 + 4 * kMaxSide,
                 taps2 + 6 * kMaxSide, (const T*)nullptr, (const T*)nullptr);
  for (int e = threadIdx.x; e < tot; e += kWT) {
    const int i = e / N, j = e - i * N;
    M[e] = s.tmp[i * ld + j];
  }
}

// ---------------------------------------------------------------------------
// Drift check: drift[c] = max(drift[c], max|Gw - G64| / max|G64|), then the
// working G is replaced by the stabilised one.  One CTA per chain.
// ---------------------------------------------------------------------------
// One cluster of kDriftCS CTAs per chain, each over an interleaved share of
// the elements: max |Gw - G64| and max |G64| are taken on the bit patterns of
// the absolute values (non-negative doubles order as integers), so the only
// FP64 work per element is the conversion and the difference; non-finite
// entries of G64 are left out of the maxima and flagged, an infinite
// difference counts, a NaN difference does not (as fmax would have it).  CTA 0 combines the
// partial maxima of the cluster through distributed shared memory.
constexpr int kDriftCS = 2;
template <typename T>
__global__ void __launch_bounds__(256) k_drift_reset(const double* G64, T* Gw, int N, double* drift,
                                                    int* status) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = static_cast<int>(cl.block_rank());
  const int c = blockIdx.x / kDriftCS;
  const size_t nn = static_cast<size_t>(N) * N;
  const double* g = G64 + c * nn;
  T* w = Gw + c * nn;
  unsigned long long md = 0ull, mg = 0ull;
  bool bad = false;
  constexpr unsigned long long kAbs = 0x7FFFFFFFFFFFFFFFull;
  for (size_t e = rank * blockDim.x + threadIdx.x; e < nn; e += kDriftCS * blockDim.x) {
    const double ge = g[e];
    const unsigned long long ga = static_cast<unsigned long long>(__double_as_longlong(ge)) & kAbs;
    if (ga >= 0x7FF0000000000000ull) {  // Inf or NaN
      bad = true;
    } else {
      const unsigned long long da =
          static_cast<unsigned long long>(__double_as_longlong(static_cast<double>(w[e]) - ge)) & kAbs;
      md = (da <= 0x7FF0000000000000ull && da > md) ? da : md;  // Inf counts, NaN not
      mg = ga > mg ? ga : mg;
    }
    w[e] = static_cast<T>(ge);
  }
  __shared__ unsigned long long s1[32], s2[32];
  __shared__ int sb;
  if (threadIdx.x == 0) sb = 0;
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long m1 = __shfl_xor_sync(0xFFFFFFFFu, md, o);
    const unsigned long long m2 = __shfl_xor_sync(0xFFFFFFFFu, mg, o);
    md = m1 > md ? m1 : md;
    mg = m2 > mg ? m2 : mg;
  }
  __syncthreads();
  if (bad) atomicOr(&sb, 1);
  if ((threadIdx.x & 31) == 0) {
    s1[threadIdx.x >> 5] = md;
    s2[threadIdx.x >> 5] = mg;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w2 = 1; w2 < static_cast<int>(blockDim.x >> 5); ++w2) {
      md = s1[w2] > md ? s1[w2] : md;
      mg = s2[w2] > mg ? s2[w2] : mg;
    }
    s1[0] = md;
    s2[0] = mg;
    if (sb) atomicExch(status, kDevNonFinite);
  }
  cl.sync();
  if (rank == 0 && threadIdx.x == 0) {
    for (int r = 1; r < kDriftCS; ++r) {
      const unsigned long long m1 = *cl.map_shared_rank(&s1[0], r);
      const unsigned long long m2 = *cl.map_shared_rank(&s2[0], r);
      md = m1 > md ? m1 : md;
      mg = m2 > mg ? m2 : mg;
    }
    const double mdd = __longlong_as_double(static_cast<long long>(md));
    const double mgd = __longlong_as_double(static_cast<long long>(mg));
    const double dr = mgd > 0.0 ? mdd / mgd : mdd;
    if (!(dr <= drift[c])) drift[c] = dr;
  }
  cl.sync();  // the peers' shared memory stays until CTA 0 has read it
}

// ---------------------------------------------------------------------------
// Equal-time observables of one configuration from the stabilised G_up
// (G_dn = I - P G_up^T P):  n = (1/N) sum_i [(1 - G_ii) + G_ii],
// docc = (1/N) sum_i (1 - G_ii) G_ii,
// ekin = (1/N) sum_sigma sum_ij K_ij <c^dag_i c_j> = (2t/N) sum_j sum_delta G_{j, j+delta},
// and the translation-averaged spin correlation of Sec. 4 (Fig. 5),
// C(r) = (1/N) sum_i <S^z_i S^z_{i+r}>, S^z = (n_up - n_dn)/2, accumulated into
// spin[c][r], r = dx + Lx dy.  Wick's theorem per spin with G_dn = I - P G_up^T P
// gives, for a = G_ij, b = G_ji, d = delta_ij, p = p_i p_j = (-1)^(dx+dy) (even
// sides) and m_i = n_i,up - n_i,dn = 1 - 2 G_ii:
//   4 <S^z_i S^z_j> = m_i m_j + (d - b) a + p a (d - p b)
// (spin-up exchange, then spin-down exchange).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_observables(const double* G64, int Lx, int Ly, double t,
                                                    double* obs, double* spin) {
  const int c = blockIdx.x;
  const int N = Lx * Ly;
  const double* G = G64 + static_cast<size_t>(c) * N * N;
  __shared__ double m[kMaxN];
  for (int i = threadIdx.x; i < N; i += blockDim.x) m[i] = 1.0 - 2.0 * G[static_cast<size_t>(i) * N + i];
  __syncthreads();
  for (int r = threadIdx.x; r < N; r += blockDim.x) {
    const int dx = r % Lx, dy = r / Lx;
    const double p = ((dx + dy) & 1) ? -1.0 : 1.0;
    double acc = 0.0;
    int y = 0, yj = dy;
    for (; y < Ly; ++y) {
      const int row0 = Lx * y, rowj = Lx * yj;
#pragma unroll 4
      for (int x = 0; x < Lx; ++x) {
        const int xj = (x + dx < Lx) ? x + dx : x + dx - Lx;
        const int i = row0 + x, j = rowj + xj;
        const double a = G[static_cast<size_t>(i) * N + j];
        const double b = G[static_cast<size_t>(j) * N + i];
        const double d = (i == j) ? 1.0 : 0.0;
        acc += m[i] * m[j] + (d - b) * a + p * a * (d - p * b);
      }
      yj = (yj + 1 == Ly) ? 0 : yj + 1;
    }
    spin[static_cast<size_t>(c) * N + r] += acc / (4.0 * N);
  }
  double n = 0.0, dc = 0.0, ek = 0.0;
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    const double g = G[static_cast<size_t>(j) * N + j];
    n += (1.0 - g) + g;
    dc += (1.0 - g) * g;
    const int x = j % Lx, y = j / Lx;
    const int nb[4] = {(x + 1) % Lx + Lx * y, (x + Lx - 1) % Lx + Lx * y, x + Lx * ((y + 1) % Ly),
                       x + Lx * ((y + Ly - 1) % Ly)};
    for (int q = 0; q < 4; ++q) ek += G[static_cast<size_t>(j) * N + nb[q]];
  }
  __shared__ double sm[3][32];
  for (int o = 16; o > 0; o >>= 1) {
    n += __shfl_xor_sync(0xFFFFFFFFu, n, o);
    dc += __shfl_xor_sync(0xFFFFFFFFu, dc, o);
    ek += __shfl_xor_sync(0xFFFFFFFFu, ek, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sm[0][threadIdx.x >> 5] = n;
    sm[1][threadIdx.x >> 5] = dc;
    sm[2][threadIdx.x >> 5] = ek;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) {
      n += sm[0][w];
      dc += sm[1][w];
      ek += sm[2][w];
    }
    double* o = obs + static_cast<size_t>(c) * 4;
    o[0] += n / N;
    o[1] += dc / N;
    o[2] += 2.0 * t * ek / N;
    o[3] += 1.0;
  }
}

// ---------------------------------------------------------------------------
// Correlation length of Sec. 4 (Fig. 5): least-squares line through
// (|r|, ln c(r)), c(r) = (-1)^(dx+dy) C(r) the staggered correlation,
// |r| = sqrt(min(dx, Lx-dx)^2 + min(dy, Ly-dy)^2), over 0 < |r| <= dmax and
// c(r) > 0; xi = -1/slope (+inf for a slope >= 0, nan below two distinct
// distances).  C(r) = spin[c][r] / obs[c][3] for block c < C; block C takes
// the chain average sum_c spin[c][r] / sum_c obs[c][3].  One thread per r.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_corr_length(const double* spin, const double* obs, int C,
                                                    int Lx, int Ly, double dmax, double* out) {
  const int b = blockIdx.x, N = Lx * Ly;
  __shared__ double cnt_sh;
  if (threadIdx.x == 0) {
    double cnt = 0.0;
    if (b < C) {
      cnt = obs[static_cast<size_t>(b) * 4 + 3];
    } else {
      for (int c = 0; c < C; ++c) cnt += obs[static_cast<size_t>(c) * 4 + 3];
    }
    cnt_sh = cnt;
  }
  __syncthreads();
  double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};  // n, S_d, S_y, S_dd, S_dy
  double dmin = CUDART_INF, dmaxp = -1.0;     // smallest / largest distance used
  for (int r = threadIdx.x; r < N; r += blockDim.x) {
    double v = 0.0;
    if (b < C) {
      v = spin[static_cast<size_t>(b) * N + r];
    } else {
      for (int c = 0; c < C; ++c) v += spin[static_cast<size_t>(c) * N + r];
    }
    const int dx = r % Lx, dy = r / Lx;
    const double cr = (((dx + dy) & 1) ? -v : v) / cnt_sh;
    const int ax = min(dx, Lx - dx), ay = min(dy, Ly - dy);
    const double d = sqrt(static_cast<double>(ax * ax + ay * ay));
    if (d > 0.0 && d <= dmax && cr > 0.0) {
      const double y = log(cr);
      s[0] += 1.0;
      s[1] += d;
      s[2] += y;
      s[3] += d * d;
      s[4] += d * y;
      dmin = fmin(dmin, d);
      dmaxp = fmax(dmaxp, d);
    }
  }
  __shared__ double red[8][7];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int q = 0; q < 5; ++q) s[q] += __shfl_xor_sync(0xFFFFFFFFu, s[q], o);
    dmin = fmin(dmin, __shfl_xor_sync(0xFFFFFFFFu, dmin, o));
    dmaxp = fmax(dmaxp, __shfl_xor_sync(0xFFFFFFFFu, dmaxp, o));
  }
  if (lane == 0) {
    for (int q = 0; q < 5; ++q) red[w][q] = s[q];
    red[w][5] = dmin;
    red[w][6] = dmaxp;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int nw = blockDim.x >> 5;
    double t[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    double lo = CUDART_INF, hi = -1.0;
    for (int q = 0; q < nw; ++q) {
      for (int k = 0; k < 5; ++k) t[k] += red[q][k];
      lo = fmin(lo, red[q][5]);
      hi = fmax(hi, red[q][6]);
    }
    double xi = CUDART_NAN;
    const double den = t[0] * t[3] - t[1] * t[1];
    if (t[0] >= 2.0 && hi > lo && den > 0.0) {
      const double slope = (t[0] * t[4] - t[1] * t[2]) / den;
      xi = (slope < 0.0) ? -1.0 / slope : CUDART_INF;
    }
    out[b] = xi;
  }
}

// ---------------------------------------------------------------------------
// Host launch wrappers.
// ---------------------------------------------------------------------------
cudaError_t launch_init_field(int8_t* field, int C, int L, int N, int chain0, uint64_t seed,
                              cudaStream_t st) {
  const long long total = static_cast<long long>(C) * L * N;
  const int blocks = static_cast<int>(std::min<long long>((total + 255) / 256, kSMs * 16));
  k_init_field<<<blocks, 256, 0, st>>>(field, C, L, N, chain0, static_cast<uint32_t>(seed),
                                       static_cast<uint32_t>(seed >> 32));
  return cudaGetLastError();
}

template <typename T>
size_t metropolis_smem(int N, int k) {
  const int NP = ((N + 31) / 32) * 32;
  return static_cast<size_t>(NP) * (sizeof(double) + sizeof(float)) + 2ull * k * NP * sizeof(T) +
         static_cast<size_t>(NP) * (sizeof(T) + sizeof(float) + sizeof(int)) +
         static_cast<size_t>(kWin) * (NP + 1) * sizeof(T) +
         (std::is_same<T, float>::value ? static_cast<size_t>(kRing) * NP * sizeof(T) : 0);
}

template <typename T>
cudaError_t launch_metropolis(T* G, int8_t* field, int C, const MetroArgs& a, cudaStream_t st) {
  const int NP = ((a.N + 31) / 32) * 32;
  const int threads = NP * kHalves + (kScalarWarp<T>() ? 32 : 0);
  const size_t sm = metropolis_smem<T>(a.N, a.k);
  cudaError_t e = cudaFuncSetAttribute(k_metropolis<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  if (a.cs <= 1) {
    k_metropolis<T><<<C, threads, sm, st>>>(G, field, a);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C * a.cs, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = a.cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_metropolis<T>, G, field, a);
}

template <typename T>
size_t kron_smem(int N, int nv) {
  return (2ull * nv * (N + 1) + 8 * kMaxSide + N) * sizeof(T);
}

template <typename T>
cudaError_t launch_kron_rows(const T* in, T* out, int batch, const KronArgs& a, cudaStream_t st) {
  const size_t sm = kron_smem<T>(a.N, a.nv);
  cudaError_t e = cudaFuncSetAttribute(k_kron_rows<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  dim3 grid((a.N + a.nv - 1) / a.nv, batch);
  k_kron_rows<T><<<grid, 256, sm, st>>>(in, out, a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_kron_cols(T* X, int batch, const KronArgs& a, cudaStream_t st) {
  const size_t sm = kron_smem<T>(a.N, a.nv);
  cudaError_t e = cudaFuncSetAttribute(k_kron_cols<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  dim3 grid((a.N + a.nv - 1) / a.nv, batch);
  k_kron_cols<T><<<grid, 256, sm, st>>>(X, a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wrap_smem(T* X, int batch, const KronArgs& a, cudaStream_t st) {
  const size_t sm = (2ull * a.N * (a.N + 1) + 16 * kMaxSide + 2 * a.N) * sizeof(T);
  cudaError_t e = cudaFuncSetAttribute(k_wrap_smem<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sm));
  if (e != cudaSuccess) return e;
  k_wrap_smem<T><<<batch, kWT, sm, st>>>(X, a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_drift_reset(const double* G64, T* Gw, int C, int N, double* drift, int* status,
                               cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C * kDriftCS, 1, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kDriftCS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_drift_reset<T>, G64, Gw, N, drift, status);
}

cudaError_t launch_observables(const double* G64, int C, int Lx, int Ly, double t, double* obs,
                               double* spin, cudaStream_t st) {
  k_observables<<<C, 256, 0, st>>>(G64, Lx, Ly, t, obs, spin);
  return cudaGetLastError();
}

cudaError_t launch_corr_length(const double* spin, const double* obs, int C, int Lx, int Ly,
                               double dmax, double* out, cudaStream_t st) {
  k_corr_length<<<C + 1, 256, 0, st>>>(spin, obs, C, Lx, Ly, dmax, out);
  return cudaGetLastError();
}

#define DQMC_INST(T)                                                                              \
  template cudaError_t launch_metropolis<T>(T*, int8_t*, int, const MetroArgs&, cudaStream_t);   \
  template cudaError_t launch_kron_rows<T>(const T*, T*, int, const KronArgs&, cudaStream_t);    \
  template cudaError_t launch_kron_cols<T>(T*, int, const KronArgs&, cudaStream_t);              \
  template cudaError_t launch_wrap_smem<T>(T*, int, const KronArgs&, cudaStream_t);              \
  template cudaError_t launch_drift_reset<T>(const double*, T*, int, int, double*, int*,         \
                                             cudaStream_t);                                      \
  template size_t metropolis_smem<T>(int, int);
DQMC_INST(double)
DQMC_INST(float)
DQMC_INST(df32)
#undef DQMC_INST

}  // namespace dqmc
