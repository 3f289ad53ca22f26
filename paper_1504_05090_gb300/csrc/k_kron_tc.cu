// Kronecker products with exp(-+dtau K) = E_y (x) E_x of Eq. (2) on the
// tcgen05 tensor cores, for the FP64 UDV stack products X = B_l ... B_1 (U D)
// (Sec. 2: the O(Lambda N^3) stabilised matrix work behind Eq. (3)).
//
// A vector v of length N = Lx Ly is the Ly x Lx grid V[y][x] = v[x + Lx y],
// and E v = E_y V E_x^T with the circulant E_x[x][x'] = ex[(x - x') mod Lx].
// Eight (in general 128 / max(Lx, Ly)) vectors of one matrix stay in shared
// memory for all the slices of a call.  Per slice:
//   x step: rows (vector, y) of length Lx times E_x^T      (M = 128, N = K = 16)
//   y step: rows (vector, x) of length Ly times E_y^T      (M = 128, N = K = 16)
// each one digit-sliced product in integer arithmetic: every row of the left
// operand and the taps are aligned to their largest exponent (55 bits) and cut
// into seven signed 8-bit digits, -128 .. 127, exact in BF16; the 28 digit
// products with p + q <= 6 accumulate in seven FP32 TMEM accumulators (sums of
// 16 products of two digits: exact), and the epilogue puts them together in one
// 64-bit integer and rounds that to FP64.  What is left out, the products with
// p + q = 7 of balanced digits, is below that of eight unsigned 7-bit digits
// with p + q = 8, which need 36 products.  Rows and columns past Lx, Ly are
// zero padding.  The diagonal factor e^{+-c s_l} is an FP64 product per
// element, taken with the load of the x step (B, B^{-T}) or the store of the y
// step (B^T).
//
// What bounds it: the integer and FP32 instructions of the split and the
// recombination (about 80 per element and step).  The FP64 pipe, which issues a
// warp instruction in 64 to 76 clocks, is left to the diagonal factor: digits,
// sums and the rounding use integer and FP32 instructions only, no conversion
// instruction (15 lanes per clock and SM) among them.  The vectors lie in
// shared memory with rows of odd length, so that lanes along y and along x both
// find different banks.  One launch of the 16 x 16 sweep (64 chains x 256
// vectors x 10 slices): 1.32 ms with eight 7-bit digits, FP64 conversions and
// rows of Lx, 0.61 ms now.
//
// Eight 7-bit digits (TcDigits8: 53 bits, truncated, 36 products, rounded once
// from two 64-bit integers) stay for the groups whose stack steps stretch a
// vector so far that single entries of G(tau) carry the rounding of a step
// amplified to 1e-8 and more (long_step in dqmc.cu): their numbers depend on
// every rounding and are kept as they are.
#include "common.cuh"
#include "kernels.h"
#include "oz_compose.cuh"

namespace dqmc {
namespace {

constexpr int kR = 128;     // rows of one product (TMEM lanes)
constexpr int kK = 16;      // inner dimension (padded side)
constexpr int kTC = 128;    // threads
constexpr long long kWaitLimit = 1LL << 26;
constexpr int kASlice = kR * kK * 2;   // bytes of one digit slice of the rows (4 KB)
constexpr int kBSlice = kK * kK * 2;   // of the taps (512 B)

__device__ __forceinline__ uint32_t tc_smem(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// No-swizzle K-major descriptor: core matrices of 8 rows x 16 bytes, the next
// one along K 128 bytes on, the next 8 rows 256 bytes on (K = 16).
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) {
  constexpr uint32_t lbo = 128, sbo = 256;
  return static_cast<uint64_t>((addr >> 4) & 0x3FFF) |
         (static_cast<uint64_t>((lbo >> 4) & 0x3FFF) << 16) |
         (static_cast<uint64_t>((sbo >> 4) & 0x3FFF) << 32) | (1ULL << 46);
}

// Element offset of (row r, k) in one digit slice.
__device__ __forceinline__ int tc_off(int r, int k) {
  return (r >> 3) * (kK / 8 * 64) + (k >> 3) * 64 + (r & 7) * 8 + (k & 7);
}

__device__ __forceinline__ bool tc_wait(uint64_t* bar, int parity) {
  uint32_t done = 0;
  for (long long it = 0; it < kWaitLimit && !done; ++it)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(tc_smem(bar)), "r"(parity));
  return done != 0;
}

// Two floats with at most eight significant bits as a BF16 pair: their high
// halves.
__device__ __forceinline__ uint32_t tc_pack(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// The number W 2^(e - 2102), W the integer sum of the accumulators, rounded to
// FP64 (W's leading 53 bits; e: the sum of the two biased exponents).
__device__ __forceinline__ double tc_compose(long long W, int e) {
  const unsigned long long x = static_cast<unsigned long long>(W < 0 ? -W : W);
  const int lz = __clzll(static_cast<long long>(x));
  const unsigned long long m = ((x << (lz - 1)) + 0x200u) >> 10;  // 2^52 .. 2^53
  const int ef = e - 1016 - lz;
  if (x != 0 && (ef < 1 || ef > 2045)) return ldexp(static_cast<double>(W), e - 2102);
  unsigned long long r = (static_cast<unsigned long long>(ef - 1) << 52) + m;
  if (W < 0) r |= 0x8000000000000000ULL;
  return (x == 0) ? 0.0 : __longlong_as_double(static_cast<long long>(r));
}

// Seven balanced digits of eight bits.
struct TcDigits7 {
  static constexpr int kS = 7;  // digit slices

  // Exponent to align a vector to: the largest biased exponent, one higher where
  // the leading seven bits of the significand are all ones, so that the top
  // digit of the aligned number, rounded up by the digits below it, stays below
  // 128.
  static __device__ __forceinline__ int expo(double x) {
    return ((__double2hiint(x) & 0x7FFFFFFF) + 0x4000) >> 20;
  }

  // x as the integer round-down(|x| 2^(1077 - emax)) with x's sign, below 2^55,
  // plus 128 in each of its seven bytes: byte 6 - p is then digit p plus 128.
  static __device__ __forceinline__ unsigned long long align(double x, int emax) {
    const long long bits = __double_as_longlong(x);
    const int E = static_cast<int>((bits >> 52) & 0x7FF);
    long long m = 0;
    if (E != 0) {  // zero and subnormal inputs contribute zero digits
      const unsigned long long mant =
          ((static_cast<unsigned long long>(bits) & ((1ULL << 52) - 1)) | (1ULL << 52)) << 2;
      const int sh = emax - E;
      m = (sh < 64) ? static_cast<long long>(mant >> sh) : 0LL;
      if (bits < 0) m = -m;
    }
    return static_cast<unsigned long long>(m) + 0x0080808080808080ULL;
  }

  // Digit p of an aligned number as a float: the byte in the low bits of 2^23,
  // minus 2^23 + 128.
  static __device__ __forceinline__ float digit(unsigned long long t, int p) {
    const uint32_t w = (p < 3) ? static_cast<uint32_t>(t >> 32) : static_cast<uint32_t>(t);
    const int byte = (p < 3) ? 2 - p : 6 - p;
    return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440u | byte)) - 8388736.0f;
  }

  // The result from the accumulators P_d, integers below 2^21, read off the low
  // bits of 1.5 2^23 + P_d (as P_d + kM): W = sum_d P_d 2^(44 - 8 d) (d = 6
  // rounded), below 2^63; ea, eb: the exponents of the two operands.
  static __device__ __forceinline__ double compose(const uint32_t (&acc)[kS], int ea, int eb) {
    constexpr uint32_t kM = 0x4B400000u;
    uint32_t u[kS];
#pragma unroll
    for (int d = 0; d < kS; ++d) u[d] = __float_as_uint(__uint_as_float(acc[d]) + 12582912.0f);
    const int a = static_cast<int>(u[0] * 256u + u[1] - kM * 257u);
    const int b = static_cast<int>(u[2] * 256u + u[3] - kM * 257u);
    const int c = static_cast<int>(u[4] * 256u + u[5] - kM * 257u);
    const int g = static_cast<int>(u[6] - kM);
    const long long W = ((static_cast<long long>(a) * 65536 + b) << 20) +
                        (static_cast<long long>(c) << 4) + ((g + 8) >> 4);
    return tc_compose(W, ea + eb);
  }
};

// Eight digits of seven bits (the last of four), of the magnitude with x's sign.
struct TcDigits8 {
  static constexpr int kS = 8;

  static __device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

  // the significand shifted down to emax, x's sign on top
  static __device__ __forceinline__ unsigned long long align(double x, int emax) {
    const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
    const int E = static_cast<int>((bits >> 52) & 0x7FF), sh = emax - E;
    unsigned long long al = 0ULL;
    if (E != 0 && sh < 64) al = ((bits & ((1ULL << 52) - 1)) | (1ULL << 52)) >> sh;
    return al | (bits & 0x8000000000000000ULL);
  }

  static __device__ __forceinline__ float digit(unsigned long long t, int p) {
    const uint32_t d = (p < 7) ? static_cast<uint32_t>(t >> (46 - 7 * p)) & 127u
                               : (static_cast<uint32_t>(t) & 15u) << 3;
    const uint32_t sign = static_cast<uint32_t>(t >> 32) & 0x80000000u;
    return __uint_as_float(__float_as_uint(__uint_as_float(0x4B000000u | d) - 8388608.0f) | sign);
  }

  // (hi + 2^-28 lo) 2^{e - 21} with e the sum of the operands' exponents less
  // 6 each, rounded once (FP64 products where it leaves the normal range)
  static __device__ __forceinline__ double compose(const uint32_t (&acc)[kS], int ea, int eb) {
    int n[kS];
#pragma unroll
    for (int d = 0; d < kS; ++d)
      n[d] = __float_as_int(__uint_as_float(acc[d]) + 12582912.0f) - 0x4B400000;
    long long hi = 0, lo = 0;
#pragma unroll
    for (int d = 0; d < 4; ++d) hi += static_cast<long long>(n[d]) * (1 << (7 * (3 - d)));
#pragma unroll
    for (int d = 4; d < kS; ++d) lo += static_cast<long long>(n[d]) * (1 << (7 * (7 - d)));
    const int fa = ea - 1029, fb = eb - 1029 - 21;
    bool ok;
    const double v = oz_compose(hi, lo, fa + fb, false, ok);
    if (ok) return v;
    return fma(static_cast<double>(lo), 0x1p-28, static_cast<double>(hi)) * ldexp(1.0, fa) * ldexp(1.0, fb);
  }
};

// Digits of the taps as the right operand: column j, inner index k,
// t[(j - k) mod n] for j, k < n (zero padding beyond); the columns hold the same
// taps, so they share one exponent, which is returned.
template <class Dg>
__device__ int tc_tap_digits(const double* t, int n, unsigned char* bs) {
  int emax = 0;
  for (int k = 0; k < n; ++k) emax = max(emax, Dg::expo(t[k]));
  for (int e = threadIdx.x; e < kK * kK; e += blockDim.x) {
    const int j = e / kK, k = e - j * kK;
    const unsigned long long v = Dg::align((j < n && k < n) ? t[(j - k + n) % n] : 0.0, emax);
    for (int p = 0; p < Dg::kS; ++p)
      reinterpret_cast<uint16_t*>(bs + p * kBSlice)[tc_off(j, k)] =
          static_cast<uint16_t>(__float_as_uint(Dg::digit(v, p)) >> 16);
  }
  return emax;
}

// Shared-memory state of one CTA of the tensor-core Kronecker kernels.
struct TcState {
  unsigned char* as;  // digit slices of the rows (kS x 4 KB)
  unsigned char* bx;  // digit slices of the taps along x (kS x 512 B)
  unsigned char* by;  // along y
  double* V;          // the CTA's vectors, element (vi, x, y) at vi VP + y LP + x
  double* sc;         // diagonal of the slice, (x, y) at y LP + x
  uint64_t* mbar;     // MMA completion
  int* fail;          // a bounded wait gave up
  int ex, ey;         // exponents of the taps
  int Lx, Ly, LP, VP;
  uint32_t tbase;     // TMEM accumulators (kS x 16 columns)
};

__host__ __device__ __forceinline__ int tc_pitch(int Lx) { return Lx | 1; }

template <class Dg>
__device__ __forceinline__ void tc_layout(TcState& s, unsigned char* sm, int nvpc, int Lx, int Ly) {
  s.as = sm;
  s.bx = s.as + Dg::kS * kASlice;
  s.by = s.bx + Dg::kS * kBSlice;
  s.Lx = Lx;
  s.Ly = Ly;
  s.LP = tc_pitch(Lx);
  s.VP = Ly * s.LP;
  s.V = reinterpret_cast<double*>(s.by + Dg::kS * kBSlice);
  s.sc = s.V + nvpc * s.VP;
}

// TMEM, barrier and the digits of the taps of E_x, E_y (kind: E or E^{-1}).
template <class Dg>
__device__ void tc_setup(TcState& s, uint32_t* tmem_sh, const KronTaps& taps, bool inv, double* tx,
                         double* ty) {
  const int warp = threadIdx.x >> 5;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(
        tc_smem(tmem_sh)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(s.mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
    *s.fail = 0;
  }
  if (threadIdx.x < kMaxSide) {
    tx[threadIdx.x] = inv ? taps.exi[threadIdx.x] : taps.ex[threadIdx.x];
    ty[threadIdx.x] = inv ? taps.eyi[threadIdx.x] : taps.ey[threadIdx.x];
  }
  // zero digits of k = 8 .. 15, which sides of at most 8 never write
  for (int e = threadIdx.x; e < Dg::kS * kASlice / 16; e += blockDim.x)
    reinterpret_cast<uint4*>(s.as)[e] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  s.ex = tc_tap_digits<Dg>(tx, s.Lx, s.bx);
  s.ey = tc_tap_digits<Dg>(ty, s.Ly, s.by);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  s.tbase = *tmem_sh;
}

__device__ void tc_teardown(const TcState& s) {
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(s.tbase));
}

// One factor B on the nv vectors in s.V: the diagonal s.sc before the taps
// (post = false: B, B^{-T}) or after them (post = true: B^T), then the x and
// y steps as digit-sliced products.  All threads, which have synchronised since
// s.V and s.sc were written; false if a wait gave up.
template <class Dg>
__device__ bool tc_slice(TcState& s, bool post, int nv, int& phase) {
  constexpr int kS = Dg::kS;
  const int warp = threadIdx.x >> 5;
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((kK >> 3) << 17) | ((kR >> 4) << 24);
  const int r = threadIdx.x;  // the row of both products this thread owns
  const bool wide = max(s.Lx, s.Ly) > 8;
  for (int dir = 0; dir < 2; ++dir) {
    // row r: (vector, y) with elements x' (x step) or (vector, x) with y' (y step)
    const int side = dir == 0 ? s.Ly : s.Lx, klen = dir == 0 ? s.Lx : s.Ly;
    const int vi = r / side, o = r - vi * side;
    const bool live = vi < nv;
    const int base = dir == 0 ? o * s.LP : o, step = dir == 0 ? 1 : s.LP;
    double* v = s.V + vi * s.VP + base;
    const double* scp = s.sc + base;
    int emax = 0;
    {
      double row[kK];
#pragma unroll
      for (int k = 0; k < kK; ++k) {
        double x = 0.0;
        if (live && k < klen) {
          x = v[k * step];
          if (!post && dir == 0) x *= scp[k];
        }
        row[k] = x;
        emax = max(emax, Dg::expo(x));
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        if (half == 1 && !wide) break;
        unsigned long long t[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) t[q] = Dg::align(row[half * 8 + q], emax);
#pragma unroll
        for (int p = 0; p < kS; ++p)
          *reinterpret_cast<uint4*>(s.as + p * kASlice + 2 * tc_off(r, half * 8)) =
              make_uint4(tc_pack(Dg::digit(t[0], p), Dg::digit(t[1], p)),
                         tc_pack(Dg::digit(t[2], p), Dg::digit(t[3], p)),
                         tc_pack(Dg::digit(t[4], p), Dg::digit(t[5], p)),
                         tc_pack(Dg::digit(t[6], p), Dg::digit(t[7], p)));
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const unsigned char* bs = dir == 0 ? s.bx : s.by;
    if (threadIdx.x == 0) {
      for (int d = 0; d < kS; ++d)
        for (int p = 0; p <= d; ++p) {
          const int q = d - p;
          const uint64_t ad = tc_desc(tc_smem(s.as + p * kASlice));
          const uint64_t bd = tc_desc(tc_smem(bs + q * kBSlice));
          const uint32_t acc = p > 0 ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred pa;\n setp.ne.u32 pa, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pa;\n}" ::"r"(s.tbase + d * kK),
              "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
        }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          tc_smem(s.mbar)));
    }
    if (!tc_wait(s.mbar, phase)) *s.fail = 1;
    phase ^= 1;
    const bool ok = __syncthreads_and(*s.fail == 0) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (!ok) return false;
    // recombination, eight columns at a time
    const int eb = dir == 0 ? s.ex : s.ey;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (half * 8 >= klen) break;
      uint32_t acc[kS][8];
#pragma unroll
      for (int d = 0; d < kS; ++d) {
        const uint32_t ta = s.tbase + (static_cast<uint32_t>(warp * 32) << 16) + d * kK + half * 8;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=r"(acc[d][0]), "=r"(acc[d][1]), "=r"(acc[d][2]), "=r"(acc[d][3]), "=r"(acc[d][4]),
              "=r"(acc[d][5]), "=r"(acc[d][6]), "=r"(acc[d][7])
            : "r"(ta));
      }
      asm volatile("tcgen05.wait::ld.sync.aligned;");
      if (live) {
#pragma unroll
        for (int jq = 0; jq < 8; ++jq) {
          const int j = half * 8 + jq;
          if (j >= klen) continue;
          uint32_t pd[kS];
#pragma unroll
          for (int d = 0; d < kS; ++d) pd[d] = acc[d][jq];
          double val = Dg::compose(pd, emax, eb);
          // rows are read above and written only here, each by its owner
          if (post && dir == 1) val *= scp[j * step];
          v[j * step] = val;
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
  }
  return true;
}

}  // namespace

// One CTA per (group of nvpc vectors, batch entry); the arguments and slice
// ranges are those of k_kron_rows<double>.
template <class Dg>
__global__ void __launch_bounds__(kTC) k_kron_tc(const double* in, double* out, KronArgs a,
                                                int nvpc, int* status) {
  const int b = blockIdx.y;
  int chain, first, count;
  chain = b / a.per_chain;
  if (a.cp) {
    const int blk = b - chain * a.per_chain;
    const int lo = a.cp[blk] + a.step, hi = a.cp[blk + 1];
    first = lo;
    count = (lo < hi) ? 1 : 0;
  } else {
    first = a.l0_first;
    count = a.n_slices;
  }
  const int N = a.N;
  const int v0 = blockIdx.x * nvpc;
  const int nv = min(nvpc, N - v0);
  extern __shared__ __align__(1024) unsigned char tc_sm[];
  __shared__ uint64_t mbar;
  __shared__ uint32_t tmem_sh;
  __shared__ int fail_sh;
  __shared__ double tx[kMaxSide], ty[kMaxSide];
  TcState s;
  tc_layout<Dg>(s, tc_sm, nvpc, a.Lx, a.Ly);
  s.mbar = &mbar;
  s.fail = &fail_sh;
  const double* src = in + static_cast<size_t>(b) * a.mat_stride;
  for (int e = threadIdx.x; e < nv * N; e += blockDim.x) {
    const int vi = e / N, i = e - vi * N, y = i / a.Lx;
    double val = src[static_cast<size_t>(v0) * N + e];
    if (a.vscale) val *= a.vscale[static_cast<size_t>(b) * a.vscale_stride + v0 + vi];
    s.V[vi * s.VP + y * s.LP + i - y * a.Lx] = val;
  }
  tc_setup<Dg>(s, &tmem_sh, a.taps, a.kind == kBIT, tx, ty);
  const double up = (a.kind == kBIT) ? a.emc : a.ec, dn = (a.kind == kBIT) ? a.ec : a.emc;
  const int8_t* f = a.field + static_cast<size_t>(chain) * a.L * N;
  int phase = 0;
  bool ok = true;
  for (int stp = 0; stp < count && ok; ++stp) {
    const int l0 = first + stp * a.dir;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const int y = i / a.Lx;
      s.sc[y * s.LP + i - y * a.Lx] = f[static_cast<size_t>(l0) * N + i] > 0 ? up : dn;
    }
    __syncthreads();
    ok = tc_slice<Dg>(s, a.kind == kBT, nv, phase);
  }
  if (!ok && threadIdx.x == 0) atomicExch(status, kDevTimeout);
  __syncthreads();
  double* dst = out + static_cast<size_t>(b) * a.out_stride;
  for (int e = threadIdx.x; e < nv * N; e += blockDim.x) {
    const int vi = e / N, i = e - vi * N, y = i / a.Lx;
    dst[static_cast<size_t>(v0) * N + e] = s.V[vi * s.VP + y * s.LP + i - y * a.Lx];
  }
  tc_teardown(s);
}

// Unequal-time propagation of k_gtau_propagate on the tensor cores: the rows
// of one stabilisation point's G(c,0)^T (kind B) or Y (kind B^{-T}) are
// propagated over the slices of its block, and after each slice every
// element is added to the bin of its separation (spin-up G(l,0) bins or Y
// bins of slice l): one thread per bin sums its element of each of the CTA's
// vectors and adds the sum to bins[chain][l][slot].
template <class Dg>
__global__ void __launch_bounds__(kTC) k_gtau_tc(const double* Xall, GtauArgs a, int nvpc,
                                                int* status) {
  const int b = blockIdx.y;
  const int chain = b / a.per_chain, blk = b - chain * a.per_chain;
  const int N = a.N;
  const int v0 = blockIdx.x * nvpc;
  const int nv = min(nvpc, N - v0);
  const int lo = a.cp[blk], hi = a.cp[blk + 1];
  extern __shared__ __align__(1024) unsigned char tc_sm[];
  __shared__ uint64_t mbar;
  __shared__ uint32_t tmem_sh;
  __shared__ int fail_sh;
  __shared__ double tx[kMaxSide], ty[kMaxSide];
  TcState s;
  tc_layout<Dg>(s, tc_sm, nvpc, a.Lx, a.Ly);
  s.mbar = &mbar;
  s.fail = &fail_sh;
  const double* X = Xall + static_cast<size_t>(b) * a.mat_stride;
  for (int e = threadIdx.x; e < nv * N; e += blockDim.x) {
    const int vi = e / N, i = e - vi * N, y = i / a.Lx;
    s.V[vi * s.VP + y * s.LP + i - y * a.Lx] = X[static_cast<size_t>(v0) * N + e];
  }
  tc_setup<Dg>(s, &tmem_sh, a.taps, a.kind == kBIT, tx, ty);
  const int8_t* f = a.field + static_cast<size_t>(chain) * a.L * N;
  const double up = (a.kind == kBIT) ? a.emc : a.ec, dn = (a.kind == kBIT) ? a.ec : a.emc;
  int phase = 0;
  bool ok = true;
  for (int l = lo; l < hi && ok; ++l) {
    if (l > lo) {
      for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int y = i / a.Lx;
        s.sc[y * s.LP + i - y * a.Lx] = f[static_cast<size_t>(l - 1) * N + i] > 0 ? up : dn;
      }
      __syncthreads();
      ok = tc_slice<Dg>(s, false, nv, phase);
      if (!ok) break;
    }
    double* out = a.bins + ((static_cast<size_t>(chain) * (a.L + 1) + l) * 2 + a.bin_slot) * N;
    for (int r = threadIdx.x; r < N; r += blockDim.x) {
      const int ry = r / a.Lx, rx = r - ry * a.Lx;
      int qy = v0 / a.Lx, qx = v0 - qy * a.Lx;
      double sum = 0.0;
      for (int vi = 0; vi < nv; ++vi) {
        // vec_is_col: r = r_el - r_q, else r = r_q - r_el
        int x = a.vec_is_col ? qx + rx : qx - rx, y = a.vec_is_col ? qy + ry : qy - ry;
        if (x < 0) x += a.Lx;
        if (x >= a.Lx) x -= a.Lx;
        if (y < 0) y += a.Ly;
        if (y >= a.Ly) y -= a.Ly;
        sum += s.V[vi * s.VP + y * s.LP + x];
        if (++qx == a.Lx) {
          qx = 0;
          ++qy;
        }
      }
      atomicAdd(&out[r], sum);
    }
    __syncthreads();
  }
  if (!ok && threadIdx.x == 0) atomicExch(status, kDevTimeout);
  tc_teardown(s);
}

int kron_tc_vectors(int Lx, int Ly) { return kR / max(Lx, Ly); }

template <class Dg>
static size_t tc_bytes(int nvpc, int Lx, int Ly) {
  return static_cast<size_t>(Dg::kS) * kASlice + 2ull * Dg::kS * kBSlice +
         static_cast<size_t>(nvpc + 1) * Ly * tc_pitch(Lx) * sizeof(double);
}

template <class Dg>
static cudaError_t tc_launch_kron(const double* in, double* out, int batch, const KronArgs& a,
                                  int* status, cudaStream_t st) {
  const int nvpc = kron_tc_vectors(a.Lx, a.Ly);
  const size_t smem = tc_bytes<Dg>(nvpc, a.Lx, a.Ly);
  cudaError_t e = cudaFuncSetAttribute(k_kron_tc<Dg>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  dim3 grid((a.N + nvpc - 1) / nvpc, batch);
  k_kron_tc<Dg><<<grid, kTC, smem, st>>>(in, out, a, nvpc, status);
  return cudaGetLastError();
}

template <class Dg>
static cudaError_t tc_launch_gtau(const double* X, int batch, const GtauArgs& a, int* status,
                                  cudaStream_t st) {
  const int nvpc = kron_tc_vectors(a.Lx, a.Ly);
  const size_t smem = tc_bytes<Dg>(nvpc, a.Lx, a.Ly);
  cudaError_t e = cudaFuncSetAttribute(k_gtau_tc<Dg>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  dim3 grid((a.N + nvpc - 1) / nvpc, batch);
  k_gtau_tc<Dg><<<grid, kTC, smem, st>>>(X, a, nvpc, status);
  return cudaGetLastError();
}

cudaError_t launch_kron_tc(const double* in, double* out, int batch, const KronArgs& a, int* status,
                           cudaStream_t st) {
  if (a.Lx > kK || a.Ly > kK) return cudaErrorInvalidValue;
  return a.digits8 ? tc_launch_kron<TcDigits8>(in, out, batch, a, status, st)
                   : tc_launch_kron<TcDigits7>(in, out, batch, a, status, st);
}

cudaError_t launch_gtau_tc(const double* X, int batch, const GtauArgs& a, int* status,
                           cudaStream_t st) {
  if (a.Lx > kK || a.Ly > kK) return cudaErrorInvalidValue;
  return a.digits8 ? tc_launch_gtau<TcDigits8>(X, batch, a, status, st)
                   : tc_launch_gtau<TcDigits7>(X, batch, a, status, st);
}

}  // namespace dqmc
