// Device code shared by the class-sorted H|psi> kernels (paper Eq. (2)):
// the kernel parameter block, the arithmetic policies (FP32, FP64, exact
// 64-bit fixed point, fixed-point sums with FP64 weights), the fixed-point
// <-> FP64 conversions done by
// bit manipulation.
#pragma once

#include <cstdint>
#include <cstring>

#include "ed_internal.h"

namespace edk {
struct P3 {
  Dev3 t;
  const DevBlock* blocks;
  int nblk;
  int ncross;
  const double* xd;  // FP64 input of a split diagonal (PI64S)
};

// kSplit: the diagonal is not part of the integer sums; the last store of an
// element adds it in FP64 from the FP64 input (P3::xd).
// Policy types: S = staged / gathered values (and per-class sums), Y = the
// partial output kept in y between the passes, A = the accumulator, D = the
// diagonal, W = the per-class weights; dmul / wmul combine them.
struct PF32 {
  static constexpr bool kSplit = false;
  using S = float;
  using Y = float;
  using A = float;
  using D = float;
  using W = float;
  __device__ static float dmul(float d, float x) { return d * x; }
  __device__ static float wmul(float w, float s) { return w * s; }
  __device__ static float w(const Dev3& t, int c) { return t.w32[c]; }
  __device__ static float bw(const Dev3& t, int k) { return t.bond_w32[k]; }
  __device__ static float diagA(const Dev3& t, long long gA) { return t.A_d32[gA] + t.dc0_32; }
  __device__ static float diagB(const Dev3& t, long long gB) { return t.B_d32[gB]; }
  __device__ static float vab(const Dev3& t, unsigned z) {
    float v = 0.f;
    for (int q = 0; q < t.ncls_d; ++q) v += t.dw32[q] * (float)__popc(z & t.dmask[q]);
    return v;
  }
  __device__ static float diag(const Dev3& t, long long gA, long long gB, unsigned z) {
    float v = t.A_d32[gA] + t.B_d32[gB] + t.dc0_32;
    for (int q = 0; q < t.ncls_d; ++q) v += t.dw32[q] * (float)__popc(z & t.dmask[q]);
    return v;
  }
};
struct PF64 {
  static constexpr bool kSplit = false;
  using S = double;
  using Y = double;
  using A = double;
  using D = double;
  using W = double;
  __device__ static double dmul(double d, double x) { return d * x; }
  __device__ static double wmul(double w, double s) { return w * s; }
  __device__ static double w(const Dev3& t, int c) { return t.w64[c]; }
  __device__ static double bw(const Dev3& t, int k) { return t.bond_w64[k]; }
  __device__ static double diagA(const Dev3& t, long long gA) { return t.A_d64[gA] + t.dc0_64; }
  __device__ static double diagB(const Dev3& t, long long gB) { return t.B_d64[gB]; }
  __device__ static double vab(const Dev3& t, unsigned z) {
    double v = 0.0;
    for (int q = 0; q < t.ncls_d; ++q) v += t.dw64[q] * (double)__popc(z & t.dmask[q]);
    return v;
  }
  __device__ static double diag(const Dev3& t, long long gA, long long gB, unsigned z) {
    double v = t.A_d64[gA] + t.B_d64[gB] + t.dc0_64;
    for (int q = 0; q < t.ncls_d; ++q) v += t.dw64[q] * (double)__popc(z & t.dmask[q]);
    return v;
  }
};
// The integer diagonal and weights are 32-bit: every weight is at most 2^24 in
// magnitude (dyadic couplings), the diagonal a sum of three such terms and 32
// such weights, so a product with x takes a 64 x 32-bit multiplication.
struct PI64 {
  static constexpr bool kSplit = false;
  using S = long long;
  using Y = long long;
  using A = long long;
  using D = int;
  using W = int;
  __device__ static long long dmul(int d, long long x) { return d * x; }
  __device__ static long long wmul(int w, long long s) { return w * s; }
  __device__ static int w(const Dev3& t, int c) { return (int)t.wI[c]; }
  __device__ static int bw(const Dev3& t, int k) { return (int)t.bond_wI[k]; }
  __device__ static int diagA(const Dev3& t, long long gA) { return t.A_dI[gA] + (int)t.dc0_I; }
  __device__ static int diagB(const Dev3& t, long long gB) { return t.B_dI[gB]; }
  __device__ static int vab(const Dev3& t, unsigned z) {
    int v = 0;
    for (int q = 0; q < t.ncls_d; ++q) v += (int)t.dwI[q] * __popc(z & t.dmask[q]);
    return v;
  }
};

// dyadic off-diagonal terms with a diagonal that is not (disordered on-site
// energies): the integer passes take the off-diagonal terms
struct PI64S : PI64 {
  static constexpr bool kSplit = true;
};

// Fixed-point gathers with FP64 weights (models whose couplings are not
// dyadic): x is summed exactly per value class on the integer pipe as in
// PI64, and each class sum is multiplied by its FP64 weight once per
// element, the diagonal likewise (a few FP64 operations per element instead
// of one per matrix element).  The partial result between the passes is FP64
// in fixed-point units; the last store scales it by one power of two.
struct PC64 {
  static constexpr bool kSplit = false;
  using S = long long;
  using Y = double;
  using A = double;
  using D = double;
  using W = double;
  __device__ static double dmul(double d, long long x) { return d * (double)x; }
  __device__ static double wmul(double w, long long s) { return w * (double)s; }
  __device__ static double w(const Dev3& t, int c) { return t.w64[c]; }
  __device__ static double bw(const Dev3& t, int k) { return t.bond_w64[k]; }
  __device__ static double diagA(const Dev3& t, long long gA) { return t.A_d64[gA] + t.dc0_64; }
  __device__ static double diagB(const Dev3& t, long long gB) { return t.B_d64[gB]; }
  __device__ static double vab(const Dev3& t, unsigned z) { return PF64::vab(t, z); }
};

// 128-bit two's-complement integer: sums of products of 64-bit integers
struct I128 {
  unsigned long long lo;
  long long hi;
};
__host__ __device__ __forceinline__ I128 operator+(I128 a, I128 b) {
  I128 r;
  r.lo = a.lo + b.lo;
  r.hi = a.hi + b.hi + (r.lo < a.lo ? 1 : 0);
  return r;
}
__host__ __device__ __forceinline__ I128 mul_wide(long long a, long long b) {
  I128 r;
  r.lo = (unsigned long long)a * (unsigned long long)b;
#ifdef __CUDA_ARCH__
  r.hi = __mul64hi(a, b);
#else
  r.hi = (long long)(((__int128)a * (__int128)b) >> 64);
#endif
  return r;
}

// Wide integer weights (models whose couplings are not dyadic): every
// coupling and diagonal value is an FP64 number, i.e. an integer multiple of
// 2^-q_shift for one q_shift that covers them all; the class sums of the
// fixed-point x are multiplied by these 64-bit integer weights into an exact
// 128-bit sum, rounded once to FP64 per pass by bit manipulation (no FP64
// instruction per matrix element).  The row pass's partial result is kept in
// y as FP64 and the panel pass adds its own rounded sum to it.
struct AccW {
  I128 s;    // exact sum of this pass
  double p;  // partial result of the row pass (panel pass only)
  __device__ AccW() {}
  __device__ AccW(I128 v) : s(v), p(0.0) {}
  __device__ AccW(double v) : p(v) { s.lo = 0ull; s.hi = 0ll; }
  __device__ AccW& operator+=(I128 v) {
    s = s + v;
    return *this;
  }
};
struct PW {
  static constexpr bool kSplit = false;
  using S = long long;
  using Y = double;
  using A = AccW;
  using D = long long;
  using W = long long;
  __device__ static I128 dmul(long long d, long long x) { return mul_wide(d, x); }
  __device__ static I128 wmul(long long w, long long s) { return mul_wide(w, s); }
  __device__ static long long w(const Dev3& t, int c) { return t.wI[c]; }
  __device__ static long long bw(const Dev3& t, int k) { return t.bond_wI[k]; }
  __device__ static long long diagA(const Dev3& t, long long gA) { return t.A_dW[gA] + t.dc0_I; }
  __device__ static long long diagB(const Dev3& t, long long gB) { return t.B_dW[gB]; }
  __device__ static long long vab(const Dev3& t, unsigned z) {
    long long v = 0;
    for (int q = 0; q < t.ncls_d; ++q) v += t.dwI[q] * (long long)__popc(z & t.dmask[q]);
    return v;
  }
};

// ---------------------------------------------------------------- fixed point <-> FP64 by bit manipulation

__host__ __device__ __forceinline__ unsigned long long f64_bits(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(v);
#else
  unsigned long long u;
  memcpy(&u, &v, 8);
  return u;
#endif
}
__host__ __device__ __forceinline__ double bits_f64(unsigned long long u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double v;
  memcpy(&v, &u, 8);
  return v;
#endif
}
__host__ __device__ __forceinline__ int clz64(unsigned long long u) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)u);
#else
  return __builtin_clzll(u);
#endif
}

// round(v * 2^sh_base) (ties away from zero) for |v| < 2^E, sh_base = P - E
__host__ __device__ __forceinline__ long long to_fixed(double v, int sh_base) {
  const unsigned long long u = f64_bits(v);
  const int s = (int)(u >> 63);
  int e = (int)((u >> 52) & 0x7ffull);
  unsigned long long m = u & 0xFFFFFFFFFFFFFull;
  if (e == 0) {
    if (m == 0) return 0;
    e = 1;
  } else {
    m |= 1ull << 52;
  }
  const int sh = e - 1075 + sh_base;
  long long X;
  if (sh >= 0) X = (long long)(m << sh);
  else if (sh > -64) X = (long long)((m + (1ull << (-sh - 1))) >> (-sh));
  else X = 0;
  return s ? -X : X;
}

// Y * 2^e2 rounded to nearest (ties to even) FP64: the magnitude's leading one
// moved to bit 63, its top 53 bits and the rounding increment added to the
// exponent field (the implicit bit and a mantissa overflow carry into it).
// Exponents outside the normal range give zero or infinity.
__host__ __device__ __forceinline__ double from_fixed(long long Y, int e2) {
  if (Y == 0) return 0.0;
  const unsigned long long s = Y < 0 ? 1ull << 63 : 0ull;
  const unsigned long long u = s ? 0ull - (unsigned long long)Y : (unsigned long long)Y;
  const int n = clz64(u);
  const unsigned long long h = u << n;
  unsigned long long m = h >> 11;
  m += (((unsigned)h & 0x7FFu) + 0x3FFu + ((unsigned)m & 1u)) >> 11;
  const int ex = 63 - n + e2 + 1023 + (int)(m >> 53);  // after rounding
  if (ex <= 0) return bits_f64(s);
  if (ex >= 2047) return bits_f64(s | (0x7ffull << 52));
  return bits_f64(s | (((unsigned long long)(63 - n + e2 + 1022) << 52) + m));
}

// v * 2^e2 rounded to nearest (ties to even) FP64, v a 128-bit integer
__host__ __device__ __forceinline__ double from_fixed128(I128 v, int e2) {
  const unsigned long long s = v.hi < 0 ? 1ull : 0ull;
  unsigned long long lo = v.lo, hi = (unsigned long long)v.hi;
  if (s) {  // magnitude
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0ull ? 1ull : 0ull);
  }
  if (hi == 0ull && lo == 0ull) return 0.0;
  // normalise: leading one at bit 63 of h, the bits below it in h then l
  int p;
  unsigned long long h, l;
  if (hi != 0ull) {
    const int n = clz64(hi);
    p = 127 - n;
    h = n == 0 ? hi : (hi << n) | (lo >> (64 - n));
    l = lo << n;
  } else {
    const int n = clz64(lo);
    p = 63 - n;
    h = lo << n;
    l = 0ull;
  }
  unsigned long long mant = h >> 11;  // 53 bits
  const unsigned long long rbit = (h >> 10) & 1ull;
  const bool sticky = (h & 0x3FFull) != 0ull || l != 0ull;
  if (rbit && (sticky || (mant & 1ull))) {
    ++mant;
    if (mant >> 53) {
      mant >>= 1;
      ++p;
    }
  }
  const int ex = p + e2 + 1023;
  if (ex <= 0) return s ? -0.0 : 0.0;
  if (ex >= 2047) return bits_f64((s << 63) | (0x7ffull << 52));
  return bits_f64((s << 63) | ((unsigned long long)ex << 52) | (mant & 0xFFFFFFFFFFFFFull));
}

__device__ __forceinline__ int out_exp(const Dev3& t, int emax) { return (emax - 1022) - t.P - t.q_shift; }

template <class Pol>
__device__ __forceinline__ void store_out(typename Pol::Y* y, long long i, typename Pol::A v, bool final_,
                                          int e2) {
  y[i] = v;
}
template <>
__device__ __forceinline__ void store_out<PI64>(long long* y, long long i, long long v, bool final_, int e2) {
  if (final_) reinterpret_cast<double*>(y)[i] = from_fixed(v, e2);
  else y[i] = v;
}
template <>
__device__ __forceinline__ void store_out<PI64S>(long long* y, long long i, long long v, bool final_, int e2) {
  store_out<PI64>(y, i, v, final_, e2);
}
template <>
__device__ __forceinline__ void store_out<PC64>(double* y, long long i, double v, bool final_, int e2) {
  y[i] = final_ ? ldexp(v, e2) : v;
}
template <>
__device__ __forceinline__ void store_out<PW>(double* y, long long i, AccW v, bool final_, int e2) {
  y[i] = v.p + from_fixed128(v.s, e2);  // both passes store real values
}

// ---------------------------------------------------------------- dependent launches

// Programmatic dependent launch: the kernel is set up while the previous one
// of the stream drains, and waits here until that one has finished and its
// writes are visible.  Called before any access to global memory.  (H|psi> of
// 12,870 / 853,776 states: 22.5 -> 16.3 / 32.8 -> 25.6 us.  Releasing the next
// kernel earlier, by launch_dependents, costs the large sectors 7 %: its CTAs
// take slots from the running kernel's last wave.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// lets the next kernel of the stream start on the SMs that this one leaves
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// kernel launch with programmatic stream serialization (see pdl_wait)
template <class... KArgs, class... Args>
inline cudaError_t launch_pdl(void (*k)(KArgs...), long long grid, int block, size_t smem, cudaStream_t st,
                              Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<KArgs>(args)...);
}

// ---------------------------------------------------------------- exponents

constexpr int kExpParts = 2048;  // partial exponents of k_exp_max, behind the first 16 ints of the scratch

__device__ __forceinline__ int biased_exp(double v) {
  return (int)(((unsigned long long)__double_as_longlong(v) >> 52) & 0x7ffull);
}

// largest of the CTA's values, in every thread (blockDim a multiple of 32)
__device__ __forceinline__ int block_max(int m) {
  __shared__ int red[32];
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  const int w = threadIdx.x & 31;
  return __reduce_max_sync(0xffffffffu, w < (int)(blockDim.x >> 5) ? red[w] : 0);
}

// largest biased exponent of each CTA's share of x into part[blockIdx.x] (apply3.cu)
__global__ void k_exp_max(const double* __restrict__ x, long long n, int* __restrict__ part);

// the largest exponent from k_exp_max's partial results, in every thread; CTA
// 0 leaves it in emax[0] for the kernels after this one
__device__ __forceinline__ int finish_exp(const int* __restrict__ part, int npart, int* emax) {
  int m = 0;
  for (int i = threadIdx.x; i < npart; i += blockDim.x) m = max(m, part[i]);
  m = block_max(m);
  if (blockIdx.x == 0 && threadIdx.x == 0) emax[0] = m;
  return m;
}

__device__ __forceinline__ int find_blk(const long long* row_start, int nblk, long long row) {
  int lo = 0, hi = nblk - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (row_start[mid] <= row) lo = mid; else hi = mid - 1;
  }
  return lo;
}

inline int n_sms(int dev) {
  int n = 0;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    n = 148;
  }
  return n;
}

}  // namespace edk
