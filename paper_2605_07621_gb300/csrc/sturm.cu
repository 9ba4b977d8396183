// All eigenvalues of a batch of symmetric tridiagonal matrices on the GPU, by
// counting: the number of negative pivots of T - x I = L D L^T, q_i = (d_i -
// x) - e_{i-1}^2 / q_{i-1}, is the number of eigenvalues below x (Sturm;
// Givens 1954; Barth, Martin and Wilkinson, "Calculation of the eigenvalues
// of a symmetric tridiagonal matrix by the method of bisection", Numer. Math.
// 9, 1967; Kahan 1966 for its backward stability).  Every eigenvalue is
// bracketed on its own, so the whole batch is one launch per stage:
//   k_sturm_df   brackets of 2^-49 of the norm (of the unreduced part, see
//                k_sturm_prep).  The recurrence runs in
//                float-float on the FP32 pipe: a step is about 30 FP32
//                instructions and a chain of about 60 cycles.
//   k_sturm_f64  from there to 2^-53 of the norm in FP64, whose pipe takes 64
//                cycles for a warp's instruction: 7 of them per step, for the
//                last 6 of 53 bits.  A bracket whose end the FP64 counts never
//                moved is checked there and widened if need be, so the result
//                is that of bisection in FP64 alone.
// A group of S lanes (a power of two) takes one eigenvalue and S shifts at
// once, which cut its bracket into S + 1 parts: log2(S + 1) bits per pass over
// the matrix.  S shifts cost S / log2(S + 1) times the work of plain bisection,
// so S only fills the GPU: about four warps per scheduler for the float-float
// stage (latency), one for the FP64 stage (throughput).
//
// It replaces the QL iteration on the host as the spectrum's last stage: for
// m = 3432, about 10^7 rotations of two dependent divisions each took 130 ms
// against 5.7 ms here (2.9 float-float, 2.8 FP64); the 16,384 levels of a
// 15-block spectrum (m up to 3432) take 10.3 ms (4.7 + 5.5), FP64 alone would
// take about 48.
#include <algorithm>
#include <cmath>
#include <vector>

#include "dfloat.cuh"
#include "eigsym.h"

namespace edk {
namespace {

constexpr int kStThreads = 128;
constexpr int kStPrep = 1024;   // threads of k_sturm_prep
constexpr int kStPasses = 200;  // most passes of a bracket (S = 1 needs about 60)

// The matrix falls apart where an off-diagonal entry is no larger than eps times
// its two neighbours on the diagonal, or than eps times the norm of the whole
// matrix (the rule of the QL iteration in eigsym.cu).  Every part is scaled and
// counted by itself: a part of one row is its own eigenvalue, so a block without
// weight has exact zeros and a diagonal one keeps levels far below its norm
// (counted as one matrix they all came out at 2^-53 of the norm, or of 1 for a
// zero matrix), and the others' brackets are as narrow as their own norm asks.
//
// Per block: its parts (row: first row, end, exponent of the part's norm
// max(|d_i| + |e_{i-1}| + |e_i|)), and the matrix with each part's norm scaled
// into [1/2, 1): d and e^2 as float-float (tf) and FP64 (td), e2 of row i
// coupling it to row i - 1, zero in a part's first row.  nrm: the norm, NaN if
// an entry is not finite.  A thread takes a run of consecutive rows; the first
// row of each row's part is a prefix maximum over the threads, the end a suffix
// minimum, the norms are the maxima of the bits (pn, one word per row).
__global__ void __launch_bounds__(kStPrep) k_sturm_prep(const SturmBlk* __restrict__ blk, const double* __restrict__ de,
                                                        float4* __restrict__ tf, double2* __restrict__ td,
                                                        SturmRow* __restrict__ row, unsigned long long* __restrict__ pn,
                                                        double* nrm) {
  const SturmBlk B = blk[blockIdx.x];
  const double *d = de + 2 * B.off, *e = d + B.n;
  row += B.off;
  pn += B.off;
  const int tid = threadIdx.x, n = B.n;
  __shared__ double s_m[kStPrep / 32];
  __shared__ int s_bad, s_first[kStPrep], s_end[kStPrep];
  if (tid == 0) s_bad = 0;
  __syncthreads();
  double mx = 0.0;
  for (int i = tid; i < n; i += kStPrep) {
    const double t = fabs(d[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0) + (i < n - 1 ? fabs(e[i]) : 0.0);
    if (!isfinite(t)) s_bad = 1;
    mx = fmax(mx, t);
    pn[i] = 0;
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((tid & 31) == 0) s_m[tid >> 5] = mx;
  __syncthreads();
  mx = s_m[0];
  for (int w = 1; w < kStPrep / 32; ++w) mx = fmax(mx, s_m[w]);
  if (tid == 0) nrm[blockIdx.x] = s_bad ? __longlong_as_double(0x7ff8000000000000ll) : mx;
  // a part starts at row i
  auto starts = [&](int i) {
    if (i == 0) return true;
    const double a = fabs(e[i - 1]);
    return a <= 0x1p-53 * (fabs(d[i - 1]) + fabs(d[i])) || a <= 0x1p-53 * mx;
  };
  const int per = (n + kStPrep - 1) / kStPrep, i0 = min(n, tid * per), i1 = min(n, i0 + per);
  int first = -1, end = n;  // the last start in this thread's rows, and the first
  for (int i = i0; i < i1; ++i)
    if (starts(i)) {
      if (first < 0) end = i;
      first = i;
    }
  s_first[tid] = first;
  s_end[tid] = end;
  __syncthreads();
  for (int o = 1; o < kStPrep; o *= 2) {
    const int f = tid >= o ? s_first[tid - o] : -1, z = tid + o < kStPrep ? s_end[tid + o] : n;
    __syncthreads();
    s_first[tid] = max(s_first[tid], f);
    s_end[tid] = min(s_end[tid], z);
    __syncthreads();
  }
  int at = tid > 0 ? s_first[tid - 1] : 0;  // the part of the row before this thread's
  double pm = 0.0;
  auto put = [&] {
    if (pm > 0.0) atomicMax(pn + at, (unsigned long long)__double_as_longlong(pm));
    pm = 0.0;
  };
  for (int i = i0; i < i1; ++i) {
    if (starts(i)) {
      put();
      at = i;
    }
    row[i].first = at;
    const double t = fabs(d[i]) + (i > at ? fabs(e[i - 1]) : 0.0) + (i < n - 1 && !starts(i + 1) ? fabs(e[i]) : 0.0);
    if (isfinite(t)) pm = fmax(pm, t);
  }
  put();
  int z = tid + 1 < kStPrep ? s_end[tid + 1] : n;  // the end of the part of this thread's last row
  for (int i = i1 - 1; i >= i0; --i) {
    row[i].end = z;
    if (row[i].first == i) z = i;
  }
  __syncthreads();
  for (int i = tid; i < n; i += kStPrep) {
    const int r0 = row[i].first;
    int ex = 0;
    if (pn[r0]) frexp(__longlong_as_double((long long)pn[r0]), &ex);
    row[i].ex = ex;
    const double ds = ldexp(d[i], -ex), es = i > r0 ? ldexp(e[i - 1], -ex) : 0.0, e2 = es * es;
    td[B.off + i] = make_double2(ds, e2);
    const float2 a = split_scaled(ds, 0), b = split_scaled(e2, 0);
    tf[B.off + i] = make_float4(a.x, a.y, b.x, b.y);
  }
}

// eigenvalues below x of the n x n matrix t, in float-float.  A pivot below
// 2^-100 counts as -2^-100 (the matrix's norm is 1), so no quotient overflows.
__device__ __forceinline__ int count_df(const float4* __restrict__ t, int n, double x) {
  const float xh = (float)x, xl = (float)(x - (double)xh);
  float qh = 1.f, ql = 0.f;
  int c = 0;
#pragma unroll 8
  for (int i = 0; i < n; ++i) {
    const float4 v = __ldg(t + i);
    // u = d - x
    const float u = __fsub_rn(v.x, xh), zu = __fsub_rn(u, v.x);
    const float ul = __fadd_rn(__fsub_rn(__fsub_rn(v.x, __fsub_rn(u, zu)), __fadd_rn(xh, zu)), __fsub_rn(v.y, xl));
    // w = e^2 / q: a quotient of the leading parts and its remainder's
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(qh));
    const float w = __fmul_rn(v.z, r);
    const float rem = __fadd_rn(fmaf(-w, ql, fmaf(-w, qh, v.z)), v.w);
    const float wl = __fmul_rn(rem, r);
    // q = u - w, normalised
    const float s = __fsub_rn(u, w), zs = __fsub_rn(s, u);
    const float e = __fsub_rn(__fsub_rn(u, __fsub_rn(s, zs)), __fadd_rn(w, zs));
    const float l = __fadd_rn(e, __fsub_rn(ul, wl));
    qh = __fadd_rn(s, l);
    ql = __fsub_rn(l, __fsub_rn(qh, s));
    if (fabsf(qh) < 0x1p-100f) {
      qh = -0x1p-100f;
      ql = 0.f;
    }
    c += qh < 0.f;
  }
  return c;
}

// the same in FP64.  The quotient: the hardware's approximate reciprocal, one
// Newton step, and the residual of e^2 / q with that (40 + 40 bits, rounded to
// FP64: the plain division is about twice the instructions).
__device__ __forceinline__ int count_f64(const double2* __restrict__ t, int n, double x) {
  double q = 1.0;
  int c = 0;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const double2 v = __ldg(t + i);
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(q));
    r = fma(r, fma(-q, r, 1.0), r);
    const double w0 = v.y * r, w = fma(r, fma(-w0, q, v.y), w0);
    q = (v.x - x) - w;
    // |q| < 2^-300, by its exponent bits
    if ((__double2hiint(q) & 0x7fffffff) < (1023 - 300) << 20) q = -0x1p-300;
    c += (unsigned)__double2hiint(q) >> 31;
  }
  return c;
}

// the block and row of this group of S lanes, whose eigenvalue is the one that
// stands as many places up in the row's part; warp w of the launch belongs to
// the block b with first[b] <= w
template <int STAGE>
__device__ __forceinline__ bool group_of(const SturmBlk* __restrict__ blk, int nb, int S, int& b, int& k) {
  const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  int lo = 0, hi = nb;
  while (hi - lo > 1) {
    const int mid = (lo + hi) / 2;
    if ((STAGE == 0 ? blk[mid].w0 : blk[mid].w1) <= w)
      lo = mid;
    else
      hi = mid;
  }
  b = lo;
  const int lane = threadIdx.x & 31;
  k = (w - (STAGE == 0 ? blk[b].w0 : blk[b].w1)) * (32 / S) + lane / S;
  const bool mine = k < blk[b].n;
  k = min(k, blk[b].n - 1);
  return mine;
}

// point i of the S that cut (lo, hi) into S + 1 parts
__device__ __forceinline__ double cut(double lo, double hi, int i, double inv) { return fma((hi - lo) * inv, i + 1.0, lo); }

// the part of (lo, hi) that holds eigenvalue k, from the counts of the group's S points
__device__ __forceinline__ void narrow(double& lo, double& hi, int cnt, int k, int S, double inv) {
  const int lane = threadIdx.x & 31, base = lane & ~(S - 1);
  const unsigned mask = S == 32 ? 0xffffffffu : (1u << S) - 1u;
  const unsigned above = (__ballot_sync(0xffffffffu, cnt > k) >> base) & mask;
  const int i = above ? __ffs((int)above) - 1 : S;
  const double a = i == 0 ? lo : cut(lo, hi, i - 1, inv), b = i == S ? hi : cut(lo, hi, i, inv);
  lo = a;
  hi = b;
}

__global__ void __launch_bounds__(kStThreads) k_sturm_df(const SturmBlk* __restrict__ blk, int nb, int S, int warps,
                                                         const float4* __restrict__ tf,
                                                         const SturmRow* __restrict__ row, double2* __restrict__ br) {
  if ((int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) >= warps) return;
  int b, k;
  const bool mine = group_of<0>(blk, nb, S, b, k);
  const SturmRow R = row[blk[b].off + k];
  const int n = R.end - R.first, sub = threadIdx.x & (S - 1);
  const float4* t = tf + blk[b].off + R.first;
  const double inv = 1.0 / (S + 1);
  double lo = -1.0, hi = n > 1 ? 1.0 : -1.0;  // (a part of one row needs no bracket)
  for (int p = 0; p < kStPasses && __any_sync(0xffffffffu, hi - lo > 0x1p-49); ++p)
    narrow(lo, hi, n > 1 ? count_df(t, n, cut(lo, hi, sub, inv)) : 0, k - R.first, S, inv);
  if (mine && sub == 0) br[blk[b].off + k] = make_double2(lo, hi);
}

__global__ void __launch_bounds__(kStThreads) k_sturm_f64(const SturmBlk* __restrict__ blk, int nb, int S, int warps,
                                                          const double2* __restrict__ td,
                                                          const double2* __restrict__ br,
                                                          const SturmRow* __restrict__ row,
                                                          const double* __restrict__ de, double* __restrict__ lam) {
  if ((int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) >= warps) return;
  int b, k;
  const bool mine = group_of<1>(blk, nb, S, b, k);
  const SturmRow R = row[blk[b].off + k];
  const int n = R.end - R.first, sub = threadIdx.x & (S - 1);
  const double2* t = td + blk[b].off + R.first;
  const double inv = 1.0 / (S + 1);
  const double2 v = br[blk[b].off + k];
  double lo = v.x - 0x1p-49, hi = v.y + 0x1p-49, grow = 0x1p-45;
  // whether the FP64 counts put the eigenvalue above lo, below hi
  bool lok = false, hok = false, stuck = false;  // stuck: no FP64 value in between
  const int nth = k - R.first;                   // the eigenvalue's number in its part
  for (int p = 0; p < kStPasses; ++p) {
    const bool wide = n > 1 && hi - lo > 0x1p-53 && !stuck, ends = n > 1 && !wide && !(lok && hok);
    if (!__any_sync(0xffffffffu, wide || ends)) break;
    const double x = wide ? cut(lo, hi, sub, inv) : !lok ? lo : hi;
    const int cnt = wide || ends ? count_f64(t, n, x) : 0;
    const double lo0 = lo, hi0 = hi;
    double a = lo, c = hi;
    narrow(a, c, cnt, nth, S, inv);
    if (wide) {
      lo = a;
      hi = c;
      lok |= lo != lo0;
      hok |= hi != hi0;
      stuck = lo == lo0 && hi == hi0;
    } else if (ends) {
      const bool in = !lok ? cnt <= nth : cnt > nth;
      if (in) {
        (!lok ? lok : hok) = true;
      } else if (!lok) {  // below lo: that is an upper end
        hi = lo;
        lo -= grow;
        hok = true;
      } else {  // not below hi
        lo = hi;
        hi += grow;
        hok = false;
      }
      if (!in) {
        grow *= 16.0;
        stuck = false;
      }
    }
  }
  if (mine && sub == 0)
    lam[blk[b].off + blk[b].n - 1 - k] = n == 1 ? de[2 * blk[b].off + k] : ldexp(0.5 * (lo + hi), R.ex);
}

}  // namespace

ed_status sturm_eigenvalues(const SturmBatch& B, cudaStream_t st) {
  const int nb = (int)B.nb;
  if (nb == 0) return ED_OK;
  k_sturm_prep<<<nb, kStPrep, 0, st>>>(B.d_blk, B.de, B.tf, B.td, B.row, (unsigned long long*)B.br, B.nrm);
  const int per = kStThreads / 32;
  k_sturm_df<<<(B.warps0 + per - 1) / per, kStThreads, 0, st>>>(B.d_blk, nb, B.S0, B.warps0, B.tf, B.row,
                                                               B.br);
  k_sturm_f64<<<(B.warps1 + per - 1) / per, kStThreads, 0, st>>>(B.d_blk, nb, B.S1, B.warps1, B.td, B.br, B.row, B.de,
                                                                B.lam);
  ED_CUDA_TRY(cudaGetLastError());
  return ED_OK;
}

void sturm_plan(std::vector<SturmBlk>& blk, int sms, SturmBatch* B) {
  long long total = 0;
  for (const SturmBlk& x : blk) total += x.n;
  // lanes per eigenvalue: the largest power of two with at most `warps` per
  // scheduler (four to an SM) over the whole batch
  auto lanes = [&](int warps) {
    int S = 1;
    while (S < 32 && total * 2 * S <= 32LL * 4 * warps * sms) S *= 2;
    return S;
  };
  B->S0 = lanes(4);
  B->S1 = lanes(1);
  B->warps0 = B->warps1 = 0;
  for (SturmBlk& x : blk) {
    x.w0 = B->warps0;
    x.w1 = B->warps1;
    B->warps0 += (x.n * B->S0 + 31) / 32;
    B->warps1 += (x.n * B->S1 + 31) / 32;
  }
  B->nb = blk.size();
}

}  // namespace edk
