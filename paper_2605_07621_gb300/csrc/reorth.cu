// Full orthogonalisation of an FP64 Lanczos vector against the kept basis:
// classical Gram-Schmidt applied twice (h = V^T w, w -= V h), with the norm of
// the result.  Bound: the dots by the FP64 pipe (two products per clock and SM,
// about 183 us for 150 vectors of 731,808 elements), which the update's
// products would occupy as long again.  So the update runs in FP32 on an FP32
// copy of the basis (a plane of rows of fp32_ld(n) elements, written with each
// vector) where that costs no digit of w: the rounding of the m coefficients,
// of the plane and of the m FP32 additions of an element is at most (m + 3)
// 2^-24 sum_j |h_j| |V_j|, over all elements in norm (m + 3) 2^-24 sum_j |h_j|
// for unit vectors V_j, and the update takes the plane while that is at most
// 2^-54 |w|, below the rounding of w itself (kRoSmall).  |w| is the norm before
// this very pass, so the second pass after a large first one is judged by what
// the first one left.  After a Lanczos step the coefficients are at rounding
// level, 300 of them at about 2^-52: 2^-59.  Otherwise, and without the plane,
// the FP64 basis.
// 300-step Green's function of the 12-site Hubbard ring (two sectors of
// 731,808 states): 554 -> 394 ms (dots 210 us at 0.54 T products/s, update 75
// us).  Not kept: float-float dots on two FP32 planes (325 ms, but G of the
// reference test scattered about 20 % more) and exact integer dots on
// fixed-point planes (416 ms: bound by the 32 x 32 + 64-bit multiply-adds).
#include <algorithm>

#include "apply3.cuh"
#include "krylov.h"
#include "reduce.cuh"

namespace edk {

constexpr int kRoBatch = 8;  // basis vectors per CTA of the dots
constexpr double kRoSmall = 0x1p-30;  // (m + 3) sum |h_j| / |w| up to which the update takes the FP32 plane

// part[j * gridDim.x + blockIdx.x] = the share of <V_j, w> of the CTA's column
// range, for the kRoBatch vectors of blockIdx.y: w is read once for eight
// vectors, eight independent sums per thread
__global__ void __launch_bounds__(256, 4) k_reorth_dots(const double* __restrict__ V, long long ldv, int m,
                                                     const double* __restrict__ w, long long n,
                                                     double* __restrict__ part) {
  pdl_wait();
  __shared__ double red[8][kRoBatch];
  const int j0 = blockIdx.y * kRoBatch, nj = min(kRoBatch, m - j0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* vp = V + (long long)j0 * ldv;
  double s[kRoBatch];
#pragma unroll
  for (int u = 0; u < kRoBatch; ++u) s[u] = 0.0;
  const long long step = gridDim.x * 256ll;
  if (nj == kRoBatch) {
#pragma unroll 4
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += step) {
      const double x = __ldg(w + i);
      double v[kRoBatch];
#pragma unroll
      for (int u = 0; u < kRoBatch; ++u) v[u] = __ldg(vp + (long long)u * ldv + i);
#pragma unroll
      for (int u = 0; u < kRoBatch; ++u) s[u] = fma(v[u], x, s[u]);
    }
  } else {
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += step) {
      const double x = __ldg(w + i);
#pragma unroll
      for (int u = 0; u < kRoBatch; ++u)
        if (u < nj) s[u] = fma(__ldg(vp + (long long)u * ldv + i), x, s[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < kRoBatch; ++u) {
    for (int o = 16; o > 0; o >>= 1) s[u] += __shfl_down_sync(0xffffffffu, s[u], o);
    if (lane == 0) red[warp][u] = s[u];
  }
  __syncthreads();
  if (threadIdx.x < nj) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += red[k][threadIdx.x];
    part[(long long)(j0 + threadIdx.x) * gridDim.x + blockIdx.x] = t;
  }
}

// h_j = sum of its partial results, one warp per j
__global__ void __launch_bounds__(256) k_reorth_sum(const double* __restrict__ part, int g, int m,
                                                    double* __restrict__ h) {
  pdl_wait();
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= m) return;
  double s = 0.0;
  for (int i = lane; i < g; i += 32) s += part[(long long)j * g + i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) h[j] = s;
}

// w -= sum_j h_j V_j, four elements per thread and U vectors in flight; LAST, or
// where the coefficients are large: then beta = ||w|| by the last CTA (small ones
// leave the norm as it was, to 2^-60).  *beta holds the norm of w before.  F: the
// FP32 plane (row stride ldf), or null.
template <bool LAST>
__global__ void __launch_bounds__(128) k_reorth_update(const double* __restrict__ V, long long ldv,
                                                       const float* __restrict__ F, long long ldf, int m,
                                                       double* __restrict__ w, long long n,
                                                       const double* __restrict__ h, double* beta, double* npart,
                                                       unsigned* ctr) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char ro_smem[];
  double* hs = reinterpret_cast<double*>(ro_smem);  // [m]
  float* hf = reinterpret_cast<float*>(hs + m);     // [m] h_j 2^sh
  constexpr int U = 8;
  const double b0 = beta[0];
  const int sh = min(900, max(-900, 1022 - biased_exp(b0)));  // the norm near 1
  double hsum = 0.0;
  for (int j = threadIdx.x; j < m; j += 128) {
    const double v = h[j];
    hs[j] = v;
    hf[j] = (float)ldexp(v, sh);
    hsum += fabs(v);
  }
  hsum = block_sum(hsum);
  const bool big = __syncthreads_or(threadIdx.x == 0 && !(F && (m + 3) * hsum <= kRoSmall * b0));
  double nacc = 0.0;
  for (long long i = 4 * (blockIdx.x * 128ll + threadIdx.x); i < n; i += 4 * gridDim.x * 128ll) {
    double s[4];
    if (!big) {
      float a[4] = {0.f, 0.f, 0.f, 0.f};
      auto add = [&](float f, float4 v) {
        a[0] = fmaf(f, v.x, a[0]);
        a[1] = fmaf(f, v.y, a[1]);
        a[2] = fmaf(f, v.z, a[2]);
        a[3] = fmaf(f, v.w, a[3]);
      };
      int j = 0;
      for (; j + U <= m; j += U) {
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = __ldg(reinterpret_cast<const float4*>(F + (long long)(j + u) * ldf + i));
#pragma unroll
        for (int u = 0; u < U; ++u) add(hf[j + u], v[u]);
      }
      for (; j < m; ++j) add(hf[j], __ldg(reinterpret_cast<const float4*>(F + (long long)j * ldf + i)));
#pragma unroll
      for (int q = 0; q < 4; ++q) s[q] = ldexp((double)a[q], -sh);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) s[q] = 0.0;
#pragma unroll 4
      for (int j = 0; j < m; ++j) {
        const double* vp = V + (long long)j * ldv + i;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (i + q < n) s[q] = fma(hs[j], __ldg(vp + q), s[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i + q < n) {
        const double v = w[i + q] - s[q];
        w[i + q] = v;
        if (LAST || big) nacc = fma(v, v, nacc);
      }
  }
  if (!LAST && !big) return;
  const double s = block_sum(nacc);
  __shared__ unsigned s_last;
  if (threadIdx.x == 0) {
    npart[blockIdx.x] = s;
    __threadfence();
    s_last = atomicAdd(ctr, 1u) == gridDim.x - 1 ? 1u : 0u;
    if (s_last) {
      *ctr = 0u;
      __threadfence();
    }
  }
  __syncthreads();
  if (!s_last) return;
  double v = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += 128) v += __ldcg(npart + i);
  const double t = block_sum(v);
  if (threadIdx.x == 0) beta[0] = sqrt(t > 0.0 ? t : 0.0);
}

long long fp32_ld(long long n) { return (n + 3) / 4 * 4; }

constexpr int kRoParts = 256;  // most column ranges of the dots

long long reorth64_doubles(int cap) { return (long long)cap * (kRoParts + 1); }

ed_status launch_reorth64(ed_ctx* c, const double* V, const float* F, int m, double* w, long long n, double* scratch,
                          cudaStream_t st) {
  if (m <= 0) return ED_OK;
  const int sms = n_sms(c->device), jg = (m + kRoBatch - 1) / kRoBatch;
  // column ranges: one wave of four CTAs per SM, no range shorter than one pass
  const int g = (int)std::max<long long>(
      1, std::min<long long>({(n + 255) / 256, (long long)4 * sms / jg, (long long)kRoParts}));
  const int gu = (int)std::min<long long>({(n + 511) / 512, (long long)sms * 16, (long long)kMaxPartials});
  double* part = scratch;
  double* h = scratch + (long long)m * g;
  double* beta = slot(c, 1);
  unsigned* ctr = (unsigned*)c->d_err + 2;
  for (int pass = 0; pass < 2; ++pass) {
    k_reorth_dots<<<dim3(g, jg), 256, 0, st>>>(V, n, m, w, n, part);
    ED_CUDA_TRY(cudaGetLastError());
    ED_CUDA_TRY(launch_pdl(k_reorth_sum, (m + 7) / 8, 256, 0, st, (const double*)part, g, m, h));
    ED_CUDA_TRY(launch_pdl(pass ? k_reorth_update<true> : k_reorth_update<false>, gu, 128, (size_t)m * 12, st, V, n, F,
                           fp32_ld(n), m, w, n, (const double*)h, beta, c->d_partials, ctr));
  }
  return ED_OK;
}

}  // namespace edk
