// Class-sorted H|psi> (paper Eq. (2)) in these arithmetic flavours:
//   FP32  storage and accumulation;
//   FP64  storage and accumulation (fallback);
//   I64   FP64 storage, exact 64-bit fixed-point accumulation: when every
//         matrix element is a small integer multiple of 2^-q_shift, x is
//         scaled by one power of two per vector, summed exactly on the
//         integer pipe and rounded once back to FP64.  FP64 adds and FP64
//         conversions run at about 0.5 T/s on this GPU, the integer pipe at
//         tens of T/s, so no FP64 instruction is issued per matrix element;
//   W128  the same for couplings that are not dyadic: FP64 values are
//         integer multiples of 2^-q_shift with up to 53-bit integers, so the
//         class sums are weighted by 64-bit integers into exact 128-bit sums,
//         rounded to FP64 once per pass;
//   C64   fixed-point class sums weighted in FP64 (value ranges too wide
//         for 64-bit integer weights).
// Row pass (k_row5): the diagonal, the H_B (column-mixing) term and the
// cross-cut terms of whole rows.  A few rows psi_s[a,:] are staged in shared
// memory, then each column b sums, class by class, its H_B
// neighbours (16-bit column indices) and the cross-cut gathers from x in
// global memory, plus the diagonal.
// Panel pass: the H_A (row-mixing) term over column panels that stay
// resident in L2.
#include <mutex>
#include <type_traits>

#include "apply3.cuh"

namespace edk {

// host entry points of the two conversions (used by the CPU tests)
long long host_to_fixed(double v, int sh_base) { return to_fixed(v, sh_base); }
double host_from_fixed(long long Y, int e2) { return from_fixed(Y, e2); }
double host_from_fixed128(long long hi, unsigned long long lo, int e2) {
  I128 v;
  v.hi = hi;
  v.lo = lo;
  return from_fixed128(v, e2);
}
void host_mul_wide(long long a, long long b, long long* hi, unsigned long long* lo) {
  const I128 v = mul_wide(a, b);
  *hi = v.hi;
  *lo = v.lo;
}

// largest biased exponent of each CTA's share of x into part[blockIdx.x];
// the next kernel takes the largest of them (no atomics, nothing to clear).
// x is 16-byte aligned.  Bound by HBM: 0.67 ms for 4.8 GB (7.2 TB/s).
__global__ void __launch_bounds__(256) k_exp_max(const double* __restrict__ x, long long n, int* __restrict__ part) {
  pdl_wait();
  const double2* x2 = reinterpret_cast<const double2*>(x);
  const long long n2 = n >> 1, step = (long long)gridDim.x * 256;
  int m = 0;
  long long i = blockIdx.x * 256ll + threadIdx.x;
  for (; i + 3 * step < n2; i += 4 * step) {
    double2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = x2[i + u * step];
#pragma unroll
    for (int u = 0; u < 4; ++u) m = max(m, max(biased_exp(v[u].x), biased_exp(v[u].y)));
  }
  for (; i < n2; i += step) {
    const double2 v = x2[i];
    m = max(m, max(biased_exp(v.x), biased_exp(v.y)));
  }
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) m = max(m, biased_exp(x[n - 1]));
  m = block_max(m);
  if (threadIdx.x == 0) part[blockIdx.x] = m;
}

// |x| < 2^E with E = emax - 1022; X = round(x * 2^(P - E)).  Bound by HBM
// (16 bytes per element): 16-byte accesses, four in flight per thread; 601 M
// elements 1.80 -> 1.46 ms (6.6 TB/s) against one 8-byte access at a time.
__global__ void __launch_bounds__(256) k_to_fixed(const double* __restrict__ x, long long* __restrict__ X, long long n,
                                                  const int* __restrict__ part, int npart, int* emax, int P) {
  pdl_wait();
  const int sh = P - (finish_exp(part, npart, emax) - 1022);
  const double2* x2 = reinterpret_cast<const double2*>(x);
  longlong2* X2 = reinterpret_cast<longlong2*>(X);
  const long long n2 = n >> 1, step = (long long)gridDim.x * 256;
  long long i = blockIdx.x * 256ll + threadIdx.x;
  for (; i + 3 * step < n2; i += 4 * step) {
    double2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = x2[i + u * step];
#pragma unroll
    for (int u = 0; u < 4; ++u) X2[i + u * step] = make_longlong2(to_fixed(v[u].x, sh), to_fixed(v[u].y, sh));
  }
  for (; i < n2; i += step) {
    const double2 v = x2[i];
    X2[i] = make_longlong2(to_fixed(v.x, sh), to_fixed(v.y, sh));
  }
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) X[n - 1] = to_fixed(x[n - 1], sh);
}

// R rows of the staged group at one column: one 16-byte shared-memory access
template <class S, int R>
struct alignas(16) RowVec {
  S v[R];
};

__device__ __forceinline__ void l2_prefetch(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// *p under the predicate, else zero.  8-byte types: a predicated load, without
// a branch (row pass of J1-J2 4x8: 17.0 -> 15.8 ms); FP32, with twice the rows
// per bond, is faster as the compiler schedules it (9.2 against 9.6 ms)
__device__ __forceinline__ long long ldg_if(const long long* p, bool on) {
  long long v = 0;
  asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q ld.global.nc.b64 %0, [%1]; }" : "+l"(v) : "l"(p), "r"((unsigned)on));
  return v;
}
__device__ __forceinline__ double ldg_if(const double* p, bool on) {
  return __longlong_as_double(ldg_if(reinterpret_cast<const long long*>(p), on));
}
__device__ __forceinline__ float ldg_if(const float* p, bool on) { return on ? __ldg(p) : 0.f; }

// Row pass: work unit = R consecutive rows of one block ("row group", R = 16
// bytes / element), staged in shared memory with the R rows of a column side
// by side, so that one 16-byte access serves R matrix elements and every
// B-side index, map and diagonal load is shared by the R rows.  A warp takes
// 32 columns (one slab) at a time:
//  * H_B: the slab's pair rows (Dev3::B_pair) are read with one coalesced
//    4-byte load per lane, four rows a step and a step ahead of their use;
//    the slab's row counts are the same for all lanes, so the loops neither
//    diverge nor run past the slab's longest list;
//  * cross terms: per octet of cross-bond sites one 16-byte load brings a
//    column's eight maps, one word its 32 bond bits; each present slot
//    gathers the R source rows under the predicate that the bond flips, all
//    gathers of a site before their sums, one weight per value class and
//    column;
//  * the diagonal from per-row constants and popcounts of packed words.
// Bound: the L1 / shared-memory data path (69 % of its wavefronts on J1-J2 4x7),
// then issue (63 %).  A 16-byte access
// takes four wavefronts at best; the lists are ordered so that it takes 4.06
// (order_lists).  Measured, FP64 fixed point / FP32: J1-J2 4x8 (601 M states)
// 22.9 -> 16.4 / 14.3 -> 9.2 ms, Hubbard 4x4 (166 M states) 2.75 -> 1.63 /
// 1.48 -> 0.92 ms, against lists of 8-byte groups per column, scattered over the
// lanes and padded to 16 entries.  The digit-split dense products on the
// tensor cores that could take the terms inside a group of sites would cost
// about 28 instructions per state and group for the split and the
// recombination, as much as the gathers they replace.
// CVT (contexts without cross terms): the rows are staged from the FP64 input
// and converted on the way; the fixed-point copy xw, which only the panel
// pass then reads, is written here instead of by k_to_fixed.
template <class Pol, int R, int NT, bool CVT>
__global__ void __launch_bounds__(NT, 1024 / NT)
    k_row5(P3 p, const long long* __restrict__ grp_start, long long n_groups,
           const std::conditional_t<CVT, double, typename Pol::S>* __restrict__ x, typename Pol::Y* __restrict__ y,
           int* emax, typename Pol::S* __restrict__ xw, const int* __restrict__ part, int npart) {
  using S = typename Pol::S;
  using V = RowVec<S, R>;
  static_assert(sizeof(V) == 16, "one 16-byte word per column");
  extern __shared__ __align__(16) unsigned char smem5[];
  V* const xs = reinterpret_cast<V*>(smem5);
  // source row of each (slot or bond, row), null where there is none; the
  // A-side bits of the slots and the mask of slots with a source row
  __shared__ __align__(16) const S* s_ptr[kMaxOct][32][R];
  __shared__ unsigned s_ax[kMaxOct][R], s_vm[kMaxOct][R];
  const Dev3& t = p.t;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_wait();
  int sh = 0, e2 = 0;
  if constexpr (CVT) {
    const int em = finish_exp(part, npart, emax);
    sh = t.P - (em - 1022);
    e2 = out_exp(t, em);
  } else {
    e2 = emax ? out_exp(t, emax[0]) : 0;
  }
  const int n_oct = !CVT && p.ncross ? (t.xs_ok ? t.n_oct : 1) : 0;
  for (long long g = blockIdx.x; g < n_groups; g += gridDim.x) {
    const int bi = find_blk(grp_start, p.nblk, g);
    const DevBlock bl = p.blocks[bi];
    const long long a0 = (g - grp_start[bi]) * R;
    const int nr = (int)min((long long)R, bl.dA - a0);
    const int dB = (int)bl.dB;
    const long long row0 = bl.off + a0 * dB;
    __syncthreads();  // the previous group's columns are done
    {
      const auto* r0 = x + row0;
#pragma unroll 4
      for (int b = threadIdx.x; b < dB; b += NT) {
        V w;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if constexpr (CVT) w.v[r] = r < nr ? to_fixed(r0[(long long)r * dB + b], sh) : 0;
          else w.v[r] = r < nr ? r0[(long long)r * dB + b] : (S)0;
        }
        xs[b] = w;
        if constexpr (CVT) {
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (r < nr && bl.has_hA) xw[row0 + (long long)r * dB + b] = w.v[r];
        }
      }
      if (threadIdx.x < 8) {  // zero slots addressed by the padding indices, one per bank group
        V w;
#pragma unroll
        for (int r = 0; r < R; ++r) w.v[r] = 0;
        xs[dB + threadIdx.x] = w;
      }
    }
    // one warp per (octet, row): lane = slot (or bond, without slots)
    for (int q = warp; q < n_oct * R; q += NT / 32) {
      const int h = q / R, r = q % R;
      const int k = t.xs_ok ? t.xs_k[32 * h + lane] : (lane < p.ncross ? lane : 255);
      const S* sp = nullptr;
      const long long gA = bl.gA0 + a0 + r;
      if (r < nr && k != 255) {
        const int sb = ((t.A_pack[gA] >> k) & 1u) ? bl.nbr_lo : bl.nbr_hi;
        if (sb >= 0) {
          const DevBlock& so = p.blocks[sb];
          const unsigned rr = t.mapA[(long long)t.bond_ia[k] * t.A_total + gA];
          if constexpr (!CVT)
            if (rr != 0xFFFFu) sp = x + so.off + (long long)rr * so.dB;
        }
      }
      s_ptr[h][lane][r] = sp;
      const unsigned vm = __ballot_sync(0xffffffffu, sp != nullptr);
      if (lane == 0) {
        s_vm[h][r] = vm;
        s_ax[h][r] = r < nr ? (t.xs_ok ? t.A_xs[h * t.A_total + gA] : t.A_pack[gA]) : 0u;
      }
    }
    // the next group's rows on their way into L2 while this one is summed
    if (threadIdx.x == 0 && g + gridDim.x < n_groups) {
      const long long gn = g + gridDim.x;
      const int bn = find_blk(grp_start, p.nblk, gn);
      const DevBlock& nb = p.blocks[bn];
      const long long an = (gn - grp_start[bn]) * R;
      const char* p0 = reinterpret_cast<const char*>(x + nb.off + an * nb.dB);
      const char* p1 = p0 + (size_t)(min((long long)R, nb.dA - an) * nb.dB) * sizeof(*x);
      const char* q0 = reinterpret_cast<const char*>(((uintptr_t)p0 + 15) & ~(uintptr_t)15);
      const char* q1 = reinterpret_cast<const char*>((uintptr_t)p1 & ~(uintptr_t)15);
      if (q1 > q0) l2_prefetch(q0, (unsigned)(q1 - q0));
    }
    unsigned pa[R];
    typename Pol::D da[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const long long gA = bl.gA0 + a0 + (r < nr ? r : 0);
      pa[r] = t.A_pack[gA];
      da[r] = Pol::diagA(t, gA);
    }
    const bool final_ = !bl.has_hA;
    __syncthreads();
    const int nslab = (dB + 31) >> 5;
    for (int sl = warp; sl < nslab; sl += NT / 32) {
      const int b = 32 * sl + lane;
      const bool in = b < dB;
      const long long gB = bl.gB0 + (in ? b : dB - 1);
      const uint2 m = t.B_slab[bl.slabB0 + sl];
      const unsigned* cp = t.B_pair + (size_t)m.x * 32 + lane;
      unsigned qn[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) qn[u] = __ldg(cp + 32 * u);
      const unsigned pb = t.B_pack[gB];
      uint4 mv = make_uint4(0u, 0u, 0u, 0u);
      unsigned bx = 0u;
      if (n_oct && t.xs_ok) {
        mv = __ldg(t.B_xmap + gB);
        bx = __ldg(t.B_xs + gB);
      }
      typename Pol::A acc[R];
      {
        const typename Pol::D dbv = Pol::diagB(t, gB);
        const V xb = xs[in ? b : dB];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const unsigned z = t.vab_and ? (pa[r] & pb) : (pa[r] ^ pb);
          if constexpr (Pol::kSplit) acc[r] = 0;
          else acc[r] = Pol::dmul(da[r] + dbv + Pol::vab(t, z), xb.v[r]);
        }
      }
#pragma unroll
      for (int c = 0; c < kMaxCls; ++c) {
        const int n = (int)((m.y >> (8 * c)) & 255u);
        if (!n) continue;
        S sum[R];
#pragma unroll
        for (int r = 0; r < R; ++r) sum[r] = 0;
        auto add_pair = [&](unsigned q) {
          const V v0 = xs[q & 0xFFFFu], v1 = xs[q >> 16];
#pragma unroll
          for (int r = 0; r < R; ++r) sum[r] += v0.v[r] + v1.v[r];
        };
        int i = n;
        for (; i >= 4; i -= 4) {
          unsigned q[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) q[u] = qn[u];
          cp += 128;
#pragma unroll
          for (int u = 0; u < 4; ++u) qn[u] = __ldg(cp + 32 * u);
#pragma unroll
          for (int u = 0; u < 4; ++u) add_pair(q[u]);
        }
        if (i > 0) {
          const unsigned q0 = qn[0], q1 = qn[1], q2 = qn[2];
          cp += 32 * i;
#pragma unroll
          for (int u = 0; u < 4; ++u) qn[u] = __ldg(cp + 32 * u);
          add_pair(q0);
          if (i > 1) add_pair(q1);
          if (i > 2) add_pair(q2);
        }
        const typename Pol::W wc = Pol::w(t, c);
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] += Pol::wmul(wc, sum[r]);
      }
      if (n_oct && t.xs_ok) {
        S s0[R], s1[R];
#pragma unroll
        for (int r = 0; r < R; ++r) s0[r] = s1[r] = 0;
        for (int h = 0; h < n_oct; ++h) {
          unsigned z[R];
#pragma unroll
          for (int r = 0; r < R; ++r) z[r] = in ? (s_ax[h][r] ^ bx) & s_vm[h][r] : 0u;
          const unsigned pm = t.xs_present[h];
          const uint4 mc = mv;
          if (h + 1 < n_oct) {
            mv = __ldg(t.B_xmap + (h + 1) * t.B_total + gB);
            bx = __ldg(t.B_xs + (h + 1) * t.B_total + gB);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const unsigned pj = (pm >> (4 * j)) & 15u;
            if (!pj) break;
            const unsigned mw = j < 2 ? mc.x : j < 4 ? mc.y : j < 6 ? mc.z : mc.w;
            const unsigned mq = (j & 1) ? mw >> 16 : mw & 0xFFFFu;
            S v[4][R];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
#pragma unroll
              for (int r = 0; r < R; ++r) v[s][r] = 0;
              if ((pj >> s) & 1u) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                  v[s][r] = ldg_if(s_ptr[h][4 * j + s][r] + mq, (z[r] & (1u << (4 * j + s))) != 0u);
              }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
              s0[r] += v[0][r] + v[1][r];
              s1[r] += v[2][r] + v[3][r];
            }
          }
        }
        const typename Pol::W w0 = Pol::w(t, t.xl_c[0]), w1 = Pol::w(t, t.xl_c[1]);
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] += Pol::wmul(w0, s0[r]) + Pol::wmul(w1, s1[r]);
      } else if (n_oct) {
        // more than two value classes on the cut: bond by bond
        unsigned z[R];
#pragma unroll
        for (int r = 0; r < R; ++r) z[r] = in ? (s_ax[0][r] ^ pb) & s_vm[0][r] : 0u;
        for (int k = 0; k < p.ncross; ++k) {
          const unsigned mq = __ldg(t.mapB + (long long)t.bond_ib[k] * t.B_total + gB);
          const typename Pol::W wk = Pol::bw(t, k);
#pragma unroll
          for (int r = 0; r < R; ++r)
            if ((z[r] >> k) & 1u) acc[r] += Pol::wmul(wk, __ldg(s_ptr[0][k][r] + mq));
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (in && r < nr) store_out<Pol>(y, row0 + (long long)r * dB + b, acc[r], final_, e2);
      if constexpr (Pol::kSplit) {
        if (final_ && in)  // no H_A pass: the FP64 diagonal is added here
          for (int r = 0; r < nr; ++r) {
            const long long i = row0 + (long long)r * dB + b;
            double* yd = reinterpret_cast<double*>(y) + i;
            const unsigned z = t.vab_and ? (pa[r] & pb) : (pa[r] ^ pb);
            *yd = fma(PF64::diag(t, bl.gA0 + a0 + r, gB, z), p.xd[i], *yd);
          }
      }
    }
  }
}

constexpr int kPanelCtas = 3;  // resident CTAs of the panel pass per SM

// H_A panel pass: work item = a run of rows of one block times a panel of
// 32 * NC columns.  A warp owns one output row of the panel at a time, a CTA
// the item's rows in ascending order: side-A neighbours that differ in low
// bits are a few rows away, so their panel segments (1 KB each) are found in
// L1, the others in L2, where the whole column panel stays resident.  The
// column indices of up to 32 entries are read by the 32 lanes at once and
// their row offsets broadcast entry by entry; U neighbour rows (U x NC
// independent loads per lane) are in flight before any is summed.  One CTA
// per item, started in item order, keeps every SM on the same one or two
// panels; a persistent grid drifts apart over many panels and loses the L2
// residency (J1-J2 4x8: 17 ms).
// Bound: latency of L2 (56 % of its throughput) and issue (53 %).  Measured,
// FP64 fixed point / FP32: J1-J2 4x8 (601 M states) 9.8 -> 7.8 / 5.4 -> 4.1 ms,
// Hubbard 4x4 (166 M states) 2.04 -> 1.65 / 1.16 -> 0.84 ms against one row and
// 256 columns per warp with per-entry index loads and 64-bit offsets.  Runs of
// 16 and 32 rows: 8.5 and 7.9 ms; two or four resident CTAs: 10.5 and 8.4 ms.
template <class Pol, int NC, int U>
__global__ void __launch_bounds__(256, kPanelCtas) k_panel4(P3 p, const long long* __restrict__ item_start, int rows,
                                                const typename Pol::S* __restrict__ x, typename Pol::Y* __restrict__ y,
                                                const int* __restrict__ emax) {
  using S = typename Pol::S;
  constexpr int W = 32 * NC;
  const Dev3& t = p.t;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();
  const int e2 = emax ? out_exp(t, emax[0]) : 0;
  // split diagonal: the weighted popcounts of the packed cut words from a
  // table (an FP64 conversion and product per element would double the FP64
  // instructions, which bound this store)
  __shared__ double s_vab[Pol::kSplit ? kMaxClasses : 1][33];
  if constexpr (Pol::kSplit) {
    for (int i = threadIdx.x; i < 33 * t.ncls_d; i += 256) s_vab[i / 33][i % 33] = t.dw64[i / 33] * (i % 33);
    __syncthreads();
  }
  const long long w = blockIdx.x;
  const int bi = find_blk(item_start, p.nblk, w);
  const DevBlock& bl = p.blocks[bi];
  const int nrun = (int)((bl.dA + rows - 1) / rows), q = (int)(w - item_start[bi]);
  const int col0 = q / nrun * W, row0 = q % nrun * rows, row1 = min(row0 + rows, (int)bl.dA);
  const unsigned dB = (unsigned)bl.dB;
  const long long off = bl.off, gA0 = bl.gA0;
  const unsigned b0 = col0 + lane;
  const bool full = col0 + W <= (int)dB;
  const S* xb0 = x + off + min(b0, dB - 1);
  for (int a = row0 + warp; a < row1; a += 8) {
    typename Pol::Y* yrow = y + off + (long long)a * dB + b0;
    const uint2 m = t.A_meta[gA0 + a];
    typename Pol::A acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c)
      acc[c] = typename Pol::A(full || b0 + 32 * c < dB ? yrow[32 * c] : (typename Pol::Y)0);
    const uint16_t* ep = t.A_col + m.x;
    const int tot = (int)((m.y & 255u) + ((m.y >> 8) & 255u) + ((m.y >> 16) & 255u) + (m.y >> 24));
    int pos = 0, cb = 0;
    unsigned ro = lane < tot ? (unsigned)ep[lane] * dB : 0u;  // row offset of entry cb + lane
    auto run = [&](auto FULL) {
      unsigned cc[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c)
        cc[c] = decltype(FULL)::value ? 32u * c : (b0 + 32 * c < dB ? 32u * c : 0u);
#pragma unroll
      for (int cl = 0; cl < kMaxCls; ++cl) {
        const int n = (int)((m.y >> (8 * cl)) & 255u);
        if (!n) continue;
        S sum[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) sum[c] = 0;
        for (int i = 0; i < n; i += U) {
          if (pos + U > cb + 32) {
            cb = pos;
            ro = cb + lane < tot ? (unsigned)ep[cb + lane] * dB : 0u;
          }
          S v[U][NC];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const S* rp = xb0 + __shfl_sync(0xffffffffu, ro, (pos - cb + u) & 31);
            if (u == 0 || i + u < n) {
#pragma unroll
              for (int c = 0; c < NC; ++c) v[u][c] = __ldg(rp + cc[c]);
            } else {
#pragma unroll
              for (int c = 0; c < NC; ++c) v[u][c] = 0;
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u)
#pragma unroll
            for (int c = 0; c < NC; ++c) sum[c] += v[u][c];
          pos += min(U, n - i);
        }
        const typename Pol::W wc = Pol::w(t, cl);
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] += Pol::wmul(wc, sum[c]);
      }
    };
    if (full) run(std::true_type{});
    else run(std::false_type{});
    if constexpr (Pol::kSplit) {
      const double da = t.A_d64[gA0 + a] + t.dc0_64;
      const unsigned pa = t.A_pack[gA0 + a];
      const double* xr = p.xd + (off + (long long)a * dB + b0);
      double xv[NC], d[NC];
      unsigned pb[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const bool in = full || b0 + 32 * c < dB;
        xv[c] = in ? xr[32 * c] : 0.0;
        d[c] = in ? t.B_d64[bl.gB0 + b0 + 32 * c] : 0.0;
        pb[c] = in ? t.B_pack[bl.gB0 + b0 + 32 * c] : 0u;
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const unsigned z = t.vab_and ? (pa & pb[c]) : (pa ^ pb[c]);
        double v = da + d[c];
        for (int q = 0; q < t.ncls_d; ++q) v += s_vab[q][__popc(z & t.dmask[q])];
        if (full || b0 + 32 * c < dB)
          reinterpret_cast<double*>(yrow)[32 * c] = fma(v, xv[c], from_fixed(acc[c], e2));
      }
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (full || b0 + 32 * c < dB) store_out<Pol>(yrow, 32 * c, acc[c], true, e2);
    }
  }
}

static P3 make_p3(const ed_ctx* c) {
  P3 p;
  p.t = c->t3;
  p.blocks = c->d_blocks;
  p.nblk = (int)c->blocks.size();
  p.ncross = c->kind == ED_SPIN ? (int)c->cross.size() : 0;
  p.xd = nullptr;
  return p;
}

// dynamic shared memory of the row pass: the R rows (16 bytes a column) of the
// widest block and eight zero slots
static size_t v3_smem(const ed_ctx* c) {
  long long mdb = 1;
  for (const auto& b : c->blocks) mdb = std::max<long long>(mdb, b.dB);
  return (size_t)(mdb + 8) * 16;
}

constexpr size_t kRowMax = 220 * 1024;      // most row bytes of the row pass
constexpr size_t kRowHalf = 106 * 1024;     // for two CTAs of it per SM
constexpr size_t kRowQuarter = 50 * 1024;   // for four

bool v3_usable(const ed_ctx* c, ed_dtype dt, const void* x) {
  (void)dt;
  return c->v3_ok && ((uintptr_t)x % 16) == 0 && v3_smem(c) <= kRowMax;
}

// events bracketing the stages of one apply when profiling is on
struct ProfMarks {
  cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  bool on = false;
  void begin(ed_ctx* c) {
    on = c->prof;
    if (!on) return;
    for (auto& e : ev) cudaEventCreate(&e);
  }
  void mark(int i, cudaStream_t st) {
    if (on) cudaEventRecord(ev[i], st);
  }
  void end(ed_ctx* c) {
    if (!on) return;
    for (auto& e : ev) c->prof_ev.push_back(e);
  }
};

// x: the pass's input (CVT: the FP64 vector, whose fixed-point copy goes to
// xw); xd: the FP64 vector of a split diagonal
template <class Pol, bool CVT = false>
static ed_status run_v3(ed_ctx* c, const std::conditional_t<CVT, double, typename Pol::S>* x, typename Pol::Y* y,
                        int* emax, cudaStream_t st, ProfMarks& pm, const double* xd = nullptr,
                        typename Pol::S* xw = nullptr, const int* part = nullptr, int npart = 0) {
  P3 p = make_p3(c);
  p.xd = xd;
  if (c->n_rows == 0) return ED_OK;
  constexpr int R = 16 / (int)sizeof(typename Pol::S);
  const size_t smem = v3_smem(c);
  const int sms = n_sms(c->device);
  pm.mark(2, st);
  {
    const long long* gs = R == 4 ? c->d_grp4_start : c->d_grp2_start;
    const long long ng = R == 4 ? c->n_grp4 : c->n_grp2;
    // 1024 threads per SM: in one CTA while its rows need more than half of
    // the shared memory, else in two or four CTAs, so that one stages its
    // rows while another sums.  (The attribute is the function's: the same value
    // for every context, so that another thread's cannot come between it and
    // the launch.)
    auto go = [&](auto kern, int nt, size_t most) -> ed_status {
      ED_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
      const long long grid = std::min<long long>(ng, (long long)sms * (1024 / nt));
      ED_CUDA_TRY(launch_pdl(kern, grid, nt, smem, st, p, gs, ng, x, y, emax, xw, part, npart));
      return ED_OK;
    };
    if (smem > kRowHalf) ED_TRY(go(k_row5<Pol, R, 1024, CVT>, 1024, kRowMax));
    else if (smem > kRowQuarter) ED_TRY(go(k_row5<Pol, R, 512, CVT>, 512, kRowHalf));
    else ED_TRY(go(k_row5<Pol, R, 256, CVT>, 256, kRowQuarter));
  }
  pm.mark(3, st);
  constexpr int q = sizeof(typename Pol::S) == 4 ? 1 : 0;
  if (c->n_panel[q] > 0) {
    // 1 KB of a row per panel: 128 columns of 8-byte types with four neighbour
    // rows in flight, 256 of FP32 with two
    const long long* is = c->d_panel_start + q * (c->blocks.size() + 1);
    const typename Pol::S* xp;
    if constexpr (CVT) xp = xw;
    else xp = x;
    ED_CUDA_TRY(launch_pdl(k_panel4<Pol, q ? 8 : 4, q ? 2 : 4>, c->n_panel[q], 256, 0, st, p, is, c->panel_rows[q], xp,
                           y, (const int*)emax));
  }
  return ED_OK;
}

// fixed-point passes of the context's arithmetic: x is the fixed-point copy
// (CVT: the FP64 vector), xd the FP64 vector
template <bool CVT>
static ed_status run_fixed(ed_ctx* c, const std::conditional_t<CVT, double, long long>* x, const double* xd, double* y,
                           int* emax, cudaStream_t st, ProfMarks& pm, long long* xw = nullptr,
                           const int* part = nullptr, int npart = 0) {
  if (c->diag_split) return run_v3<PI64S, CVT>(c, x, (long long*)y, emax, st, pm, xd, xw, part, npart);
  if (c->dyadic) return run_v3<PI64, CVT>(c, x, (long long*)y, emax, st, pm, xd, xw, part, npart);
  if (c->wide) return run_v3<PW, CVT>(c, x, y, emax, st, pm, xd, xw, part, npart);
  return run_v3<PC64, CVT>(c, x, y, emax, st, pm, xd, xw, part, npart);
}

// exact fixed-point FP64 apply with explicit scratch: `fixed` holds D 64-bit
// integers; the exponents go through the context's exponent scratch
static ed_status apply_fixed(ed_ctx* c, const double* x, double* y, long long* fixed, cudaStream_t st, ProfMarks& pm) {
  const long long n = c->D;
  if (n < 1) return ED_OK;
  const int sms = n_sms(c->device);
  int* emax = c->d_exp;
  int* part = c->d_exp + 16;
  const int g = (int)std::min<long long>({(n + 511) / 512, (long long)sms * 8, (long long)kExpParts});
  pm.mark(0, st);
  ED_CUDA_TRY(launch_pdl(k_exp_max, g, 256, 0, st, x, n, part));
  pm.mark(1, st);
  // without cross terms only whole rows and the panel pass read the copy: the
  // row pass makes it, where several CTAs per SM hide the conversion (12-site
  // Hubbard ring 30 -> 26 us, 41 M-state impurity 0.45 -> 0.39 ms for the two;
  // with one CTA per SM, Hubbard 4x4, it is 2.08 against 1.65 + 0.41 ms)
  if ((c->kind != ED_SPIN || c->cross.empty()) && v3_smem(c) <= kRowHalf)
    return run_fixed<true>(c, x, x, y, emax, st, pm, fixed, part, g);
  ED_CUDA_TRY(launch_pdl(k_to_fixed, g, 256, 0, st, x, fixed, n, (const int*)part, g, emax, c->t3.P));
  return run_fixed<false>(c, fixed, x, y, emax, st, pm);
}

// fixed-point input: exact integer sums, with small integer weights (dyadic
// couplings), with 64-bit integer weights into 128-bit sums (other couplings)
// or, when their range is too wide for that, with FP64 weights per value class
static bool fixed_mode(const ed_ctx* c) { return c->dyadic || c->classed; }

bool fixed_path(const ed_ctx* c, const void* x) { return fixed_mode(c) && v3_usable(c, ED_F64, x); }

ed_status apply_prepared_fixed(ed_ctx* c, const double* x, double* y, cudaStream_t st) {
  if (!c->d_fixed) {
    set_error("fixed-point input was not prepared");
    return ED_EINVAL;
  }
  ProfMarks pm;
  pm.begin(c);
  pm.mark(0, st);
  pm.mark(1, st);
  const ed_status r = run_fixed<false>(c, c->d_fixed, x, y, c->d_exp, st, pm);
  pm.mark(4, st);
  pm.end(c);
  return r;
}

ed_status apply_v3(ed_ctx* c, const void* x, void* y, ed_dtype dt, cudaStream_t st) {
  ProfMarks pm;
  pm.begin(c);
  ed_status r;
  if (dt == ED_F32 || !fixed_mode(c)) {
    pm.mark(0, st);
    pm.mark(1, st);
    r = dt == ED_F32 ? run_v3<PF32>(c, (const float*)x, (float*)y, nullptr, st, pm)
                     : run_v3<PF64>(c, (const double*)x, (double*)y, nullptr, st, pm);
  } else {
    // exact fixed point: exponent of max|x|, scaled copy, integer passes
    if (!c->d_fixed) ED_TRY(dev_alloc(c, (void**)&c->d_fixed, (size_t)std::max<long long>(c->D, 2) * 8));
    r = apply_fixed(c, (const double*)x, (double*)y, c->d_fixed, st, pm);
  }
  pm.mark(4, st);
  pm.end(c);
  return r;
}

// ---------------------------------------------------------------- apply without allocation

// Scratch of ed_apply_H_noalloc: a file-scope device array (a header that the
// size limit counts, then the 64-bit fixed-point copy of x; the exponents go
// through the context's own scratch).  Every GPU
// that loads this library holds it until the process exits.
constexpr size_t kNoAllocScratchBytes = (size_t)32 << 20;
constexpr size_t kNoAllocHeader = 256;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kNoAllocMaxDevices = 64;
static std::mutex g_noalloc_mu;
static void* g_noalloc_ptr[kNoAllocMaxDevices] = {};

// device address of the scratch on the current device; the first call on a
// device looks it up (cudaGetSymbolAddress) and caches it
static ed_status noalloc_scratch(int dev, unsigned char** out) {
  if (dev < 0 || dev >= kNoAllocMaxDevices) {
    set_error("device %d outside the %d devices the scratch table covers", dev, kNoAllocMaxDevices);
    return ED_EUNSUPPORTED;
  }
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      set_error("cudaGetSymbolAddress of the static scratch failed on device %d: %s", dev, cudaGetErrorString(e));
      return ED_ECUDA;
    }
    g_noalloc_ptr[dev] = p;
  }
  *out = (unsigned char*)g_noalloc_ptr[dev];
  return ED_OK;
}

}  // namespace edk

using namespace edk;

extern "C" ed_status ed_apply_H_noalloc(ed_ctx* c, const void* x, void* y, void* stream) {
  if (!c) { set_error("ctx is NULL"); return ED_EINVAL; }
  if (!c->ops_built) { set_error("ed_build_local_ops has not been called"); return ED_EINVAL; }
  if (c->D > 0 && (!x || !y)) { set_error("x or y is NULL"); return ED_EINVAL; }
  const size_t need = kNoAllocHeader + (size_t)c->D * sizeof(long long);
  if (fixed_mode(c) && need > kNoAllocScratchBytes) {
    set_error("ed_apply_H_noalloc: %lld states need %zu bytes of scratch, the static scratch holds %zu "
              "(at most %zu states)", (long long)c->D, need, kNoAllocScratchBytes,
              (kNoAllocScratchBytes - kNoAllocHeader) / sizeof(long long));
    return ED_EINVAL;
  }
  const char* xb = (const char*)x;
  const char* yb = (const char*)y;
  if (c->D > 0 && xb < yb + c->D * 8 && yb < xb + c->D * 8) { set_error("x and y overlap"); return ED_EINVAL; }
  if (!v3_usable(c, ED_F64, x)) {
    set_error("ed_apply_H_noalloc needs the class-sorted kernels (16-byte aligned x, at most 4 value classes, "
              "32 cross bonds and 65534 states per side charge)");
    return ED_EUNSUPPORTED;
  }
  ED_DEVICE_SCOPE(c->device);
  cudaStream_t st = (cudaStream_t)stream;
  ProfMarks pm;  // no profiling events here
  if (!fixed_mode(c)) return run_v3<PF64>(c, (const double*)x, (double*)y, nullptr, st, pm);
  unsigned char* base = nullptr;
  ED_TRY(noalloc_scratch(c->device, &base));
  return apply_fixed(c, (const double*)x, (double*)y, (long long*)(base + kNoAllocHeader), st, pm);
}



extern "C" int ed_row_pass(const ed_ctx* c, ed_dtype dt) {
  if (!c || !c->ops_built) return -1;
  if (!v3_usable(c, dt, (const void*)(uintptr_t)256)) return 0;  // any 16-byte aligned x
  return 1;
}

extern "C" int ed_fp64_mode(const ed_ctx* c) {
  if (!c || !c->ops_built) return -1;
  if (c->dyadic) return 1;
  if (c->classed) return c->wide ? 2 : 3;
  return 0;
}

extern "C" ed_status ed_profile_enable(ed_ctx* c, int enable) {
  if (!c) { set_error("ctx is NULL"); return ED_EINVAL; }
  c->prof = enable != 0;
  return ED_OK;
}

extern "C" ed_status ed_profile_read(ed_ctx* c, double* ms, int64_t* count, int reset) {
  if (!c) { set_error("ctx is NULL"); return ED_EINVAL; }
  for (size_t i = 0; i + 5 <= c->prof_ev.size(); i += 5) {
    cudaEvent_t* e = &c->prof_ev[i];
    ED_CUDA_TRY(cudaEventSynchronize(e[4]));
    for (int k = 0; k < 4; ++k) {
      float t = 0.f;
      ED_CUDA_TRY(cudaEventElapsedTime(&t, e[k], e[k + 1]));
      c->prof_ms[k] += t;
    }
    ++c->prof_count;
    for (int k = 0; k < 5; ++k) cudaEventDestroy(e[k]);
  }
  c->prof_ev.clear();
  if (ms)
    for (int k = 0; k < 4; ++k) ms[k] = c->prof_ms[k];
  if (count) *count = c->prof_count;
  if (reset) {
    for (double& v : c->prof_ms) v = 0.0;
    c->prof_count = 0;
  }
  return ED_OK;
}
