// Dense H|psi> of small batched instances on the tensor cores.
//
// An instance is one block Psi (d_A x d_B, row-major) of a Hubbard model
// with the spin cut, which leaves no cross terms, so Eq. (2) reads
//   H psi = H_A Psi + Psi H_B^T + V o Psi
// with the side operators H_A, H_B (hopping of the up and of the down
// electrons) and the diagonal V.  Both products run as BF16 tcgen05 MMAs with
// FP32 accumulation in TMEM.  Every FP32 value v (of H_A, H_B and Psi) is
// split into three BF16 pieces v = h0 + h1 + h2 (8 significant bits each,
// 24 in all, each piece the rounding of what the previous ones leave); the
// piece products h_p(H) h_q(Psi) with p + q <= 2 are accumulated in FP32,
// the dropped ones (p + q >= 3) being below 2^-24 of the leading product.
// The leading products (p = q = 0) and the corrections (p + q = 1, 2) go into
// separate accumulators (64-wide tiles: one per order), so the rounding of the
// many small correction sums does not fall on the large leading sum; both
// products of an output tile (they add) share them, and the epilogue adds them
// and the diagonal.
//
// Per output tile (128 rows a x BN columns b): the K steps of H_A Psi
// (A operand: H_A's pieces, rows a, K = a' contiguous; B operand: Psi's pieces,
// rows a' of BN columns, the MN-major form, so no transposed copy of Psi is
// written or read) and then those of Psi H_B^T (A: Psi's pieces, rows a; B:
// H_B's pieces, rows b, both K = b' contiguous).  Tiles staged by TMA with
// 128-byte swizzle, one thread issues the MMAs, eight warps drain the
// accumulators (those of two tiles alternate, so the epilogue of one tile
// overlaps the products of the next).  Persistent: the CTAs take the tiles of
// the active instances from a counter, those with the most K steps first.
#include <cuda_bf16.h>

#include <cstring>

#include "apply3.cuh"  // pdl_wait, launch_pdl
#include "batch.h"
#include "batch_dev.cuh"
#include "tc.cuh"

namespace edk {

constexpr int kBdEpiWarps = 8;   // two per TMEM lane quarter, splitting the columns
// warps 0-7 epilogue, 8 TMA producer, 9 MMA issuer, 10 tile list
constexpr int kBdThreads = 32 * (kBdEpiWarps + 3);
constexpr int kBdWarpTma = kBdEpiWarps, kBdWarpMma = kBdEpiWarps + 1, kBdWarpList = kBdEpiWarps + 2;
constexpr int kBdTiles = 4;      // tiles that the list warp is ahead
constexpr int kBdTrans = 32 * 9;  // floats of one warp's transpose buffer (32 rows x 8 columns, odd stride)
constexpr int kBdBM = 128;       // output rows per tile (UMMA M)
constexpr int kBdBK = 64;        // K per pipeline step: one 128-byte swizzle row of BF16
constexpr int kBdPieces = 3;
constexpr int kBdXTile = 64 * kBdBK * 2;  // a box of Psi in the B role: 8 KB
constexpr long long kBdSpin = 1ll << 26;  // bounded waits (about a second)

// tensor maps of one slot: the A roles (H_A, Psi) with 128-row boxes, Psi in
// the B role with 64-row boxes, H_B with BN-row boxes
enum { kMapHA = 0, kMapXN = 1, kMapXB = 2, kMapHB64 = 3, kMapHB128 = 4 };

template <int BN>
struct BdCfg {
  static constexpr int kStages = BN == 64 ? 3 : 2;
  static constexpr int kATile = kBdBM * kBdBK * 2;  // one piece: 16 KB
  static constexpr int kBTile = BN * kBdBK * 2;
  static constexpr int kStage = kBdPieces * (kATile + kBTile);  // 72 or 96 KB
  // accumulators of a tile: the leading products, and the corrections p + q =
  // 1 and 2 (one accumulator for both at BN = 128, where TMEM has no more)
  static constexpr int kAcc = BN == 64 ? 3 : 2;
  static constexpr int kTmemCols = 512;  // two tiles in flight (a power of two of columns)
  static constexpr size_t kSmem = 1024 + (size_t)kStages * kStage + 512 + (size_t)kBdEpiWarps * kBdTrans * 4;
};

// ---------------------------------------------------------------- pieces

__device__ __forceinline__ void split3_dev(float v, uint16_t& h0, uint16_t& h1, uint16_t& h2) {
  const __nv_bfloat16 a = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(a);
  const __nv_bfloat16 b = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(b);
  const __nv_bfloat16 c = __float2bfloat16_rn(r2);
  h0 = __bfloat16_as_ushort(a);
  h1 = __bfloat16_as_ushort(b);
  h2 = __bfloat16_as_ushort(c);
}

// the pieces of two neighbours, each pair in one word (the first in its low half)
__device__ __forceinline__ void split3_pair(float a, float b, uint32_t& h0, uint32_t& h1, uint32_t& h2) {
  auto pack = [](float lo, float hi) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    uint32_t u;
    memcpy(&u, &t, 4);
    return u;
  };
  auto low = [](uint32_t u) { return __uint_as_float(u << 16); };
  auto high = [](uint32_t u) { return __uint_as_float(u & 0xffff0000u); };
  h0 = pack(a, b);
  const float a1 = a - low(h0), b1 = b - high(h0);
  h1 = pack(a1, b1);
  h2 = pack(a1 - low(h1), b1 - high(h1));
}

// Pieces of Psi for every dense instance, in units of 64 x 64 elements; a warp
// takes eight rows, whose loads are all in flight, a lane two neighbouring
// columns, so a warp writes 128 bytes along a row.  The piece rows start on
// multiples of 64 elements: pairs at even columns are 4-byte aligned.
__global__ void __launch_bounds__(256) k_bslice(BDenseArgs g) {
  if (blockIdx.x == 0 && threadIdx.x < 2) g.next[threadIdx.x] = 0;  // the tile counters of the products
  const int n = g.cnt[1];
  if (n <= 0) return;
  const long long total = g.dspref[n];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (long long u = blockIdx.x; u < total; u += gridDim.x) {
    const int ai = find_pref(g.dspref, n, u);
    const BInst& I = g.insts[g.didx[ai]];
    const int dA = I.dA, dB = I.dB;
    const long long t = u - g.dspref[ai];
    const int tnb = (dB + 63) >> 6;
    const int a0 = (int)(t / tnb) * 64 + warp, b = (int)(t % tnb) * 64 + 2 * lane;
    if (b >= dB) continue;
    const bool two = b + 1 < dB;
    const float* __restrict__ x = (g.user_mode ? g.ux + I.uoff : g.arena + I.voff + I.D) + b;
    uint32_t* __restrict__ d = reinterpret_cast<uint32_t*>(I.XN + b);
    const long long kw = I.KpB / 2, pw = (long long)dA * kw;  // words of a row, of a piece
    float v[8], w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int a = a0 + 8 * i;
      v[i] = a < dA ? __ldg(x + (long long)a * dB) : 0.f;
      w[i] = a < dA && two ? __ldg(x + (long long)a * dB + 1) : 0.f;  // zero past d_B: the padding of the row
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int a = a0 + 8 * i;
      if (a < dA) {
        uint32_t h0, h1, h2;
        split3_pair(v[i], w[i], h0, h1, h2);
        d[a * kw] = h0;
        d[a * kw + pw] = h1;
        d[a * kw + 2 * pw] = h2;
      }
    }
  }
}

// ---------------------------------------------------------------- tables

// Dense H_A, H_B pieces and their nonzero-K-block masks from the instance's
// CSR rows (zeroed beforehand): one thread per row of either side; entries
// with the same column are summed before the split.
__global__ void k_btables(BInst I) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool onA = r < I.dA;
  if (r >= (long long)I.dA + I.dB) return;
  const long long row = onA ? r : r - I.dA;
  const int d = onA ? I.dA : I.dB;
  const int* rp = onA ? I.A_rp : I.B_rp;
  const int* col = onA ? I.A_col : I.B_col;
  const float* val = onA ? I.A_val : I.B_val;
  uint16_t* P = const_cast<uint16_t*>(onA ? I.HA : I.HB);
  const int kp = onA ? I.KpA : I.KpB;
  const long long plane = (long long)d * kp;
  uint32_t* km = const_cast<uint32_t*>(I.kmask);
  const int tmA = (I.dA + kBdBM - 1) / kBdBM, tn64 = (I.dB + 63) / 64;
  for (int e = rp[row]; e < rp[row + 1]; ++e) {
    const int c = col[e];
    bool seen = false;
    for (int f = rp[row]; f < e; ++f) seen = seen || col[f] == c;
    if (seen) continue;
    float v = 0.f;
    for (int f = e; f < rp[row + 1]; ++f)
      if (col[f] == c) v += val[f];
    uint16_t h0, h1, h2;
    split3_dev(v, h0, h1, h2);
    P[row * kp + c] = h0;
    P[plane + row * kp + c] = h1;
    P[2 * plane + row * kp + c] = h2;
    const uint32_t bit = 1u << (c / kBdBK);
    if (onA) {
      atomicOr(&km[row / kBdBM], bit);
    } else {
      atomicOr(&km[tmA + row / 64], bit);
      atomicOr(&km[tmA + tn64 + row / 128], bit);
    }
  }
}

ed_status bdense_tables(const BInst& I, cudaStream_t st) {
  const long long n = (long long)I.dA + I.dB;
  k_btables<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(I);
  ED_CUDA_TRY(cudaGetLastError());
  return ED_OK;
}

// ---------------------------------------------------------------- products

// K steps of one output tile: the nonzero 64-wide K blocks of H_A's row
// tile (H_A Psi), then those of H_B's row tile (Psi H_B^T); entry = kb, plus
// 32 for the second product (kb < 16 as d <= 1024).  A tile with none gets
// one zero block (which clears its accumulators).
template <int BN>
__device__ __forceinline__ int tile_steps(const BInst& I, int m0, int n0, unsigned char* ks, int& nA) {
  const int tmA = (I.dA + kBdBM - 1) / kBdBM, tn64 = (I.dB + 63) / 64;
  const uint32_t ma = I.kmask[m0 / kBdBM];
  const uint32_t mb = BN == 64 ? I.kmask[tmA + n0 / 64] : I.kmask[tmA + tn64 + n0 / 128];
  int n = 0;
  for (uint32_t m = ma; m; m &= m - 1) ks[n++] = (unsigned char)__ffs(m) - 1;
  if (ma == 0 && mb == 0) ks[n++] = 0;
  nA = n;
  for (uint32_t m = mb; m; m &= m - 1) ks[n++] = (unsigned char)(32 + __ffs(m) - 1);
  return n;
}

// one entry of a CTA's tile list
struct BdTile {
  int slot, m0, n0, nk, nA;
  unsigned char ks[32];  // the K steps, the first nA of H_A Psi (tile_steps)
};

// Bound: operands from L2 (a K step moves 72 KB for a 128 x 64 tile, 96 KB for
// 128 x 128; 5.7 and 4.1 GB for 512 Hubbard instances of 26 M states, 16 and 11
// TB/s), the tensor pipe active 44 and 47 % of the time.  Of that batch's
// H|psi>, with 64-wide / 128-wide tiles: 694 / 537 us with two stages, N = BN
// instructions, Psi^T sliced beside Psi and every CTA looking up its own tiles;
// 538 / 542 with three stages (64-wide), N up to 192 and no prefetch into L2,
// which moved every operand twice through L2's ports; 506 / 545 with the list
// warp; 449 / 462 without Psi^T (slicing 114 -> 59 us, 0.2 GB less from HBM);
// 439 / 451 with the launches overlapped; 432 / 448 without 64-bit divisions and
// with ready descriptors in the issuing thread.  Tried and slower: barriers per piece
// instead of per K step (608 / 549), operands prefetched once per row or column
// of tiles (531 / 560).
template <int BN>
__global__ void __launch_bounds__(kBdThreads, 1) k_bgemm(BDenseArgs g, int which) {
  using C = BdCfg<BN>;
  // Both widths wait for the kernel before them in the stream, and so does
  // k_bapply: a grid that was released early sees what earlier grids wrote only
  // after its own wait.  The early release still lets the 128-wide launch be set
  // up while the last 64-wide tiles run.
  pdl_wait();
  if (BN == 64) pdl_trigger();
  const int n = g.cnt[which];
  const int* vidx = BN == 64 ? g.idx64 : g.idx128;
  const long long* tpref = BN == 64 ? g.tpref64 : g.tpref128;
  const long long total = n > 0 ? tpref[n] : 0;
  if (total <= 0) return;

  extern __shared__ unsigned char sm_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)sm_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(sm + C::kStages * C::kStage);  // kStages
  uint64_t* empty = full + C::kStages;                       // kStages
  uint64_t* acc_full = empty + C::kStages;                   // 2
  uint64_t* acc_empty = acc_full + 2;                        // 2
  uint64_t* mma_done = acc_empty + 2;
  uint64_t* ti_full = mma_done + 1;                          // kBdTiles
  uint64_t* ti_empty = ti_full + kBdTiles;                   // kBdTiles
  float* trans = (float*)(sm + C::kStages * C::kStage + 512);  // kBdEpiWarps x [32][9]
  __shared__ BdTile s_tile[kBdTiles];
  __shared__ unsigned s_tmem;
  __shared__ volatile int s_abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < C::kStages; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < kBdTiles; ++i) {
      tc::mbar_init(&ti_full[i], 1);
      tc::mbar_init(&ti_empty[i], 2 + kBdEpiWarps);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&acc_full[i], 1);
      tc::mbar_init(&acc_empty[i], 32 * kBdEpiWarps);
    }
    tc::mbar_init(mma_done, 1);
    tc::fence_mbar_init();
    s_abort = 0;
  }
  if (warp == 0) tc::tmem_alloc(&s_tmem, C::kTmemCols);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const unsigned tmem = s_tmem;

  // the list entry of this CTA's tile tl, once it is written; nullptr at the
  // list's end and when the wait ran out
  auto tile_at = [&](int tl) -> const BdTile* {
    if (!tc::mbar_wait(&ti_full[tl % kBdTiles], (unsigned)((tl / kBdTiles) & 1), kBdSpin)) {
      s_abort = 1;
      return nullptr;
    }
    const BdTile* T = &s_tile[tl % kBdTiles];
    return T->nk > 0 ? T : nullptr;
  };

  if (warp == kBdWarpList) {
    // ---- tile list: a tile's instance (a binary search in global memory),
    // origin and K steps are looked up tiles ahead of their use -- done by the
    // producer itself, the lookups (5,000 cycles) drained its stages -- and
    // its tensor maps fetched
    if (lane == 0) {
      for (int tl = 0; !s_abort; ++tl) {
        const long long tile = (long long)atomicAdd(&g.next[BN == 64 ? 0 : 1], 1ull);
        const int e = tl % kBdTiles, u = tl / kBdTiles;
        if (u > 0 && !tc::mbar_wait(&ti_empty[e], (unsigned)((u - 1) & 1), kBdSpin)) {
          s_abort = 1;
          break;
        }
        if (tile >= total) {  // no K steps: the end of the list
          s_tile[e].nk = 0;
          tc::mbar_arrive(&ti_full[e]);
          break;
        }
        const int ai = find_pref(tpref, n, tile);
        const int slot = vidx[ai];
        const BInst& I = g.insts[slot];
        const int tn = (I.dB + BN - 1) / BN;
        const long long t = tile - tpref[ai];
        BdTile& T = s_tile[e];
        T.slot = slot;
        T.m0 = (int)(t / tn) * kBdBM;
        T.n0 = (int)(t % tn) * BN;
        const CUtensorMap* mp = g.maps + (long long)slot * kBMaps;
        tc::tma_prefetch_map(mp + kMapHA);
        tc::tma_prefetch_map(mp + kMapXN);
        tc::tma_prefetch_map(mp + kMapXB);
        tc::tma_prefetch_map(mp + (BN == 64 ? kMapHB64 : kMapHB128));
        T.nk = tile_steps<BN>(I, T.m0, T.n0, T.ks, T.nA);
        tc::mbar_arrive(&ti_full[e]);
      }
      if (s_abort) atomicExch(g.err, 1);
    }
  } else if (warp == kBdWarpTma) {
    // ---- TMA producer: per K step the three pieces of the A tile and of the B tile
    if (lane == 0) {
      int s = 0;  // the stage, and the parity of its phase
      unsigned ph = 0;
      for (int tl = 0; !s_abort; ++tl) {
        const BdTile* T = tile_at(tl);
        if (!T) break;
        const int m0 = T->m0, n0 = T->n0, nk = T->nk;
        const CUtensorMap* mp = g.maps + (long long)T->slot * kBMaps;
        const CUtensorMap* mHB = mp + (BN == 64 ? kMapHB64 : kMapHB128);
        for (int ks = 0; ks < nk; ++ks) {
          // (a fresh barrier passes the wait for the phase before its first)
          if (!tc::mbar_wait(&empty[s], ph ^ 1u, kBdSpin)) {
            s_abort = 1;
            break;
          }
          unsigned char* sa = sm + s * C::kStage;
          unsigned char* sb = sa + kBdPieces * C::kATile;
          const bool first = ks < T->nA;  // H_A Psi, then Psi H_B^T
          const int kc = (T->ks[ks] & 31) * kBdBK;
          const CUtensorMap* ma = first ? mp + kMapHA : mp + kMapXN;
          tc::mbar_expect_tx(&full[s], C::kStage);
#pragma unroll
          for (int p = 0; p < kBdPieces; ++p) tc::tma_load_3d(sa + p * C::kATile, ma, kc, m0, p, &full[s]);
          if (first) {  // Psi, 64 rows a' of 64 columns b each
#pragma unroll
            for (int q = 0; q < kBdPieces * BN / 64; ++q)
              tc::tma_load_3d(sb + q * kBdXTile, mp + kMapXB, n0 + 64 * (q % (BN / 64)), kc, q / (BN / 64), &full[s]);
          } else {
#pragma unroll
            for (int q = 0; q < kBdPieces; ++q) tc::tma_load_3d(sb + q * C::kBTile, mHB, kc, n0, q, &full[s]);
          }
          if (++s == C::kStages) {
            s = 0;
            ph ^= 1u;
          }
        }
        tc::mbar_arrive(&ti_empty[tl % kBdTiles]);
      }
      if (s_abort) atomicExch(g.err, 1);
    }
  } else if (warp == kBdWarpMma) {
    // ---- MMA issuer: piece pairs p + q <= 2 into the tile's accumulators
    if (lane == 0) {
      // descriptors of the first stage: A, and B as rows of Psi or of H_B
      const uint64_t dA = tc::sdesc_kmajor_sw128(sm);
      const uint64_t dX = tc::sdesc_mnmajor_sw128(sm + kBdPieces * C::kATile, kBdXTile);
      const uint64_t dH = tc::sdesc_kmajor_sw128(sm + kBdPieces * C::kATile);
      int s = 0;  // the stage, and the parity of its phase
      unsigned ph = 0;
      for (int tl = 0; !s_abort; ++tl) {
        const BdTile* T = tile_at(tl);
        if (!T) break;
        const int nk = T->nk, nA = T->nA;
        tc::mbar_arrive(&ti_empty[tl % kBdTiles]);
        const int buf = tl & 1, use = tl >> 1;
        if (use > 0 && !tc::mbar_wait(&acc_empty[buf], (unsigned)((use - 1) & 1), kBdSpin)) {
          s_abort = 1;
          break;
        }
        tc::tc_fence_after();
        const unsigned dt = tmem + (unsigned)(C::kAcc * buf * BN);
        for (int ks = 0; ks < nk; ++ks) {
          if (!tc::mbar_wait(&full[s], ph, kBdSpin)) {
            s_abort = 1;
            break;
          }
          tc::tc_fence_after();
          // B's pieces lie behind one another in shared memory and the
          // accumulators in TMEM, so one instruction of N = np BN takes np
          // pairs (p, q), (p, q + 1), ... whose accumulators differ
          const bool first = ks < nA;
          auto pairs = [&](int p, int q, int np, int acc) {
            const unsigned idesc = tc::idesc_bf16_f32(kBdBM, np * BN) | (first ? tc::kIdescBMnMajor : 0u);
            const uint64_t da = dA + (unsigned)((s * C::kStage + p * C::kATile) / 16);
            const uint64_t db = (first ? dX : dH) + (unsigned)((s * C::kStage + q * C::kBTile) / 16);
            // 16 of K per instruction: 32 bytes along a K-major row, 16 rows of Psi
            const int kb = first ? 16 * 128 / 16 : 2;
#pragma unroll
            for (int kk = 0; kk < kBdBK / 16; ++kk)
              tc::mma_bf16(dt + (unsigned)(acc * BN), da + 2 * kk, db + kb * kk, idesc,
                           !(ks == 0 && p == 0 && q == 0 && kk == 0));
          };
          if (BN == 64) {
            pairs(0, 0, 3, 0);
            pairs(1, 0, 2, 1);
            pairs(2, 0, 1, 2);
          } else {
            pairs(0, 0, 2, 0);
            pairs(0, 2, 1, 1);
            pairs(1, 0, 1, 1);
            pairs(1, 1, 1, 1);
            pairs(2, 0, 1, 1);
          }
          tc::mma_commit(&empty[s]);
          if (++s == C::kStages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (s_abort) break;
        tc::mma_commit(&acc_full[buf]);
      }
      // every issued MMA finishes before the accumulators are released
      tc::mma_commit(mma_done);
      if (!tc::mbar_wait(mma_done, 0, kBdSpin)) s_abort = 1;
      if (s_abort) atomicExch(g.err, 1);
    }
  } else {
    // ---- epilogue: warp w drains TMEM lanes 32 (w % 4) .. + 31 (tile rows)
    // for every other 32-column chunk; each 32 x 8 part of it goes through
    // shared memory so the loads of x and the stores of y = accumulators + V x
    // move whole 32-byte sectors along rows
    const int quarter = warp & 3, half = warp >> 2;
    float* tr = trans + warp * kBdTrans;
    for (int tl = 0;; ++tl) {
      const BdTile* T = tile_at(tl);
      if (!T) break;
      const int m0 = T->m0, n0 = T->n0;
      const BInst& I = g.insts[T->slot];
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ti_empty[tl % kBdTiles]);
      const int buf = tl & 1, use = tl >> 1;
      bool ok = false;
      for (long long i = 0; i < kBdSpin && !ok; ++i) {
        ok = tc::mbar_try(&acc_full[buf], (unsigned)(use & 1));
        if (!ok && s_abort) break;
      }
      if (!ok) {
        s_abort = 1;
        break;
      }
      tc::tc_fence_after();
      // the instance's fields in registers (y stores could alias them otherwise)
      const int dA = I.dA, dB = I.dB;
      const int r0 = m0 + quarter * 32;  // this warp's first row
      const float* __restrict__ x = g.user_mode ? g.ux + I.uoff : g.arena + I.voff + I.D;
      float* __restrict__ y = g.user_mode ? g.uy + I.uoff : g.arena + I.voff + 2 * I.D;
      const uint32_t* __restrict__ Bs = I.B_str;
      const float* __restrict__ Bd = I.B_diag;
      const int ncls = I.ncls, vand = I.vab_and;
      float w[kMaxClasses];
      unsigned mk[kMaxClasses];
#pragma unroll
      for (int q = 0; q < kMaxClasses; ++q) {
        w[q] = I.w[q];
        mk[q] = I.mask[q];
      }
      // lane r holds row r0 + r's side-A string and diagonal
      const int nr = min(32, dA - r0);  // rows of this warp inside the block (may be <= 0)
      float dal = 0.f;
      uint32_t sal = 0;
      if (lane < nr) {
        dal = I.A_diag[r0 + lane] + I.c0;
        sal = I.A_str[r0 + lane];
      }
#pragma unroll 1
      for (int c = half; c < BN / 32; c += 2) {
        float v[32], u[32];
        const unsigned ta = tmem + ((unsigned)(quarter * 32) << 16) + (unsigned)(C::kAcc * buf * BN + c * 32);
        tc::tmem_ld32(ta + BN, v);
        if (C::kAcc == 3) {
          tc::tmem_ld32(ta + 2 * BN, u);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] += u[j];
        }
        tc::tmem_ld32(ta, u);
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] += u[j];
        // 8 columns at a time through shared memory: lane = (row 4 i + lane /
        // 8, column lane % 8), so x and y move in whole 32-byte sectors
        const int lr = lane >> 3, lc = lane & 7;
#pragma unroll
        for (int s8 = 0; s8 < 4; ++s8) {
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 8; ++j) tr[lane * 9 + j] = v[8 * s8 + j];
          const int col = n0 + c * 32 + 8 * s8 + lc;
          const bool cv = col < dB;
          const uint32_t sb = cv ? Bs[col] : 0u;
          const float bd = cv ? Bd[col] : 0.f;
          const float* __restrict__ xc = x + (long long)r0 * dB + col;
          float* __restrict__ yc = y + (long long)r0 * dB + col;
          // the 32 rows' x loads in flight before any is used (x is read from
          // DRAM here: one load at a time per warp would leave the epilogue
          // bound by memory latency)
          float xv[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = 4 * i + lr;
            xv[i] = (r < nr && cv) ? xc[(long long)r * dB] : 0.f;
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = 4 * i + lr;
            const uint32_t sa = __shfl_sync(0xffffffffu, sal, r);
            const float da = __shfl_sync(0xffffffffu, dal, r);
            if (r < nr && cv) {
              const uint32_t z = vand ? (sa & sb) : (sa ^ sb);
              float dg = da + bd;
#pragma unroll
              for (int q = 0; q < kMaxClasses; ++q)  // unrolled: w, mk stay in registers
                if (q < ncls) dg += w[q] * (float)__popc(z & mk[q]);
              yc[(long long)r * dB] = fmaf(dg, xv[i], tr[r * 9 + lc]);
            }
          }
        }
        __syncwarp();
      }
      tc::tc_fence_before();
      tc::mbar_arrive(&acc_empty[buf]);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, C::kTmemCols);
  }
}

ed_status bdense_prepare() {
  ED_CUDA_TRY(cudaFuncSetAttribute(k_bgemm<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BdCfg<64>::kSmem));
  ED_CUDA_TRY(cudaFuncSetAttribute(k_bgemm<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BdCfg<128>::kSmem));
  return ED_OK;
}

ed_status bdense_apply(const BDenseArgs& a, cudaStream_t st) {
  k_bslice<<<a.sms * 8, 256, 0, st>>>(a);
  ED_CUDA_TRY(launch_pdl(k_bgemm<64>, a.sms, kBdThreads, BdCfg<64>::kSmem, st, a, 2));
  ED_CUDA_TRY(launch_pdl(k_bgemm<128>, a.sms, kBdThreads, BdCfg<128>::kSmem, st, a, 3));
  ED_CUDA_TRY(cudaGetLastError());
  return ED_OK;
}

}  // namespace edk
