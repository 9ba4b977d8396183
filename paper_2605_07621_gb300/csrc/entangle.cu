// Entanglement spectrum across the cut: the spectrum xi = -log(lambda) of
// the entanglement Hamiltonian H_E = -log(rho_A), rho_A = Tr_B |psi><psi|,
// resolved by the conserved charge of side A (the paper's discussion of
// its figure "Distributed entanglement spectrum", with the sector weights W_q).
//
// In the block layout rho_A is block diagonal, rho_A(s) = Psi_s Psi_s^T, and
// its nonzero eigenvalues are those of the Gram matrix of Psi_s in the
// smaller of its two dimensions (the squared singular values of Psi_s).
// The Gram matrix is formed on the tensor cores by the FP64-accurate
// digit-split GEMM (ozaki.cu; one digit-plane buffer serves as both
// factors, only the tiles on or below the diagonal), reduced to tridiagonal
// form on the GPU by Householder reflections (eigsym.cu), the blocks
// concurrently on a few streams; then the eigenvalues of all blocks'
// tridiagonal matrices by counting, in one batch (sturm.cu).
#include <cmath>
#include <algorithm>
#include <string>
#include <thread>

#include "krylov.h"
#include "eigsym.h"
#include "ozaki.h"

namespace edk {
namespace {

struct DevMem {
  std::vector<void*> p;
  ~DevMem() {
    for (void* q : p) cudaFree(q);
  }
  ed_status get(void** out, size_t bytes) {
    cudaError_t e = cudaMalloc(out, bytes < 16 ? 16 : bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      set_error("cudaMalloc(%zu) for the entanglement spectrum failed: %s", bytes, cudaGetErrorString(e));
      return ED_ENOMEM;
    }
    p.push_back(*out);
    return ED_OK;
  }
};

}  // namespace

// The lane of each of nb blocks (of m[i] rows) and the share of the SMs of each
// lane: the blocks, largest first, to the lane with the least work so far, and
// the SMs so that the lanes end together.  A reduction on g SMs takes about
// serial(m) + spread(m) / g microseconds (m = 1716 / 3003 / 3432 alone on 25 to
// 152 SMs: within 5 %).  No lane gets fewer SMs than the panels of up to
// kShareRows rows of its blocks need to run as one launch each
// (tridiag_panel_ctas): by their work alone the lanes of a few hundred to two
// thousand rows beside larger ones got so few that their panels went back to
// three kernels per column.  28 sites with 11 / 9 up spins (m up to 2,002 / 1,001):
// 42.0 -> 33.0 / 17.2 -> 15.1 ms, 30 sites with 12 (5,005): 204 -> 183.  Larger
// panels on few SMs are better off with those kernels, which use the whole GPU:
// with the line at 4,096 rows, or for all, 32 sites with 12 up spins (8,008) 514
// -> 573 / 591, 30 with 15 623 -> 632 / 690, 32 with 16 3,174 -> 3,232 / 3,459; at
// 2,048: 520, 620, 3,178.  On a GPU with fewer SMs than the needs add up to, a
// lane's launches wait for another's.
constexpr long long kShareRows = 2048;
void entangle_shares(const long long* m, int nb, int lanes, int sms, int* lane_of, int* share) {
  std::vector<int> order(nb), need(lanes, 0);
  for (int i = 0; i < nb; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int u, int v) { return m[u] > m[v]; });
  auto serial = [](double x) { return x * (9.0 + 0.6e-3 * x); };
  auto spread = [](double x) { return 1.45e6 * std::pow(x / 3432.0, 2.5); };
  std::vector<double> lane_serial(lanes, 0.0), lane_spread(lanes, 0.0), load(lanes, 0.0);
  for (int i : order) {
    const double x = (double)m[i];
    const int k = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    lane_of[i] = k;
    load[k] += serial(x) + spread(x) * lanes / sms;
    lane_serial[k] += serial(x);
    lane_spread[k] += spread(x);
    need[k] = std::max(need[k], std::min(sms, tridiag_panel_ctas((int)std::min(m[i], kShareRows))));
  }
  // the lanes end together, at T: bisection for the least T at which the shares fit
  double lo = *std::max_element(lane_serial.begin(), lane_serial.end()), hi = lo + 1.0;
  auto shares = [&](double T) {
    int sum = 0;
    for (int k = 0; k < lanes; ++k) {
      share[k] = (int)std::min((double)sms, std::max((double)need[k], std::floor(lane_spread[k] / (T - lane_serial[k]))));
      sum += share[k];
    }
    return sum;
  };
  for (int i = 0; i < 60 && shares(hi) > sms; ++i) hi = lo + 2.0 * (hi - lo);
  for (int i = 0; i < 40; ++i) {
    const double mid = 0.5 * (lo + hi);
    if (shares(mid) > sms) lo = mid; else hi = mid;
  }
  shares(hi);
}

}  // namespace edk

using namespace edk;

// panels: the reductions may take one cooperative launch per panel.  late: a wait
// of those launches ran out (the status is then not ED_OK).
static ed_status spectrum(ed_ctx* c, const double* psi, double* lambda, int64_t cap, int64_t* n_lambda, double* weight,
                          double* entropy, double* stage_ms, void* stream, bool panels, bool* late) {
  if (!c || !n_lambda) {
    set_error("ctx or n_lambda is NULL");
    return ED_EINVAL;
  }
  int64_t need = 0, mmax = 0;
  for (const Block& b : c->blocks) {
    const int64_t m = std::min(b.dA, b.dB);
    need += m;
    mmax = std::max(mmax, m);
  }
  *n_lambda = need;
  if (!lambda) return ED_OK;  // size query
  if (!psi) {
    set_error("psi is NULL");
    return ED_EINVAL;
  }
  if (cap < need) {
    set_error("lambda holds %lld values, %lld needed", (long long)cap, (long long)need);
    return ED_EINVAL;
  }
  if (mmax > 46340) {  // m * m must fit 32-bit index arithmetic of the reduction
    set_error("block Gram dimension %lld exceeds the dense eigensolver's limit", (long long)mmax);
    return ED_EUNSUPPORTED;
  }
  ED_DEVICE_SCOPE(c->device);
  ED_TRY(ensure_scratch(c));
  cudaStream_t st = (cudaStream_t)stream;
  const size_t nb = c->blocks.size();
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
    cudaGetLastError();
    sms = 148;
  }

  // The blocks are reduced concurrently on up to kLanes streams ("lanes"): a
  // column is mostly latency and leaves most of the GPU idle.  They go, largest
  // first, to the lane with the least work so far; each lane has its own
  // buffers, sized for its largest block, and a share of the SMs for its panel
  // kernels (one CTA per SM).  Spectrum of 15 blocks with m up to 3432 / of 13
  // with m up to 924, in equal shares: 2 lanes 146 / 27 ms, 3: 130 / 19.6, 4:
  // 134 / 16.7, 6: 154 / 15.9; shared out by their work: 3: 127 / 19.5, 4: 122 /
  // 17.1, 5: 114 / 16.2, 6: 134 / 20.5; with a fifth of the SMs left to the
  // trailing updates, 5: 122 / 17.1.
  constexpr int kLanes = 5;
  std::vector<size_t> order(nb);
  for (size_t i = 0; i < nb; ++i) order[i] = i;
  auto bm = [&](size_t i) { return (long long)std::min(c->blocks[i].dA, c->blocks[i].dB); };
  auto bl = [&](size_t i) { return (long long)std::max(c->blocks[i].dA, c->blocks[i].dB); };
  std::stable_sort(order.begin(), order.end(), [&](size_t u, size_t v) { return bm(u) > bm(v); });
  // device bytes of a lane sized for blocks up to (m, m x Lpad elements)
  auto lane_bytes = [&](long long m, long long xel) {
    const long long ldF = tridiag_ldF((int)m);
    return (double)m * m * 8 + (double)m * ldF * 8 + 3.0 * m * 2 * kTriNb * 8 +
           8.0 * tridiag_blocked_work_doubles((int)m) +
           2.0 * kOzDigits * xel + 2.0 * 2 * kOzDigits * m * 2 * kTriNb + 4.0 * m;
  };
  int lanes = kLanes;
  {
    size_t fr = 0, tot_mem = 0;
    if (cudaMemGetInfo(&fr, &tot_mem) != cudaSuccess) {
      cudaGetLastError();
      fr = 0;
    }
    long long m0 = nb ? bm(order[0]) : 1, x0 = 1;
    for (size_t i = 0; i < nb; ++i) x0 = std::max(x0, bm(i) * ((bl(i) + 7) / 8 * 8));
    const double one = lane_bytes(m0, x0);
    while (lanes > 1 && one * lanes > 0.8 * (double)fr) --lanes;
  }
  std::vector<long long> mb(nb);
  for (size_t bi = 0; bi < nb; ++bi) mb[bi] = bm(bi);
  std::vector<int> lane_of(nb, 0), share(lanes, 1);
  entangle_shares(mb.data(), (int)nb, lanes, sms, lane_of.data(), share.data());
  std::vector<std::vector<size_t>> lane_blocks(lanes);
  for (size_t bi : order) lane_blocks[lane_of[bi]].push_back(bi);
  while (lanes > 1 && lane_blocks[lanes - 1].empty()) --lanes;

  DevMem mem;
  OzContext oz;
  oz.device = c->device;
  struct Lane {
    long long mmax = 1, xel = 1;
    double *G = nullptr, *work = nullptr, *NVW = nullptr, *WV = nullptr;
    float2 *F = nullptr, *WVf = nullptr;
    OzOperand X, opA, opB;
    cudaStream_t s = nullptr;
  };
  std::vector<Lane> L(lanes);
  for (int k = 0; k < lanes; ++k) {
    for (size_t bi : lane_blocks[k]) {
      L[k].mmax = std::max(L[k].mmax, bm(bi));
      L[k].xel = std::max(L[k].xel, bm(bi) * ((bl(bi) + 7) / 8 * 8));
    }
    const long long mk = L[k].mmax;
    ED_TRY(mem.get((void**)&L[k].G, (size_t)mk * mk * sizeof(double)));
    ED_TRY(mem.get((void**)&L[k].work, (size_t)tridiag_blocked_work_doubles((int)mk) * sizeof(double)));
    ED_TRY(mem.get((void**)&L[k].F, (size_t)mk * tridiag_ldF((int)mk) * sizeof(float2)));
    ED_TRY(mem.get((void**)&L[k].WVf, (size_t)mk * 2 * kTriNb * sizeof(float2)));
    ED_TRY(oz_alloc(&oz, (void**)&L[k].NVW, (size_t)mk * 2 * kTriNb * sizeof(double)));
    ED_TRY(oz_alloc(&oz, (void**)&L[k].WV, (size_t)mk * 2 * kTriNb * sizeof(double)));
    ED_TRY(oz_operand_buffer(&oz, L[k].xel, mk, &L[k].X));
    ED_TRY(oz_operand_buffer(&oz, mk * 2 * kTriNb, mk, &L[k].opA));
    ED_TRY(oz_operand_buffer(&oz, mk * 2 * kTriNb, mk, &L[k].opB));
  }

  // per block: its Gram matrix (digit planes of Psi_s as both factors, the
  // tiles on or below the diagonal) and the trailing updates of its
  // reduction, in its lane's buffers; tensor maps and launch lists up front
  std::vector<OzSliceJob> jobs(nb);
  std::vector<OzProblem> probs(nb);
  std::vector<long long> units(nb), tiles(nb);
  std::vector<OzSliceJob> tjobs;
  std::vector<OzProblem> tprobs;
  std::vector<size_t> toff(nb);
  for (size_t bi = 0; bi < nb; ++bi) {
    const Block& b = c->blocks[bi];
    Lane& ln = L[lane_of[bi]];
    const int m = (int)bm(bi), Lg = (int)bl(bi);
    int ma = 0, mb = 0;
    ED_TRY(oz_map(&oz, &ln.X, m, Lg, true, &ma));
    ED_TRY(oz_map(&oz, &ln.X, m, Lg, false, &mb));
    OzSliceJob j{};
    j.src = psi + b.off;
    j.sbase = 0;
    j.ld = b.dB;
    j.rows = (int)b.dA;
    j.cols = (int)b.dB;
    j.dst = ln.X.slices;
    j.exps = ln.X.exps;
    j.Kpad = (Lg + 7) / 8 * 8;
    j.first = 0;
    jobs[bi] = j;
    // Psi Psi^T (rows, dA <= dB) or Psi^T Psi (columns)
    units[bi] = b.dA <= b.dB ? (long long)b.dA : (b.dB + 31) / 32;
    OzProblem p{};
    p.mapA = ma;
    p.mapB = mb;
    p.ea = ln.X.exps;
    p.eb = ln.X.exps;
    p.C = ln.G;
    p.cbase = 0;
    p.ldc = m;
    p.M = p.N = m;
    p.K = Lg;
    p.acc = 0;
    p.tiles_n = (m + kOzBN - 1) / kOzBN;
    p.tri = 1;  // the lower triangle: all the reduction reads
    p.tile0 = 0;
    probs[bi] = p;
    tiles[bi] = oz_tiles(m, m, 1);
    toff[bi] = tprobs.size();
    ED_TRY(tridiag_blocked_setup(&oz, ln.G, m, ln.opA, ln.opB, ln.NVW, ln.WV, tjobs, tprobs));
  }
  ED_TRY(oz_finish(&oz));
  OzSliceJob *d_tjobs = nullptr, *d_jobs = nullptr;
  OzProblem *d_tprobs = nullptr, *d_probs = nullptr;
  if (!tprobs.empty()) {
    ED_TRY(oz_alloc(&oz, (void**)&d_tjobs, tjobs.size() * sizeof(OzSliceJob)));
    ED_TRY(oz_alloc(&oz, (void**)&d_tprobs, tprobs.size() * sizeof(OzProblem)));
    ED_CUDA_TRY(cudaMemcpy(d_tjobs, tjobs.data(), tjobs.size() * sizeof(OzSliceJob), cudaMemcpyHostToDevice));
    ED_CUDA_TRY(cudaMemcpy(d_tprobs, tprobs.data(), tprobs.size() * sizeof(OzProblem), cudaMemcpyHostToDevice));
  }
  ED_TRY(oz_alloc(&oz, (void**)&d_jobs, nb * sizeof(OzSliceJob)));
  ED_TRY(oz_alloc(&oz, (void**)&d_probs, nb * sizeof(OzProblem)));
  ED_CUDA_TRY(cudaMemcpy(d_jobs, jobs.data(), nb * sizeof(OzSliceJob), cudaMemcpyHostToDevice));
  ED_CUDA_TRY(cudaMemcpy(d_probs, probs.data(), nb * sizeof(OzProblem), cudaMemcpyHostToDevice));

  // the batch of tridiagonal matrices, largest first (the empty blocks have none)
  std::vector<size_t> boff(nb + 1, 0);
  for (size_t bi = 0; bi < nb; ++bi) boff[bi + 1] = boff[bi] + (size_t)bm(bi);
  std::vector<SturmBlk> sblk;
  for (size_t bi : order)
    if (bm(bi) > 0) sblk.push_back(SturmBlk{(int)bm(bi), (long long)boff[bi], 0, 0});
  SturmBatch sb{};
  sturm_plan(sblk, sms, &sb);
  double* d_de = nullptr;
  SturmBlk* d_sblk = nullptr;
  {
    const size_t n1 = std::max<size_t>((size_t)need, 1), b1 = std::max<size_t>(sblk.size(), 1);
    ED_TRY(mem.get((void**)&d_de, 2 * n1 * sizeof(double)));
    ED_TRY(mem.get((void**)&sb.lam, (n1 + b1) * sizeof(double)));
    ED_TRY(mem.get((void**)&sb.tf, n1 * sizeof(float4)));
    ED_TRY(mem.get((void**)&sb.td, n1 * sizeof(double2)));
    ED_TRY(mem.get((void**)&sb.br, n1 * sizeof(double2)));
    ED_TRY(mem.get((void**)&sb.row, n1 * sizeof(SturmRow)));
    ED_TRY(mem.get((void**)&d_sblk, b1 * sizeof(SturmBlk)));
    sb.nrm = sb.lam + need;
    sb.de = d_de;
    sb.d_blk = d_sblk;
    if (!sblk.empty())
      ED_CUDA_TRY(cudaMemcpy(d_sblk, sblk.data(), sblk.size() * sizeof(SturmBlk), cudaMemcpyHostToDevice));
  }
  struct EventSet {
    std::vector<cudaEvent_t> e;
    ~EventSet() {
      for (cudaEvent_t x : e)
        if (x) cudaEventDestroy(x);
    }
    ed_status make(size_t n) {
      e.assign(n, nullptr);
      for (cudaEvent_t& x : e) ED_CUDA_TRY(cudaEventCreate(&x));
      return ED_OK;
    }
  } ev_g0, ev_g1, ev_lane, ev_se;
  ED_TRY(ev_g0.make(nb));
  ED_TRY(ev_g1.make(nb));
  ED_TRY(ev_lane.make(lanes));
  ED_TRY(ev_se.make(2));
  struct Streams {
    std::vector<cudaStream_t> s;
    ~Streams() {
      for (cudaStream_t x : s) cudaStreamDestroy(x);
    }
  } own;
  ED_CUDA_TRY(cudaEventRecord(ev_se.e[0], st));
  for (int k = 0; k < lanes; ++k) {
    cudaStream_t s = nullptr;
    ED_CUDA_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    own.s.push_back(s);
    L[k].s = s;
    ED_CUDA_TRY(cudaStreamWaitEvent(s, ev_se.e[0], 0));  // after the caller's work on its stream
  }
  // the reduction reads entries of F outside the trailing triangle (times
  // zero): every value must be finite
  for (int k = 0; k < lanes; ++k)
    ED_CUDA_TRY(cudaMemsetAsync(L[k].F, 0, (size_t)L[k].mmax * tridiag_ldF((int)L[k].mmax) * sizeof(float2), L[k].s));

  // per lane one host thread enqueues its blocks
  std::vector<std::thread> workers;
  struct Joiner {
    std::vector<std::thread>* t;
    int n;
    ~Joiner() {
      for (int i = 0; i < n; ++i)
        for (auto& x : t[i])
          if (x.joinable()) x.join();
    }
  };
  Joiner jw{&workers, 1};
  std::vector<ed_status> lst(lanes, ED_OK);
  std::vector<std::string> lmsg(lanes);
  auto lane_fn = [&](int k) {
    auto fail = [&](ed_status s) {
      lst[k] = s;
      lmsg[k] = ed_last_error();
    };
    DeviceGuard dg(c->device);
    if (dg.status() != ED_OK) return fail(ED_ECUDA);
    Lane& ln = L[k];
    for (size_t bi : lane_blocks[k]) {
      const Block& b = c->blocks[bi];
      const int m = (int)bm(bi);
      double* bd = d_de + 2 * boff[bi];
      ed_status s = ED_OK;
      if (cudaEventRecord(ev_g0.e[bi], ln.s) != cudaSuccess) return fail(ED_ECUDA);
      if ((s = oz_slice(&oz, d_jobs + bi, 1, units[bi], b.dA > b.dB, b.dA, nullptr, ln.s)) != ED_OK) return fail(s);
      if ((s = oz_gemm(&oz, d_probs + bi, 1, tiles[bi], nullptr, ln.s)) != ED_OK) return fail(s);
      if (cudaEventRecord(ev_g1.e[bi], ln.s) != cudaSuccess) return fail(ED_ECUDA);
      TriBlocked tb{&oz, ln.NVW, ln.WV, ln.WVf, ln.F, tridiag_ldF(m), {}, oz.d_err, d_tjobs + 2 * toff[bi],
                    d_tprobs + toff[bi], panels ? share[k] : 0};
      if (m >= 3 && (s = tmap_8b_2d(&tb.tmF, ln.F, m, m, tb.ldF, 34, 32)) != ED_OK) return fail(s);
      if ((s = tridiag_reduce_blocked(ln.G, m, ln.work, bd, bd + m, ln.s, sms, tb)) != ED_OK) return fail(s);
    }
    if (cudaEventRecord(ev_lane.e[k], ln.s) != cudaSuccess) return fail(ED_ECUDA);
  };
  for (int k = 0; k < lanes; ++k) {
    try {
      workers.emplace_back(lane_fn, k);
    } catch (...) {
      lane_fn(k);  // no thread to be had: enqueue this lane from here
    }
  }
  for (auto& x : workers) x.join();
  for (int k = 0; k < lanes; ++k)
    if (lst[k] != ED_OK) {
      for (int i = 0; i < lanes; ++i) cudaStreamSynchronize(L[i].s);  // nothing of this call left in flight
      set_error("%s", lmsg[k].c_str());
      return lst[k];
    }
  for (int k = 0; k < lanes; ++k) ED_CUDA_TRY(cudaStreamWaitEvent(st, ev_lane.e[k], 0));
  ED_TRY(sturm_eigenvalues(sb, st));
  ED_CUDA_TRY(cudaEventRecord(ev_se.e[1], st));
  std::vector<double> lam((size_t)need + std::max<size_t>(sblk.size(), 1));
  ED_CUDA_TRY(cudaMemcpyAsync(lam.data(), sb.lam, lam.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
  // ||Psi_s||^2 (the trace of rho_A(s)) with the library's FP64 reduction
  std::vector<double> wt(nb);
  for (size_t bi = 0; bi < nb; ++bi) {
    const Block& b = c->blocks[bi];
    ED_TRY(dot_dev<double>(c, psi + b.off, psi + b.off, b.dA * b.dB, slot(c, 3), st, 0));
    ED_TRY(read_scalars(c, 3, 1, &wt[bi], st));  // synchronises the stream
  }
  int code = 0;
  const ed_status waits = oz_status(&oz, st, &code);  // no bounded wait of the reduction's kernels ran out
  *late = code == kPanelLate;
  ED_TRY(waits);
  double t_gram = 0.0;
  float t_all = 0.f;
  for (size_t bi = 0; bi < nb; ++bi) {
    float t1 = 0.f;
    ED_CUDA_TRY(cudaEventElapsedTime(&t1, ev_g0.e[bi], ev_g1.e[bi]));
    t_gram += t1;
  }
  ED_CUDA_TRY(cudaEventElapsedTime(&t_all, ev_se.e[0], ev_se.e[1]));
  for (size_t i = 0; i < sblk.size(); ++i) {
    double* w = lam.data() + sblk[i].off;
    const size_t n = (size_t)sblk[i].n;
    if (!std::isfinite(lam[need + i])) {  // entries that are not finite: the host iteration's answer
      std::vector<double> dd(n), ee(n);
      ED_CUDA_TRY(cudaMemcpy(dd.data(), d_de + 2 * sblk[i].off, n * sizeof(double), cudaMemcpyDeviceToHost));
      ED_CUDA_TRY(cudaMemcpy(ee.data(), d_de + 2 * sblk[i].off + n, (n - 1) * sizeof(double), cudaMemcpyDeviceToHost));
      ee.resize(n - 1);
      if (!tridiag_eigenvalues(dd, ee)) {
        set_error("tridiagonal QL did not converge on a block of %zu levels", n);
        return ED_ENOCONV;
      }
      std::copy(dd.begin(), dd.end(), w);
    }
    // descending (the parts of a matrix follow one another, and neighbours within
    // the brackets' width may be swapped)
    if (!std::is_sorted(w, w + n, std::greater<double>())) std::sort(w, w + n, std::greater<double>());
  }
  std::copy(lam.begin(), lam.begin() + need, lambda);
  if (stage_ms) {
    // with the blocks on several streams the Gram products overlap other
    // blocks' reductions: [0] = the Gram products' own device time, [1] =
    // the rest of the call's device time
    stage_ms[0] = t_gram;
    stage_ms[1] = std::max(0.0, (double)t_all - t_gram);
  }
  double tot = 0.0;
  for (double v : wt) tot += v;
  if (weight)
    for (size_t bi = 0; bi < wt.size(); ++bi) weight[bi] = wt[bi];
  if (entropy) {
    // von Neumann entropy of the normalised spectrum; eigenvalues at or below
    // zero (rounding of a rank-deficient block) carry no weight
    double s = 0.0;
    if (tot > 0.0)
      for (int64_t i = 0; i < need; ++i) {
        const double p = lambda[i] / tot;
        if (p > 0.0) s -= p * std::log(p);
      }
    *entropy = s;
  }
  return ED_OK;
}

extern "C" ed_status ed_entanglement_spectrum(ed_ctx* c, const double* psi, double* lambda, int64_t cap,
                                              int64_t* n_lambda, double* weight, double* entropy, double* stage_ms,
                                              void* stream) {
  bool late = false;
  const ed_status s = spectrum(c, psi, lambda, cap, n_lambda, weight, entropy, stage_ms, stream, true, &late);
  // other work held SMs for seconds: once more, with kernels that do not wait
  return late ? spectrum(c, psi, lambda, cap, n_lambda, weight, entropy, stage_ms, stream, false, &late) : s;
}
