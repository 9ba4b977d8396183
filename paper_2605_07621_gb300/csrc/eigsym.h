// Eigenvalues of dense symmetric FP64 matrices: Householder tridiagonal
// reduction (eigsym.cu), then the tridiagonal matrix's by counting (sturm.cu).
#pragma once

#include <vector>

#include "ed_internal.h"
#include "ozaki.h"

namespace edk {
// Blocked reduction: panels of kTriNb reflectors, each followed by the
// trailing update A -= V W^T + W V^T as one FP64-accurate tensor-core product
constexpr int kTriNb = 64;
struct TriPanel {
  int k0, jb, t0;  // first column, reflectors, first row of the trailing matrix
};
std::vector<TriPanel> tridiag_panels(int m);
// the panel buffers (device [m][2 kTriNb] FP64 each, and WVf), the float-float copy
// of the matrix (device [m][ldF] float2, ldF = tridiag_ldF(m); every value
// finite, since the reduction also reads entries outside the trailing
// triangle, multiplied by zero), a 2-D tensor map over it (m x m 8-byte
// elements, row stride ldF, box 34 x 32), the flag that bounded waits set,
// and, per panel, two slicing jobs and one product (built by
// tridiag_blocked_setup, on device)
inline long long tridiag_ldF(int m) { return m + (m & 1); }
// fewest CTAs with which an m x m reduction takes one launch for every panel of
// up to kPtMax rows (eigsym.cu)
int tridiag_panel_ctas(int m);
constexpr int kPanelLate = 4;  // TriBlocked::err: a wait of the panel kernel ran out
// entangle.cu
void entangle_shares(const long long* m, int nb, int lanes, int sms, int* lane_of, int* share);
struct TriBlocked {
  OzContext* oz;
  double* NVW;
  double* WV;
  float2* WVf;  // the panel's W and sigma V as float-float pairs (device [m][2 kTriNb])
  float2* F;
  long long ldF;
  CUtensorMap tmF;
  int* err;
  const OzSliceJob* d_jobs;
  const OzProblem* d_probs;
  int ctas;  // most CTAs of the panel kernel (they wait for one another: all must be resident); 0: none
};
// appends the jobs and products of an m x m reduction of A (tensor maps in oz;
// opA / opB: digit-plane buffers for m x 2 kTriNb operands)
ed_status tridiag_blocked_setup(OzContext* oz, double* A, int m, const OzOperand& opA, const OzOperand& opB,
                                const double* NVW, const double* WV, std::vector<OzSliceJob>& jobs,
                                std::vector<OzProblem>& probs);
inline long long tridiag_blocked_work_doubles(int m) {
  return 7LL * m + 2LL * ((m + 63) / 64) * m + 128LL * (2 * kTriNb + 1) + 2 * kTriNb + 4096 + 1024 + 8 +
         4LL * kTriNb + 2 + (2 * kTriNb + 1) + 160 + 160LL * (2 * kTriNb + 4) + 4;
}
// Reduce the symmetric m x m row-major A (device; only its lower triangle,
// diagonal included, is read and overwritten) to tridiagonal form; the
// diagonal (m) and off-diagonal (m - 1) entries go to the device arrays d_out
// and e_out.
// work: device scratch of tridiag_blocked_work_doubles(m) doubles.
ed_status tridiag_reduce_blocked(double* A, int m, double* work, double* d_out, double* e_out, cudaStream_t st,
                                 int sms, const TriBlocked& tb);
// all eigenvalues of a batch of tridiagonal matrices on the device (sturm.cu):
// block b's diagonal (n) and off-diagonal (n - 1) from de + 2 off, its
// eigenvalues into lam + off, in descending order within each unreduced part of
// the matrix; nrm[b] receives the matrix's norm, NaN where an entry is not
// finite (lam is then undefined)
struct SturmBlk {
  int n;
  long long off;
  int w0, w1;  // first warp of each stage (sturm_plan)
};
struct SturmRow {
  int first, end, ex;  // the unreduced part of a row: rows first .. end - 1, norm in [2^(ex-1), 2^ex)
};
struct SturmBatch {
  const SturmBlk* d_blk;  // device, nb entries, n >= 1
  size_t nb;
  int S0, S1, warps0, warps1;  // lanes per eigenvalue and warps of each stage (sturm_plan)
  const double* de;            // device [2 sum n]
  double* lam;                 // device [sum n]
  double* nrm;                 // device [nb]
  float4* tf;                  // device scratch [sum n] each
  double2 *td, *br;
  SturmRow* row;
};
void sturm_plan(std::vector<SturmBlk>& blk, int sms, SturmBatch* B);
ed_status sturm_eigenvalues(const SturmBatch& B, cudaStream_t st);
// all eigenvalues of the tridiagonal (d, e) on the host into d (unordered);
// false if the iteration did not converge
bool tridiag_eigenvalues(std::vector<double>& d, std::vector<double>& e);
}  // namespace edk
