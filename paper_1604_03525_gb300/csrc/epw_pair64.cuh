// Per-pair FP64 work on fixed-point contractions (epw_pair64.cu).
#pragma once
#include "epw_fx.cuh"

struct Pair64Args {
  int nq, nw, nm;
  int k0, nk;                  // k-points [k0, k0 + nk) of the call, the chunk that CH, CG hold
  const long long *CH, *CG;    // [nk nw^2][ldc] H(k+q) (fx_hermitian's rows), [nk 2 nm nw^2][ldc] g_a(k,q) U_k
  const short *eH, *eG;        // their exponents (value = I 2^(e - F))
  int FH, FG;
  size_t ldc;
  const double2 *ET;           // mode factors [nm nm][nq]
  const double *omK, *nbT;     // frequencies (-1 for modes that are left out) and Bose factors [nm][nq]
  const double *wmax;          // [nq] largest frequency of the kept modes (-1: none)
  const double *eps_k;         // [nk of the call][nw]
  const double *wq;            // [nq] or null (1/nq)
  double T, EF, sigma;
  double inv_kT, inv_sigma, gnorm, inv_nq;  // 1/kT (T > 0), 1/sigma, 1/(sigma sqrt pi), 1/nq
  double *partial;             // [nk of the call][ceil(nq/128)][nw]
  unsigned *dstatus;
  const double *exptab;        // 2^(-j/EPW_EXPTAB)
  const int *bad;              // nonzero: some operand held an infinity or a NaN
  const double2 *Cpol;         // long-range factors [nm][nq] or null
  const cx<double> *Uk;        // [nk of the call][nw][nw]
  // adjoint: cotangent [nk of the call][nw], Xbar [nk nm nw^2][nq] (zeroed by the caller), sums [nk][ceil(nq/128)]
  const double *cot;
  double2 *xbar;
  double *partialT, *partialE;
  // phonon side: weights of the call's k-points (null: 1/nk_total), k per block, sums
  // [chunk][nq][2 nm + 1] (the layout of k_ph_finalize)
  const double *wk;
  int nk_total, nkc;
  // interpolation: eigenvalues and eigenvectors of H(k+q) [nq][nk][nw], [nq][nk][nw][nw]
  const double *wkq;
  const cx<double> *Ukq;
  double *eps_kq;              // [nk of the call][nq][nw] or null
  cx<double> *gout;            // [nk of the call][nq][nm][nw][nw] or null
};

// Im Sigma_nk terms of the chunk's pairs, summed over blocks of 128 q.
epw_status launch_lw64(const Pair64Args &a, cudaStream_t st);
// Adjoint of the linewidth per pair: Xbar and the sums for dL/dT, dL/dE_F.
epw_status launch_adj64(const Pair64Args &a, cudaStream_t st);
// Sums over the chunk's k per (q, nu): Pi'', lambda and nesting terms (nw <= 8, 3nat <= 9), a.nkc k per warp.
epw_status launch_ph64(const Pair64Args &a, int nchunk, cudaStream_t st);
// e_k+q and g_mn,nu from given eigenvectors.
epw_status launch_g64(const Pair64Args &a, cudaStream_t st);
// The adjoint's k side: B[split][nk nm nw^2][2 nRp] (sum over q of conj(P_q(Rp)) Xbar, in parts) is
// rotated by U_k^dagger into G1[nRp nm nw^2][nk].
void launch_adj_rotate64(int nk, int k0, int nRp, int nm, int nw, int splits, size_t stride, const double *B,
                         const cx<double> *Uk, cx<double> *G1, cudaStream_t st);
// dg[Re][c] = wRe wRp gT[c][Re]
void launch_dg64(const epw_model *m, const cx<double> *gT, double *dg, cudaStream_t st);
// omK, nbT [nm][nq] and wmax [nq] from the frequencies omegaT [nm][nq]
void launch_tables64(int nq, int nm, const double *omegaT, double omega_min, double T, double *omK, double *nbT,
                     double *wmax, cudaStream_t st);
