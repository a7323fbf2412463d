// FP64-accurate contractions on the tensor cores: operands as digit planes, results as
// fixed-point integers (epw_fx.cu; the error-free splitting of Ozaki, Ogita, Oishi and Rump,
// Numer. Algorithms 59, 95 (2012), with integer digits).
#pragma once
#include <cuda_bf16.h>

#include "epw_internal.cuh"

constexpr int FX_S = 7;         // digit planes, 8 bits each: x = 2^e sum_i d_i 2^(-7-8(i-1)), |d_i| <= 128
constexpr int FX_NT = 64;       // columns (rows of B) of a tile
constexpr int FX_EMIN = -900;   // smallest row exponent (keeps 2^(e - F) normal)
constexpr int FX_BAD = 0x4000;  // row exponent of a row that holds an infinity or a NaN

// An operand [rows][kpad] (K contiguous) as FX_S planes of bf16 integers, one exponent per row.
struct FxOp {
  __nv_bfloat16 *d;  // [FX_S][rows][kpad]
  short *e;          // [rows], or null: all 0 (phases)
  int rows, kpad;
};
inline int fx_kpad(int nR) { return (2 * nR + 31) / 32 * 32; }
FxOp fx_plan(Arena &A, size_t rows, int kpad, bool exps);

// Phases e^{2 pi i x.R} (conjugated with conj), K index 2r + (re, im), of npt points.
void fx_phases(int npt, const double *x, int nR, const int *R, int rmax, const FxOp &o, cudaStream_t st);
// Columns of a complex array src[nk][nR][ld], the first ncol of each row, as rows
// 2 (k ncol + c) + s, s = re/im: K index 2r + t holds (Re, -Im) for s = 0 and (Im, Re) for s = 1.
void fx_columns(int nk, int nR, int ncol, size_t ld, const cx<double> *src, const FxOp &o, int *bad, cudaStream_t st);
// Rows of a complex array src[nrow][ld], K of them per row: row m holds (Re, Im) at K index 2j + t.
void fx_rows(size_t nrow, int K, size_t ld, const cx<double> *src, const FxOp &o, cudaStream_t st);
// Conjugate phases over points, rows 2r + s: K index 2p + t holds (cos, sin) for s = 0 and
// (-sin, cos) for s = 1, so that a row (Re, Im) of fx_rows gives sum_p conj(P_p(R_r)) x_p.
void fx_phases_conj(int npt, const double *x, int nR, const int *R, const FxOp &o, cudaStream_t st);
// The Hermitian part of sum_r P(r) X_r, P given as phases p[nk][nR] times X[nR][n][n] (p null:
// X alone, nk = 1): n^2 rows per k, h(i,i) the diagonal's real part, h(i,j) and h(j,i), i < j, the
// real and imaginary part of element (i, j).
void fx_hermitian(int nk, int nR, int n, const cx<double> *p, const cx<double> *X, const FxOp &o, int *bad,
                  cudaStream_t st);
__host__ __device__ __forceinline__ int fx_hrow(int n, int i, int j) { return i * n + j; }

// Bits of the fixed point for sums over nR complex terms: |sum| <= sqrt(2) nR 2^e, value = I 2^(e - F).
inline int fx_bits(int nR) {
  int l = 0;
  while ((1 << l) < 1.5 * nR + 1) l++;
  return 62 - l < 54 ? 62 - l : 54;
}

// I[col][ldc] (64-bit integers, col a row of B, ldc >= the rows of A padded to 128)
epw_status fx_gemm_i64(const FxOp &A, const FxOp &B, int F, long long *C, size_t ldc, unsigned *dstatus,
                       cudaStream_t st);
// out[row][ldo] FP64, row a row of A, columns the rows of B (acc: added to what is there).  With
// ostride > 0 the K range goes in fx_splits parts to out + part * ostride.
epw_status fx_gemm_f64(const FxOp &A, const FxOp &B, int F, double *out, size_t ldo, unsigned *dstatus,
                       cudaStream_t st, bool acc = false, size_t ostride = 0);
// Parts of a long K: at most FX_KMAX elements each (their sum's fixed point keeps F near 50 bits).
constexpr int FX_KMAX = 4096;
inline int fx_kb_split(int kpad) {  // 32-element K blocks per part
  const int kb = kpad / 32, s = (kb + FX_KMAX / 32 - 1) / (FX_KMAX / 32);
  return (kb + s - 1) / s;
}
inline int fx_splits(int kpad) { return (kpad / 32 + fx_kb_split(kpad) - 1) / fx_kb_split(kpad); }
// scale[i] = 2^(e[i] - F), NaN for rows that are not finite
void fx_scales(size_t n, const short *e, int F, double *scale, cudaStream_t st);

// Unpacks the Hermitian matrices of fx_hermitian's rows: out[i][n][n] complex from in[i][n^2].
void fx_unpack_hermitian(int npt, int n, const double *in, cx<double> *out, cudaStream_t st);
