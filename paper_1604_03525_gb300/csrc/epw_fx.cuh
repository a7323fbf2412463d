// FP64-accurate contractions on the tensor cores: operands as digit planes, results as
// fixed-point integers (epw_fx.cu; the error-free splitting of Ozaki, Ogita, Oishi and Rump,
// Numer. Algorithms 59, 95 (2012), with integer digits).
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

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

// The digits of X (|X| <= 2^55), most significant first, as bf16 pairs (x in the low half).
// Balanced base 256: adding 128 to each of the six lower bytes makes them unsigned, the rest is d_1.
__device__ __forceinline__ void fx_digits2(long long X, long long Y, uint32_t (&p)[FX_S]) {
  const long long bias = 0x0000808080808080LL;
  const long long xb = X + bias, yb = Y + bias;
  const uint32_t x0 = (uint32_t)xb, x1 = (uint32_t)(xb >> 32), y0 = (uint32_t)yb, y1 = (uint32_t)(yb >> 32);
  auto pack = [](float a, float b) { return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632); };
  p[0] = pack((float)((int)x1 >> 16), (float)((int)y1 >> 16));
#pragma unroll
  for (int i = 1; i < FX_S; i++) {
    const int b = FX_S - 1 - i;  // byte
    const uint32_t xs = b >= 4 ? x1 : x0, ys = b >= 4 ? y1 : y0;
    const uint32_t fx = __byte_perm(xs, 0x4B000000u, 0x7440 | (b & 3)), fy = __byte_perm(ys, 0x4B000000u, 0x7440 | (b & 3));
    p[i] = pack(__uint_as_float(fx) - 8388736.0f, __uint_as_float(fy) - 8388736.0f);  // byte - 128
  }
}
// |c|, |s| exceed 1 by rounding at most, which the leading digit has room for
__device__ __forceinline__ void fx_phase_digits(double c, double s, uint32_t (&p)[FX_S]) {
  fx_digits2(__double2ll_rn(c * 36028797018963968.0), __double2ll_rn(s * 36028797018963968.0), p);  // 2^55
}

constexpr int FX_PPB = 16;    // points per block
struct FxFactors {
  double2 f[FX_PPB][3][2 * PH_RMAX + 1];
};
// Phases e^{2 pi i x.R} of a block's FX_PPB points: the one-axis factors e^{2 pi i (x_j n mod 1)},
// n = 1..rmax (n < 0: the conjugate), one per thread, then a warp per point, lanes over R (contiguous
// K on the way out) up to `half` (0 beyond nR).  rmax > PH_RMAX: the phase of each R by itself.
// row(point, finite) once per point, put(point, r, cos, sin) for every r.  Blocks of 128 threads.
template <class ROW, class PUT>
__device__ __forceinline__ void fx_point_phases(int npt, const double *__restrict__ x, int nR,
                                                const int *__restrict__ R, int rmax, int half, FxFactors &F, ROW row,
                                                PUT put) {
  const int p0 = blockIdx.x * FX_PPB, np = min(FX_PPB, npt - p0);
  const bool fact = rmax <= PH_RMAX;
  if (fact) {
    const int per = 3 * (rmax + 1);
    for (int t = threadIdx.x; t < np * per; t += 128) {
      const int p = t / per, j = (t - p * per) / (rmax + 1), n = t % (rmax + 1);
      double a = x[3 * (size_t)(p0 + p) + j] * n;
      a -= rint(a);
      double s, c;
      sincospi(2.0 * a, &s, &c);
      F.f[p][j][PH_RMAX + n] = make_double2(c, s);
      F.f[p][j][PH_RMAX - n] = make_double2(c, -s);
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int p = warp; p < np; p += 4) {
    const size_t pt = (size_t)(p0 + p);
    const double q0 = x[3 * pt], q1 = x[3 * pt + 1], q2 = x[3 * pt + 2];
    const bool fin = isfinite(q0) && isfinite(q1) && isfinite(q2);
    if (lane == 0) row(pt, fin);
    for (int r = lane; r < half; r += 32) {
      double c = 0.0, s = 0.0;
      if (r < nR && fin) {
        if (fact) {
          const double2 f0 = F.f[p][0][R[3 * r] + PH_RMAX], f1 = F.f[p][1][R[3 * r + 1] + PH_RMAX],
                        f2 = F.f[p][2][R[3 * r + 2] + PH_RMAX];
          const cx<double> f = phase_product(mkc(f0.x, f0.y), mkc(f1.x, f1.y), mkc(f2.x, f2.y));
          c = f.x;
          s = f.y;
        } else {
          double a = q0 * R[3 * r] + q1 * R[3 * r + 1] + q2 * R[3 * r + 2];
          a -= rint(a);
          sincospi(2.0 * a, &s, &c);
        }
      }
      put(pt, r, c, s);
    }
  }
}

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
// Unpacks the Hermitian matrices of fx_hermitian's rows: out[i][n][n] complex from in[i][n^2].
void fx_unpack_hermitian(int npt, int n, const double *in, cx<double> *out, cudaStream_t st);
