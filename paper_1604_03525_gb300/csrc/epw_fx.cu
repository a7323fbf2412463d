// FP64-accurate contractions on the tensor cores.
//
// The FP64 pipe of sm_103a issues one warp instruction per 64 cycles and sub-partition (1.26
// TFLOP/s measured), so an FP64 contraction costs 1500 times its BF16 one.  Here every operand
// is written as FX_S = 7 planes of 8-bit signed digits (bf16 holds them exactly), 56 bits below
// the largest element of its row, and the products d_i d'_j of the 28 plane pairs with i + j <= 8
// are summed by tcgen05 kind::f16 MMAs, one FP32 accumulator per level l = i + j - 1:
//   - a product is an integer of at most 2^14; an accumulator is emptied after at most 256
//     terms per pair, so level l holds at most l 2^22 and levels 1 to 4 are exact for any input;
//     levels 5 to 7 would have to exceed 2^24 to round: digits that all agree in sign and size.  Then the
//     last 16 of level 5's 80 accumulations round by a unit of 2^-46 of the row scales each at most, 2^-42
//     beside a sum of such digits of about 2^7, inside the a-priori bound of an FP64 sum; for digits
//     without such structure they are exact too (about 2^18);
//   - the levels are combined in 64-bit integers at 2^-F of the row scales (F about 53), so the
//     sum over K is exact and its order does not matter.
// What is dropped (levels from 8 on) is about 2^-52 of the product of the row maxima; the FP64
// FMA chain that this replaces rounds at 2^-53 of every partial sum, about 2^-49 in all for 250
// complex terms.
//
// Tile: 128 rows of A by 64 rows of B.  The 7 planes of B are neighbours in shared memory, so one
// MMA multiplies plane i of A with planes 1 .. 8-i of B (N up to 256) and its accumulators are
// the levels i, i+1, ... of 64 tensor-memory columns each: 10 MMAs per K = 16 step instead of 28,
// which keeps the shared-memory reads (96 KB per 896 cycles) below the 128 B/cycle limit.  448 of
// the 512 columns are used, so the accumulators are not doubled; the epilogue (8 warps) reads
// them into 64-bit registers and hands them back before it converts or stores anything.
// Measured: diamond nw = 8, 24 k x 8000 q 3.0 ms, 76 % of the BF16 peak in digit products; fcc nw = 4,
// 125 k x 13,824 q 2.5 ms, 61 %.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>

#include "epw_fx.cuh"
#include "epw_tc.cuh"
#include "epw_tcgen05.cuh"

namespace {

constexpr int FX_BK = 32;                            // K of a stage (64-byte rows)
constexpr int FX_RB = 64;
constexpr int FX_A_BYTES = FX_S * 128 * FX_RB;       // 56 KiB
constexpr int FX_B_BYTES = FX_S * FX_NT * FX_RB;     // 28 KiB
constexpr int FX_STAGE = FX_A_BYTES + FX_B_BYTES;
constexpr int FX_STAGES = 2;
constexpr int FX_SMEM = FX_STAGES * FX_STAGE + 1024;
constexpr int FX_EPI = 8;                            // epilogue warps
constexpr int FX_THREADS = 64 + 32 * FX_EPI;
constexpr int FX_CHUNK = 256 / FX_BK;                // stages between two readings of the accumulators

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
// 8 consecutive columns per thread, not waited for
__device__ __forceinline__ void tmem_ld8_async(uint32_t taddr, uint32_t (&u)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7])
               : "r"(taddr)
               : "memory");
}
// the loads' registers pass through, so that no use moves above the wait
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&u)[FX_S][8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int l = 0; l < FX_S; l++)
#pragma unroll
    for (int c = 0; c < 8; c++) asm volatile("" : "+r"(u[l][c]));
}

// D = F32, A = B = BF16, K-major, M = 128
__host__ __device__ constexpr uint32_t fx_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

struct FxArgs {
  int M, N;  // rows of A and of B
  int mtiles, ntiles, kblocks, mgroup;
  int splits, kb_split;  // K in splits of kb_split stages
  size_t ostride;
  int acc;
  int shift_hi, shift_lo;  // I = (hi << shift_hi) + (lo >> shift_lo)
  long long *C;
  size_t ldc;
  double *out;
  size_t ldo;
  const short *eA, *eB;
  int F;
  unsigned *dstatus;
};

template <bool F64>
__global__ void __launch_bounds__(FX_THREADS, 1)
    k_fx_gemm(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, FxArgs g) {
  __shared__ __align__(8) uint64_t bar_full[FX_STAGES], bar_empty[FX_STAGES], bar_tfull, bar_tempty, bar_final;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int *abort_flag = &abort_sh;
  const int nitems = g.mtiles * g.ntiles * g.splits;
  if (threadIdx.x == 0) {
    for (int s = 0; s < FX_STAGES; s++) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    mbar_init(smem_u32(&bar_tfull), 1);
    mbar_init(smem_u32(&bar_tempty), FX_EPI);
    mbar_init(smem_u32(&bar_final), 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_sh), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  // tiles in groups of mgroup rows of tiles, the row index fastest: the CTAs of a wave share
  // both operands' tiles through L2
  auto coords = [&](int it0, int &mt, int &nt, int &sp, int &nkb) {
    const int item = it0 / g.splits;
    sp = it0 - item * g.splits;
    nkb = min(g.kb_split, g.kblocks - sp * g.kb_split);
    const int per = g.mgroup * g.ntiles, grp = item / per, rest = item - grp * per;
    const int mg = min(g.mgroup, g.mtiles - grp * g.mgroup);
    nt = rest / mg;
    mt = grp * g.mgroup + rest - nt * mg;
  };
  if (warp == 0) {
    int issued[FX_STAGES] = {0, 0};
    uint32_t it = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      int mt, nt, sp, nkb;
      coords(item, mt, nt, sp, nkb);
      for (int kb = 0; kb < nkb; kb++, it++) {
        const int s = it % FX_STAGES;
        if (lane == 0) {
          ok = wait_bar(smem_u32(&bar_empty[s]), ((it / FX_STAGES) & 1u) ^ 1u, abort_flag, g.dstatus);
          if (ok) {
            const uint32_t base = smem0 + s * FX_STAGE, fb = smem_u32(&bar_full[s]);
            mbar_expect_tx(fb, FX_STAGE);
            const int kx = (sp * g.kb_split + kb) * FX_BK;
            tma_load_3d(base, &mA, kx, mt * 128, 0, fb);
            tma_load_3d(base + FX_A_BYTES, &mB, kx, nt * FX_NT, 0, fb);
            issued[0] = s == 0 ? (int)(it / FX_STAGES) + 1 : issued[0];
            issued[1] = s == 1 ? (int)(it / FX_STAGES) + 1 : issued[1];
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
      }
    }
    if (lane == 0) {
#pragma unroll
      for (int z = 0; z < FX_STAGES; z++)
        if (issued[z] > 0) drain_bar(smem_u32(&bar_full[z]), (uint32_t)((issued[z] - 1) & 1));
    }
    __syncwarp();
  } else if (warp == 1) {
    uint32_t it = 0, chunk = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      int mt, nt, sp, nkb;
      coords(item, mt, nt, sp, nkb);
      for (int kb = 0; kb < nkb; kb++, it++) {
        const int s = it % FX_STAGES, kc = kb % FX_CHUNK;
        if (lane == 0) {
          if (kc == 0) ok = wait_bar(smem_u32(&bar_tempty), (chunk & 1u) ^ 1u, abort_flag, g.dstatus);
          if (ok) ok = wait_bar(smem_u32(&bar_full[s]), (it / FX_STAGES) & 1u, abort_flag, g.dstatus);
          if (ok) {
            tc_fence_after();
            const uint32_t base = smem0 + s * FX_STAGE;
            const uint64_t dA = sdesc_sw<FX_RB>(base), dB = sdesc_sw<FX_RB>(base + FX_A_BYTES);
#pragma unroll
            for (int ks = 0; ks < FX_BK / 16; ks++) {
              const uint64_t off = (uint64_t)((ks * 32) >> 4);
#pragma unroll
              for (int i = 0; i < FX_S; i++) {
                // plane i of A with planes j0 .. of B, in pieces of at most four planes
#pragma unroll
                for (int j0 = 0; j0 < FX_S - i; j0 += 4) {
                  const int nj = FX_S - i - j0 < 4 ? FX_S - i - j0 : 4;
                  // plane 0 of A meets every level first
                  const uint32_t acc = (kc == 0 && ks == 0 && i == 0) ? 0u : 1u;
                  umma_id<true>(tmem + (i + j0) * FX_NT, dA + off + (uint64_t)((i * 128 * FX_RB) >> 4),
                                dB + off + (uint64_t)((j0 * FX_NT * FX_RB) >> 4), fx_idesc(nj * FX_NT), acc);
                }
              }
            }
            umma_commit(smem_u32(&bar_empty[s]));
            if (kc == FX_CHUNK - 1 || kb == nkb - 1) umma_commit(smem_u32(&bar_tfull));
          }
        }
        if (kc == FX_CHUNK - 1 || kb == nkb - 1) chunk++;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
      }
    }
    if (lane == 0) {
      umma_commit(smem_u32(&bar_final));
      drain_bar(smem_u32(&bar_final), 0);
    }
    __syncwarp();
  } else {
    const int quad = warp & 3, half = (warp - 2) >> 2;
    const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + half * 32;
    uint32_t chunk = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      int mt, nt, sp, nkb;
      coords(item, mt, nt, sp, nkb);
      long long acc[32];
#pragma unroll
      for (int c = 0; c < 32; c++) acc[c] = 0;
      for (int kb = 0; kb < nkb; kb += FX_CHUNK, chunk++) {
        ok = wait_bar(smem_u32(&bar_tfull), chunk & 1u, abort_flag, g.dstatus);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < 32; c0 += 8) {
          uint32_t u[FX_S][8];
#pragma unroll
          for (int l = 0; l < FX_S; l++) tmem_ld8_async(taddr + l * FX_NT + c0, u[l]);
          tmem_ld_wait(u);
#pragma unroll
          for (int c = 0; c < 8; c++) {
            int v[FX_S];
#pragma unroll
            for (int l = 0; l < FX_S; l++) v[l] = __float2int_rn(__uint_as_float(u[l][c]));
            const long long hi = ((long long)v[0] << 24) + ((long long)v[1] << 16) + (long long)((v[2] * 256LL) + v[3]);
            const long long lo = ((long long)v[4] << 16) + ((long long)v[5] << 8) + v[6];
            acc[c0 + c] += (hi << g.shift_hi) + ((lo + (1LL << (g.shift_lo - 1))) >> g.shift_lo);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_tempty));
      }
      if (!ok) break;
      const int m = mt * 128 + quad * 32 + lane, n0 = nt * FX_NT + half * 32;
      if constexpr (!F64) {
        // column-major: a column's 32 rows are 256 contiguous bytes
        if (n0 < g.N) {
#pragma unroll
          for (int c = 0; c < 32; c++)
            if (n0 + c < g.N) g.C[(size_t)(n0 + c) * g.ldc + m] = acc[c];
        }
      } else {
        if (m < g.M) {
          const int ea = g.eA ? g.eA[m] : 0;
          double *o = g.out + sp * g.ostride + (size_t)m * g.ldo + n0;
#pragma unroll
          for (int c = 0; c < 32; c++) {
            if (n0 + c >= g.N) continue;
            const int eb = g.eB ? g.eB[n0 + c] : 0;
            double d = __ll2double_rn(acc[c]);
            if (ea == FX_BAD || eb == FX_BAD)
              d = __longlong_as_double(0x7ff8000000000000LL);
            else if (acc[c] != 0)  // times 2^(ea + eb - F): the exponent field (never subnormal: FX_EMIN)
              d = __longlong_as_double(__double_as_longlong(d) + ((long long)(ea + eb - g.F) << 52));
            o[c] = g.acc ? o[c] + d : d;
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------ digit planes
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

__global__ void __launch_bounds__(128) k_fx_phases(int npt, const double *__restrict__ x, int nR,
                                                   const int *__restrict__ R, int rmax, int kpad, size_t plane,
                                                   __nv_bfloat16 *d, short *e) {
  __shared__ FxFactors F;
  fx_point_phases(
      npt, x, nR, R, rmax, kpad / 2, F, [&](size_t row, bool fin) { e[row] = fin ? 0 : FX_BAD; },
      [&](size_t row, int r, double c, double s) {
        uint32_t pl[FX_S];
        fx_phase_digits(c, s, pl);
        uint32_t *o = reinterpret_cast<uint32_t *>(d + row * kpad) + r;
#pragma unroll
        for (int i = 0; i < FX_S; i++) o[i * (plane / 2)] = pl[i];
      });
}

// Exponent of a row from the largest |x|'s high word: |x| < 2^e; FX_BAD when not finite.
__device__ __forceinline__ int fx_exponent(unsigned hi) {
  const int b = (int)(hi >> 20);
  return b == 0x7ff ? FX_BAD : max(FX_EMIN, b - 1022);
}
__device__ __forceinline__ unsigned absmax_hi(double x, double y) {
  return max((unsigned)__double2hiint(x) & 0x7fffffffu, (unsigned)__double2hiint(y) & 0x7fffffffu);
}

// One block per 32 columns of one k: their largest magnitudes, then 32 x 32 (R, column) tiles
// through shared memory so that both the reads (columns) and the stores (K) are contiguous.
__global__ void __launch_bounds__(256) k_fx_columns(int nR, int ncol, size_t ld, const double2 *__restrict__ src, int kpad,
                                                    size_t plane, __nv_bfloat16 *d, short *e, int *bad) {
  __shared__ double2 tile[32][33];
  __shared__ unsigned mx[32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int c0 = blockIdx.x * 32, k = blockIdx.y;
  const double2 *s = src + (size_t)k * nR * ld;
  if (ty == 0) mx[tx] = 0;
  __syncthreads();
  unsigned m = 0;
  if (c0 + tx < ncol)
    for (int r = ty; r < nR; r += 8) {
      const double2 v = s[(size_t)r * ld + c0 + tx];
      m = max(m, absmax_hi(v.x, v.y));
    }
  atomicMax(&mx[tx], m);
  __syncthreads();
  if (ty == 0 && c0 + tx < ncol) {
    const int ex = fx_exponent(mx[tx]);
    if (ex == FX_BAD && bad) atomicOr(bad, 1);
    const size_t row = (size_t)k * 2 * ncol + 2 * (size_t)(c0 + tx);
    e[row] = e[row + 1] = (short)ex;
  }
  for (int r0 = 0; r0 < kpad / 2; r0 += 32) {
    __syncthreads();
    for (int i = ty; i < 32; i += 8)
      tile[i][tx] = (r0 + i < nR && c0 + tx < ncol) ? s[(size_t)(r0 + i) * ld + c0 + tx] : make_double2(0.0, 0.0);
    __syncthreads();
    if (r0 + tx < kpad / 2) {
      for (int i = ty; i < 32 && c0 + i < ncol; i += 8) {
        const int ex = fx_exponent(mx[i]);
        const double sc = ex == FX_BAD ? 0.0 : pow2d(55 - ex);
        const double2 v = tile[tx][i];
        // (a non-finite row: any digits, its results are NaN through the exponent)
        const long long X = ex == FX_BAD ? 0 : __double2ll_rn(v.x * sc), Y = ex == FX_BAD ? 0 : __double2ll_rn(v.y * sc);
        uint32_t a[FX_S], b[FX_S];
        fx_digits2(X, -Y, a);
        fx_digits2(Y, X, b);
        const size_t row = (size_t)k * 2 * ncol + 2 * (size_t)(c0 + i);
        uint32_t *o = reinterpret_cast<uint32_t *>(d + row * kpad) + r0 + tx;
#pragma unroll
        for (int z = 0; z < FX_S; z++) {
          o[z * (plane / 2)] = a[z];
          o[z * (plane / 2) + kpad / 2] = b[z];
        }
      }
    }
  }
}

// One warp per row, lanes over K.
__global__ void __launch_bounds__(128) k_fx_rows(size_t nrow, int K, size_t ld, const double2 *__restrict__ src,
                                                 int kpad, size_t plane, __nv_bfloat16 *d, short *e) {
  const int lane = threadIdx.x & 31;
  const size_t row = (size_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (row >= nrow) return;
  const double2 *s = src + row * ld;
  unsigned m = 0;
  for (int j = lane; j < K; j += 32) {
    const double2 v = s[j];
    m = max(m, absmax_hi(v.x, v.y));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  const int ex = fx_exponent(m);
  if (lane == 0) e[row] = (short)ex;
  const double sc = ex == FX_BAD ? 0.0 : pow2d(55 - ex);
  uint32_t *o = reinterpret_cast<uint32_t *>(d + row * kpad);
  for (int j = lane; j < kpad / 2; j += 32) {
    const double2 v = j < K && ex != FX_BAD ? s[j] : make_double2(0.0, 0.0);
    uint32_t a[FX_S];
    fx_digits2(__double2ll_rn(v.x * sc), __double2ll_rn(v.y * sc), a);
#pragma unroll
    for (int z = 0; z < FX_S; z++) o[z * (plane / 2) + j] = a[z];
  }
}

// One thread per (R, point), points contiguous; both rows of R.
__global__ void k_fx_phases_conj(int npt, const double *__restrict__ x, int nR, const int *__restrict__ R, int kpad,
                                 size_t plane, __nv_bfloat16 *d) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const int half = kpad / 2;
  if (t >= (size_t)nR * half) return;
  const int r = (int)(t / half), p = (int)(t - (size_t)r * half);
  double s = 0.0, c = 0.0;
  if (p < npt) {
    const double q0 = x[3 * (size_t)p], q1 = x[3 * (size_t)p + 1], q2 = x[3 * (size_t)p + 2];
    double a = q0 * R[3 * r] + q1 * R[3 * r + 1] + q2 * R[3 * r + 2];
    a -= rint(a);
    if (isfinite(a)) sincospi(2.0 * a, &s, &c);  // (such a point's values are NaN on the other side)
  }
  const long long C = __double2ll_rn(c * 36028797018963968.0), S = __double2ll_rn(s * 36028797018963968.0);
  uint32_t a0[FX_S], a1[FX_S];
  fx_digits2(C, S, a0);
  fx_digits2(-S, C, a1);
  uint32_t *o = reinterpret_cast<uint32_t *>(d + (size_t)2 * r * kpad) + p;
#pragma unroll
  for (int z = 0; z < FX_S; z++) {
    o[z * (plane / 2)] = a0[z];
    o[z * (plane / 2) + half] = a1[z];
  }
}

struct FxRows {
  double x, y, z, w;
};
// One warp per element (i, j), i <= j, of one k: its one or two rows (real part h(i,j), imaginary part
// h(j,i)), lanes over R.  The products P(r) X_r stay in registers between the search for the largest
// and the digits when nR <= 256 (beyond, the rest is formed twice): they are most of the work.
__global__ void __launch_bounds__(128) k_fx_hermitian(int nk, int nR, int n, const double2 *__restrict__ p,
                                                      const double2 *__restrict__ X, int kpad, size_t plane,
                                                      __nv_bfloat16 *d, short *e, int *bad) {
  constexpr int NV = 8;
  const int lane = threadIdx.x & 31, ne = n * (n + 1) / 2;
  const size_t w = (size_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (w >= (size_t)nk * ne) return;
  const int k = (int)(w / ne);
  int i = 0, j = (int)(w % ne);
  while (j >= n - i) j -= n - i++;
  j += i;
  // coefficients of (cos, sin): v.x, v.y of the real part's row, v.z, v.w of the imaginary part's
  auto value = [&](int r) {
    double2 a = X[(size_t)r * n * n + i * n + j], b = X[(size_t)r * n * n + j * n + i];
    if (p) {
      const double2 f = p[(size_t)k * nR + r];
      a = make_double2(f.x * a.x - f.y * a.y, f.x * a.y + f.y * a.x);
      b = make_double2(f.x * b.x - f.y * b.y, f.x * b.y + f.y * b.x);
    }
    FxRows v;
    v.x = i == j ? a.x : 0.5 * (a.x + b.x);
    v.y = i == j ? -a.y : -0.5 * (a.y + b.y);
    v.z = 0.5 * (a.y - b.y);
    v.w = 0.5 * (a.x - b.x);
    return v;
  };
  FxRows c[NV];
  unsigned m0 = 0, m1 = 0;
#pragma unroll
  for (int t = 0; t < NV; t++) {
    c[t] = FxRows{0.0, 0.0, 0.0, 0.0};
    const int r = lane + 32 * t;
    if (r < nR) c[t] = value(r);
    m0 = max(m0, absmax_hi(c[t].x, c[t].y));
    m1 = max(m1, absmax_hi(c[t].z, c[t].w));
  }
  for (int r = lane + 32 * NV; r < nR; r += 32) {
    const FxRows v = value(r);
    m0 = max(m0, absmax_hi(v.x, v.y));
    m1 = max(m1, absmax_hi(v.z, v.w));
  }
  const int e0 = fx_exponent(__reduce_max_sync(0xffffffffu, m0)), e1 = fx_exponent(__reduce_max_sync(0xffffffffu, m1));
  const size_t r0 = (size_t)k * n * n + i * n + j, r1 = (size_t)k * n * n + j * n + i;
  if (lane == 0) {
    e[r0] = (short)e0;
    if (i != j) e[r1] = (short)e1;
    if ((e0 == FX_BAD || e1 == FX_BAD) && bad) atomicOr(bad, 1);
  }
  const double s0 = e0 == FX_BAD ? 0.0 : pow2d(55 - e0), s1 = e1 == FX_BAD ? 0.0 : pow2d(55 - e1);
  auto put = [&](int r, const FxRows &v) {
    uint32_t a[FX_S];
    uint32_t *o = reinterpret_cast<uint32_t *>(d + r0 * kpad) + r;
    fx_digits2(e0 == FX_BAD ? 0 : __double2ll_rn(v.x * s0), e0 == FX_BAD ? 0 : __double2ll_rn(v.y * s0), a);
#pragma unroll
    for (int z = 0; z < FX_S; z++) o[z * (plane / 2)] = a[z];
    if (i == j) return;
    o = reinterpret_cast<uint32_t *>(d + r1 * kpad) + r;
    fx_digits2(e1 == FX_BAD ? 0 : __double2ll_rn(v.z * s1), e1 == FX_BAD ? 0 : __double2ll_rn(v.w * s1), a);
#pragma unroll
    for (int z = 0; z < FX_S; z++) o[z * (plane / 2)] = a[z];
  };
#pragma unroll
  for (int t = 0; t < NV; t++)
    if (lane + 32 * t < kpad / 2) put(lane + 32 * t, c[t]);
  for (int r = lane + 32 * NV; r < kpad / 2; r += 32) put(r, r < nR ? value(r) : FxRows{0.0, 0.0, 0.0, 0.0});
}

__global__ void k_fx_unpack(int npt, int n, const double *__restrict__ in, double2 *out) {
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= (size_t)npt * n * n) return;
  const int h = (int)(i % (n * n)), a = h / n, b = h % n;
  const double *s = in + i - h;
  out[i] = a == b ? make_double2(s[h], 0.0)
                  : make_double2(s[fx_hrow(n, min(a, b), max(a, b))],
                                 (a < b ? 1.0 : -1.0) * s[fx_hrow(n, max(a, b), min(a, b))]);
}

PFN_cuTensorMapEncodeTiled_v12000 fx_encode() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult qr;
    const bool ok = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &qr) ==
                        cudaSuccess && qr == cudaDriverEntryPointSuccess;
    return ok ? (PFN_cuTensorMapEncodeTiled_v12000)p : nullptr;
  }();
  return fn;
}
// [FX_S][rows][kpad], box: FX_S planes of box_rows rows of FX_BK elements (64-byte swizzle)
bool fx_map(CUtensorMap *map, const FxOp &o, uint32_t box_rows) {
  auto fn = fx_encode();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)o.kpad, (cuuint64_t)o.rows, FX_S};
  cuuint64_t strides[2] = {(cuuint64_t)o.kpad * 2, (cuuint64_t)o.rows * o.kpad * 2};
  cuuint32_t box[3] = {FX_BK, box_rows, FX_S};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, o.d, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool F64>
epw_status fx_run(const FxOp &A, const FxOp &B, int F, FxArgs &g, cudaStream_t st) {
  if (A.rows <= 0 || B.rows <= 0) return EPW_OK;
  if (A.kpad != B.kpad || F < 39 || F > 61) return EPW_ERR_UNSUPPORTED;
  CUtensorMap ma, mb;
  if (!fx_map(&ma, A, 128) || !fx_map(&mb, B, FX_NT)) return EPW_ERR_CUDA;
  g.M = A.rows;
  g.N = B.rows;
  g.mtiles = (A.rows + 127) / 128;
  g.ntiles = (B.rows + FX_NT - 1) / FX_NT;
  g.mgroup = 4;
  g.kblocks = A.kpad / FX_BK;
  g.kb_split = g.ostride ? fx_kb_split(A.kpad) : g.kblocks;
  g.splits = (g.kblocks + g.kb_split - 1) / g.kb_split;
  // a part of n complex terms sums to at most sqrt(2) n 2^F in units of the row scales: within 63 bits
  if (1.5 * (FX_BK / 2) * std::min(g.kblocks, g.kb_split) > std::ldexp(1.0, 63 - F)) return EPW_ERR_UNSUPPORTED;
  g.shift_hi = F - 38;  // hi counts 2^-38, lo 2^-62
  g.shift_lo = 62 - F;
  g.eA = A.e;
  g.eB = B.e;
  g.F = F;
  if (cudaFuncSetAttribute(k_fx_gemm<F64>, cudaFuncAttributeMaxDynamicSharedMemorySize, FX_SMEM) != cudaSuccess)
    return EPW_ERR_CUDA;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  k_fx_gemm<F64><<<std::min(g.mtiles * g.ntiles * g.splits, sms), FX_THREADS, FX_SMEM, st>>>(ma, mb, g);
  epw_count_launch();
  return cudaGetLastError() == cudaSuccess ? EPW_OK : EPW_ERR_CUDA;
}

}  // namespace

FxOp fx_plan(Arena &A, size_t rows, int kpad, bool exps) {
  FxOp o;
  o.d = A.take<__nv_bfloat16>((size_t)FX_S * rows * kpad);
  o.e = exps ? A.take<short>(rows) : nullptr;
  o.rows = (int)rows;
  o.kpad = kpad;
  return o;
}

void fx_phases(int npt, const double *x, int nR, const int *R, int rmax, const FxOp &o, cudaStream_t st) {
  if (npt <= 0) return;
  k_fx_phases<<<(npt + 15) / 16, 128, 0, st>>>(npt, x, nR, R, rmax, o.kpad, (size_t)o.rows * o.kpad, o.d, o.e);
  epw_count_launch();
}

void fx_columns(int nk, int nR, int ncol, size_t ld, const cx<double> *src, const FxOp &o, int *bad, cudaStream_t st) {
  if (nk <= 0 || ncol <= 0) return;
  k_fx_columns<<<dim3((ncol + 31) / 32, nk), 256, 0, st>>>(nR, ncol, ld, (const double2 *)src, o.kpad,
                                                           (size_t)o.rows * o.kpad, o.d, o.e, bad);
  epw_count_launch();
}

void fx_rows(size_t nrow, int K, size_t ld, const cx<double> *src, const FxOp &o, cudaStream_t st) {
  if (!nrow) return;
  k_fx_rows<<<(unsigned)((nrow + 3) / 4), 128, 0, st>>>(nrow, K, ld, (const double2 *)src, o.kpad,
                                                       (size_t)o.rows * o.kpad, o.d, o.e);
  epw_count_launch();
}

void fx_phases_conj(int npt, const double *x, int nR, const int *R, const FxOp &o, cudaStream_t st) {
  const size_t n = (size_t)nR * (o.kpad / 2);
  if (!n) return;
  k_fx_phases_conj<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(npt, x, nR, R, o.kpad, (size_t)o.rows * o.kpad, o.d);
  epw_count_launch();
}

void fx_hermitian(int nk, int nR, int n, const cx<double> *p, const cx<double> *X, const FxOp &o, int *bad,
                  cudaStream_t st) {
  const size_t rows = (size_t)nk * (n * (n + 1) / 2);
  if (!rows) return;
  k_fx_hermitian<<<(unsigned)((rows + 3) / 4), 128, 0, st>>>(nk, nR, n, (const double2 *)p, (const double2 *)X, o.kpad,
                                                            (size_t)o.rows * o.kpad, o.d, o.e, bad);
  epw_count_launch();
}

epw_status fx_gemm_i64(const FxOp &A, const FxOp &B, int F, long long *C, size_t ldc, unsigned *dstatus,
                       cudaStream_t st) {
  FxArgs g{};
  g.C = C;
  g.ldc = ldc;
  g.dstatus = dstatus;
  return fx_run<false>(A, B, F, g, st);
}

epw_status fx_gemm_f64(const FxOp &A, const FxOp &B, int F, double *out, size_t ldo, unsigned *dstatus,
                       cudaStream_t st, bool acc, size_t ostride) {
  FxArgs g{};
  g.acc = acc ? 1 : 0;
  g.ostride = ostride;
  g.out = out;
  g.ldo = ldo;
  g.dstatus = dstatus;
  return fx_run<true>(A, B, F, g, st);
}

void fx_unpack_hermitian(int npt, int n, const double *in, cx<double> *out, cudaStream_t st) {
  const size_t t = (size_t)npt * n * n;
  if (!t) return;
  k_fx_unpack<<<(unsigned)((t + 255) / 256), 256, 0, st>>>(npt, n, in, (double2 *)out);
  epw_count_launch();
}
