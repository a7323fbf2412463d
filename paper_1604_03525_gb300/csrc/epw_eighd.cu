// Batched FP64 Hermitian eigensolves of the preparation: H(k) (nw x nw) and D(q) (3nat x 3nat).
//
// Cyclic two-sided complex Jacobi, the rotations of jacobi_herm in the same order, so the
// eigenvectors' phases do not depend on which kernel ran.  What bounds it on sm_103a: the FP64
// pipe issues one warp instruction per 64 cycles and SM sub-partition, whatever the number of
// active lanes (measured: a dependent DFMA chain of one lane runs at 65 cycles per step, four
// warps per SM at 76).  So the cost of a rotation is its FP64 instruction count, and a matrix
// that fills only some lanes of a warp wastes the rest:
//   - rotation parameters from three reciprocal square roots (about 7 instructions each)
//     instead of three square roots and three divisions (about 57): jrot_d (not with X: 13,824 of
//     9 x 9 3.2 ms against 2.4);
//   - few matrices: L lanes per matrix, each taking rows of A and of V (k_eigh_coop), so a
//     rotation costs 12 ceil((2n-2)/L) instructions beside its parameters instead of 12 (2n-2);
//   - many matrices: one thread per matrix, in registers for n <= 6 (k_eigh_reg).
// launch_eigh_d takes the form whose count times waves of warps is smallest (eigh_cost).
#include <algorithm>
#include <cmath>

#include "epw_internal.cuh"

namespace {

// X: jacobi_herm's arithmetic to the bit (three square roots and divisions, its order of products, of a
// product's imaginary part the second term fused), whatever the number of matrices: for the FP32 adjoint,
// whose gradient is summed and rounded in FP32, so that one phonon that is cast to FP32 the other way
// moves a few percent of its entries by a last place.
//
// The rotation that zeroes a_pq: c, (sx, sy) = s a_pq/|a_pq|, and the new diagonal.  With theta =
// (aqq - app) / (2 |a_pq|) and h = 1/sqrt(1 + theta^2): c^2 = (1 + |theta| h) / 2, s = sign(theta) h
// / (2c), t = s / c.
template <bool X>
__device__ __forceinline__ void jrot_d(double &app, double &aqq, double ax, double ay, double m2, double &c, double &sx,
                                       double &sy) {
  if constexpr (X) {
    const double mag = sqrt(m2), rinv = 1.0 / mag;
    const double th = (aqq - app) * (0.5 * rinv);
    double t = 1.0 / (fabs(th) + sqrt(fma(th, th, 1.0)));
    t = th < 0.0 ? -t : t;
    c = 1.0 / sqrt(fma(t, t, 1.0));
    const double s = t * c;
    app = fma(-t, mag, app);
    aqq = fma(t, mag, aqq);
    sx = s * (ax * rinv);
    sy = s * (ay * rinv);
  } else {
    const double r = rsqrt(m2);
    const double th = (aqq - app) * (0.5 * r);
    // clamped: theta^2 must not overflow (a rotation that small changes nothing)
    const double at = fmin(fabs(th), 1e150);
    const double h = rsqrt(fma(at, at, 1.0));
    const double rc = rsqrt(fma(0.5 * at, h, 0.5));  // 1/c
    c = fma(0.5 * at, h, 0.5) * rc;
    double s = 0.5 * h * rc;
    s = th < 0.0 ? -s : s;
    const double tm = s * rc * (m2 * r);
    const double sr = s * r;
    app -= tm;
    aqq += tm;
    sx = sr * ax;
    sy = sr * ay;
  }
}

// off + |a|^2 (X: jacobi_herm's roundings; a sweep more or less is a last place of every entry)
template <bool X>
__device__ __forceinline__ double joff_d(double off, double2 a) {
  return X ? off + fma(a.x, a.x, __dmul_rn(a.y, a.y)) : fma(a.x, a.x, fma(a.y, a.y, off));
}

// (u, v) <- (c u - conj(se) v, se u + c v), se = sx + i sy
template <bool X>
__device__ __forceinline__ void jrow_d(double c, double sx, double sy, double2 &u, double2 &v) {
  const double2 a = u, b = v;
  if constexpr (X) {
    u.x = fma(c, a.x, -fma(sx, b.x, __dmul_rn(sy, b.y)));
    u.y = fma(c, a.y, -fma(-sy, b.x, __dmul_rn(sx, b.y)));
    v.x = fma(c, b.x, fma(sx, a.x, -__dmul_rn(sy, a.y)));
    v.y = fma(c, b.y, fma(sy, a.x, __dmul_rn(sx, a.y)));
  } else {
    u.x = fma(-sx, b.x, fma(-sy, b.y, c * a.x));
    u.y = fma(-sx, b.y, fma(sy, b.x, c * a.y));
    v.x = fma(sx, a.x, fma(-sy, a.y, c * b.x));
    v.y = fma(sx, a.y, fma(sy, a.x, c * b.y));
  }
}

// ------------------------------------------------------ one thread per matrix
// A (upper triangle) and V in registers: every index is a compile-time constant.
template <int N, bool X>
__global__ void __launch_bounds__(64) k_eigh_reg(int nmat, const double2 *__restrict__ Ain, double *w, double2 *V,
                                                 unsigned *dstatus) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nmat) return;
  double d[N];
  double2 A[N][N], U[N][N];  // A[i][j], i < j
  const double2 *a = Ain + (size_t)t * N * N;
#pragma unroll
  for (int i = 0; i < N; i++) {
    d[i] = a[i * N + i].x;
#pragma unroll
    for (int j = i + 1; j < N; j++) {
      const double2 x = a[i * N + j], y = a[j * N + i];
      A[i][j] = make_double2(0.5 * (x.x + y.x), 0.5 * (x.y - y.y));
    }
#pragma unroll
    for (int j = 0; j < N; j++) U[i][j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
  }
  bool done = false;
  for (int sweep = 0; sweep <= jacobi_tol<double>::maxsweep; sweep++) {
    double off = 0.0, dg = 0.0;
#pragma unroll
    for (int i = 0; i < N; i++) {
      dg = fma(d[i], d[i], dg);
#pragma unroll
      for (int j = i + 1; j < N; j++) off = joff_d<X>(off, A[i][j]);
    }
    done = off <= jacobi_tol<double>::tol2 * (dg + 2.0 * off);
    if (done || sweep == jacobi_tol<double>::maxsweep) break;
#pragma unroll
    for (int p = 0; p < N - 1; p++)
#pragma unroll
      for (int q = p + 1; q < N; q++) {
        const double ax = A[p][q].x, ay = A[p][q].y, m2 = fma(ax, ax, ay * ay);
        if (m2 != 0.0) {
          double c, sx, sy;
          jrot_d<X>(d[p], d[q], ax, ay, m2, c, sx, sy);
          A[p][q] = make_double2(0.0, 0.0);
#pragma unroll
          for (int r = 0; r < N; r++) {
            if (r == p || r == q) continue;
            // A[r][p], A[r][q] from the stored upper triangle (lower entries are conjugates)
            double2 u = r < p ? A[r][p] : make_double2(A[p][r].x, -A[p][r].y);
            double2 v = r < q ? A[r][q] : make_double2(A[q][r].x, -A[q][r].y);
            jrow_d<X>(c, sx, sy, u, v);
            if (r < p)
              A[r][p] = u;
            else
              A[p][r] = make_double2(u.x, -u.y);
            if (r < q)
              A[r][q] = v;
            else
              A[q][r] = make_double2(v.x, -v.y);
          }
#pragma unroll
          for (int r = 0; r < N; r++) jrow_d<X>(c, sx, sy, U[r][p], U[r][q]);
        }
      }
  }
  if (!done) atomicOr(dstatus, EPW_DEV_NOT_CONVERGED);
  // ascending order by rank (ties keep their order)
#pragma unroll
  for (int i = 0; i < N; i++) {
    int rank = 0;
#pragma unroll
    for (int j = 0; j < N; j++) rank += (d[j] < d[i] || (d[j] == d[i] && j < i)) ? 1 : 0;
    w[(size_t)t * N + rank] = d[i];
#pragma unroll
    for (int r = 0; r < N; r++) V[(size_t)t * N * N + r * N + rank] = U[r][i];
  }
}

// The same with indexed (local-memory) arrays, for n beyond the registers.
template <int N, bool X>
__global__ void __launch_bounds__(64) k_eigh_loc(int nmat, const double2 *__restrict__ Ain, double *w, double2 *V,
                                                 unsigned *dstatus) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nmat) return;
  double d[N];
  double2 A[N][N], U[N][N];
  const double2 *a = Ain + (size_t)t * N * N;
#pragma unroll 1
  for (int i = 0; i < N; i++) {
    d[i] = a[i * N + i].x;
#pragma unroll 1
    for (int j = 0; j < N; j++) {
      const double2 x = a[i * N + j], y = a[j * N + i];
      A[i][j] = make_double2(0.5 * (x.x + y.x), 0.5 * (x.y - y.y));
      U[i][j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
    }
  }
  bool done = false;
#pragma unroll 1
  for (int sweep = 0; sweep <= jacobi_tol<double>::maxsweep; sweep++) {
    double off = 0.0, dg = 0.0;
#pragma unroll 1
    for (int i = 0; i < N; i++) {
      dg = fma(d[i], d[i], dg);
#pragma unroll 1
      for (int j = i + 1; j < N; j++) off = joff_d<X>(off, A[i][j]);
    }
    done = off <= jacobi_tol<double>::tol2 * (dg + 2.0 * off);
    if (done || sweep == jacobi_tol<double>::maxsweep) break;
#pragma unroll 1
    for (int p = 0; p < N - 1; p++)
#pragma unroll 1
      for (int q = p + 1; q < N; q++) {
        const double ax = A[p][q].x, ay = A[p][q].y, m2 = fma(ax, ax, ay * ay);
        if (m2 == 0.0) continue;
        double c, sx, sy;
        jrot_d<X>(d[p], d[q], ax, ay, m2, c, sx, sy);
        A[p][q] = A[q][p] = make_double2(0.0, 0.0);
#pragma unroll
        for (int r = 0; r < N; r++) {
          if (r != p && r != q) {
            double2 u = A[r][p], v = A[r][q];
            jrow_d<X>(c, sx, sy, u, v);
            A[r][p] = u;
            A[p][r] = make_double2(u.x, -u.y);
            A[r][q] = v;
            A[q][r] = make_double2(v.x, -v.y);
          }
          jrow_d<X>(c, sx, sy, U[r][p], U[r][q]);
        }
      }
  }
  if (!done) atomicOr(dstatus, EPW_DEV_NOT_CONVERGED);
#pragma unroll 1
  for (int i = 0; i < N; i++) {
    int rank = 0;
#pragma unroll 1
    for (int j = 0; j < N; j++) rank += (d[j] < d[i] || (d[j] == d[i] && j < i)) ? 1 : 0;
    w[(size_t)t * N + rank] = d[i];
#pragma unroll 1
    for (int r = 0; r < N; r++) V[(size_t)t * N * N + r * N + rank] = U[r][i];
  }
}

// ---------------------------------------------------- L lanes per matrix (n <= 18)
// A and V of a matrix in shared memory; of the 2n rows that a rotation changes (A's, then V's)
// lane l of the group takes l, l + L, ...  Control flow is uniform over the warp (__syncwarp):
// a group whose matrix has converged only keeps step with the others.
constexpr int EC_WARPS = 4;  // one warp per SM sub-partition
template <int L, bool X>
__global__ void __launch_bounds__(EC_WARPS * 32) k_eigh_coop(int nmat, int n, const double2 *__restrict__ Ain,
                                                             double *w, double2 *V, unsigned *dstatus) {
  extern __shared__ __align__(16) double2 ec_sm[];
  constexpr int GW = 32 / L;  // groups per warp
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane / L, l = lane % L;
  const int t0 = (blockIdx.x * EC_WARPS + warp) * GW;
  if (t0 >= nmat) return;  // the whole warp
  const int t = t0 + g;
  const bool have = t < nmat;
  const int nn = n * n, stride = 2 * nn + 1;  // odd: groups on different banks
  double2 *A = ec_sm + (size_t)(warp * GW + g) * stride, *U = A + nn;
  const double2 *a = Ain + (size_t)(have ? t : t0) * nn;
  for (int e = l; e < nn; e += L) {
    const int i = e / n, j = e - i * n;
    const double2 x = a[e], y = a[j * n + i];
    A[e] = make_double2(0.5 * (x.x + y.x), 0.5 * (x.y - y.y));
    U[e] = make_double2(i == j ? 1.0 : 0.0, 0.0);
  }
  __syncwarp();
  bool done = false;
  for (int sweep = 0; sweep <= jacobi_tol<double>::maxsweep; sweep++) {
    double off = 0.0, dg = 0.0;
    for (int i = l; i < n; i += L) {
      const double x = A[i * n + i].x;
      dg = fma(x, x, dg);
      for (int j = i + 1; j < n; j++) off = joff_d<X>(off, A[i * n + j]);
    }
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      dg += __shfl_xor_sync(0xffffffffu, dg, o);
    }
    if constexpr (X) {
      // the lanes' sums come in another order than jacobi_herm's (n^2 / 2 roundings of 2^-53): where that could
      // decide, its order
      const double thr = jacobi_tol<double>::tol2 * (dg + 2.0 * off);
      if (fabs(off - thr) <= 1e-12 * thr) {
        off = dg = 0.0;
        for (int i = 0; i < n; i++) {
          dg = fma(A[i * n + i].x, A[i * n + i].x, dg);
          for (int j = i + 1; j < n; j++) off = joff_d<X>(off, A[i * n + j]);
        }
      }
    }
    done = off <= jacobi_tol<double>::tol2 * (dg + 2.0 * off);
    if (__all_sync(0xffffffffu, done) || sweep == jacobi_tol<double>::maxsweep) break;
    for (int p = 0; p < n - 1; p++)
      for (int q = p + 1; q < n; q++) {
        const double2 apq = A[p * n + q];
        double app = A[p * n + p].x, aqq = A[q * n + q].x;
        const double m2 = fma(apq.x, apq.x, apq.y * apq.y);
        const bool act = !done && m2 != 0.0;
        __syncwarp();
        if (act) {
          double c, sx, sy;
          jrot_d<X>(app, aqq, apq.x, apq.y, m2, c, sx, sy);
          for (int it = l; it < 2 * n; it += L) {
            const bool isA = it < n;
            const int r = isA ? it : it - n;
            if (isA && (r == p || r == q)) {
              // the 2 x 2 block
              A[r * n + r].x = r == p ? app : aqq;
              A[r * n + (r == p ? q : p)] = make_double2(0.0, 0.0);
              continue;
            }
            double2 *row = (isA ? A : U) + r * n;
            double2 u = row[p], v = row[q];
            jrow_d<X>(c, sx, sy, u, v);
            row[p] = u;
            row[q] = v;
            if (isA) {
              A[p * n + r] = make_double2(u.x, -u.y);
              A[q * n + r] = make_double2(v.x, -v.y);
            }
          }
        }
        __syncwarp();
      }
  }
  if (!have) return;
  if (!done && l == 0) atomicOr(dstatus, EPW_DEV_NOT_CONVERGED);
  for (int i = l; i < n; i += L) {
    const double di = A[i * n + i].x;
    int rank = 0;
    for (int j = 0; j < n; j++) {
      const double dj = A[j * n + j].x;
      rank += (dj < di || (dj == di && j < i)) ? 1 : 0;
    }
    w[(size_t)t * n + rank] = di;
    for (int r = 0; r < n; r++) V[(size_t)t * nn + r * n + rank] = U[r * n + i];
  }
}

template <int L, bool X>
void eigh_coop(int nmat, int n, const cx<double> *A, double *w, cx<double> *V, unsigned *dstatus, cudaStream_t st) {
  constexpr int per = EC_WARPS * (32 / L);  // matrices per block
  const size_t smem = (size_t)per * (2 * n * n + 1) * sizeof(double2);
  if (smem > 48 * 1024)
    cudaFuncSetAttribute(k_eigh_coop<L, X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_eigh_coop<L, X><<<(nmat + per - 1) / per, EC_WARPS * 32, smem, st>>>(nmat, n, (const double2 *)A, w, (double2 *)V,
                                                                      dstatus);
}

// FP64 instructions of a rotation times the waves of warps over the GPU's 608 sub-partitions,
// for L lanes per matrix (L = 1: one thread per matrix).  Measured alone, us: 37 of 8 x 8, L = 1
// 1629, 16 413; 37 of 18 x 18, 8 6012, 32 3594; 1000 of 4 x 4, 1 125, 8 82; 9001 of 6 x 6, 1 518,
// 4 567; 13,824 of 9 x 9, 1 2950, 4 3710; 316,000 of 6 x 6, 1 8917, 4 17,679.  The other kernels
// of the preparation share the FP64 pipe, so more lanes have to win by a quarter.
double eigh_cost(long nmat, int n, int L) {
  // (the L-lane form in blocks of four warps, one per sub-partition)
  const double waves = L == 1 ? std::max(1.0, std::ceil((nmat + 31) / 32 / 608.0))
                              : std::max(1.0, std::ceil((nmat * L + 127) / 128 / 152.0));
  const double rows = L == 1 ? 2.0 * n - 2.0 : (double)((2 * n + L - 1) / L);
  return waves * (40.0 + 12.0 * rows) * (L == 1 ? 1.0 : 1.25);
}

template <bool X>
void eigh_d(int nmat, int n, cx<double> *A, double *w, cx<double> *V, unsigned *dstatus, cudaStream_t st) {
  if (!nmat) return;
  const double2 *Ad = (const double2 *)A;
  double2 *Vd = (double2 *)V;
  int L = 1;
  for (int c : {4, 8, 16, 32}) {
    if (eigh_cost(nmat, n, c) < eigh_cost(nmat, n, L)) L = c;
  }
  // the widest matrices do not fit one thread's arrays: always L lanes
  if (n > 9 && L == 1) L = 8;
  if (n > 9 && L == 4) L = 8;  // 8 matrices of 18 x 18 per warp exceed shared memory
  const int s = nmat <= 608 * 32 ? 32 : 64;  // a block per warp while sub-partitions would idle
  const int grid = (nmat + s - 1) / s;
  if (L == 32)
    eigh_coop<32, X>(nmat, n, A, w, V, dstatus, st);
  else if (L == 16)
    eigh_coop<16, X>(nmat, n, A, w, V, dstatus, st);
  else if (L == 8)
    eigh_coop<8, X>(nmat, n, A, w, V, dstatus, st);
  else if (L == 4)
    eigh_coop<4, X>(nmat, n, A, w, V, dstatus, st);
  else {
    if (n > 6) {
      // indexed arrays live in L1, but not in all of it: with no shared memory left on an SM no
      // block that needs some can join it while this kernel runs
      const void *f = n == 7 ? (const void *)k_eigh_loc<7, X> : n == 8 ? (const void *)k_eigh_loc<8, X> : (const void *)k_eigh_loc<9, X>;
      cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 50);
    }
    switch (n) {
      case 1: k_eigh_reg<1, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
      case 2: k_eigh_reg<2, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
      case 3: k_eigh_reg<3, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
      case 4: k_eigh_reg<4, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
      case 5: k_eigh_reg<5, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
      case 6: k_eigh_reg<6, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
      case 7: k_eigh_loc<7, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
      case 8: k_eigh_loc<8, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
      default: k_eigh_loc<9, X><<<grid, s, 0, st>>>(nmat, Ad, w, Vd, dstatus); break;
    }
  }
  epw_count_launch();
}

}  // namespace

void launch_eigh_d(int nmat, int n, cx<double> *A, double *w, cx<double> *V, unsigned *dstatus, cudaStream_t st,
                   bool exact) {
  exact ? eigh_d<true>(nmat, n, A, w, V, dstatus, st) : eigh_d<false>(nmat, n, A, w, V, dstatus, st);
}
