// Per-pair adjoint of the linewidth for the staged FP32 forms (nw <= 8, 3nat <= 9): one thread per
// (k, q) pair diagonalises H(k+q), then each warp takes its pairs' reachable terms together.
//
// The kernel that this replaces evaluated every (m, n, nu) with per-thread arrays of 9 x 8 x 8
// complex in local memory and about 2,200 FP64 instructions a pair for dL/dT and dL/dE_F, nearly
// all of them on Gaussians that underflow.  A term whose FP32 Gaussians are zero adds exact zeros,
// so here
//   - H(k+q) is diagonalised in registers by the same Jacobi rotations (bit-identical bands);
//   - the (m, n) with |e_nk - e_mk+q| <= max_nu w_qnu + 10.3 sigma (beyond, expf(-y^2) = 0 in every
//     one of a mode's three Gaussians) are listed per warp and taken 32 at a time;
//   - Xbar is row-major over q (zeroed before), each term adding its column's entries in memory:
//     the terms that a warp handles between two barriers differ in (pair, n).
// It is bound by the listed terms' FP64 sums and by Xbar's traffic: hex nw = 5, 9 modes, 216 k x 13,824 q
// 9.1 ms (82 with every term).
#include "epw_internal.cuh"

namespace {

constexpr float A32_CUT = 10.3f;

template <int W>
struct A32Warp {
  cx<float> u[W][32];  // each lane's current eigenvector
  float em[32];
  bool all[32];          // every term, also those whose Gaussians are zero
  unsigned short list[32 * W];
};

template <int W, bool EX, int MM>
__global__ void __launch_bounds__(128) k_adj32(PairArgs a) {
  constexpr bool REG = W <= 5;  // matrices in registers, every loop over bands unrolled
  constexpr int UW = REG ? W : 1;
  constexpr int UM = MM;
  __shared__ double sh[2][4];
  __shared__ A32Warp<W> sws[4];
  const int qi = blockIdx.x * 128 + threadIdx.x, kl = blockIdx.y, k = a.k0 + kl;
  const bool valid = qi < a.nq;
  const int q = valid ? qi : 0;  // lanes past the last q keep step with their warp
  const int n = EX ? W : a.nw, nm = MM, n2 = n * n, nq = a.nq;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, qw = qi - lane;
  const float *Ck = a.Cq + (size_t)kl * a.cpk * a.ldc;
  const cx<float> *ET = (const cx<float> *)a.ET;
  A32Warp<W> &sw = sws[warp];
  // bands at k+q
  cx<float> A[W][W], U[W][W];
  float ekq[W];
  {
    const float *C = Ck + q;
#pragma unroll UW
    for (int i = 0; i < W; i++)
#pragma unroll UW
      for (int j = 0; j < W; j++) {
        A[i][j] = mkc(0.0f, 0.0f);
        if (i < n && j < n) {
          const size_t ij = 2 * (size_t)(i * n + j), ji = 2 * (size_t)(j * n + i);
          A[i][j] = mkc(0.5f * (C[ij * a.ldc] + C[ji * a.ldc]), 0.5f * (C[(ij + 1) * a.ldc] - C[(ji + 1) * a.ldc]));
        }
      }
  }
  bool nc = false;
  jacobi_herm<float, W, UW>(A, U, n, jacobi_tol<float>::tol2, jacobi_tol<float>::maxsweep, nc);
  sort_eig<float, W, UW>(A, U, ekq, n);
  if (nc && valid) atomicOr(a.dstatus, EPW_DEV_NOT_CONVERGED);

  const double *ek = a.eps_k + (size_t)k * n, *cot = a.cot + (size_t)k * n;
  // a vertex, weight or cotangent that is not finite shows in every term, zero Gaussians too
  bool all = *a.bad != 0 || (a.wq && !isfinite(a.wq[q]));
  for (int j = 0; j < n; j++) all |= !isfinite(cot[j]);
  const float inv_sigma = (float)(1.0 / a.sigma);
  const float gnorm = (float)(1.0 / (a.sigma * 1.7724538509055160273));
  const double kT = EPW_KB * a.T, ikT2 = 1.0 / (kT * a.T), ikT = 1.0 / kT, inq = 1.0 / nq;
  float wmax = -1.0f;
  for (int v = 0; v < nm; v++) {
    const float w = (float)a.omegaT[(size_t)v * nq + q];
    if (w >= (float)a.omega_min && w > 0.0f) wmax = fmaxf(wmax, w);
  }
  // (a band that is not a number reaches everything)
  const float thr = !valid ? -1.0f
                    : all ? __int_as_float(0x7f800000)
                    : wmax >= 0.0f ? (wmax + A32_CUT * (float)a.sigma) * 1.00001f : -1.0f;
  unsigned need = 0;
#pragma unroll UW
  for (int m = 0; m < W; m++) {
    if (m >= n) continue;
    for (int j = 0; j < n; j++)
      if (thr >= 0.0f && !(fabsf((float)ek[j] - ekq[m]) > thr)) need |= 1u << m;
  }
  double sT = 0.0, sE = 0.0;
  cx<float> *xb = (cx<float> *)a.xbar + (size_t)kl * nm * n2 * nq;
  while (__any_sync(0xffffffffu, need != 0)) {
    // each lane its own next band m: its eigenvector for the warp, its terms to the list
    unsigned todo = 0;
    if (need) {
      const int m = __ffs(need) - 1;
      need &= need - 1;
      float em = 0.0f;
      cx<float> u[W];
      if constexpr (REG) {
#pragma unroll
        for (int c = 0; c < W; c++)
          if (c == m) {
            em = ekq[c];
#pragma unroll
            for (int i = 0; i < W; i++) u[i] = U[i][c];
          }
      } else {
        em = ekq[m];
        for (int i = 0; i < n; i++) u[i] = U[i][m];
      }
      for (int j = 0; j < n; j++)
        if (!(fabsf((float)ek[j] - em) > thr)) todo |= 1u << j;
#pragma unroll UW
      for (int i = 0; i < W; i++)
        if (i < n) sw.u[i][lane] = u[i];
      sw.em[lane] = em;
      sw.all[lane] = all;
    }
    const int cnt = __popc(todo);
    int off = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, off, o);
      if (lane >= o) off += y;
    }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    off -= cnt;
    while (todo) {
      sw.list[off++] = (unsigned short)((lane << 8) | (__ffs(todo) - 1));
      todo &= todo - 1;
    }
    __syncwarp();
    for (int j = lane; j < total; j += 32) {
      const int sl = sw.list[j] >> 8, nb = sw.list[j] & 255, qs = qw + sl;
      const float *C = Ck + qs;
      // g_nu = sum_a E[a][nu] (u^dagger X_a)_n
      cx<float> g[MM];
#pragma unroll UM
      for (int v = 0; v < MM; v++) g[v] = mkc(0.0f, 0.0f);
#pragma unroll 1
      for (int al = 0; al < nm; al++) {
        const float *X = C + 2 * (size_t)(n2 * (1 + al) + nb) * a.ldc;
        cx<float> y = mkc(0.0f, 0.0f);
#pragma unroll UW
        for (int i = 0; i < W; i++)
          if (i < n) cfma(y, conjc(sw.u[i][sl]), mkc(X[2 * (size_t)i * n * a.ldc], X[(2 * (size_t)i * n + 1) * a.ldc]));
#pragma unroll UM
        for (int v = 0; v < MM; v++)
          if (v < nm) cfma(g[v], ET[((size_t)al * nm + v) * nq + qs], y);
      }
      if (a.Cpol) {
        const cx<double> *Uk = a.Uk + (size_t)k * n2;
        cx<float> o = mkc(0.0f, 0.0f);
#pragma unroll UW
        for (int i = 0; i < W; i++)
          if (i < n) cfma(o, conjc(sw.u[i][sl]), ccast<float>(Uk[i * n + nb]));
#pragma unroll UM
        for (int v = 0; v < MM; v++)
          if (v < nm) {
            const cx<float> c = ((const cx<float> *)a.Cpol)[(size_t)v * nq + qs];
            cfma(g[v], mkc(-c.y, c.x), o);
          }
      }
      const float em = sw.em[sl], x = (float)ek[nb] - em;
      const float f = occ_fermi<float>(em, a.EF, a.T);
      const double ff = fermi_ff_d((double)em - a.EF, a.T);
      const double dfE = ff * ikT, dfT = ff * ((double)em - a.EF) * ikT2;
      const double c = cot[nb] * EPW_PI * (a.wq ? a.wq[qs] : inq);
      const bool als = sw.all[sl];
      double tT = 0.0, tE = 0.0;
#pragma unroll UM
      for (int v = 0; v < MM; v++) {
        if (v >= nm) continue;
        const float w = (float)a.omegaT[(size_t)v * nq + qs];
        const bool keep = w >= (float)a.omega_min && w > 0.0f;
        const float dp = gauss_r<float>(x + w, inv_sigma, gnorm), dm = gauss_r<float>(x - w, inv_sigma, gnorm);
        float Wv = 0.0f;
        if (als || (keep && !(dp == 0.0f && dm == 0.0f))) {
          const float nb_ = keep ? occ_bose<float>(w, a.T) : 0.0f;
          const double dn = (double)nb_ * ((double)nb_ + 1.0) * (double)w * ikT2;
          Wv = (float)((keep ? c : 0.0) * ((double)(nb_ + f) * dp + (double)(nb_ + 1.0f - f) * dm));
          // (cabs2 and gauss_diff_r with their fused products written out: dL/dT and dL/dE_F cancel, and
          // round as k_pair's do)
          const double g2 = (double)fmaf(g[v].x, g[v].x, __fmul_rn(g[v].y, g[v].y));
          const float as = x * inv_sigma, bs = w * inv_sigma, y2 = 2.0f * as * bs;
          const double dd = fabsf(y2) > 1.0f ? dp - dm
                                             : -2.0f * gnorm * expf(-fmaf(as, as, __fmul_rn(bs, bs))) * sinhf(y2);
          tT = fma(g2, keep ? dn * ((double)dp + (double)dm) + dfT * dd : 0.0, tT);
          tE = fma(g2, keep ? dfE * dd : 0.0, tE);
        }
        g[v] = (2.0f * Wv) * g[v];
      }
      sT = fma(c, tT, sT);
      sE = fma(c, tE, sE);
      // Xbar_a[i][n] += u_i sum_nu conj(E[a][nu]) Gbar_nu
#pragma unroll 1
      for (int al = 0; al < nm; al++) {
        cx<float> y = mkc(0.0f, 0.0f);
#pragma unroll UM
        for (int v = 0; v < MM; v++)
          if (v < nm) cfma(y, conjc(ET[((size_t)al * nm + v) * nq + qs]), g[v]);
        cx<float> *o = xb + (size_t)((al * n) * n + nb) * nq + qs;
#pragma unroll UW
        for (int i = 0; i < W; i++)
          if (i < n) {
            cx<float> t = o[(size_t)i * n * nq];
            cfma(t, sw.u[i][sl], y);
            o[(size_t)i * n * nq] = t;
          }
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sT += __shfl_down_sync(0xffffffffu, sT, o);
    sE += __shfl_down_sync(0xffffffffu, sE, o);
  }
  if (lane == 0) {
    sh[0][warp] = sT;
    sh[1][warp] = sE;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    const double *t = sh[threadIdx.x];
    (threadIdx.x ? a.partialE : a.partialT)[(size_t)kl * gridDim.x + blockIdx.x] = ((t[0] + t[1]) + t[2]) + t[3];
  }
}

}  // namespace

// By bounds: the modes of one, two or three atoms as a constant; widths 4 and 5 in registers, 8 in local memory.
template <int W, bool EX>
static void adj32_modes(const PairArgs &a, cudaStream_t st) {
  const dim3 grid((a.nq + 127) / 128, a.nkc);
  if (a.nm == 3)
    k_adj32<W, EX, 3><<<grid, 128, 0, st>>>(a);
  else if (a.nm == 6)
    k_adj32<W, EX, 6><<<grid, 128, 0, st>>>(a);
  else
    k_adj32<W, EX, 9><<<grid, 128, 0, st>>>(a);
}

epw_status launch_adj_staged(const PairArgs &a, cudaStream_t st) {
  if (a.nkc <= 0 || a.nq <= 0) return EPW_OK;
  if (!a.Cq || a.nw > 8 || a.nm > 9) return EPW_ERR_UNSUPPORTED;
  if (a.nw < 4)
    adj32_modes<4, false>(a, st);
  else if (a.nw == 4)
    adj32_modes<4, true>(a, st);
  else if (a.nw == 5)
    adj32_modes<5, true>(a, st);
  else
    adj32_modes<8, false>(a, st);
  epw_count_launch();
  return cudaGetLastError() == cudaSuccess ? EPW_OK : EPW_ERR_CUDA;
}
