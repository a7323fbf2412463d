// Per-pair FP64 kernels of the linewidth path on contractions that epw_fx.cu has summed on the
// tensor cores.  One thread per (k, q) pair, 128 consecutive q of one k per block.
//
// What bounds them: FP64 issue (one warp instruction per 64 cycles and sub-partition), so two
// warps per sub-partition are enough and only the count of FP64 instructions matters:
//   - the fixed-point values become FP64 with one conversion (the scale is an integer addition
//     to the exponent field);
//   - H(k+q) is diagonalised by Householder reduction and implicit QR (about 5,500 instructions
//     for nw = 8) instead of cyclic Jacobi (about 50,000);
//   - only the eigenvectors and the (m, n) terms are formed whose Gaussians do not underflow in
//     FP64 (|e_nk - e_mk+q| <= max_nu w_qnu + 27.35 sigma; beyond, exp(-y^2) is exactly 0), so
//     every sum equals the dense one; a warp takes its pairs' terms together, 32 at a time.
// Measured: fcc nw = 4, 125 k x 13,824 q 7 ms, diamond nw = 8, 24 k x 8000 q 4.8 ms (contraction, Jacobi
// and every term in one kernel on the CUDA cores: 126 and 181); k_ph64 fcc 8000 k x 216 q 9.0 ms (203).
#include "epw_pair64.cuh"

namespace {

constexpr int P64_REGW = 5;        // matrices up to this order live in registers
constexpr double P64_CUT = 27.35;  // exp(-27.35^2) < 2^-1075

__device__ __forceinline__ double fx_value(long long I, int e, int F) {
  const double d = __ll2double_rn(I);
  const double v = __longlong_as_double(__double_as_longlong(d) + ((long long)(e - F) << 52));
  return e == FX_BAD ? __longlong_as_double(0x7ff8000000000000LL) : (I == 0 ? 0.0 : v);
}

// exp(-z) for z >= 0, table-driven (Tang, ACM Trans. Math. Softw. 15, 144 (1989)): z = n ln2/512 + r,
// exp(-z) = 2^(-n div 512) T[n mod 512] (1 + p(r)), |r| <= ln2/1024, p the Taylor polynomial of
// exp(-r) - 1 to r^4 (the next term is 1e-18).  Nine FP64 instructions; CUDA's exp takes 16 or 17.
// Below 2^-1020 the result is 0.
__device__ __forceinline__ double exp64n(const double *__restrict__ tab, double z) {
  const double magic = 6755399441055744.0;  // 1.5 2^52: the sum's low bits are the rounded integer
  const double t = fma(z, 738.6598609351493, magic);                        // 512 / ln 2
  const int n = __double2loint(t);
  const double nf = t - magic;
  double r = fma(nf, -0.001353803086658445, z);                           // ln 2 / 512: 32 bits and the rest
  r = fma(nf, -3.7269822837316166e-13, r);
  const double p = r * fma(r, fma(r, fma(r, 1.0 / 24.0, -1.0 / 6.0), 0.5), -1.0);
  const double T = tab[n & (EPW_EXPTAB - 1)], v = fma(T, p, T);
  const double s = __hiloint2double(__double2hiint(v) - ((n >> 9) << 20), __double2loint(v));
  // (z <= 707 by its high word, an integer comparison; NaN compares above)
  return __double2hiint(z) <= 0x40861800 ? s : (z != z ? z : 0.0);
}

__device__ __forceinline__ double wsum64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// p ? x : 0, OR-ed into r: a value picked at a runtime index by masks (a chain of selects becomes an
// indexed access, which moves the array to local memory)
__device__ __forceinline__ void pick64(unsigned long long &r, bool p, double x) {
  r |= (p ? ~0ull : 0ull) & (unsigned long long)__double_as_longlong(x);
}
__device__ __forceinline__ double picked(unsigned long long r) { return __longlong_as_double((long long)r); }

// (c, s) of length 1 to the last place: a reciprocal square root and a product leave about two, which the
// rotations of a matrix add up (orders 4, 5, 8, against FP64 Jacobi: orthogonality 3.2, 3.3, 3.2 units of
// 2^-53 without and 2.3, 2.4, 2.4 with, Jacobi 2.6, 2.9, 3.6; v^dagger A v 1.5, 1.4, 1.1 and 1.3, 1.2, 1.0, Jacobi
// 1.4, 1.35, 1.3).
__device__ __forceinline__ void unit64(double &c, double &s) {
  const double d = 0.5 * fma(-c, c, fma(-s, s, 1.0));
  c = fma(c, d, c);
  s = fma(s, d, s);
}

// Hermitian eigenproblem of one thread (n <= W; EX: n = W): Householder reduction
// A = Q T_c Q^dagger (reflector k below the diagonal of column k), a diagonal phase that makes the
// subdiagonal real, implicit QR with Wilkinson shifts (Golub & Van Loan, Sec. 8.3).  Small W in
// registers (every loop unrolled), else in local memory.
template <int W, bool EX>
struct Eig64 {
  static constexpr int U = W <= P64_REGW ? W : 1;  // outer loops
  static constexpr int UI = W <= 9 ? W : 3;  // inner loops
  double2 A[W][W];  // lower triangle; then the reflectors
  double d[W], e[W];
  double V[W][W];   // V[c][r]: eigenvector column c of T
  double tau[W];
  double2 phi[W];

  __device__ __forceinline__ void tridiag(int n) {
    double2 t[W];
    const int nn = EX ? W : n;
#pragma unroll U
    for (int k = 0; k < W - 2; k++) {
      if (k >= nn - 2) continue;
      const double2 x0 = A[k + 1][k];
      double sr = 0.0;
#pragma unroll UI
      for (int i = 2; i < W; i++)
        if (i >= k + 2 && i < nn) sr = fma(A[i][k].x, A[i][k].x, fma(A[i][k].y, A[i][k].y, sr));
      tau[k] = 0.0;
      t[k] = x0;
      if (sr > 0.0) {
        const double n0s = fma(x0.x, x0.x, x0.y * x0.y), tot = n0s + sr;
        const double al = tot * rsqrt(tot);
        const double rn = n0s > 0.0 ? rsqrt(n0s) : 0.0, n0 = n0s * rn;
        const double2 ph = n0s > 0.0 ? make_double2(x0.x * rn, x0.y * rn) : make_double2(1.0, 0.0);
        const double2 v1 = make_double2(ph.x * (n0 + al), ph.y * (n0 + al));
        const double tk = 2.0 / fma(v1.x, v1.x, fma(v1.y, v1.y, sr));  // of the v that is used
        tau[k] = tk;
        t[k] = make_double2(-ph.x * al, -ph.y * al);
        A[k + 1][k] = v1;
        // p = tau B v, K = tau/2 Re(v^dagger p), w = p - K v; B -= v w^dagger + w v^dagger
        double2 p[W];
        double vp = 0.0;
#pragma unroll U
        for (int i = 1; i < W; i++) {
          if (i < k + 1 || i >= nn) continue;
          double2 s = make_double2(0.0, 0.0);
#pragma unroll UI
          for (int j = 1; j < W; j++) {
            if (j < k + 1 || j >= nn) continue;
            const double2 v = A[j][k];
            if (j == i) {
              s.x = fma(A[i][i].x, v.x, s.x);
              s.y = fma(A[i][i].x, v.y, s.y);
            } else {
              const double2 b = j < i ? A[i][j] : make_double2(A[j][i].x, -A[j][i].y);
              s.x = fma(b.x, v.x, fma(-b.y, v.y, s.x));
              s.y = fma(b.x, v.y, fma(b.y, v.x, s.y));
            }
          }
          p[i] = make_double2(tk * s.x, tk * s.y);
          vp = fma(A[i][k].x, p[i].x, fma(A[i][k].y, p[i].y, vp));
        }
        const double K = 0.5 * tk * vp;
#pragma unroll UI
        for (int i = 1; i < W; i++)
          if (i >= k + 1 && i < nn) p[i] = make_double2(fma(-K, A[i][k].x, p[i].x), fma(-K, A[i][k].y, p[i].y));
#pragma unroll U
        for (int i = 1; i < W; i++) {
          if (i < k + 1 || i >= nn) continue;
          const double2 vi = A[i][k], wi = p[i];
#pragma unroll UI
          for (int j = 1; j < W; j++) {
            if (j < k + 1 || j > i) continue;
            const double2 vj = A[j][k], wj = p[j];
            // v_i conj(w_j) + w_i conj(v_j)
            A[i][j].x -= fma(vi.x, wj.x, fma(vi.y, wj.y, fma(wi.x, vj.x, wi.y * vj.y)));
            A[i][j].y = j == i ? 0.0
                               : A[i][j].y - fma(vi.y, wj.x, fma(-vi.x, wj.y, fma(wi.y, vj.x, -wi.x * vj.y)));
          }
        }
      }
    }
    if (nn >= 2) {
#pragma unroll U
      for (int k = 0; k < W - 1; k++)
        if (k == nn - 2) t[k] = A[k + 1][k];
    }
    phi[0] = make_double2(1.0, 0.0);
#pragma unroll U
    for (int i = 0; i < W; i++) {
      if (i >= nn) continue;
      d[i] = A[i][i].x;
      e[i] = 0.0;
      if (i < W - 1 && i < nn - 1) {
        const double m2 = fma(t[i].x, t[i].x, t[i].y * t[i].y);
        const double rm = m2 > 0.0 ? rsqrt(m2) : 0.0;
        double2 u = m2 > 0.0 ? make_double2(t[i].x * rm, t[i].y * rm) : make_double2(1.0, 0.0);
        unit64(u.x, u.y);
        phi[i + 1 < W ? i + 1 : 0] =
            make_double2(fma(phi[i].x, u.x, -phi[i].y * u.y), fma(phi[i].x, u.y, phi[i].y * u.x));
        e[i] = m2 * rm;
      }
    }
  }

  // false: not converged.  Every lane of the warp calls it.
  __device__ __forceinline__ bool qr(int n) {
    const int nn = EX ? W : n;
#pragma unroll U
    for (int c = 0; c < W; c++)
#pragma unroll UI
      for (int r = 0; r < W; r++) V[c][r] = c == r ? 1.0 : 0.0;
    if (nn == 1) return d[0] == d[0];
    double scale = 0.0;
#pragma unroll U
    for (int i = 0; i < W; i++)
      if (i < nn) scale = fmax(scale, fmax(fabs(d[i]), fabs(e[i])));
    const double tol = 1.1102230246251565e-16 * scale;  // 2^-53
    bool conv = false;
    const int maxit = 10 * nn;
#pragma unroll 1
    for (int it = 0;; it++) {
      int h = 0, l = 0;
#pragma unroll U
      for (int i = 0; i < W - 1; i++) {
        if (i >= nn - 1) continue;
        if (fabs(e[i]) <= tol) e[i] = 0.0;
        if (e[i] != 0.0) h = i + 1;  // (a NaN never converges)
      }
      conv = h == 0;
      if (__all_sync(0xffffffffu, conv) || it == maxit) break;
#pragma unroll U
      for (int i = 0; i < W - 1; i++)
        if (i < h && e[i] == 0.0) l = i + 1;
      double x = 0.0, z = 0.0, pa = 0.0, pc = 0.0, b = 0.0;
      if constexpr (W <= P64_REGW) {
        unsigned long long ra = 0, rc = 0, rb = 0, rx = 0, rz = 0;
#pragma unroll
        for (int i = 0; i < W - 1; i++) {
          pick64(ra, i == h - 1, d[i]);
          pick64(rc, i == h - 1, d[i + 1]);
          pick64(rb, i == h - 1, e[i]);
          pick64(rx, i == l, d[i]);
          pick64(rz, i == l, e[i]);
        }
        pa = picked(ra);
        pc = picked(rc);
        b = picked(rb);
        x = picked(rx);
        z = picked(rz);
      } else if (!conv) {
        pa = d[h - 1];
        pc = d[h];
        b = e[h - 1];
        x = d[l];
        z = e[l];
      }
      // Wilkinson shift of the trailing 2 x 2 block [[pa, b], [b, pc]]
      const double del = 0.5 * (pa - pc), b2 = b * b, q2 = fma(del, del, b2);
      const double rr = q2 > 0.0 ? q2 * rsqrt(q2) : 0.0;
      const double den = del >= 0.0 ? del + rr : del - rr;
      x -= den != 0.0 ? pc - b2 / den : pc;
      const int k0 = __reduce_min_sync(0xffffffffu, conv ? W : l), k1 = __reduce_max_sync(0xffffffffu, h);
#pragma unroll U
      for (int k = 0; k < W - 1; k++) {
        if (k < k0 || k >= k1) continue;
        if (!conv && k >= l && k < h) {
          const double r2 = fma(x, x, z * z);
          const double ri = r2 > 0.0 ? rsqrt(r2) : 0.0;
          double c = r2 > 0.0 ? x * ri : 1.0, s = -z * ri;
          unit64(c, s);
          if (k > l) e[k > 0 ? k - 1 : 0] = r2 * ri;
          // the diagonal by corrections (c^2 + s^2 = 1 used, not rounded twice)
          const double diff = d[k] - d[k + 1], ok = e[k], co = c * ok;
          const double w2 = fma(s, diff, co + co), t = s * w2;
          d[k] -= t;
          d[k + 1] += t;
          const double o = fma(c, w2, -ok);
          e[k] = o;
          x = o;
          if (k + 1 < W - 1 && k + 1 < h) {
            const double en = e[k + 1 < W ? k + 1 : 0];
            z = -s * en;
            e[k + 1 < W ? k + 1 : 0] = c * en;
          }
#pragma unroll UI
          for (int r = 0; r < W; r++) {
            if (!EX && r >= nn) continue;
            const double v0 = V[k][r], v1 = V[k + 1][r];
            V[k][r] = fma(-s, v1, c * v0);
            V[k + 1][r] = fma(s, v0, c * v1);
          }
        }
      }
    }
    double sum = 0.0;  // a NaN on the diagonal alone
#pragma unroll U
    for (int i = 0; i < W; i++)
      if (i < nn) sum += d[i];
    return conv && sum == sum;
  }

  __device__ __forceinline__ double eigenvalue(int m) const {
    if constexpr (W <= P64_REGW) {
      unsigned long long r = 0;
#pragma unroll
      for (int i = 0; i < W; i++) pick64(r, m == i, d[i]);
      return picked(r);
    } else {
      return d[m];
    }
  }

  // eigenvector m: u = Q D V e_m
  __device__ __forceinline__ void vector(int n, int m, double2 (&u)[W]) const {
    const int nn = EX ? W : n;
#pragma unroll UI
    for (int i = 0; i < W; i++) {
      double y = 0.0;
      if constexpr (W <= P64_REGW) {
        unsigned long long r = 0;
#pragma unroll
        for (int c = 0; c < W; c++) pick64(r, m == c, V[c][i]);
        y = picked(r);
      } else {
        y = V[m][i];
      }
      u[i] = i < nn ? make_double2(phi[i].x * y, phi[i].y * y) : make_double2(0.0, 0.0);
    }
#pragma unroll U
    for (int k = W - 3; k >= 0; k--) {
      if (k > nn - 3) continue;
      double2 s = make_double2(0.0, 0.0);
#pragma unroll UI
      for (int i = 1; i < W; i++) {
        if (i < k + 1 || i >= nn) continue;
        const double2 v = A[i][k];
        s.x = fma(v.x, u[i].x, fma(v.y, u[i].y, s.x));
        s.y = fma(v.x, u[i].y, fma(-v.y, u[i].x, s.y));
      }
      s = make_double2(tau[k] * s.x, tau[k] * s.y);
#pragma unroll UI
      for (int i = 1; i < W; i++) {
        if (i < k + 1 || i >= nn) continue;
        const double2 v = A[i][k];
        u[i].x = fma(-v.x, s.x, fma(v.y, s.y, u[i].x));
        u[i].y = fma(-v.x, s.y, fma(-v.y, s.x, u[i].y));
      }
    }
  }
};

// H(k+q) of pair (kl, q) and its eigenproblem.
template <int W, bool EX>
__device__ __forceinline__ bool pair64_eig(const Pair64Args &a, int kl, int q, Eig64<W, EX> &S) {
  const int n = EX ? W : a.nw;
  const long long *C = a.CH + (size_t)kl * n * n * a.ldc + q;
  const short *e = a.eH + (size_t)kl * n * n;
#pragma unroll(W <= P64_REGW ? W : 1)
  for (int j = 0; j < W; j++) {
    if (j >= n) continue;
#pragma unroll(W <= P64_REGW ? W : 1)
    for (int i = 0; i < W; i++) {
      if (i < j || i >= n) continue;
      const int hr = fx_hrow(n, j, i), hi = fx_hrow(n, i, j);
      const double x = fx_value(C[(size_t)hr * a.ldc], e[hr], a.FH);
      // rows hold element (j, i), j < i: the lower triangle is its conjugate
      S.A[i][j] = i == j ? make_double2(x, 0.0) : make_double2(x, -fx_value(C[(size_t)hi * a.ldc], e[hi], a.FH));
    }
  }
  S.tridiag(n);
  return S.qr(n);
}

constexpr int P64_MM = 18;  // modes

// What a warp shares while it works through the terms of its 32 pairs: eigenvectors (component i of
// lane l's at u[s][i][l]), eigenvalues and occupations of MS bands per lane (all of them, or the
// current one), and the list of terms: lane, slot s, band n.
template <int W, int MS, bool OCC = true>
struct P64Warp {
  double2 u[MS][W][32];
  double em[MS][32], f[OCC ? MS : 1][32];
  unsigned short list[32 * W * MS];
};

// f(e) with one exponential and one reciprocal for either sign of e - E_F
__device__ __forceinline__ double fermi64(const Pair64Args &a, double e) {
  const double d = e - a.EF;
  if (!(a.T > 0.0)) return d < 0.0 ? 1.0 : (d > 0.0 ? 0.0 : 0.5);
  const double t = exp64n(a.exptab, fabs(d) * a.inv_kT), r = 1.0 / (1.0 + t);
  return __double2hiint(d) < 0 ? r : t * r;
}

// |e_nk - e_mk+q| <= thr, in FP32 with a margin for the rounding of all three (a term too many
// adds an exact 0)
__device__ __forceinline__ bool p64_reach(float ek, float em, float thr) {
  return fabsf(ek - em) <= fmaf(3e-7f, fabsf(ek) + fabsf(em), thr);
}

// g_mn,nu of one term (pair (kl, q), band n = nb, eigenvector u[.][sl]):
// t_a = u^dagger X_a[:, n], g_nu = sum_a E[a][nu] t_a (plus i C_nu u^dagger U_k[:, n])
template <int W, bool EX, int MM>
__device__ __forceinline__ void pair64_g(const Pair64Args &a, int kl, int q, int nb, const double2 (*u)[32], int sl,
                                         double2 (&g)[MM]) {
  const int n = EX ? W : a.nw, nm = MM <= 9 ? MM : a.nm;
  constexpr int UM = MM <= 9 ? MM : 1;
  const size_t c0 = (size_t)kl * 2 * nm * n * n + 2 * nb;
#pragma unroll UM
  for (int v = 0; v < MM; v++) g[v] = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int al = 0; al < nm; al++) {
    double2 t = make_double2(0.0, 0.0);
    if constexpr (W == 1) {  // the eigenvector is 1
      const size_t c = c0 + 2 * (size_t)al;
      t = make_double2(fx_value(a.CG[c * a.ldc + q], a.eG[c], a.FG), fx_value(a.CG[(c + 1) * a.ldc + q], a.eG[c], a.FG));
    } else
#pragma unroll(W <= 9 ? W : 2)
    for (int i = 0; i < W; i++) {
      if (i >= n) continue;
      const size_t c = c0 + 2 * (size_t)((al * n + i) * n);
      const int e = a.eG[c];
      const double2 ui = u[i][sl];
      const double xr = fx_value(a.CG[c * a.ldc + q], e, a.FG), xi = fx_value(a.CG[(c + 1) * a.ldc + q], e, a.FG);
      t.x = fma(ui.x, xr, fma(ui.y, xi, t.x));
      t.y = fma(ui.x, xi, fma(-ui.y, xr, t.y));
    }
    const double2 *E = a.ET + (size_t)al * nm * a.nq + q;
#pragma unroll UM
    for (int v = 0; v < MM; v++) {
      if (v >= nm) continue;
      const double2 f = E[(size_t)v * a.nq];
      g[v].x = fma(f.x, t.x, fma(-f.y, t.y, g[v].x));
      g[v].y = fma(f.x, t.y, fma(f.y, t.x, g[v].y));
    }
  }
  if (a.Cpol) {
    const cx<double> *Uk = a.Uk + (size_t)(a.k0 + kl) * n * n;
    double2 t = make_double2(0.0, 0.0);
#pragma unroll(W <= 9 ? W : 1)
    for (int i = 0; i < W; i++) {
      if (i >= n) continue;
      const cx<double> w = Uk[i * n + nb];
      const double2 ui = u[i][sl];
      t.x = fma(ui.x, w.x, fma(ui.y, w.y, t.x));
      t.y = fma(ui.x, w.y, fma(-ui.y, w.x, t.y));
    }
#pragma unroll UM
    for (int v = 0; v < MM; v++) {
      if (v >= nm) continue;
      const double2 c = a.Cpol[(size_t)v * a.nq + q];
      g[v].x = fma(-c.y, t.x, fma(-c.x, t.y, g[v].x));
      g[v].y = fma(-c.y, t.y, fma(c.x, t.x, g[v].y));
    }
  }
}

// Walks the reachable terms of a warp's pairs, 32 at a time whichever pair they belong to (on the fcc
// model a pair has about 5 of 16 terms, the busiest lane of a warp twice that).  MS = 1: each lane
// takes its next band m that some n reaches and forms its eigenvector, then the lanes' terms of that
// step go through the warp; MS = W (narrow matrices, whose eigenvectors all fit shared memory): one
// list of all terms, so that only its last 32 can be short.  term(lane of the pair, slot, n) runs for
// every term; step(r0, own0, own1) after the terms r0 .. r0 + 31, with this lane's own range.
// (reach: whether a term (band n = j with FP32 energy ek, e_mk+q = em in FP32) is wanted)
struct P64Window {
  float thr;
  __device__ __forceinline__ bool operator()(float ek, float em) const { return p64_reach(ek, em, thr); }
};
struct P64NoStep {
  __device__ __forceinline__ void operator()(int, int, int) const {}
};
template <int W, bool EX, bool OCC, int MS, class R, class F, class G = P64NoStep>
__device__ __forceinline__ void p64_terms(const Pair64Args &a, const Eig64<W, EX> &S, const float *ekf, bool any,
                                          R reach, P64Warp<W, MS, OCC> &sw, F &&term,
                                          G step = G{}) {
  const int lane = threadIdx.x & 31;
  const int n = EX ? W : a.nw;
  unsigned need = 0;
  if (any) {
#pragma unroll(W <= P64_REGW ? W : 1)
    for (int m = 0; m < W; m++) {
      if (m >= n) continue;
      const float em = (float)S.eigenvalue(m);
      for (int j = 0; j < n; j++)
        if (reach(ekf[j], em)) need |= 1u << m;
    }
  }
  // band m of this lane into slot s; its terms as a mask
  auto band = [&](int m, int s) {
    const double em = S.eigenvalue(m);
    const float emf = (float)em;
    unsigned todo = 0;
    for (int j = 0; j < n; j++)
      if (reach(ekf[j], emf)) todo |= 1u << j;
    double2 u[W];
    S.vector(n, m, u);
#pragma unroll(W <= 9 ? W : 1)
    for (int i = 0; i < W; i++)
      if (i < n) sw.u[s][i][lane] = u[i];
    sw.em[s][lane] = em;
    if constexpr (OCC) sw.f[s][lane] = fermi64(a, em);
    return todo;
  };
  auto run = [&](int cnt, auto &&fill) {
    int off = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, off, o);
      if (lane >= o) off += y;
    }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    off -= cnt;
    fill(off);  // this lane's terms: off .. off + cnt
    __syncwarp();
    for (int r0 = 0; r0 < total; r0 += 32) {
      const int j = r0 + lane;
      if (j < total) {
        const unsigned e = sw.list[j];
        term((int)(e >> 10), (int)((e >> 5) & 31), (int)(e & 31));
      }
      step(r0, off, off + cnt);
    }
    __syncwarp();
  };
  if constexpr (MS > 1) {
    static_assert(MS == W, "a slot per band");
    unsigned todo[W];
    int cnt = 0, left = need;
    // (the lanes' bands in step, so that the eigenvectors are formed together)
#pragma unroll
    for (int t = 0; t < W; t++) todo[t] = 0;
#pragma unroll 1
    for (int t = 0; __any_sync(0xffffffffu, left != 0); t++) {
      if (left) {
        const int m = __ffs(left) - 1;
        left &= left - 1;
        const unsigned d = band(m, t);
#pragma unroll
        for (int c = 0; c < W; c++) todo[c] |= c == t ? d : 0u;
        cnt += __popc(d);
      }
    }
    run(cnt, [&](int off) {
#pragma unroll
      for (int t = 0; t < W; t++) {
        unsigned d = todo[t];
        while (d) {
          sw.list[off++] = (unsigned short)((lane << 10) | (t << 5) | (__ffs(d) - 1));
          d &= d - 1;
        }
      }
    });
  } else {
    while (__any_sync(0xffffffffu, need != 0)) {
      unsigned todo = 0;
      if (need) {
        const int m = __ffs(need) - 1;
        need &= need - 1;
        todo = band(m, 0);
      }
      run(__popc(todo), [&](int off) {
        while (todo) {
          sw.list[off++] = (unsigned short)((lane << 10) | (__ffs(todo) - 1));
          todo &= todo - 1;
        }
      });
    }
  }
}

// Reach of a pair's terms: the largest kept frequency and a Gaussian's width; everything (all) where a
// vertex or a weight that is not finite has to show in terms whose Gaussians are zero too.
__device__ __forceinline__ double p64_threshold(const Pair64Args &a, bool valid, double wmax, bool all) {
  if (!valid) return -1.0;
  if (all) return __longlong_as_double(0x7ff0000000000000LL);
  return __double2hiint(wmax) >= 0 ? wmax + P64_CUT * a.sigma : -1.0;
}

template <int W, bool EX, int MM>
__global__ void __launch_bounds__(128, 2) k_lw64(Pair64Args a) {
  __shared__ double sh[4][W];
  __shared__ float ekf[W];
  constexpr int MS = W <= 4 ? W : 1;
  __shared__ P64Warp<W, MS> sws[4];
  const int qi = blockIdx.x * 128 + threadIdx.x, kl = blockIdx.y, k = a.k0 + kl;
  const bool valid = qi < a.nq;
  const int q = valid ? qi : 0;  // lanes past the last q keep step with their warp
  const int n = EX ? W : a.nw, nm = MM <= 9 ? MM : a.nm;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double *ek = a.eps_k + (size_t)k * n;
  if (threadIdx.x < n) ekf[threadIdx.x] = (float)ek[threadIdx.x];
  __syncthreads();
  Eig64<W, EX> S;
  const bool conv = pair64_eig<W, EX>(a, kl, q, S);
  if (!conv && valid) atomicOr(a.dstatus, EPW_DEV_NOT_CONVERGED);
  const double wm = a.wmax[q];
  const double thr = p64_threshold(a, valid, wm, *a.bad || (a.wq && !isfinite(a.wq[q])));
  double acc[W];
#pragma unroll(W <= P64_REGW ? W : 1)
  for (int j = 0; j < W; j++) acc[j] = 0.0;
  P64Warp<W, MS> &sw = sws[warp];
  const int qw = qi - lane;
  p64_terms<W, EX, true, MS>(a, S, ekf, thr >= 0.0, P64Window{__double2float_ru(thr)}, sw, [&](int sl, int ms, int nb) {
    const int qs = qw + sl;
    double2 g[MM];
    pair64_g<W, EX, MM>(a, kl, qs, nb, sw.u[ms], sl, g);
    const double x = ek[nb] - sw.em[ms][sl], f = sw.f[ms][sl];
    double s = 0.0;
#pragma unroll(MM <= 9 ? MM : 1)
    for (int v = 0; v < MM; v++) {
      if (v >= nm) continue;
      const double w = a.omK[(size_t)v * a.nq + qs];
      if (__double2hiint(w) < 0) continue;
      const double nbv = a.nbT[(size_t)v * a.nq + qs];
      const double yp = (x + w) * a.inv_sigma, ym = (x - w) * a.inv_sigma;
      const double t =
          fma(nbv + f, exp64n(a.exptab, yp * yp), (nbv + 1.0 - f) * exp64n(a.exptab, ym * ym));
      s = fma(fma(g[v].x, g[v].x, g[v].y * g[v].y), t, s);
    }
    s *= a.wq ? a.wq[qs] : a.inv_nq;
    if constexpr (W <= P64_REGW) {
#pragma unroll
      for (int j = 0; j < W; j++)
        if (j == nb) acc[j] += s;
    } else {
      acc[nb] += s;
    }
  });
#pragma unroll(W <= P64_REGW ? W : 1)
  for (int j = 0; j < W; j++) {
    if (j >= n) continue;
    const double s = wsum64(acc[j]);
    if (lane == 0) sh[warp][j] = s;
  }
  __syncthreads();
  if (threadIdx.x < n)
    a.partial[((size_t)k * gridDim.x + blockIdx.x) * n + threadIdx.x] =
        a.gnorm * (((sh[0][threadIdx.x] + sh[1][threadIdx.x]) + sh[2][threadIdx.x]) + sh[3][threadIdx.x]);
}

// delta(x + w) - delta(x - w) without cancellation for soft modes (the identity of gauss_diff_r),
// dp and dm the two Gaussians with their norm
__device__ __forceinline__ double gauss_diff64(const Pair64Args &a, double x, double w, double dp, double dm) {
  const double p = x * a.inv_sigma, b = w * a.inv_sigma, y = 2.0 * p * b;
  return fabs(y) > 1.0 ? dp - dm : -2.0 * a.gnorm * exp64n(a.exptab, fma(p, p, b * b)) * sinh(y);
}

// Adjoint of L = sum c_nk Im Sigma_nk per pair.  With W_nu,mn = c_nk pi w_q [(n+f) d+ + (n+1-f) d-]:
// Gbar_nu = 2 W g_nu, Xbar_a[i][n] = sum_m u_m[i] sum_nu conj(E[a][nu]) Gbar_nu,mn.  A term adds to
// its pair's Xbar column in memory; the terms that a warp handles between two barriers have
// different (pair, n), so no two lanes meet, and a column's terms come in ascending m.
template <int W, bool EX, int MM>
__global__ void __launch_bounds__(128, 2) k_adj64(Pair64Args a) {
  __shared__ double sh[2][4];
  __shared__ float ekf[W];
  constexpr int MS = 1;  // (a barrier between the terms of a pair's bands m: they add to the same Xbar)
  __shared__ P64Warp<W, MS> sws[4];
  const int qi = blockIdx.x * 128 + threadIdx.x, kl = blockIdx.y, k = a.k0 + kl;
  const bool valid = qi < a.nq;
  const int q = valid ? qi : 0;
  const int n = EX ? W : a.nw, nm = MM <= 9 ? MM : a.nm;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double *ek = a.eps_k + (size_t)k * n, *cot = a.cot + (size_t)k * n;
  if (threadIdx.x < n) ekf[threadIdx.x] = (float)ek[threadIdx.x];
  __syncthreads();
  Eig64<W, EX> S;
  const bool conv = pair64_eig<W, EX>(a, kl, q, S);
  if (!conv && valid) atomicOr(a.dstatus, EPW_DEV_NOT_CONVERGED);
  const double wm = a.wmax[q];
  bool all = *a.bad || (a.wq && !isfinite(a.wq[q]));
  for (int j = 0; j < n; j++) all |= !isfinite(cot[j]);
  const double thr = p64_threshold(a, valid, wm, all);
  P64Warp<W, MS> &sw = sws[warp];
  const int qw = qi - lane;
  double sT = 0.0, sE = 0.0;
  double2 *xb = a.xbar + (size_t)kl * nm * n * n * a.nq;
  p64_terms<W, EX, true, MS>(a, S, ekf, thr >= 0.0, P64Window{__double2float_ru(thr)}, sw, [&](int sl, int ms, int nb) {
    const int qs = qw + sl;
    double2 g[MM];
    pair64_g<W, EX, MM>(a, kl, qs, nb, sw.u[ms], sl, g);
    const double em = sw.em[ms][sl], f = sw.f[ms][sl], x = ek[nb] - em;
    const double c = cot[nb] * EPW_PI * (a.wq ? a.wq[qs] : a.inv_nq);
    const double ff = fermi_ff_d(em - a.EF, a.T);
    const double dfE = ff * a.inv_kT, dfT = dfE * (em - a.EF) / a.T;
    double tT = 0.0, tE = 0.0;
#pragma unroll(MM <= 9 ? MM : 1)
    for (int v = 0; v < MM; v++) {
      if (v >= nm) continue;
      const double w = a.omK[(size_t)v * a.nq + qs];
      if (__double2hiint(w) < 0) {  // left out (0 times a vertex that is not finite is not 0)
        g[v] = make_double2(0.0 * g[v].x, 0.0 * g[v].y);
        tT = fma(g[v].x, g[v].y, tT);
        tE = fma(g[v].x, g[v].y, tE);
        continue;
      }
      const double nbv = a.nbT[(size_t)v * a.nq + qs];
      const double yp = (x + w) * a.inv_sigma, ym = (x - w) * a.inv_sigma;
      const double dp = a.gnorm * exp64n(a.exptab, yp * yp), dm = a.gnorm * exp64n(a.exptab, ym * ym);
      const double g2 = fma(g[v].x, g[v].x, g[v].y * g[v].y);
      const double dn = nbv * (nbv + 1.0) * w * a.inv_kT / a.T;
      const double dd = gauss_diff64(a, x, w, dp, dm);
      tT = fma(g2, fma(dn, dp + dm, dfT * dd), tT);
      tE = fma(g2, dfE * dd, tE);
      const double W2 = 2.0 * c * fma(nbv + f, dp, (nbv + 1.0 - f) * dm);
      g[v] = make_double2(W2 * g[v].x, W2 * g[v].y);
    }
    sT = fma(c, tT, sT);
    sE = fma(c, tE, sE);
#pragma unroll 1
    for (int al = 0; al < nm; al++) {
      const double2 *E = a.ET + (size_t)al * nm * a.nq + qs;
      double2 y = make_double2(0.0, 0.0);
#pragma unroll(MM <= 9 ? MM : 1)
      for (int v = 0; v < MM; v++) {
        if (v >= nm) continue;
        const double2 e = E[(size_t)v * a.nq];
        y.x = fma(e.x, g[v].x, fma(e.y, g[v].y, y.x));
        y.y = fma(e.x, g[v].y, fma(-e.y, g[v].x, y.y));
      }
#pragma unroll(W <= 9 ? W : 1)
      for (int i = 0; i < W; i++) {
        if (i >= n) continue;
        double2 *o = xb + (size_t)((al * n + i) * n + nb) * a.nq + qs;
        const double2 u = sw.u[ms][i][sl];
        double2 t = *o;
        t.x = fma(u.x, y.x, fma(-u.y, y.y, t.x));
        t.y = fma(u.x, y.y, fma(u.y, y.x, t.y));
        *o = t;
      }
    }
  });
  sT = wsum64(sT);
  sE = wsum64(sE);
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

// Phonon-side sums (see k_pair_ph): each warp 32 q against a.nkc of the chunk's k-points (few q are
// the rule here: blocks of 128 q left lanes and sub-partitions idle).  The terms of a q go back to
// its lane through shared memory, in order.
template <int W, bool EX, int MM>
__global__ void __launch_bounds__(128, 2) k_ph64(Pair64Args a) {
  __shared__ float ekf_s[4][W];
  __shared__ double dn_w[4][W], ia_w[4][W];
  constexpr int MS = W <= 3 || (W == 4 && MM <= 3) ? W : 1;  // (what fits 48 KB with the terms' results)
  __shared__ P64Warp<W, MS, false> sws[4];
  __shared__ double res[4][32][2 * MM];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nqw = (a.nq + 31) / 32, w_ = blockIdx.x * 4 + warp, chunk = w_ / nqw, qw = (w_ - chunk * nqw) * 32;
  const int nchunk = (a.nk + a.nkc - 1) / a.nkc;
  if (chunk >= nchunk) return;  // the whole warp; only warp-level synchronisation below
  float *ekf = ekf_s[warp];
  double *dn_s = dn_w[warp], *ia_s = ia_w[warp];
  const int qi = qw + lane;
  const bool valid = qi < a.nq;
  const int q = valid ? qi : 0;
  const int n = EX ? W : a.nw, nm = MM <= 9 ? MM : a.nm;
  P64Warp<W, MS, false> &sw = sws[warp];
  const double wm = a.wmax[q];
  double sp[MM], sl_[MM], sz = 0.0;
#pragma unroll
  for (int v = 0; v < MM; v++) sp[v] = sl_[v] = 0.0;
  const int kc1 = min(a.nk, (chunk + 1) * a.nkc);
  for (int kl = chunk * a.nkc; kl < kc1; kl++) {
    const int k = a.k0 + kl;
    const double *ek = a.eps_k + (size_t)k * n;
    __syncwarp();
    if (lane < n) {
      const double e = ek[lane], y = (e - a.EF) * a.inv_sigma;
      ekf[lane] = (float)e;
      dn_s[lane] = a.gnorm * exp64n(a.exptab, y * y);
      ia_s[lane] = a.T > 0.0 ? 1.0 / (1.0 + exp64n(a.exptab, fabs(e - a.EF) * a.inv_kT)) : 0.0;
    }
    __syncwarp();
    Eig64<W, EX> S;
    const bool conv = pair64_eig<W, EX>(a, kl, q, S);
    if (!conv && valid) atomicOr(a.dstatus, EPW_DEV_NOT_CONVERGED);
    const double wk = a.wk ? a.wk[k] : 1.0 / a.nk_total;
    const bool all = *a.bad || !isfinite(wk);
    const double thr = p64_threshold(a, valid, wm, all);
    // nesting: (sum_n delta(e_nk - E_F)) (sum_m delta(e_mk+q - E_F))
    double zn = 0.0, zm = 0.0;
    for (int j = 0; j < n; j++) zn += dn_s[j];
    if (zn != 0.0 || all) {
#pragma unroll(W <= P64_REGW ? W : 1)
      for (int m = 0; m < W; m++) {
        if (m >= n) continue;
        const double y = (S.eigenvalue(m) - a.EF) * a.inv_sigma;
        zm += exp64n(a.exptab, y * y);
      }
      sz = fma(wk * zn, a.gnorm * zm, sz);
    }
    // Pi'': |e_nk - e_mk+q - w| within the Gaussian; lambda: both bands within that of E_F
    const float thrf = __double2float_ru(thr), cutf = __double2float_ru(P64_CUT * a.sigma), ef = (float)a.EF;
    p64_terms<W, EX, false, MS>(
        a, S, ekf, thr >= 0.0,
        [&](float en, float em) {
          return p64_reach(en, em, thrf) || (p64_reach(en, ef, cutf) && p64_reach(em, ef, cutf));
        },
        sw,
        [&](int sl, int ms, int nb) {
          const int qs = qw + sl;
          const double em = sw.em[ms][sl], en = ek[nb], x = en - em, dn = dn_s[nb];
          const double ym = (em - a.EF) * a.inv_sigma;
          const double z = dn != 0.0 ? dn * a.gnorm * exp64n(a.exptab, ym * ym) : 0.0;
          double *r = res[warp][lane];
          // the Gaussians of e_nk - e_mk+q - w; with all of them and z zero the term is
          double gs[MM], any = z;
#pragma unroll
          for (int v = 0; v < MM; v++) {
            gs[v] = 0.0;
            if (v >= nm) continue;
            const double w = a.omK[(size_t)v * a.nq + qs];
            if (__double2hiint(w) < 0) continue;
            const double y = (x - w) * a.inv_sigma;
            gs[v] = a.gnorm * exp64n(a.exptab, y * y);
            any += gs[v];
          }
          if (any == 0.0 && !all) {
#pragma unroll
            for (int v = 0; v < 2 * MM; v++) r[v] = 0.0;
            return;
          }
          // f_nk - f_mk+q = 2 sinh(d/2) e^{-S/2} / ((1 + e^{-|a|}) (1 + e^{-|b|})) (fermi_diff_d)
          double fd;
          if (a.T > 0.0) {
            const double aa = (en - a.EF) * a.inv_kT, bb = (em - a.EF) * a.inv_kT;
            const double d = bb - aa, S2 = fabs(aa) + fabs(bb), ad = fabs(d);
            const double num = exp64n(a.exptab, fmax(0.5 * (S2 - ad), 0.0)) * expm1(-ad);
            const double ib = 1.0 / (1.0 + exp64n(a.exptab, fabs(bb)));
            fd = (d >= 0.0 ? -num : num) * ia_s[nb] * ib;
          } else {
            fd = fermi_d(en, a.EF, a.T) - fermi_d(em, a.EF, a.T);
          }
          double2 g[MM];
          pair64_g<W, EX, MM>(a, kl, qs, nb, sw.u[ms], sl, g);
#pragma unroll
          for (int v = 0; v < MM; v++) {
            const bool keep = v < nm && __double2hiint(a.omK[(size_t)(v < nm ? v : 0) * a.nq + qs]) >= 0;
            const double g2 = fma(g[v].x, g[v].x, g[v].y * g[v].y);
            r[v] = keep ? g2 * fd * gs[v] : 0.0;
            r[MM + v] = keep ? g2 * z : 0.0;
          }
        },
        [&](int r0, int own0, int own1) {
          __syncwarp();
          for (int j = max(own0, r0); j < min(own1, r0 + 32); j++) {
            const double *r = res[warp][j - r0];
#pragma unroll
            for (int v = 0; v < MM; v++) {
              sp[v] = fma(wk, r[v], sp[v]);
              sl_[v] = fma(wk, r[MM + v], sl_[v]);
            }
          }
          __syncwarp();
        });
  }
  if (!valid) return;
  double *o = a.partial + ((size_t)chunk * a.nq + q) * (2 * nm + 1);
#pragma unroll
  for (int v = 0; v < MM; v++)
    if (v < nm) {
      o[v] = sp[v];
      o[nm + v] = sl_[v];
    }
  o[2 * nm] = sz;
}

// e_k+q and g_mn,nu = sum_a E[a][nu] (U_k+q^dagger X_a)_mn (plus the long-range part): lanes over q
// (the contractions' contiguous index), one (m, n) per row of the block.
__global__ void __launch_bounds__(256) k_g64(Pair64Args a) {
  const int q = blockIdx.x * 32 + threadIdx.x, kl = blockIdx.y, k = a.k0 + kl;
  if (q >= a.nq) return;
  const int n = a.nw, nm = a.nm, n2 = n * n;
  const size_t pr = (size_t)q * a.nk + kl;
  if (a.eps_kq && threadIdx.y == 0 && blockIdx.z == 0)
    for (int m = 0; m < n; m++) a.eps_kq[((size_t)k * a.nq + q) * n + m] = a.wkq[pr * n + m];
  if (!a.gout) return;
  const cx<double> *U = a.Ukq + pr * n2, *Uk = a.Uk + (size_t)k * n2;
  const int mn = blockIdx.z * 8 + threadIdx.y;
  if (mn < n2) {
    const int m = mn / n, nb = mn - m * n;
    double2 g[P64_MM];
#pragma unroll
    for (int v = 0; v < P64_MM; v++) g[v] = make_double2(0.0, 0.0);
    for (int al = 0; al < nm; al++) {
      double2 t = make_double2(0.0, 0.0);
      for (int i = 0; i < n; i++) {
        const size_t c = (size_t)kl * 2 * nm * n2 + 2 * (size_t)((al * n + i) * n + nb);
        const int e = a.eG[c];
        const double xr = fx_value(a.CG[c * a.ldc + q], e, a.FG), xi = fx_value(a.CG[(c + 1) * a.ldc + q], e, a.FG);
        const cx<double> u = U[i * n + m];
        t.x = fma(u.x, xr, fma(u.y, xi, t.x));
        t.y = fma(u.x, xi, fma(-u.y, xr, t.y));
      }
#pragma unroll
      for (int v = 0; v < P64_MM; v++) {
        if (v >= nm) break;
        const double2 f = a.ET[((size_t)al * nm + v) * a.nq + q];
        g[v].x = fma(f.x, t.x, fma(-f.y, t.y, g[v].x));
        g[v].y = fma(f.x, t.y, fma(f.y, t.x, g[v].y));
      }
    }
    if (a.Cpol) {
      double2 t = make_double2(0.0, 0.0);
      for (int i = 0; i < n; i++) {
        const cx<double> u = U[i * n + m], w = Uk[i * n + nb];
        t.x = fma(u.x, w.x, fma(u.y, w.y, t.x));
        t.y = fma(u.x, w.y, fma(-u.y, w.x, t.y));
      }
#pragma unroll
      for (int v = 0; v < P64_MM; v++) {
        if (v >= nm) break;
        const double2 c = a.Cpol[(size_t)v * a.nq + q];
        g[v].x = fma(-c.y, t.x, fma(-c.x, t.y, g[v].x));
        g[v].y = fma(-c.y, t.y, fma(c.x, t.x, g[v].y));
      }
    }
    cx<double> *o = a.gout + ((size_t)k * a.nq + q) * nm * n2 + mn;
#pragma unroll
    for (int v = 0; v < P64_MM; v++) {
      if (v >= nm) break;
      o[(size_t)v * n2] = mkc(g[v].x, g[v].y);
    }
  }
}

// One thread per (k, aj, Rp), Rp contiguous in B.
__global__ void k_adj_rotate64(int nk, int k0, int nRp, int nm, int nw, int splits, size_t stride,
                               const double *__restrict__ B, const cx<double> *__restrict__ Uk, cx<double> *G1) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const int naj = nm * nw;
  if (t >= (size_t)naj * nRp) return;
  const int r = (int)(t % nRp), aj = (int)(t / nRp);
  for (int k = blockIdx.y; k < nk; k += gridDim.y) {
    double2 b[EPW_MAX_NW];
    for (int n = 0; n < nw; n++) {
      const double *s = B + ((size_t)k * naj * nw + (size_t)aj * nw + n) * 2 * nRp + 2 * r;
      double2 v = make_double2(0.0, 0.0);
      for (int sp = 0; sp < splits; sp++) {
        const double2 x = *reinterpret_cast<const double2 *>(s + sp * stride);
        v.x += x.x;
        v.y += x.y;
      }
      b[n] = v;
    }
    const cx<double> *U = Uk + (size_t)(k0 + k) * nw * nw;
    for (int i = 0; i < nw; i++) {
      cx<double> acc = mkc(0.0, 0.0);
      for (int n = 0; n < nw; n++) cfma(acc, mkc(b[n].x, b[n].y), conjc(U[i * nw + n]));
      G1[(((size_t)r * naj + aj) * nw + i) * nk + k] = acc;
    }
  }
}

// 32 x 32 tiles through shared memory (Re contiguous on one side, the vertex index on the other).
__global__ void k_dg64(int nRe, int nRp, size_t per, const double *__restrict__ wRe, const double *__restrict__ wRp,
                       const double2 *__restrict__ gT, double2 *dg) {
  __shared__ double2 tile[32][33];
  const size_t nc = (size_t)nRp * per, c0 = (size_t)blockIdx.x * 32;
  const int e0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += 8)
    if (c0 + i < nc && e0 + threadIdx.x < nRe) tile[i][threadIdx.x] = gT[(c0 + i) * nRe + e0 + threadIdx.x];
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8)
    if (e0 + i < nRe && c0 + threadIdx.x < nc) {
      const double s = wRe[e0 + i] * wRp[(c0 + threadIdx.x) / per];
      const double2 v = tile[threadIdx.x][i];
      dg[(size_t)(e0 + i) * nc + c0 + threadIdx.x] = make_double2(s * v.x, s * v.y);
    }
}

__global__ void k_tables64(int nq, int nm, const double *__restrict__ om, double omega_min, double T, double *omK,
                           double *nb, double *wmax) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  double m = -1.0;
  for (int v = 0; v < nm; v++) {
    const size_t i = (size_t)v * nq + q;
    const double w = om[i];
    const bool keep = w >= omega_min && w > 0.0;
    omK[i] = keep ? w : -1.0;
    nb[i] = keep ? bose_d(w, T) : 0.0;
    if (keep) m = fmax(m, w);
  }
  wmax[q] = m;
}

}  // namespace

// The instances go by bounds.  Modes come in threes: 3, 6 and 9 (one to three atoms) are constants of the
// kernel, more take its 18.  Bands take the widths 1, 4, 5 (matrices in registers), 8 and 18 (in local memory);
// a band count that is the width itself is a constant too.  Measured, 57 R each (before: 18 modes and the widths
// 4, 8, 18 for all but four sizes): linewidth 4 bands 3 atoms, 75 k x 4000 q 4.4 -> 4.1 ms, 5 bands 1 atom, 60 k
// 2.9 -> 2.5, 8 bands 3 atoms, 37 k 10.2 -> 9.1 (as a bound instead of a constant 10.3); gradients 1.02 to
// 1.25 times as fast, phonon side 1.02 to 1.27.  Six and seven bands with 9 modes keep the 18 in the linewidth
// (8.3 ms, the constant 9.0: more registers live over the local matrices).
template <template <int, bool, int> class K, int MMAX, int W, bool EX>
static void p64_modes(const Pair64Args &a, dim3 grid, cudaStream_t st) {
  if (a.nm == 3)
    K<W, EX, 3>::run(a, grid, st);
  else if (a.nm == 6)
    K<W, EX, 6>::run(a, grid, st);
  else if (a.nm == 9 && (MMAX == 9 || W != 8 || EX)) {
    if constexpr (MMAX == 9 || W != 8 || EX) K<W, EX, 9>::run(a, grid, st);
  } else if constexpr (MMAX > 9) {
    K<W, EX, MMAX>::run(a, grid, st);
  }
}
template <template <int, bool, int> class K, int WMAX, int MMAX>
static epw_status p64_launch(const Pair64Args &a, dim3 grid, cudaStream_t st) {
  if (a.nw > WMAX || a.nm > MMAX) return EPW_ERR_UNSUPPORTED;
  const int n = a.nw;
  if (n == 1)
    p64_modes<K, MMAX, 1, true>(a, grid, st);
  else if (n < 4)
    p64_modes<K, MMAX, 4, false>(a, grid, st);
  else if (n == 4)
    p64_modes<K, MMAX, 4, true>(a, grid, st);
  else if (n == 5)
    p64_modes<K, MMAX, 5, true>(a, grid, st);
  else if (n < 8)
    p64_modes<K, MMAX, 8, false>(a, grid, st);
  else if (n == 8)
    p64_modes<K, MMAX, 8, true>(a, grid, st);
  else if constexpr (WMAX > 8)
    p64_modes<K, MMAX, WMAX, false>(a, grid, st);
  epw_count_launch();
  return cudaGetLastError() == cudaSuccess ? EPW_OK : EPW_ERR_CUDA;
}

template <int W, bool EX, int MM>
struct Lw64 {
  static void run(const Pair64Args &a, dim3 grid, cudaStream_t st) { k_lw64<W, EX, MM><<<grid, 128, 0, st>>>(a); }
};
template <int W, bool EX, int MM>
struct Adj64 {
  static void run(const Pair64Args &a, dim3 grid, cudaStream_t st) { k_adj64<W, EX, MM><<<grid, 128, 0, st>>>(a); }
};
template <int W, bool EX, int MM>
struct Ph64 {
  static void run(const Pair64Args &a, dim3 grid, cudaStream_t st) { k_ph64<W, EX, MM><<<grid, 128, 0, st>>>(a); }
};

epw_status launch_lw64(const Pair64Args &a, cudaStream_t st) {
  if (a.nk <= 0 || a.nq <= 0) return EPW_OK;
  return p64_launch<Lw64, 18, P64_MM>(a, dim3((a.nq + 127) / 128, a.nk), st);
}

epw_status launch_adj64(const Pair64Args &a, cudaStream_t st) {
  if (a.nk <= 0 || a.nq <= 0) return EPW_OK;
  return p64_launch<Adj64, 8, 9>(a, dim3((a.nq + 127) / 128, a.nk), st);
}

epw_status launch_ph64(const Pair64Args &a, int nchunk, cudaStream_t st) {
  if (a.nk <= 0 || a.nq <= 0) return EPW_OK;
  return p64_launch<Ph64, 8, 9>(a, dim3((unsigned)(((size_t)((a.nq + 31) / 32) * nchunk + 3) / 4)), st);
}

epw_status launch_g64(const Pair64Args &a, cudaStream_t st) {
  if (a.nk <= 0 || a.nq <= 0) return EPW_OK;
  k_g64<<<dim3((a.nq + 31) / 32, a.nk, a.gout ? (a.nw * a.nw + 7) / 8 : 1), dim3(32, 8), 0, st>>>(a);
  epw_count_launch();
  return cudaGetLastError() == cudaSuccess ? EPW_OK : EPW_ERR_CUDA;
}

void launch_adj_rotate64(int nk, int k0, int nRp, int nm, int nw, int splits, size_t stride, const double *B,
                         const cx<double> *Uk, cx<double> *G1, cudaStream_t st) {
  const size_t n = (size_t)nm * nw * nRp;
  if (nk <= 0) return;
  k_adj_rotate64<<<dim3((unsigned)((n + 127) / 128), nk < 65535 ? nk : 65535), 128, 0, st>>>(nk, k0, nRp, nm, nw, splits, stride, B, Uk, G1);
  epw_count_launch();
}

void launch_dg64(const epw_model *m, const cx<double> *gT, double *dg, cudaStream_t st) {
  const size_t per = (size_t)m->nm * m->nw * m->nw, nc = (size_t)m->nRp * per;
  k_dg64<<<dim3((unsigned)((nc + 31) / 32), (m->nRe + 31) / 32), dim3(32, 8), 0, st>>>(
      m->nRe, m->nRp, per, m->wRe, m->wRp, (const double2 *)gT, (double2 *)dg);
  epw_count_launch();
}

void launch_tables64(int nq, int nm, const double *omegaT, double omega_min, double T, double *omK, double *nbT,
                     double *wmax, cudaStream_t st) {
  if (nq <= 0) return;
  k_tables64<<<(nq + 63) / 64, 64, 0, st>>>(nq, nm, omegaT, omega_min, T, omK, nbT, wmax);
  epw_count_launch();
}
