// C ABI of the linewidth library: model ownership, workspace, argument
// checking and orchestration of the kernels (declared in include/epw.h).
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "epw_host.cuh"

// ------------------------------------------------------------------ errors
static thread_local char g_err[512] = "";
static std::atomic<uint64_t> g_launches{0};

void epw_count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

static epw_status fail(epw_status s, const char *fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return s;
}
epw_status epwi_fail(epw_status s, const char *fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return s;
}

#define CK(call)                                                                                    \
  do {                                                                                              \
    cudaError_t e_ = (call);                                                                        \
    if (e_ != cudaSuccess) {                                                                        \
      return fail(e_ == cudaErrorMemoryAllocation ? EPW_ERR_OOM : EPW_ERR_CUDA, "%s: %s (%s:%d)", #call, \
                  cudaGetErrorString(e_), __FILE__, __LINE__);                                      \
    }                                                                                               \
  } while (0)

#define CKS(expr)                      \
  do {                                 \
    epw_status s_ = (expr);            \
    if (s_ != EPW_OK) return s_;       \
  } while (0)

bool epwi_is_device_ptr(const void *p) {
  if (!p) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

static bool is_device_ptr(const void *p) { return epwi_is_device_ptr(p); }

// ------------------------------------------------------------------ model
static bool same_set(int n1, const int32_t *a, int n2, const int32_t *b) {
  return n1 == n2 && std::memcmp(a, b, sizeof(int32_t) * 3 * (size_t)n1) == 0;
}

template <typename T>
static epw_status upload(T **dst, const T *src, size_t n) {
  *dst = nullptr;
  if (n == 0) return EPW_OK;
  CK(cudaMalloc((void **)dst, n * sizeof(T)));
  CK(cudaMemcpy(*dst, src, n * sizeof(T), cudaMemcpyHostToDevice));
  return EPW_OK;
}

static void free_model_arrays(epw_model *m) {
  void *ptrs[] = {m->Re, m->Rp, m->Rph, m->wRe, m->wRp, m->Hw, m->Phiw, m->Phidf, m->gw, m->mass, m->exptab, m->dstatus,
                  m->ws, m->pZ};
  for (void *p : ptrs)
    if (p) cudaFree(p);
  if (m->aux) cudaStreamDestroy(m->aux);
  if (m->ev_fork) cudaEventDestroy(m->ev_fork);
  if (m->ev_join) cudaEventDestroy(m->ev_join);
  if (m->ev_phase) cudaEventDestroy(m->ev_phase);
  if (m->ev_gate) cudaEventDestroy(m->ev_gate);
  if (m->ev_vertex) cudaEventDestroy(m->ev_vertex);
  if (m->aux2) cudaStreamDestroy(m->aux2);
  if (m->ev_fork2) cudaEventDestroy(m->ev_fork2);
  if (m->ev_join2) cudaEventDestroy(m->ev_join2);
  m->aux = m->aux2 = nullptr;
  m->ev_fork = m->ev_join = m->ev_phase = m->ev_gate = m->ev_vertex = m->ev_fork2 = m->ev_join2 = nullptr;
  if (m->ev) {
    for (int i = 0; i < 2 * EPW_MAX_TIMED; i++)
      if (m->ev[i]) cudaEventDestroy(m->ev[i]);
    free(m->ev);
    m->ev = nullptr;
  }
  free(m->ev_tag);
  m->ev_tag = nullptr;
  tc_free(m);
}

extern "C" epw_status epw_load_wannier(const epw_wannier_desc *d, epw_model **out) {
  g_err[0] = 0;
  if (!d || !out) return fail(EPW_ERR_INVALID_ARG, "null descriptor or output");
  *out = nullptr;
  const int nw = d->nw, nat = d->nat, nm = 3 * nat;
  if (nw < 1 || nw > EPW_MAX_NW) return fail(EPW_ERR_INVALID_ARG, "nw=%d outside [1,%d]", nw, EPW_MAX_NW);
  if (nat < 1 || nm > EPW_MAX_MODES) return fail(EPW_ERR_INVALID_ARG, "3*nat=%d outside [3,%d]", nm, EPW_MAX_MODES);
  if (d->nRe < 1 || d->nRp < 1 || d->nRph < 1) return fail(EPW_ERR_INVALID_ARG, "empty R set");
  if (!d->mass || !d->Re || !d->H || !d->Rph || !d->Phi || !d->Rp || !d->g)
    return fail(EPW_ERR_INVALID_ARG, "null array in descriptor");
  for (int a = 0; a < nat; a++)
    if (!(d->mass[a] > 0.0)) return fail(EPW_ERR_INVALID_ARG, "mass[%d] must be > 0", a);
  int dev = 0;
  CK(cudaGetDevice(&dev));

  const size_t nw2 = (size_t)nw * nw, nm2 = (size_t)nm * nm;
  std::vector<cx<double>> Hw((size_t)d->nRe * nw2), Phiw((size_t)d->nRph * nm2);
  for (int r = 0; r < d->nRe; r++) {
    double w = d->wRe ? d->wRe[r] : 1.0;
    for (size_t e = 0; e < nw2; e++)
      Hw[r * nw2 + e] = mkc(w * d->H[2 * (r * nw2 + e)], w * d->H[2 * (r * nw2 + e) + 1]);
  }
  for (int r = 0; r < d->nRph; r++) {
    double w = d->wRph ? d->wRph[r] : 1.0;
    for (int a = 0; a < nm; a++)
      for (int b = 0; b < nm; b++) {
        size_t e = r * nm2 + a * nm + b;
        double s = w / std::sqrt(d->mass[a / 3] * d->mass[b / 3]);
        Phiw[e] = mkc(s * d->Phi[2 * e], s * d->Phi[2 * e + 1]);
      }
  }
  // the same force constants as double-float pairs (hi = fl32(x), lo = fl32(x - hi))
  std::vector<float4> Phidf(Phiw.size());
  for (size_t e = 0; e < Phiw.size(); e++) {
    const float rh = (float)Phiw[e].x, ih = (float)Phiw[e].y;
    Phidf[e] = make_float4(rh, (float)(Phiw[e].x - (double)rh), ih, (float)(Phiw[e].y - (double)ih));
  }
  const size_t per = nm * nw2;
  std::vector<cx<double>> gw((size_t)d->nRe * d->nRp * per);
  std::vector<double> wRe(d->nRe, 1.0), wRp(d->nRp, 1.0);
  if (d->wRe) std::memcpy(wRe.data(), d->wRe, sizeof(double) * d->nRe);
  if (d->wRp) std::memcpy(wRp.data(), d->wRp, sizeof(double) * d->nRp);
  for (int a = 0; a < d->nRe; a++)
    for (int b = 0; b < d->nRp; b++) {
      double s = wRe[a] * wRp[b];
      size_t o = ((size_t)a * d->nRp + b) * per;
      for (size_t e = 0; e < per; e++) {
        double re, im;
        if (d->g_is_c64) {
          re = ((const float *)d->g)[2 * (o + e)];
          im = ((const float *)d->g)[2 * (o + e) + 1];
        } else {
          re = ((const double *)d->g)[2 * (o + e)];
          im = ((const double *)d->g)[2 * (o + e) + 1];
        }
        gw[o + e] = mkc(s * re, s * im);
      }
    }

  std::vector<double> exptab(EPW_EXPTAB);
  for (int j = 0; j < EPW_EXPTAB; j++) exptab[j] = std::exp2(-(double)j / EPW_EXPTAB);

  epw_model *m = (epw_model *)calloc(1, sizeof(epw_model));
  if (!m) return fail(EPW_ERR_OOM, "host allocation failed");
  m->device = dev;
  m->nw = nw;
  m->nat = nat;
  m->nm = nm;
  m->nRe = d->nRe;
  m->nRp = d->nRp;
  m->nRph = d->nRph;
  m->same_ep = same_set(d->nRe, d->Re, d->nRp, d->Rp);
  m->same_eph = same_set(d->nRe, d->Re, d->nRph, d->Rph);
  m->rmax = 0;
  for (int t = 0; t < 3; t++) {
    const int n = t == 0 ? d->nRe : t == 1 ? d->nRp : d->nRph;
    const int32_t *R = t == 0 ? d->Re : t == 1 ? d->Rp : d->Rph;
    for (long i = 0; i < 3L * n; i++) m->rmax = std::max(m->rmax, std::abs((int)R[i]));
  }
  epw_status s = EPW_OK;
  if ((s = upload(&m->Re, (const int *)d->Re, 3 * (size_t)d->nRe)) != EPW_OK ||
      (s = upload(&m->Rp, (const int *)d->Rp, 3 * (size_t)d->nRp)) != EPW_OK ||
      (s = upload(&m->Rph, (const int *)d->Rph, 3 * (size_t)d->nRph)) != EPW_OK ||
      (s = upload(&m->wRe, wRe.data(), wRe.size())) != EPW_OK || (s = upload(&m->wRp, wRp.data(), wRp.size())) != EPW_OK ||
      (s = upload(&m->Hw, Hw.data(), Hw.size())) != EPW_OK || (s = upload(&m->Phiw, Phiw.data(), Phiw.size())) != EPW_OK ||
      (s = upload(&m->Phidf, Phidf.data(), Phidf.size())) != EPW_OK ||
      (s = upload(&m->gw, gw.data(), gw.size())) != EPW_OK ||
      (s = upload(&m->mass, d->mass, (size_t)nat)) != EPW_OK ||
      (s = upload(&m->exptab, exptab.data(), exptab.size())) != EPW_OK) {
    free_model_arrays(m);
    free(m);
    return s;
  }
  cudaError_t e = cudaMalloc((void **)&m->dstatus, 16);
  if (e == cudaSuccess) e = cudaMemset(m->dstatus, 0, 16);
  if (e != cudaSuccess) {
    free_model_arrays(m);
    free(m);
    return fail(EPW_ERR_CUDA, "status word: %s", cudaGetErrorString(e));
  }
  *out = m;
  return EPW_OK;
}

extern "C" void epw_free_model(epw_model *m) {
  if (!m) return;
  int cur = 0;
  cudaGetDevice(&cur);
  cudaSetDevice(m->device);
  cudaDeviceSynchronize();
  free_model_arrays(m);
  free(m);
  cudaSetDevice(cur);
}

static epw_status ensure_ws(epw_model *m, size_t bytes);

extern "C" epw_status epw_set_vertex(epw_model *m, const void *g, int g_is_c64, void *stream) {
  g_err[0] = 0;
  if (!m || !g) return fail(EPW_ERR_INVALID_ARG, "null model or vertex");
  int cur = -1;
  CK(cudaGetDevice(&cur));
  if (cur != m->device) return fail(EPW_ERR_INVALID_ARG, "model lives on device %d, current device is %d", m->device, cur);
  cudaStream_t st = (cudaStream_t)stream;
  const size_t bytes = (size_t)m->nRe * m->nRp * m->nm * m->nw * m->nw * (g_is_c64 ? 8 : 16);
  const void *gd = g;
  if (!is_device_ptr(g)) {
    CKS(ensure_ws(m, bytes));
    CK(cudaMemcpyAsync(m->ws, g, bytes, cudaMemcpyHostToDevice, st));
    gd = m->ws;
  }
  launch_set_vertex(m, gd, g_is_c64, st);
  CK(cudaGetLastError());
  if (gd != g) CK(cudaStreamSynchronize(st));
  return EPW_OK;
}

extern "C" epw_status epw_set_polar(epw_model *m, const epw_polar_desc *d) {
  g_err[0] = 0;
  if (!m) return fail(EPW_ERR_INVALID_ARG, "null model");
  if (!d) {
    m->polar = 0;
    return EPW_OK;
  }
  if (!d->Zstar) return fail(EPW_ERR_INVALID_ARG, "null Born charges");
  if (!(d->alpha > 0.0) || !std::isfinite(d->alpha)) return fail(EPW_ERR_INVALID_ARG, "alpha must be > 0");
  if (d->gmax < 0 || d->gmax > 16) return fail(EPW_ERR_INVALID_ARG, "gmax must be in [0, 16]");
  if (!std::isfinite(d->prefactor)) return fail(EPW_ERR_INVALID_ARG, "prefactor must be finite");
  const double *A = &d->A[0][0];
  const double det = A[0] * (A[4] * A[8] - A[5] * A[7]) - A[1] * (A[3] * A[8] - A[5] * A[6]) +
                     A[2] * (A[3] * A[7] - A[4] * A[6]);
  if (!(std::fabs(det) > 0.0) || !std::isfinite(det)) return fail(EPW_ERR_INVALID_ARG, "singular lattice vectors");
  double inv[9];
  inv[0] = (A[4] * A[8] - A[5] * A[7]) / det;
  inv[1] = (A[2] * A[7] - A[1] * A[8]) / det;
  inv[2] = (A[1] * A[5] - A[2] * A[4]) / det;
  inv[3] = (A[5] * A[6] - A[3] * A[8]) / det;
  inv[4] = (A[0] * A[8] - A[2] * A[6]) / det;
  inv[5] = (A[2] * A[3] - A[0] * A[5]) / det;
  inv[6] = (A[3] * A[7] - A[4] * A[6]) / det;
  inv[7] = (A[1] * A[6] - A[0] * A[7]) / det;
  inv[8] = (A[0] * A[4] - A[1] * A[3]) / det;
  for (int i = 0; i < 3; i++)
    for (int c = 0; c < 3; c++) m->pb[i * 3 + c] = 2.0 * EPW_PI * inv[c * 3 + i];
  for (int i = 0; i < 9; i++) m->peps[i] = (&d->eps_inf[0][0])[i];
  int cur = -1;
  CK(cudaGetDevice(&cur));
  if (cur != m->device) return fail(EPW_ERR_INVALID_ARG, "model lives on device %d, current device is %d", m->device, cur);
  if (!m->pZ) CK(cudaMalloc((void **)&m->pZ, sizeof(double) * 9 * m->nat));
  CK(cudaMemcpy(m->pZ, d->Zstar, sizeof(double) * 9 * m->nat, cudaMemcpyHostToDevice));
  m->palpha = d->alpha;
  m->ppref = d->prefactor;
  m->pgmax = d->gmax;
  m->polar = 1;
  return EPW_OK;
}

extern "C" epw_status epw_model_info(const epw_model *m, int *nw, int *nat, int *nRe, int *nRp, int *nRph) {
  if (!m) return fail(EPW_ERR_INVALID_ARG, "null model");
  if (nw) *nw = m->nw;
  if (nat) *nat = m->nat;
  if (nRe) *nRe = m->nRe;
  if (nRp) *nRp = m->nRp;
  if (nRph) *nRph = m->nRph;
  return EPW_OK;
}

extern "C" uint64_t epw_launch_count(void) { return g_launches.load(); }

// ------------------------------------------------------ measurement hook
// Timed launches carry a tag: 0 the dominant kernel, 1 a secondary one (the
// per-pair eigensolve kernel of the wide-shape form).
void epw_timing_begin_tag(epw_model *m, cudaStream_t st, int tag) {
  if (!m->timing || !m->ev || m->nev >= EPW_MAX_TIMED) return;
  cudaEventRecord(m->ev[2 * m->nev], st);
  m->ev_tag[m->nev] = (unsigned char)(tag & 1);
}
void epw_timing_begin(epw_model *m, cudaStream_t st) { epw_timing_begin_tag(m, st, 0); }
void epw_timing_end(epw_model *m, cudaStream_t st) {
  if (!m->timing || !m->ev || m->nev >= EPW_MAX_TIMED) return;
  cudaEventRecord(m->ev[2 * m->nev + 1], st);
  m->nev++;
}

extern "C" epw_status epw_timing_enable(epw_model *m, int enable) {
  if (!m) return fail(EPW_ERR_INVALID_ARG, "null model");
  if (enable && !m->ev) {
    m->ev = (cudaEvent_t *)calloc(2 * EPW_MAX_TIMED, sizeof(cudaEvent_t));
    m->ev_tag = (unsigned char *)calloc(EPW_MAX_TIMED, 1);
    if (!m->ev || !m->ev_tag) return fail(EPW_ERR_OOM, "host allocation failed");
    for (int i = 0; i < 2 * EPW_MAX_TIMED; i++) CK(cudaEventCreate(&m->ev[i]));
  }
  m->timing = enable ? 1 : 0;
  m->nev = 0;
  return EPW_OK;
}

extern "C" epw_status epw_timing_read_tags(epw_model *m, double *ms2, int *n2) {
  if (!m) return fail(EPW_ERR_INVALID_ARG, "null model");
  double tot[2] = {0.0, 0.0};
  int cnt[2] = {0, 0};
  for (int i = 0; i < m->nev; i++) {
    float ms = 0.0f;
    CK(cudaEventSynchronize(m->ev[2 * i + 1]));
    CK(cudaEventElapsedTime(&ms, m->ev[2 * i], m->ev[2 * i + 1]));
    tot[m->ev_tag[i]] += ms;
    cnt[m->ev_tag[i]]++;
  }
  for (int t = 0; t < 2; t++) {
    if (ms2) ms2[t] = tot[t];
    if (n2) n2[t] = cnt[t];
  }
  m->nev = 0;
  return EPW_OK;
}

extern "C" epw_status epw_timing_read(epw_model *m, double *total_ms, int *launches) {
  double ms2[2];
  int n2[2];
  CKS(epw_timing_read_tags(m, ms2, n2));
  if (total_ms) *total_ms = ms2[0];
  if (launches) *launches = n2[0];
  return EPW_OK;
}
extern "C" const char *epw_last_error(void) { return g_err; }
extern "C" int epw_abi_version(void) { return EPW_ABI_VERSION; }

// -------------------------------------------------------------- workspace
static epw_status ensure_ws(epw_model *m, size_t bytes) {
  if (bytes <= m->ws_bytes) return EPW_OK;
  size_t avail = 0, total = 0;
  CK(cudaMemGetInfo(&avail, &total));
  // what would not fit even in place of the old workspace leaves that one where it is
  if (bytes > avail + m->ws_bytes)
    return fail(EPW_ERR_OOM, "workspace of %zu bytes: %zu are free", bytes, avail + m->ws_bytes);
  CK(cudaDeviceSynchronize());
  if (m->ws) cudaFree(m->ws);
  m->ws = nullptr;
  m->ws_bytes = 0;
  for (size_t b : {bytes + bytes / 8 + (1 << 20), bytes}) {  // with room to grow, if there is any
    const cudaError_t e = cudaMalloc(&m->ws, b);
    if (e == cudaSuccess) {
      m->ws_bytes = b;
      return EPW_OK;
    }
    m->ws = nullptr;
    cudaGetLastError();
    if (e != cudaErrorMemoryAllocation) return fail(EPW_ERR_CUDA, "workspace: %s", cudaGetErrorString(e));
  }
  return fail(EPW_ERR_OOM, "workspace of %zu bytes: out of memory", bytes);
}

// The fixed-point forms take more workspace than the CUDA cores' (digit planes, the contractions of at
// least one k over all q; 18 bands, 18 modes: 93 KB a q and k).  Plans beyond this, or beyond what the device
// has left, keep the CUDA cores' form, so that a q list of any length that fits without them still does.
static const size_t FX_WS_BYTES = (size_t)64 << 30;

// Plans a call's workspace (plan(A), twice: its size, then its pointers).  The fixed-point forms are
// taken (fx_on) while the whole plan stays within FX_WS_BYTES and can be allocated.
template <class PLAN>
static epw_status plan_ws(epw_model *m, Arena &A, const Fx64 &fx, bool &fx_on, PLAN plan) {
  A = Arena{nullptr, 0, 0};
  CKS(plan(A));
  if (A.off > FX_WS_BYTES && (fx.dq || fx.g1)) {
    fx_on = false;
    A = Arena{nullptr, 0, 0};
    CKS(plan(A));
  }
  epw_status s = ensure_ws(m, A.off);
  if (s == EPW_ERR_OOM && fx_on && (fx.dq || fx.g1)) {
    fx_on = false;
    A = Arena{nullptr, 0, 0};
    CKS(plan(A));
    s = ensure_ws(m, A.off);
    if (s == EPW_OK) g_err[0] = 0;
  }
  CKS(s);
  A = Arena{(char *)m->ws, m->ws_bytes, 0};
  return plan(A);
}

static size_t rsize(int prec) { return prec == EPW_FP64 ? sizeof(cx<double>) : sizeof(cx<float>); }

// Lay out (or, with a null base, measure) the preparation buffers.
static void plan_prep(Arena &A, const epw_model *m, int nk, int nq, int prec, bool stage_k, bool stage_q,
                      bool stage_wq, bool need_B, Prep &p, const Fx64 *fx = nullptr) {
  const size_t sR = rsize(prec);
  const size_t nw2 = (size_t)m->nw * m->nw, nm2 = (size_t)m->nm * m->nm;
  p.bad = nullptr;
  p.kd = stage_k ? A.take<double>(3 * (size_t)nk) : nullptr;
  p.qd = stage_q ? A.take<double>(3 * (size_t)nq) : nullptr;
  p.wqd = stage_wq ? A.take<double>((size_t)nq) : nullptr;
  p.PkRM = A.take<cx<double>>((size_t)nk * m->nRe);
  p.PkT = A.take<cx<double>>((size_t)nk * m->nRe);
  p.Hk = A.take<cx<double>>((size_t)nk * nw2);
  p.epsk = A.take<double>((size_t)nk * m->nw);
  p.Uk = A.take<cx<double>>((size_t)nk * nw2);
  if (fx && fx->pair) {
    p.PqTe = p.PqTp = nullptr;  // the phases are digit planes
    p.PqTph = nullptr;
  } else {
    p.PqTe = A.take<char>(sR * m->nRe * (size_t)nq);
    p.PqTp = m->same_ep ? p.PqTe : A.take<char>(sR * m->nRp * (size_t)nq);
    p.PqTph = (m->same_eph && prec == EPW_FP64) ? (cx<double> *)p.PqTe : A.take<cx<double>>((size_t)m->nRph * nq);
  }
  p.D = A.take<cx<double>>((size_t)nq * nm2);
  p.w2 = A.take<double>((size_t)nq * m->nm);
  p.ev = A.take<cx<double>>((size_t)nq * nm2);
  p.omegaT = A.take<double>((size_t)nq * m->nm);
  p.ET = A.take<char>(sR * nm2 * (size_t)nq);
  p.Cpol = m->polar ? A.take<char>(sR * (size_t)m->nm * nq) : nullptr;
  if (need_B) {
    size_t nbg = (size_t)nk * m->nRp * m->nm * nw2;
    p.G1 = A.take<char>(sR * nbg);
    p.Bg = A.take<char>(sR * nbg);
    p.BH = fx && fx->pair ? nullptr : A.take<char>(sR * (size_t)nk * m->nRe * nw2);
    if (prec != EPW_FP64) {
      p.Pk32 = A.take<cx<float>>((size_t)nk * m->nRe);
      p.gw32 = A.take<cx<float>>((size_t)m->nRe * m->nRp * m->nm * nw2);
    } else {
      p.Pk32 = nullptr;
      p.gw32 = nullptr;
    }
  } else {
    p.G1 = p.Bg = p.BH = nullptr;
    p.Pk32 = p.gw32 = nullptr;
  }
}

// --------------------------------------------- fixed-point contractions
// FP64 instructions (64 cycles a warp on each of 608 sub-partitions) in microseconds at 2 GHz.
static double fp64_us(double per_thread, double threads) {
  return per_thread * 0.032 * std::max(1.0, threads / (32.0 * 608.0));
}
// D(q) as digit planes costs two passes over them and about 30 us of launches; the CUDA cores
// take 4 nR nm^2 FP64 instructions per q (316,000 q of 249 R and 6 modes: 18.6 ms).
static bool fx_dq(const epw_model *m, int nq) {
  return fp64_us(4.0 * m->nRph * m->nm * m->nm, nq) > 150.0;
}
// The pairs: the CUDA cores take 4 nw^2 (nRe + nm nRp) instructions per pair; the planes of both
// sides, the GEMMs and their launches take about 100 us at least.
static bool fx_pair(const epw_model *m, int nk, int nq) {
  return fp64_us(4.0 * m->nw * m->nw * (m->nRe + (double)m->nm * m->nRp), (double)nk * nq) > 150.0;
}

// g(k,Rp) = sum_Re P_k(Re) g(Re,Rp) in FP64: the CUDA cores take 4 nRe instructions per k and
// column; the digit planes of g are 90 bytes of traffic per entry, their GEMM 2,490 cycles per
// 128 k x 32 columns x 16 Re.
static bool fx_g1(const epw_model *m, int nk) {
  const double ncol = (double)m->nRp * m->nm * m->nw * m->nw;
  const double simt = fp64_us(4.0 * m->nRe, ncol * nk);
  const double tiles = (double)((nk + 127) / 128) * std::ceil(ncol / 32.0) * (fx_kpad(m->nRe) / 32);
  return 25.0 + m->nRe * ncol * 90.0 / 4e6 + tiles * 2490.0 / (152.0 * 1900.0) < simt;
}
// Planes of g per block of columns.
static const size_t FX_GW_BYTES = (size_t)2 << 30;

// Contraction chunk of the FP64 form.
static const size_t FX_CT_BYTES = (size_t)2 << 30;

// more: further bytes per k of a chunk (the adjoint's and the interpolation's buffers); kmax: most k of a
// chunk (the adjoint sums over its k in one fixed point; the kernels have k on the grid's second axis).
static const int FX_KC_MAX = 65535;
static void plan_fx(Arena &A, const epw_model *m, int nk, int nq, bool dq, bool pair, bool g1, Fx64 &f,
                    size_t more = 0, int kmax = FX_KC_MAX) {
  f = Fx64{};
  f.dq = dq || pair;
  f.pair = pair;
  f.g1 = g1;
  if (g1) {
    const int kp = fx_kpad(m->nRe);
    const size_t ncol = (size_t)m->nRp * m->nm * m->nw * m->nw;
    f.gcols = (int)std::min<size_t>(ncol, std::max<size_t>(32, FX_GW_BYTES / ((size_t)28 * kp) / 32 * 32));
    f.Ak = fx_plan(A, nk, kp, true);
    f.Gw = fx_plan(A, 2 * (size_t)f.gcols, kp, true);
  }
  if (!f.dq) return;
  const size_t nm2 = (size_t)m->nm * m->nm, nw2 = (size_t)m->nw * m->nw;
  f.Aph = fx_plan(A, nq, fx_kpad(m->nRph), true);
  f.Phi = fx_plan(A, nm2, fx_kpad(m->nRph), true);
  f.Dh = A.take<double>(nm2 * nq);
  if (!pair) return;
  f.Ae = m->same_eph ? f.Aph : fx_plan(A, nq, fx_kpad(m->nRe), true);
  f.Ap = m->same_ep ? f.Ae : fx_plan(A, nq, fx_kpad(m->nRp), true);
  f.ldc = (size_t)(nq + 127) / 128 * 128;
  const size_t cols = nw2 * (1 + 2 * (size_t)m->nm);
  const size_t kplanes = 2 * FX_S * nw2 * ((size_t)fx_kpad(m->nRe) + 2 * (size_t)m->nm * fx_kpad(m->nRp));
  f.kc = (int)std::min<size_t>((size_t)std::min(nk, kmax),
                               std::max<size_t>(1, FX_CT_BYTES / (cols * f.ldc * 8 + kplanes + more)));
  f.BH = fx_plan(A, f.kc * nw2, fx_kpad(m->nRe), true);
  f.BG = fx_plan(A, f.kc * nw2 * 2 * m->nm, fx_kpad(m->nRp), true);
  f.CH = A.take<long long>(f.kc * nw2 * f.ldc);
  f.CG = A.take<long long>(f.kc * nw2 * 2 * m->nm * f.ldc);
  f.omK = A.take<double>((size_t)m->nm * nq);
  f.nbT = A.take<double>((size_t)m->nm * nq);
  f.wmax = A.take<double>(nq);
  f.bad = A.take<int>(1);
}

struct PhaseA;
static PhaseA staged_a(const epw_model *m, TcStaged &s);
// The A operand of a tensor-core form that takes the phases of one R set, Re = Rp: built with the
// planes of D(q) when there are any and Re = Rph.
struct PhaseA {
  int op, kpad;
  void *hi, *lo;
  bool *done;
};
static PhaseA staged_a(const epw_model *m, TcStaged &s) {
  // (with two R sets the operand is built from q: no destination here)
  return m->same_ep ? PhaseA{s.op, s.kpad, s.Ahi, s.Alo, &s.a_done} : PhaseA{s.op, s.kpad, nullptr, nullptr, &s.a_done};
}
// q side: the phases' planes and D(q).
static epw_status run_fx_q(const epw_model *m, int nq, const double *q, Fx64 &f, cx<double> *D, cudaStream_t st,
                           const PhaseA *pa) {
  if (pa)
    tc_phases_a(pa->op, nq, q, m->nRe, m->Re, m->rmax, f.Aph, pa->kpad, pa->hi, pa->lo, st);
  else
    fx_phases(nq, q, m->nRph, m->Rph, m->rmax, f.Aph, st);
  fx_hermitian(1, m->nRph, m->nm, nullptr, m->Phiw, f.Phi, nullptr, st);
  CKS(fx_gemm_f64(f.Aph, f.Phi, fx_bits(m->nRph), f.Dh, (size_t)m->nm * m->nm, m->dstatus, st));
  fx_unpack_hermitian(nq, m->nm, f.Dh, D, st);
  if (f.pair) {
    if (!m->same_eph) fx_phases(nq, q, m->nRe, m->Re, m->rmax, f.Ae, st);
    if (!m->same_ep) fx_phases(nq, q, m->nRp, m->Rp, m->rmax, f.Ap, st);
  }
  return EPW_OK;
}

// G1[k][Rp a j i] = sum_Re P_k(Re) g(Re, Rp)_aji in FP64.
static epw_status run_vertex64(const epw_model *m, int nk, const double *k, const Prep &p, Fx64 *f, cudaStream_t st) {
  const int ncol = m->nRp * m->nm * m->nw * m->nw;
  if (!f || !f->g1) {
    launch_vertex_fewk(nk, m->nRe, ncol, p.PkRM, m->gw, (cx<double> *)p.G1, st);
    return EPW_OK;
  }
  FxOp ak = f->Ak;
  ak.rows = nk;
  fx_phases(nk, k, m->nRe, m->Re, m->rmax, ak, st);
  for (int c0 = 0; c0 < ncol; c0 += f->gcols) {
    const int nc = std::min(f->gcols, ncol - c0);
    FxOp gw = f->Gw;
    gw.rows = 2 * nc;
    fx_columns(1, m->nRe, nc, ncol, m->gw + c0, gw, nullptr, st);
    CKS(fx_gemm_f64(ak, gw, fx_bits(m->nRe), (double *)p.G1 + 2 * (size_t)c0, 2 * (size_t)ncol, m->dstatus, st));
  }
  return EPW_OK;
}

// H(k+q) of the k-points [k0, k0 + kc): as fixed point into f.CH, or as FP64 into f.Hq [nq][kc][nw^2].
static FxOp fx_bh(const epw_model *m, int k0, int kc, const Prep &p, Fx64 &f, cudaStream_t st) {
  FxOp bh = f.BH;  // a last, shorter chunk has fewer rows (and tighter planes)
  bh.rows = kc * m->nw * m->nw;
  fx_hermitian(kc, m->nRe, m->nw, p.PkRM + (size_t)k0 * m->nRe, m->Hw, bh, f.bad, st);
  return bh;
}
static epw_status run_fx_hmat(const epw_model *m, int k0, int kc, const Prep &p, Fx64 &f, cudaStream_t st) {
  const FxOp bh = fx_bh(m, k0, kc, p, f, st);
  return fx_gemm_f64(f.Ae, bh, fx_bits(m->nRe), f.Hq, (size_t)kc * m->nw * m->nw, m->dstatus, st);
}
// g(k,q) U_k into f.CG.
static epw_status run_fx_vertex(const epw_model *m, int k0, int kc, const Prep &p, Fx64 &f, cudaStream_t st) {
  const int ncol = m->nm * m->nw * m->nw;
  FxOp bg = f.BG;
  bg.rows = kc * 2 * ncol;
  fx_columns(kc, m->nRp, ncol, ncol, (const cx<double> *)p.Bg + (size_t)k0 * m->nRp * ncol, bg, f.bad, st);
  return fx_gemm_i64(f.Ap, bg, fx_bits(m->nRp), f.CG, f.ldc, m->dstatus, st);
}
// Both of a chunk.
static epw_status run_fx_contract(const epw_model *m, int k0, int kc, const Prep &p, Fx64 &f, cudaStream_t st) {
  const FxOp bh = fx_bh(m, k0, kc, p, f, st);
  CKS(fx_gemm_i64(f.Ae, bh, fx_bits(m->nRe), f.CH, f.ldc, m->dstatus, st));
  return run_fx_vertex(m, k0, kc, p, f, st);
}

static Pair64Args pair64_args(const epw_model *m, int k0, int kc, int nq, const double *wq, const epw_params *par,
                              const Prep &p, const Fx64 &f) {
  Pair64Args a;
  std::memset(&a, 0, sizeof(a));
  a.nq = nq;
  a.nw = m->nw;
  a.nm = m->nm;
  a.k0 = k0;
  a.nk = kc;
  a.CH = f.CH;
  a.CG = f.CG;
  a.eH = f.BH.e;
  a.eG = f.BG.e;
  a.FH = fx_bits(m->nRe);
  a.FG = fx_bits(m->nRp);
  a.ldc = f.ldc;
  a.ET = (const double2 *)p.ET;
  a.omK = f.omK;
  a.nbT = f.nbT;
  a.wmax = f.wmax;
  a.eps_k = p.epsk;
  a.wq = wq;
  a.T = par->T_K;
  a.EF = par->EF_eV;
  a.sigma = par->sigma_eV;
  a.inv_kT = par->T_K > 0.0 ? 1.0 / (EPW_KB * par->T_K) : 0.0;
  a.inv_sigma = 1.0 / par->sigma_eV;
  a.gnorm = 1.0 / (par->sigma_eV * 1.7724538509055160273);
  a.inv_nq = 1.0 / nq;
  a.dstatus = m->dstatus;
  a.bad = f.bad;
  a.exptab = m->exptab;
  a.Cpol = m->polar ? (const double2 *)p.Cpol : nullptr;
  a.Uk = p.Uk;
  return a;
}

// Phases, k-side bands, phonons and the k-side vertex (Bg, BH).
// The k side (bands at k, k-side vertex) and the q side (phases, phonons, long-range factors) are
// independent: the q side runs on the model's second stream, forked from and joined back into st.
static epw_status prep_streams(epw_model *m) {
  if (m->aux) return EPW_OK;
  CK(cudaStreamCreateWithFlags(&m->aux, cudaStreamNonBlocking));
  CK(cudaEventCreateWithFlags(&m->ev_fork, cudaEventDisableTiming));
  CK(cudaEventCreateWithFlags(&m->ev_join, cudaEventDisableTiming));
  CK(cudaEventCreateWithFlags(&m->ev_phase, cudaEventDisableTiming));
  CK(cudaEventCreateWithFlags(&m->ev_gate, cudaEventDisableTiming));
  CK(cudaEventCreateWithFlags(&m->ev_vertex, cudaEventDisableTiming));
  CK(cudaStreamCreateWithFlags(&m->aux2, cudaStreamNonBlocking));
  CK(cudaEventCreateWithFlags(&m->ev_fork2, cudaEventDisableTiming));
  CK(cudaEventCreateWithFlags(&m->ev_join2, cudaEventDisableTiming));
  return EPW_OK;
}

// tcb (optional): the fused tensor-core kernel's operands are built here, B on the
// main stream after the k side and A after the q phases, both while the q-side
// phonon work (FP64) still runs on the second stream.
static epw_status run_prep(const epw_model *mc, int nk, const double *k, int nq, const double *q, int prec,
                           double omega_min, bool need_B, Prep &p, double *omega_out, cudaStream_t st,
                           bool fork = true, TcBuffers *tcb = nullptr, Fx64 *fx = nullptr,
                           const PhaseA *pa = nullptr) {
  epw_model *m = const_cast<epw_model *>(mc);
  const int nw = m->nw, nm = m->nm;
  const size_t nw2 = (size_t)nw * nw;
  const bool exact = fx && fx->exact;
  // The k side of the FP32 and split forms, always: it is cast to FP32 and split, and a value that is cast
  // the other way moves every q of its k alike (up to 4e-8 of that k's linewidths, 1.5e-9 of a list of 256
  // k); a q's casts are one term of many (316,000 q: below 5e-12).
  const bool exact_k = exact || prec != EPW_FP64;
  cudaStream_t sq = st;
  fork = fork && nq > 0 && nk > 0;
  if (fork) {
    CKS(prep_streams(m));
    CK(cudaEventRecord(m->ev_fork, st));
    CK(cudaStreamWaitEvent(m->aux, m->ev_fork, 0));
    sq = m->aux;
  }
  // q side: phases in working precision (+ FP64 for phonons); the fused tensor-core
  // form takes phases, A operand and D(q) from one double-float kernel instead
  const bool qs = tcb && prec != EPW_FP64 && tc_qside(m, nq, q, *tcb, p.D, sq);
  if (qs) {
    tcb->prebuilt_a = true;
  } else if (fx && fx->pair) {
    CK(cudaMemsetAsync(fx->bad, 0, sizeof(int), st));
  } else if (prec == EPW_FP64) {
    launch_phases(nq, q, m->nRe, m->Re, m->rmax, nullptr, (cx<double> *)p.PqTe, nullptr, sq, exact);
    if (!m->same_ep) launch_phases(nq, q, m->nRp, m->Rp, m->rmax, nullptr, (cx<double> *)p.PqTp, nullptr, sq, exact);
    if (!m->same_eph) launch_phases(nq, q, m->nRph, m->Rph, m->rmax, nullptr, p.PqTph, nullptr, sq, exact);
  } else if (pa) {
    // staged and wide forms read no phase arrays: the A operand (from FP64 phases when Re = Rph)
    const bool dq = fx && fx->dq;
    *pa->done = dq && m->same_eph && pa->hi;
    if (!*pa->done && (!dq || (m->same_eph && pa->hi)))
      launch_phases(nq, q, m->nRph, m->Rph, m->rmax, nullptr, p.PqTph, nullptr, sq, exact);
  } else {
    launch_phases(nq, q, m->nRe, m->Re, m->rmax, nullptr, m->same_eph ? p.PqTph : nullptr, (cx<float> *)p.PqTe, sq, exact);
    if (!m->same_ep) launch_phases(nq, q, m->nRp, m->Rp, m->rmax, nullptr, nullptr, (cx<float> *)p.PqTp, sq, exact);
    if (!m->same_eph) launch_phases(nq, q, m->nRph, m->Rph, m->rmax, nullptr, p.PqTph, nullptr, sq, exact);
  }
  if (tcb && fork && !qs) CK(cudaEventRecord(m->ev_phase, sq));
  // phonons (FP64 eigensolve)
  if (!qs && fx && fx->dq) {
    CKS(run_fx_q(m, nq, q, *fx, p.D, sq, pa && *pa->done ? pa : nullptr));
  } else if (!qs) {
    launch_fourier_d(nq, m->nRph, p.PqTph, m->Phiw, nm * nm, p.D, sq, exact);
  }
  // The eigensolves are one long wave of FP64-bound warps that has to start on a GPU with room on every
  // SM: launched while a GEMM fills it, their blocks share the few SMs that happen to have room
  // (13,824 of 9 x 9: 6.6 ms against 2.4; 1728: 3.3 against 0.8).  So the k-side vertex starts after
  // them where it runs on the tensor cores (FP64), and they start after it where it runs on the CUDA
  // cores, which they slow down threefold (FP32: 809 us beside 9001 of 6 x 6, 284 alone); the kernels
  // after that vertex wait until they are launched (13,824 of 9 x 9 among them: 16.8 ms).
  const bool gate = fork && fx && (fx->dq || exact);
  const bool after_vertex = gate && need_B && prec != EPW_FP64;
  if (gate) CK(cudaEventRecord(m->ev_gate, sq));
  auto q_tail = [&]() {
    launch_eigh_d(nq, nm, p.D, p.w2, p.ev, m->dstatus, sq, exact);
    launch_phonon_post(nq, nm, p.w2, p.ev, m->mass, omega_min, p.omegaT,
                       prec == EPW_FP64 ? (cx<double> *)p.ET : nullptr,
                       prec == EPW_FP64 ? nullptr : (cx<float> *)p.ET, omega_out, sq);
    if (m->polar) {
      if (prec == EPW_FP64)
        launch_polar_factors<double>(m, nq, q, (const cx<double> *)p.ET, (cx<double> *)p.Cpol, sq);
      else
        launch_polar_factors<float>(m, nq, q, (const cx<float> *)p.ET, (cx<float> *)p.Cpol, sq);
    }
    if (fx && fx->pair && fx->omK)
      launch_tables64(nq, nm, p.omegaT, omega_min, fx->T, fx->omK, fx->nbT, fx->wmax, sq);
  };
  if (!after_vertex) q_tail();
  // k side (FP64): phases, H(k), eigensolve, then the k-side vertex; with a fork the
  // bands (H(k), eigensolve) run on a third stream beside the vertex GEMM, which
  // needs only the phases, and are joined before the U_k rotation
  launch_phases(nk, k, m->nRe, m->Re, m->rmax, p.PkRM, p.PkT, nullptr, st, exact_k);
  const bool fork2 = fork && need_B;
  cudaStream_t sk = st;
  if (fork2) {
    CK(cudaEventRecord(m->ev_fork2, st));
    CK(cudaStreamWaitEvent(m->aux2, m->ev_fork2, 0));
    sk = m->aux2;
  }
  launch_fourier_d(nk, m->nRe, p.PkT, m->Hw, (int)nw2, p.Hk, sk, exact_k);
  launch_eigh_d(nk, nw, p.Hk, p.epsk, p.Uk, m->dstatus, sk, exact_k);
  if (fork2) CK(cudaEventRecord(m->ev_join2, sk));
  if (need_B && nk > 0) {
    const int ncol = m->nRp * nm * (int)nw2;
    if (gate && !after_vertex) CK(cudaStreamWaitEvent(st, m->ev_gate, 0));
    if (prec == EPW_FP64) {
      CKS(run_vertex64(m, nk, k, p, fx, st));
      if (fork2) CK(cudaStreamWaitEvent(st, m->ev_join2, 0));
      launch_build_B<double>(m, nk, p.PkRM, (const cx<double> *)p.G1, p.Uk, (cx<double> *)p.Bg, (cx<double> *)p.BH,
                             st);
    } else {
      launch_cast_c64_to_c32((size_t)nk * m->nRe, p.PkRM, p.Pk32, st);
      launch_vertex32(nk, m->nRe, ncol, p.Pk32, m->gw, p.gw32, (cx<float> *)p.G1, st);
      if (after_vertex) {
        CK(cudaEventRecord(m->ev_vertex, st));
        CK(cudaStreamWaitEvent(sq, m->ev_vertex, 0));
        CK(cudaEventRecord(m->ev_gate, sq));
        q_tail();
        CK(cudaStreamWaitEvent(st, m->ev_gate, 0));
      }
      if (fork2) CK(cudaStreamWaitEvent(st, m->ev_join2, 0));
      if (p.bad) CK(cudaMemsetAsync(p.bad, 0, sizeof(int), st));
      launch_build_B<float>(m, nk, p.PkRM, (const cx<float> *)p.G1, p.Uk, (cx<float> *)p.Bg, (cx<float> *)p.BH, st,
                            p.bad);
    }
  }
  if (tcb && nk > 0 && nq > 0) {
    tc_build_b(m, nk, (const cx<float> *)p.Bg, (const cx<float> *)p.BH, *tcb, st);
    tcb->prebuilt_b = true;
    if (!qs) {
      tcb->Pq64 = m->same_eph ? p.PqTph : nullptr;
      if (fork) CK(cudaStreamWaitEvent(st, m->ev_phase, 0));
      tc_build_a(m, nq, q, *tcb, st);
      tcb->prebuilt_a = true;
    }
  }
  if (fork) {
    CK(cudaEventRecord(m->ev_join, sq));
    if (fx) fx->late = fx->late && gate;
    if (fx && fx->late)
      CK(cudaStreamWaitEvent(st, m->ev_gate, 0));  // the q phases' operands; the phonons follow
    else
      CK(cudaStreamWaitEvent(st, m->ev_join, 0));
  } else if (fx) {
    fx->late = false;
  }
  CK(cudaGetLastError());
  return EPW_OK;
}
// With fx.late: joins the q side's phonons into st (contractions that read only its operands have
// run beside its eigensolves).
static epw_status prep_join(const epw_model *m, Fx64 &fx, cudaStream_t st) {
  if (fx.late) CK(cudaStreamWaitEvent(st, m->ev_join, 0));
  fx.late = false;
  return EPW_OK;
}

epw_status epwi_check_common(const epw_model *m, int nk, const double *k, int nq, const double *q) {
  if (!m) return fail(EPW_ERR_INVALID_ARG, "null model");
  if (nk < 0 || nq < 0) return fail(EPW_ERR_INVALID_ARG, "negative nk or nq");
  if ((nk > 0 && !k) || (nq > 0 && !q)) return fail(EPW_ERR_INVALID_ARG, "null k or q");
  if ((size_t)nk * (size_t)nq > (size_t)1 << 44) return fail(EPW_ERR_INVALID_ARG, "nk*nq too large");
  int cur = -1;
  CK(cudaGetDevice(&cur));
  if (cur != m->device) return fail(EPW_ERR_INVALID_ARG, "model lives on device %d, current device is %d", m->device, cur);
  return EPW_OK;
}

epw_status epwi_check_params(const epw_params *p) {
  if (!p) return fail(EPW_ERR_INVALID_ARG, "null params");
  if (!(p->T_K >= 0.0) || !std::isfinite(p->T_K)) return fail(EPW_ERR_INVALID_ARG, "T_K must be finite and >= 0");
  if (!(p->sigma_eV > 0.0) || !std::isfinite(p->sigma_eV)) return fail(EPW_ERR_INVALID_ARG, "sigma_eV must be > 0");
  if (!(p->omega_min_eV >= 0.0)) return fail(EPW_ERR_INVALID_ARG, "omega_min_eV must be >= 0");
  if (!std::isfinite(p->EF_eV)) return fail(EPW_ERR_INVALID_ARG, "EF_eV must be finite");
  if (p->precision < EPW_FP64 || p->precision > EPW_TF32X3) return fail(EPW_ERR_INVALID_ARG, "unknown precision");
  if (p->reserved != 0) return fail(EPW_ERR_INVALID_ARG, "reserved field must be 0");
  return EPW_OK;
}

static epw_status check_common(const epw_model *m, int nk, const double *k, int nq, const double *q) {
  return epwi_check_common(m, nk, k, nq, q);
}
static epw_status check_params(const epw_params *p) { return epwi_check_params(p); }

static epw_status read_status(const epw_model *m, cudaStream_t st) {
  unsigned h[4] = {0, 0, 0, 0};
  CK(cudaMemcpyAsync(h, m->dstatus, sizeof(h), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  CK(cudaMemsetAsync(m->dstatus, 0, sizeof(h), st));
  CK(cudaStreamSynchronize(st));
  if (h[0] & EPW_DEV_NOT_CONVERGED) return fail(EPW_ERR_NOT_CONVERGED, "an eigensolve did not converge");
  if (h[0] & EPW_DEV_TIMEOUT) return fail(EPW_ERR_TIMEOUT, "a device wait ran out of its iteration budget");
  if (h[0] & EPW_DEV_BAD_SHAPE) return fail(EPW_ERR_UNSUPPORTED, "kernel met an unsupported shape");
  return EPW_OK;
}

extern "C" epw_status epw_sync(const epw_model *m, void *stream) {
  if (!m) return fail(EPW_ERR_INVALID_ARG, "null model");
  return read_status(m, (cudaStream_t)stream);
}

// ------------------------------------------------------------- linewidth
// Contraction buffer of the staged tensor-core form (per chunk of k).
static const size_t STAGED_CT_BYTES = (size_t)4 << 30;
// Buffers that grow with the k count stay within this (the larger uneven-batch systems need
// up to ~19 MB per k for g(k,Rp) U_k alone); EPW_K_SIDE_BYTES overrides it.
static const size_t K_SIDE_BYTES = (size_t)8 << 30;

// EPW_WIDE_FORM selects the wide-shape form: unset or "pair", the fused kernel on CTA pairs;
// "single", the fused kernel on single CTAs; "split", the two-kernel form.
EpwTune epwi_default_tune() {
  const char *w = getenv("EPW_WIDE_FORM");
  const char *kb = getenv("EPW_K_SIDE_BYTES");
  const size_t kside = (kb && *kb) ? (size_t)strtoull(kb, nullptr, 10) : K_SIDE_BYTES;
  const int form = !w ? TCW_FORM_PAIR
                 : strcmp(w, "split") == 0 ? TCW_FORM_SPLIT
                 : strcmp(w, "single") == 0 ? TCW_FORM_SINGLE
                                            : TCW_FORM_PAIR;
  return EpwTune{0, STAGED_CT_BYTES, form, kside, false, false, false};
}

// The buffers of one pass over nk k-points (k and output staging excluded).
static epw_status plan_linewidth_pass(Arena &A, const epw_model *m, int nk, int nq, int prec, bool sq, bool swq,
                                      const EpwTune &tune, LwPlan &L) {
  const bool tc = prec == EPW_BF16X3 || prec == EPW_TF32X3;
  const int op = prec == EPW_BF16X3 ? TC_OP_BF16 : TC_OP_TF32;
  L.sg = TcStaged{};
  L.tc = TcBuffers{};
  L.w = TcwBuffers{};
  const bool narrow = tc && tc_supported(m);
  plan_fx(A, m, nk, nq, !tune.simt64 && !narrow && fx_dq(m, nq), tune.pair64, tune.g1_64, L.fx);
  plan_prep(A, m, nk, nq, tc ? EPW_FP32 : prec, false, sq, swq, true, L.p, &L.fx);
  if (narrow) {
    CKS(tc_plan(A, m, nk, nq, op, L.tc));
    L.tc.a_block_bytes = tune.a_block_bytes;
    L.partial = nullptr;
  } else if (tc && tcw_supported(m)) {
    CKS(tcw_plan(A, m, nk, nq, op, 0, L.w, tune.wide_form));
    L.partial = nullptr;
  } else {
    if (tc) CKS(tc_staged_plan(A, m, nk, nq, op, tune.staged_ct_bytes ? tune.staged_ct_bytes : STAGED_CT_BYTES, L.sg));
    int nqb = (nq + 127) / 128;
    L.partial = A.take<double>((size_t)nk * nqb * m->nw);
  }
  return EPW_OK;
}

// k per pass: the k list runs in equal passes when the buffers that grow with nk (k-side
// bands and vertex g(k,Rp) U_k, partial sums, operands and contraction chunks) would exceed
// tune.k_side_bytes: the longest pass whose plan exceeds the plan of one k by at most that
// budget (a binary search over the plans; a staged contraction chunk is capped by its own
// budget, so it stops growing at one chunk and each pass repeats the q-side preparation only
// when the k-side buffers really do not fit).
static int k_per_pass(const epw_model *m, int nk, int nq, int prec, const EpwTune &tune) {
  if (tune.k_side_bytes == 0 || nk <= 1) return nk;
  auto bytes = [&](int nkp) -> size_t {
    Arena a{nullptr, 0, 0};
    LwPlan t;
    return plan_linewidth_pass(a, m, nkp, nq, prec, false, false, tune, t) == EPW_OK ? a.off : SIZE_MAX;
  };
  const size_t b1 = bytes(1);
  if (b1 == SIZE_MAX) return nk;
  auto fits = [&](int nkp) {
    const size_t b = bytes(nkp);
    return b != SIZE_MAX && b - b1 <= tune.k_side_bytes;
  };
  if (fits(nk)) return nk;
  int lo = 1, hi = nk;  // fits(lo), not fits(hi)
  while (hi - lo > 1) {
    const int mid = lo + (hi - lo) / 2;
    if (fits(mid))
      lo = mid;
    else
      hi = mid;
  }
  const int npass = (nk + lo - 1) / lo;
  return (nk + npass - 1) / npass;
}

epw_status epwi_plan_linewidth(Arena &A, const epw_model *m, int nk, int nq, int prec, bool sk, bool sq, bool swq,
                               bool sout, const EpwTune &tune0, LwPlan &L) {
  // the form is chosen from the whole k list, so that results do not depend on the passes
  EpwTune tune = tune0;
  tune.pair64 = !tune.simt64 && prec == EPW_FP64 && fx_pair(m, nk, nq);
  tune.g1_64 = !tune.simt64 && prec == EPW_FP64 && fx_g1(m, nk);
  L.kchunk = k_per_pass(m, nk, nq, prec, tune);
  if (!tune.simt64) {
    Arena a{nullptr, 0, 0};
    LwPlan t;
    CKS(plan_linewidth_pass(a, m, L.kchunk, nq, prec, false, false, tune, t));
    if (a.off > FX_WS_BYTES && (t.fx.dq || t.fx.g1)) {
      tune.simt64 = true;
      tune.pair64 = tune.g1_64 = false;
      L.kchunk = k_per_pass(m, nk, nq, prec, tune);
    }
  }
  double *kd = sk ? A.take<double>(3 * (size_t)nk) : nullptr;  // the whole k list, staged from the host
  CKS(plan_linewidth_pass(A, m, L.kchunk, nq, prec, sq, swq, tune, L));
  L.p.kd = kd;
  L.out_d = sout ? A.take<double>((size_t)nk * m->nw) : nullptr;
  return EPW_OK;
}

static epw_status plan_linewidth(Arena &A, const epw_model *m, int nk, int nq, int prec, bool sk, bool sq, bool swq,
                                 bool sout, LwPlan &L) {
  return epwi_plan_linewidth(A, m, nk, nq, prec, sk, sq, swq, sout, epwi_default_tune(), L);
}

// The plan of a linewidth call and its workspace; with tune.simt64 where the fixed-point forms' would not fit
// the device.
static epw_status plan_linewidth_ws(epw_model *m, int nk, int nq, int prec, bool sk, bool sq, bool swq, bool sout,
                                    EpwTune &tune, LwPlan &L) {
  for (tune = epwi_default_tune();; tune.simt64 = true) {
    Arena A{nullptr, 0, 0};
    CKS(epwi_plan_linewidth(A, m, nk, nq, prec, sk, sq, swq, sout, tune, L));
    const epw_status s = ensure_ws(m, A.off);
    if (s == EPW_ERR_OOM && (L.fx.dq || L.fx.g1)) continue;
    if (s == EPW_OK) g_err[0] = 0;
    return s;
  }
}

extern "C" epw_status epw_reserve(epw_model *m, int nk, int nq, int precision) {
  CKS(check_common(m, nk, (const double *)1, nq, (const double *)1));
  if (precision < EPW_FP64 || precision > EPW_TF32X3) return fail(EPW_ERR_INVALID_ARG, "unknown precision");
  EpwTune tune;
  LwPlan L;
  return plan_linewidth_ws(m, nk, nq, precision, true, true, true, true, tune, L);
}

// Planning by shape alone: the same plan as epw_reserve on a host-side model that holds the
// shape and no device state (the planners only compute offsets).
extern "C" epw_status epw_plan_linewidth(int nw, int nat, int nRe, int nRp, int nRph, int same_ep, int same_eph,
                                         int polar, int nk, int nq, int precision, size_t *ws_bytes,
                                         int *k_per_pass) {
  g_err[0] = 0;
  if (nw < 1 || nw > EPW_MAX_NW) return fail(EPW_ERR_INVALID_ARG, "nw=%d outside [1,%d]", nw, EPW_MAX_NW);
  if (nat < 1 || 3 * nat > EPW_MAX_MODES) return fail(EPW_ERR_INVALID_ARG, "3*nat=%d outside [3,%d]", 3 * nat, EPW_MAX_MODES);
  if (nRe < 1 || nRp < 1 || nRph < 1) return fail(EPW_ERR_INVALID_ARG, "empty R set");
  if ((same_ep && nRe != nRp) || (same_eph && nRe != nRph))
    return fail(EPW_ERR_INVALID_ARG, "identical R sets need equal sizes");
  if (nk < 1 || nq < 1) return fail(EPW_ERR_INVALID_ARG, "nk and nq must be positive");
  if ((size_t)nk * (size_t)nq > (size_t)1 << 44) return fail(EPW_ERR_INVALID_ARG, "nk*nq too large");
  if (precision < EPW_FP64 || precision > EPW_TF32X3) return fail(EPW_ERR_INVALID_ARG, "unknown precision");
  epw_model m{};
  m.device = -1;
  m.nw = nw;
  m.nat = nat;
  m.nm = 3 * nat;
  m.nRe = nRe;
  m.nRp = nRp;
  m.nRph = nRph;
  m.same_ep = same_ep ? 1 : 0;
  m.same_eph = same_eph ? 1 : 0;
  m.polar = polar ? 1 : 0;
  Arena A{nullptr, 0, 0};
  LwPlan L;
  CKS(plan_linewidth(A, &m, nk, nq, precision, true, true, true, true, L));
  const bool tcp = precision == EPW_BF16X3 || precision == EPW_TF32X3;
  if (tcp && !L.tc.ok && !L.sg.ok && !L.w.ok)
    return fail(EPW_ERR_UNSUPPORTED, "no tensor-core form for nw=%d, 3nat=%d", nw, 3 * nat);
  if (ws_bytes) *ws_bytes = A.off;
  if (k_per_pass) *k_per_pass = L.kchunk;
  return EPW_OK;
}

extern "C" epw_status epw_linewidth(const epw_model *mc, int nk, const double *k, int nq, const double *q,
                                    const double *wq, const epw_params *par, double *imsigma, void *stream) {
  g_err[0] = 0;
  epw_model *m = const_cast<epw_model *>(mc);
  CKS(check_common(m, nk, k, nq, q));
  CKS(check_params(par));
  if (nk > 0 && !imsigma) return fail(EPW_ERR_INVALID_ARG, "null imsigma");
  cudaStream_t st = (cudaStream_t)stream;
  if (nk == 0) return EPW_OK;
  const int prec = par->precision;
  const bool sk = !is_device_ptr(k), sq = nq > 0 && !is_device_ptr(q), swq = wq && nq > 0 && !is_device_ptr(wq);
  const bool sout = !is_device_ptr(imsigma);
  if (nq == 0) {
    if (sout) {
      std::memset(imsigma, 0, sizeof(double) * (size_t)nk * m->nw);
      return EPW_OK;
    }
    CK(cudaMemsetAsync(imsigma, 0, sizeof(double) * (size_t)nk * m->nw, st));
    return EPW_OK;
  }
  EpwTune tune;
  LwPlan L;
  CKS(plan_linewidth_ws(m, nk, nq, prec, sk, sq, swq, sout, tune, L));
  Arena A{(char *)m->ws, m->ws_bytes, 0};
  CKS(epwi_plan_linewidth(A, m, nk, nq, prec, sk, sq, swq, sout, tune, L));
  Prep &p = L.p;
  const double *kd = k, *qd = q, *wqd = wq;
  if (sk) {
    CK(cudaMemcpyAsync(p.kd, k, sizeof(double) * 3 * nk, cudaMemcpyHostToDevice, st));
    kd = p.kd;
  }
  if (sq) {
    CK(cudaMemcpyAsync(p.qd, q, sizeof(double) * 3 * nq, cudaMemcpyHostToDevice, st));
    qd = p.qd;
  }
  if (swq) {
    CK(cudaMemcpyAsync(p.wqd, wq, sizeof(double) * nq, cudaMemcpyHostToDevice, st));
    wqd = p.wqd;
  }
  double *out = sout ? L.out_d : imsigma;
  CKS(epwi_linewidth_exec(m, nk, kd, nq, qd, wqd, par, L, out, st));
  if (sout) {
    CK(cudaMemcpyAsync(imsigma, out, sizeof(double) * (size_t)nk * m->nw, cudaMemcpyDeviceToHost, st));
  }
  if (sk || sq || swq || sout) return read_status(m, st);
  return EPW_OK;
}

static epw_status linewidth_pass(epw_model *m, int nk, const double *kd, int nq, const double *qd, const double *wqd,
                                 const epw_params *par, LwPlan &L, double *out, cudaStream_t st);

epw_status epwi_linewidth_exec(epw_model *m, int nk, const double *kd, int nq, const double *qd, const double *wqd,
                               const epw_params *par, LwPlan &L, double *out, cudaStream_t st) {
  const int kc = L.kchunk > 0 ? std::min(L.kchunk, nk) : nk;
  for (int k0 = 0; k0 < nk; k0 += kc)
    CKS(linewidth_pass(m, std::min(kc, nk - k0), kd + 3 * (size_t)k0, nq, qd, wqd, par, L,
                       out + (size_t)k0 * m->nw, st));
  return EPW_OK;
}

// One pass over nk <= L.kchunk k-points (q side recomputed per pass: it costs a small
// fraction of the pass's pairs).
static epw_status linewidth_pass(epw_model *m, int nk, const double *kd, int nq, const double *qd, const double *wqd,
                                 const epw_params *par, LwPlan &L, double *out, cudaStream_t st) {
  const int prec = par->precision;
  Prep &p = L.p;
  const bool tcp = prec == EPW_BF16X3 || prec == EPW_TF32X3;
  if (tcp && !L.tc.ok && !L.sg.ok && !L.w.ok)
    return fail(EPW_ERR_UNSUPPORTED, "no tensor-core form for nw=%d, 3nat=%d", m->nw, m->nm);
  if (tcp && L.tc.ok) {
    CKS(run_prep(m, nk, kd, nq, qd, EPW_FP32, par->omega_min_eV, true, p, nullptr, st, true, &L.tc));
    L.tc.Cpol = m->polar ? (const float2 *)p.Cpol : nullptr;
    L.tc.Uk64 = p.Uk;
    L.tc.Pq64 = m->same_eph ? p.PqTph : nullptr;
    epw_status s = tc_linewidth(m, nk, kd, nq, qd, wqd, par, p.PkRM, p.epsk, p.Uk, p.omegaT, (const cx<float> *)p.ET,
                                (const cx<float> *)p.Bg, (const cx<float> *)p.BH, L.tc, out, st);
    if (s != EPW_OK) return fail(s, "tensor-core path: %s", g_err[0] ? g_err : "unsupported shape");
  } else if (tcp && L.w.ok) {
    // wide-shape fused form: per chunk of k, the H(k+q) eigensolve kernel and the vertex kernel
    const PhaseA pa{L.w.op, L.w.kpad, L.w.Ahi, L.w.Alo, &L.w.a_done};
    CKS(run_prep(m, nk, kd, nq, qd, EPW_FP32, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &L.fx, &pa));
    epw_status s = tcw_linewidth(m, nk, nq, qd, wqd, par, p.epsk, p.omegaT, (const cx<float> *)p.ET,
                                 (const cx<float> *)p.Bg, (const cx<float> *)p.BH, m->same_eph ? p.PqTph : nullptr,
                                 p.Uk, m->polar ? (const float2 *)p.Cpol : nullptr, L.w, out, st);
    if (s != EPW_OK) return fail(s, "wide tensor-core path: %s", g_err[0] ? g_err : "launch failed");
  } else if (tcp) {
    // staged tensor-core form: contraction per chunk of k on the tensor cores, per-pair work from HBM
    const PhaseA pa = staged_a(m, L.sg);
    L.fx.late = true;
    CKS(run_prep(m, nk, kd, nq, qd, EPW_FP32, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &L.fx, &pa));
    L.sg.Pq64 = m->same_eph ? p.PqTph : nullptr;
    CKS(tc_staged_phases(m, nq, qd, L.sg, st));
    epw_timing_begin(m, st);
    for (int k0 = 0; k0 < nk; k0 += L.sg.kc) {
      const int kc = std::min(L.sg.kc, nk - k0);
      epw_status s = tc_staged_contract(m, k0, kc, nq, (const cx<float> *)p.Bg, (const cx<float> *)p.BH, L.sg, st);
      if (s != EPW_OK) return fail(s, "staged tensor-core contraction failed");
      CKS(prep_join(m, L.fx, st));
      PairArgs a;
      std::memset(&a, 0, sizeof(a));
      a.nk = kc;
      a.nq = nq;
      a.nw = m->nw;
      a.nm = m->nm;
      a.nRe = m->nRe;
      a.nRp = m->nRp;
      a.k0 = k0;
      a.ET = p.ET;
      a.omegaT = p.omegaT;
      a.eps_k = p.epsk;
      a.wq = wqd;
      a.T = par->T_K;
      a.EF = par->EF_eV;
      a.sigma = par->sigma_eV;
      a.omega_min = par->omega_min_eV;
      a.partial = L.partial;
      a.dstatus = m->dstatus;
      a.Cpol = m->polar ? p.Cpol : nullptr;
      a.Uk = p.Uk;
      a.Cq = L.sg.Ct;
      a.ldc = L.sg.pair_ld();
      a.cpk = L.sg.cpk;
      s = launch_pair_staged(a, 0, st);
      if (s != EPW_OK) return fail(s, "no staged per-pair kernel for nw=%d, 3nat=%d", m->nw, m->nm);
    }
    epw_timing_end(m, st);
    launch_finalize(nk, (nq + 127) / 128, m->nw, L.partial, out, st);
  } else if (L.fx.pair) {
    // FP64: the contractions of a chunk of k as digit planes on the tensor cores, per-pair work in FP64
    L.fx.T = par->T_K;
    L.fx.late = true;
    CKS(run_prep(m, nk, kd, nq, qd, prec, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &L.fx));
    epw_timing_begin(m, st);
    for (int k0 = 0; k0 < nk; k0 += L.fx.kc) {
      const int kc = std::min(L.fx.kc, nk - k0);
      CKS(run_fx_contract(m, k0, kc, p, L.fx, st));
      CKS(prep_join(m, L.fx, st));
      Pair64Args a = pair64_args(m, k0, kc, nq, wqd, par, p, L.fx);
      a.partial = L.partial;
      epw_status s = launch_lw64(a, st);
      if (s != EPW_OK) return fail(s, "FP64 per-pair kernel failed for nw=%d, 3nat=%d", m->nw, m->nm);
    }
    epw_timing_end(m, st);
    launch_finalize(nk, (nq + 127) / 128, m->nw, L.partial, out, st);
  } else {
    CKS(run_prep(m, nk, kd, nq, qd, prec, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &L.fx));
    PairArgs a;
    std::memset(&a, 0, sizeof(a));
    a.nk = nk;
    a.nq = nq;
    a.nw = m->nw;
    a.nm = m->nm;
    a.nRe = m->nRe;
    a.nRp = m->nRp;
    a.k0 = 0;
    a.PqTe = p.PqTe;
    a.PqTp = p.PqTp;
    a.BH = p.BH;
    a.Bg = p.Bg;
    a.ET = p.ET;
    a.omegaT = p.omegaT;
    a.eps_k = p.epsk;
    a.wq = wqd;
    a.T = par->T_K;
    a.EF = par->EF_eV;
    a.sigma = par->sigma_eV;
    a.omega_min = par->omega_min_eV;
    a.partial = L.partial;
    a.dstatus = m->dstatus;
    a.Cpol = m->polar ? p.Cpol : nullptr;
    a.Uk = p.Uk;
    epw_timing_begin(m, st);
    epw_status s = prec == EPW_FP64 ? launch_pair<double>(a, 0, st) : launch_pair<float>(a, 0, st);
    epw_timing_end(m, st);
    if (s != EPW_OK) return fail(s, "no per-pair kernel for nw=%d, 3nat=%d in this precision", m->nw, m->nm);
    launch_finalize(nk, (nq + 127) / 128, m->nw, L.partial, out, st);
  }
  CK(cudaGetLastError());
  return EPW_OK;
}

// ---------------------------------------------------------------- interp
extern "C" epw_status epw_interp_g(const epw_model *mc, int nk, const double *k, int nq, const double *q,
                                   int precision, double omega_min, double *eps_k, double *eps_kq, double *omega,
                                   double *g, void *stream) {
  g_err[0] = 0;
  epw_model *m = const_cast<epw_model *>(mc);
  CKS(check_common(m, nk, k, nq, q));
  if (precision < EPW_FP64 || precision > EPW_TF32X3) return fail(EPW_ERR_INVALID_ARG, "unknown precision");
  const bool tcp = precision == EPW_BF16X3 || precision == EPW_TF32X3;
  const bool tc = tcp && tc_supported(m), staged = tcp && tc_staged_supported(m);
  if (tcp && !tc && !staged)
    return fail(EPW_ERR_UNSUPPORTED, "no tensor-core form for nw=%d, 3nat=%d", m->nw, m->nm);
  const int wprec = tcp ? EPW_FP32 : precision;  // precision of the shared preparation
  if (!(omega_min >= 0.0)) return fail(EPW_ERR_INVALID_ARG, "omega_min must be >= 0");
  cudaStream_t st = (cudaStream_t)stream;
  if (nk == 0 && nq == 0) return EPW_OK;
  const bool sk = nk > 0 && !is_device_ptr(k), sq = nq > 0 && !is_device_ptr(q);
  const size_t nw = m->nw, nm = m->nm;
  const bool s_ek = eps_k && !is_device_ptr(eps_k), s_ekq = eps_kq && !is_device_ptr(eps_kq);
  const bool s_om = omega && !is_device_ptr(omega), s_g = g && !is_device_ptr(g);
  TcBuffers tcb;
  TcStaged sg{};
  Fx64 fx;
  const bool want_pairs = nk > 0 && nq > 0 && (eps_kq || g);
  bool need_B = true;
  cx<double> *Hq = nullptr, *Uq = nullptr;
  double *wkq = nullptr;
  Prep p;
  double *ekd, *ekqd, *omd, *gd;
  bool fx_on = true;
  auto plan = [&](Arena &A) -> epw_status {
    const size_t per = (size_t)nq * nw * (40 * nw + 8);  // H(k+q) twice, its eigenvectors and eigenvalues
    plan_fx(A, m, nk > 0 ? nk : 1, nq > 0 ? nq : 1, fx_on && precision == EPW_FP64 && fx_dq(m, nq),
            fx_on && precision == EPW_FP64 && want_pairs && fx_pair(m, nk, nq),
            fx_on && precision == EPW_FP64 && nk > 0 && g && fx_g1(m, nk), fx, per);
    fx.exact = precision != EPW_FP64;
    if (fx.pair) {
      const size_t np = (size_t)nq * fx.kc;
      fx.omK = nullptr;  // (no tables: no occupations here)
      fx.Hq = A.take<double>(np * nw * nw);
      Hq = A.take<cx<double>>(np * nw * nw);
      Uq = A.take<cx<double>>(np * nw * nw);
      wkq = A.take<double>(np * nw);
    }
    need_B = nk > 0 && (g || !fx.pair);  // bands alone need no vertex
    plan_prep(A, m, nk > 0 ? nk : 1, nq > 0 ? nq : 1, wprec, sk, sq, false, need_B || nk == 0, p, &fx);
    ekd = s_ek ? A.take<double>((size_t)nk * nw) : eps_k;
    ekqd = s_ekq ? A.take<double>((size_t)nk * nq * nw) : eps_kq;
    omd = s_om ? A.take<double>((size_t)nq * nm) : omega;
    gd = s_g ? (double *)A.take<cx<double>>((size_t)nk * nq * nm * nw * nw) : g;
    const int op = precision == EPW_BF16X3 ? TC_OP_BF16 : TC_OP_TF32;
    if (tc) return tc_plan(A, m, nk > 0 ? nk : 1, nq > 0 ? nq : 1, op, tcb);
    if (staged) return tc_staged_plan(A, m, nk > 0 ? nk : 1, nq > 0 ? nq : 1, op, STAGED_CT_BYTES, sg);
    return EPW_OK;
  };
  Arena A;
  CKS(plan_ws(m, A, fx, fx_on, plan));
  const double *kd = k, *qd = q;
  if (sk) {
    CK(cudaMemcpyAsync(p.kd, k, sizeof(double) * 3 * nk, cudaMemcpyHostToDevice, st));
    kd = p.kd;
  }
  if (sq) {
    CK(cudaMemcpyAsync(p.qd, q, sizeof(double) * 3 * nq, cudaMemcpyHostToDevice, st));
    qd = p.qd;
  }
  fx.late = fx.pair;
  CKS(run_prep(m, nk, kd, nq, qd, wprec, omega_min, need_B, p, omd, st, true, tc ? &tcb : nullptr, &fx));
  if (ekd && nk > 0) CK(cudaMemcpyAsync(ekd, p.epsk, sizeof(double) * nk * nw, cudaMemcpyDeviceToDevice, st));
  if (tc && nk > 0 && nq > 0 && (ekqd || gd)) {
    tcb.Cpol = m->polar ? (const float2 *)p.Cpol : nullptr;
    tcb.Uk64 = p.Uk;
    tcb.Pq64 = m->same_eph ? p.PqTph : nullptr;
    epw_status s = tc_interp(m, nk, nq, qd, omega_min, p.epsk, p.omegaT, (const cx<float> *)p.ET,
                             (const cx<float> *)p.Bg, (const cx<float> *)p.BH, tcb, ekqd, gd, st);
    if (s != EPW_OK) return fail(s, "tensor-core interpolation failed");
  } else if (staged && nk > 0 && nq > 0 && (ekqd || gd)) {
    sg.Pq64 = m->same_eph ? p.PqTph : nullptr;
    CKS(tc_staged_phases(m, nq, qd, sg, st));
    for (int k0 = 0; k0 < nk; k0 += sg.kc) {
      const int kc = std::min(sg.kc, nk - k0);
      epw_status s = tc_staged_contract(m, k0, kc, nq, (const cx<float> *)p.Bg, (const cx<float> *)p.BH, sg, st);
      if (s != EPW_OK) return fail(s, "staged tensor-core contraction failed");
      PairArgs a;
      std::memset(&a, 0, sizeof(a));
      a.nk = kc;
      a.nq = nq;
      a.nw = m->nw;
      a.nm = m->nm;
      a.nRe = m->nRe;
      a.nRp = m->nRp;
      a.k0 = k0;
      a.ET = p.ET;
      a.omegaT = p.omegaT;
      a.eps_k = p.epsk;
      a.omega_min = omega_min;
      a.sigma = 1.0;
      a.eps_kq = ekqd;
      a.gout = (cx<double> *)gd;
      a.dstatus = m->dstatus;
      a.Cpol = m->polar ? p.Cpol : nullptr;
      a.Uk = p.Uk;
      a.Cq = sg.Ct;
      a.ldc = sg.pair_ld();
      a.cpk = sg.cpk;
      s = launch_pair_staged(a, 1, st);
      if (s != EPW_OK) return fail(s, "no staged per-pair kernel for nw=%d, 3nat=%d", m->nw, m->nm);
    }
  } else if (fx.pair) {
    // FP64: H(k+q) as matrices, the batched Jacobi (the eigenvectors' phases are its), then g
    for (int k0 = 0; k0 < nk; k0 += fx.kc) {
      const int kc = std::min(fx.kc, nk - k0);
      CKS(run_fx_hmat(m, k0, kc, p, fx, st));
      fx_unpack_hermitian(nq * kc, m->nw, fx.Hq, Hq, st);
      launch_eigh_d(nq * kc, m->nw, Hq, wkq, Uq, m->dstatus, st);
      if (gd) CKS(run_fx_vertex(m, k0, kc, p, fx, st));
      CKS(prep_join(m, fx, st));
      epw_params par{0.0, 0.0, 1.0, omega_min, precision, 0};
      Pair64Args a = pair64_args(m, k0, kc, nq, nullptr, &par, p, fx);
      a.wkq = wkq;
      a.Ukq = Uq;
      a.eps_kq = ekqd;
      a.gout = (cx<double> *)gd;
      epw_status s = launch_g64(a, st);
      if (s != EPW_OK) return fail(s, "FP64 vertex kernel failed");
    }
  } else if (nk > 0 && nq > 0 && (ekqd || gd)) {
    PairArgs a;
    std::memset(&a, 0, sizeof(a));
    a.nk = nk;
    a.nq = nq;
    a.nw = m->nw;
    a.nm = m->nm;
    a.nRe = m->nRe;
    a.nRp = m->nRp;
    a.PqTe = p.PqTe;
    a.PqTp = p.PqTp;
    a.BH = p.BH;
    a.Bg = p.Bg;
    a.ET = p.ET;
    a.omegaT = p.omegaT;
    a.eps_k = p.epsk;
    a.omega_min = omega_min;
    a.sigma = 1.0;
    a.eps_kq = ekqd;
    a.gout = (cx<double> *)gd;
    a.dstatus = m->dstatus;
    a.Cpol = m->polar ? p.Cpol : nullptr;
    a.Uk = p.Uk;
    epw_status s = precision == EPW_FP64 ? launch_pair<double>(a, 1, st) : launch_pair<float>(a, 1, st);
    if (s != EPW_OK) return fail(s, "no per-pair kernel for nw=%d, 3nat=%d", m->nw, m->nm);
  }
  CK(cudaGetLastError());
  if (s_ek) CK(cudaMemcpyAsync(eps_k, ekd, sizeof(double) * nk * nw, cudaMemcpyDeviceToHost, st));
  if (s_ekq) CK(cudaMemcpyAsync(eps_kq, ekqd, sizeof(double) * nk * nq * nw, cudaMemcpyDeviceToHost, st));
  if (s_om) CK(cudaMemcpyAsync(omega, omd, sizeof(double) * nq * nm, cudaMemcpyDeviceToHost, st));
  if (s_g) CK(cudaMemcpyAsync(g, gd, sizeof(cx<double>) * nk * nq * nm * nw * nw, cudaMemcpyDeviceToHost, st));
  if (sk || sq || s_ek || s_ekq || s_om || s_g) return read_status(m, st);
  return EPW_OK;
}

// -------------------------------------------------------------- backward
extern "C" epw_status epw_linewidth_backward(const epw_model *mc, int nk, const double *k, int nq, const double *q,
                                             const double *wq, const epw_params *par, const double *cot, double *dg,
                                             double *dT, double *dEF, void *stream) {
  g_err[0] = 0;
  epw_model *m = const_cast<epw_model *>(mc);
  CKS(check_common(m, nk, k, nq, q));
  CKS(check_params(par));
  if (!(par->T_K > 0.0)) return fail(EPW_ERR_INVALID_ARG, "the adjoint needs T_K > 0");
  if (nk > 0 && !cot) return fail(EPW_ERR_INVALID_ARG, "null grad_imsigma");
  const int prec = par->precision >= EPW_BF16X3 ? EPW_FP32 : par->precision;
  // tensor-core adjoint (TF32 split) for shapes the fused kernel serves (Re == Rp: its
  // q-contraction of the adjoint runs over one R set)
  const bool tcp = par->precision == EPW_BF16X3 || par->precision == EPW_TF32X3;
  const bool tcb = tcp && m->same_ep && tc_supported(m);
  // other shapes, and Re != Rp: the forward contraction of the recompute staged on the
  // tensor cores (its K layout carries both R sets)
  const bool staged = tcp && !tcb && m->nw <= 18 && m->nm <= 18;
  if (tcp && !tcb && !staged)
    return fail(EPW_ERR_UNSUPPORTED, "no tensor-core form for nw=%d, 3nat=%d", m->nw, m->nm);
  if (m->nw > 8 || m->nm > 9)
    return fail(EPW_ERR_UNSUPPORTED, "the adjoint has no kernel for nw=%d, 3nat=%d (at most 8 and 9)", m->nw, m->nm);
  cudaStream_t st = (cudaStream_t)stream;
  const size_t nw2 = (size_t)m->nw * m->nw, per = (size_t)m->nm * nw2;
  const size_t ng = (size_t)m->nRe * m->nRp * per;
  const bool sk = nk > 0 && !is_device_ptr(k), sq = nq > 0 && !is_device_ptr(q);
  const bool swq = wq && nq > 0 && !is_device_ptr(wq), scot = nk > 0 && !is_device_ptr(cot);
  const bool sdg = dg && !is_device_ptr(dg), sdT = dT && !is_device_ptr(dT), sdE = dEF && !is_device_ptr(dEF);
  const size_t sR = rsize(prec);
  bool fx_on = true, pair64 = false;
  // k chunk so that the per-chunk adjoint buffers stay near 1 GiB
  size_t per_k = (size_t)nq * per * sR + 2 * (size_t)m->nRp * per * sR;
  int nkc = (int)std::max<size_t>(1, std::min<size_t>((size_t)std::max(nk, 1), ((size_t)1 << 30) / std::max<size_t>(per_k, 1)));
  const int nqb = (nq + 127) / 128;
  struct B {
    Prep p;
    double *cotd, *xbar, *Bbar, *G1bar, *gwbar, *pT, *pE, *sc, *dgd;
    TcBuffers tc;
    TcBwdBuffers tw;
    TcStaged sg;
    TcBwdBuffers sw;  // staged shapes: the q contraction of Xbar on the tensor cores
    // FP64 in fixed point: Xbar's columns and the conjugate phases of Rp over q, the rotated sums and
    // the conjugate phases of Re over k, the gradient [nRp 3nat nw^2][nRe]
    Fx64 fx;
    FxOp Xq, Pq, Gk, Pk;
    cx<double> *xb64, *G1b, *gT;
    double *Bq;
  } b;
  b.sg = TcStaged{};
  auto plan = [&](Arena &A) -> epw_status {
    const int kpq = fx_kpad(nq);
    pair64 = fx_on && prec == EPW_FP64 && nk > 0 && nq > 0 && fx_pair(m, nk, nq);
    plan_fx(A, m, nk > 0 ? nk : 1, nq > 0 ? nq : 1, fx_on && prec == EPW_FP64 && fx_dq(m, nq), pair64,
            fx_on && prec == EPW_FP64 && nk > 0 && fx_g1(m, nk), b.fx,
            per * ((size_t)nq * 16 + 2 * FX_S * (size_t)kpq + 16 * (size_t)fx_splits(kpq) * m->nRp + 16 * (size_t)m->nRp),
            FX_KMAX / 2);
    b.fx.exact = prec != EPW_FP64;
    plan_prep(A, m, nk > 0 ? nk : 1, nq > 0 ? nq : 1, prec, sk, sq, swq, true, b.p, &b.fx);
    if (staged) b.p.bad = A.take<int>(1);
    b.cotd = scot ? A.take<double>((size_t)nk * m->nw) : (double *)cot;
    if (pair64) {
      const size_t kc = b.fx.kc, kpk = fx_kpad((int)kc);
      b.xb64 = A.take<cx<double>>(kc * per * nq);
      b.Xq = fx_plan(A, kc * per, kpq, true);
      b.Pq = fx_plan(A, 2 * (size_t)m->nRp, kpq, false);
      b.Bq = A.take<double>((size_t)fx_splits(kpq) * kc * per * 2 * m->nRp);
      b.G1b = A.take<cx<double>>((size_t)m->nRp * per * kc);
      b.Gk = fx_plan(A, m->nRp * per, (int)kpk, true);
      b.Pk = fx_plan(A, 2 * (size_t)m->nRe, (int)kpk, false);
      b.gT = A.take<cx<double>>(ng);
      b.pT = A.take<double>(kc * nqb);
      b.pE = A.take<double>(kc * nqb);
      b.gwbar = nullptr;
      b.sc = A.take<double>(2);
      b.dgd = sdg ? A.take<double>(2 * ng) : dg;
      return EPW_OK;
    }
    if (tcb) {
      b.xbar = b.Bbar = b.G1bar = b.pT = b.pE = nullptr;
      CKS(tc_bwd_plan(A, m, nk > 0 ? nk : 1, nq > 0 ? nq : 1, b.tc, b.tw));
    } else {
      if (staged) {
        CKS(tc_staged_plan(A, m, nk > 0 ? nk : 1, nq > 0 ? nq : 1,
                           par->precision == EPW_BF16X3 ? TC_OP_BF16 : TC_OP_TF32, (size_t)2 << 30, b.sg, true));
        nkc = std::min(nkc, b.sg.kc);
        CKS(tc_sbwd_plan(A, m, nq > 0 ? nq : 1, nkc, b.sw));
      }
      b.xbar = (double *)A.take<char>(sR * (size_t)nq * nkc * per);
      b.Bbar = (double *)A.take<char>(sR * (size_t)m->nRp * nkc * per);
      b.G1bar = (double *)A.take<char>(sR * (size_t)m->nRp * nkc * per);
      b.pT = A.take<double>((size_t)nkc * nqb);
      b.pE = A.take<double>((size_t)nkc * nqb);
    }
    b.gwbar = (double *)A.take<char>(sR * ng);
    b.sc = A.take<double>(2);
    b.dgd = sdg ? A.take<double>(2 * ng) : dg;
    return EPW_OK;
  };
  Arena A;
  CKS(plan_ws(m, A, b.fx, fx_on, plan));
  Prep &p = b.p;
  const double *kd = k, *qd = q, *wqd = wq;
  if (sk) {
    CK(cudaMemcpyAsync(p.kd, k, sizeof(double) * 3 * nk, cudaMemcpyHostToDevice, st));
    kd = p.kd;
  }
  if (sq) {
    CK(cudaMemcpyAsync(p.qd, q, sizeof(double) * 3 * nq, cudaMemcpyHostToDevice, st));
    qd = p.qd;
  }
  if (swq) {
    CK(cudaMemcpyAsync(p.wqd, wq, sizeof(double) * nq, cudaMemcpyHostToDevice, st));
    wqd = p.wqd;
  }
  if (scot) CK(cudaMemcpyAsync(b.cotd, cot, sizeof(double) * nk * m->nw, cudaMemcpyHostToDevice, st));
  CK(cudaMemsetAsync(b.sc, 0, 2 * sizeof(double), st));
  if (!pair64) CK(cudaMemsetAsync(b.gwbar, 0, sR * ng, st));
  if (pair64) {
    b.fx.T = par->T_K;
    b.fx.late = true;
    CKS(run_prep(m, nk, kd, nq, qd, prec, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &b.fx));
    if (b.dgd) fx_phases_conj(nq, qd, m->nRp, m->Rp, b.Pq, st);
    const int splits = fx_splits(b.Xq.kpad);
    for (int k0 = 0; k0 < nk; k0 += b.fx.kc) {
      const int kc = std::min(b.fx.kc, nk - k0);
      CKS(run_fx_contract(m, k0, kc, p, b.fx, st));
      CKS(prep_join(m, b.fx, st));
      CK(cudaMemsetAsync(b.xb64, 0, sizeof(cx<double>) * kc * per * nq, st));
      Pair64Args a = pair64_args(m, k0, kc, nq, wqd, par, p, b.fx);
      a.cot = b.cotd;
      a.xbar = (double2 *)b.xb64;
      a.partialT = b.pT;
      a.partialE = b.pE;
      epw_status s = launch_adj64(a, st);
      if (s != EPW_OK) return fail(s, "no FP64 adjoint kernel for nw=%d, 3nat=%d", m->nw, m->nm);
      launch_sum_scalar(kc * nqb, b.pT, 1.0, b.sc, st);
      launch_sum_scalar(kc * nqb, b.pE, 1.0, b.sc + 1, st);
      if (!b.dgd) continue;
      // sum over q of conj(P_q(Rp)) Xbar, U_k^dagger, then the sum over k of conj(P_k(Re))
      FxOp xq = b.Xq, gk = b.Gk, pk = b.Pk;
      xq.rows = kc * (int)per;
      const size_t stride = (size_t)xq.rows * 2 * m->nRp;
      fx_rows(xq.rows, nq, nq, b.xb64, xq, st);
      CKS(fx_gemm_f64(xq, b.Pq, fx_bits(std::min(nq, FX_KMAX / 2)), b.Bq, 2 * (size_t)m->nRp, m->dstatus, st, false,
                      stride));
      launch_adj_rotate64(kc, k0, m->nRp, m->nm, m->nw, splits, stride, b.Bq, p.Uk, b.G1b, st);
      gk.kpad = pk.kpad = fx_kpad(kc);
      fx_rows(m->nRp * per, kc, kc, b.G1b, gk, st);
      fx_phases_conj(kc, kd + 3 * (size_t)k0, m->nRe, m->Re, pk, st);
      CKS(fx_gemm_f64(gk, pk, fx_bits(kc), (double *)b.gT, 2 * (size_t)m->nRe, m->dstatus, st,
                      k0 > 0));
    }
  } else if (nk > 0 && nq > 0 && tcb) {
    CKS(run_prep(m, nk, kd, nq, qd, EPW_FP32, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &b.fx));
    b.tc.Cpol = m->polar ? (const float2 *)p.Cpol : nullptr;
    b.tc.Uk64 = p.Uk;
    b.tc.Pq64 = m->same_eph ? p.PqTph : nullptr;
    epw_status s = tc_linewidth_backward(m, nk, nq, qd, wqd, par, p.epsk, p.Uk, p.Pk32, p.omegaT,
                                         (const cx<float> *)p.ET, (const cx<float> *)p.Bg, (const cx<float> *)p.BH,
                                         b.cotd, b.tc, b.tw, (cx<float> *)b.gwbar, b.sc, st);
    if (s != EPW_OK) return fail(s, "tensor-core adjoint failed");
  } else if (nk > 0 && nq > 0) {
    b.fx.late = staged;
    CKS(run_prep(m, nk, kd, nq, qd, prec, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &b.fx));
    b.sg.Pq64 = m->same_eph ? p.PqTph : nullptr;
    if (staged) {
      CKS(tc_staged_phases(m, nq, qd, b.sg, st));
      CKS(tc_sbwd_phases(m, nq, qd, b.sw, st));
    }
    for (int k0 = 0; k0 < nk; k0 += nkc) {
      const int kc = std::min(nkc, nk - k0);
      if (staged) {
        epw_status s = tc_staged_contract(m, k0, kc, nq, (const cx<float> *)p.Bg, (const cx<float> *)p.BH, b.sg, st);
        if (s != EPW_OK) return fail(s, "staged tensor-core contraction failed");
        CKS(prep_join(m, b.fx, st));
      }
      PairArgs a;
      std::memset(&a, 0, sizeof(a));
      a.nk = nk;
      a.nq = nq;
      a.nw = m->nw;
      a.nm = m->nm;
      a.nRe = m->nRe;
      a.nRp = m->nRp;
      a.k0 = k0;
      a.PqTe = p.PqTe;
      a.PqTp = p.PqTp;
      a.BH = p.BH;
      a.Bg = p.Bg;
      a.ET = p.ET;
      a.omegaT = p.omegaT;
      a.eps_k = p.epsk;
      a.wq = wqd;
      a.T = par->T_K;
      a.EF = par->EF_eV;
      a.sigma = par->sigma_eV;
      a.omega_min = par->omega_min_eV;
      a.cot = b.cotd;
      a.xbar = b.xbar;
      a.partialT = b.pT;
      a.partialE = b.pE;
      a.nkc = kc;
      a.dstatus = m->dstatus;
      a.Cpol = m->polar ? p.Cpol : nullptr;
      a.Uk = p.Uk;
      if (staged) {
        a.Cq = b.sg.Ct;
        a.ldc = b.sg.pair_ld();
        a.cpk = b.sg.cpk;
        a.bad = p.bad;
      }
      if (staged) CK(cudaMemsetAsync(b.xbar, 0, sR * (size_t)nq * kc * per, st));
      epw_status s = staged ? launch_adj_staged(a, st)
                            : prec == EPW_FP64 ? launch_pair<double>(a, 2, st) : launch_pair<float>(a, 2, st);
      if (s != EPW_OK) return fail(s, "no per-pair kernel for nw=%d, 3nat=%d", m->nw, m->nm);
      launch_sum_scalar(kc * nqb, b.pT, 1.0, b.sc, st);
      launch_sum_scalar(kc * nqb, b.pE, 1.0, b.sc + 1, st);
      const int ncol = kc * (int)per;
      const int ncol2 = m->nRp * (int)per;
      if (prec == EPW_FP64) {
        launch_cgemm<double>(m->nRp, ncol, nq, (const cx<double> *)p.PqTp, nq, false, true,
                             (const cx<double> *)b.xbar, ncol, (cx<double> *)b.Bbar, ncol, false, st);
        launch_bg_adjoint_rotate_k0<double>(kc, k0, m->nRp, m->nm, m->nw, (const cx<double> *)b.Bbar, p.Uk,
                                            (cx<double> *)b.G1bar, st);
        launch_cgemm<double>(m->nRe, ncol2, kc, p.PkRM + (size_t)k0 * m->nRe, m->nRe, true, true,
                             (const cx<double> *)b.G1bar, ncol2, (cx<double> *)b.gwbar, ncol2, true, st);
      } else {
        if (staged) {
          epw_status s = tc_sbwd_contract(m, kc, nq, (const cx<float> *)b.xbar, b.sw, (cx<float> *)b.Bbar, st);
          if (s != EPW_OK) return fail(s, "tensor-core adjoint contraction failed");
        } else {
          launch_cgemm<float>(m->nRp, ncol, nq, (const cx<float> *)p.PqTp, nq, false, true,
                              (const cx<float> *)b.xbar, ncol, (cx<float> *)b.Bbar, ncol, false, st);
        }
        launch_bg_adjoint_rotate_k0<float>(kc, k0, m->nRp, m->nm, m->nw, (const cx<float> *)b.Bbar, p.Uk,
                                           (cx<float> *)b.G1bar, st);
        launch_cgemm<float>(m->nRe, ncol2, kc, p.Pk32 + (size_t)k0 * m->nRe, m->nRe, true, true,
                            (const cx<float> *)b.G1bar, ncol2, (cx<float> *)b.gwbar, ncol2, true, st);
      }
    }
  }
  if (b.dgd) {
    if (pair64)
      launch_dg64(m, b.gT, b.dgd, st);
    else if (prec == EPW_FP64)
      launch_dg_scale<double>(m, (const cx<double> *)b.gwbar, b.dgd, false, st);
    else
      launch_dg_scale<float>(m, (const cx<float> *)b.gwbar, b.dgd, false, st);
  }
  CK(cudaGetLastError());
  if (sdg) CK(cudaMemcpyAsync(dg, b.dgd, sizeof(double) * 2 * ng, cudaMemcpyDeviceToHost, st));
  if (dT) CK(cudaMemcpyAsync(dT, b.sc, sizeof(double), sdT ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st));
  if (dEF)
    CK(cudaMemcpyAsync(dEF, b.sc + 1, sizeof(double), sdE ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st));
  if (sk || sq || swq || scot || sdg || sdT || sdE) return read_status(m, st);
  return EPW_OK;
}

// ------------------------------------------------- phonon self-energy
// Per (q, nu) sums over the k list: Pi''_qnu (Eq. (linewidthph), on shell), lambda_qnu
// (Eq. (lambdaEQ)) and the nesting function (Eq. (nestingfct)); see include/epw.h.
extern "C" epw_status epw_phonon_selfenergy(const epw_model *mc, int nk, const double *k, const double *wk, int nq,
                                            const double *q, const epw_params *par, double *pi_im, double *lam,
                                            double *zeta, double *dos, void *stream) {
  g_err[0] = 0;
  epw_model *m = const_cast<epw_model *>(mc);
  CKS(check_common(m, nk, k, nq, q));
  CKS(check_params(par));
  cudaStream_t st = (cudaStream_t)stream;
  const int nm = m->nm;
  const bool tcp = par->precision == EPW_BF16X3 || par->precision == EPW_TF32X3;
  if (m->nw > 8 || nm > 9)
    return fail(EPW_ERR_UNSUPPORTED, "the phonon-side sums have no kernel for nw=%d, 3nat=%d (at most 8 and 9)",
                m->nw, nm);
  const int wprec = tcp ? EPW_FP32 : par->precision;
  const bool sk = nk > 0 && !is_device_ptr(k), sq = nq > 0 && !is_device_ptr(q);
  const bool swk = wk && nk > 0 && !is_device_ptr(wk);
  const bool spi = pi_im && nq > 0 && !is_device_ptr(pi_im), slam = lam && nq > 0 && !is_device_ptr(lam);
  const bool sz = zeta && nq > 0 && !is_device_ptr(zeta), sd = dos && !is_device_ptr(dos);
  // chunks of k per q block: enough blocks to fill the GPU a few times over
  const int nqb = (std::max(nq, 1) + 127) / 128;
  const int want = std::max(1, (4 * 152 + nqb - 1) / nqb);
  const int kper0 = std::max(1, (std::max(nk, 1) + want - 1) / want);
  int kper = kper0;
  // (FP64 in fixed point: warps of 32 q x kper k, about eight waves of two per sub-partition)
  const int kper64 = (int)std::max<long>(1, (long)std::max(nk, 1) * ((std::max(nq, 1) + 31) / 32) / 9728);
  struct B {
    Prep p;
    Fx64 fx;
    TcStaged sg;
    double *partial, *pid, *lamd, *zd, *dosd, *terms, *wkd;
    int nchunk;
  } b;
  bool fx_on = true;
  auto plan = [&](Arena &A) -> epw_status {
    plan_fx(A, m, std::max(nk, 1), std::max(nq, 1), fx_on && par->precision == EPW_FP64 && fx_dq(m, nq),
            fx_on && par->precision == EPW_FP64 && nk > 0 && nq > 0 && fx_pair(m, nk, nq),
            fx_on && par->precision == EPW_FP64 && nk > 0 && fx_g1(m, nk), b.fx);
    b.fx.exact = par->precision != EPW_FP64;
    plan_prep(A, m, std::max(nk, 1), std::max(nq, 1), wprec, sk, sq, false, true, b.p, &b.fx);
    b.wkd = swk ? A.take<double>((size_t)nk) : nullptr;  // k weights staged from the host
    b.sg = TcStaged{};
    kper = b.fx.pair ? kper64 : kper0;
    int nchunk = (std::max(nk, 1) + kper - 1) / kper;
    if (b.fx.pair) {
      nchunk = 0;
      for (int k0 = 0; k0 < nk; k0 += b.fx.kc) nchunk += (std::min(b.fx.kc, nk - k0) + kper - 1) / kper;
    }
    if (tcp) {
      CKS(tc_staged_plan(A, m, std::max(nk, 1), std::max(nq, 1), par->precision == EPW_BF16X3 ? TC_OP_BF16 : TC_OP_TF32,
                         STAGED_CT_BYTES, b.sg, true));
      if (!b.sg.ok) return fail(EPW_ERR_UNSUPPORTED, "no staged tensor-core form for this model");
      nchunk = 0;  // chunks of kper inside each staged chunk of sg.kc
      for (int k0 = 0; k0 < std::max(nk, 1); k0 += b.sg.kc) {
        const int kc = std::min(b.sg.kc, std::max(nk, 1) - k0);
        nchunk += (kc + kper - 1) / kper;
      }
    }
    b.nchunk = nchunk;
    b.partial = A.take<double>((size_t)nchunk * std::max(nq, 1) * (2 * nm + 1));
    b.pid = spi ? A.take<double>((size_t)nq * nm) : pi_im;
    b.lamd = slam ? A.take<double>((size_t)nq * nm) : lam;
    b.zd = sz ? A.take<double>((size_t)nq) : zeta;
    b.dosd = A.take<double>(1);
    b.terms = A.take<double>((size_t)std::max(nk, 1));
    return EPW_OK;
  };
  Arena A;
  CKS(plan_ws(m, A, b.fx, fx_on, plan));
  Prep &p = b.p;
  const double *kd = k, *qd = q, *wkd = wk;
  if (sk) {
    CK(cudaMemcpyAsync(p.kd, k, sizeof(double) * 3 * nk, cudaMemcpyHostToDevice, st));
    kd = p.kd;
  }
  if (sq) {
    CK(cudaMemcpyAsync(p.qd, q, sizeof(double) * 3 * nq, cudaMemcpyHostToDevice, st));
    qd = p.qd;
  }
  if (swk) {
    CK(cudaMemcpyAsync(b.wkd, wk, sizeof(double) * nk, cudaMemcpyHostToDevice, st));
    wkd = b.wkd;
  }
  CK(cudaMemsetAsync(b.dosd, 0, sizeof(double), st));
  if (nq > 0) {
    if (b.pid) CK(cudaMemsetAsync(b.pid, 0, sizeof(double) * (size_t)nq * nm, st));
    if (b.lamd) CK(cudaMemsetAsync(b.lamd, 0, sizeof(double) * (size_t)nq * nm, st));
    if (b.zd) CK(cudaMemsetAsync(b.zd, 0, sizeof(double) * (size_t)nq, st));
  }
  if (nk > 0 && nq > 0) {
    b.fx.T = par->T_K;
    b.fx.late = b.fx.pair;
    CKS(run_prep(m, nk, kd, nq, qd, wprec, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &b.fx));
  } else if (nk > 0) {
    // bands at k only (N(E_F))
    launch_phases(nk, kd, m->nRe, m->Re, m->rmax, p.PkRM, p.PkT, nullptr, st);
    launch_fourier_d(nk, m->nRe, p.PkT, m->Hw, m->nw * m->nw, p.Hk, st);
    launch_eigh_d(nk, m->nw, p.Hk, p.epsk, p.Uk, m->dstatus, st);
  }
  if (nk > 0) {
    launch_dos_terms(nk, m->nw, p.epsk, wkd, par->EF_eV, par->sigma_eV, b.terms, st);
    launch_sum_scalar(nk, b.terms, 1.0, b.dosd, st);
  }
  if (nk > 0 && nq > 0 && b.fx.pair) {
    int chunk0 = 0;
    for (int k0 = 0; k0 < nk; k0 += b.fx.kc) {
      const int kc = std::min(b.fx.kc, nk - k0), nch = (kc + kper - 1) / kper;
      CKS(run_fx_contract(m, k0, kc, p, b.fx, st));
      CKS(prep_join(m, b.fx, st));
      Pair64Args a = pair64_args(m, k0, kc, nq, nullptr, par, p, b.fx);
      a.wk = wkd;
      a.nk_total = nk;
      a.nkc = kper;
      a.partial = b.partial + (size_t)chunk0 * nq * (2 * nm + 1);
      epw_status s = launch_ph64(a, nch, st);
      if (s != EPW_OK) return fail(s, "no phonon-side kernel for nw=%d, 3nat=%d", m->nw, nm);
      chunk0 += nch;
    }
    launch_ph_finalize(nq, nm, b.nchunk, b.partial, p.omegaT, par->omega_min_eV, b.dosd, b.pid, b.lamd, b.zd, st);
  } else if (nk > 0 && nq > 0) {
    PairArgs a;
    std::memset(&a, 0, sizeof(a));
    a.nq = nq;
    a.nw = m->nw;
    a.nm = nm;
    a.nRe = m->nRe;
    a.nRp = m->nRp;
    a.PqTe = p.PqTe;
    a.PqTp = p.PqTp;
    a.BH = p.BH;
    a.Bg = p.Bg;
    a.ET = p.ET;
    a.omegaT = p.omegaT;
    a.eps_k = p.epsk;
    a.wq = wkd;  // the k weights
    a.nk_total = nk;
    a.T = par->T_K;
    a.EF = par->EF_eV;
    a.sigma = par->sigma_eV;
    a.omega_min = par->omega_min_eV;
    a.dstatus = m->dstatus;
    a.Cpol = m->polar ? p.Cpol : nullptr;
    a.Uk = p.Uk;
    a.nkc = kper;
    if (tcp) {
      b.sg.Pq64 = m->same_eph ? p.PqTph : nullptr;
      CKS(tc_staged_phases(m, nq, qd, b.sg, st));
      int chunk0 = 0;
      for (int k0 = 0; k0 < nk; k0 += b.sg.kc) {
        const int kc = std::min(b.sg.kc, nk - k0);
        epw_status s = tc_staged_contract(m, k0, kc, nq, (const cx<float> *)p.Bg, (const cx<float> *)p.BH, b.sg, st);
        if (s != EPW_OK) return fail(s, "staged tensor-core contraction failed");
        const int nch = (kc + kper - 1) / kper;
        a.k0 = k0;
        a.nk = kc;
        a.Cq = b.sg.Ct;
        a.ldc = b.sg.pair_ld();
        a.cpk = b.sg.cpk;
        a.partial = b.partial + (size_t)chunk0 * nq * (2 * nm + 1);
        s = launch_pair_ph<float>(a, nch, st);
        if (s != EPW_OK) return fail(s, "no phonon-side kernel for nw=%d, 3nat=%d", m->nw, nm);
        chunk0 += nch;
      }
    } else {
      a.k0 = 0;
      a.nk = nk;
      a.partial = b.partial;
      epw_status s = wprec == EPW_FP64 ? launch_pair_ph<double>(a, b.nchunk, st) : launch_pair_ph<float>(a, b.nchunk, st);
      if (s != EPW_OK) return fail(s, "no phonon-side kernel for nw=%d, 3nat=%d", m->nw, nm);
    }
    launch_ph_finalize(nq, nm, b.nchunk, b.partial, p.omegaT, par->omega_min_eV, b.dosd, b.pid, b.lamd, b.zd, st);
  }
  CK(cudaGetLastError());
  if (spi) CK(cudaMemcpyAsync(pi_im, b.pid, sizeof(double) * (size_t)nq * nm, cudaMemcpyDeviceToHost, st));
  if (slam) CK(cudaMemcpyAsync(lam, b.lamd, sizeof(double) * (size_t)nq * nm, cudaMemcpyDeviceToHost, st));
  if (sz) CK(cudaMemcpyAsync(zeta, b.zd, sizeof(double) * (size_t)nq, cudaMemcpyDeviceToHost, st));
  if (dos) CK(cudaMemcpyAsync(dos, b.dosd, sizeof(double), sd ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st));
  if (sk || sq || swk || spi || slam || sz || sd) return read_status(m, st);
  return EPW_OK;
}

// ------------------------------------------ complex self-energy, spectral function
extern "C" epw_status epw_selfenergy(const epw_model *mc, int nk, const double *k, int nq, const double *q,
                                     const double *wq, const epw_params *par, double delta, int nomega,
                                     const double *omega, double *sigma, double *spectral, void *stream) {
  g_err[0] = 0;
  epw_model *m = const_cast<epw_model *>(mc);
  CKS(check_common(m, nk, k, nq, q));
  CKS(check_params(par));
  if (!(delta > 0.0) || !std::isfinite(delta)) return fail(EPW_ERR_INVALID_ARG, "delta must be > 0");
  if (nomega < 0 || (nomega > 0 && (!omega || (nk > 0 && !sigma))))
    return fail(EPW_ERR_INVALID_ARG, "bad frequency grid or null output");
  if (m->nw > 8 || m->nm > 9)
    return fail(EPW_ERR_UNSUPPORTED, "the self-energy has no kernel for nw=%d, 3nat=%d (at most 8 and 9)", m->nw,
                m->nm);
  const bool tcp = par->precision == EPW_BF16X3 || par->precision == EPW_TF32X3;
  cudaStream_t st = (cudaStream_t)stream;
  const int nw = m->nw;
  const size_t nout = (size_t)nk * nw * nomega;
  if (nk == 0 || nomega == 0) return EPW_OK;
  const int wprec = tcp ? EPW_FP32 : par->precision;
  const bool sk = !is_device_ptr(k), sq = nq > 0 && !is_device_ptr(q), swq = wq && nq > 0 && !is_device_ptr(wq);
  const bool som = !is_device_ptr(omega), ssig = !is_device_ptr(sigma), ssp = spectral && !is_device_ptr(spectral);
  const int nqw = (std::max(nq, 1) + 31) / 32;
  const size_t per_k = (size_t)nqw * nw * (nomega + 1) * sizeof(double2);
  int kc = (int)std::max<size_t>(1, std::min<size_t>((size_t)nk, ((size_t)1 << 30) / per_k));
  struct B {
    Prep p;
    Fx64 fx;
    TcStaged sg;
    double *omd, *sigd, *specd, *re0;
    double2 *part;
  } b;
  bool fx_on = true;
  auto plan = [&](Arena &A) -> epw_status {
    plan_fx(A, m, nk, std::max(nq, 1), fx_on && fx_dq(m, nq), false,
            fx_on && wprec == EPW_FP64 && nq > 0 && fx_g1(m, nk), b.fx);
    plan_prep(A, m, nk, std::max(nq, 1), wprec, sk, sq, swq, true, b.p, &b.fx);
    b.sg = TcStaged{};
    if (tcp) {
      CKS(tc_staged_plan(A, m, nk, std::max(nq, 1), par->precision == EPW_BF16X3 ? TC_OP_BF16 : TC_OP_TF32,
                         STAGED_CT_BYTES, b.sg, true));
      if (!b.sg.ok) return fail(EPW_ERR_UNSUPPORTED, "no staged tensor-core form for this model");
      kc = std::min(kc, b.sg.kc);
    }
    b.omd = som ? A.take<double>((size_t)nomega) : const_cast<double *>(omega);
    b.sigd = ssig ? (double *)A.take<double2>(nout) : sigma;
    b.specd = ssp ? A.take<double>(nout) : spectral;
    b.part = A.take<double2>((size_t)kc * nqw * nw * (nomega + 1));
    b.re0 = A.take<double>((size_t)kc * nw);
    return EPW_OK;
  };
  Arena A;
  CKS(plan_ws(m, A, b.fx, fx_on, plan));
  Prep &p = b.p;
  const double *kd = k, *qd = q, *wqd = wq;
  if (sk) {
    CK(cudaMemcpyAsync(p.kd, k, sizeof(double) * 3 * nk, cudaMemcpyHostToDevice, st));
    kd = p.kd;
  }
  if (sq) {
    CK(cudaMemcpyAsync(p.qd, q, sizeof(double) * 3 * nq, cudaMemcpyHostToDevice, st));
    qd = p.qd;
  }
  if (swq) {
    CK(cudaMemcpyAsync(p.wqd, wq, sizeof(double) * nq, cudaMemcpyHostToDevice, st));
    wqd = p.wqd;
  }
  if (som) CK(cudaMemcpyAsync(b.omd, omega, sizeof(double) * nomega, cudaMemcpyHostToDevice, st));
  if (nq == 0) {
    // no q: Sigma = 0, and the spectral function's numerator |Sigma''| is 0 on the grid
    CK(cudaMemsetAsync(b.sigd, 0, nout * sizeof(double2), st));
    if (b.specd) CK(cudaMemsetAsync(b.specd, 0, nout * sizeof(double), st));
  } else {
    const PhaseA pa = staged_a(m, b.sg);
    CKS(run_prep(m, nk, kd, nq, qd, wprec, par->omega_min_eV, true, p, nullptr, st, true, nullptr, &b.fx,
                 tcp ? &pa : nullptr));
    b.sg.Pq64 = m->same_eph ? p.PqTph : nullptr;
    if (tcp) CKS(tc_staged_phases(m, nq, qd, b.sg, st));
    PairArgs a;
    std::memset(&a, 0, sizeof(a));
    a.nq = nq;
    a.nw = nw;
    a.nm = m->nm;
    a.nRe = m->nRe;
    a.nRp = m->nRp;
    a.PqTe = p.PqTe;
    a.PqTp = p.PqTp;
    a.BH = p.BH;
    a.Bg = p.Bg;
    a.ET = p.ET;
    a.omegaT = p.omegaT;
    a.eps_k = p.epsk;
    a.wq = wqd;
    a.T = par->T_K;
    a.EF = par->EF_eV;
    a.sigma = par->sigma_eV;
    a.omega_min = par->omega_min_eV;
    a.dstatus = m->dstatus;
    a.Cpol = m->polar ? p.Cpol : nullptr;
    a.Uk = p.Uk;
    for (int k0 = 0; k0 < nk; k0 += kc) {
      const int n = std::min(kc, nk - k0);
      a.k0 = k0;
      a.nk = n;
      if (tcp) {
        epw_status s = tc_staged_contract(m, k0, n, nq, (const cx<float> *)p.Bg, (const cx<float> *)p.BH, b.sg, st);
        if (s != EPW_OK) return fail(s, "staged tensor-core contraction failed");
        a.Cq = b.sg.Ct;
        a.ldc = b.sg.pair_ld();
        a.cpk = b.sg.cpk;
      }
      epw_status s = wprec == EPW_FP64 ? launch_pair_se<double>(a, nomega, b.omd, delta, b.part, st)
                                       : launch_pair_se<float>(a, nomega, b.omd, delta, b.part, st);
      if (s != EPW_OK) return fail(s, "no self-energy kernel for nw=%d, 3nat=%d", nw, m->nm);
      launch_se_finalize(n, k0, nw, nqw, nomega, b.part, b.omd, p.epsk, par->EF_eV, (double2 *)b.sigd, b.specd, b.re0, st);
    }
  }
  CK(cudaGetLastError());
  if (ssig) CK(cudaMemcpyAsync(sigma, b.sigd, nout * sizeof(double2), cudaMemcpyDeviceToHost, st));
  if (ssp) CK(cudaMemcpyAsync(spectral, b.specd, nout * sizeof(double), cudaMemcpyDeviceToHost, st));
  if (sk || sq || swq || som || ssig || ssp) return read_status(m, st);
  return EPW_OK;
}

// ---------------------------------------------------- failure-path self-test
extern "C" epw_status epw_selftest_wait_timeout(long long cycles, int *waited_out) {
  g_err[0] = 0;
  if (cycles < 1 || cycles > 4000000000LL) return fail(EPW_ERR_INVALID_ARG, "cycles must be in [1, 4e9]");
  struct D {
    unsigned st[4];
    int w;
  };
  D *d = nullptr;
  CK(cudaMalloc((void **)&d, sizeof(D)));
  epw_status s = EPW_OK;
  cudaError_t e = cudaMemset(d, 0, sizeof(D));
  if (e == cudaSuccess) {
    s = tc_wait_selftest(cycles, d->st, &d->w, 0);
    e = cudaDeviceSynchronize();
  }
  D h;
  std::memset(&h, 0, sizeof(h));
  if (e == cudaSuccess) e = cudaMemcpy(&h, d, sizeof(D), cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return fail(EPW_ERR_CUDA, "self-test: %s", cudaGetErrorString(e));
  if (s != EPW_OK) return fail(s, "self-test launch failed");
  if (waited_out) *waited_out = h.w;
  if (h.st[0] & EPW_DEV_TIMEOUT) return fail(EPW_ERR_TIMEOUT, "the bounded wait ran out (expected)");
  return EPW_OK;
}

// ---------------------------------------------------- Eliashberg function
extern "C" epw_status epw_eliashberg(int nq, int nmodes, const double *omega, const double *lambda,
                                     const double *wq, int ngrid, const double *grid, double sigma_ph, double *a2f,
                                     void *stream) {
  g_err[0] = 0;
  if (nq < 0 || nmodes < 0 || ngrid < 0) return fail(EPW_ERR_INVALID_ARG, "negative size");
  if (ngrid > 0 && (!grid || !a2f)) return fail(EPW_ERR_INVALID_ARG, "null grid or output");
  if ((size_t)nq * nmodes > 0 && (!omega || !lambda)) return fail(EPW_ERR_INVALID_ARG, "null omega or lambda");
  if (!(sigma_ph > 0.0) || !std::isfinite(sigma_ph)) return fail(EPW_ERR_INVALID_ARG, "sigma_ph must be > 0");
  if (ngrid == 0) return EPW_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t nt = (size_t)nq * nmodes;
  const bool so = nt && !is_device_ptr(omega), sl = nt && !is_device_ptr(lambda);
  const bool sw = wq && nq > 0 && !is_device_ptr(wq), sg = !is_device_ptr(grid), sa = !is_device_ptr(a2f);
  // scratch of this call only (the function has no model and no workspace)
  size_t bytes = 0;
  auto room = [&](bool need, size_t n) { size_t o = bytes; if (need) bytes += (n * sizeof(double) + 255) & ~size_t(255); return o; };
  const size_t oo = room(so, nt), ol = room(sl, nt), ow = room(sw, nq), og = room(sg, ngrid), oa = room(sa, ngrid);
  char *buf = nullptr;
  if (bytes) CK(cudaMallocAsync((void **)&buf, bytes, st));
  const double *om = so ? (const double *)(buf + oo) : omega, *la = sl ? (const double *)(buf + ol) : lambda;
  const double *w = sw ? (const double *)(buf + ow) : wq, *gr = sg ? (const double *)(buf + og) : grid;
  double *out = sa ? (double *)(buf + oa) : a2f;
  if (so) CK(cudaMemcpyAsync((void *)om, omega, nt * sizeof(double), cudaMemcpyHostToDevice, st));
  if (sl) CK(cudaMemcpyAsync((void *)la, lambda, nt * sizeof(double), cudaMemcpyHostToDevice, st));
  if (sw) CK(cudaMemcpyAsync((void *)w, wq, nq * sizeof(double), cudaMemcpyHostToDevice, st));
  if (sg) CK(cudaMemcpyAsync((void *)gr, grid, ngrid * sizeof(double), cudaMemcpyHostToDevice, st));
  launch_eliashberg(nq, nmodes, om, la, w, ngrid, gr, sigma_ph, out, st);
  CK(cudaGetLastError());
  if (sa) CK(cudaMemcpyAsync(a2f, out, ngrid * sizeof(double), cudaMemcpyDeviceToHost, st));
  if (buf) CK(cudaFreeAsync(buf, st));
  if (sa) CK(cudaStreamSynchronize(st));
  return EPW_OK;
}

// ------------------------------------------------ allocation-free linewidth
// Scratch for epw_linewidth_noalloc: a fixed device array that exists on every
// GPU on which this library is loaded, for the life of the process.  Host code
// must not hand the symbol itself to a kernel (in host code it names a host-side
// stand-in); it uses the device address obtained once per device below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[EPW_NOALLOC_SCRATCH_BYTES];

#define EPW_NOALLOC_MAX_DEVICES 64
static std::atomic<uintptr_t> g_noalloc_ptr[EPW_NOALLOC_MAX_DEVICES];

// Device address of the scratch array on the current device (looked up on the
// first call for that device, with that device current).
static epw_status noalloc_scratch(int dev, char **out) {
  if (dev < 0 || dev >= EPW_NOALLOC_MAX_DEVICES) return fail(EPW_ERR_UNSUPPORTED, "device index %d too large", dev);
  uintptr_t p = g_noalloc_ptr[dev].load(std::memory_order_acquire);
  if (!p) {
    void *addr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
    if (e != cudaSuccess || !addr)
      return fail(EPW_ERR_CUDA, "cudaGetSymbolAddress(scratch): %s", cudaGetErrorString(e));
    p = (uintptr_t)addr;
    g_noalloc_ptr[dev].store(p, std::memory_order_release);
  }
  *out = (char *)p;
  return EPW_OK;
}

extern "C" epw_status epw_linewidth_noalloc(const epw_model *mc, int nk, const double *k, int nq, const double *q,
                                            const double *wq, const epw_params *par, double *imsigma,
                                            void *stream) {
  g_err[0] = 0;
  epw_model *m = const_cast<epw_model *>(mc);
  CKS(check_common(m, nk, k, nq, q));
  CKS(check_params(par));
  const int prec = par->precision;
  if (prec != EPW_FP64 && prec != EPW_FP32)
    return fail(EPW_ERR_UNSUPPORTED, "epw_linewidth_noalloc runs EPW_FP64 or EPW_FP32");
  if ((nk > 0 && !is_device_ptr(k)) || (nq > 0 && !is_device_ptr(q)) || (wq && nq > 0 && !is_device_ptr(wq)) ||
      (nk > 0 && !is_device_ptr(imsigma)))
    return fail(EPW_ERR_INVALID_ARG, "epw_linewidth_noalloc takes device pointers only");
  cudaStream_t st = (cudaStream_t)stream;
  if (nk == 0) return EPW_OK;
  if (nq == 0) {
    CK(cudaMemsetAsync(imsigma, 0, sizeof(double) * (size_t)nk * m->nw, st));
    return EPW_OK;
  }
  // measure, then lay the buffers out inside the fixed scratch array
  LwPlan L;
  Arena A{nullptr, 0, 0};
  EpwTune tune = epwi_default_tune();
  tune.simt64 = true;  // the smallest buffers
  CKS(epwi_plan_linewidth(A, m, nk, nq, prec, false, false, false, false, tune, L));
  if (A.off > EPW_NOALLOC_SCRATCH_BYTES)
    return fail(EPW_ERR_INVALID_ARG, "problem needs %zu bytes of scratch; epw_linewidth_noalloc holds %zu", A.off,
                (size_t)EPW_NOALLOC_SCRATCH_BYTES);
  char *scratch = nullptr;
  CKS(noalloc_scratch(m->device, &scratch));
  A = Arena{scratch, (size_t)EPW_NOALLOC_SCRATCH_BYTES, 0};
  CKS(epwi_plan_linewidth(A, m, nk, nq, prec, false, false, false, false, tune, L));
  Prep &p = L.p;
  CKS(run_prep(m, nk, k, nq, q, prec, par->omega_min_eV, true, p, nullptr, st, /*fork=*/false));
  PairArgs a;
  std::memset(&a, 0, sizeof(a));
  a.nk = nk;
  a.nq = nq;
  a.nw = m->nw;
  a.nm = m->nm;
  a.nRe = m->nRe;
  a.nRp = m->nRp;
  a.PqTe = p.PqTe;
  a.PqTp = p.PqTp;
  a.BH = p.BH;
  a.Bg = p.Bg;
  a.ET = p.ET;
  a.omegaT = p.omegaT;
  a.eps_k = p.epsk;
  a.wq = wq;
  a.T = par->T_K;
  a.EF = par->EF_eV;
  a.sigma = par->sigma_eV;
  a.omega_min = par->omega_min_eV;
  a.partial = L.partial;  // every entry is written before it is read
  a.dstatus = m->dstatus;
  a.Cpol = m->polar ? p.Cpol : nullptr;
  a.Uk = p.Uk;
  epw_status s = prec == EPW_FP64 ? launch_pair<double>(a, 0, st) : launch_pair<float>(a, 0, st);
  if (s != EPW_OK) return fail(s, "no per-pair kernel for nw=%d, 3nat=%d in this precision", m->nw, m->nm);
  launch_finalize(nk, (nq + 127) / 128, m->nw, L.partial, imsigma, st);
  CK(cudaGetLastError());
  return EPW_OK;
}
