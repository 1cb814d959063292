// Calls the even-odd stencil's passes (csrc/schur.cu) on device buffers given by
// address, for tests/schur_driver.py.  prec: mglma_prec of the field named.
#include "internal.h"
#include "solver.h"

using namespace mglma;

static Spinor half_of(const mglma_gauge_s* G, void* p, int prec, int nrhs) {
  Spinor f;
  f.p = p;
  f.prec = prec;
  f.nrhs = nrhs;
  f.V = G->g.V / 2;
  return f;
}
static int done(mglma_ctx c, mglma_status st) {
  const cudaError_t e = cudaStreamSynchronize(c->stream);
  return st != MGLMA_OK ? (int)st : e == cudaSuccess ? 0 : (int)MGLMA_ERR_CUDA;
}
// sums' scratch, zeroed work of the call
struct Part {
  double* p = nullptr;
  explicit Part(const mglma_gauge_s* G, int n) { cudaMalloc(&p, schur_part_doubles(G->g.V, n) * sizeof(double)); }
  ~Part() { cudaFree(p); }
};

extern "C" {
int drv_ready(mglma_ctx c, mglma_gauge G, int* usable) {
  bool u = false;
  const int st = done(c, fine_eo_ready(c, G, &u, c->stream));
  *usable = u;
  return st;
}
int drv_odd(mglma_ctx c, mglma_gauge G, int n, void* in, int prec, void* w) {
  Spinor W = half_of(G, w, MGLMA_FP32, n);
  return done(c, schur_odd(c, G, half_of(G, in, prec, n), W, c->stream));
}
int drv_odd_solution(mglma_ctx c, mglma_gauge G, int n, void* xe, void* bo, void* xo) {
  Spinor e = half_of(G, xe, MGLMA_FP32, n), o = half_of(G, xo, MGLMA_FP32, n);
  return done(c, schur_odd_solution(c, G, xe ? &e : nullptr, half_of(G, bo, MGLMA_FP32, n), o, c->stream));
}
int drv_prepare(mglma_ctx c, mglma_gauge G, int n, void* be, void* vo, void* out) {
  Spinor o = half_of(G, out, MGLMA_FP32, n);
  return done(c, schur_prepare(c, G, half_of(G, be, MGLMA_FP32, n), half_of(G, vo, MGLMA_FP32, n), o, c->stream));
}
int drv_apply(mglma_ctx c, mglma_gauge G, int n, void* w, void* x, void* out) {
  Spinor o = half_of(G, out, MGLMA_FP32, n);
  return done(c, schur_apply(c, G, half_of(G, w, MGLMA_FP32, n), half_of(G, x, MGLMA_FP32, n), o, c->stream));
}
int drv_resid(mglma_ctx c, mglma_gauge G, int n, void* w, void* x, void* b, void* out, int prec) {
  Spinor o = half_of(G, out, prec, n);
  return done(c, schur_resid(c, G, half_of(G, w, MGLMA_FP32, n), half_of(G, x, MGLMA_FP32, n), half_of(G, b, MGLMA_FP32, n), o,
                             c->stream));
}
int drv_dot(mglma_ctx c, mglma_gauge G, int n, void* w, void* x, void* out, int prec, float2* alpha) {
  Spinor o = half_of(G, out, prec, n);
  Part part(G, n);
  return done(c, schur_dot(c, G, half_of(G, w, MGLMA_FP32, n), half_of(G, x, prec, n), o, part.p, alpha, c->stream));
}
int drv_mr(mglma_ctx c, mglma_gauge G, int n, void* w, void* t, void* tn, void* sk, void* sn, int prec,
           const float2* alpha, float2* alpha_n) {
  Spinor T = half_of(G, tn, prec, n), S = half_of(G, sn, prec, n);
  Part part(G, n);
  return done(c, schur_mr_step(c, G, half_of(G, w, MGLMA_FP32, n), half_of(G, t, prec, n), T, half_of(G, sk, prec, n), S, alpha,
                               alpha_n, part.p, c->stream));
}
int drv_gcr(mglma_ctx c, mglma_gauge G, int n, void* w, void* x, void* out, int k, void* W0, void* r, double* nw,
            double2* num, double2* dots) {
  Spinor o = half_of(G, out, MGLMA_FP32, n);
  Part part(G, n);
  return done(c, schur_gcr(c, G, half_of(G, w, MGLMA_FP32, n), half_of(G, x, MGLMA_FP32, n), o, k, W0, (size_t)12 * G->g.V * n,
                           r, part.p, nw, num, dots, c->stream));
}
}
