// Autotuner of the RHS tile widths: the stencil's tile shape (RHS per thread
// 1, 2, 4 times RHS tiles per CTA 1, 2, 4, or the staged-tile kernel with 4, 8
// or 16 RHS per CTA) and the tensor-core coarse
// kernel's RHS per tile (8, 16, 32) are timed with
// CUDA events on the context stream for a given RHS count, and the fastest
// is kept per (kernel, RHS bucket, lattice volume) in the context; the table
// can be saved to and loaded from a text file keyed by GPU name.  The stencil is
// timed as mglma_dirac_apply runs it, between canonical fields: a lone stencil
// is within 5 % for several shapes, but all except (1,1) need an unpack pass (16
// RHS of 32x16^3: 348 us at (1,1), 398 to 452 at the others).  The solver
// tunes the shapes of a (lattice, RHS bucket) on its first batch
// (autotune_for_batch; the stencil only on lattices with an odd extent, the
// others solve on the even-odd one); with MGLMA_TUNE_CACHE naming a file, a context loads
// that file when created and saves the table after each automatic tuning.
#include <cstdio>
#include <cstring>
#include <fstream>
#include <functional>
#include <sstream>
#include <string>
#include <tuple>

#include "internal.h"
#include "solver.h"
#include "subspace.h"

namespace mglma {

// the least of `tries` averages over `reps` calls, after a warm-up call
static mglma_status time_ms(mglma_ctx ctx, cudaStream_t s, int reps, const std::function<mglma_status()>& f,
                            double* ms, int tries = 1) {
  cudaEvent_t a, b;
  MG_CUDA(cudaEventCreate(&a));
  MG_CUDA(cudaEventCreate(&b));
  mglma_status st = f();  // warm-up
  for (int k = 0; k < tries && st == MGLMA_OK; ++k) {
    cudaEventRecord(a, s);
    for (int i = 0; i < reps && st == MGLMA_OK; ++i) st = f();
    cudaEventRecord(b, s);
    cudaEventSynchronize(b);
    float t = 0;
    cudaEventElapsedTime(&t, a, b);
    if (k == 0 || t / reps < *ms) *ms = t / reps;
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  (void)ctx;
  return st;
}

static std::string gpu_name(int dev) {
  cudaDeviceProp p;
  if (cudaGetDeviceProperties(&p, dev) != cudaSuccess) return "unknown";
  std::string n = p.name;
  for (auto& c : n)
    if (c == ' ') c = '_';
  return n;
}

// Tunes the tile shapes of this (lattice, RHS bucket) unless the context
// holds them already, and saves the table to the context's cache file.
mglma_status autotune_for_batch(mglma_ctx ctx, mglma_gauge_s* G, mglma_coarse_s* C, int nrhs) {
  bool even = G->eo_state >= 0;
  for (int m = 0; m < 4; ++m) even = even && G->g.L[m] % 2 == 0;
  const bool need_d = !even && !has_tuned(ctx, TUNE_DSLASH32_NR, nrhs, G->g.V);
  const bool need_c = C && C->Aimg && !has_tuned(ctx, TUNE_COARSE_NT, nrhs, C->geo.V1);
  if (!need_d && !need_c) return MGLMA_OK;
  MG_CHECK(mglma_autotune(ctx, need_d ? G : nullptr, need_c ? C : nullptr, nrhs));
  if (!ctx->tune_cache.empty()) mglma_autotune_save(ctx, ctx->tune_cache.c_str());  // best effort
  return MGLMA_OK;
}

}  // namespace mglma

using namespace mglma;

extern "C" {

mglma_status mglma_autotune(mglma_ctx ctx, mglma_gauge G, mglma_coarse C, int nrhs) {
  if (!ctx || nrhs < 1) return fail(MGLMA_ERR_INVALID, "autotune: bad arguments");
  MG_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t s = ctx->stream;
  const bool prof = ctx->profile;
  ctx->profile = false;
  const int bucket = rhs_bucket(nrhs);
  mglma_status st = MGLMA_OK;
  const auto key_d = std::make_tuple((int)TUNE_DSLASH32_NR, bucket, G ? G->g.V : (int64_t)0);
  const auto key_c = std::make_tuple((int)TUNE_COARSE_NT, bucket, C ? C->geo.V1 : (int64_t)0);
  if (G && G->ready) {
    // one canonical field, applied in place (an FP32 application has read all of
    // its input before it writes), and two FP32 work fields; without room for
    // them the stencil alone between the work fields
    Spinor a, b;
    FreeList fl(ctx, s);
    const size_t field = (size_t)nrhs * G->g.V * 24;
    void *work = nullptr, *canon = nullptr;
    a.prec = b.prec = MGLMA_FP32;
    a.nrhs = b.nrhs = nrhs;
    a.V = b.V = G->g.V;
    const size_t off = (a.bytes() + 255) / 256 * 256;
    st = dalloc(ctx, &work, off + b.bytes(), s);
    fl.add(work);
    if (st == MGLMA_OK) {
      a.p = work;
      b.p = (char*)work + off;
      MG_CUDA(cudaMemsetAsync(work, 0, off + b.bytes(), s));
      if (dalloc(ctx, &canon, field * sizeof(double), s) == MGLMA_OK)
        MG_CUDA(cudaMemsetAsync(canon, 0, field * sizeof(double), s));
      fl.add(canon);
    }
    auto apply = [&] {
      double* c = (double*)canon;
      return c ? dirac_canonical(ctx, G, MGLMA_OP_D, nrhs, c, c, MGLMA_FP32, work, s)
               : dslash(ctx, G, a, b, false, false, s);
    };
    double best = 1e30;
    int choice = 1;
    // {NR, RW} of the one-site-per-thread kernel; {0, NRT} the staged-tile kernel
    const int shapes[][2] = {{1, 1}, {2, 1}, {4, 1}, {1, 2}, {1, 4}, {2, 2}, {2, 4}, {0, 4}, {0, 8}, {0, 16}};
    for (const auto& sh : shapes) {
      if (st != MGLMA_OK) break;
      const int width = sh[0] ? sh[0] * sh[1] : sh[1];
      if (width > 1 && width > nrhs) continue;  // tiles mostly idle
      const int code = sh[0] ? dslash32_tile_code(sh[0], sh[1]) : 64 + sh[1];
      ctx->tune[key_d] = {code, 0.0};
      double ms = 0;
      st = time_ms(ctx, s, 5, apply, &ms, 3);  // a hiccup must not decide
      if (st == MGLMA_OK && ms < best) {
        best = ms;
        choice = code;
      }
    }
    ctx->tune[key_d] = {choice, best};
  }
  if (st == MGLMA_OK && C && C->Aimg) {
    const size_t n = (size_t)nrhs * C->geo.V1 * C->n2;
    FreeList fl(ctx, s);
    void *X = nullptr, *Y = nullptr;
    st = dalloc(ctx, &X, n * sizeof(float2), s);
    if (st == MGLMA_OK) st = dalloc(ctx, &Y, n * sizeof(float2), s);
    fl.add(X);
    fl.add(Y);
    if (st == MGLMA_OK) MG_CUDA(cudaMemsetAsync(X, 0, n * sizeof(float2), s));
    double best = 1e30;
    int choice = 8;
    for (int nt : {8, 16, 32}) {
      if (st != MGLMA_OK || (nt > 8 && nt >= 2 * nrhs)) break;  // tiles mostly padding
      ctx->tune[key_c] = {nt, 0.0};
      double ms = 0;
      st = time_ms(ctx, s, 5, [&] { return coarse_apply(ctx, C, X, Y, nrhs, MGLMA_FP32, CMODE_D, s); }, &ms);
      if (st == MGLMA_OK && ms < best) {
        best = ms;
        choice = nt;
      }
    }
    ctx->tune[key_c] = {choice, best};
    if (st == MGLMA_OK) st = coarse_tc_check(C, s);
  }
  ctx->profile = prof;
  return st;
}

mglma_status mglma_autotune_get(mglma_ctx ctx, int kernel, int nrhs, int* choice, double* ms) {
  if (!ctx) return fail(MGLMA_ERR_INVALID, "autotune_get: NULL context");
  if (choice) *choice = 0;
  if (ms) *ms = 0;
  // the entry set for every lattice (volume 0), else the one of the largest
  // tuned lattice (the map is ordered by volume within a kernel and bucket)
  const int b = rhs_bucket(nrhs);
  const std::pair<int, double>* hit = nullptr;
  for (auto& kv : ctx->tune) {
    if (std::get<0>(kv.first) != kernel || std::get<1>(kv.first) != b) continue;
    if (std::get<2>(kv.first) == 0) {
      hit = &kv.second;
      break;
    }
    hit = &kv.second;
  }
  if (hit) {
    if (choice) *choice = hit->first;
    if (ms) *ms = hit->second;
  }
  return MGLMA_OK;
}

mglma_status mglma_autotune_set(mglma_ctx ctx, int kernel, int nrhs, int choice) {
  if (!ctx || nrhs < 1) return fail(MGLMA_ERR_INVALID, "autotune_set: bad arguments");
  const bool ok = (kernel == TUNE_DSLASH32_NR && dslash32_tile_valid(choice)) ||
                  (kernel == TUNE_COARSE_NT && (choice == 8 || choice == 16 || choice == 32));
  if (!ok) return fail(MGLMA_ERR_INVALID, "autotune_set: unknown kernel or choice");
  ctx->tune[std::make_tuple(kernel, rhs_bucket(nrhs), (int64_t)0)] = {choice, 0.0};
  return MGLMA_OK;
}

mglma_status mglma_autotune_save(mglma_ctx ctx, const char* path) {
  if (!ctx || !path) return fail(MGLMA_ERR_INVALID, "autotune_save: NULL argument");
  std::ofstream f(path);
  if (!f) return fail(MGLMA_ERR_INVALID, std::string("autotune_save: cannot write ") + path);
  const std::string gpu = gpu_name(ctx->device);
  for (auto& kv : ctx->tune)
    f << gpu << ' ' << std::get<0>(kv.first) << ' ' << std::get<1>(kv.first) << ' ' << std::get<2>(kv.first) << ' '
      << kv.second.first << ' ' << kv.second.second << '\n';
  return MGLMA_OK;
}

mglma_status mglma_autotune_load(mglma_ctx ctx, const char* path) {
  if (!ctx || !path) return fail(MGLMA_ERR_INVALID, "autotune_load: NULL argument");
  std::ifstream f(path);
  if (!f) return fail(MGLMA_ERR_INVALID, std::string("autotune_load: cannot read ") + path);
  const std::string gpu = gpu_name(ctx->device);
  std::string line;
  while (std::getline(f, line)) {
    std::istringstream is(line);
    std::string g;
    int k, b, c;
    long long vol;
    double ms;
    if (!(is >> g >> k >> b >> vol >> c >> ms) || g != gpu) continue;
    const bool ok = (k == TUNE_DSLASH32_NR && dslash32_tile_valid(c)) ||
                    (k == TUNE_COARSE_NT && (c == 8 || c == 16 || c == 32));
    if (ok && b >= 1 && b <= 64 && vol >= 0) ctx->tune[std::make_tuple(k, b, (int64_t)vol)] = {c, ms};
  }
  return MGLMA_OK;
}

}  // extern "C"
