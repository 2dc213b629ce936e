// Dispatch of the fixed-point form of the FP64 precision over N and over
// groups of instances, and its tables (lin_fx.cuh and quad_fx.cuh have the
// kernels).
#include <algorithm>
#include <cmath>
#include <vector>

#include "fx64.cuh"
#include "lin_fx.h"

namespace lbo {
namespace fx {

#define LBO_FX_DECL(n)                                                                                            \
  size_t workspace_bytes_##n(int B, int G, int J, bool own_u);                                                    \
  lbo_status apply_##n(lbo_plan* p, const Tables& tb, const double* params, const double* g, double* out, int B,  \
                       int G, void* ws, const Cache* mc);                                                         \
  lbo_status precompute_##n(lbo_plan* p, const Tables& tb, const double* params, int B, void* ws, const Cache& mc); \
  size_t cache_bytes_##n(int B, int J);                                                                           \
  Cache cache_at_##n(void* base, int B, int J, int b0);
#define LBO_FX_QDECL(n)                                                                                            \
  size_t q_workspace_bytes_##n(int B, int J, const QuadRule& rule);                                             \
  lbo_status q_apply_##n(lbo_plan* p, const Tables& tb, const QuadRule& rule, const double* f, double* out, int B, \
                         void* ws);
LBO_FX_QDECL(16)
LBO_FX_QDECL(24)
LBO_FX_QDECL(32)
LBO_FX_QDECL(48)
LBO_FX_QDECL(64)
#undef LBO_FX_QDECL
LBO_FX_DECL(16)
LBO_FX_DECL(24)
LBO_FX_DECL(32)
LBO_FX_DECL(48)
LBO_FX_DECL(64)
#undef LBO_FX_DECL

namespace {

size_t workspace_bytes(int N, int B, int G, int J, bool own_u) {
  switch (N) {
    case 16: return workspace_bytes_16(B, G, J, own_u);
    case 24: return workspace_bytes_24(B, G, J, own_u);
    case 32: return workspace_bytes_32(B, G, J, own_u);
    case 48: return workspace_bytes_48(B, G, J, own_u);
    default: return workspace_bytes_64(B, G, J, own_u);
  }
}

lbo_status apply_part(lbo_plan* p, const Tables& tb, const double* params, const double* g, double* out, int B, int G,
                      const Cache* mc) {
  switch (p->N) {
    case 16: return apply_16(p, tb, params, g, out, B, G, p->ws, mc);
    case 24: return apply_24(p, tb, params, g, out, B, G, p->ws, mc);
    case 32: return apply_32(p, tb, params, g, out, B, G, p->ws, mc);
    case 48: return apply_48(p, tb, params, g, out, B, G, p->ws, mc);
    case 64: return apply_64(p, tb, params, g, out, B, G, p->ws, mc);
    default: return LBO_EUNSUPPORTED;
  }
}

lbo_status precompute_part(lbo_plan* p, const Tables& tb, const double* params, int B, const Cache& mc) {
  switch (p->N) {
    case 16: return precompute_16(p, tb, params, B, p->ws, mc);
    case 24: return precompute_24(p, tb, params, B, p->ws, mc);
    case 32: return precompute_32(p, tb, params, B, p->ws, mc);
    case 48: return precompute_48(p, tb, params, B, p->ws, mc);
    case 64: return precompute_64(p, tb, params, B, p->ws, mc);
    default: return LBO_EUNSUPPORTED;
  }
}

// Instances per group of the gain loop: their J half spectra together at most
// 1 GB; n instances are spread evenly over the fewest groups.  The kernels wait
// for latencies, not for memory bandwidth, so full waves of blocks count for
// more than keeping a group in the L2 cache (N = 32, batch 256: 7.30 ms per
// application at 64 MB, 6.40 at 143 MB, 5.74 at 572 MB, 5.58 at 1.1 GB, 5.54 at
// 2.3 GB; N = 64, batch 64: 39.9, 39.8, 35.2, 32.9, 32.3).
int largest_group(const lbo_plan* p) {
  const size_t unit = (size_t)p->N * p->N * (p->N / 2 + 1) * sizeof(ci64) * p->J;
  return (int)std::max<size_t>(1, ((size_t)1 << 30) / unit);
}
int group_size(const lbo_plan* p, int n) {
  const int most = largest_group(p);
  const int groups = (n + most - 1) / most;
  return (n + groups - 1) / groups;
}

// Instances per part of a call: their head and combination buffers (about 6
// half spectra each) stay below 2 GB.
int part_size(const lbo_plan* p, int B) {
  const size_t inst = (size_t)p->N * p->N * (p->N / 2 + 1) * sizeof(ci64) * 6;
  const int most = (int)std::max<size_t>(1, ((size_t)2 << 30) / inst);
  return std::min(B, most);
}

size_t cache_bytes(int N, int B, int J) {
  switch (N) {
    case 16: return cache_bytes_16(B, J);
    case 24: return cache_bytes_24(B, J);
    case 32: return cache_bytes_32(B, J);
    case 48: return cache_bytes_48(B, J);
    default: return cache_bytes_64(B, J);
  }
}

// The cache of B instances (p->mc_uh; the loss factor in p->mc_w) from instance b0 on.
Cache cache_at(const lbo_plan* p, int B, int b0) {
  Cache c;
  switch (p->N) {
    case 16: c = cache_at_16(p->mc_uh, B, p->J, b0); break;
    case 24: c = cache_at_24(p->mc_uh, B, p->J, b0); break;
    case 32: c = cache_at_32(p->mc_uh, B, p->J, b0); break;
    case 48: c = cache_at_48(p->mc_uh, B, p->J, b0); break;
    default: c = cache_at_64(p->mc_uh, B, p->J, b0);
  }
  c.w = (const double*)p->mc_w + (size_t)b0 * p->N * p->N * p->N;
  c.eps = p->mc_eps;
  return c;
}

// Multipliers value 2^-exponent of n doubles, largest in [2^61, 2^62).
int to_multipliers(const double* x, size_t n, double scale, long long* m, double* top) {
  double t = 0.0;
  for (size_t k = 0; k < n; ++k) t = std::max(t, std::fabs(x[k] * scale));
  const int e = t > 0.0 ? 61 - std::ilogb(t) : 0;
  for (size_t k = 0; k < n; ++k) m[k] = pack_mult(std::llrint(std::scalbn(x[k] * scale, e)));
  if (top) *top = t;
  return e;
}

lbo_status tables(lbo_plan* p, Tables* tb) {
  const int J = p->J, Q = 3 * (p->N / 2) * (p->N / 2) + 1;
  const size_t words = (size_t)J * Q;
  if (!p->d_fx) {
    // from the plan's FP64 multipliers; a further 1 / N^3 on phi_j normalises
    // the inverse transform of u^_j r^
    std::vector<double> x(words + Q);
    cudaError_t e = cudaMemcpy(x.data(), p->d_phi64, sizeof(double) * words, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess)
      e = cudaMemcpy(x.data() + words, p->d_omega64, sizeof(double) * Q, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "fixed-point tables");
    std::vector<long long> buf(words + Q + 2 * J);
    double* pm = (double*)(buf.data() + words + Q);
    int* qe = (int*)(buf.data() + words + Q + J);
    const double inv_n3 = 1.0 / ((double)p->N * p->N * p->N);
    for (int j = 0; j < J; ++j)
      qe[j] = to_multipliers(x.data() + (size_t)j * Q, Q, inv_n3, buf.data() + (size_t)j * Q, pm + j);
    p->fx_omega_exp = to_multipliers(x.data() + words, Q, 1.0, buf.data() + words, nullptr);
    e = cudaMalloc(&p->d_fx, sizeof(long long) * buf.size());
    if (e == cudaSuccess) e = upload_table(p->d_fx, buf.data(), sizeof(long long) * buf.size());
    if (e != cudaSuccess) {
      free_fx_tables(p);
      return cuda_fail(e, "fixed-point tables");
    }
  }
  tb->phi = (const long long*)p->d_fx;
  tb->omega = tb->phi + words;
  tb->phi_max = (const double*)(tb->omega + Q);
  tb->phi_exp = (const int*)(tb->omega + Q + J);
  tb->omega_exp = p->fx_omega_exp;
  return LBO_OK;
}

lbo_status ensure(void** ws, size_t* have, size_t bytes) {
  if (*ws && bytes <= *have) return LBO_OK;
  if (*ws) cudaFree(*ws);
  *ws = nullptr;
  *have = 0;
  if (cudaMalloc(ws, bytes) != cudaSuccess) {
    *ws = nullptr;
    cudaGetLastError();
    set_error_text("workspace allocation");
    return LBO_ENOMEM;
  }
  *have = bytes;
  return LBO_OK;
}

size_t q_workspace_bytes(int N, int B, int J, const QuadRule& rule) {
  switch (N) {
    case 16: return q_workspace_bytes_16(B, J, rule);
    case 24: return q_workspace_bytes_24(B, J, rule);
    case 32: return q_workspace_bytes_32(B, J, rule);
    case 48: return q_workspace_bytes_48(B, J, rule);
    default: return q_workspace_bytes_64(B, J, rule);
  }
}

lbo_status q_apply_part(lbo_plan* p, const Tables& tb, const QuadRule& rule, const double* f, double* out, int B,
                        void* ws) {
  switch (p->N) {
    case 16: return q_apply_16(p, tb, rule, f, out, B, ws);
    case 24: return q_apply_24(p, tb, rule, f, out, B, ws);
    case 32: return q_apply_32(p, tb, rule, f, out, B, ws);
    case 48: return q_apply_48(p, tb, rule, f, out, B, ws);
    case 64: return q_apply_64(p, tb, rule, f, out, B, ws);
    default: return LBO_EUNSUPPORTED;
  }
}

}  // namespace
}  // namespace fx

size_t fx_cache_bytes(const lbo_plan* p, int B) { return fx::cache_bytes(p->N, B, p->J); }

void free_fx_tables(lbo_plan* p) {
  if (p->d_fx) cudaFree(p->d_fx);
  p->d_fx = nullptr;
}

lbo_status run_linearized_fx(lbo_plan* p, const double* params, const double* g, double* out, int B, bool cached) {
  fx::Tables tb;
  lbo_status st = fx::tables(p, &tb);
  const int part = fx::part_size(p, B), G = fx::group_size(p, part);
  // the same buffer for cached and uncached calls and never more for a smaller
  // batch: graphs captured with a plan keep its address
  const size_t bytes = fx::workspace_bytes(p->N, part, std::min(part, fx::largest_group(p)), p->J, true);
  if (st == LBO_OK) st = fx::ensure(&p->ws, &p->ws_bytes, bytes);
  const size_t n3 = (size_t)p->N * p->N * p->N;
  p->last_launches = 0;
  for (int b0 = 0; b0 < B && st == LBO_OK; b0 += part) {
    const fx::Cache mc = cached ? fx::cache_at(p, B, b0) : fx::Cache{};
    st = fx::apply_part(p, tb, params + 5 * (size_t)b0, g + b0 * n3, out + b0 * n3, std::min(part, B - b0), G,
                        cached ? &mc : nullptr);
  }
  if (st == LBO_OK && (p->mass_fix || p->moment_fix))
    st = launch_fixes(p, out, B, p->N, 2.0 * p->L / p->N, p->stream, &p->last_launches);
  return st;
}

lbo_status precompute_fx(lbo_plan* p, const double* params, int B) {
  fx::Tables tb;
  lbo_status st = fx::tables(p, &tb);
  const int part = fx::part_size(p, B);
  if (st == LBO_OK) st = fx::ensure(&p->ws, &p->ws_bytes, fx::workspace_bytes(p->N, part, 0, p->J, false));
  if (st != LBO_OK) return st;
  cudaError_t e = cudaMemsetAsync((void*)fx::cache_at(p, B, 0).bad, 0, sizeof(int) * (size_t)B, p->stream);
  if (e != cudaSuccess) return cuda_fail(e, "fixed-point flags");
  p->mc_eps = p->eps;
  p->last_launches = 0;
  for (int b0 = 0; b0 < B && st == LBO_OK; b0 += part)
    st = fx::precompute_part(p, tb, params + 5 * (size_t)b0, std::min(part, B - b0), fx::cache_at(p, B, b0));
  return st;
}

lbo_status run_quadratic_fx(lbo_plan* p, const fx::QuadRule& rule, const double* f, double* out, int B, void** ws,
                            size_t* ws_bytes) {
  fx::Tables tb;
  lbo_status st = fx::tables(p, &tb);
  const int part = fx::part_size(p, B);
  if (st == LBO_OK)
    st = fx::ensure(ws, ws_bytes, fx::q_workspace_bytes(p->N, part, p->J, rule));
  const size_t n3 = (size_t)p->N * p->N * p->N;
  p->last_launches = 0;
  for (int b0 = 0; b0 < B && st == LBO_OK; b0 += part)
    st = fx::q_apply_part(p, tb, rule, f + b0 * n3, out + b0 * n3, std::min(part, B - b0), *ws);
  if (st == LBO_OK && (p->mass_fix || p->moment_fix))
    st = launch_fixes(p, out, B, p->N, 2.0 * p->L / p->N, p->stream, &p->last_launches);
  return st;
}

}  // namespace lbo
