// build-variants: LBO_FX_N=16 LBO_FX_N=24 LBO_FX_N=32 LBO_FX_N=48 LBO_FX_N=64
//
// L[g] in the FP64 precision in 64-bit fixed point on the integer pipe
// (lin_fx.cuh), one translation unit per N; lin_fx_plan.cu
// dispatches to the functions defined here.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "lin_fx.cuh"
#include "lin_fx.h"

#define LBO_CAT_(a, b) a##b
#define LBO_CAT(a, b) LBO_CAT_(a, b)

namespace lbo {
namespace fx {

namespace {

constexpr int N = LBO_FX_N;
constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC, T = Geo<N>::T;
constexpr size_t H = (size_t)N * NC, n3 = (size_t)N * N * N, HC3 = (size_t)HC * HC * HC;
constexpr int ACC_WARPS = 8;

// Buffers of a call's instances (head and combination) and of a group of them
// (the gain loop), carved from the plan's workspace.
struct Buffers {
  // of B instances
  ci64 *R, *F, *MH;  // r^; fields L+, u, w (first: FFT(r), FFT(g) of the planes); M's factors
  i64* mh;
  double* inst;
  float *rm, *ub;
  int *eR, *em, *eM, *EPh, *EC, *bad;
  // of G instances
  ci64* W;
  i64* U;
  float* BP;
  int *eU, *EA, *EP;
  size_t bytes;
  Buffers(void* base, size_t B, size_t G, size_t J, bool own_u) {
    unsigned char* p = (unsigned char*)base;
    auto take = [&](auto*& ptr, size_t count) {
      ptr = (std::remove_reference_t<decltype(ptr)>)p;
      p += (count * sizeof(*ptr) + 255) / 256 * 256;
    };
    take(R, B * H);
    take(F, 3 * B * H);
    take(MH, B * 3 * N);
    take(mh, B * n3);
    take(inst, B * Inst<N>::SIZE);
    take(rm, B * BANDS * NC);
    take(eR, B * NC);
    take(em, B * N);
    take(eM, B * 3);
    take(EPh, 2 * B * N);
    take(EC, 3 * B * NC);
    take(bad, B);
    take(W, G * J * H);
    take(U, own_u ? G * J * HC3 : 0);
    take(BP, G * J * N);
    take(eU, own_u ? G * J : 0);
    take(ub, own_u ? G * J * BANDS * HC * HC : 0);
    take(EA, G * J);
    take(EP, G * J * N);
    bytes = (size_t)(p - (unsigned char*)base);
  }
};

// The Maxwellian cache of B instances in one buffer.
struct CacheBuffers {
  i64 *U, *mh;
  double* inst;
  float* ub;
  int *eU, *em, *bad;
  size_t bytes;
  CacheBuffers(void* base, size_t B, size_t J) {
    unsigned char* p = (unsigned char*)base;
    auto take = [&](auto*& ptr, size_t count) {
      ptr = (std::remove_reference_t<decltype(ptr)>)p;
      p += (count * sizeof(*ptr) + 255) / 256 * 256;
    };
    take(U, B * J * HC3);
    take(mh, B * n3);
    take(inst, B * Inst<N>::SIZE);
    take(ub, B * J * BANDS * HC * HC);
    take(eU, B * J);
    take(em, B * N);
    take(bad, B);
    bytes = (size_t)(p - (unsigned char*)base);
  }
};

// planes per block (LBO_OPT_PLANES at N = 32, default 4)
constexpr int PPC = PlanesPPC<N>::v;

template <typename K>
void smem_of(K kernel, size_t bytes) { raise_smem_limit((const void*)kernel, bytes); }

void launch_tables(lbo_plan* p, double* inst, int* em, i64* mh, ci64* MH, int* eM, int* bad, const double* params, int B,
                   const char* name1, const char* name2) {
  LBO_LAUNCH(p, name1, p->stream, k_instance<N>, B, kInstanceThreads<N>, 0, params, 2.0 * p->L / N,
             std::log(1.0 / p->eps), inst, em, bad);
  LBO_LAUNCH(p, name2, p->stream, k_mh<N>, dim3(N + 1, B), 256, 0, inst, em, mh, MH, eM);
}

void launch_uhat(lbo_plan* p, const double* inst, i64* U, int* eU, float* ub, int* bad, int B, const char* name) {
  smem_of(k_uhat<N>, Octant<N>::SMEM);
  using O = Octant<N>;
  if constexpr (O::CL == 1) {
    LBO_LAUNCH(p, name, p->stream, k_uhat<N>, dim3(p->J, B), O::BLOCK, O::SMEM, inst, p->d_phit64, U, eU, ub, bad,
               p->J);
  } else {
    ProfScope scope(p, name, p->stream);
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(O::CL * p->J, B);
    c.blockDim = dim3(O::BLOCK);
    c.dynamicSmemBytes = O::SMEM;
    c.stream = p->stream;
    cudaLaunchAttribute a{};
    a.id = cudaLaunchAttributeClusterDimension;
    a.val.clusterDim = {O::CL, 1, 1};
    c.attrs = &a;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, k_uhat<N>, inst, (const double*)p->d_phit64, U, eU, ub, bad, p->J);  // errors: cudaGetLastError
  }
}

template <int P>
void launch_planes(lbo_plan* p, const Buffers& w, const i64* mh, const int* em, int B) {
  smem_of(k_plane<N, P>, Planes<N, P>::BYTES);
  LBO_LAUNCH(p, "fx_plane_inv_mh_fwd", p->stream, (k_plane<N, P>), dim3(N / P, p->J, B), (Planes<N, P>::THREADS),
             (Planes<N, P>::BYTES), w.W, w.EA, mh, em, w.EP, w.BP);
}

void launch_head(lbo_plan* p, const Tables& tb, const Buffers& w, int B, int z0, int count, const char* name) {
  LBO_LAUNCH(p, name, p->stream, k_axis1_head<N>, dim3((NC * T + 63) / 64, B, count), 64, 0, w.F, w.EPh, w.MH, w.eM,
             tb.omega, 0, tb.omega_exp, 1, w.R, w.eR, w.rm, w.EC, z0);
}

constexpr int CPPC = CombinePPC<N>::v;

template <int MODE>
void launch_combine(lbo_plan* p, const Buffers& w, const double* inst, const double* g, const double* wc, const int* bad, double* out, int B,
                    const char* name) {
  using C = Combine<N, CPPC, MODE>;
  smem_of(k_combine_planes<N, CPPC, MODE>, C::BYTES);
  LBO_LAUNCH(p, name, p->stream, (k_combine_planes<N, CPPC, MODE>), dim3(N / CPPC, B), C::THREADS, C::BYTES, inst, g,
             w.F, w.EC, wc, bad, out);
}

}  // namespace

size_t LBO_CAT(cache_bytes_, LBO_FX_N)(int B, int J) { return CacheBuffers(nullptr, B, J).bytes; }

Cache LBO_CAT(cache_at_, LBO_FX_N)(void* base, int B, int J, int b0) {
  const CacheBuffers c(base, B, J);
  const size_t o = b0;
  return Cache{c.U + o * J * HC3, c.eU + o * J, c.ub + o * J * BANDS * HC * HC, c.bad + o, c.inst + o * Inst<N>::SIZE,
               c.em + o * N, c.mh + o * n3, nullptr, 0.0};
}

size_t LBO_CAT(workspace_bytes_, LBO_FX_N)(int B, int G, int J, bool own_u) {
  return Buffers(nullptr, B, G, J, own_u).bytes;
}

lbo_status LBO_CAT(apply_, LBO_FX_N)(lbo_plan* p, const Tables& tb, const double* params, const double* g, double* out,
                                     int B, int G, void* ws, const Cache* mc) {
  cudaStream_t s = p->stream;
  const int J = p->J;
  const Buffers w(ws, B, G, J, mc == nullptr);
  const size_t sb = sizeof(int) * B;
  cudaError_t e = mc ? cudaMemcpyAsync(w.bad, mc->bad, sb, cudaMemcpyDeviceToDevice, s)
                     : cudaMemsetAsync(w.bad, 0, sb, s);
  if (e != cudaSuccess) return cuda_fail(e, "fixed-point flags");
  // the instances' tables, unless the cache holds them for this cut-off
  const bool have = mc && mc->eps == p->eps;
  const double* inst = have ? mc->inst : w.inst;
  const i64* mh = have ? mc->mh : w.mh;
  const int* em = have ? mc->em : w.em;
  if (!have) launch_tables(p, w.inst, w.em, w.mh, w.MH, w.eM, w.bad, params, B, "fx_instance", "fx_mh_table");
  // r^ = FFT(r); InvFFT_1 of g^ omega and of M^ omega
  smem_of(k_fwd_planes<N, PPC>, Planes<N, PPC>::BYTES);
  LBO_LAUNCH(p, "fx_plane_fwd", s, (k_fwd_planes<N, PPC>), dim3(N / PPC, B, 2), (Planes<N, PPC>::THREADS),
             (Planes<N, PPC>::BYTES), g, inst, 1, p->cutoff, w.F, w.EPh, w.bad);
  launch_head(p, tb, w, B, 0, mc ? 2 : 3, "fx_axis1_head");
  int launches = have ? 3 : 5;
  static_assert(acc_smem<N, ACC_WARPS>(256) <= 226 * 1024, "shared memory of k_axis1_acc at the most radial nodes");
  const size_t smem = acc_smem<N, ACC_WARPS>(J);
  smem_of(k_axis1_acc<N, ACC_WARPS>, acc_smem<N, ACC_WARPS>(256));
  // the gain loop, all radial nodes of a group of instances at once
  for (int b0 = 0; b0 < B; b0 += G) {
    const int n = std::min(G, B - b0);
    const i64* U = mc ? mc->U + b0 * (size_t)J * HC3 : w.U;
    const int* eU = mc ? mc->eU + b0 * (size_t)J : w.eU;
    const float* ub = mc ? mc->ub + b0 * (size_t)J * BANDS * HC * HC : w.ub;
    const ci64* R = w.R + b0 * H;
    const int* eR = w.eR + b0 * (size_t)NC;
    if (!mc) {
      launch_uhat(p, inst + b0 * (size_t)Inst<N>::SIZE, w.U, w.eU, w.ub, w.bad + b0, n, "fx_uhat");
      launches += 1;
    }
    LBO_LAUNCH(p, "fx_unit_scale", s, k_unit_scale<N>, dim3(J, n), 256, 0, ub, eU, w.rm + b0 * (size_t)BANDS * NC, eR, w.EA, J);
    LBO_LAUNCH(p, "fx_axis1_uhat_inv", s, k_axis1_inv<N>, dim3((NC * T + 63) / 64, J, n), 64, 0, R, eR, U, eU, w.EA, w.W);
    if (N == 32 && p->planes_per_cta == 2) launch_planes<N == 32 ? 2 : PPC>(p, w, mh + b0 * n3, em + b0 * N, n);
    else if (N == 32 && p->planes_per_cta == 8) launch_planes<N == 32 ? 8 : PPC>(p, w, mh + b0 * n3, em + b0 * N, n);
    else launch_planes<PPC>(p, w, mh + b0 * n3, em + b0 * N, n);
    LBO_LAUNCH(p, "fx_axis1_fwd_acc", s, (k_axis1_acc<N, ACC_WARPS>), dim3((NC * T + 31) / 32, n), 32 * ACC_WARPS,
               smem, w.W, w.EP, w.BP, tb.phi, tb.phi_exp, tb.phi_max, w.F + b0 * H, w.EC + b0 * (size_t)NC, J);
    launches += 4;
  }
  // L+ - u M - w g
  if (mc) launch_combine<CACHED>(p, w, inst, g, mc->w, w.bad, out, B, "fx_combine");
  else launch_combine<COMBINE>(p, w, inst, g, nullptr, w.bad, out, B, "fx_combine");
  p->last_launches += launches;
  e = cudaGetLastError();
  return e == cudaSuccess ? LBO_OK : cuda_fail(e, "fixed-point launch");
}

lbo_status LBO_CAT(precompute_, LBO_FX_N)(lbo_plan* p, const Tables& tb, const double* params, int B, void* ws,
                                          const Cache& mc) {
  const Buffers w(ws, B, 0, p->J, false);
  launch_tables(p, (double*)mc.inst, (int*)mc.em, (i64*)mc.mh, w.MH, w.eM, (int*)mc.bad, params, B, "cache_fx_instance",
                "cache_fx_mh_table");
  launch_uhat(p, mc.inst, (i64*)mc.U, (int*)mc.eU, (float*)mc.ub, (int*)mc.bad, B, "cache_fx_uhat");
  launch_head(p, tb, w, B, 2, 1, "cache_fx_axis1_head");
  launch_combine<FACTOR>(p, w, nullptr, nullptr, nullptr, mc.bad, (double*)mc.w, B, "cache_fx_combine");
  p->last_launches += 5;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LBO_OK : cuda_fail(e, "fixed-point cache launch");
}

}  // namespace fx
}  // namespace lbo
