// The fixed-point form of the FP64 precision (lin_fx.cuh): what the plan's
// entry points (lbo.cu), the per-N units (lin_fx.cu) and their dispatch
// (lin_fx_plan.cu) share.
#pragma once
#include "lbo_internal.h"

namespace lbo {
namespace fx {

// phi_j(|k|^2) / N^6 as multipliers (fx64.cuh pack_mult) with one exponent
// per radial node: phi = value 2^-phi_exp[j], largest value in [2^61, 2^62).
struct Tables {
  const long long* phi = nullptr;   // [J][3(N/2)^2+1]
  const int* phi_exp = nullptr;     // [J]
  const double* phi_max = nullptr;  // [J] max |phi_j| / N^6
  const long long* omega = nullptr;  // [3(N/2)^2+1] omega(|k|^2) / N^3, the same with exponent omega_exp
  int omega_exp = 0;
};

// The Maxwellian-dependent factors of a set of instances.
struct Cache {
  const long long* U;  // [B][J][(N/2+1)^3] u^_j
  const int* eU;       // [B][J] its exponents
  const float* ub;     // [B][J][BANDS][(N/2+1)^2] its magnitudes (lin_fx.cuh)
  const int* bad;      // [B] 1: not finite
  const double* inst;  // the instances' tables (lin_fx.cuh) for the cut-off level eps
  const int* em;
  const long long* mh;
  const double* w;     // [B][N^3] InvFFT(FFT(M) omega)
  double eps;
};

// The hemisphere rule of Q(f,f) on the device, and optionally the loss
// multiplier of Eq. (2.16) per half-spectrum position (FP64, positions of
// fft.cuh) with a bound of its magnitude.
struct QuadRule {
  const double *gj, *sig, *wm;  // [J] radial nodes, [M][3] directions, [M] weights
  int M;
  const int4* node;        // [M], ordered by class: (node, class, sigma_1 < 0, first of its class)
  const int* class_begin;  // host, [classes + 1]: a class shares |sigma_1| and w_m
  int classes;
  double wmax;
  const double* omega3;
  double omega3_bound;
};

}  // namespace fx

// Q(f,f) of FP64 on the integer pipe; ws: a buffer grown as needed
lbo_status run_quadratic_fx(lbo_plan* p, const fx::QuadRule& rule, const double* f, double* out, int B, void** ws,
                            size_t* ws_bytes);
// L[g] of FP64 on the integer pipe (lin_fx_plan.cu)
lbo_status run_linearized_fx(lbo_plan* p, const double* params, const double* g, double* out, int B, bool cached);
lbo_status precompute_fx(lbo_plan* p, const double* params, int B);
size_t fx_cache_bytes(const lbo_plan* p, int B);
void free_fx_tables(lbo_plan* p);

}  // namespace lbo
