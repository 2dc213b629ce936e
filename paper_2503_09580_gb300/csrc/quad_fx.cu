// build-variants: LBO_FX_N=16 LBO_FX_N=24 LBO_FX_N=32 LBO_FX_N=48 LBO_FX_N=64
//
// Q(f,f) in the FP64 precision in 64-bit fixed point on the integer pipe
// (quad_fx.cuh), one translation unit per N; lin_fx_plan.cu dispatches to the
// functions defined here.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "lin_fx.h"
#include "quad_fx.cuh"

#define LBO_CAT_(a, b) a##b
#define LBO_CAT(a, b) LBO_CAT_(a, b)

namespace lbo {
namespace fx {

namespace {

constexpr int N = LBO_FX_N;
constexpr int NC = Geo<N>::NC, T = Geo<N>::T;
constexpr size_t H = (size_t)N * NC, n3 = (size_t)N * N * N;
constexpr int kSMs = 152;
constexpr int ACC_WARPS = 8, PPC = PlanesPPC<N>::v, CPPC = CombinePPC<N>::v;

// How a call is cut: G instances at a time whose J plane spectra PW stay below
// 512 MB; of a pair's hemisphere nodes as many classes per launch as keep their
// Z and the table of e_2 e_3 below 1 GB each, and of the (instance, radial node)
// pairs as many as 1 GB of Z holds, spread evenly over the launches.
struct Cut {
  int G, classes, nodes, most, pairs;  // nodes, most: the most nodes and pairs of a launch
  int few;  // launches of at most so many pairs store their products first (k_q_plane)
  Cut(int B, int J, const QuadRule& r) {
    const size_t z = 2 * sizeof(ci64) * H, gb = (size_t)1 << 30;
    G = (int)std::min<size_t>(B, std::max<size_t>(1, (gb / 2) / (sizeof(ci64) * H * J)));
    int wide = 1;
    for (int c = 0; c < r.classes; ++c) wide = std::max(wide, r.class_begin[c + 1] - r.class_begin[c]);
    classes = (int)std::min<size_t>(r.classes, std::max<size_t>(1, std::min(gb / z, gb / (sizeof(ci64) * NC * J * wide))));
    nodes = std::min(r.M, classes * wide);
    const size_t all = (size_t)G * J;
    most = (int)std::min<size_t>(all, std::max<size_t>(1, gb / (z * classes)));
    const size_t launches = (all + most - 1) / most;
    pairs = (int)((all + launches - 1) / launches);
    // fewer blocks than SMs, and products of at most 1 GB
    few = (int)std::min<size_t>((kSMs - 1) / (N / GeoQ<N>::PPC), gb / (sizeof(i64) * n3 * nodes));
    few = std::min(few, most);
  }
};

// Sized by the most pairs of a launch, not by the even share: a smaller batch
// never needs more, so what was captured with a larger one keeps its buffer.
struct Buffers {
  ci64 *R, *F, *PW, *Z, *tab1, *tab;
  i64 *accG, *om3, *prod;
  float *rm, *BP;
  int *eR, *EF, *EPh, *EC, *bad, *EP, *accE, *prodE;
  size_t bytes;
  Buffers(void* base, size_t B, size_t J, const QuadRule& r, const Cut& c) {
    unsigned char* p = (unsigned char*)base;
    auto take = [&](auto*& ptr, size_t count) {
      ptr = (std::remove_reference_t<decltype(ptr)>)p;
      p += (count * sizeof(*ptr) + 255) / 256 * 256;
    };
    const bool rest = c.classes < r.classes;
    take(R, B * H);
    take(F, 2 * B * H);
    take(PW, c.G * J * H);
    take(Z, (size_t)c.most * c.classes * 2 * H);
    take(tab1, J * c.classes * N);
    take(tab, J * c.nodes * NC);
    take(accG, rest ? c.most * n3 : 0);
    take(om3, r.omega3 ? H : 0);
    take(BP, c.G * J * N);
    take(rm, B * BANDS * NC);
    take(eR, B * NC);
    take(EF, B);
    take(EPh, B * N);
    take(EC, 2 * B * NC);
    take(bad, B);
    take(EP, c.G * J * N);
    take(accE, rest ? (size_t)c.most * N * N : 0);
    take(prod, (size_t)c.few * c.nodes * n3);
    take(prodE, (size_t)c.few * c.nodes * N * N);
    bytes = (size_t)(p - (unsigned char*)base);
  }
};

template <typename K>
void smem_of(K kernel, size_t bytes) { raise_smem_limit((const void*)kernel, bytes); }

}  // namespace

size_t LBO_CAT(q_workspace_bytes_, LBO_FX_N)(int B, int J, const QuadRule& rule) {
  return Buffers(nullptr, B, J, rule, Cut(B, J, rule)).bytes;
}

lbo_status LBO_CAT(q_apply_, LBO_FX_N)(lbo_plan* p, const Tables& tb, const QuadRule& rule, const double* f, double* out,
                                       int B, void* ws) {
  cudaStream_t s = p->stream;
  const int J = p->J, M = rule.M;
  const Cut cut(B, J, rule);
  const Buffers w(ws, B, J, rule, cut);
  cudaError_t e = cudaMemsetAsync(w.bad, 0, sizeof(int) * B, s);
  if (e != cudaSuccess) return cuda_fail(e, "fixed-point flags");
  const double pi = 3.141592653589793238462643383279502884;
  // phi_j carries 4 pi^2 w_j B_j s_j / N^6 (one 1 / N^3 for T+ or T-, one for
  // the last transform); Eq. (2.14): 16 pi^2, and T+ T- a second 1 / N^3
  const double a0 = 4.0 / (double)n3, a0_lo = std::fma(-a0, (double)n3, 4.0) / (double)n3;
  int ke = 0;
  std::frexp(std::sqrt(rule.wmax * a0), &ke);  // the largest s_m is 2^ke times a number in [0.5, 1)
  const double a = std::scalbn(a0, -2 * ke), a_lo = std::scalbn(a0_lo, -2 * ke);
  int launches = 4;
  auto phases = [&](int first, int last) {  // classes [first, last)
    const int m0 = rule.class_begin[first];
    LBO_LAUNCH(p, "q_fx_phase_table", s, k_q_phase_table<N>, dim3(rule.class_begin[last] - m0, J), 256, 0, rule.gj, rule.sig,
               rule.wm, rule.node + m0, first, last - first, pi, 2.0 * p->L, a, a_lo, w.tab1, w.tab);
    launches += 1;
  };
  if (cut.classes == rule.classes) phases(0, rule.classes);
  const i64* omega = tb.omega;
  int omega_exp = tb.omega_exp;
  if (rule.omega3) {
    omega = w.om3;
    omega_exp = 61 - std::ilogb(rule.omega3_bound);
    LBO_LAUNCH(p, "q_fx_multipliers", s, k_q_position_multipliers<N>, 152, 256, 0, rule.omega3, omega_exp, w.om3);
    launches += 1;
  }
  // F = FFT(f); InvFFT_1(F omega)
  smem_of(k_fwd_planes<N, PPC>, Planes<N, PPC>::BYTES);
  LBO_LAUNCH(p, "q_fx_plane_fwd", s, (k_fwd_planes<N, PPC>), dim3(N / PPC, B, 1), (Planes<N, PPC>::THREADS),
             (Planes<N, PPC>::BYTES), f, (const double*)nullptr, 0, 0, w.F, w.EPh, w.bad);
  LBO_LAUNCH(p, "q_fx_axis1_head", s, k_axis1_head<N>, dim3((NC * T + 63) / 64, B, 2), 64, 0, w.F, w.EPh,
             (const ci64*)nullptr, (const int*)nullptr, omega, rule.omega3 ? 1 : 0, omega_exp, 0, w.R, w.eR, w.rm, w.EC, 0);
  LBO_LAUNCH(p, "q_fx_rescale", s, k_q_rescale<N>, dim3((NC + 63) / 64, B), 64, 0, w.R, w.eR, w.rm, w.EF);
  const bool carry = M >= 64;
  const auto k_whole = carry ? k_q_plane<N, true, WHOLE> : k_q_plane<N, false, WHOLE>;
  const auto k_sum = carry ? k_q_plane<N, true, SUM> : k_q_plane<N, false, SUM>;
  const auto k_products = k_q_plane<N, false, PRODUCTS>;
  for (const auto k : {k_whole, k_sum, k_products}) smem_of(k, GeoQ<N>::BYTES);
  smem_of(k_axis1_acc<N, ACC_WARPS>, acc_smem<N, ACC_WARPS>(256));
  // head room of the sum over m: products of at most 2^60, a sum below 2^63
  int guard = 0;
  while ((8 << guard) <= M) ++guard;
  for (int b0 = 0; b0 < B; b0 += cut.G) {
    const int n = std::min(cut.G, B - b0);
    const ci64* R = w.R + b0 * H;
    for (int q0 = 0; q0 < n * J; q0 += cut.pairs) {
      const int np = std::min(cut.pairs, n * J - q0);
      for (int c0 = 0; c0 < rule.classes; c0 += cut.classes) {
        const int c1 = std::min(c0 + cut.classes, rule.classes), m0 = rule.class_begin[c0], m1 = rule.class_begin[c1];
        if (cut.classes < rule.classes) phases(c0, c1);
        LBO_LAUNCH(p, "q_fx_axis1_phase", s, k_q_axis1<N>, dim3((NC * T + 31) / 32, c1 - c0, np), 32, 0, R, w.tab1, J, q0,
                   w.Z);
        const int planes = N / GeoQ<N>::PPC, mc = m1 - m0, f0 = c0 == 0 ? 1 : 0, l1 = c1 == rule.classes ? 1 : 0;
        auto plane = [&](const char* name, decltype(k_whole) k, dim3 grid, int share) {
          LBO_LAUNCH(p, name, s, k, grid, GeoQ<N>::THREADS, GeoQ<N>::BYTES, w.Z, w.tab, rule.node + m0, c0, c1 - c0,
                     w.EF + b0, J, mc, q0, f0, l1, guard, ke, share, w.prod, w.prodE, w.accG, w.accE, w.PW, w.EP, w.BP);
        };
        if (np > cut.few) {
          plane("q_fx_plane_prod", k_whole, dim3(planes, np), 0);
        } else {  // one wave of blocks
          const int wave = kSMs * std::max(GeoQ<N>::BLOCKS, 2), share = (mc * planes * np + wave - 1) / wave;
          plane("q_fx_plane_prod", k_products, dim3(planes, np, (mc + share - 1) / share), share);
          plane("q_fx_plane_sum", k_sum, dim3(planes, np), 0);
          launches += 1;
        }
        launches += 2;
      }
    }
    LBO_LAUNCH(p, "q_fx_axis1_fwd_acc", s, (k_axis1_acc<N, ACC_WARPS>), dim3((NC * T + 31) / 32, n), 32 * ACC_WARPS,
               (acc_smem<N, ACC_WARPS>(J)), w.PW, w.EP, w.BP, tb.phi, tb.phi_exp, tb.phi_max, w.F + b0 * H,
               w.EC + b0 * (size_t)NC, J);
    launches += 1;
  }
  using C = Combine<N, CPPC, QUAD>;
  smem_of(k_combine_planes<N, CPPC, QUAD>, C::BYTES);
  LBO_LAUNCH(p, "q_fx_combine", s, (k_combine_planes<N, CPPC, QUAD>), dim3(N / CPPC, B), C::THREADS, C::BYTES,
             (const double*)nullptr, f, w.F, w.EC, (const double*)nullptr, w.bad, out);
  p->last_launches += launches;
  e = cudaGetLastError();
  return e == cudaSuccess ? LBO_OK : cuda_fail(e, "fixed-point quadratic launch");
}

}  // namespace fx
}  // namespace lbo
