// Kernels of Q(f,f) in the FP64 precision on the integer pipe: the M-point
// form of Eq. (2.14) in 64-bit block fixed point (fx64.cuh), with the head,
// accumulation and combination kernels of L[g] (lin_fx.cuh).
//
// For radial node j and hemisphere node m the two translated fields T+ =
// InvFFT(F E), T- = InvFFT(F conj E), E = e_1 e_2 e_3, are real, so one complex
// field Z = T+ + i T- carries both through the planes: no packing of columns or
// rows, and the product T+ T- is the product of a value's two parts.  Since
// E + i conj(E) = (1 + i) (Re E + Im E), Z = (1 + i) InvFFT(F (Re E + Im E)), and
// with e_1 = c1 + i s1, e_2 e_3 = c + i s the multiplier is
// c (c1 + s1) + s (c1 - s1): axis 1 only sees e_1, once for all nodes that share
// |sigma_1|, four nodes of a ring as a rule (sigma and -sigma exchange T+ and
// T-, so sigma_1 < 0 is taken as -sigma).
//
//   k_q_phase_table  the phase factors of every radial node and hemisphere node
//   k_q_rescale      F to one exponent per instance
//   k_q_axis1        the axis-1 transforms of Z for every class of nodes of a launch
//   k_q_plane        axes 2 and 3 of Z, sum_m w_m T+ T- on chip, and the
//                    forward transforms of axes 3 and 2 of the sum
#pragma once
#include "lin_fx.cuh"

namespace lbo {
namespace fx {

// Full complex planes: N pencils per axis.
template <int N>
struct GeoQ {
  static constexpr int T = Geo<N>::T, TPP = N * T;
  static constexpr bool WARP = TPP == 16 || TPP == 32;
  static constexpr int PPC = WARP ? 32 / TPP * 2 : (TPP == 24 ? 4 : 1);  // planes per block
  static constexpr int THREADS = TPP * PPC;
  static constexpr int BLOCKS = Geo<N>::V == 16 ? 384 / THREADS : 1;  // per SM: 12 warps of 168 registers
  static constexpr int RS = T == 2 ? N + 2 : N + 1;  // row stride of the exchange buffer (Geo::RS)
  static constexpr size_t BYTES = (size_t)PPC * (sizeof(ci64) * N * RS + sizeof(i64) * N * N);
};

// Phase factors of radial node j and the nodes (-sigma where sigma_1 < 0) of a
// launch, as packed multipliers.  e_d(k) = exp(i alpha_d centred(k)), alpha_d = pi g_j
// sigma_(m,d) / (2 L), at the Nyquist index cos(alpha_d N / 2), the average of
// the two images.  With e_1 = c + i s of a class, axis 1 takes
//   tab1[(j classes + class) N + k1] = ((c + s) s_m, (c - s) s_m), 1 = 2^61,
// where s_m = sqrt(w_m a): T+ T- then carries w_m and the constant a; the planes
//   tab[(j nodes + node) NC + (k2, k3)] = +- e_2(k2) e_3(k3), 1 = 2^62,
// negative for every other node: the product T+ T- is the same, and the mean
// error that the transforms' roundings leave in T+ and T- changes sides.  The
// large radial nodes, whose T+ and T- hardly meet, weigh it by some hundreds:
// without this and with ties all rounded up, the mass of Q+ was off by 1 to 5e-15
// at N = 16 to 32, now by 2e-16 to 2e-15 (FP64 kernels: up to 1e-15).
// a + a_lo: the constant in two parts.  s_m multiplies every mode of every radial
// node, so its rounding does not average out: the factors of axis 1 are formed
// in pairs of FP64 from the FP64 values of c, s and w_m.
// grid = (nodes, J), block = 256.
template <int N>
__global__ void __launch_bounds__(256) k_q_phase_table(const double* __restrict__ gj, const double* __restrict__ sig,
                                                       const double* __restrict__ wm, const int4* __restrict__ node,
                                                       int class0, int classes, double pi, double two_l, double a,
                                                       double a_lo,
                                                       ci64* __restrict__ tab1, ci64* __restrict__ tab) {
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC;
  __shared__ double2 e[2][N];
  const int j = blockIdx.y;
  const int4 nd = node[blockIdx.x];
  const double f = (pi * gj[j] / two_l);
  for (int t = threadIdx.x; t < 3 * N; t += 256) {
    const int d = t / N, k = t % N;
    if (d == 0 && !nd.w) continue;
    const double sg = sig[3 * nd.x + d], al = f * (d == 0 ? fabs(sg) : nd.z ? -sg : sg);
    double s = 0.0, co;
    if (k == N / 2) co = cos(al * (N / 2));
    else sincos(al * (double)centred<N>(k), &s, &co);
    if (d == 0) {
      const double w = wm[nd.x], x = __dmul_rn(w, a), xl = fma(w, a, -x) + w * a_lo;
      const double sm = sqrt(x), sl = (fma(-sm, sm, x) + xl) / (2.0 * sm);
      auto factor = [&](double b) {  // (co + b) s_m 2^61
        const double t = __dadd_rn(co, b), u = __dsub_rn(t, co);
        const double tl = __dadd_rn(__dsub_rn(co, __dsub_rn(t, u)), __dsub_rn(b, u));
        const double hi = __dmul_rn(t, sm), lo = fma(t, sm, -hi) + (t * sl + tl * sm);
        return pack_mult(__double2ll_rn(hi * 0x1p61) + __double2ll_rn(lo * 0x1p61));
      };
      tab1[((size_t)j * classes + nd.y - class0) * N + k] = ci64{factor(s), factor(-s)};
    } else {
      e[d - 1][k] = double2{co, s};
    }
  }
  __syncthreads();
  ci64* out = tab + ((size_t)j * gridDim.x + blockIdx.x) * NC;
  for (int t = threadIdx.x; t < NC; t += 256) {
    const double2 u = e[0][t / HC], v = e[1][t % HC];
    const double one = blockIdx.x % 2 ? -0x1p62 : 0x1p62;
    const i64 s = __double2ll_rn((u.x * v.y + u.y * v.x) * one);
    // the planes negate the words of s: its low one is not -2^31
    out[t] = ci64{pack_mult(__double2ll_rn((u.x * v.x - u.y * v.y) * one)),
                  pack_mult((unsigned)(u64)s == 0x80000000u ? s + 1 : s)};
  }
}

// The Eq. (2.16) loss multiplier (FP64, positions of fft.cuh along axes 1 and
// 2) as multipliers value 2^-e in natural order.  grid = any, block = 256.
template <int N>
__global__ void __launch_bounds__(256) k_q_position_multipliers(const double* __restrict__ om, int e,
                                                              i64* __restrict__ out) {
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC;
  for (int t = blockIdx.x * 256 + threadIdx.x; t < N * NC; t += gridDim.x * 256) {
    const int k1 = t / NC, k2 = (t % NC) / HC, k3 = t % HC;
    const double v = om[(size_t)pos_of_freq<N>(k1) * NC + pos_of_freq<N>(k2) * HC + k3];
    out[t] = pack_mult(__double2ll_rn(scalbn(v, e)));
  }
}

// R[b][k1][col] from its columns' exponents eR to the instance's EF[b], chosen
// so that sum(|re| + |im|) over every axis-1 pencil is at most 2^62.
// grid = (ceil(NC / 64), B), block = 64.
template <int N>
__global__ void __launch_bounds__(64) k_q_rescale(ci64* __restrict__ R, const int* __restrict__ eR,
                                                  const float* __restrict__ rm, int* __restrict__ EF) {
  constexpr int NC = Geo<N>::NC;
  __shared__ int top;
  const int b = blockIdx.y, col = blockIdx.x * 64 + threadIdx.x;
  if (threadIdx.x == 0) top = kZeroExp;
  __syncthreads();
  int e = kZeroExp;
  for (int c = threadIdx.x; c < NC; c += 64) {
    float s = 0x1p-30f;
    for (int k = 0; k < BANDS; ++k) s += rm[((size_t)b * BANDS + k) * NC + c];  // 2^-62 of the pencil's sum
    if (eR[b * NC + c] != kZeroExp) e = max(e, eR[b * NC + c] + ilogbf(s * 1.0001f) + 1);
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&top, e);
  __syncthreads();
  const int E = top == kZeroExp ? 0 : top;
  if (blockIdx.x == 0 && threadIdx.x == 0) EF[b] = E;
  if (col >= NC) return;
  const int d = E - eR[b * NC + col];
  ci64* p = R + (size_t)b * N * NC + col;
#pragma unroll 8
  for (int k = 0; k < N; ++k) {
    const ci64 v = p[(size_t)k * NC];
    p[(size_t)k * NC] = ci64{shift_any(v.x, d), shift_any(v.y, d)};
  }
}

// Axis 1 of Z for a class of hemisphere nodes, one thread per column (k2, k3)
// of the half spectrum: S+- = InvFFT_1(F (c +- s)), stored as (1 + i) S+- in
// Z[pair][class][i1][2][k2][k3]; real multipliers, two transforms for all nodes
// of the class.  F (c - s) waits in shared memory.
// Bound by the writes of Z (4.6 GB at N = 32, M = 32, 32 instances, 1.15 ms, 4.0
// TB/s); one pass per node instead, with its own axis-1 products and 17 GB of Z,
// took 7.3 ms.
// tab1: [j][classes][N]; bj0: the launch's first (instance, radial node) pair.
// grid = (ceil(NC T / 32), classes, pairs), block = 32, shared memory V 32 words.
template <int N>
__global__ void __launch_bounds__(32) k_q_axis1(const ci64* __restrict__ R, const ci64* __restrict__ tab1, int J,
                                                int bj0, ci64* __restrict__ Z) {
  constexpr int NC = Geo<N>::NC, T = Geo<N>::T, V = Geo<N>::V;
  __shared__ ci64 S[V][32];
  const int lane = threadIdx.x, id = blockIdx.x * 32 + lane, h = T == 2 ? id & 1 : 0;
  const bool on = id / T < NC;
  const int col = on ? id / T : NC - 1;
  const int bj = bj0 + blockIdx.z, b = bj / J, j = bj % J;
  const ci64* mf = tab1 + ((size_t)j * gridDim.y + blockIdx.y) * N;
  const ci64* src = R + (size_t)b * N * NC + col;
  ci64* dst = Z + ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * N * 2 * NC + col;
  ci64 x[V];
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const int k = idx_parity<N>(i, h);
    const ci64 f = src[(size_t)k * NC], e = mf[k];
    const SignedMult p = signed_of(e.x), q = signed_of(e.y);
    x[i] = ci64{mul_signed(f.x, p.m, p.neg), mul_signed(f.y, p.m, p.neg)};
    S[i][lane] = ci64{mul_signed(f.x, q.m, q.neg), mul_signed(f.y, q.m, q.neg)};
  }
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    dft_time<N, true>(x, h);
    if (on) {
#pragma unroll
      for (int i = 0; i < V; ++i)  // (1 + i) x
        dst[((size_t)idx_halves<N>(i, h) * 2 + pass) * NC] = ci64{x[i].x - x[i].y, x[i].x + x[i].y};
    }
    if (pass == 0) {
#pragma unroll
      for (int i = 0; i < V; ++i) x[i] = S[i][lane];
    }
  }
}

// One plane i1 of one (instance, radial node) pair: of every hemisphere node m of
// the launch, Z from its class (k_q_axis1) and e_2 e_3, the inverse axes 2 and 3, the sum over m of the products of its two parts
// (kept in shared memory, each row i2 at the largest exponent it met so far and
// `guard` bits below a product's top), and after the last m the forward transforms of
// axes 3 and 2 of the sum, two rows per pencil, into PW[bj][i1].  Between the
// launches of a chunked m the sum rests in accG, accE.
// node: the launch's mc nodes, of `classes` classes from class0 on.
// Bound by instruction issue: 54 % of the slots at 12 warps per SM (168
// registers; without the bound on registers, 8 warps, 14.8 ms), its integer pipe
// 55 %; stalls are fixed latencies and instruction fetch.  N = 32, M = 32, 32
// instances: 13.8 ms, where the kernel that read a ready Z per node took 10.1
// and left 7.3 to axis 1.  The exponents of the sum belong to a row, not to the
// plane: the largest T of a row needs a shuffle, that of a plane a barrier.
// CARRY, from 64 nodes on: the sum's unit is 2^guard of a product's, and products
// rounded each by itself would leave more than FP64 transforms do (N = 32, M =
// 288, hard spheres: up to 3.5 times their error); costs 1 %.
// A launch with few pairs would leave SMs idle while its blocks walk the nodes
// one after the other.  PRODUCTS takes `share` of them per block and stores
// the products (prod, prodE: [pair][node][i1]) that SUM then adds in the same
// order: the same bits.  N = 16, one instance, one radial node, M = 32: 206 us as
// a whole, 87 in two (153 in FP64 registers or shared memory).
// EF[b]: exponent of F; 2^ke: factor of the phase table; EP, BP as k_plane's.
// grid = (N / PPC, pairs), for PRODUCTS (N / PPC, pairs, ceil(mc / share)), block = GeoQ<N>::THREADS.
enum QMode { WHOLE, PRODUCTS, SUM };
template <int N, bool CARRY, int MODE>
__global__ void __launch_bounds__(GeoQ<N>::THREADS, GeoQ<N>::BLOCKS) k_q_plane(const ci64* __restrict__ Z,
                                                            const ci64* __restrict__ tab, const int4* __restrict__ node,
                                                            int class0, int classes, const int* __restrict__ EF,
                                                            int J, int mc, int bj0, int first, int last, int guard, int ke,
                                                            int share, i64* __restrict__ prod, int* __restrict__ prodE,
                                                            i64* __restrict__ accG, int* __restrict__ accE,
                                                            ci64* __restrict__ PW, int* __restrict__ EP,
                                                            float* __restrict__ BP) {
  using G = GeoQ<N>;
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC, T = Geo<N>::T, V = Geo<N>::V, TPP = G::TPP, RS = G::RS, FT = Geo<N>::TPP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[5 * G::PPC];
  const int pp = threadIdx.x / TPP, tp = threadIdx.x % TPP, h = T == 2 ? tp & 1 : 0, q = tp / T;
  const int i1 = blockIdx.x * G::PPC + pp, bj = bj0 + blockIdx.y;
  ci64* Bs = (ci64*)smem_raw + (size_t)pp * N * RS;
  i64* acc = (i64*)((ci64*)smem_raw + (size_t)G::PPC * N * RS) + (size_t)pp * N * N;  // [i3][i2]
  const size_t pl = (size_t)blockIdx.y * N + i1;
  auto sync = [&]() {
    if (G::WARP) __syncwarp();
    else __syncthreads();
  };
  // maxima over the plane's threads; the slots of a pass are cleared two syncs ahead
  auto group_max = [&](unsigned v, int slot) -> unsigned {
    if constexpr (G::WARP) {
#pragma unroll
      for (int o = TPP / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
      return v;
    } else {
      atomicMax(&red[slot * G::PPC + pp], v);
      __syncthreads();
      return red[slot * G::PPC + pp];
    }
  };
  if (threadIdx.x < 5 * G::PPC) red[threadIdx.x] = 0;
  int EA = kZeroExp;  // exponent of the pencil's sum
  if (first) {
#pragma unroll
    for (int i = 0; i < V; ++i) acc[idx_halves<N>(i, h) * N + q] = 0;
  } else if (MODE != PRODUCTS) {
#pragma unroll
    for (int i = 0; i < V; ++i) acc[idx_halves<N>(i, h) * N + q] = accG[pl * N * N + idx_halves<N>(i, h) * N + q];
    EA = accE[pl * N + q];
  }
  __syncthreads();
  // products with the 2^61-scaled axis-1 factors, which carry 2^ke, and with e_2 e_3
  const int E0 = EF[bj / J] + 5 + ke;
  const PlaneThread t{pp, tp, h, q};
  const bool fwd = tp < FT;  // threads of the forward pencils
  ci64 x[V];
  int E = 0, s = 0;
  float top = 0.f;
  // the sum += product(i) 2^(EPr - guard), i < V, of the thread's part of a row
  int carryE = kZeroExp;
  unsigned carry = 0;
  auto add = [&](int EPr, auto product) {
    if (EPr > EA) {  // the sum moves to the larger exponent; ties go up and down in turn
      const int d = min(EPr - EA, 63);
#pragma unroll
      for (int i = 0; i < V; ++i) {
        i64& a = acc[idx_halves<N>(i, h) * N + q];
        a = (a + ((i64)1 << (d - 1)) - i % 2) >> d;
      }
      EA = EPr;
    }
    const int d = min(EA - EPr + guard, 62);
    const i64 half = d > 0 ? (i64)1 << (d - 1) : 0;
    if (CARRY && d < 32) {
      // what a product loses in the sum's units goes to the row's next point, and
      // what is left at its end to the next node's
      unsigned c = (unsigned)half;
      if (carryE != kZeroExp) c = EPr >= carryE ? carry >> min(EPr - carryE, 31) : carry << (carryE - EPr);
      const unsigned mask = (1u << d) - 1;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const i64 p = product(i) + (i64)c;
        acc[idx_halves<N>(i, h) * N + q] += p >> d;
        c = (unsigned)(u64)p & mask;
      }
      carry = c;
      carryE = EPr;
    } else {
      const i64 down = d > 0 ? half - 1 : 0;
#pragma unroll
      for (int i = 0; i < V; ++i) acc[idx_halves<N>(i, h) * N + q] += (product(i) + (i % 2 ? down : half)) >> d;
      carryE = kZeroExp;
    }
  };
  if (MODE == SUM) {
#pragma unroll 1
    for (int m = 0; m < mc; ++m) {
      const size_t pm = ((size_t)blockIdx.y * mc + m) * N + i1;
#pragma unroll
      for (int i = 0; i < V; ++i) x[i].x = prod[pm * N * N + idx_halves<N>(i, h) * N + q];
      add(prodE[pm * N + q], [&](int i) { return x[i].x; });
    }
  }
  const int begin = MODE == PRODUCTS ? 2 * share * (int)blockIdx.z : (MODE == SUM ? 2 * mc : 0);
  const int passes = MODE == PRODUCTS ? min(begin + 2 * share, 2 * mc) : 2 * mc + (last ? 2 : 0);
#pragma unroll 1
  for (int it = begin; it < passes; ++it) {
    const int kind = it >= 2 * mc ? 2 + (it - 2 * mc) : it & 1;
    if (MODE != SUM && kind == 0) {
      // Z(k2, q) = c Z1 + s Z2, e_2 e_3 = c + i s.  Beyond the half spectrum,
      // from its mirrored entry: the parts of c Z2 - s Z1, exchanged.
      const int4 nd = node[it >> 1];
      const bool mir = q > N / 2;
      const size_t o = (mir ? (size_t)N * HC + N - q : (size_t)q);
      const int step = mir ? -HC : HC;
      const ci64* z = Z + ((((size_t)blockIdx.y * classes + nd.y - class0) * N + i1) * 2) * NC;
      const ci64 *z1 = z + (mir ? NC : 0) + o, *z2 = z + (mir ? 0 : NC) + o;
      const ci64* ph = tab + ((size_t)(bj % J) * mc + (it >> 1)) * NC + o;
      const int flip = mir ? -1 : 0;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int k = idx_parity<N>(i, h), r = (mir && k == 0 ? N : k) * step;
        const ci64 u = z1[r], v = z2[r], e = ph[r];
        const Mult c = unpack_mult(e.x), sw = unpack_mult(e.y), sn = Mult{(sw.th ^ flip) - flip, (sw.tl ^ flip) - flip};
        const i64 zx = mul_pair(u.x, c, v.x, sn), zy = mul_pair(u.y, c, v.y, sn);
        x[i] = ci64{mir ? zy : zx, mir ? zx : zy};
      }
      E = E0;
    } else if (MODE != SUM && kind == 1) {
#pragma unroll
      for (int i = 0; i < V; ++i) x[i] = Bs[q * RS + idx_parity<N>(i, h)];
    } else if (MODE != PRODUCTS && kind == 2) {
      // the rows to one exponent; rows q and q + N/2 of the sum, parts exchanged
      const int top = (int)group_max((unsigned)(EA - 2 * kZeroExp), 4) + 2 * kZeroExp, d = min(top - EA, 63);
#pragma unroll
      for (int i = 0; i < V; ++i) {
        i64& a = acc[idx_halves<N>(i, h) * N + q];
        a = shift_right(a, d);
      }
      EA = top;
      sync();
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const i64* a = acc + idx_halves<N>(i, h) * N;
        x[i] = fwd ? ci64{a[q + N / 2], a[q]} : ci64{0, 0};
      }
      E = EA == kZeroExp ? 0 : EA;
    } else if (MODE != PRODUCTS && fwd) {
      load_columns<N>(x, t, Bs);
    }
    top = __uint_as_float(group_max(__float_as_uint(pencil_sum<N>(abs_sum<V>(x))), kind));
    s = shift_for(top, kSumBits);
    shift_all<V>(x, s);
    E += s;
    pencil_inverse<N>(x, h, MODE == PRODUCTS || (MODE == WHOLE && kind < 2));
    if (MODE != SUM && kind == 0) {
#pragma unroll
      for (int i = 0; i < V; ++i) Bs[idx_halves<N>(i, h) * RS + q] = x[i];
      if (!G::WARP && threadIdx.x < G::PPC) red[G::PPC + threadIdx.x] = 0;
      sync();
      if (!G::WARP && threadIdx.x < G::PPC) red[threadIdx.x] = 0;
    } else if (MODE != SUM && kind == 1) {
      // T+ and T- of the pencil to at most 2^62, their product, and the sum over m
      int m = 0;
#pragma unroll
      for (int i = 0; i < V; ++i) m = max(m, max(abs((int)(x[i].x >> 32)), abs((int)(x[i].y >> 32))));
      if (T == 2) m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
      const int l = max(__clz(m) - 2, 0);
      const int EPr = m ? 2 * (E - l) + 64 + guard : kZeroExp;
      auto product = [&](int i) {
        const SignedMult a = signed_mult((i64)((u64)x[i].y << l));
        return mul_signed_rounded((i64)((u64)x[i].x << l), a.m, a.neg);
      };
      if (MODE == PRODUCTS) {
        const size_t pm = ((size_t)blockIdx.y * mc + (it >> 1)) * N + i1;
#pragma unroll
        for (int i = 0; i < V; ++i) prod[pm * N * N + idx_halves<N>(i, h) * N + q] = product(i);
        if (h == 0) prodE[pm * N + q] = EPr;
      } else {
        if constexpr (T == 2) {  // all products first: 1 to 3 % faster here, 2 % slower with all values in one thread
#pragma unroll
          for (int i = 0; i < V; ++i) x[i].x = product(i);
          add(EPr, [&](int i) { return x[i].x; });
        } else {
          add(EPr, product);
        }
      }
    } else if (MODE != PRODUCTS && kind == 2) {
      sync();
      if (fwd) store_rows<N>(x, t, Bs);
      sync();
    }
  }
  if (MODE == PRODUCTS) return;
  if (!last) {
#pragma unroll
    for (int i = 0; i < V; ++i) accG[pl * N * N + idx_halves<N>(i, h) * N + q] = acc[idx_halves<N>(i, h) * N + q];
    if (h == 0) accE[pl * N + q] = EA;
    return;
  }
  if (!fwd) return;
  E -= 1;  // load_columns doubles
  store_spectrum<N>(x, t, PW + ((size_t)bj * N + i1) * NC);
  if (tp == 0) {
    EP[(size_t)bj * N + i1] = E;
    BP[(size_t)bj * N + i1] = plane_bound(top);
  }
}

}  // namespace fx
}  // namespace lbo
