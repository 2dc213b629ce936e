// Kernels of Q(f,f) in the FP64 precision on the integer pipe: the M-point
// form of Eq. (2.14) in 64-bit block fixed point (fx64.cuh), with the head,
// accumulation and combination kernels of L[g] (lin_fx.cuh).
//
// For radial node j and hemisphere node m the two translated fields T+ =
// InvFFT(F E), T- = InvFFT(F conj E) are real, so one complex field Z = T+ + i T-
// carries both through the planes: no packing of columns or rows, and the
// product T+ T- is the product of a value's two parts.
//
//   k_q_phase_table  the per-axis phase factors of every (j, m)
//   k_q_rescale      F to one exponent per instance
//   k_q_axis1        the axis-1 transform of Z for every m of a chunk
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
  static constexpr int RS = T == 2 ? N + 2 : N + 1;  // row stride of the exchange buffer (Geo::RS)
  static constexpr size_t BYTES = (size_t)PPC * (sizeof(ci64) * N * RS + sizeof(i64) * N * N);
};

// tab[((j M + m) 3 + d) N + k] = exp(i alpha_d centred(k)) as two packed
// multipliers (1 = 2^62), alpha_d = pi g_j sigma_(m,d) / (2 L), at the Nyquist
// index cos(alpha_d N / 2), the average of the two images.  Axis 1 carries
// s_m = sqrt(w_m c): T+ T- then carries w_m and the constant c.
// grid = J M, block = 3 N.
template <int N>
__global__ void __launch_bounds__(3 * N) k_q_phase_table(const double* __restrict__ gj, const double* __restrict__ sig,
                                                         const double* __restrict__ wm, int M, double pi, double two_l,
                                                         double c, ci64* __restrict__ tab) {
  const int j = blockIdx.x / M, m = blockIdx.x % M, d = threadIdx.x / N, k = threadIdx.x % N;
  const double al = (pi * gj[j] / two_l) * sig[3 * m + d];
  double s = 0.0, co;
  if (k == N / 2) co = cos(al * (N / 2));
  else sincos(al * (double)centred<N>(k), &s, &co);
  const double f = d == 0 ? sqrt(wm[m] * c) : 1.0;
  tab[(size_t)blockIdx.x * 3 * N + threadIdx.x] =
      ci64{pack_mult(__double2ll_rn(co * f * 0x1p62)), pack_mult(__double2ll_rn(s * f * 0x1p62))};
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

__device__ __forceinline__ i64 raw_mult(i64 packed) {
  const Mult m = unpack_mult(packed);
  return ((i64)m.th << 32) + m.tl;
}
// (a, b) -> 4 a as a multiplier: products of two 2^62-scaled factors are 2^60-scaled
__device__ __forceinline__ SignedMult times4_mult(i64 a) { return signed_mult((i64)((u64)a << 2)); }

// Axis 1 of Z for the columns (k2, k3) of the half spectrum: Y+- =
// InvFFT_1(F E), InvFFT_1(F conj E); Z(i1, k2, k3) = Y+ + i Y-, and at the
// mirrored column Z(i1, -k2, -k3) = conj(Y+) + i conj(Y-).  One pass over F
// forms both products, F conj E waits in shared memory.  E(-k1) shares E(k1)'s
// four products.
// Z: [bj][m][i1][k2][k3] of the launch; bj0: its first (instance, node) pair.
// grid = (ceil(NC T / 32), mc, pairs), block = 32, shared memory V 32 words.
template <int N>
__global__ void __launch_bounds__(32) k_q_axis1(const ci64* __restrict__ R, const ci64* __restrict__ tab, int J, int M,
                                                int m0, int bj0, ci64* __restrict__ Z) {
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC, T = Geo<N>::T, V = Geo<N>::V;
  __shared__ ci64 S[V][32];
  const int lane = threadIdx.x, id = blockIdx.x * 32 + lane, h = T == 2 ? id & 1 : 0;
  const bool on = id / T < NC;
  const int col = on ? id / T : NC - 1, k2 = col / HC, k3 = col % HC;
  const int bj = bj0 + blockIdx.z, b = bj / J, j = bj % J, m = m0 + blockIdx.y;
  const ci64* mf = tab + (size_t)(j * M + m) * 3 * N;
  const ci64* src = R + (size_t)b * N * NC + col;
  const ci64 e2 = mf[N + k2], e3 = mf[2 * N + k3];
  const Mult e2x = unpack_mult(e2.x), e2y = unpack_mult(e2.y);
  const ci64 c0 = cmul_mult(SignedMult{e2x, e2x.th >> 31}, SignedMult{e2y, e2y.th >> 31},
                            ci64{raw_mult(e3.x), raw_mult(e3.y)});
  const SignedMult cx = times4_mult(c0.x), cy = times4_mult(c0.y);
  ci64 x[V];
  // value i at k1 = k: F E in x, F conj(E) in S
  auto product = [&](int i, int k, ci64 e) {
    const ci64 f = src[(size_t)k * NC];
    const SignedMult ex = times4_mult(e.x), ey = times4_mult(e.y);
    const i64 ac = mul_signed(f.x, ex.m, ex.neg), bd = mul_signed(f.y, ey.m, ey.neg);
    const i64 bc = mul_signed(f.y, ex.m, ex.neg), ad = mul_signed(f.x, ey.m, ey.neg);
    x[i] = ci64{ac - bd, bc + ad};
    S[i][lane] = ci64{ac + bd, bc - ad};
  };
  auto phase = [&](int k, ci64& e, ci64& em) {  // e1(k) c and conj(e1(k)) c
    const ci64 a = mf[k];
    const i64 ax = raw_mult(a.x), ay = raw_mult(a.y);
    const i64 xx = mul_signed(ax, cx.m, cx.neg), yy = mul_signed(ay, cy.m, cy.neg);
    const i64 xy = mul_signed(ax, cy.m, cy.neg), yx = mul_signed(ay, cx.m, cx.neg);
    e = ci64{xx - yy, xy + yx};
    em = ci64{xx + yy, xy - yx};
  };
  if constexpr (T == 1) {
#pragma unroll
    for (int k = 0; k <= N / 2; ++k) {
      ci64 e, em;
      phase(k, e, em);
      product(k, k, e);
      if (k > 0 && k < N / 2) product(N - k, N - k, em);
    }
  } else {
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int k = idx_parity<N>(i, h);
      ci64 e, em;
      phase(k, e, em);
      product(i, k, e);
    }
  }
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    dft_time<N, true>(x, h);
    if (pass == 0) {
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const ci64 v = S[i][lane];
        S[i][lane] = x[i];
        x[i] = v;
      }
    }
  }
  if (!on) return;
  ci64* dst = Z + ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * N * N * N;
  const size_t o = (size_t)k2 * N + k3, om = (size_t)((N - k2) % N) * N + (N - k3) % N;
  const bool mirror = k3 > 0 && k3 < N / 2;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const ci64 p = S[i][lane], q = x[i];
    const size_t plane = (size_t)idx_halves<N>(i, h) * N * N;
    dst[plane + o] = ci64{p.x - q.y, p.y + q.x};
    if (mirror) dst[plane + om] = ci64{p.x + q.y, q.x - p.y};
  }
}

// One plane i1 of one (instance, node) pair: Z of every m of the launch through
// the inverse axes 2 and 3, the sum over m of the products of its two parts
// (kept in shared memory at the largest exponent met so far, `guard` bits
// below a product's top), and after the last m the forward transforms of
// axes 3 and 2 of the sum, two rows per pencil, into PW[bj][i1].  Between the
// launches of a chunked m the sum rests in accG, accE.
// EF[b]: exponent of F; 2^ke: factor of the phase table; EP, BP as k_plane's.
// grid = (N / PPC, pairs), block = GeoQ<N>::THREADS.
template <int N>
__global__ void __launch_bounds__(GeoQ<N>::THREADS) k_q_plane(const ci64* __restrict__ Z, const int* __restrict__ EF,
                                                            int J, int mc, int bj0, int first, int last, int guard, int ke,
                                                            i64* __restrict__ accG, int* __restrict__ accE,
                                                            ci64* __restrict__ PW, int* __restrict__ EP,
                                                            double* __restrict__ BP) {
  using G = GeoQ<N>;
  constexpr int NC = Geo<N>::NC, T = Geo<N>::T, V = Geo<N>::V, TPP = G::TPP, RS = G::RS, FT = Geo<N>::TPP;
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
  int EA = kZeroExp;  // exponent of the sum
  if (first) {
#pragma unroll
    for (int i = 0; i < V; ++i) acc[idx_halves<N>(i, h) * N + q] = 0;
  } else {
#pragma unroll
    for (int i = 0; i < V; ++i) acc[idx_halves<N>(i, h) * N + q] = accG[pl * N * N + idx_halves<N>(i, h) * N + q];
    EA = accE[pl];
  }
  __syncthreads();
  const int E0 = EF[bj / J] + 2 + ke;  // products with the 2^62-scaled phases, 2^ke in axis 1's
  const PlaneThread t{pp, tp, h, q};
  const bool fwd = tp < FT;  // threads of the forward pencils
  ci64 x[V];
  int E = 0, s = 0;
  float top = 0.f;
  const int passes = 2 * mc + (last ? 2 : 0);
#pragma unroll 1
  for (int it = 0; it < passes; ++it) {
    const int kind = it >= 2 * mc ? 2 + (it - 2 * mc) : it & 1;
    if (kind == 0) {
      const ci64* src = Z + (((size_t)blockIdx.y * mc + (it >> 1)) * N + i1) * N * N + q;
#pragma unroll
      for (int i = 0; i < V; ++i) x[i] = src[(size_t)idx_parity<N>(i, h) * N];
      E = E0;
    } else if (kind == 1) {
#pragma unroll
      for (int i = 0; i < V; ++i) x[i] = Bs[q * RS + idx_parity<N>(i, h)];
    } else if (kind == 2) {
      // rows q and q + N/2 of the sum, parts exchanged
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const i64* a = acc + idx_halves<N>(i, h) * N;
        x[i] = fwd ? ci64{a[q + N / 2], a[q]} : ci64{0, 0};
      }
      E = EA == kZeroExp ? 0 : EA;
    } else if (fwd) {
      load_columns<N>(x, t, Bs);
    }
    top = __uint_as_float(group_max(__float_as_uint(pencil_sum<N>(abs_sum<V>(x))), kind));
    s = shift_for(top, kSumBits);
    shift_all<V>(x, s);
    E += s;
    pencil_inverse<N>(x, h, kind < 2);
    if (kind == 0) {
#pragma unroll
      for (int i = 0; i < V; ++i) Bs[idx_halves<N>(i, h) * RS + q] = x[i];
      if (!G::WARP && threadIdx.x < G::PPC) red[4 * G::PPC + threadIdx.x] = red[G::PPC + threadIdx.x] = 0;
      sync();
    } else if (kind == 1) {
      // T+ and T- to a top bit of 2^61, their product, and the sum over m
      unsigned m = top_bits<V>(x);
      m = group_max(m, 4);
      if (!G::WARP && threadIdx.x < G::PPC) red[threadIdx.x] = 0;
      const int l = m ? __clz(m) - 1 : 0;
      const int EPr = 2 * (E - l) + 64 + guard;
      if (EPr > EA) {  // the sum moves to the larger exponent
        const int d = min(EPr - EA, 63);
#pragma unroll
        for (int i = 0; i < V; ++i) acc[idx_halves<N>(i, h) * N + q] >>= d;
        EA = EPr;
      }
      const int d = min(EA - EPr + guard, 62);
      const i64 half = d > 0 ? (i64)1 << (d - 1) : 0;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const SignedMult a = signed_mult((i64)((u64)x[i].y << l));
        const i64 p = mul_signed_rounded((i64)((u64)x[i].x << l), a.m, a.neg);
        acc[idx_halves<N>(i, h) * N + q] += (p + half) >> d;
      }
      sync();
    } else if (kind == 2) {
      sync();
      if (fwd) store_rows<N>(x, t, Bs);
      sync();
    }
  }
  if (!last) {
#pragma unroll
    for (int i = 0; i < V; ++i) accG[pl * N * N + idx_halves<N>(i, h) * N + q] = acc[idx_halves<N>(i, h) * N + q];
    if (tp == 0) accE[pl] = EA;
    return;
  }
  if (!fwd) return;
  E -= 1;  // load_columns doubles
  store_spectrum<N>(x, t, PW + ((size_t)bj * N + i1) * NC);
  if (tp == 0) {
    EP[(size_t)bj * N + i1] = E;
    BP[(size_t)bj * N + i1] = plane_bound(top, E, s);
  }
}

}  // namespace fx
}  // namespace lbo
