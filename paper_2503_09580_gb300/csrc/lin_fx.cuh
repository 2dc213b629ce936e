// Kernels of L[g] in the FP64 precision on the integer pipe: Algorithm 1 in
// 64-bit block fixed point (fx64.cuh).  Inputs, Maxwellians, the ratio r = g/M,
// the weights of u^_j and the final combination are FP64.
//
// A unit u = (instance b, radial node j) is one pass psi_j = InvFFT(u^_j r^),
// psi^_j = FFT(M^h psi_j).  All units of a group of instances run in one
// launch per kernel, so a single instance still fills the chip with its J
// nodes:
//
//   k_instance       per-instance tables (all exponentials)
//   k_mh             the table of M^h, the 1-D transforms of M's factors
//   k_fwd_planes     axes 3 and 2 of FFT(r) and FFT(g)
//   k_axis1_head     axis 1 of r^; InvFFT_1(FFT(g) omega), InvFFT_1(FFT(M) omega)
//   k_uhat           u^_j of a unit on its (N/2+1)^3 octant (three DCT-I passes)
//   k_unit_scale     the exponent of u^_j r^, from a bound of its axis-1 pencils
//   k_axis1_inv      psi_j <- InvFFT_1(u^_j r^)
//   k_plane          inverse axes 2 and 3, x M^h, forward axes 3 and 2, in place
//   k_axis1_acc      InvFFT_1(sum_j phi_j FFT_1(psi^_j))
//   k_combine_planes inverse axes 2 and 3 of L+, u and w, and L+ - u M - w g
//
// N = 32, 256 instances, J = 32: 5.6 ms (30.4 ms in FP64 registers, where the
// FP64 pipe was the bound).  Arithmetic alone would take 2.0 ms at the
// rate of register transforms, HBM 0.02 ms for inputs and outputs and about 1.5
// for the spectra that pass between the kernels.
//
// Layout: half spectra [u][i1 or k1][k2][k3], all indices natural, k3 =
// 0..N/2, ci64.  One thread transforms one pencil in registers (two threads,
// joined by shuffles, for N = 32, 48 and 64).
#pragma once
#include "fx64.cuh"
#include "lin_kernels.cuh"

namespace lbo {
namespace fx {

template <int N>
struct Geo {
  static constexpr int HC = N / 2 + 1, NC = N * HC;
  static constexpr int T = N >= 32 ? 2 : 1;  // threads per pencil
  static constexpr int V = N / T;           // values per thread
  // row stride of a plane in shared memory: odd, or 2 mod 8 for pairs of
  // threads, so that the row pass is free of bank conflicts
  static constexpr int RS = T == 2 ? HC + 1 : HC;
  static constexpr int PEN = N / 2;         // pencils per plane and pass
  static constexpr int TPP = PEN * T;       // threads per plane
  // the threads of a plane are consecutive lanes of one warp
  static constexpr bool WARP = TPP == 8 || TPP == 16 || TPP == 32;
};

// The axis-1 frequencies |k| in BANDS bands, [0, N/2) in quarters and N/2: the
// magnitudes of r^ and of u^_j that bound their products' pencil sums.
constexpr int BANDS = 5;
template <int N>
__device__ __forceinline__ constexpr int band(int k) { return k / (N / 8); }

constexpr int kSumBits = 60;       // sum(|re| + |im|) of a pencil before its transform, at most 2^60
constexpr int kZeroExp = -100000;  // exponent of an all-zero column

// Index of value i of thread h of a pencil: PARITY 2 i + h, HALVES the
// indices [h V/2, (h+1) V/2) of the lower and of the upper half.  A
// decimation-in-time transform takes PARITY to HALVES, one in frequency
// HALVES to PARITY; one thread per pencil holds all indices in order.
template <int N>
__device__ __forceinline__ int idx_parity(int i, int h) { return Geo<N>::T == 1 ? i : 2 * i + h; }
template <int N>
__device__ __forceinline__ int idx_halves(int i, int h) {
  constexpr int V = Geo<N>::V;
  return Geo<N>::T == 1 ? i : (i < V / 2 ? 0 : V) + h * (V / 2) + i % (V / 2);
}

__device__ __forceinline__ ci64 shfl_xor1(ci64 v) {
  return ci64{__shfl_xor_sync(0xffffffffu, v.x, 1), __shfl_xor_sync(0xffffffffu, v.y, 1)};
}
__device__ __forceinline__ ci64 select(bool c, ci64 a, ci64 b) { return ci64{c ? a.x : b.x, c ? a.y : b.y}; }

template <int N, bool INV, int I>
__device__ __forceinline__ void join_time(ci64 (&x)[N / 2], int h) {
  constexpr int V = N / 2;
  if constexpr (I < V / 2) {
    const ci64 lo = x[I], hi = x[V / 2 + I];
    const ci64 recv = shfl_xor1(select(h, lo, hi)), keep = select(h, hi, lo);
    const ci64 e = select(h, recv, keep);
    ci64 o = twiddle_n<I, N, INV>(select(h, keep, recv));
    o = select(h, quarter<INV>(o), o);
    x[I] = e + o;
    x[V / 2 + I] = e - o;
    join_time<N, INV, I + 1>(x, h);
  }
}
template <int N, bool INV, int I>
__device__ __forceinline__ void join_freq(ci64 (&x)[N / 2], int h) {
  constexpr int V = N / 2;
  if constexpr (I < V / 2) {
    const ci64 e = x[I] + x[V / 2 + I];
    ci64 o = twiddle_n<I, N, INV>(x[I] - x[V / 2 + I]);
    o = select(h, quarter<INV>(o), o);
    const ci64 recv = shfl_xor1(select(h, e, o)), keep = select(h, o, e);
    x[I] = select(h, recv, keep);
    x[V / 2 + I] = select(h, keep, recv);
    join_freq<N, INV, I + 1>(x, h);
  }
}
// PARITY -> HALVES
template <int N, bool INV>
__device__ __forceinline__ void dft_time(ci64 (&x)[Geo<N>::V], int h) {
  dft<Geo<N>::V, INV>(x);
  if constexpr (Geo<N>::T == 2) join_time<N, INV, 0>(x, h);
}
// HALVES -> PARITY
template <int N, bool INV>
__device__ __forceinline__ void dft_freq(ci64 (&x)[Geo<N>::V], int h) {
  if constexpr (Geo<N>::T == 2) join_freq<N, INV, 0>(x, h);
  dft<Geo<N>::V, INV>(x);
}

// sum(|re| + |im|) of a thread's values in units of 2^32, rounded up past the
// dropped low words and the float sum's rounding
template <int V>
__device__ __forceinline__ float abs_sum(const ci64 (&x)[V]) {
  float a = 0.f, b = 0.f;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    a += fabsf((float)(int)(x[i].x >> 32));
    b += fabsf((float)(int)(x[i].y >> 32));
  }
  return (a + b) * 1.00002f + (float)(2 * V);
}
// sum of a pencil's threads
template <int N>
__device__ __forceinline__ float pencil_sum(float v) {
  if constexpr (Geo<N>::T == 2) v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v;
}
// the right shift (negative: left) that brings a sum of `s` 2^32 to at most 2^BITS
__device__ __forceinline__ int shift_for(float s, int bits) {
  return (int)(__float_as_uint(s) >> 23) - 127 + 1 - (bits - 32);
}
__device__ __forceinline__ i64 shifted(i64 x, int s) { return s >= 0 ? x >> s : (i64)((u64)x << -s); }
// round(x 2^-s) for any s; the PTX shifts take amounts above 63 as 63 or 64
__device__ __forceinline__ i64 shift_any(i64 x, int s) {
  i64 r, l, half;
  const int right = max(s, 0);
  asm("shl.b64 %0, %1, %2;" : "=l"(half) : "l"(1LL), "r"(right));
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x + (i64)((u64)half >> 1)), "r"(right));
  asm("shl.b64 %0, %1, %2;" : "=l"(l) : "l"(r), "r"(max(-s, 0)));
  return right > 62 ? 0 : l;
}
// The values of a block by one shift.  Rounded, not floored: a mean error of
// half a unit over a field would meet in its zero mode, 2^7 times what
// random errors leave there; ties go up and down in turn for the same reason.
template <int V>
__device__ __forceinline__ void shift_all(ci64 (&x)[V], int s) {
  if (s > 0) {
    const i64 up = (i64)1 << (s - 1), down = up - 1;
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const i64 h = i % 2 ? down : up;
      x[i] = ci64{(x[i].x + h) >> s, (x[i].y + h) >> s};
    }
  } else if (s < 0) {
#pragma unroll
    for (int i = 0; i < V; ++i) x[i] = ci64{(i64)((u64)x[i].x << -s), (i64)((u64)x[i].y << -s)};
  }
}
// The same floored: where the following inverse transforms gather the mean
// error in the corner of the grid and M^h takes it away.
template <int V>
__device__ __forceinline__ void shift_floor(ci64 (&x)[V], int s) {
  if (s > 0) {
#pragma unroll
    for (int i = 0; i < V; ++i) x[i] = ci64{x[i].x >> s, x[i].y >> s};
  } else if (s < 0) {
#pragma unroll
    for (int i = 0; i < V; ++i) x[i] = ci64{(i64)((u64)x[i].x << -s), (i64)((u64)x[i].y << -s)};
  }
}
// round(x 2^-s), 0 <= s <= 63 (the PTX shift by 0xffffffff gives 0)
__device__ __forceinline__ i64 shift_right(i64 x, int s) {
  i64 half;
  asm("shl.b64 %0, %1, %2;" : "=l"(half) : "l"(1LL), "r"(s - 1));
  return (x + half) >> s;
}
// 2^-e as a float, 0 beyond its normal range (e >= 0)
__device__ __forceinline__ float exp2_neg(int e) { return e > 126 ? 0.f : __uint_as_float((unsigned)(127 - e) << 23); }
// x 2^e as FP64, rounded to nearest even; the integer pipe does it (a
// conversion of 64 bits and a product would take two slots of the FP64 pipe)
__device__ __forceinline__ double to_double(i64 x, int e) {
  const u64 m = x < 0 ? (u64)-x : (u64)x;
  const int l = __clzll((i64)m);
  const u64 n = m << (l & 63);  // top bit at 63
  const u64 r = n >> 11, mant = r + ((n & 0x7ff) + (r & 1) > 0x400);  // 53 bits, or 2^53
  const int ex = 63 - l + e + 1023;  // exponent field of the top bit
  if (m == 0) return 0.0;
  if (ex < 1 || ex > 2045) return scalbn((double)x, e);
  const u64 bits = ((u64)(unsigned)(ex - 1) << 52) + mant;
  return __longlong_as_double((i64)(x < 0 ? bits | 0x8000000000000000ULL : bits));
}
// round(v 2^-E), ties away from zero; |v 2^-E| < 2^62, v finite
__device__ __forceinline__ i64 to_fixed(double v, int E) {
  const u64 w = (u64)__double_as_longlong(v);
  const int f = (int)(w >> 52) & 0x7ff;
  const u64 m = (w & 0x000fffffffffffffULL) | (f ? 0x0010000000000000ULL : 0);
  const int s = (f ? f : 1) - 1075 - E;  // v = m 2^(s + E)
  u64 y;
  if (s >= 0) y = s > 10 ? 0 : m << s;
  else y = s < -54 ? 0 : ((m >> (-s - 1)) + 1) >> 1;
  return (i64)w < 0 ? -(i64)y : (i64)y;
}

// ------------------------------------------------------------ tables
// Per instance, once per application: everything that takes an exponential or
// a division, so that the kernels with many blocks only load.  Offsets in
// doubles from inst[b]:
template <int N>
struct Inst {
  static constexpr int EM = 0;           // [3][N] factors of M (fill_maxwellian_tables)
  static constexpr int EI = 3 * N;       // [3][N] factors of 1/M (fill_ratio_tables)
  static constexpr int SQ = 6 * N;       // [3][N] (v_i - u_d)^2, every operation rounded
  static constexpr int EH = 9 * N;       // [3][N] factors of |M^h|
  static constexpr int MG = 12 * N;      // [N/2+1] exp(-(i h)^2 / theta), then |rho| (pi theta)^(-3/2)
  static constexpr int DSTAR = 12 * N + N / 2 + 2;  // the cut-off's distance (fill_ratio_tables)
  static constexpr int SIZE = DSTAR + 1;
};

// inst as above; em[b][i1]: exponent of the plane i1 of M^h (see k_mh).
// |rho| in M^h and in the weights of u^_j: multipliers are not negative, and
// L^+ has the product of the two.
// bad[b]: 1 where a factor is not finite (the output is then NaN).
// grid = B, block = kInstanceThreads.
template <int N>
constexpr int kInstanceThreads = (9 * N + N / 2 + 1 + 3 + 31) / 32 * 32;
template <int N>
__global__ void __launch_bounds__(kInstanceThreads<N>) k_instance(const double* __restrict__ params, double h, double log_inv_eps,
                                                  double* __restrict__ inst, int* __restrict__ em1,
                                                  int* __restrict__ bad) {
  constexpr int HC = Geo<N>::HC;
  // tasks: every exponential, power and the cut-off's distance in a thread of
  // its own, side by side, then the products
  constexpr int TI = 3 * N, TH = 6 * N, TG = 9 * N, TP = 9 * N + HC;  // ends of M, 1/M, M^h, M^g
  static_assert(TP + 3 <= kInstanceThreads<N>, "one thread per task");
  __shared__ double pre[2];
  __shared__ unsigned long long top[3];  // largest factor of M^h per axis (bits of a positive double)
  const int b = blockIdx.x, t = threadIdx.x;
  const InstanceParams q = load_params(params, b);
  double* I = inst + (size_t)b * Inst<N>::SIZE;
  if (t < 3) top[t] = 0;
  double e = 0.0;
  const int ti = t % (3 * N), d = ti / N;  // axis and index of the factor tasks
  if (t < TG) {
    const double ud = d == 0 ? q.u1 : (d == 1 ? q.u2 : q.u3), vi = __dmul_rn((double)(ti % N - N / 2), h);
    const double dv = __dsub_rn(vi, ud);
    if (t < TI) {  // as fill_maxwellian_tables
      const double v = (double)(ti % N - N / 2) * h - ud;
      e = exp(-(v * v) / (2.0 * q.theta));
    } else if (t < TH) {  // as fill_ratio_tables
      e = exp(__dmul_rn(dv, dv) / (2.0 * q.theta));
      I[Inst<N>::SQ + ti] = sq_rn(dv);
    } else {  // as fill_mh_tables
      const double v = (double)(ti % N - N / 2) * h - ud;
      e = exp(-(v * v) / q.theta);
    }
  } else if (t < TP) {
    const double x = (t - TG) * h;
    I[Inst<N>::MG + t - TG] = exp(-(x * x) / q.theta);
  } else if (t == TP) {
    pre[0] = q.rho * pow(2.0 * 3.141592653589793 * q.theta, -1.5);
  } else if (t == TP + 1) {
    pre[1] = q.rho * pow(3.141592653589793 * q.theta, -1.5);
    I[Inst<N>::MG + HC] = fabs(pre[1]);
  } else if (t == TP + 2) {
    I[Inst<N>::DSTAR] = cut_distance(q.theta, log_inv_eps);
  }
  __syncthreads();
  if (t < TI) {
    if (d == 0) e *= pre[0];
    I[Inst<N>::EM + ti] = e;
    if (!isfinite(e)) atomicOr(bad + b, 1);
  } else if (t < TH) {
    if (d == 0) e /= pre[0];
    I[Inst<N>::EI + ti] = e;
  } else if (t < TG) {
    if (d == 0) e *= pre[1];
    e = fabs(e);
    if (!isfinite(e)) atomicOr(bad + b, 1);
    else atomicMax(&top[d], (unsigned long long)__double_as_longlong(e));
    I[Inst<N>::EH + ti] = isfinite(e) ? e : 0.0;
  }
  __syncthreads();
  if (t >= TH && t < TH + N) {
    const double m = (e * __longlong_as_double((i64)top[1])) * __longlong_as_double((i64)top[2]);
    // a plane where every entry underflows has no magnitude: its bound must not
    // set the exponent of the sum over the planes
    em1[b * N + ti] = !(m > 0.0) ? kZeroExp : (isfinite(m) ? ilogb(m) - 59 : 0);
  }
}

// |M^h(v)| = mh[b][i1][i3][i2] 2^em[b][i1] as a multiplier (pack_finer), every
// plane's largest entry in [2^59, 2^60).  i2 runs fastest so that the row
// threads of k_plane read consecutive entries.  The last block of an instance:
// MH[b][d][k] 2^eM[b][d] = the 1-D transforms of M's factors, whose product is
// FFT(M).
// grid = (N + 1, B), block = 256.
template <int N>
__global__ void __launch_bounds__(256) k_mh(const double* __restrict__ inst, const int* __restrict__ em,
                                            i64* __restrict__ mh, ci64* __restrict__ MH, int* __restrict__ eM) {
  const int b = blockIdx.y, i1 = blockIdx.x, t = threadIdx.x;
  const double* I = inst + (size_t)b * Inst<N>::SIZE;
  if (i1 < N) {
    const double* eh = I + Inst<N>::EH;
    const int E = em[b * N + i1];
    i64* dst = mh + ((size_t)b * N + i1) * N * N;
    for (int e = t; e < N * N; e += 256)
      dst[e] = pack_finer(to_fixed((eh[i1] * eh[N + e % N]) * eh[2 * N + e / N], E));
    return;
  }
  constexpr int T = Geo<N>::T, V = Geo<N>::V;
  if (t >= 32) return;
  const int h = T == 2 ? t & 1 : 0, d = min(t / T, 2);
  const double* m = I + Inst<N>::EM + d * N;
  unsigned top = 0;
#pragma unroll 8
  for (int i = 0; i < N; ++i) top = max(top, (unsigned)__double2hiint(m[i]) & 0x7fffffffu);
  const bool fin = top < 0x7ff00000u;
  const int E = (int)(top >> 20) - 1023 - 57;  // the largest factor in [2^57, 2^58)
  ci64 x[V];
#pragma unroll
  for (int i = 0; i < V; ++i) x[i] = ci64{fin ? to_fixed(m[idx_parity<N>(i, h)], E) : 0, 0};
  const int s = shift_for(pencil_sum<N>(abs_sum<V>(x)), kSumBits);
  shift_all<V>(x, s);
  dft_time<N, false>(x, h);
  if (t < 3 * T) {
#pragma unroll
    for (int i = 0; i < V; ++i) MH[((size_t)b * 3 + d) * N + idx_halves<N>(i, h)] = x[i];
    if (h == 0) eM[b * 3 + d] = E + s;
  }
}

// ------------------------------------------------------------ u^_j
// One unit's octant U[u][k1][k2][k3] 2^eU[u] = FFT(M^g phit_j), scaled to a
// largest entry in [2^61, 2^62), and ub[u][band][k2][k3], its largest magnitude
// over a band of k1 times 2^-62: the weight in FP64 as k_uhat_planes forms it,
// then the three DCT-I passes, each after a shift by its own largest pencil
// sum.  One thread per pencil, the octant in shared memory; at N = 64, where
// that takes 287 KB, a cluster of two blocks holds half of the planes d1 each
// and reads the other's for axis 1.
// Bound by latencies between its three passes (one block of (N/2+1)^2 pencils
// holds the whole octant); N = 32, 256 instances: 0.60 ms, 3.0 in FP64.  At N =
// 64 the pencils of 33 values spill 1 to 2 KB; a cluster of four instead of two
// took 127 us where two take 98.
// grid = (CL J, B), cluster CL, block = BLOCK, shared memory SMEM.
template <int N>
struct Octant {
  static constexpr int HC = Geo<N>::HC, HC2 = HC * HC, HC3 = HC2 * HC;
  static constexpr int CL = sizeof(i64) * HC3 > 200 * 1024 ? 2 : 1;
  static constexpr int D1 = (HC + CL - 1) / CL;       // planes d1 of a block
  static constexpr int PENCILS = (HC2 + CL - 1) / CL;  // axis-1 pencils of a block
  static constexpr int BLOCK = (PENCILS + 31) / 32 * 32;
  static constexpr size_t SMEM = sizeof(i64) * D1 * HC2;
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_map(const void* p, int rank) {  // shared::cluster address of p in block `rank`
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ i64 cluster_load(unsigned a) {
  i64 v;
  asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(a));
  return v;
}
// *red becomes the maximum over the unit's threads (every block's copy)
template <int CL>
__device__ __forceinline__ unsigned unit_max(unsigned v, unsigned* red) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) {
    if (CL == 1) {
      atomicMax(red, v);
    } else {
      for (int r = 0; r < CL; ++r)
        asm volatile("red.shared::cluster.max.u32 [%0], %1;" ::"r"(cluster_map(red, r)), "r"(v) : "memory");
    }
  }
  if (CL == 1) __syncthreads();
  else cluster_sync();
  return *red;
}

template <int H, int STRIDE>
__device__ __forceinline__ float dct_abs_sum(const i64* x) {
  float s = 0.f;
#pragma unroll
  for (int d = 0; d <= H; ++d) s += (d == 0 || d == H ? 1.f : 2.f) * fabsf((float)(int)(x[d * STRIDE] >> 32));
  return s * 1.00002f + (float)(2 * H);
}
template <int H>
__device__ __forceinline__ void dct_shifted(i64 (&x)[H + 1], int s) {  // the shift rounds: no bias of the sums
  const i64 half = s > 0 ? (i64)1 << (s - 1) : 0;
#pragma unroll
  for (int d = 0; d <= H; ++d) x[d] = shifted(x[d] + half, s);
  dct1<H, 1>(x);
}

template <int N>
__global__ void __launch_bounds__(Octant<N>::BLOCK) k_uhat(const double* __restrict__ inst,
                                                         const double* __restrict__ phit, i64* __restrict__ U,
                                                         int* __restrict__ eU, float* __restrict__ ub,
                                                         int* __restrict__ bad, int J) {
  using O = Octant<N>;
  constexpr int H = N / 2, HC = O::HC, HC2 = O::HC2, HC3 = O::HC3, CL = O::CL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  i64* W = (i64*)smem_raw;  // [d1 - first][d2][d3]
  __shared__ double mg[HC + 1], row[O::D1 * HC];
  __shared__ unsigned red[5];
  const int rank = CL == 1 ? 0 : blockIdx.x % CL, j = blockIdx.x / CL, b = blockIdx.y, t = threadIdx.x;
  const int first = rank * O::D1, planes = min(O::D1, HC - first);
  const size_t u = (size_t)b * J + j;
  if (t <= HC) mg[t] = inst[(size_t)b * Inst<N>::SIZE + Inst<N>::MG + t];
  if (t < 5) red[t] = 0;
  __syncthreads();
  for (int e = t; e < planes * HC; e += O::BLOCK) row[e] = mg[HC] * (mg[first + e / HC] * mg[e % HC]);
  if (CL == 1) __syncthreads();
  else cluster_sync();  // red is ready in both blocks
  unsigned top = 0;
  for (int e = t; e < planes * HC2; e += O::BLOCK) {
    const int d3 = e % HC, r = e / HC, d2 = r % HC, d1 = first + r / HC;
    const i64 w = __double_as_longlong((row[r] * mg[d3]) * phit[(((size_t)j * N + d1) * N + d2) * N + d3]);
    W[e] = w;
    top = max(top, (unsigned)(w >> 32) & 0x7fffffffu);
  }
  top = unit_max<CL>(top, &red[0]);
  int E = (int)(top >> 20) - 1023 - 57;  // the largest weight in [2^57, 2^58)
  const bool fin = top < 0x7ff00000u;
  if (!fin && t == 0) atomicOr(bad + b, 1);
  for (int e = t; e < planes * HC2; e += O::BLOCK) W[e] = fin ? to_fixed(__longlong_as_double(W[e]), E) : 0;
  __syncthreads();
  i64 x[HC];
  // axes 3 and 2 of the block's planes, in place
#pragma unroll 1
  for (int axis = 3; axis >= 2; --axis) {
    const int stride = axis == 3 ? 1 : HC;
    float m = 0.f;
    for (int q = t; q < planes * HC; q += O::BLOCK) {
      const i64* p = W + (axis == 3 ? q * HC : (q / HC) * HC2 + q % HC);
#pragma unroll
      for (int d = 0; d < HC; ++d) x[d] = p[d * stride];
      m = fmaxf(m, dct_abs_sum<H, 1>(x));
    }
    const int s = shift_for(__uint_as_float(unit_max<CL>(__float_as_uint(m), &red[axis - 1])), kSumBits);
    for (int q = t; q < planes * HC; q += O::BLOCK) {
      i64* p = W + (axis == 3 ? q * HC : (q / HC) * HC2 + q % HC);
#pragma unroll
      for (int d = 0; d < HC; ++d) x[d] = p[d * stride];
      dct_shifted<H>(x, s);
#pragma unroll
      for (int d = 0; d < HC; ++d) p[d * stride] = x[d];
    }
    E += s;
    if (CL == 1) __syncthreads();
    else cluster_sync();
  }
  // axis 1: one pencil per thread, kept in registers for the final scale
  const int q = rank * O::PENCILS + t;
  const bool on = t < O::PENCILS && q < HC2;
#pragma unroll
  for (int d = 0; d < HC; ++d) {
    if (CL == 1) x[d] = on ? W[d * HC2 + q] : 0;
    else x[d] = on ? cluster_load(cluster_map(W + (d % O::D1) * HC2 + q, d / O::D1)) : 0;
  }
  const int s = shift_for(__uint_as_float(unit_max<CL>(__float_as_uint(dct_abs_sum<H, 1>(x)), &red[3])), kSumBits);
  dct_shifted<H>(x, s);
  E += s;
  unsigned m = 0;
#pragma unroll
  for (int d = 0; d < HC; ++d) m = max(m, (unsigned)((x[d] ^ (x[d] >> 63)) >> 31));
  m = unit_max<CL>(m, &red[4]);  // also: every block has read its neighbour's planes
  const int l = m ? __clz(m) - 1 : 0;  // left shift to a top bit of 2^61
  if (on) {
    i64* dst = U + u * HC3 + q;
    unsigned top[BANDS] = {};
#pragma unroll
    for (int d = 0; d < HC; ++d) {
      const i64 v = (i64)((u64)x[d] << l);
      dst[d * HC2] = v;
      top[band<N>(d)] = max(top[band<N>(d)], (unsigned)((v ^ (v >> 63)) >> 32));
    }
#pragma unroll
    for (int d = 0; d < BANDS; ++d) ub[(u * BANDS + d) * HC2 + q] = ((float)top[d] + 1.f) * (1.00001f * 0x1p-30f);
  }
  if (t == 0 && rank == 0) eU[u] = E - l;
}

// ------------------------------------------------------------ exponents
// EA[u]: the exponent of the products u^_j r^ of unit u, such that
// sum(|re| + |im|) over every axis-1 pencil is at most 2^60; from the largest
// sum over the bands of ub (k_uhat) times rm (k_axis1_head) over the columns.
// Bands, not one bound per column: u^_j falls steeply, and the bits that one
// bound of |u^_j| |r^| gives away are error.  Latency: 17 us at N = 32 for 86
// instances, 9 us for 8.
// grid = (J, B), block = 256.
template <int N>
__global__ void __launch_bounds__(256) k_unit_scale(const float* __restrict__ ub, const int* __restrict__ eU,
                                                    const float* __restrict__ rm, const int* __restrict__ eR,
                                                    int* __restrict__ EA, int J) {
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC;
  __shared__ int top;
  __shared__ unsigned red;
  const int j = blockIdx.x, b = blockIdx.y, t = threadIdx.x;
  const size_t u = (size_t)b * J + j;
  if (t == 0) {
    top = kZeroExp;
    red = 0;
  }
  __syncthreads();
  int e = kZeroExp;
  for (int c = t; c < NC; c += 256) e = max(e, eR[b * NC + c]);
  e = __reduce_max_sync(0xffffffffu, e);
  if ((t & 31) == 0) atomicMax(&top, e);
  __syncthreads();
  const int et = top;
  float f = 0.f;
  for (int c = t; c < NC; c += 256) {
    const int k2 = c / HC, k3 = c % HC, a2 = k2 <= N / 2 ? k2 : N - k2;
    const float* r = rm + (size_t)b * BANDS * NC + c;
    const float* uc = ub + u * BANDS * HC * HC + a2 * HC + k3;
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < BANDS; ++k) s += uc[(size_t)k * HC * HC] * r[(size_t)k * NC];
    const int d = et - eR[b * NC + c];
    if (d < 120) f = fmaxf(f, s * __uint_as_float((unsigned)(127 - d) << 23));
  }
  f = f * 1.0001f + 0x1p-60f;
  atomicMax(&red, __float_as_uint(f));
  __syncthreads();
  if (t == 0) {
    const int lg = (int)(red >> 23) - 127 + 1;  // f < 2^lg
    EA[u] = et == kZeroExp ? 0 : eU[u] + et + 124 + lg - kSumBits;
  }
}

// ------------------------------------------------------------ axis 1, inverse
// W[u][i1][col] 2^EA[u] = InvFFT_1(u^_j r^).  The octant's entries carry the
// shift from the column's exponent to EA, the data are not shifted.
// Bound by load latency and issue: two threads per pencil and blocks of 64 put
// 12 warps on an SM at N = 32.  256 instances: 0.92 ms, 4.3 in FP64; r^ kept in
// registers over four nodes took as long (32.4 against 32.2 us per 7 instances).
// grid = (ceil(NC T / 64), J, B), block = 64.
template <int N>
__global__ void __launch_bounds__(64) k_axis1_inv(const ci64* __restrict__ R, const int* __restrict__ eR,
                                                  const i64* __restrict__ U, const int* __restrict__ eU,
                                                  const int* __restrict__ EA, ci64* __restrict__ W) {
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC, T = Geo<N>::T, V = Geo<N>::V;
  const int j = blockIdx.y, b = blockIdx.z, id = blockIdx.x * 64 + threadIdx.x, h = T == 2 ? id & 1 : 0;
  const bool on = id / T < NC;
  const int col = on ? id / T : NC - 1;
  const size_t u = (size_t)b * gridDim.y + j;
  const int k2 = col / HC, k3 = col % HC, a2 = k2 <= N / 2 ? k2 : N - k2;
  const i64* uc = U + u * HC * HC * HC + a2 * HC + k3;
  const ci64* src = R + (size_t)b * N * NC + col;
  // U' = U 2^sh; beyond the headroom of this pencil's entries (r^ tiny where
  // u^ is large) the rest of the shift is applied to the products
  int sh = 64 + eR[b * NC + col] + eU[u] - EA[u], rest = 0;
  sh = sh < -63 ? -63 : sh;
  if (sh > 0) {
    unsigned m = 1;
    for (int k = 0; k < HC; ++k) {
      const i64 v = uc[(size_t)k * HC * HC];
      m = max(m, (unsigned)((v ^ (v >> 63)) >> 31));
    }
    const int room = max(__clz(m) - 1, 0);
    rest = min(max(sh - room, 0), 62);
    sh = min(sh, room);
  }
  ci64 x[V];
#pragma unroll
  for (int i = 0; i < V; ++i) x[i] = src[(size_t)idx_parity<N>(i, h) * NC];
  if constexpr (T == 1) {
#pragma unroll
    for (int k = 0; k <= N / 2; ++k) {
      const Mult m = split_mult(shifted(uc[(size_t)k * HC * HC], -sh));
      const int neg = m.th >> 31;
      x[k] = ci64{mul_signed(x[k].x, m, neg), mul_signed(x[k].y, m, neg)};
      if (k > 0 && k < N / 2) x[N - k] = ci64{mul_signed(x[N - k].x, m, neg), mul_signed(x[N - k].y, m, neg)};
    }
  } else {
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int k = idx_parity<N>(i, h);
      const Mult m = split_mult(shifted(uc[(size_t)(k <= N / 2 ? k : N - k) * HC * HC], -sh));
      const int neg = m.th >> 31;
      x[i] = ci64{mul_signed(x[i].x, m, neg), mul_signed(x[i].y, m, neg)};
    }
  }
  if (rest > 0) shift_all<V>(x, -rest);
  dft_time<N, true>(x, h);
  if (on) {
    ci64* dst = W + u * N * NC + col;
#pragma unroll
    for (int i = 0; i < V; ++i) dst[(size_t)idx_halves<N>(i, h) * NC] = x[i];
  }
}

// ------------------------------------------------------------ planes
// planes per block of the L kernels, and of the combination (up to three
// fields per block)
template <int N>
struct PlanesPPC { static constexpr int v = N == 64 ? 1 : (N == 48 ? 2 : (N == 32 ? 4 : 8)); };
template <int N>
struct CombinePPC { static constexpr int v = N == 32 ? 2 : (N < 32 ? 4 : 1); };
template <int N, int PPC>
struct Planes {
  static constexpr int THREADS = Geo<N>::TPP * PPC;
  // blocks per SM asked of the compiler: 168 registers where a thread holds 16 values
  static constexpr int BLOCKS = Geo<N>::V == 16 ? 384 / THREADS : 1;
  static constexpr size_t BYTES = sizeof(ci64) * (size_t)PPC * N * Geo<N>::RS;
};

// Barrier and maximum over the threads of a plane.  Where a plane is part of
// one warp no block barrier is needed.
template <int N>
__device__ __forceinline__ void plane_sync() {
  if constexpr (Geo<N>::WARP) __syncwarp();
  else __syncthreads();
}
template <int N>
__device__ __forceinline__ float plane_max(float v, unsigned* slot) {
  if constexpr (Geo<N>::WARP) {
#pragma unroll
    for (int o = Geo<N>::TPP / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
  } else {
    atomicMax(slot, __float_as_uint(v));
    __syncthreads();
    return __uint_as_float(*slot);
  }
}
// Column pencil q of a plane: q = 0 is the pair of columns 0 and N/2, whose
// transforms along axis 2 are of real sequences, packed as x_0 + i x_(N/2);
// q > 0 is column k3 = q.  Row pencil q holds the rows q and q + N/2 as
// x_q + i x_(q+N/2) (an odd row stride keeps consecutive q on distinct
// shared-memory banks).  Every pass: load, shift by the plane's largest pencil
// sum, transform, store.
struct PlaneThread {
  int pp, tp, h, q;  // plane of the block, thread of the plane, thread of the pencil, pencil
};
template <int N>
__device__ __forceinline__ PlaneThread plane_thread(int t) {
  constexpr int T = Geo<N>::T, TPP = Geo<N>::TPP;
  const int tp = t % TPP;
  return PlaneThread{t / TPP, tp, T == 2 ? tp & 1 : 0, tp / T};
}

// shift by the plane's largest pencil sum (returned); E is the values' exponent
template <int N>
__device__ __forceinline__ float normalise(ci64 (&x)[Geo<N>::V], int& s, int& E, unsigned* slot, bool round) {
  const float top = plane_max<N>(pencil_sum<N>(abs_sum<Geo<N>::V>(x)), slot);
  s = shift_for(top, kSumBits);
  if (round) shift_all<Geo<N>::V>(x, s);
  else shift_floor<Geo<N>::V>(x, s);
  E += s;
  return top;
}

// The transforms of a plane run in a loop with one copy of the pencil
// transform: four inlined copies (158 KB of code) spent 46 % of the issue
// slots on instruction fetches.  A forward transform is the inverse one of the
// values with their parts exchanged.
template <bool SWAP>
__device__ __forceinline__ ci64 parts(i64 re, i64 im) { return SWAP ? ci64{im, re} : ci64{re, im}; }

// inverse transform, PARITY -> HALVES (time) or HALVES -> PARITY
template <int N>
__device__ __forceinline__ void pencil_inverse(ci64 (&x)[Geo<N>::V], int h, bool time) {
  if constexpr (Geo<N>::T == 2) {
    if (!time) join_freq<N, true, 0>(x, h);
  }
  dft<Geo<N>::V, true>(x);
  if constexpr (Geo<N>::T == 2) {
    if (time) join_time<N, true, 0>(x, h);
  }
}

// column pencil after its inverse transform (i2 in HALVES) -> Bs[i2][q]
template <int N>
__device__ __forceinline__ void store_columns(const ci64 (&x)[Geo<N>::V], const PlaneThread& t, ci64* Bs) {
#pragma unroll
  for (int i = 0; i < Geo<N>::V; ++i) Bs[idx_halves<N>(i, t.h) * Geo<N>::RS + t.q] = x[i];
}

// Bs -> the row pair's packed spectrum (k3 in PARITY); its inverse transform
// has the reals of row q in x.x, of row q + N/2 in x.y (i3 in HALVES)
template <int N>
__device__ __forceinline__ void load_rows(ci64 (&x)[Geo<N>::V], const PlaneThread& t, const ci64* Bs) {
  constexpr int RS = Geo<N>::RS, V = Geo<N>::V;
  const ci64* ra = Bs + t.q * RS;
  const ci64* rb = ra + (N / 2) * RS;
  if constexpr (Geo<N>::T == 1) {
    const ci64 a0 = ra[0], b0 = rb[0];  // (x_0, x_(N/2)) of each row
    x[0] = ci64{a0.x, b0.x};
    x[N / 2] = ci64{a0.y, b0.y};
#pragma unroll
    for (int k = 1; k < N / 2; ++k) {
      const ci64 a = ra[k], c = rb[k];
      x[k] = ci64{a.x - c.y, a.y + c.x};
      x[N - k] = ci64{a.x + c.y, c.x - a.y};
    }
  } else {
#pragma unroll
    for (int i = 0; i < V / 2; ++i) {
      const int k = 2 * i + t.h, m = N / 2 - k;  // x[i]: index k, x[V/2 + i]: index N/2 + k = N - m
      const ci64 a = ra[k], c = rb[k];
      x[i] = ci64{a.x - c.y, a.y + c.x};
      const ci64 am = ra[m % (N / 2)], cm = rb[m % (N / 2)];
      x[V / 2 + i] = ci64{am.x + cm.y, cm.x - am.y};
      if (i == 0 && t.h == 0) {
        x[0] = ci64{a.x, c.x};
        x[V / 2] = ci64{a.y, c.y};
      }
    }
  }
}

// a row pair's forward transform z(k) (k in PARITY, parts exchanged) in the
// pair's own slots of Bs: k < N/2 in row q, the others in row q + N/2
template <int N>
__device__ __forceinline__ void store_rows(const ci64 (&x)[Geo<N>::V], const PlaneThread& t, ci64* Bs) {
  ci64* ra = Bs + t.q * Geo<N>::RS;
  ci64* rb = ra + (N / 2) * Geo<N>::RS;
#pragma unroll
  for (int i = 0; i < Geo<N>::V; ++i)
    (i < Geo<N>::V / 2 ? ra : rb)[idx_parity<N>(i, t.h) % (N / 2)] = ci64{x[i].y, x[i].x};
}

// Bs after store_rows -> column pencil q (i2 in HALVES, parts exchanged) at
// twice its value, from z(q) and z(N - q) of every row pair
template <int N>
__device__ __forceinline__ void load_columns(ci64 (&x)[Geo<N>::V], const PlaneThread& t, const ci64* Bs) {
  constexpr int RS = Geo<N>::RS, V = Geo<N>::V;
  const bool packed = t.q == 0;
#pragma unroll
  for (int i = 0; i < V / 2; ++i) {
    const int r = Geo<N>::T == 1 ? i : t.h * (V / 2) + i;
    const ci64 z1 = Bs[r * RS + t.q], z2 = Bs[(r + N / 2) * RS + (packed ? 0 : N / 2 - t.q)];
    x[i] = packed ? ci64{z2.x, z1.x} : ci64{z1.y - z2.y, z1.x + z2.x};
    x[V / 2 + i] = packed ? ci64{z2.y, z1.y} : ci64{z2.x - z1.x, z1.y + z2.y};
  }
}

// column pencil after its forward transform (k2 in PARITY, parts exchanged) ->
// the plane's half spectrum; the packed pair is split
template <int N>
__device__ __forceinline__ void store_spectrum(const ci64 (&x)[Geo<N>::V], const PlaneThread& t,
                                               ci64* __restrict__ gw) {
  constexpr int HC = Geo<N>::HC, V = Geo<N>::V;
  if (t.q == 0) {
    // X_0(k) = Z(k) + conj Z(-k), X_(N/2)(k) = -i (Z(k) - conj Z(-k))
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int k = idx_parity<N>(i, t.h);
      ci64 zm = x[(V - i) % V];
      if (Geo<N>::T == 2) zm = select(t.h, x[V - 1 - i], zm);
      gw[k * HC] = ci64{x[i].y + zm.y, x[i].x - zm.x};
      gw[k * HC + N / 2] = ci64{x[i].x + zm.x, zm.y - x[i].y};
    }
  } else {
#pragma unroll
    for (int i = 0; i < V; ++i) gw[idx_parity<N>(i, t.h) * HC + t.q] = ci64{x[i].y, x[i].x};
  }
}

// a bound of a plane's entries in its own units: twice (the packed pair's sum) the
// largest pencil sum `top` 2^32, after the shift that brings it to [2^59, 2^60) and
// the halving of the plane's unit: the bits of `top` at the exponent 60
__device__ __forceinline__ float plane_bound(float top) {
  return __uint_as_float((__float_as_uint(top) & 0x7fffffu) | (127u + 60u) << 23);
}

// In place on W[u][i1]: psi <- M^h psi between the inverse and the forward
// transforms of axes 2 and 3.  EP, BP [u][i1]: the plane's exponent and a bound
// of its entries, |entry| <= BP 2^EP.
// Bound by instruction issue (56 % of the slots at N = 32, integer pipe 55 %, 12
// warps per SM) and instruction fetch.  The four passes are one loop around one
// transform body: written out, 158 KB of code waited for instructions 46 % of
// the time.  Two threads per pencil from N = 32 on, so that 168 registers and 12
// warps per SM are enough: one thread per pencil took 105 us where this takes
// 75.8 (7 instances), 16 warps of 128 registers 79.7.  A plane of 8, 16 or 32
// threads stays within a warp and needs no block barrier.  256 instances: 2.51
// ms, 15.2 in FP64; 5.55 TFLOP/s, 0.42 of the rate of register transforms.
// grid = (N / PPC, J, B), block = Planes<N, PPC>::THREADS.
template <int N, int PPC>
__global__ void __launch_bounds__(Planes<N, PPC>::THREADS, Planes<N, PPC>::BLOCKS) k_plane(ci64* __restrict__ W, const int* __restrict__ EA,
                                                                 const i64* __restrict__ mh,
                                                                 const int* __restrict__ em, int* __restrict__ EP,
                                                                 float* __restrict__ BP) {
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC, V = Geo<N>::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[4 * PPC];
  const PlaneThread t = plane_thread<N>(threadIdx.x);
  const int j = blockIdx.y, b = blockIdx.z, i1 = blockIdx.x * PPC + t.pp;
  const size_t u = (size_t)b * gridDim.y + j;
  ci64* Bs = (ci64*)smem_raw + (size_t)t.pp * N * Geo<N>::RS;
  ci64* gw = W + (u * N + i1) * NC;
  if (threadIdx.x < 4 * PPC) red[threadIdx.x] = 0;
  __syncthreads();
  int E = EA[u], s = 0;
  float top = 0.f;
  ci64 x[V];
#pragma unroll 1
  for (int pass = 0; pass < 4; ++pass) {
    if (pass == 2) {
      // x M^h (parts exchanged from here on).  psi_j is largest in the tails,
      // where M^h is smallest, so the products are far below the product of
      // the largest values; they are formed with as many more bits as a bound
      // of their own pencil sum leaves room for.  Without these the products'
      // rounding drowned the result (25 times the error in the 2-norm).
      const i64* mp = mh + ((size_t)b * N + i1) * N * N + t.q;
      float sum = 0.f;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const i64* m = mp + idx_halves<N>(i, t.h) * N;
        sum += (fabsf((float)(int)(x[i].x >> 32)) + 1.f) * (float)((int)(__ldg(m) >> 32) + 1);
        sum += (fabsf((float)(int)(x[i].y >> 32)) + 1.f) * (float)((int)(__ldg(m + N / 2) >> 32) + 1);
      }
      sum = sum * (1.00002f * 0x1p-33f) + 1.f;  // of the products / 2^64, in units of 2^32
      s = shift_for(plane_max<N>(pencil_sum<N>(sum), red + 2 * PPC + t.pp), kSumBits);
      const int bits = min(max(-s, 1), 31);
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const i64* m = mp + idx_halves<N>(i, t.h) * N;
        x[i] = ci64{mul_finer(x[i].y, __ldg(m + N / 2), bits), mul_finer(x[i].x, __ldg(m), bits)};
      }
      E += 64 + em[b * N + i1] - bits;
      s += bits;
      if (s > 0) {  // one bit was too many
        shift_all<V>(x, s);
        E += s;
      }
    } else {
      if (pass == 0) {
#pragma unroll
        for (int i = 0; i < V; ++i) x[i] = gw[idx_parity<N>(i, t.h) * HC + t.q];
        if (t.q == 0) {
#pragma unroll
          for (int i = 0; i < V; ++i) x[i] = x[i] + mul_i(gw[idx_parity<N>(i, t.h) * HC + N / 2]);
        }
      } else if (pass == 1) {
        load_rows<N>(x, t, Bs);
      } else {
        load_columns<N>(x, t, Bs);
      }
      top = normalise<N>(x, s, E, red + pass * PPC + t.pp, pass == 3);
    }
    pencil_inverse<N>(x, t.h, pass < 2);
    if (pass == 0) {
      store_columns<N>(x, t, Bs);
      plane_sync<N>();
    } else if (pass == 2) {
      store_rows<N>(x, t, Bs);
      plane_sync<N>();
    }
  }
  E -= 1;  // load_columns doubles
  store_spectrum<N>(x, t, gw);
  if (t.tp == 0) {
    EP[u * N + i1] = E;
    BP[u * N + i1] = plane_bound(top);
  }
}

// ------------------------------------------------------------ head
// the plane's maximum of an unsigned value
template <int N>
__device__ __forceinline__ unsigned plane_umax(unsigned v, unsigned* slot) {
  if constexpr (Geo<N>::WARP) {
#pragma unroll
    for (int o = Geo<N>::TPP / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
  } else {
    atomicMax(slot, v);
    __syncthreads();
    return *slot;
  }
}
// Axes 3 and 2 of FFT(r) (blockIdx.z = 0 with with_ratio; r = g/M with the
// cut-off) or of FFT(g): F[z][b][i1][k2][k3], EP [z][b][i1].  The field's plane is
// read coalesced into shared memory as FP64, converted at the plane's own
// exponent by the row threads.  Latency-bound: 0.19 ms for 256 instances at N =
// 32 (1.4 in FP64).
// grid = (N / PPC, B, 2 or 1), block = Planes<N, PPC>::THREADS.
template <int N, int PPC>
__global__ void __launch_bounds__(Planes<N, PPC>::THREADS) k_fwd_planes(const double* __restrict__ field,
                                                                      const double* __restrict__ inst, int with_ratio, int cutoff,
                                                                      ci64* __restrict__ F, int* __restrict__ EP,
                                                                      int* __restrict__ bad) {
  constexpr int NC = Geo<N>::NC, V = Geo<N>::V, TPP = Geo<N>::TPP, RS = N + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[3 * PPC];
  __shared__ double em[6 * N];  // factors of 1/M, squared distances
  const double* sq = em + 3 * N;
  const PlaneThread t = plane_thread<N>(threadIdx.x);
  const int b = blockIdx.y, i1 = blockIdx.x * PPC + t.pp;
  const size_t u = (size_t)blockIdx.z * gridDim.y + b;
  ci64* Bs = (ci64*)smem_raw + (size_t)t.pp * N * Geo<N>::RS;
  double* D = (double*)Bs;  // [i2][i3], row stride N + 1
  const bool ratio = with_ratio && blockIdx.z == 0;
  if (threadIdx.x < 3 * PPC) red[threadIdx.x] = 0;
  static_assert(Inst<N>::SQ == Inst<N>::EI + 3 * N, "the two tables follow each other");
  double dstar = 0.0;
  if (ratio) {
    const double* I = inst + (size_t)b * Inst<N>::SIZE;
    dstar = I[Inst<N>::DSTAR];
    for (int i = threadIdx.x; i < 6 * N; i += Planes<N, PPC>::THREADS) em[i] = I[Inst<N>::EI + i];
  }
  __syncthreads();
  const double* g = field + ((size_t)b * N + i1) * N * N;
  unsigned top = 0;
  // the loads of several points in flight: one at a time took 10 of 20 us for a single instance
#pragma unroll 8
  for (int it = 0; it < N * N / TPP; ++it) {
    const int e = t.tp + it * TPP, i3 = e % N, i2 = e / N;
    double v = g[e];
    if (ratio) {
      const bool cut = cutoff && __dadd_rn(__dadd_rn(sq[i1], sq[N + i2]), sq[2 * N + i3]) >= dstar;
      v = cut ? 0.0 : v * ((em[i1] * em[N + i2]) * em[2 * N + i3]);
    }
    D[i2 * RS + i3] = v;
    top = max(top, (unsigned)__double2hiint(v) & 0x7fffffffu);
  }
  plane_sync<N>();
  top = plane_umax<N>(top, red + t.pp);
  const bool fin = top < 0x7ff00000u;
  if (!fin && t.tp == 0) atomicOr(bad + b, 1);
  int E = (int)(top >> 20) - 1023 - 57;  // the plane's largest value in [2^57, 2^58)
  int s = 0;
  ci64 x[V];
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 0) {
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int i3 = idx_halves<N>(i, t.h);
        x[i] = fin ? ci64{to_fixed(D[(t.q + N / 2) * RS + i3], E), to_fixed(D[t.q * RS + i3], E)} : ci64{0, 0};
      }
    } else {
      load_columns<N>(x, t, Bs);
    }
    normalise<N>(x, s, E, red + (1 + pass) * PPC + t.pp, true);
    pencil_inverse<N>(x, t.h, false);
    if (pass == 0) {
      plane_sync<N>();  // D has been read
      store_rows<N>(x, t, Bs);
      plane_sync<N>();
    }
  }
  E -= 1;
  store_spectrum<N>(x, t, F + (u * N + i1) * NC);
  if (t.tp == 0) EP[u * N + i1] = E;
}

// a value as a multiplier with its sign mask
struct SignedMult {
  Mult m;
  int neg;
};
__device__ __forceinline__ SignedMult signed_mult(i64 y) {
  const Mult m = split_mult(y);
  return SignedMult{m, m.th >> 31};
}
__device__ __forceinline__ SignedMult signed_of(i64 packed) {
  const Mult m = unpack_mult(packed);
  return SignedMult{m, m.th >> 31};
}
// a z / 2^64 with a's parts as multipliers
__device__ __forceinline__ ci64 cmul_mult(SignedMult ax, SignedMult ay, ci64 z) {
  return ci64{mul_signed(z.x, ax.m, ax.neg) - mul_signed(z.y, ay.m, ay.neg),
              mul_signed(z.y, ax.m, ax.neg) + mul_signed(z.x, ay.m, ay.neg)};
}
template <int V>
__device__ __forceinline__ unsigned top_bits(const ci64 (&x)[V]) {  // bits 31.. of the largest magnitude
  unsigned m = 0;
#pragma unroll
  for (int i = 0; i < V; ++i)
    m = max(m, max((unsigned)((x[i].x ^ (x[i].x >> 63)) >> 31), (unsigned)((x[i].y ^ (x[i].y >> 63)) >> 31)));
  return m;
}

// Axis 1 of the head, one column per pencil.  z = 0: r^ = FFT_1 of F[0], every
// column scaled to a top bit of 2^61 with its exponent eR; rm[b][band][col]:
// sum of (|re| + |im|) 2^-62 over the band's |k1| (k_unit_scale).  z = 1: F[1] <- InvFFT_1(FFT_1(F[src1]) omega) (src1 = 1: in
// place).  z = 2: F[2] = InvFFT_1(FFT(M) omega), FFT(M) from its factors.  Of
// F[1], F[2] every column has its exponent EC[z][b][col].  z0: the first z of
// the launch.  omega: multipliers indexed by |k|^2, or with omega3 by the
// position (k1, k2, k3).
// grid = (ceil(NC T / 64), B, count), block = 64.
template <int N>
__global__ void __launch_bounds__(64) k_axis1_head(ci64* __restrict__ F, const int* __restrict__ EP,
                                                   const ci64* __restrict__ MH, const int* __restrict__ eM,
                                                   const i64* __restrict__ omega, int omega3, int omega_exp,
                                                   int src1, ci64* __restrict__ R,
                                                   int* __restrict__ eR, float* __restrict__ rm, int* __restrict__ EC,
                                                   int z0) {
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC, T = Geo<N>::T, V = Geo<N>::V;
  __shared__ int se[N];
  __shared__ float fe[N];
  const int z = z0 + blockIdx.z, B = gridDim.y, b = blockIdx.y;
  const int id = blockIdx.x * 64 + threadIdx.x, h = T == 2 ? id & 1 : 0;
  const bool on = id / T < NC;
  const int col = on ? id / T : NC - 1, k2 = col / HC, k3 = col % HC;
  const size_t u = (size_t)z * B + b, us = (size_t)(z == 1 ? src1 : z) * B + b;
  ci64 x[V];
  int E;
  if (z < 2) {
    // the planes' exponents below the largest
    int base = kZeroExp;
    for (int i = 0; i < N; ++i) base = max(base, EP[us * N + i]);
    for (int i = threadIdx.x; i < N; i += 64) {
      se[i] = base - EP[us * N + i];
      fe[i] = exp2_neg(se[i]);
    }
    __syncthreads();
    const ci64* src = F + us * N * NC + col;
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int i1 = idx_parity<N>(i, h);
      x[i] = src[(size_t)i1 * NC];
      sum += (fabsf((float)(int)(x[i].x >> 32)) + fabsf((float)(int)(x[i].y >> 32))) * fe[i1];
    }
    const int s = shift_for(pencil_sum<N>(sum * 1.00002f + (float)(2 * V)), kSumBits);
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int d = se[idx_parity<N>(i, h)] + s;
      x[i] = ci64{shift_any(x[i].x, d), shift_any(x[i].y, d)};
    }
    E = base + s;
    dft_time<N, false>(x, h);  // k1 in HALVES
  } else {
    const ci64 m2 = MH[((size_t)b * 3 + 1) * N + k2], m3 = MH[((size_t)b * 3 + 2) * N + k3];
    ci64 c = cmul_mult(signed_mult(m2.x), signed_mult(m2.y), m3);
    const i64 m = (c.x ^ (c.x >> 63)) | (c.y ^ (c.y >> 63));
    const int l = max(__clzll(m) - 2, 0);
    const SignedMult cx = signed_mult((i64)((u64)c.x << l)), cy = signed_mult((i64)((u64)c.y << l));
#pragma unroll
    for (int i = 0; i < V; ++i) x[i] = cmul_mult(cx, cy, MH[(size_t)b * 3 * N + idx_halves<N>(i, h)]);
    E = eM[b * 3] + eM[b * 3 + 1] + eM[b * 3 + 2] + 128 - l;
  }
  if (z == 0) {
    unsigned m = top_bits<V>(x);
    if (T == 2) m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    const int l = m ? __clz(m) - 1 : 0;
    ci64* dst = R + (size_t)b * N * NC + col;
    float sums[BANDS] = {};
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const ci64 v = ci64{(i64)((u64)x[i].x << l), (i64)((u64)x[i].y << l)};
      if (on) dst[(size_t)idx_halves<N>(i, h) * NC] = v;
      const float w = (fabsf((float)(int)(v.x >> 32)) + fabsf((float)(int)(v.y >> 32)) + 2.f) * 0x1p-30f;
      if (T == 1) {
        sums[band<N>(i <= N / 2 ? i : N - i)] += w;
      } else {  // |k| of value i of thread 0, 1: i, N/4 + i below, N/2 - i, N/4 - i above N/2
        constexpr int Q = N / 4;
        const float w0 = h ? 0.f : w, w1 = h ? w : 0.f;
        sums[band<N>(i < Q ? i : (i == Q ? N / 2 : N / 2 - (i - Q)))] += w0;
        sums[band<N>(i < Q ? Q + i : Q - (i - Q))] += w1;
      }
    }
#pragma unroll
    for (int d = 0; d < BANDS; ++d) {
      const float w = pencil_sum<N>(sums[d]);
      if (on && h == 0) rm[((size_t)b * BANDS + d) * NC + col] = w;
    }
    if (!on) return;
    if (h == 0) eR[b * NC + col] = m ? E - l : kZeroExp;
    return;
  }
  const int c2 = k2 <= N / 2 ? k2 : N - k2, q23 = c2 * c2 + k3 * k3;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const int k = idx_halves<N>(i, h), c = k <= N / 2 ? k : N - k;
    const Mult m = unpack_mult(__ldg(omega3 ? omega + (size_t)k * NC + col : omega + q23 + c * c));
    x[i] = ci64{mul_signed_rounded(x[i].x, m, m.th >> 31), mul_signed_rounded(x[i].y, m, m.th >> 31)};
  }
  const int s = shift_for(pencil_sum<N>(abs_sum<V>(x)), kSumBits);
  shift_all<V>(x, s);
  E += 64 - omega_exp + s;
  dft_freq<N, true>(x, h);  // i1 in PARITY
  if (!on) return;
  if (h == 0) EC[u * NC + col] = E;
  ci64* dst = F + u * N * NC + col;
#pragma unroll
  for (int i = 0; i < V; ++i) dst[(size_t)idx_parity<N>(i, h) * NC] = x[i];
}

// ------------------------------------------------------------ accumulation
__device__ __forceinline__ int log2_above(double x) { return x > 0.0 ? ilogb(x) + 1 : kZeroExp; }
// 2^-e as FP64, 0 beyond its normal range (e >= 0)
__device__ __forceinline__ double exp2_neg64(int e) { return e > 1022 ? 0.0 : __hiloint2double((1023 - e) << 20, 0); }

// InvFFT_1(L^+) of one instance for a block of columns.
//
// The exponent EL of L^+ and the right shift sp of every plane of every node
// into units where phi_j x / 2^64 carries EL: with S_j the sum over planes of
// the bounds BP 2^EP (an axis-1 pencil of psi^_j at most), S_j <= 2^60 of those
// units and sum_j S_j max|phi_j| <= 2^61 of EL's.  q[j], pm[j]: the exponent and
// the largest value of the multipliers phi_j.  S_j is kept as a value and the
// largest exponent of its planes: as one FP64 number it overflowed, unlike the
// result, for inputs 2^20 below FP64's own limit.
//
// Warp w takes the nodes j = w, w + WARPS, ...; their phi_j psi^_j add up in the
// warp's shared memory, and the warps' sums at the end (integer sums: any
// order gives the same result).  Then warp 0 transforms each column back, at
// its own exponent EC[b][col].
// Bound by issue and load latency; the sum over j stays on chip, where a launch
// per node read and wrote it 32 times: 0.89 ms for 256 instances at N = 32, 4.5
// in FP64.
// grid = (ceil(NC T / 32), B), block = 32 WARPS, shared memory acc_smem(J).
template <int N, int WARPS>
constexpr size_t acc_smem(int J) {
  return sizeof(ci64) * WARPS * Geo<N>::V * 32 + (sizeof(double) + sizeof(int) * (N + 1)) * (size_t)J;
}
template <int N, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_axis1_acc(const ci64* __restrict__ W, const int* __restrict__ EP,
                                                        const float* __restrict__ BP, const i64* __restrict__ phi,
                                                        const int* __restrict__ q, const double* __restrict__ pm,
                                                        ci64* __restrict__ F, int* __restrict__ EC, int J) {
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC, T = Geo<N>::T, V = Geo<N>::V, Q = 3 * (N / 2) * (N / 2) + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* part = (double*)(smem_raw + sizeof(ci64) * WARPS * V * 32);  // [J] S_j max|phi_j|
  int* pe = (int*)(part + J);                                         // [J] the exponents of part
  int* sp = pe + J;                                                   // [J][N]
  __shared__ int el;
  const int b = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int id = blockIdx.x * 32 + lane, h = T == 2 ? id & 1 : 0;
  const bool on = id / T < NC;
  const int col = on ? id / T : NC - 1, k2 = col / HC, k3 = col % HC, c2 = k2 <= N / 2 ? k2 : N - k2;
  const int q23 = c2 * c2 + k3 * k3;
  if (threadIdx.x == 0) el = kZeroExp;
  __syncthreads();
#pragma unroll(N >= 48 ? 1 : 4)
  for (int j = w; j < J; j += WARPS) {
    const size_t u = ((size_t)b * J + j) * N;
    constexpr int R = (N + 31) / 32;  // planes per lane
    int e[R], base = kZeroExp;
    unsigned f[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = lane + 32 * r;
      e[r] = i < N ? EP[u + i] : 2 * kZeroExp;
      f[r] = i < N ? __float_as_uint(BP[u + i]) : 0u;
      base = max(base, e[r]);
    }
    base = __reduce_max_sync(0xffffffffu, base);
    // the bounds' 24-bit mantissas at 2^37 (their exponent is 60), added as
    // integers with 32 bits below: FP64 sums took 3.5 us of the SM's pipe per block at
    // N = J = 64
    u64 s = 0;
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (base - e[r] < 64) s += ((u64)(f[r] & 0x7fffffu | 0x800000u) << 32) >> (base - e[r]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      s += N;  // past what the shifts dropped
      part[j] = (double)s * pm[j];
      pe[j] = base + 5;
      atomicMax(&el, base + 5 + 64 - __clzll((i64)s) - kSumBits - q[j] + 64);
    }
  }
  __syncthreads();
  if (w == 0) {
    int base = pe[lane % J];
    for (int j = lane + 32; j < J; j += 32) base = max(base, pe[j]);
    base = __reduce_max_sync(0xffffffffu, base);
    double s = 0.0;
    for (int j = lane; j < J; j += 32) s += part[j] * exp2_neg64(base - pe[j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      const int e = max(el, base + log2_above(s * 1.0001) - 61);
      el = e < kZeroExp / 2 ? 0 : e;
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < J * N; e += 32 * WARPS) {
    // >= 0: BP is at least 2^60 of its plane's units
    sp[e] = min(max(el + q[e / N] - 64 - EP[(size_t)b * J * N + e], 0), 63);
  }
  __syncthreads();
  ci64* acc = (ci64*)smem_raw + w * V * 32 + lane;
#pragma unroll
  for (int i = 0; i < V; ++i) acc[i * 32] = ci64{0, 0};
  ci64 x[V];
  for (int j = w; j < J; j += WARPS) {
    const size_t u = (size_t)b * J + j;
    const ci64* src = W + u * N * NC + col;
    const int* su = sp + j * N;
    const i64* tab = phi + (size_t)j * Q + q23;
#pragma unroll
    for (int i = 0; i < V; ++i) x[i] = src[(size_t)idx_parity<N>(i, h) * NC];
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int s = su[idx_parity<N>(i, h)];
      x[i] = ci64{shift_right(x[i].x, s), shift_right(x[i].y, s)};
    }
    dft_time<N, false>(x, h);
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int k = idx_halves<N>(i, h), c = k <= N / 2 ? k : N - k;
      const Mult m = unpack_mult(__ldg(tab + c * c));
      const int neg = m.th >> 31;
      ci64 a = acc[i * 32];
      a.x += mul_signed_rounded(x[i].x, m, neg);
      a.y += mul_signed_rounded(x[i].y, m, neg);
      acc[i * 32] = a;
    }
  }
  __syncthreads();
  ci64* all = (ci64*)smem_raw + lane;
  for (int i = w; i < V; i += WARPS) {
    ci64 a{0, 0};
    for (int v = 0; v < WARPS; ++v) a = a + all[(v * V + i) * 32];
    all[i * 32] = a;
  }
  __syncthreads();
  if (w > 0) return;
#pragma unroll
  for (int i = 0; i < V; ++i) x[i] = all[i * 32];
  const int s = shift_for(pencil_sum<N>(abs_sum<V>(x)), kSumBits);
  shift_all<V>(x, s);
  dft_freq<N, true>(x, h);
  if (!on) return;
  if (h == 0) EC[b * NC + col] = el + s;
#pragma unroll
  for (int i = 0; i < V; ++i) F[((size_t)b * N + idx_parity<N>(i, h)) * NC + col] = x[i];
}

// ------------------------------------------------------------ combination
// Inverse axes 2 and 3 of the fields of the mode, and the output:
//   COMBINE  out = L+ - u M - w g, fields L+ = 0, u = 1, w = 2
//   CACHED   the same with w read from wc
//   FACTOR   out = w (field 2 alone, for the Maxwellian cache)
//   QUAD     out = Q+ - u g (Q(f,f): fields Q+ = 0, u = 1, g = f)
// A group of threads for each field transforms the block's planes of it, then
// all threads combine.  Columns of F carry their own exponents EC[f][b][col];
// they meet at the plane's largest.  NaN for a marked instance (bad).
// The results become FP64 on the integer pipe (to_double).  Latency-bound: 0.33
// ms for 256 instances at N = 32, 15 % of HBM; 1.0 in FP64.
// grid = (N / PPC, B), block = FIELDS Planes<N, PPC>::THREADS.
enum CombineMode { COMBINE, CACHED, FACTOR, QUAD };
template <int N, int PPC, int MODE>
struct Combine {
  static constexpr int F0 = MODE == FACTOR ? 2 : 0, FIELDS = MODE == FACTOR ? 1 : (MODE == COMBINE ? 3 : 2);
  static constexpr bool MAXW = MODE == COMBINE || MODE == CACHED;  // u is multiplied by M
  static constexpr int GROUP = Planes<N, PPC>::THREADS, THREADS = FIELDS * GROUP;
  static constexpr size_t BYTES = FIELDS * Planes<N, PPC>::BYTES;
};
template <int N, int PPC, int MODE>
__global__ void __launch_bounds__(Combine<N, PPC, MODE>::THREADS)
    k_combine_planes(const double* __restrict__ inst, const double* __restrict__ g, const ci64* __restrict__ F,
                     const int* __restrict__ EC, const double* __restrict__ wc, const int* __restrict__ bad,
                     double* __restrict__ out) {
  using C = Combine<N, PPC, MODE>;
  constexpr int HC = Geo<N>::HC, NC = Geo<N>::NC, V = Geo<N>::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned red[3 * C::FIELDS * PPC];
  __shared__ double em[3 * N];
  const int fl = threadIdx.x / C::GROUP, f = C::F0 + fl;
  const PlaneThread t = plane_thread<N>(threadIdx.x % C::GROUP);
  const int B = gridDim.y, b = blockIdx.y, i1 = blockIdx.x * PPC + t.pp;
  ci64* Bs = (ci64*)smem_raw + (size_t)(fl * PPC + t.pp) * N * Geo<N>::RS;
  for (int i = threadIdx.x; i < 3 * C::FIELDS * PPC; i += C::THREADS) red[i] = 0;
  if constexpr (C::MAXW) {
    for (int i = threadIdx.x; i < 3 * N; i += C::THREADS) em[i] = inst[(size_t)b * Inst<N>::SIZE + Inst<N>::EM + i];
  }
  __syncthreads();
  const size_t u = (size_t)f * B + b;
  const ci64* src = F + (u * N + i1) * NC + t.q;
  const int* ec = EC + u * NC + t.q;
  unsigned* slot = red + fl * 3 * PPC + t.pp;
  // the largest column exponent (offset to stay positive), then the pencils' sums below it
  int top = kZeroExp;
  for (int i = 0; i < V; ++i) {
    const int k = idx_parity<N>(i, t.h) * HC;
    top = max(top, ec[k]);
    if (t.q == 0) top = max(top, ec[k + N / 2]);
  }
  const int base = (int)plane_umax<N>((unsigned)(top - 2 * kZeroExp), slot) + 2 * kZeroExp;
  ci64 x[V];
  int E = base, s = 0;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 0) {
      float sum = 0.f;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int k = idx_parity<N>(i, t.h) * HC;
        x[i] = src[k];
        sum += (fabsf((float)(int)(x[i].x >> 32)) + fabsf((float)(int)(x[i].y >> 32))) * exp2_neg(base - ec[k]);
        if (t.q == 0) {
          const ci64 v = src[k + N / 2];
          sum += (fabsf((float)(int)(v.x >> 32)) + fabsf((float)(int)(v.y >> 32))) * exp2_neg(base - ec[k + N / 2]);
        }
      }
      sum = sum * 1.00002f + (float)(4 * V);
      const int sc = shift_for(plane_max<N>(pencil_sum<N>(sum), slot + PPC), kSumBits);
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int k = idx_parity<N>(i, t.h) * HC, d = base - ec[k] + sc;
        x[i] = ci64{shift_any(x[i].x, d), shift_any(x[i].y, d)};
        if (t.q == 0) {
          const ci64 v = src[k + N / 2];
          const int d2 = base - ec[k + N / 2] + sc;
          x[i] = x[i] + mul_i(ci64{shift_any(v.x, d2), shift_any(v.y, d2)});
        }
      }
      E += sc;
    } else {
      load_rows<N>(x, t, Bs);
      normalise<N>(x, s, E, slot + 2 * PPC, true);
    }
    pencil_inverse<N>(x, t.h, true);
    if (pass == 0) {
      store_columns<N>(x, t, Bs);
      plane_sync<N>();
    }
  }
  plane_sync<N>();
  // the field as FP64 (u already times M) in the rows' own slots of Bs
  double* ra = (double*)(Bs + t.q * Geo<N>::RS);
  double* rb = (double*)(Bs + (t.q + N / 2) * Geo<N>::RS);
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const int i3 = idx_halves<N>(i, t.h);
    double va = to_double(x[i].x, E), vb = to_double(x[i].y, E);
    if (C::MAXW && f == 1) {
      va *= em[i1] * em[N + t.q] * em[2 * N + i3];
      vb *= em[i1] * em[N + N / 2 + t.q] * em[2 * N + i3];
    }
    ra[i3] = va;
    rb[i3] = vb;
  }
  __syncthreads();
  const size_t o = ((size_t)b * N + blockIdx.x * PPC) * N * N;
  const bool nan = MODE != FACTOR && bad[b] != 0;
#pragma unroll 4
  for (int e = threadIdx.x; e < PPC * N * N; e += C::THREADS) {
    const int i3 = e % N, r = e / N;  // row r of the block's planes
    const double* v = (const double*)((ci64*)smem_raw + (size_t)r * Geo<N>::RS) + i3;
    constexpr size_t FS = (size_t)PPC * N * Geo<N>::RS * 2;  // doubles from one field's planes to the next
    double y = v[0];
    if constexpr (MODE == QUAD) y = y - g[o + e] * v[FS];
    if constexpr (C::MAXW) y = y - v[FS] - (MODE == CACHED ? wc[o + e] : v[2 * FS]) * g[o + e];
    if constexpr (MODE != FACTOR) {
      if (nan) y = __longlong_as_double(0x7ff8000000000000LL);
    }
    out[o + e] = y;
  }
}

}  // namespace fx
}  // namespace lbo
