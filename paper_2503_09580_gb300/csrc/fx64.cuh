// 64-bit block fixed-point arithmetic on the integer pipe: the transforms of
// the FP64 precision on GB300, whose FP64 pipe issues two lanes per clock per
// SM while its integer pipe adds about 58 and multiplies (to the high 64 bits)
// about 7 pairs of 64-bit numbers per clock.  A 32-point transform in
// registers takes 19 SM clocks per lane here (lbo_measure_fx_peak) against 245 in
// FP64.
//
// A number is an integer x with the value x 2^E; E is shared by a block of
// numbers (a plane, a column, an instance).  Before every transform the block
// is shifted so that sum(|re| + |im|) over each of its pencils is at most
// 2^60.  That sum bounds every partial sum of the transform, so no operation
// overflows, and the rounding of one operation (at most one unit in the last
// place) is then 2^-57 to 2^-60 of the pencil's largest result, where FP64
// rounds at 2^-53.
//
// Multiplications: y t / 2^64 with t = th 2^32 + tl, th >= 0 and tl signed,
// from the two high cross products and the wide main product; the product
// yl tl is left out and the two floors are balanced by + 1, so the error is
// below 1.5 units and unbiased.  |t| < 0.46 2^64 and |y| < 2^60 keep the sum of
// the cross products within 32 bits; larger constants are held as their
// distance to 1/2 or to 1 (fx_constants.h).  Rotations by a < 45 degrees are
// three lifting steps (tan(a/2), sin(a), tan(a/2)), each one such product.
//
// Host code can include this header (the tests check the transforms there).
#pragma once
#include <cstdint>

#include "fx_constants.h"

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
#endif

namespace lbo {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

struct alignas(16) ci64 {
  i64 x, y;
};

FX_FN ci64 operator+(ci64 a, ci64 b) { return ci64{a.x + b.x, a.y + b.y}; }
FX_FN ci64 operator-(ci64 a, ci64 b) { return ci64{a.x - b.x, a.y - b.y}; }
FX_FN ci64 mul_i(ci64 a) { return ci64{-a.y, a.x}; }
FX_FN ci64 mul_mi(ci64 a) { return ci64{a.y, -a.x}; }
template <bool INV>
FX_FN ci64 quarter(ci64 a) {  // a exp(-+ i pi / 2)
  return INV ? mul_i(a) : mul_mi(a);
}

FX_FN unsigned umulhi32(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (unsigned)(((u64)a * b) >> 32);
#endif
}
FX_FN int mulhi32(int a, int b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((i64)a * b) >> 32);
#endif
}

// A multiplier t = th 2^32 + tl split for mul(): th >= 0, tl signed.
struct Mult {
  int th, tl;
};
FX_FN constexpr Mult split_mult(i64 t) { return Mult{(int)((t + 0x80000000LL) >> 32), (int)(unsigned)(u64)t}; }
// the same packed into the two words of one 64-bit table entry
FX_FN i64 pack_mult(i64 t) { return (i64)((u64)(t + 0x80000000LL) & 0xffffffff00000000ULL) | (i64)(unsigned)(u64)t; }
FX_FN Mult unpack_mult(i64 w) { return Mult{(int)(w >> 32), (int)(unsigned)(u64)w}; }

// round(y t / 2^64), th >= 0.  The 1 that balances the two floors is left out
// for y = 0: whole pencils are zero (r beyond the cut-off), and what a unit in
// each of their products adds up to was ten times the other rounding errors.
FX_FN i64 mul(i64 y, Mult t) {
  const unsigned yl = (unsigned)(u64)y;
  const int yh = (int)(y >> 32);
  const int c = (int)umulhi32(yl, (unsigned)t.th) + mulhi32(yh, t.tl) + (int)(yl < 1u ? yl : 1u);
  return (i64)yh * t.th + (i64)c;
}
// round(y t / 2^64), th of either sign; neg = th >> 31 (|t| <= 2^62)
FX_FN i64 mul_signed(i64 y, Mult t, int neg) {
  const unsigned yl = (unsigned)(u64)y;
  const int yh = (int)(y >> 32);
  const int c = (int)(umulhi32(yl, (unsigned)t.th) - (yl & (unsigned)neg)) + mulhi32(yh, t.tl) + (int)(yl < 1u ? yl : 1u);
  return (i64)yh * t.th + (i64)c;
}
// round((y t + z w) / 2^64) for |y|, |z| <= 2^60 and a pair of multipliers whose
// th have a norm of at most 2^30: the cross products together then stay below
// 1.8 2^30.  Their four floors are balanced by 2 unless y = z = 0.
FX_FN i64 mul_pair(i64 y, Mult t, i64 z, Mult w) {
  const unsigned yl = (unsigned)(u64)y, zl = (unsigned)(u64)z, any = yl | zl;
  const int yh = (int)(y >> 32), zh = (int)(z >> 32);
  const int c = (int)(umulhi32(yl, (unsigned)t.th) - (yl & (unsigned)(t.th >> 31))) + mulhi32(yh, t.tl) +
                (int)(umulhi32(zl, (unsigned)w.th) - (zl & (unsigned)(w.th >> 31))) + mulhi32(zh, w.tl) +
                (int)(any < 2u ? any : 2u);
  return (i64)yh * t.th + ((i64)zh * w.th + (i64)c);
}
// y m 2^(b - 64) for a multiplier 0 <= m < 2^60 split at bit 31 (pack_finer), 1 <= b
// <= 31: b more bits than mul() keeps, all four partial products taken.
FX_FN i64 pack_finer(i64 m) { return (i64)(((u64)m >> 31) << 32 | ((u64)m & 0x7fffffffULL)); }
FX_FN i64 mul_finer(i64 y, i64 packed, int b) {
  const unsigned yl = (unsigned)(u64)y, th = (unsigned)((u64)packed >> 32), tl = (unsigned)(u64)packed;
  const int yh = (int)(y >> 32);
  const u64 t0 = (u64)(yl >> 1) * th + umulhi32(yl, tl);
  const i64 t1 = (i64)yh * (int)tl + (i64)t0;
  return (i64)((u64)((i64)yh * (int)th) << (b - 1)) + ((t1 + ((i64)1 << (31 - b))) >> (32 - b));
}
// mul_signed() rounded once, from the exact sum of the cross products: unbiased
// also where th = 0 (a multiplier far below its table's largest entry), where
// the + 1 of mul_signed() would add half a unit to every product.
FX_FN i64 mul_signed_rounded(i64 y, Mult t, int neg) {
  const unsigned yl = (unsigned)(u64)y;
  const int yh = (int)(y >> 32);
  const u64 t0 = (u64)yl * (unsigned)t.th + 0x80000000ULL - ((u64)(yl & (unsigned)neg) << 32);
  const i64 t1 = (i64)yh * t.tl + (i64)t0;
  return (i64)yh * t.th + (t1 >> 32);
}
// y t for a compile-time constant 0 < |t| < 0.46 2^64
template <i64 T>
FX_FN i64 mulc(i64 y) {
  constexpr Mult k = split_mult(T < 0 ? -T : T);
  return T < 0 ? -mul(y, k) : mul(y, k);
}
// y x for a constant 0 < x < 1 held as (form, value), see gen_fx_constants.py
template <int FORM, i64 V>
FX_FN i64 mul_formed(i64 y) {
  if constexpr (FORM == 0) return mulc<V>(y);
  else if constexpr (FORM == 1) return V == 0 ? (y >> 1) : (y >> 1) + mulc<(V == 0 ? 1 : V)>(y);
  else return y - mulc<V>(y);
}

// z exp(-i 2 pi M / NN), |M| <= NN / 8 (NN = 64 or 48): three lifting steps
template <int M, int NN>
FX_FN ci64 rotate(ci64 z) {
  constexpr int A = M < 0 ? -M : M;
  static_assert((NN == 64 || NN == 48) && A <= NN / 8, "angle of a rotation");
  if constexpr (M == 0) {
    return z;
  } else if constexpr (8 * A == NN) {  // 45 degrees: (x + y, y - x) / sqrt 2
    const ci64 s = M > 0 ? ci64{z.x + z.y, z.y - z.x} : ci64{z.x - z.y, z.x + z.y};
    return ci64{s.x - mulc<kFxOneMinusSqrtHalf>(s.x), s.y - mulc<kFxOneMinusSqrtHalf>(s.y)};
  } else {
    constexpr i64 t = NN == 64 ? fx_tan_half64(A) : fx_tan_half48(A);
    constexpr i64 s = NN == 64 ? fx_sin64(A) : fx_sin48(A);
    constexpr int f = NN == 64 ? fx_sin64_form(A) : fx_sin48_form(A);
    if constexpr (M > 0) {  // x' = c x + s y, y' = c y - s x
      z.x += mulc<t>(z.y);
      z.y -= mul_formed<f, s>(z.x);
      z.x += mulc<t>(z.y);
    } else {
      z.x -= mulc<t>(z.y);
      z.y += mul_formed<f, s>(z.x);
      z.x -= mulc<t>(z.y);
    }
    return z;
  }
}

// z W_NN^M, W_NN = exp(-2 pi i / NN) (INV: its conjugate), any M >= 0
template <int M, int NN, bool INV>
FX_FN ci64 twiddle(ci64 z) {
  constexpr int m = INV ? (NN - M % NN) % NN : M % NN;
  constexpr int q = (m + NN / 8 - 1) / (NN / 4), r = m - q * (NN / 4);  // r in (-NN/8, NN/8]
  z = rotate<r, NN>(z);
  if constexpr ((q & 3) == 1) return mul_mi(z);
  else if constexpr ((q & 3) == 2) return ci64{-z.x, -z.y};
  else if constexpr ((q & 3) == 3) return mul_i(z);
  else return z;
}

// W_N^M through the table of 64ths or 48ths
template <int M, int N, bool INV>
FX_FN ci64 twiddle_n(ci64 z) {
  if constexpr (64 % N == 0) return twiddle<M * (64 / N), 64, INV>(z);
  else return twiddle<M * (48 / N), 48, INV>(z);
}

template <bool INV>
FX_FN void dft3(ci64& a0, ci64& a1, ci64& a2) {
  const ci64 t1 = a1 + a2, t2 = a1 - a2;
  const ci64 m = ci64{a0.x - (t1.x >> 1), a0.y - (t1.y >> 1)};
  const i64 sx = t2.x - mulc<kFxOneMinusSqrt34>(t2.x), sy = t2.y - mulc<kFxOneMinusSqrt34>(t2.y);
  const ci64 s = INV ? ci64{-sy, sx} : ci64{sy, -sx};
  a0 = a0 + t1;
  a1 = m + s;
  a2 = m - s;
}

template <bool INV>
FX_FN void dft4(ci64& a0, ci64& a1, ci64& a2, ci64& a3) {
  const ci64 t0 = a0 + a2, t1 = a0 - a2, t2 = a1 + a3, t3 = quarter<INV>(a1 - a3);
  a0 = t0 + t2;
  a2 = t0 - t2;
  a1 = t1 + t3;
  a3 = t1 - t3;
}

template <bool INV>
FX_FN void dft8(ci64 (&a)[8]) {
  ci64 e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6], o0 = a[1], o1 = a[3], o2 = a[5], o3 = a[7];
  dft4<INV>(e0, e1, e2, e3);
  dft4<INV>(o0, o1, o2, o3);
  o1 = twiddle<8, 64, INV>(o1);
  o2 = quarter<INV>(o2);
  o3 = twiddle<24, 64, INV>(o3);
  a[0] = e0 + o0;
  a[4] = e0 - o0;
  a[1] = e1 + o1;
  a[5] = e1 - o1;
  a[2] = e2 + o2;
  a[6] = e2 - o2;
  a[3] = e3 + o3;
  a[7] = e3 - o3;
}

// column n1 of the first stage of an (R1 x R2)-point transform: the R2-point
// transform over x[n1 + R1 i] and its twiddles W_N^(n1 k)
template <int N, int R1, int N1, bool INV>
FX_FN void stage_a(const ci64 (&x)[N], ci64 (&y)[N / R1]) {
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int i = 0; i < N / R1; ++i) y[i] = x[N1 + R1 * i];
  if constexpr (N / R1 == 8) dft8<INV>(y);
  else dft4<INV>(y[0], y[1], y[2], y[3]);
  y[1] = twiddle_n<N1 * 1, N, INV>(y[1]);
  y[2] = twiddle_n<N1 * 2, N, INV>(y[2]);
  y[3] = twiddle_n<N1 * 3, N, INV>(y[3]);
  if constexpr (N / R1 == 8) {
    y[4] = twiddle_n<N1 * 4, N, INV>(y[4]);
    y[5] = twiddle_n<N1 * 5, N, INV>(y[5]);
    y[6] = twiddle_n<N1 * 6, N, INV>(y[6]);
    y[7] = twiddle_n<N1 * 7, N, INV>(y[7]);
  }
}

// x <- DFT_N(x), N = 16 (4 x 4), 24 (3 x 8) or 32 (4 x 8), natural order in
// and out: forward exp(-2 pi i n k / N), inverse the conjugate (unnormalised)
template <int N, bool INV>
FX_FN void dft(ci64 (&x)[N]) {
  static_assert(N == 16 || N == 24 || N == 32, "transform length");
  constexpr int R1 = N == 24 ? 3 : 4, R2 = N / R1;
  ci64 y0[R2], y1[R2], y2[R2], y3[R2];
  stage_a<N, R1, 0, INV>(x, y0);
  stage_a<N, R1, 1, INV>(x, y1);
  stage_a<N, R1, 2, INV>(x, y2);
  if constexpr (R1 == 4) stage_a<N, R1, 3, INV>(x, y3);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int k = 0; k < R2; ++k) {
    if constexpr (R1 == 4) dft4<INV>(y0[k], y1[k], y2[k], y3[k]);
    else dft3<INV>(y0[k], y1[k], y2[k]);
    x[k] = y0[k];
    x[k + R2] = y1[k];
    x[k + 2 * R2] = y2[k];
    if constexpr (R1 == 4) x[k + 3 * R2] = y3[k];
  }
}

// DCT-I of length H + 1 (H even), in place: U(k) = x_0 + (-1)^k x_H
// + 2 sum_(0<d<H) x_d cos(pi k d / H), by pairing d with H - d: the even
// outputs are the DCT-I of length H / 2 + 1 of the pair sums, the odd ones
// H / 2 terms each over the pair differences.
template <int H, int K, int D>
FX_FN i64 dct_odd_terms(const i64* od) {  // 2 sum_(d >= D) od_d cos(pi K d / H), d < H / 2
  if constexpr (2 * D >= H) {
    return 0;
  } else {
    constexpr int N2 = 2 * H, NN = 64 % N2 == 0 ? 64 : 48;
    constexpr int m0 = (K * D) % N2;
    constexpr int m1 = m0 > H ? N2 - m0 : m0;       // cos(2 pi m / N2), m in [0, H]
    constexpr bool minus = 2 * m1 > H;
    constexpr int m = (minus ? H - m1 : m1) * (NN / N2);  // in [0, NN / 4]
    const i64 rest = dct_odd_terms<H, K, D + 1>(od);
    if constexpr (4 * m == NN) {
      return rest;
    } else if constexpr (m == 0) {
      return minus ? rest - od[D] : rest + od[D];
    } else {
      constexpr i64 v = NN == 64 ? fx_cos64(m) : fx_cos48(m);
      constexpr int f = NN == 64 ? fx_cos64_form(m) : fx_cos48_form(m);
      const i64 p = mul_formed<f, v>(od[D]);
      return minus ? rest - p : rest + p;
    }
  }
}
template <int H, int K>
FX_FN void dct_odd_outputs(const i64* od, i64* x, int stride) {
  if constexpr (K < H) {
    x[K * stride] = od[0] + 2 * dct_odd_terms<H, K, 1>(od);
    dct_odd_outputs<H, K + 2>(od, x, stride);
  }
}
template <int H, int STRIDE>
FX_FN void dct1(i64* x) {
  if constexpr (H == 1) {
    const i64 a = x[0], b = x[STRIDE];
    x[0] = a + b;
    x[STRIDE] = a - b;
  } else if constexpr (H % 2 == 1) {  // H = 3 (N = 24, 48): direct, cosines 1, 1/2
    const i64 a = x[0], b = x[STRIDE], c = x[2 * STRIDE], d = x[3 * STRIDE];
    x[0] = a + d + 2 * (b + c);
    x[STRIDE] = a - d + b - c;
    x[2 * STRIDE] = a + d - b - c;
    x[3 * STRIDE] = a - d - 2 * (b - c);
  } else {
    i64 ev[H / 2 + 1], od[H / 2];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int d = 0; d < H / 2; ++d) {
      const i64 a = x[d * STRIDE], b = x[(H - d) * STRIDE];
      ev[d] = a + b;
      od[d] = a - b;
    }
    ev[H / 2] = 2 * x[(H / 2) * STRIDE];  // cos(pi k / 2) = +-1 at weight 2
    dct1<H / 2, 1>(ev);
    dct_odd_outputs<H, 1>(od, x, STRIDE);
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k <= H / 2; ++k) x[2 * k * STRIDE] = ev[k];
  }
}

}  // namespace fx
}  // namespace lbo
