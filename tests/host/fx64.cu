// Host-only check of the 64-bit fixed-point arithmetic (csrc/fx64.cuh): the
// products against 128-bit integers, the pencil transforms against a direct
// DFT and the DCT-I against its direct sum in long double.  The worst of many
// random cases in units of the last place, one line "<what> <error> <bias>"
// each.  Runs no kernel.
#include <cmath>
#include <cstdio>
#include <random>

#include "../../paper_2503_09580_gb300/csrc/fx64.cuh"

using namespace lbo::fx;

static std::mt19937_64 rng(11);
static const long double pi = 3.141592653589793238462643383279502884L;

// inputs with sum(|re| + |im|) just below 2^60; every fifth case has half of them zero
template <int N, bool INV>
static void transform() {
  std::normal_distribution<double> nd;
  double worst = 0, bias = 0;
  for (int tr = 0; tr < 300; ++tr) {
    ci64 x[N];
    long double re[N], im[N], sum = 0;
    for (int i = 0; i < N; ++i) {
      const double w = tr % 5 == 0 ? (i % 2) : (tr % 5 == 1 ? exp(-0.5 * i) : 1.0);
      re[i] = nd(rng) * w;
      im[i] = nd(rng) * w;
      sum += fabsl(re[i]) + fabsl(im[i]);
    }
    const long double sc = 0.999L * 1152921504606846976.0L / sum;
    for (int i = 0; i < N; ++i) {
      x[i] = ci64{(i64)(re[i] * sc), (i64)(im[i] * sc)};
      re[i] = x[i].x;
      im[i] = x[i].y;
    }
    dft<N, INV>(x);
    long double e2 = 0;
    for (int k = 0; k < N; ++k) {
      long double sr = 0, si = 0;
      for (int n = 0; n < N; ++n) {
        const long double a = (INV ? 2 : -2) * pi * ((n * k) % N) / N;
        sr += re[n] * cosl(a) - im[n] * sinl(a);
        si += re[n] * sinl(a) + im[n] * cosl(a);
      }
      e2 += (x[k].x - sr) * (x[k].x - sr) + (x[k].y - si) * (x[k].y - si);
      bias += (double)(x[k].x - sr + x[k].y - si) / (2.0 * N * 300);
    }
    worst = fmax(worst, sqrt((double)(e2 / (2 * N))));
  }
  ci64 z[N] = {};
  dft<N, INV>(z);
  for (int k = 0; k < N; ++k)
    if (z[k].x || z[k].y) worst = INFINITY;  // zeros stay zeros
  std::printf("dft%d%s %.3f %.3f\n", N, INV ? "i" : "f", worst, bias);
}

template <int H>
static void cosine() {
  std::normal_distribution<double> nd;
  double worst = 0;
  for (int tr = 0; tr < 300; ++tr) {
    i64 x[H + 1];
    long double v[H + 1];
    for (int i = 0; i <= H; ++i) v[i] = x[i] = (i64)(nd(rng) * 1e16);
    dct1<H, 1>(x);
    for (int k = 0; k <= H; ++k) {
      long double s = v[0] + (k % 2 ? -v[H] : v[H]);
      for (int i = 1; i < H; ++i) s += 2 * v[i] * cosl(pi * ((k * i) % (2 * H)) / H);
      worst = fmax(worst, (double)fabsl(s - x[k]));
    }
  }
  std::printf("dct%d %.3f 0\n", H, worst);
}

template <typename F>
static void product(const char* name, bool sign, int ybits, F f) {
  double worst = 0, bias = 0;
  const int n = 200000;
  for (int tr = 0; tr < n; ++tr) {
    i64 y = (i64)(rng() >> (64 - ybits)), t = (i64)(rng() >> (2 + rng() % 40));
    if (rng() & 1) y = -y;
    if (sign && (rng() & 1)) t = -t;
    if (tr % 1000 == 0) y = 0;
    const Mult m = unpack_mult(pack_mult(t));
    const __int128 p = (__int128)y * t;
    const i64 hi = (i64)(p >> 64);
    const double frac = (double)(unsigned long long)p / 18446744073709551616.0;
    const double e = (double)(f(y, m) - hi) - frac;
    worst = fmax(worst, fabs(e));
    bias += e / n;
  }
  std::printf("%s %.3f %.4f\n", name, worst, bias);
}

// mul_pair(): random directions (t, w) of norm 2^62 and below
static void pair() {
  double worst = 0, bias = 0;
  const int n = 200000;
  for (int tr = 0; tr < n; ++tr) {
    i64 y = (i64)(rng() >> 4), z = (i64)(rng() >> 4);
    if (rng() & 1) y = -y;
    if (rng() & 1) z = -z;
    const long double a = (rng() >> 11) * 0x1p-53L * 2 * 3.14159265358979323846L;
    const i64 t = (i64)(cosl(a) * 0x1p62L), w = (i64)(sinl(a) * 0x1p62L) >> (tr % 3 == 0 ? rng() % 50 : 0);
    if (tr % 1000 == 0) y = z = 0;
    const __int128 p = (__int128)y * t + (__int128)z * w;
    const double e = (double)(mul_pair(y, unpack_mult(pack_mult(t)), z, unpack_mult(pack_mult(w))) - (i64)(p >> 64)) -
                     (double)(unsigned long long)p / 18446744073709551616.0;
    worst = fmax(worst, fabs(e));
    bias += e / n;
  }
  std::printf("mul_pair %.3f %.4f\n", worst, bias);
}

int main() {
  pair();
  product("mul", false, 60, [](i64 y, Mult m) { return mul(y, m); });
  product("mul_signed", true, 62, [](i64 y, Mult m) { return mul_signed(y, m, m.th >> 31); });
  product("mul_signed_rounded", true, 62, [](i64 y, Mult m) { return mul_signed_rounded(y, m, m.th >> 31); });
  transform<16, false>();
  transform<16, true>();
  transform<24, false>();
  transform<24, true>();
  transform<32, false>();
  transform<32, true>();
  cosine<8>();
  cosine<12>();
  cosine<16>();
  cosine<24>();
  cosine<32>();
  return 0;
}
