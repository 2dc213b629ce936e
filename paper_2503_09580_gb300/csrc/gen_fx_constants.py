"""Write fx_constants.h: the multipliers of the 64-bit fixed-point transforms
(fx64.cuh) as 64-bit integers, from 60-digit decimal arithmetic
(gen_twiddles_hi.py): tan(a/2) and sin(a) of the rotations by a = 2 pi r / n
(n = 64 and 48, a up to 45 degrees), and cos(2 pi m / n) of the DCT-I.  Each
is round(x 2^64) with |x| < 0.46: a larger x is held as its distance to 1/2 or
to 1, which the code adds back (fx_form).

    python gen_fx_constants.py > fx_constants.h
"""
from decimal import ROUND_HALF_EVEN, Decimal

from gen_twiddles_hi import cos_sin, pi

P = pi()


def q64(x):
    return int((x * Decimal(2) ** 64).to_integral_value(ROUND_HALF_EVEN))


def emit(name, n, rows, what):
    print("// %s" % (what % n))
    print("LBO_HD constexpr long long %s(int m) {" % name)
    print("  switch (m) {")
    for m, v in rows:
        print("    case %d: return %dLL;" % (m, v))
    print("    default: return 0;")
    print("  }")
    print("}")


def tan_half(m, n):
    c, s = cos_sin(2 * P * m / n)
    return s / (1 + c)


def form(x):
    """0: x itself (below 0.46), 1: x - 1/2 (0.46 .. 0.54), 2: 1 - x (above)."""
    return 0 if x < Decimal("0.46") else 2 if x > Decimal("0.54") else 1


def shrunk(x):
    x = x.quantize(Decimal(10) ** -50)
    return (x, x - Decimal("0.5"), 1 - x)[form(x)]


def emit_form(name, rows):
    print("LBO_HD constexpr int %s(int m) {" % name)
    print("  switch (m) {")
    for m, x in rows:
        print("    case %d: return %d;" % (m, form(x)))
    print("    default: return 0;")
    print("  }")
    print("}")


if __name__ == "__main__":
    print("// Generated by gen_fx_constants.py: round(x 2^64) of the fixed-point transforms' multipliers.")
    print("#pragma once")
    print("#ifndef LBO_HD")
    print("#ifdef __CUDACC__")
    print("#define LBO_HD __host__ __device__")
    print("#else")
    print("#define LBO_HD")
    print("#endif")
    print("#endif")
    for n in (64, 48):
        emit("fx_tan_half%d" % n, n, [(m, q64(tan_half(m, n))) for m in range(1, n // 8 + 1)], "tan(pi m / %d)")
        sines = [(m, cos_sin(2 * P * m / n)[1]) for m in range(1, n // 8 + 1)]
        emit("fx_sin%d" % n, n, [(m, q64(shrunk(x))) for m, x in sines], "sin(2 pi m / %d) in its form")
        emit_form("fx_sin%d_form" % n, sines)
        cosines = [(m, cos_sin(2 * P * m / n)[0]) for m in range(1, n // 4 + 1)]
        emit("fx_cos%d" % n, n, [(m, q64(shrunk(x))) for m, x in cosines], "cos(2 pi m / %d) in its form")
        emit_form("fx_cos%d_form" % n, cosines)
    r = Decimal("0.5").sqrt()
    print("constexpr long long kFxOneMinusSqrtHalf = %dLL;  // 1 - 1/sqrt 2" % q64(1 - r))
    print("constexpr long long kFxOneMinusSqrt34 = %dLL;  // 1 - sqrt(3)/2" % q64(1 - Decimal(3).sqrt() / 2))
