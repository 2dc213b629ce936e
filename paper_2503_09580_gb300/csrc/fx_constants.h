// Generated by gen_fx_constants.py: round(x 2^64) of the fixed-point transforms' multipliers.
#pragma once
#ifndef LBO_HD
#ifdef __CUDACC__
#define LBO_HD __host__ __device__
#else
#define LBO_HD
#endif
#endif
// tan(pi m / 64)
LBO_HD constexpr long long fx_tan_half64(int m) {
  switch (m) {
    case 1: return 906230424844939522LL;
    case 2: return 1816845711190106722LL;
    case 3: return 2736315999040864331LL;
    case 4: return 3669285534148243471LL;
    case 5: return 4620668848450484397LL;
    case 6: return 5595758638113189652LL;
    case 7: return 6600350569198068924LL;
    case 8: return 7640891576956012809LL;
    default: return 0;
  }
}
// sin(2 pi m / 64) in its form
LBO_HD constexpr long long fx_sin64(int m) {
  switch (m) {
    case 1: return 1808097102496279522LL;
    case 2: return 3598781241489102189LL;
    case 3: return 5354807149832443555LL;
    case 4: return 7059263338087549767LL;
    case 5: return -527637075443782536LL;
    case 6: return 8198282170225769627LL;
    case 7: return 6744253518662684480LL;
    case 8: return 5402926248376769404LL;
    default: return 0;
  }
}
LBO_HD constexpr int fx_sin64_form(int m) {
  switch (m) {
    case 1: return 0;
    case 2: return 0;
    case 3: return 0;
    case 4: return 0;
    case 5: return 1;
    case 6: return 2;
    case 7: return 2;
    case 8: return 2;
    default: return 0;
  }
}
// cos(2 pi m / 64) in its form
LBO_HD constexpr long long fx_cos64(int m) {
  switch (m) {
    case 1: return 88826114722943760LL;
    case 2: return 354449014849699498LL;
    case 3: return 794310606647799060LL;
    case 4: return 1404174782535421627LL;
    case 5: return 2178168217113098606LL;
    case 6: return 3108836930497996774LL;
    case 7: return 4187218074224949849LL;
    case 8: return 5402926248376769404LL;
    case 9: return 6744253518662684480LL;
    case 10: return 8198282170225769627LL;
    case 11: return -527637075443782536LL;
    case 12: return 7059263338087549767LL;
    case 13: return 5354807149832443555LL;
    case 14: return 3598781241489102189LL;
    case 15: return 1808097102496279522LL;
    case 16: return 0LL;
    default: return 0;
  }
}
LBO_HD constexpr int fx_cos64_form(int m) {
  switch (m) {
    case 1: return 2;
    case 2: return 2;
    case 3: return 2;
    case 4: return 2;
    case 5: return 2;
    case 6: return 2;
    case 7: return 2;
    case 8: return 2;
    case 9: return 2;
    case 10: return 2;
    case 11: return 1;
    case 12: return 0;
    case 13: return 0;
    case 14: return 0;
    case 15: return 0;
    case 16: return 0;
    default: return 0;
  }
}
// tan(pi m / 48)
LBO_HD constexpr long long fx_tan_half48(int m) {
  switch (m) {
    case 1: return 1209063484257398157LL;
    case 2: return 2428559929659355502LL;
    case 3: return 3669285534148243471LL;
    case 4: return 4942790177534073029LL;
    case 5: return 6261825837983445860LL;
    case 6: return 7640891576956012809LL;
    default: return 0;
  }
}
// sin(2 pi m / 48) in its form
LBO_HD constexpr long long fx_sin48(int m) {
  switch (m) {
    case 1: return 2407783262799110479LL;
    case 2: return 4774368686408090022LL;
    case 3: return 7059263338087549767LL;
    case 4: return 0LL;
    case 5: return 7217077790839976240LL;
    case 6: return 5402926248376769404LL;
    default: return 0;
  }
}
LBO_HD constexpr int fx_sin48_form(int m) {
  switch (m) {
    case 1: return 0;
    case 2: return 0;
    case 3: return 0;
    case 4: return 1;
    case 5: return 2;
    case 6: return 2;
    default: return 0;
  }
}
// cos(2 pi m / 48) in its form
LBO_HD constexpr long long fx_cos48(int m) {
  switch (m) {
    case 1: return 157814452752426473LL;
    case 2: return 628557561968679382LL;
    case 3: return 1404174782535421627LL;
    case 4: return 2471395088767036514LL;
    case 5: return 3811958045334532105LL;
    case 6: return 5402926248376769404LL;
    case 7: return 7217077790839976240LL;
    case 8: return 0LL;
    case 9: return 7059263338087549767LL;
    case 10: return 4774368686408090022LL;
    case 11: return 2407783262799110479LL;
    case 12: return 0LL;
    default: return 0;
  }
}
LBO_HD constexpr int fx_cos48_form(int m) {
  switch (m) {
    case 1: return 2;
    case 2: return 2;
    case 3: return 2;
    case 4: return 2;
    case 5: return 2;
    case 6: return 2;
    case 7: return 2;
    case 8: return 1;
    case 9: return 0;
    case 10: return 0;
    case 11: return 0;
    case 12: return 0;
    default: return 0;
  }
}
constexpr long long kFxOneMinusSqrtHalf = 5402926248376769404LL;  // 1 - 1/sqrt 2
constexpr long long kFxOneMinusSqrt34 = 2471395088767036514LL;  // 1 - sqrt(3)/2
