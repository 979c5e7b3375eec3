// Text helpers of the CUDA emitters (literals that read back bit-exactly,
// indented lines) and the double-double host arithmetic that the emitted
// constants are computed in.
#pragma once

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <sstream>
#include <string>

namespace kx {

inline std::string fmt(const char* f, ...) {
  va_list ap, ap2;
  va_start(ap, f);
  va_copy(ap2, ap);
  const int n = vsnprintf(nullptr, 0, f, ap);
  va_end(ap);
  std::string out(n > 0 ? n : 0, '\0');
  if (n > 0) vsnprintf(&out[0], n + 1, f, ap2);
  va_end(ap2);
  return out;
}

// float64 literal that reads back bit-exactly
inline std::string D(double v) {
  if (std::isnan(v)) return "KX_NAN";
  if (std::isinf(v)) return v > 0 ? "KX_INF" : "(-KX_INF)";
  std::string s = fmt("%.17g", v);
  if (s.find_first_of(".en") == std::string::npos) s += ".0";
  return s[0] == '-' ? "(" + s + ")" : s;
}

// float32 literal (value rounded to float first)
inline std::string F(double v) {
  float f = (float)v;
  if (std::isinf(f)) return v > 0 ? "__int_as_float(0x7f800000)" : "(-__int_as_float(0x7f800000))";
  std::string s = fmt("%.9g", (double)f);
  if (s.find_first_of(".en") == std::string::npos) s += ".0";
  s += "f";
  return s[0] == '-' ? "(" + s + ")" : s;
}

inline std::string fpair(double v) {
  const float h = (float)v;
  const float l = (float)(v - (double)h);
  return F(h) + "," + F(l);
}

inline std::string DFc(double v) { return "kx_mk(" + fpair(v) + ")"; }

struct Out {
  std::ostringstream o;
  int ind = 1;
  void operator()(const std::string& s) { o << std::string(2 * ind, ' ') << s << "\n"; }
};

// Double-double host arithmetic from error-free transformations (std::fma is exact IEEE arithmetic
// on every host), so that the emitted constants are the same bits on every platform: long double is
// 80-bit on x86-64 and 128-bit on aarch64.
struct HostDD { double hi, lo; };
inline HostDD hdd_norm(double a, double b) { const double s = a + b; return {s, b - (s - a)}; }
inline HostDD hdd_add(HostDD a, HostDD b) {
  const double s = a.hi + b.hi, bb = s - a.hi;
  const double e = (a.hi - (s - bb)) + (b.hi - bb);
  return hdd_norm(s, e + a.lo + b.lo);
}
inline HostDD hdd_mul(HostDD a, HostDD b) {
  const double p = a.hi * b.hi;
  return hdd_norm(p, std::fma(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi));
}

// p(L) = sum c_n L^n re-expanded about L0: d_m = sum_{n>=m} C(n,m) c_n L0^(n-m), in double-double
inline void shift_poly(const double* cf, double L0, double scale, double out[5]) {
  static const double binom[5][5] = {{1, 0, 0, 0, 0}, {1, 1, 0, 0, 0}, {1, 2, 1, 0, 0}, {1, 3, 3, 1, 0}, {1, 4, 6, 4, 1}};
  HostDD pw[5] = {{1.0, 0.0}};
  for (int k = 1; k < 5; ++k) pw[k] = hdd_mul(pw[k - 1], {L0, 0.0});
  for (int mm = 0; mm < 5; ++mm) {
    HostDD d = {0.0, 0.0};
    for (int n = mm; n < 5; ++n) d = hdd_add(d, hdd_mul(hdd_mul({binom[n][mm], 0.0}, {cf[n], 0.0}), pw[n - mm]));
    d = hdd_mul(d, {scale, 0.0});
    out[mm] = d.hi + d.lo;
  }
}

}  // namespace kx
