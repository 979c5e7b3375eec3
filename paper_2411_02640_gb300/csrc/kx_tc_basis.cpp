// Functions of temperature shared by a family of matrices, for the
// tensor-core transport kernels.
//
// Every mixing sum of the transport properties is a product of the state's
// mole fractions with a matrix that depends on temperature alone:
// sum_j X_j / D_kj(T) (Eq. (mix_diff)), sum_j X_j phi_kj(T) (Wilke, App.
// A.3.5; phi_kj depends on T through eta_k/eta_j only), sum_j X_j lambda_j(T)
// and sum_j X_j / lambda_j(T) (Mathur).  Divided by a common factor g(T), the
// entries are smooth in ln T, so the whole matrix is
//   c_rj(T) = c_rj,0 + sum_m c_rj,m phi_m(t),  t = (ln T - L_mid)/L_half in [-1, 1]
// with few basis functions phi_m, and the sums become products with constant
// matrices.  Here: the entries at Chebyshev nodes, their Chebyshev
// coefficients, the singular vectors of those (the shortest such basis, by
// one-sided Jacobi rotations on the triangular factor of a Householder
// factorisation), the coefficients c_rj,m and phi_m as polynomials in t.
#include "kx_tc_basis.h"

#include <algorithm>
#include <cmath>

#include "kx_emit_text.h"

namespace kx {

namespace {

HostDD dd(double x) { return {x, 0.0}; }
HostDD dd_neg(HostDD a) { return {-a.hi, -a.lo}; }

// e^x in double-double: x = k ln 2 + r, Taylor series of e^(r/16), four squarings
double exp_dd(HostDD x) {
  const HostDD ln2 = {0.6931471805599453, 2.3190468138462996e-17};
  const double k = std::nearbyint(x.hi / ln2.hi);
  HostDD r = hdd_add(x, dd_neg(hdd_mul(ln2, dd(k))));
  r = hdd_mul(r, dd(0.0625));
  HostDD s = dd(1.0);
  for (int n = 18; n >= 1; --n) {
    // s = 1 + r s / n
    HostDD q = hdd_mul(r, s);
    const double a = q.hi / n;
    const double rest = std::fma(-a, (double)n, q.hi) + q.lo;
    s = hdd_add(dd(1.0), hdd_norm(a, rest / n));
  }
  for (int j = 0; j < 4; ++j) s = hdd_mul(s, s);
  return std::ldexp(s.hi + s.lo, (int)k);
}

// cos(pi r / (2 N)) for r = 0 .. 2 N, Taylor series in double-double
double cos_dd(int r, int N) {
  const HostDD pi = {3.141592653589793, 1.2246467991473532e-16};
  const double c = (double)r / (2 * N);   // exact: N is a power of two
  const HostDD x = hdd_mul(pi, dd(c));
  HostDD x2 = dd_neg(hdd_mul(x, x));
  HostDD s = dd(1.0);
  for (int n = 26; n >= 1; --n) {
    HostDD q = hdd_mul(x2, s);
    const double d = (2.0 * n) * (2.0 * n - 1.0);
    const double a = q.hi / d;
    const double rest = std::fma(-a, d, q.hi) + q.lo;
    s = hdd_add(dd(1.0), hdd_norm(a, rest / d));
  }
  return s.hi + s.lo;
}

constexpr int kNodes = 32;

// polynomial with coefficients c[0..4] at x
HostDD poly(const double* c, double x) {
  HostDD s = dd(c[4]);
  for (int n = 3; n >= 0; --n) s = hdd_add(hdd_mul(s, dd(x)), dd(c[n]));
  return s;
}

}  // namespace

bool tc_basis(const Mechanism& m, int part, bool mixed, TcBasis& b) {
  if (m.fit_direct) return false;
  const int ns = m.ns;
  b = TcBasis();
  b.ns = ns;
  b.K = (ns + 15) / 16 * 16;
  b.first = part == 2 ? 2 : 5;
  b.rows = b.first + ns;
  const int rows = b.rows;
  double node[kNodes];
  for (int i = 0; i < kNodes; ++i) node[i] = cos_dd(2 * i + 1, kNodes);
  // the fits about L_mid, and the means that the common factors are made of
  std::vector<double> pe(5 * (size_t)ns), pl(5 * (size_t)ns), pd;
  double me[5] = {0}, ml[5] = {0}, md[5] = {0};
  for (int k = 0; k < ns; ++k) {
    shift_poly(&m.eta[5 * k], kTcLmid, 1.0, &pe[5 * k]);
    shift_poly(&m.lam[5 * k], kTcLmid, 1.0, &pl[5 * k]);
    for (int n = 0; n < 5; ++n) { me[n] += pe[5 * k + n] / ns; ml[n] += pl[5 * k + n] / ns; }
  }
  if (part == 2) {
    pd.resize(5 * (size_t)ns * ns);
    const double np = std::max(1.0, 0.5 * ns * (ns - 1.0));
    for (int k = 0; k < ns; ++k)
      for (int j = k; j < ns; ++j) {
        double d[5];
        shift_poly(&m.dif[5 * ((size_t)k * ns + j)], kTcLmid, 1.0, d);
        for (int n = 0; n < 5; ++n) {
          pd[5 * ((size_t)k * ns + j) + n] = pd[5 * ((size_t)j * ns + k) + n] = d[n];
          if (j != k) md[n] += d[n] / np;
        }
      }
  }
  // rounded to float pairs: the kernel evaluates the same polynomials
  auto fp = [](double x) { const float h = (float)x; return (double)h + (double)(float)(x - (double)h); };
  for (int n = 0; n < 5; ++n) {
    me[n] = fp(me[n]); ml[n] = fp(ml[n]); md[n] = fp(md[n]);
    b.g0[n] = part == 2 ? -md[n] : me[n];   // 1/D common factor; 1/(common factor of 1/eta)
    b.g1[n] = ml[n];
  }
  b.g0c = exp_dd(dd(b.g0[0]));
  b.g1c = exp_dd(dd(b.g1[0]));
  // entries at the nodes, [row][species][node]
  std::vector<double> f((size_t)rows * ns * kNodes, 0.0);
  auto at = [&](int r, int j) { return &f[((size_t)r * ns + j) * kNodes]; };
  for (int i = 0; i < kNodes; ++i) {
    const double x = kTcLhalf * node[i];
    if (part == 2) {
      const HostDD g = poly(md, x);
      for (int k = 0; k < ns; ++k)
        for (int j = k + 1; j < ns; ++j) {
          const double v = exp_dd(hdd_add(g, dd_neg(poly(&pd[5 * ((size_t)k * ns + j)], x))));
          at(2 + k, j)[i] = v / m.W[j];
          at(2 + j, k)[i] = v / m.W[k];
        }
    } else {
      const HostDD g = poly(me, x), gl = poly(ml, x);
      std::vector<double> u(ns), v(ns), ie(ns);
      for (int k = 0; k < ns; ++k) {
        const HostDD p = poly(&pe[5 * k], x);
        const double w4 = std::sqrt(std::sqrt(m.W[k]));
        u[k] = exp_dd(hdd_mul(p, dd(0.5))) / w4;
        v[k] = exp_dd(hdd_mul(p, dd(-0.5))) * w4;
        ie[k] = exp_dd(hdd_add(g, dd_neg(p)));   // g / eta_k
        const HostDD q = hdd_add(poly(&pl[5 * k], x), dd_neg(gl));
        at(1, k)[i] = exp_dd(q) / m.W[k];
        at(2, k)[i] = exp_dd(dd_neg(q)) / m.W[k];
      }
      for (int k = 0; k < ns; ++k)
        for (int j = 0; j < ns; ++j) {
          const double w = std::fma(u[k], v[j], 1.0);
          at(5 + k, j)[i] = w * w / std::sqrt(8.0 * (1.0 + m.W[k] / m.W[j])) * ie[k] / m.W[j];
        }
    }
    for (int j = 0; j < ns; ++j) {
      at(0, j)[i] = 1.0 / m.W[j];
      if (part == 2) at(1, j)[i] = 1.0;
    }
  }
  // powers of two that bring every column's entries, then every row's, near one
  b.ecol.assign(ns, 0);
  std::vector<double> lg(ns, 0.0);
  for (int j = 0; j < ns; ++j) {
    int cnt = 0;
    for (int k = 0; k < ns; ++k) {
      const double v = at(b.first + k, j)[kNodes / 2];
      if (v > 0) { int e; const double mn = std::frexp(v, &e); lg[j] += e + 2.0 * (mn - 1.0); ++cnt; }
    }
    if (cnt) lg[j] /= cnt;
  }
  const double top = *std::max_element(lg.begin(), lg.end());
  for (int j = 0; j < ns; ++j) {
    b.ecol[j] = (int)std::nearbyint(lg[j] - top);
    if (b.ecol[j] < -40) return false;
  }
  // the conductivities span an order of magnitude between light and heavy species: each of their two
  // rows is split in two, so that a mixture without the species of the largest entries keeps its digits
  if (part != 2)
    for (int r = 1; r <= 2; ++r) {
      double mx = 0;
      for (int j = 0; j < ns; ++j) mx = std::max(mx, std::ldexp(at(r, j)[kNodes / 2], -b.ecol[j]));
      for (int j = 0; j < ns; ++j)
        if (std::ldexp(at(r, j)[kNodes / 2], -b.ecol[j]) < 0.2 * mx)
          for (int i = 0; i < kNodes; ++i) std::swap(at(r, j)[i], at(r + 2, j)[i]);
    }
  b.rho.assign(rows, 0);
  for (int r = 0; r < rows; ++r) {
    double mx = 0;
    for (int j = 0; j < ns; ++j)
      for (int i = 0; i < kNodes; ++i) {
        const double v = std::ldexp(at(r, j)[i], -b.ecol[j]);
        if (!std::isfinite(v) || v < 0) return false;
        mx = std::max(mx, v);
      }
    int e = 0;
    if (mx > 0) std::frexp(mx, &e);
    b.rho[r] = e;
    for (int j = 0; j < ns; ++j)
      for (int i = 0; i < kNodes; ++i) at(r, j)[i] = std::ldexp(at(r, j)[i], -b.ecol[j] - e);
  }
  // Chebyshev coefficients
  // T_n(node_i) = cos(pi n (2 i + 1)/(2 N)) at the exact angles (a recurrence from the rounded nodes leaves
  // errors of 2^-50 that are alike in every entry)
  std::vector<double> cosine(2 * kNodes + 1), tn(kNodes * kNodes);
  for (int r = 0; r <= 2 * kNodes; ++r) cosine[r] = cos_dd(r, kNodes);
  for (int i = 0; i < kNodes; ++i)
    for (int n = 0; n < kNodes; ++n) {
      const int r = n * (2 * i + 1) % (4 * kNodes);
      tn[n * kNodes + i] = cosine[r <= 2 * kNodes ? r : 4 * kNodes - r];
    }
  const size_t nr = (size_t)rows * ns;
  std::vector<double> c0(nr), all(nr * kNodes);
  std::vector<double> most(kNodes, 0.0);
  for (size_t r = 0; r < nr; ++r) {
    for (int n = 0; n < kNodes; ++n) {
      double s = 0;
      for (int i = 0; i < kNodes; ++i) s += f[r * kNodes + i] * tn[n * kNodes + i];
      s *= 2.0 / kNodes;
      if (n == 0) c0[r] = 0.5 * s;
      all[r * kNodes + n] = s;
      most[n] += s * s / nr;
    }
  }
  // degrees whose coefficients stand out of the rounding of the entries (2^-52 in the mean square): 1..nc
  // enter the basis.  (The functions of the smallest coefficients would else hold high powers of t in full
  // measure, whose polynomials cancel badly at t = +-1.)
  int nc = kNodes - 1;
  while (nc > 1 && std::sqrt(most[nc]) < std::ldexp(1.0, mixed ? -28 : -52)) --nc;
  std::vector<double> C(nr * nc);
  for (size_t r = 0; r < nr; ++r)
    for (int n = 1; n <= nc; ++n) C[r * nc + n - 1] = all[r * kNodes + n];
  // Householder triangular factor of C
  std::vector<double> A = C;
  for (int k = 0; k < nc && (size_t)k < nr; ++k) {
    double s = 0;
    for (size_t r = k; r < nr; ++r) s += A[r * nc + k] * A[r * nc + k];
    const double nrm = std::sqrt(s);
    if (nrm == 0) continue;
    const double al = A[k * nc + k] > 0 ? -nrm : nrm;
    const double vk = A[k * nc + k] - al, vv = s - A[k * nc + k] * A[k * nc + k] + vk * vk;
    std::vector<double> w(nr - k);
    w[0] = vk;
    for (size_t r = k + 1; r < nr; ++r) w[r - k] = A[r * nc + k];
    std::vector<double> dots(nc, 0.0);
    for (size_t r = k; r < nr; ++r)
      for (int j = k; j < nc; ++j) dots[j] += w[r - k] * A[r * nc + j];
    for (size_t r = k; r < nr; ++r)
      for (int j = k; j < nc; ++j) A[r * nc + j] -= 2.0 / vv * dots[j] * w[r - k];
  }
  const int tr = (int)std::min<size_t>(nr, nc);
  std::vector<double> R((size_t)nc * nc, 0.0), V((size_t)nc * nc, 0.0);
  for (int i = 0; i < tr; ++i)
    for (int j = i; j < nc; ++j) R[i * nc + j] = A[i * nc + j];
  for (int j = 0; j < nc; ++j) V[j * nc + j] = 1.0;
  // one-sided Jacobi: columns of R V orthogonal
  for (int sweep = 0; sweep < 30; ++sweep) {
    bool done = true;
    for (int p = 0; p < nc; ++p)
      for (int q = p + 1; q < nc; ++q) {
        double al = 0, be = 0, ga = 0;
        for (int i = 0; i < nc; ++i) {
          al += R[i * nc + p] * R[i * nc + p];
          be += R[i * nc + q] * R[i * nc + q];
          ga += R[i * nc + p] * R[i * nc + q];
        }
        if (std::fabs(ga) <= 1e-15 * std::sqrt(al * be) || ga == 0) continue;
        done = false;
        const double ze = (be - al) / (2.0 * ga);
        const double t = (ze >= 0 ? 1.0 : -1.0) / (std::fabs(ze) + std::sqrt(1.0 + ze * ze));
        const double c = 1.0 / std::sqrt(1.0 + t * t), s = c * t;
        for (int i = 0; i < nc; ++i) {
          double x = R[i * nc + p], y = R[i * nc + q];
          R[i * nc + p] = c * x - s * y; R[i * nc + q] = s * x + c * y;
          x = V[i * nc + p]; y = V[i * nc + q];
          V[i * nc + p] = c * x - s * y; V[i * nc + q] = s * x + c * y;
        }
      }
    if (done) break;
  }
  std::vector<std::pair<double, int>> order(nc);
  for (int j = 0; j < nc; ++j) {
    double s = 0;
    for (int i = 0; i < nc; ++i) s += R[i * nc + j] * R[i * nc + j];
    order[j] = {-s, j};
  }
  std::sort(order.begin(), order.end());
  // coefficients in that basis; as many as the residual needs
  std::vector<double> P(nr * nc);
  std::vector<double> big(nc, 0.0), rest(nc + 1, 0.0);
  for (size_t r = 0; r < nr; ++r) {
    double tail = 0;
    for (int q = nc - 1; q >= 0; --q) {
      const int j = order[q].second;
      double s = 0;
      for (int n = 0; n < nc; ++n) s += C[r * nc + n] * V[n * nc + j];
      P[r * nc + q] = s;
      big[q] = std::max(big[q], std::fabs(s));
      tail += std::fabs(s);
      rest[q] = std::max(rest[q], tail);
    }
  }
  const double tol = std::ldexp(1.0, mixed ? -26 : -50);
  int M = 0;
  while (M < nc && rest[M] > tol) ++M;
  if (M > kTcMaxBasis) return false;
  b.M = M;
  b.E.assign(M + 1, 0);
  b.phi.assign(M + 1, std::vector<double>(1, 1.0));
  b.cheb = b.phi;
  for (int q = 0; q < M; ++q) {
    int e;
    std::frexp(big[q], &e);
    b.E[q + 1] = e;
    const int j = order[q].second;
    std::vector<double> ch(kNodes, 0.0);
    for (int n = 1; n <= nc; ++n) ch[n] = std::ldexp(V[(n - 1) * nc + j], e);
    // drop the highest terms below the accuracy that the basis function is needed to
    const double cut = std::ldexp(1.0, mixed ? -27 : -51);
    int deg = nc;
    double drop = 0;
    while (deg > 1 && drop + std::fabs(ch[deg]) < cut) drop += std::fabs(ch[deg--]);
    std::vector<double> mono(deg + 1, 0.0), t0(deg + 1, 0.0), t1(deg + 1, 0.0), t2(deg + 1, 0.0);
    t0[0] = 1.0;
    t1[1] = 1.0;
    for (int n = 1; n <= deg; ++n) {
      for (int i = 0; i <= n; ++i) mono[i] += ch[n] * t1[i];
      for (int i = 0; i <= deg; ++i) t2[i] = (i > 0 ? 2.0 * t1[i - 1] : 0.0) - t0[i];
      t0 = t1; t1 = t2;
    }
    b.phi[q + 1] = mono;
    b.cheb[q + 1].assign(ch.begin(), ch.begin() + deg + 1);
  }
  b.coef.assign(nr * (size_t)(M + 1), 0.0);
  for (size_t r = 0; r < nr; ++r) {
    b.coef[r * (M + 1)] = c0[r];
    if (std::fabs(c0[r]) > 1.0) return false;
    for (int q = 0; q < M; ++q) b.coef[r * (M + 1) + q + 1] = std::ldexp(P[r * nc + q], -b.E[q + 1]);
  }
  return true;
}

bool tc_thermo(const Mechanism& m, TcBasis& b, std::vector<double>& mids) {
  const int ns = m.ns;
  b = TcBasis();
  b.ns = ns;
  b.K = (ns + 15) / 16 * 16;
  mids = m.Tmid;
  std::sort(mids.begin(), mids.end());
  mids.erase(std::unique(mids.begin(), mids.end()), mids.end());
  if (mids.size() > 4) return false;
  b.rows = 12 * (int)mids.size();
  b.E.assign(1, 0);
  b.phi.assign(1, std::vector<double>(1, 1.0));
  b.cheb = b.phi;
  b.ecol.assign(ns, 0);
  double wmin = m.W[0];
  for (double w : m.W) wmin = std::min(wmin, w);
  for (int k = 0; k < ns; ++k) {
    int e;
    std::frexp(wmin / m.W[k], &e);
    b.ecol[k] = std::min(0, e);
    if (b.ecol[k] < -40) return false;
  }
  std::vector<double> f((size_t)b.rows * ns, 0.0);
  for (int k = 0; k < ns; ++k) {
    const int g = (int)(std::lower_bound(mids.begin(), mids.end(), m.Tmid[k]) - mids.begin());
    for (int rg = 0; rg < 2; ++rg) {
      const double* a = rg == 0 ? &m.a_lo[7 * k] : &m.a_hi[7 * k];
      double d[5];
      shift_poly(a, kThTc[rg], 1.0, d);
      HostDD h = {a[5], 0.0}, t = {kThTc[rg], 0.0};
      for (int n = 0; n < 5; ++n) {
        const HostDD q = hdd_mul({a[n], 0.0}, t);
        const double v = q.hi / (n + 1), r = std::fma(-v, (double)(n + 1), q.hi) + q.lo;
        h = hdd_add(h, hdd_norm(v, r / (n + 1)));
        t = hdd_mul(t, {kThTc[rg], 0.0});
      }
      double p = 1.0;
      for (int n = 0; n < 5; ++n, p *= kThHalf[rg]) f[(size_t)(12 * g + 6 * rg + n) * ns + k] = d[n] * p * (R_U / m.W[k]);
      f[(size_t)(12 * g + 6 * rg + 5) * ns + k] = (h.hi + h.lo) * (R_U / m.W[k]);
    }
  }
  b.rho.assign(b.rows, 0);
  b.coef.assign(f.size(), 0.0);
  for (int r = 0; r < b.rows; ++r) {
    double mx = 0;
    for (int k = 0; k < ns; ++k) {
      const double v = std::ldexp(f[(size_t)r * ns + k], -b.ecol[k]);
      if (!std::isfinite(v)) return false;
      mx = std::max(mx, std::fabs(v));
    }
    int e = 0;
    if (mx > 0) std::frexp(mx, &e);
    if (e > 100 || e < -100) return false;
    b.rho[r] = e;
    for (int k = 0; k < ns; ++k) b.coef[(size_t)r * ns + k] = std::ldexp(f[(size_t)r * ns + k], -b.ecol[k] - e);
  }
  return true;
}

}  // namespace kx
