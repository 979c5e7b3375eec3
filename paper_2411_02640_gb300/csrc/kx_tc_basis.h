// Temperature basis of the tensor-core transport kernels (kx_tc_basis.cpp).
#pragma once

#include <vector>

#include "kx_internal.h"

namespace kx {

// Temperatures that the basis covers: 200 to 4000 K (t = -1 .. 1).
constexpr double kTcTlo = 200.0, kTcThi = 4000.0;
constexpr double kTcLmid = 6.796183424706478;     // ln sqrt(200 * 4000)
constexpr double kTcTmid = 894.4271206813461;        // e^L_mid
constexpr double kTcLhalf = 1.4978661367769954;   // ln(4000/200) / 2
constexpr int kTcMaxBasis = 24;

// Rows: part 2 (diffusion) 0: 1/W_j, 1: one, 2 + k: 1/(W_j D_kj) over g0, j != k;
// part 1 (viscosity, conductivity) 0: 1/W_j, 1 and 3: lambda_j/W_j over g1 (of the species with
// large and small entries), 2 and 4: 1/(W_j lambda_j) times g1, 5 + k: phi_kj/(W_j eta_k) times g0; g0, g1 = exp of the polynomials below in
// ln T - L_mid.  Row r's entry of species j is
//   2^(rho_r + ecol_j) sum_m coef[(r ns + j)(M + 1) + m] phi_m(t),  |coef| <= 1, phi_0 = 1,
// phi_m scaled by 2^E_m so that the coefficients fill [-1, 1].
struct TcBasis {
  int ns = 0, K = 0, rows = 0, first = 0, M = 0;
  std::vector<int> E, ecol, rho;
  std::vector<std::vector<double>> phi, cheb;   // [M + 1] polynomials in t: of its powers, of T_n(t)
  std::vector<double> coef;
  double g0[5] = {0}, g1[5] = {0}, g0c = 1.0, g1c = 1.0;   // g0c = e^g0[0], g1c = e^g1[0]
};

bool tc_basis(const Mechanism& m, int part, bool mixed, TcBasis& b);

// Thermo: the NASA-7 blocks are polynomials in T, so their basis is exact: for every distinct T_mid and
// range six rows, R_U/W_j times the coefficients of c_p/R in x = (T - kThTc)/kThHalf (x^0 .. x^4) and
// H/R at x = 0; rows 12 g + 6 (T >= T_mid) + 0 .. 5, M = 0.  mids receives the distinct T_mid.
constexpr double kThTc[2] = {600.0, 2048.0}, kThHalf[2] = {512.0, 2048.0};
bool tc_thermo(const Mechanism& m, TcBasis& b, std::vector<double>& mids);

}  // namespace kx
