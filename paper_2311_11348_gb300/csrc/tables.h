// Reference-element tables of libswedg (host side).
#pragma once
#include "common.h"

namespace swedg {

template <typename F>
struct RefTablesOf {
  F D[2][KMAX][KMAX];          // D_k[q][i] = int phi_i d_k phi_q
  F Ds[KMAX][KMAX];            // D_1 - D_0 / 2
  F G[2][KMAX][KMAX][KMAX];    // G_k[q][i][j] = int phi_i phi_j d_k phi_q
  F T[KMAX][KMAX][KMAX];       // T[n][i][j] = int phi_n phi_i phi_j
  F M[KMAX][KMAX];             // int phi_q phi_i (identity up to rounding)
  F grad1[3][2];               // grad phihat_q for q < 3 (constant)
  F phi0;                      // phihat_1 = sqrt 2
  F Lv[3][3];                  // int lambda_v phihat_i, i < 3
  F es[9][8], ew[9][8];        // Gauss-Legendre rules on [0,1], 1..8 points
  F EB[9][3][KMAX][8];         // EB[n][k][i][g] = phihat_i(gamma_k(s_g)) with the n-point rule
  F GL[9][8][5];               // GL[n][g][l] = P_l(2 s_g - 1), l < 5
  F EL[3][KMAX][5];            // phihat_i(gamma_k(s)) = sum_l EL[k][i][l] P_l(2 s - 1)
};
using RefTables = RefTablesOf<double>;

const RefTables& tables();

}  // namespace swedg
