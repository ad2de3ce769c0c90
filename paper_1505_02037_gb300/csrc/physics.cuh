// Pointwise Bona-Masso right-hand sides at zero shift in vacuum
// (Ilseven & Mendoza, arXiv:1505.02037, Sec. "Bona-Masso evolution
// equations"; Eq. alfan for the lapse, the three-metric equation, the
// extrinsic-curvature flux lambda^k_ij and source S_ij, and Eq. Vsor for
// Omega_k).
//
// Symmetric tensors are held as their 6 independent components
// (xx, xy, xz, yy, yz, zz); D_kij as D[k][6]. All loops are unrolled so
// every index is a compile-time constant and every array lives in registers.
//
// Index placement: raised indices use the inverse three-metric g^{ij};
// D_kr^r = g^{rm} D_krm, D^r_rk = g^{rm} D_mrk, D_k^{rs} = g^{ra} g^{sb} D_kab,
// D^k_ij = g^{km} D_mij. The second term of the gamma_ij/4 bracket of S_ij is
// taken as D_kr^r D^{ks}_s: with that placement the K equation equals the ADM
// evolution minus (alpha/4) gamma_ij times the Hamiltonian constraint, as the
// paper's "Einstein evolution system" requires.
#pragma once

namespace lbnr {

// Index of the stored component (i, j) of a symmetric tensor. Not recursive,
// so that every use with constant arguments folds to an immediate and the
// arrays it indexes stay in registers.
__host__ __device__ constexpr int sym(int i, int j) {
  return (i < j ? i : j) == 0 ? (i < j ? j : i) : ((i < j ? i : j) == 1 ? 2 + (i < j ? j : i) : 5);
}

// Inverse of a symmetric 3 x 3 matrix; inv: the inverse of its determinant.
template <class T>
__device__ __forceinline__ void invert_sym3(const T g[6], T gi[6], T& inv) {
  const T c00 = g[3] * g[5] - g[4] * g[4];
  const T c01 = g[2] * g[4] - g[1] * g[5];
  const T c02 = g[1] * g[4] - g[2] * g[3];
  const T det = g[0] * c00 + g[1] * c01 + g[2] * c02;
  inv = T(1) / det;
  gi[0] = c00 * inv;
  gi[1] = c01 * inv;
  gi[2] = c02 * inv;
  gi[3] = (g[0] * g[5] - g[2] * g[2]) * inv;
  gi[4] = (g[1] * g[2] - g[0] * g[4]) * inv;
  gi[5] = (g[0] * g[3] - g[1] * g[1]) * inv;
}
template <class T>
__device__ __forceinline__ void invert_sym3(const T g[6], T gi[6]) {
  T inv;
  invert_sym3(g, gi, inv);
}

// The 16 field values in storage order: alpha, gamma(6), K(6), V(3).
enum : int { kAlpha = 0, kG = 1, kK = 7, kV = 13, kNF = 16 };

// The sources as printed, through the Christoffel symbols and over all three
// axes: the FP32 form of the 1D and 2D sets. Those runs take hundreds to
// thousands of steps at 1000 to 4096 cells a side and amplify their FP32
// rounding to 1e-5 and more of the result; another order of these sums moved
// a 4096-cell run by 3.3e-5 in 1200 steps and a 1000^2 run by 1.1e-5 in 200.
// They are bound by memory (1000^2 D2Q9: 173 us a collide, 174 us for its
// bytes at the copy rate), so the shorter form below has nothing to give.
template <class T>
__device__ __forceinline__ void bm_sources_plain(const T alpha, const T g[6], const T K[6],
                                                 const T V[3], const T A[3], const T D[3][6],
                                                 int slicing, T S[kNF], T fluidP) {
  T gi[6];
  invert_sym3(g, gi);

  // K^i_j = g^{im} K_mj (not symmetric in general)
  T Km[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      Km[i][j] = gi[sym(i, 0)] * K[sym(0, j)] + gi[sym(i, 1)] * K[sym(1, j)] +
                 gi[sym(i, 2)] * K[sym(2, j)];
  const T trK = Km[0][0] + Km[1][1] + Km[2][2];
  T trK2 = T(0);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) trK2 += Km[i][j] * Km[j][i];

  // D_ki^r = D_kim g^{mr}
  T Dl[3][3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int r = 0; r < 3; ++r)
        Dl[k][i][r] = D[k][sym(i, 0)] * gi[sym(0, r)] + D[k][sym(i, 1)] * gi[sym(1, r)] +
                      D[k][sym(i, 2)] * gi[sym(2, r)];
  // traces: D_kr^r and D^r_rk
  T tr1[3], tr2[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    tr1[k] = Dl[k][0][0] + Dl[k][1][1] + Dl[k][2][2];
    tr2[k] = Dl[0][k][0] + Dl[1][k][1] + Dl[2][k][2];
  }
  // raised vectors
  T Au[3], Vu[3], tr1u[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    Au[k] = gi[sym(k, 0)] * A[0] + gi[sym(k, 1)] * A[1] + gi[sym(k, 2)] * A[2];
    Vu[k] = gi[sym(k, 0)] * V[0] + gi[sym(k, 1)] * V[1] + gi[sym(k, 2)] * V[2];
    tr1u[k] = gi[sym(k, 0)] * tr1[0] + gi[sym(k, 1)] * tr1[1] + gi[sym(k, 2)] * tr1[2];
  }
  // D^k_ij = g^{km} D_mij (symmetric in ij)
  T Du[3][6];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int q = 0; q < 6; ++q)
      Du[k][q] = gi[sym(k, 0)] * D[0][q] + gi[sym(k, 1)] * D[1][q] + gi[sym(k, 2)] * D[2][q];
  // Christoffel symbols Gamma^k_ij = D_ij^k + D_ji^k - D^k_ij
  T Gam[3][6];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) Gam[k][sym(i, j)] = Dl[i][j][k] + Dl[j][i][k] - Du[k][sym(i, j)];
  // Gamma^k_kr
  T Gc[3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
    Gc[r] = Gam[0][sym(0, r)] + Gam[1][sym(1, r)] + Gam[2][sym(2, r)];
  // D_k^{kr} = g^{ka} D_ka^r
  T Dkk[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    T t = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int a = 0; a < 3; ++a) t += gi[sym(k, a)] * Dl[k][a][r];
    Dkk[r] = t;
  }
  // D_k^{rs} Gamma^k_rs, with D_k^{rs} = g^{ra} D_ka^s
  T DG = T(0);
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const T Duu = gi[sym(r, 0)] * Dl[k][0][s] + gi[sym(r, 1)] * Dl[k][1][s] +
                      gi[sym(r, 2)] * Dl[k][2][s];
        DG += Duu * Gam[k][sym(r, s)];
      }
  const T bracket = -DG + (tr1[0] * tr1u[0] + tr1[1] * tr1u[1] + tr1[2] * tr1u[2]) -
                    T(2) * (Vu[0] * A[0] + Vu[1] * A[1] + Vu[2] * A[2]) + trK2 - trK * trK;

  // S_ij
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const int q = sym(i, j);
      // -2 K_ik K^k_j + trK K_ij
      T t = -T(2) * (K[sym(i, 0)] * Km[0][j] + K[sym(i, 1)] * Km[1][j] + K[sym(i, 2)] * Km[2][j]) +
            trK * K[q];
      // 2 D_ik^r D_rj^k + 2 D_jk^r D_ri^k ; Gamma^k_kr Gamma^r_ij - Gamma^k_ri Gamma^r_kj
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int r = 0; r < 3; ++r)
          t += T(2) * (Dl[i][k][r] * Dl[r][j][k] + Dl[j][k][r] * Dl[r][i][k]) -
               Gam[k][sym(r, i)] * Gam[r][sym(k, j)];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        t += Gc[r] * Gam[r][q];
        // -(2 D_k^{kr} - A^r)(D_ijr + D_jir)
        t -= (T(2) * Dkk[r] - Au[r]) * (D[i][sym(j, r)] + D[j][sym(i, r)]);
        // - V^k D_kij
        t -= Vu[r] * D[r][q];
      }
      // A_i (V_j - D_jk^k / 2) + A_j (V_i - D_ik^k / 2)
      t += A[i] * (V[j] - T(0.5) * tr1[j]) + A[j] * (V[i] - T(0.5) * tr1[i]);
      t += T(0.25) * g[q] * bracket;
      t += T(0.5) * fluidP * g[q];
      S[kK + q] = alpha * t;
    }

  // Omega_k (Eq. Vsor at zero shift, vacuum)
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T t = A[0] * Km[0][k] + A[1] * Km[1][k] + A[2] * Km[2][k] - trK * A[k];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
#pragma unroll
      for (int s = 0; s < 3; ++s) t += (Dl[k][r][s] - T(2) * Dl[r][k][s]) * Km[r][s];
      t -= Km[r][k] * (tr1[r] - T(2) * tr2[r]);
    }
    S[kV + k] = alpha * t;
  }

  // Lapse (Eq. alfan, beta = 0) and metric (beta = 0, s_ij = 0)
  const T Qg = slicing == 1 ? trK : (slicing == 2 ? trK / alpha : T(0));
  S[kAlpha] = -alpha * alpha * Qg;
#pragma unroll
  for (int q = 0; q < 6; ++q) S[kG + q] = -T(2) * alpha * K[q];
}

// Sources S_F of all 16 fields (d_t of each field less its flux divergence)
// at the state (alpha, gamma, K, V) with derivatives A_k, D_kij.
//
// Matter (Sec. "Expansion of flat universe"): a perfect fluid at rest in the
// slice frame, with energy density rho = alpha^2 G^00 and pressure P:
// G_ij = P gamma_ij, tr G = 3P, G^0_k = 0. S_ij gains -R^(4)_ij +
// (gamma_ij / 4) 2 alpha^2 G^00 with R^(4)_ij = G_ij - (gamma_ij / 2)
// (-alpha^2 G^00 + tr G) = (rho - P) gamma_ij / 2, so the sum is
// (P / 2) gamma_ij and rho drops out; Omega_k gains alpha^2 G^0_k = 0.
// fluidP = 0 is vacuum.
//
// dim: the axes k along which A_k and D_kij can differ from zero (the axes the
// velocity set spans); terms with another A_k or D_kij are not formed.
//
// The Christoffel symbols of the printed S_ij are never formed either. With
// D_ki^r = D_kim g^{mr} (Dl below), tr1_k = D_kr^r and tr2_k = D^r_rk:
//   Gamma^k_kr = tr1_r and D_k^{kr} = g^{rm} tr2_m, so with
//     Z_rij = D_ijr + D_jir the terms linear in D_ij are
//     g^{rm}(tr1 - 2 tr2 + A)_m Z_rij - g^{rm}(tr1 + V)_m D_rij;
//   Gamma^k_ri Gamma^r_kj = N_ij + X_ij with N_ij = D_ir^k D_jk^r: lowered,
//     Gamma_mri = D_irm + (D_rim - D_mir), symmetric plus antisymmetric in
//     (r, m), and the mixed products vanish. The antisymmetric part is a
//     vector, D_rim - D_mir = eps_rmn x_i^n, so X_ij = -2 det(g^-1) g_np
//     x_i^n x_j^p;
//   D_k^{rs} Gamma^k_rs = g^{ij}(M_ij + M_ji - N_ij), M_ij = D_ik^r D_rj^k.
// In 3D that is 574 multiplications where the printed sums take 742, in 2D 426,
// in 1D 277. FP64 is bound by its operations (a warp's FP64 instruction holds
// its scheduler for 64 cycles, whatever the active lanes): with 200 cells of
// D1Q3 a step takes 28 us instead of 42, 64^3 with the monitor 50.3 ms instead
// of 55.4 for 40 steps. 16-bit storage waits on the latency of its instructions
// (41 % of the issue slots used), so fewer in a row help there too: 256^3
// D3Q19 FP16, 100 steps 653 instead of 697 ms, host copies included.
template <class T, int dim>
__device__ __forceinline__ void bm_sources(const T alpha, const T g[6], const T K[6],
                                           const T V[3], const T A[3], const T D[3][6],
                                           int slicing, T S[kNF], T fluidP = T(0)) {
  static_assert(dim >= 1 && dim <= 3, "one to three axes");
  if constexpr (sizeof(T) == 4 && dim <= 2) {
    bm_sources_plain<T>(alpha, g, K, V, A, D, slicing, S, fluidP);
    return;
  }
  T gi[6], idet;
  invert_sym3(g, gi, idet);

  // K^i_j = g^{im} K_mj (not symmetric in general)
  T Km[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      Km[i][j] = gi[sym(i, 0)] * K[sym(0, j)] + gi[sym(i, 1)] * K[sym(1, j)] +
                 gi[sym(i, 2)] * K[sym(2, j)];
  const T trK = Km[0][0] + Km[1][1] + Km[2][2];
  const T trK2 = Km[0][0] * Km[0][0] + Km[1][1] * Km[1][1] + Km[2][2] * Km[2][2] +
                 T(2) * (Km[0][1] * Km[1][0] + Km[0][2] * Km[2][0] + Km[1][2] * Km[2][1]);

  // D_ki^r = D_kim g^{mr}, k < dim
  T Dl[dim][3][3];
#pragma unroll
  for (int k = 0; k < dim; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int r = 0; r < 3; ++r)
        Dl[k][i][r] = D[k][sym(i, 0)] * gi[sym(0, r)] + D[k][sym(i, 1)] * gi[sym(1, r)] +
                      D[k][sym(i, 2)] * gi[sym(2, r)];
  // traces: tr1_k = D_kr^r (k < dim) and tr2_k = D^r_rk
  T tr1[dim], tr2[3];
#pragma unroll
  for (int k = 0; k < dim; ++k) tr1[k] = Dl[k][0][0] + Dl[k][1][1] + Dl[k][2][2];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    tr2[k] = Dl[0][k][0];
#pragma unroll
    for (int r = 1; r < dim; ++r) tr2[k] += Dl[r][k][r];
  }
  // Omega_k (Eq. Vsor at zero shift, vacuum):
  // (A_r - tr1_r + 2 tr2_r) K^r_k - trK A_k + (D_kr^s - 2 D_rk^s) K^r_s
  {
    T v[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) v[r] = T(2) * tr2[r] + (r < dim ? A[r] - tr1[r] : T(0));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      T t = v[0] * Km[0][k] + v[1] * Km[1][k] + v[2] * Km[2][k], u = T(0);
      if (k < dim) t -= trK * A[k];
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          if (k < dim) t += Dl[k][r][s] * Km[r][s];
          if (r < dim) u += Dl[r][k][s] * Km[r][s];
        }
      S[kV + k] = alpha * (t - T(2) * u);
    }
  }

  // E^r = g^{rm} (tr1 - 2 tr2 + A)_m, H^r = g^{rm} (tr1 + V)_m (r < dim)
  T Eu[3], Hu[dim];
  T bracket = trK2 - trK * trK;
  {
    T e[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) e[k] = (k < dim ? A[k] + tr1[k] : T(0)) - T(2) * tr2[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      Eu[k] = gi[sym(k, 0)] * e[0] + gi[sym(k, 1)] * e[1] + gi[sym(k, 2)] * e[2];
      if (k < dim) {
        T t1u = gi[sym(k, 0)] * tr1[0];
#pragma unroll
        for (int m = 1; m < dim; ++m) t1u += gi[sym(k, m)] * tr1[m];
        const T Vu = gi[sym(k, 0)] * V[0] + gi[sym(k, 1)] * V[1] + gi[sym(k, 2)] * V[2];
        Hu[k] = t1u + Vu;
        bracket += tr1[k] * t1u - T(2) * Vu * A[k];
      }
    }
  }
  // dual vectors of D_rim - D_mir, and lowered: y_i = -2 det(g^-1) g x_i.
  // In 1D only D_0im is there, so x_i^0 = 0; n0 is the first live component.
  constexpr int n0 = dim == 1 ? 1 : 0;
  T x[3][3], y[3][3];
  const T m2 = -T(2) * idet;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (dim == 3) x[i][0] = D[1][sym(i, 2)] - D[dim - 1][sym(i, 1)];
    if (dim == 2) x[i][0] = D[dim - 1][sym(i, 2)];
    x[i][1] = dim == 3 ? D[dim - 1][sym(i, 0)] - D[0][sym(i, 2)] : -D[0][sym(i, 2)];
    x[i][2] = dim >= 2 ? D[0][sym(i, 1)] - D[dim >= 2 ? 1 : 0][sym(i, 0)] : D[0][sym(i, 1)];
#pragma unroll
    for (int n = n0; n < 3; ++n) {
      T t = g[sym(n, n0)] * x[i][n0];
#pragma unroll
      for (int p = n0 + 1; p < 3; ++p) t += g[sym(n, p)] * x[i][p];
      y[i][n] = m2 * t;
    }
  }
  T h[3];  // V_i - D_ir^r / 2
#pragma unroll
  for (int i = 0; i < 3; ++i) h[i] = i < dim ? V[i] - T(0.5) * tr1[i < dim ? i : 0] : V[i];

  // S_ij less the gamma_ij / 4 bracket, whose sum over M and N is taken along
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const int q = sym(i, j);
      // -2 K_ik K^k_j + trK K_ij
      T t = -T(2) * (K[sym(i, 0)] * Km[0][j] + K[sym(i, 1)] * Km[1][j] + K[sym(i, 2)] * Km[2][j]) +
            trK * K[q];
      // M_ij + M_ji and N_ij (i <= j, so i < dim whenever j < dim)
      if (i < dim) {
        T ms = T(0), nn = T(0);
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            if (r < dim) ms += Dl[i < dim ? i : 0][k][r] * Dl[r < dim ? r : 0][j][k];
            if (r < dim && i != j && j < dim)
              ms += Dl[j < dim ? j : 0][k][r] * Dl[r < dim ? r : 0][i][k];
            if (j < dim) nn += Dl[i < dim ? i : 0][k][r] * Dl[j < dim ? j : 0][r][k];
          }
        if (i == j) ms = ms + ms;
        bracket -= (i == j ? gi[q] : T(2) * gi[q]) * (ms - nn);
        t += T(2) * ms - nn;
      }
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        if (r >= n0) t -= x[i][r] * y[j][r];
        if (i == j && i < dim)
          t += T(2) * Eu[r] * D[i][sym(i, r)];
        else if (j < dim)
          t += Eu[r] * (D[i][sym(j, r)] + D[j][sym(i, r)]);
        else if (i < dim)
          t += Eu[r] * D[i][sym(j, r)];
        if (r < dim) t -= Hu[r < dim ? r : 0] * D[r][q];
      }
      // A_i (V_j - D_jk^k / 2) + A_j (V_i - D_ik^k / 2)
      if (i == j && i < dim)
        t += T(2) * A[i] * h[i];
      else if (i < dim)
        t += A[i] * h[j];
      if (i != j && j < dim) t += A[j] * h[i];
      S[kK + q] = t;
    }
  const T quarter = T(0.25) * bracket + T(0.5) * fluidP;
#pragma unroll
  for (int q = 0; q < 6; ++q) S[kK + q] = alpha * (S[kK + q] + quarter * g[q]);

  // Lapse (Eq. alfan, beta = 0) and metric (beta = 0, s_ij = 0)
  const T Qg = slicing == 1 ? trK : (slicing == 2 ? trK / alpha : T(0));
  S[kAlpha] = -alpha * alpha * Qg;
#pragma unroll
  for (int q = 0; q < 6; ++q) S[kG + q] = -T(2) * alpha * K[q];
}

template <class T, int dim>
__device__ __forceinline__ void bm_flux_plain(const T alpha, const T g[6], const T V[3], const T A[3],
                                              const T D[3][6], T F[6][3]) {
  T gi[6];
  invert_sym3(g, gi);
  T tr1[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    tr1[k] = gi[0] * D[k][0] + gi[3] * D[k][3] + gi[5] * D[k][5] +
             T(2) * (gi[1] * D[k][1] + gi[2] * D[k][2] + gi[4] * D[k][4]);
  T e[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) e[i] = T(0.5) * (A[i] + T(2) * V[i] - tr1[i]);
#pragma unroll
  for (int k = 0; k < dim; ++k) {
    const T Vu = gi[sym(k, 0)] * V[0] + gi[sym(k, 1)] * V[1] + gi[sym(k, 2)] * V[2];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        const int q = sym(i, j);
        T l = gi[sym(k, 0)] * D[0][q] + gi[sym(k, 1)] * D[1][q] + gi[sym(k, 2)] * D[2][q] -
              T(0.5) * Vu * g[q];
        if (k == i) l += e[j];
        if (k == j) l += e[i];
        F[q][k] = alpha * l;
      }
  }
#pragma unroll
  for (int k = dim; k < 3; ++k)
#pragma unroll
    for (int q = 0; q < 6; ++q) F[q][k] = T(0);
}

// Flux of K_ij along axis k times a factor: al lambda^k_ij, with al = alpha
// (times what the caller scales its fluxes by) and
// lambda^k_ij = D^k_ij + 1/2 delta^k_i (A_j + 2 V_j - D_jr^r)
//             + 1/2 delta^k_j (A_i + 2 V_i - D_ir^r) - 1/2 V^k gamma_ij.
// al multiplies the six g^{ij} and the three brackets instead of the 18
// results (not in the FP32 form of 1D and 2D, see bm_sources_plain). Only the
// first `dim` axes are formed (the lattice has no other velocities); ddim: the
// axes along which A_k and D_kij can differ from zero.
template <class T, int dim, int ddim = dim>
__device__ __forceinline__ void bm_flux(const T al, const T g[6], const T V[3], const T A[3],
                                        const T D[3][6], T F[6][3]) {
  if constexpr (sizeof(T) == 4 && ddim <= 2) {
    bm_flux_plain<T, dim>(al, g, V, A, D, F);
    return;
  }
  T gi[6];
  invert_sym3(g, gi);
  const T ah = T(0.5) * al;
  T e[3], ga[6];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    T t = T(2) * V[i];
    if (i < ddim) {
      const T tr1 = gi[0] * D[i][0] + gi[3] * D[i][3] + gi[5] * D[i][5] +
                    T(2) * (gi[1] * D[i][1] + gi[2] * D[i][2] + gi[4] * D[i][4]);
      t += A[i] - tr1;
    }
    e[i] = ah * t;
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) ga[q] = al * gi[q];
#pragma unroll
  for (int k = 0; k < dim; ++k) {
    const T Vh = T(0.5) * (ga[sym(k, 0)] * V[0] + ga[sym(k, 1)] * V[1] + ga[sym(k, 2)] * V[2]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        const int q = sym(i, j);
        T l = ga[sym(k, 0)] * D[0][q] - Vh * g[q];
#pragma unroll
        for (int m = 1; m < ddim; ++m) l += ga[sym(k, m)] * D[m][q];
        if (k == i) l += e[j];
        if (k == j) l += e[i];
        F[q][k] = l;
      }
  }
#pragma unroll
  for (int k = dim; k < 3; ++k)
#pragma unroll
    for (int q = 0; q < 6; ++q) F[q][k] = T(0);
}

// Shift-field terms (Sec. "Bona-Masso evolution equations"; B_k^i =
// d_k beta^i / 2, B[k][i]): added to the sources S (metric, K_ij: alpha S_ij,
// V: Omega_k) at the point, with B_ij = B_i^m gamma_mj, B^r_s = g^{rl} B_ls.
//   gamma_ij: 2 (B_ij + B_ji)
//   K_ij:     2 (K_ir B_j^r + K_jr B_i^r - K_ij tr B)
//   V_k:      2 (B_k^r - delta_k^r tr B) V_r + 2 (D_rk^s - delta^s_k D^j_jr) B^r_s
template <class T>
__device__ __forceinline__ void shift_field_sources(const T g[6], const T K[6], const T V[3],
                                                    const T D[3][6], const T B[3][3],
                                                    T S[16]) {
  T gi[6];
  invert_sym3(g, gi);
  T Bl[3][3], Bul[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      Bl[i][j] = B[i][0] * g[sym(0, j)] + B[i][1] * g[sym(1, j)] + B[i][2] * g[sym(2, j)];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      Bul[i][j] = gi[sym(i, 0)] * Bl[0][j] + gi[sym(i, 1)] * Bl[1][j] + gi[sym(i, 2)] * Bl[2][j];
  const T trB = B[0][0] + B[1][1] + B[2][2];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const int q = sym(i, j);
      S[1 + q] += T(2) * (Bl[i][j] + Bl[j][i]);
      T t = -K[q] * trB;
#pragma unroll
      for (int r = 0; r < 3; ++r) t += K[sym(i, r)] * B[j][r] + K[sym(j, r)] * B[i][r];
      S[7 + q] += T(2) * t;
    }
  // D^j_jr = g^{ja} D_jar
  T Dt2[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    T t = T(0);
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int a = 0; a < 3; ++a) t += gi[sym(j, a)] * D[j][sym(a, r)];
    Dt2[r] = t;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T t = T(0);
#pragma unroll
    for (int r = 0; r < 3; ++r) t += (B[k][r] - (k == r ? trB : T(0))) * V[r];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
#pragma unroll
      for (int s2 = 0; s2 < 3; ++s2) {
        // D_rk^s = g^{sm} D_rkm
        const T Drks = gi[sym(s2, 0)] * D[r][sym(k, 0)] + gi[sym(s2, 1)] * D[r][sym(k, 1)] +
                       gi[sym(s2, 2)] * D[r][sym(k, 2)];
        t += (Drks - (s2 == k ? Dt2[r] : T(0))) * Bul[r][s2];
      }
    }
    S[13 + k] += T(2) * t;
  }
}

// Flux of V_i along k under a shift field: -beta^k V_i + B^k_i - B_i^k
// (the V equation's flux; B^k_i = g^{kl} B_l^m gamma_mi).
template <class T, int dim>
__device__ __forceinline__ void shift_field_vflux(const T g[6], const T V[3], const T beta[3],
                                                  const T B[3][3], T Fv[3][3]) {
  T gi[6];
  invert_sym3(g, gi);
  T Bl[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      Bl[i][j] = B[i][0] * g[sym(0, j)] + B[i][1] * g[sym(1, j)] + B[i][2] * g[sym(2, j)];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (k < dim) {
        const T Bki = gi[sym(k, 0)] * Bl[0][i] + gi[sym(k, 1)] * Bl[1][i] + gi[sym(k, 2)] * Bl[2][i];
        Fv[i][k] = -beta[k] * V[i] + Bki - B[i][k];
      } else {
        Fv[i][k] = T(0);
      }
    }
}

}  // namespace lbnr
