// The FP64 step with sixteen or eight lanes to a cell, for small lattices.
//
// On GB300 a warp's FP64 instruction holds its scheduler for 64 cycles however
// many of its lanes are active, and a lattice of a few thousand cells leaves
// most of the 608 schedulers idle: with a thread per cell, 200 cells of D1Q3
// are 7 warps that each run their 700-odd FP64 instructions one after the
// other (28 us a step with the shorter sources of physics.cuh). Here 16 or
// 8 lanes share a cell: each owns one or two of the 16 fields for the sums, the
// relaxation and the streaming, and the tensor algebra between them is laid
// out as rounds of equal tasks (a component each), with every intermediate
// in shared memory. About 180 (1D) to 330 (3D) instructions follow one another
// instead. The same sums and formulas as collide_body (bm_sources and bm_flux
// of physics.cuh), rounded in another order.
//
// The stencil's neighbours are summed by the cell that needs them, so one
// launch does the whole SYNC step; that reads neighbours' distributions, which
// only ping-pong buffers allow. Under LAG the planes are read as everywhere.
//
// Bound by the chain of rounds (about 16 of them, a few FP64 instructions each)
// and, as the lattice grows, by the FP64 pipe, which the half-empty rounds use
// less well than a thread per cell does. 200 cells D1Q3: 11.3 us a step, launch
// included, against 25.6 (42.0 before the shorter sources); 800 x 4 D2Q9 23.4
// against 45.
#pragma once

#include "kernels.cuh"

namespace lbnr {

// The form (lanes per cell) a context starts with, by the lattice's cells: 16
// while the schedulers have a warp each at most, 8 while they have a few, then
// a thread per cell (0). us a step with 16 lanes, 8 lanes, a thread: D1Q3 1000
// cells 11.3, 12.3, 25.6; 2500 19.4, 14.4, 25.6; 6000 36.9, 24.6, 25.6. D2Q9 32^2
// 14.3, 17.4, 45.1; 70^2 41.0, 31.8, 46.1; 90^2 61.4, 45.2, 46.1. D3Q19 8^3 17.4,
// 22.6, 69.7; 12^3 22.6, 24.6, 71.7; 16^3 47.1, 34.8, 71.7; 20^3 87.1, 77.3, 71.7.
// LAG crosses at much the same sizes: D1Q3 1500 12.3, 12.3, 21.5; 5500 34.8, 23.6,
// 22.5; D2Q9 41^2 15.4, 15.4, 40.0; 89^2 56.4, 40.0, 40.0; D3Q19 2000 cells 21.5,
// 19.5, 62.5; 19^3 65.3, 44.5, 62.5.
template <int Q>
constexpr int lanes_for(int64_t cells) {
  return cells <= (Q == 3 ? 1500 : Q == 9 ? 1700 : 2000) ? 16
         : cells <= (Q == 3 ? 5500 : Q == 9 ? 8000 : 7000) ? 8 : 0;
}

// One cell's intermediates.
struct LaneCell {
  double rt[kNF], rho[kNF], S[kNF];
  double nb[6][7];           // moments of alpha, gamma at the neighbours (k, +-)
  double A[3], D[3][6];      // zero beyond the set's axes
  double gi[6], cof[6];      // inverse metric and its cofactors
  double m[36];              // K^i_j, then D_ki^r at 9 + 9 k + 3 i + r
  double tr[4];              // tr K, then D_kr^r
  double tr2[3];             // D^r_rk
  double v[3], e[3], h[3];   // A - tr1 + 2 tr2, A + tr1 - 2 tr2, V - tr1 / 2
  double Eu[3], t1u[3], Vu[3];
  double x[3][3], y[3][3];
  double dot[24];            // M_ij (9), N_ij (6), u_k (3), w_k (3), K^i_j K^j_i
  double sk[6], mn[6];       // S_ij less its bracket, g^{ij} (M_ij + M_ji - N_ij)
  double ga[6], fe[3], Vh[3], F[6][3];
};

// Stored component (i, j) of a symmetric tensor, indices known at run time.
__device__ __forceinline__ int sym_rt(int i, int j) {
  const int lo = min(i, j), hi = max(i, j);
  return ((lo * (5 - lo)) >> 1) + hi;
}
// Row and column of pair q.
__device__ __forceinline__ int pair_row(int q) { return q < 3 ? 0 : q < 5 ? 1 : 2; }
__device__ __forceinline__ int pair_col(int q) { return q < 3 ? q : q < 5 ? q - 2 : 2; }
__device__ __forceinline__ int nibble(uint32_t w, int i) { return (w >> (4 * i)) & 15; }

// gi = inverse of the symmetric g by the lanes of a cell; returns 1 / det g.
__device__ __forceinline__ double lane_inverse(const double* g, double* cof, double* gi, int t) {
  if (t < 6) {
    // cofactors g_a g_b - g_c g_d in the order of invert_sym3
    const int a = nibble(0x010123u, t), b = nibble(0x325445u, t);
    const int c = nibble(0x102214u, t), d = nibble(0x142354u, t);
    cof[t] = g[a] * g[b] - g[c] * g[d];
  }
  __syncwarp();
  const double inv = 1.0 / (g[0] * cof[0] + g[1] * cof[1] + g[2] * cof[2]);
  if (t < 6) gi[t] = cof[t] * inv;
  __syncwarp();
  return inv;
}

// Task o of N for each lane of a cell, in rounds of G.
#define LBNR_TASKS(o, N) _Pragma("unroll") for (int r_ = 0; r_ < ((N) + G - 1) / G; ++r_) if (const int o = r_ * G + t; o < (N))
template <int Q, int G, bool LAGW>
__global__ void __launch_bounds__(32) k_lanes(const StepArgs<double, double> a) {
  using L = Lattice<Q>;
  constexpr int dim = L::kDim;
  constexpr int NL = kNF / G;  // fields per lane: t, t + G, ...
  __shared__ LaneCell shared[32 / G];
  const int t = threadIdx.x & (G - 1);
  LaneCell& s = shared[threadIdx.x / G];
  const int64_t cells = a.G.cells;
  const int64_t cell = (int64_t)blockIdx.x * (32 / G) + threadIdx.x / G;
  const bool valid = cell < cells;
  const Nbr n = make_nbr(a.G, valid ? cell : cells - 1);
  const uint32_t pc[3] = {n.at(1, 0, 0), n.at(0, 1, 0), n.at(0, 0, 1)};
  const uint32_t mc[3] = {n.at(-1, 0, 0), n.at(0, -1, 0), n.at(0, 0, -1)};

  // this lane's fields, and the neighbours' lapse and metric
  double f[NL][Q];
#pragma unroll
  for (int j = 0; j < NL; ++j)
#pragma unroll
    for (int l = 0; l < Q; ++l) f[j][l] = __ldg(a.fin + fidx<Q, double>(n.c, t + j * G, l));
  if (!LAGW) {
    LBNR_TASKS(i, 14 * dim) {
      const int side = i / 7, p = i - 7 * side;
      {
        const int k = side >> 1;
        const uint32_t c = (side & 1) ? (k == 0 ? mc[0] : k == 1 ? mc[1] : mc[2])
                                      : (k == 0 ? pc[0] : k == 1 ? pc[1] : pc[2]);
        double w[Q], sum = 0;
#pragma unroll
        for (int l = 0; l < Q; ++l) w[l] = __ldg(a.fin + fidx<Q, double>(c, p, l));
#pragma unroll
        for (int l = 0; l < Q; ++l) sum += w[l];
        s.nb[side][p] = sum;
      }
    }
  } else {
    LBNR_TASKS(i, 14 * dim) {
      const int side = i / 7, p = i - 7 * side;
      {
        const int k = side >> 1;
        const uint32_t c = (side & 1) ? (k == 0 ? mc[0] : k == 1 ? mc[1] : mc[2])
                                      : (k == 0 ? pc[0] : k == 1 ? pc[1] : pc[2]);
        s.nb[side][p] = __ldg(a.aux + (size_t)p * (size_t)cells + c);
      }
    }
  }
  double sum[NL];
  bool bad = false;
#pragma unroll
  for (int j = 0; j < NL; ++j) {
    sum[j] = 0;
#pragma unroll
    for (int l = 0; l < Q; ++l) sum[j] += f[j][l];
    s.rt[t + j * G] = sum[j];
    bad |= valid && !isfinite(sum[j]);
  }
  __syncwarp();
  if (!LAGW) {
    if (t < 2 * dim) s.nb[t][0] = log(s.nb[t][0]);
    __syncwarp();
  }
  // A_k and D_kij
  LBNR_TASKS(i, 21) {
    const int k = i / 7, p = i - 7 * k;
    double d = 0;
    if (k < dim) d = (s.nb[2 * k][p] - s.nb[2 * k + 1][p]) * (p == 0 ? a.inv2dx : a.inv4dx);
    if (p == 0)
      s.A[k] = d;
    else
      s.D[k][p - 1] = d;
  }
  __syncwarp();

  // ---- sources at rho~ ----
  const double* g = s.rt + kG;
  const double* K = s.rt + kK;
  const double* V = s.rt + kV;
  const double alpha = s.rt[0];
  const double m2 = -2.0 * lane_inverse(g, s.cof, s.gi, t);
  // K^i_j = g^{im} K_mj and D_ki^r = D_kim g^{mr}
  LBNR_TASKS(o, 9 + 9 * dim) {
    {
      const int mat = o / 9, e = o - 9 * mat, i = e / 3, j = e - 3 * i;
      const double* p = mat == 0 ? s.gi : s.D[mat - 1];
      const double* q = mat == 0 ? K : s.gi;
      s.m[o] = p[sym_rt(i, 0)] * q[sym_rt(0, j)] + p[sym_rt(i, 1)] * q[sym_rt(1, j)] +
               p[sym_rt(i, 2)] * q[sym_rt(2, j)];
    }
  }
  // dual vectors of D_rim - D_mir
  LBNR_TASKS(o, 9) {
    const int i = o / 3, c = o - 3 * i, p = c == 2 ? 0 : c + 1, q = c == 0 ? 2 : c - 1;
    s.x[i][c] = s.D[p][sym_rt(i, q)] - s.D[q][sym_rt(i, p)];
  }
  __syncwarp();
  // traces
  if (t <= 3) {
    const double* p = s.m + 9 * t;
    s.tr[t] = t <= dim ? p[0] + p[4] + p[8] : 0.0;
  } else if (t < 7) {
    const int k = t - 4;
    double d = s.m[9 + 3 * k];
#pragma unroll
    for (int r = 1; r < dim; ++r) d += s.m[9 + 9 * r + 3 * k + r];
    s.tr2[k] = d;
  }
  __syncwarp();
  LBNR_TASKS(w, 9) {
    const int o = w / 3, k = w - 3 * o;
    const double t1 = s.tr[1 + k], t2 = s.tr2[k];
    // v, e: A -+ (tr1 - 2 tr2); h = V - tr1 / 2
    const double base = o == 2 ? V[k] : s.A[k];
    const double c1 = o == 0 ? -1.0 : o == 1 ? 1.0 : -0.5, c2 = o == 0 ? 2.0 : o == 1 ? -2.0 : 0.0;
    (o == 0 ? s.v : o == 1 ? s.e : s.h)[k] = base + c1 * t1 + c2 * t2;
  }
  __syncwarp();
  // raised e, tr1, V; lowered and scaled x
  LBNR_TASKS(o, 18) {
    {
      const int w = o / 3, k = o - 3 * w;
      const double* mat = w < 3 ? s.gi : g;
      const double* vec = w == 0 ? s.e : w == 1 ? s.tr + 1 : w == 2 ? V : s.x[w - 3];
      double* out = w == 0 ? s.Eu : w == 1 ? s.t1u : w == 2 ? s.Vu : s.y[w - 3];
      out[k] = (w < 3 ? 1.0 : m2) * (mat[sym_rt(k, 0)] * vec[0] + mat[sym_rt(k, 1)] * vec[1] +
                                     mat[sym_rt(k, 2)] * vec[2]);
    }
  }
  // sums over two indices of products of K^i_j and D_ki^r:
  // M_ij = D_ik^r D_rj^k (i < dim, r < dim), N_ij = D_ir^k D_jk^r (i <= j < dim),
  // u_k = D_rk^s K^r_s (r < dim), w_k = D_kr^s K^r_s (k < dim), K^i_j K^j_i
  LBNR_TASKS(o, 22) {
    int b1 = 0, s1 = 3, t1 = 1, b2 = 0, s2 = 3, t2 = 1, lim = 3;
    bool live = true;
    if (o < 9) {
      const int i = o / 3, j = o - 3 * i;
      b1 = 9 + 9 * i, s1 = 1, t1 = 3, b2 = 9 + 3 * j, s2 = 9, t2 = 1, lim = dim;
      live = i < dim;
    } else if (o < 15) {
      const int i = pair_row(o - 9), j = pair_col(o - 9);
      b1 = 9 + 9 * i, s1 = 1, t1 = 3, b2 = 9 + 9 * j, s2 = 3, t2 = 1;
      live = j < dim;
    } else if (o < 18) {
      b1 = 9 + 3 * (o - 15), s1 = 9, lim = dim;
    } else if (o < 21) {
      b1 = 9 + 9 * (o - 18);
      live = o - 18 < dim;
    } else {
      s2 = 1, t2 = 3;
    }
    double d = 0;
    if (live) {
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        const int pp = p < lim ? p : 0;
        const double z = p < lim ? 1.0 : 0.0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const double w = p < dim ? s.m[b1 + pp * s1 + q * t1]
                                   : z * s.m[b1 + pp * s1 + q * t1];
          d += w * s.m[b2 + pp * s2 + q * t2];
        }
      }
    }
    s.dot[o] = d;
  }
  __syncwarp();
  const double trK = s.tr[0];
  if (t < 6) {
    const int i = pair_row(t), j = pair_col(t);
    const double ms = s.dot[3 * i + j] + s.dot[3 * j + i], nn = s.dot[9 + t];
    s.mn[t] = (i == j ? s.gi[t] : 2.0 * s.gi[t]) * (ms - nn);
    double d = -2.0 * (K[sym_rt(i, 0)] * s.m[j] + K[sym_rt(i, 1)] * s.m[3 + j] +
                       K[sym_rt(i, 2)] * s.m[6 + j]) +
               trK * K[t];
    d += 2.0 * ms - nn;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      if (dim > 1 || r > 0) d -= s.x[i][r] * s.y[j][r];
      d += s.Eu[r] * (s.D[i][sym_rt(j, r)] + s.D[j][sym_rt(i, r)]);
      if (r < dim) d -= (s.t1u[r] + s.Vu[r]) * s.D[r][t];
    }
    s.sk[t] = d + s.A[i] * s.h[j] + s.A[j] * s.h[i];
  }
  __syncwarp();
  {
    double bracket = s.dot[21] - trK * trK;
#pragma unroll
    for (int k = 0; k < dim; ++k) bracket += s.tr[1 + k] * s.t1u[k] - 2.0 * s.Vu[k] * s.A[k];
#pragma unroll
    for (int q = 0; q < 6; ++q) bracket -= s.mn[q];
    double half_p = 0;
    if (a.clock != nullptr) {
      const double r = a.fluid_t0 / (a.fluid_t0 + (double)(*a.clock) * a.fluid_dt);
      half_p = 0.5 * a.fluid_P0 * r * r;
    }
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const int F = t + j * G;
      double S;
      if (F == 0) {
        const double Qg = a.slicing == 1 ? trK : (a.slicing == 2 ? trK / alpha : 0.0);
        S = -alpha * alpha * Qg;
      } else if (F < kK) {
        S = -2.0 * alpha * s.rt[F + 6];
      } else if (F < kV) {
        S = alpha * (s.sk[F - kK] + (0.25 * bracket + half_p) * g[F - kK]);
      } else {
        const int k = F - kV;
        S = alpha * (s.v[0] * s.m[k] + s.v[1] * s.m[3 + k] + s.v[2] * s.m[6 + k] - trK * s.A[k] +
                     s.dot[18 + k] - 2.0 * s.dot[15 + k]);
      }
      if (!a.sources_on) S = 0;
      s.S[F] = S;
      s.rho[F] = sum[j] + a.half_dt * S;
    }
  }
  __syncwarp();

  // ---- fluxes at rho, times 3 omega and the weight of the last velocity ----
  constexpr double kWb = L::w(Q - 1);
  const double* g2 = s.rho + kG;
  const double* V2 = s.rho + kV;
  lane_inverse(g2, s.cof, s.gi, t);
  const double al = s.rho[0] * (3.0 * a.omega * kWb);
  if (t < 3) {
    const double* D = s.D[t];
    const double tr1 = s.gi[0] * D[0] + s.gi[3] * D[3] + s.gi[5] * D[5] +
                       2.0 * (s.gi[1] * D[1] + s.gi[2] * D[2] + s.gi[4] * D[4]);
    s.fe[t] = 0.5 * al * (s.A[t] + 2.0 * V2[t] - tr1);
  }
  if (t < 6) s.ga[t] = al * s.gi[t];
  __syncwarp();
  if (t < dim)
    s.Vh[t] = 0.5 * (s.ga[sym_rt(t, 0)] * V2[0] + s.ga[sym_rt(t, 1)] * V2[1] + s.ga[sym_rt(t, 2)] * V2[2]);
  __syncwarp();
  LBNR_TASKS(o, 6 * dim) {
    {
      const int k = o / 6, q = o - 6 * k, i = pair_row(q), j = pair_col(q);
      double d = -s.Vh[k] * g2[q];
#pragma unroll
      for (int m = 0; m < dim; ++m) d += s.ga[sym_rt(k, m)] * s.D[m][q];
      d += (k == i ? s.fe[j] : 0.0) + (k == j ? s.fe[i] : 0.0);
      s.F[q][k] = d;
    }
  }
  __syncwarp();

  // ---- relax, add the source, stream ----
#pragma unroll
  for (int j = 0; j < NL; ++j) {
    const int F = t + j * G;
    const double cf = a.omega * sum[j] + (a.half_dt + a.half_dt) * s.S[F];
    double b[3] = {0, 0, 0};
    if (F >= kK && F < kV) {
#pragma unroll
      for (int k = 0; k < dim; ++k) b[k] = s.F[F - kK][k];
    }
#pragma unroll
    for (int l = 0; l < Q; ++l) {
      double d = L::w(l) * cf;
#pragma unroll
      for (int k = 0; k < dim; ++k) {
        const double bk = (L::w(l) / kWb) * b[k];
        if (L::c(l, k) > 0) d += bk;
        if (L::c(l, k) < 0) d -= bk;
      }
      const uint32_t c = n.at(L::c(l, 0), L::c(l, 1), L::c(l, 2));
      if (valid) Codec<double>::store(a.fout + fidx<Q, double>(c, F, l), fma(a.omc, f[j][l], d));
    }
  }
  if (LAGW && valid && t < 7)
    a.aux_out[(size_t)t * (size_t)cells + n.c] = t == 0 ? log(s.rho[0]) : s.rho[t];
  if (bad) atomicOr(a.flag, 1);
}

#undef LBNR_TASKS

}  // namespace lbnr
