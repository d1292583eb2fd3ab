// lb_adjoint.cu -- discrete adjoint of the thermal D3Q19 step (reverse mode, FP64).
//
// Objective: J = (1/N) sum_{n=1..N} Nu_mean(x_n), the time-averaged Nusselt number of Eq. (4),
// x_n the pre-collision state at step n, x_{n+1} = Phi(x_n) the step of Eqs. (6)-(9) with the
// readings of the forward kernels. Gradients: dJ/dT_d, dJ/dT_u, dJ/dG and dJ/dT0 (the initial
// temperature field of lb_init). The adjoint state lambda_n = dJ/dx_n obeys
//   lambda_N = (1/N) dNu/dx_N,  lambda_n = (dPhi/dx_n)^T lambda_{n+1} + [n >= 1] (1/N) dNu/dx_n.
// One reverse step, for state n, in the reverse order of the forward operations:
//   streaming^T (push of lambda_{n+1}, bounce-back transposed, the thermal wall rule's density
//   and T_w terms) -> collision^T (f^eq(rho, u', T), g^eq(rho, T, u), counter term) -> the Nu
//   terms of state n -> divergence^T (radius-1 gather) -> velocities^T (u, u' -> j, F, rho) ->
//   force^T (radius-1 psi gather with the mirrored wall ghosts; dJ/dG) -> moments^T
// in three kernels: coll_adj (up to the Nu terms), vel_adj (divergence^T, velocities^T and the own
// node's part of force^T), force_adj (the gather and the new lambda).
// The forward states are recomputed per segment from checkpoints taken every K steps; the
// macroscopic fields of a state are recomputed per reverse step.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "lb_ctx.h"

namespace tlbm {
namespace adj {

struct Geom {
  int nx, ny, nz, plane, N, nb;   // nb = CTAs per plane
  unsigned div_m, div_s;          // as KArgs::div_m, div_s
};
struct Par {
  double tau, om, omk, G, gz, lam, cv, kappa, Td, Tu;
  double om1, omk1;            // 1 - om, 1 - omk
  double w[3], j3[2], q9[2];   // f: om w per class; 3 om w and 9 om w of the axis and diagonal classes
  double wg[3], j3g[2], q9g[2];  // the same of g
  double Kc;        // 1 / (N_t kappa (T_d - T_u) nx ny): weight of sum_x rho U u_z in J
  double src;       // -1 / (omk c_v)
  int include_nu;   // add (1/N_t) dNu_mean/dx of this state
};

// fields of M (forward macros of one state, MF_* of lb_kernels.cuh), each [N]
// fields of A (adjoints of the macros), each [N]: of coll_adj (first block), of vel_adj (second; RHO
// is updated): dJ/dE, dJ/dj, H = psi dJ/dF and the factor of the gathered sum in dJ/drho
enum { AF_RHO = 0, AF_T, AF_UX, AF_UY, AF_UZ, AF_VX, AF_VY, AF_VZ, AF_D,
       AF_E, AF_JX, AF_JY, AF_JZ, AF_HX, AF_HY, AF_HZ, AF_KP, AF_COUNT };
// per-block parameter partials: wall terms of dJ/dT_d and dJ/dT_u, dJ/dG, the sum of J
enum { P_TD = 0, P_TU, P_G, P_J, P_COUNT };

constexpr int kThreads = 128;     // coll_adj at 64^3: 124 us, 128 with 256

// node of this thread: one CTA covers kThreads consecutive nodes of a plane
struct Node {
  unsigned xs[3], ys[3];   // columns x-1, x, x+1 and rows (y-1) nx, y nx, (y+1) nx, periodic
  unsigned i;              // in-plane index
  int z;
  bool valid;
};
__device__ __forceinline__ Node node_of(const Geom& g) {
  Node n;
  n.z = (int)blockIdx.x / g.nb;
  n.i = (blockIdx.x - (unsigned)(n.z * g.nb)) * kThreads + threadIdx.x;
  n.valid = n.i < (unsigned)g.plane;
  const unsigned nx = (unsigned)g.nx, last = (unsigned)g.plane - nx;
  const unsigned x = n.i - (g.div_m ? (__umulhi(n.i, g.div_m) >> g.div_s) : n.i) * nx, row = n.i - x;
  n.xs[0] = x == 0 ? nx - 1 : x - 1; n.xs[1] = x; n.xs[2] = x + 1 == nx ? 0u : x + 1;
  n.ys[0] = row == 0 ? last : row - nx; n.ys[1] = row; n.ys[2] = row == last ? 0u : row + nx;
  return n;
}
__device__ __forceinline__ void coords(int idx, const Geom& g, int& x, int& y, int& z) {
  x = idx % g.nx;
  y = (idx / g.nx) % g.ny;
  z = idx / g.plane;
}
__device__ __forceinline__ int at(const Geom& g, int x, int y, int z) {
  return z * g.plane + wrapi(y, g.ny) * g.nx + wrapi(x, g.nx);
}

// Sum of v over the CTA on thread 0, in a fixed order: every warp leaves its values in shared memory
// and one adds them, kThreads / 32 per lane and then by shuffles (8 FP64 instructions of one warp
// instead of 5 of every warp). sh is the caller's own array.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = sh[threadIdx.x];
    for (int k = 32; k < kThreads; k += 32) s += sh[threadIdx.x + k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  return s;
}

// rho, j, E, T, psi of state X ([38][N]: f then g, pre-collision, float64)
__global__ void macro_kernel(const double* __restrict__ X, Geom g, double* __restrict__ M) {
  const size_t N = g.N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.N; i += gridDim.x * blockDim.x) {
    double f[Q], E = 0.0;
#pragma unroll
    for (int l = 0; l < Q; ++l) f[l] = X[l * N + i];
#pragma unroll
    for (int l = 0; l < Q; ++l) E += X[(Q + l) * N + i];
    double rho, jx, jy, jz;
    density_momentum<double>(f, rho, jx, jy, jz);
    M[MF_RHO * N + i] = rho; M[MF_JX * N + i] = jx; M[MF_JY * N + i] = jy; M[MF_JZ * N + i] = jz;
    M[MF_E * N + i] = E; M[MF_T * N + i] = E / rho; M[MF_PSI * N + i] = exp(-1.0 / rho);
  }
}

// Eq. (9): A_a = sum_{l>=1} W_l c_la psi(x + c_l) (mirrored ghosts), F = -G psi A + rho g_z z,
// u = (j + F/2)/rho, u' = (j + tau F)/rho
__global__ void force_fwd_kernel(Geom g, Par p, double* __restrict__ M) {
  const size_t N = g.N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.N; i += gridDim.x * blockDim.x) {
    int x, y, z;
    coords(i, g, x, y, z);
    double A[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int l = 1; l < Q; ++l) {
      const double nb = M[MF_PSI * N + at(g, x + CX(l), y + CY(l), mirror_z(z + CZ(l), g.nz))];
      if (CX(l)) A[0] += FW<double>(l) * CX(l) * nb;
      if (CY(l)) A[1] += FW<double>(l) * CY(l) * nb;
      if (CZ(l)) A[2] += FW<double>(l) * CZ(l) * nb;
    }
    const double rho = M[MF_RHO * N + i], psi = M[MF_PSI * N + i];
    const double F[3] = {-p.G * psi * A[0], -p.G * psi * A[1], -p.G * psi * A[2] + rho * p.gz};
    for (int a = 0; a < 3; ++a) {
      const double j = M[(MF_JX + a) * N + i];
      M[(MF_AX + a) * N + i] = A[a];
      M[(MF_FX + a) * N + i] = F[a];
      M[(MF_UX + a) * N + i] = (j + 0.5 * F[a]) / rho;
      M[(MF_VX + a) * N + i] = (j + p.tau * F[a]) / rho;
    }
  }
}

// D = sum_a [u_a(x+e_a) - u_a(x-e_a)]/2, u_z -> -u_z across the walls
__global__ void div_fwd_kernel(Geom g, double* __restrict__ M) {
  const size_t N = g.N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.N; i += gridDim.x * blockDim.x) {
    int x, y, z;
    coords(i, g, x, y, z);
    const double uz0 = M[MF_UZ * N + i];
    const double uzp = (z + 1 < g.nz) ? M[MF_UZ * N + i + g.plane] : -uz0;
    const double uzm = (z - 1 >= 0) ? M[MF_UZ * N + i - g.plane] : -uz0;
    double D = 0.5 * (M[MF_UX * N + at(g, x + 1, y, z)] - M[MF_UX * N + at(g, x - 1, y, z)]);
    D += 0.5 * (M[MF_UY * N + at(g, x, y + 1, z)] - M[MF_UY * N + at(g, x, y - 1, z)]);
    D += 0.5 * (uzp - uzm);
    M[MF_D * N + i] = D;
  }
}

// streaming^T: adjoint of the post-collision populations l = 0..18 at node n in lattice Ln (f or g):
// lambda'_l(x + c_l), or through a wall the bounce-back that delivered f*_l(x) as f'_{opp(l)}(x) (g:
// with a minus sign)
template <bool G_LATTICE>
__device__ __forceinline__ void adj_pull(double (&v)[Q], const double* Ln, const Geom& g, const Node& n) {
  const size_t N = (size_t)g.N, plane = (size_t)g.plane;
#pragma unroll
  for (int l = 0; l < Q; ++l) {
    const int zn = n.z + CZ(l);
    const bool wall = zn < 0 || zn >= g.nz;
    const double* b = wall ? Ln + OPP(l) * N + (size_t)n.z * plane : Ln + l * N + (size_t)zn * plane;
    const double x = b[wall ? n.i : n.xs[1 + CX(l)] + n.ys[1 + CY(l)]];
    v[l] = G_LATTICE && wall ? -x : x;
  }
}

// Moments in c_l of the adjoint populations, weighted as the equilibria's terms are: sums per class
// (rest, axis, diagonal), 3 sum w om c_l a_l and 9 sum w om c_l c_l a_l. Every term of collision^T is
// polynomial in c_l of degree <= 2, so these ten numbers per lattice carry all of it.
struct AdjMoments {
  double s0, s1, s2;                 // om w sum of a over the class
  double jx, jy, jz;
  double qxx, qyy, qzz, qxy, qxz, qyz;
};
__device__ __forceinline__ AdjMoments adj_moments(const double (&a)[Q], const double (&w)[3], const double (&j3)[2],
                                                  const double (&q9)[2]) {
  double S[Q / 2], D[Q / 2];
#pragma unroll
  for (int k = 0; k < Q / 2; ++k) { S[k] = a[2 * k + 1] + a[2 * k + 2]; D[k] = a[2 * k + 1] - a[2 * k + 2]; }
  // pairs: 0..2 axis x, y, z; 3, 4 xy (same, opposite signs); 5, 6 xz; 7, 8 yz
  const double Pxy = S[3] + S[4], Pxz = S[5] + S[6], Pyz = S[7] + S[8];
  AdjMoments m;
  m.s0 = w[0] * a[0];
  m.s1 = w[1] * ((S[0] + S[1]) + S[2]);
  m.s2 = w[2] * ((Pxy + Pxz) + Pyz);
  m.jx = j3[0] * D[0] + j3[1] * ((D[3] + D[4]) + (D[5] + D[6]));
  m.jy = j3[0] * D[1] + j3[1] * ((D[3] - D[4]) + (D[7] + D[8]));
  m.jz = j3[0] * D[2] + j3[1] * ((D[5] - D[6]) + (D[7] - D[8]));
  m.qxx = q9[0] * S[0] + q9[1] * (Pxy + Pxz);
  m.qyy = q9[0] * S[1] + q9[1] * (Pxy + Pyz);
  m.qzz = q9[0] * S[2] + q9[1] * (Pxz + Pyz);
  m.qxy = q9[1] * (S[3] - S[4]);
  m.qxz = q9[1] * (S[5] - S[6]);
  m.qyz = q9[1] * (S[7] - S[8]);
  return m;
}

// Wall rules^T, collision^T and the Nu terms. Bound by its FP64 instructions like everything here; the
// moment form takes about 200 of them a node where the sum over the pairs took 650 (64^3: 124 us against
// 288; the three reverse kernels 222 us against 388).
// (The reverse kernels follow each other as the step's do, and like them read through plain loads only:
// wait_for_predecessor and ld_at in lb_split.cuh.)
__global__ void __launch_bounds__(kThreads) coll_adj_kernel(const double* M, const double* Ln, Geom g, Par p,
                                                            double* A, double* part) {
  __shared__ double sh[4][kThreads];
  const Node n = node_of(g);
  wait_for_predecessor();
  const size_t N = (size_t)g.N, i = (size_t)n.z * (size_t)g.plane + n.i;
  const bool wallz = n.z == 0 || n.z == g.nz - 1;
  double pTd = 0.0, pTu = 0.0, pG = 0.0, pJ = 0.0;
  if (n.valid) {
    const double rho = M[MF_RHO * N + i], T = M[MF_T * N + i], E = rho * T;
    const double ux = M[MF_UX * N + i], uy = M[MF_UY * N + i], uz = M[MF_UZ * N + i];
    double a_rho = 0.0, a_T = 0.0, a_D = 0.0;
    double a_v[3] = {0.0, 0.0, 0.0}, a_u[3] = {0.0, 0.0, 0.0};
    if (Ln) {
      double a[Q];
      adj_pull<false>(a, Ln, g, n);
      // f* = (1 - om) f + om f^eq(rho, v, T), f^eq = w rho [1 + 3 c.v + 4.5 (c.v)^2 - 1.5 v.v + 4.5 (T - 1/3) k]
      {
        const AdjMoments m = adj_moments(a, p.w, p.j3, p.q9);
        const double vx = M[MF_VX * N + i], vy = M[MF_VY * N + i], vz = M[MF_VZ * N + i];
        const double vv = vx * vx + vy * vy + vz * vz;
        const double sf = (m.s0 + m.s1) + m.s2, sfk = m.s2 - m.s0;
        const double qx = m.qxx * vx + m.qxy * vy + m.qxz * vz, qy = m.qxy * vx + m.qyy * vy + m.qyz * vz,
                     qz = m.qxz * vx + m.qyz * vy + m.qzz * vz;
        a_rho = sf * (1.0 - 1.5 * vv) + sfk * (4.5 * T - 1.5);
        a_rho += vx * (0.5 * qx + m.jx) + vy * (0.5 * qy + m.jy) + vz * (0.5 * qz + m.jz);
        a_T = 4.5 * rho * sfk;
        const double s3 = 3.0 * sf;
        a_v[0] = rho * (m.jx + qx - s3 * vx); a_v[1] = rho * (m.jy + qy - s3 * vy); a_v[2] = rho * (m.jz + qz - s3 * vz);
      }
      // g* = (1 - omk) g + omk g^eq(rho, T, u) + w S, S = -rho T D / c_v,
      // g^eq = w [rho T (1 + 3 c.u + 4.5 (c.u)^2 - 1.5 u.u) + 4.5 (lam T - rho T/3) k]
      adj_pull<true>(a, Ln + Q * N, g, n);
      {
        const AdjMoments m = adj_moments(a, p.wg, p.j3g, p.q9g);
        const double uu = ux * ux + uy * uy + uz * uz;
        const double sg = (m.s0 + m.s1) + m.s2, sgk = m.s2 - m.s0;
        const double qx = m.qxx * ux + m.qxy * uy + m.qxz * uz, qy = m.qxy * ux + m.qyy * uy + m.qyz * uz,
                     qz = m.qxz * ux + m.qyz * uy + m.qzz * uz;
        const double X = sg * (1.0 - 1.5 * uu) +
                         (ux * (0.5 * qx + m.jx) + uy * (0.5 * qy + m.jy) + uz * (0.5 * qz + m.jz));
        const double lS = p.src * sg;          // sum_l w_l lambda_l = sg/omk, times -1/c_v
        const double D = M[MF_D * N + i];
        a_rho += T * (X - 1.5 * sgk + lS * D);
        a_T += rho * (X + lS * D) + (4.5 * p.lam - 1.5 * rho) * sgk;
        a_D = lS * E;
        const double s3 = 3.0 * sg;
        a_u[0] = E * (m.jx + qx - s3 * ux); a_u[1] = E * (m.jy + qy - s3 * uy); a_u[2] = E * (m.jz + qz - s3 * uz);
      }
      if (wallz) {
        // thermal wall rule: g'_m(x_w) = ... + 2 w_m [rho T_w + 4.5 (lam T_w - rho T_w/3)(|c_m|^2-1)]
#pragma unroll
        for (int m = 0; m < Q; ++m) {
          const bool bot = (CZ(m) > 0 && n.z == 0), top = (CZ(m) < 0 && n.z == g.nz - 1);
          if (bot || top) {
            const double Tw = bot ? p.Td : p.Tu;
            const double lm = Ln[(Q + m) * N + i];
            const double k = CSQ(m) - 1;
            a_rho += 2.0 * WT<double>(m) * Tw * (1.0 - 1.5 * k) * lm;
            const double dTw = 2.0 * WT<double>(m) * (rho + 4.5 * (p.lam - rho / 3.0) * k) * lm;
            if (bot) pTd += dTw; else pTu += dTw;
          }
        }
      }
    }
    // Nu terms: J_n = (1/N_t)[1 + sum_x rho U u_z / (kappa (T_d - T_u) nx ny)], U = c_v T + (G/4) e^{-2/rho}
    if (p.include_nu) {
      const double psi = M[MF_PSI * N + i];
      const double e2 = psi * psi;            // e^{-2/rho} = psi^2
      const double U = p.cv * T + 0.25 * p.G * e2;
      const double ku = p.Kc * uz, kr = p.Kc * rho;
      a_rho += ku * U;        // and the derivative of e^{-2/rho}, which vel_adj adds (it has 1/rho)
      a_T += kr * p.cv * uz;
      a_u[2] += kr * U;
      pG = kr * uz * 0.25 * e2;
      pJ = kr * U * uz;       // J = 1 + sum_n sum_x Kc rho U u_z (conduction telescopes)
    }
    A[AF_RHO * N + i] = a_rho; A[AF_T * N + i] = a_T; A[AF_D * N + i] = a_D;
#pragma unroll
    for (int k = 0; k < 3; ++k) { A[(AF_UX + k) * N + i] = a_u[k]; A[(AF_VX + k) * N + i] = a_v[k]; }
  }
  double* o = part + (size_t)blockIdx.x * P_COUNT;
  if (p.include_nu) {
    const double s2 = block_sum(pG, sh[0]), s3 = block_sum(pJ, sh[1]);
    if (threadIdx.x == 0) { o[P_G] += s2; o[P_J] += s3; }
  }
  if (wallz && Ln) {
    const double s0 = block_sum(pTd, sh[2]), s1 = block_sum(pTu, sh[3]);
    if (threadIdx.x == 0) { o[P_TD] += s0; o[P_TU] += s1; }
  }
}

// divergence^T (radius-1 gather), velocities^T: u = (j + F/2)/rho, u' = (j + tau F)/rho, the node's own
// factors of force^T: F = -G psi A + rho g_z z, psi = e^{-1/rho}, and T = E/rho ^T. One reciprocal per
// node serves this kernel and the next (64^3: 33 us).
__global__ void __launch_bounds__(kThreads) vel_adj_kernel(const double* M, Geom g, Par p, double* A, double* part) {
  __shared__ double sh[kThreads];
  const Node n = node_of(g);
  wait_for_predecessor();
  const size_t N = (size_t)g.N, plane = (size_t)g.plane, zo = (size_t)n.z * plane, i = zo + n.i;
  double pG = 0.0;
  if (n.valid) {
    const double* aD = A + AF_D * N;
    const double own = aD[i];
    const double dm = n.z >= 1 ? aD[i - plane] : own, dp = n.z <= g.nz - 2 ? aD[i + plane] : own;
    const double gr[3] = {aD[zo + n.xs[0] + n.ys[1]] - aD[zo + n.xs[2] + n.ys[1]],
                          aD[zo + n.xs[1] + n.ys[0]] - aD[zo + n.xs[1] + n.ys[2]], dm - dp};
    const double rho = M[MF_RHO * N + i], psi = M[MF_PSI * N + i];
    const double inv = 1.0 / rho;
    double au[3], av[3], mu[3], mv[3], ma[3];       // every load before the first store
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      au[k] = A[(AF_UX + k) * N + i]; av[k] = A[(AF_VX + k) * N + i];
      mu[k] = M[(MF_UX + k) * N + i]; mv[k] = M[(MF_VX + k) * N + i]; ma[k] = M[(MF_AX + k) * N + i];
    }
    const double aT = A[AF_T * N + i], ar = A[AF_RHO * N + i], T = M[MF_T * N + i];
    double dot = 0.0, FA = 0.0, lFz = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double lu = au[k] + 0.5 * gr[k], lv = av[k];
      A[(AF_JX + k) * N + i] = (lv + lu) * inv;
      const double lF = (p.tau * lv + 0.5 * lu) * inv;
      dot += mv[k] * lv + mu[k] * lu;
      FA += lF * ma[k];
      A[(AF_HX + k) * N + i] = psi * lF;
      if (k == 2) lFz = lF;
    }
    const double aE = aT * inv;
    const double kp = -p.G * psi * inv * inv;       // lambda_psi -> lambda_rho of the terms -G (...)
    pG = -psi * FA;
    A[AF_E * N + i] = aE;
    A[AF_KP * N + i] = kp * (1.0 / 12.0);
    double a_rho = ar - dot * inv + p.gz * lFz + kp * FA - aE * T;
    if (p.include_nu) a_rho += p.Kc * mu[2] * (0.5 * p.G * psi * psi) * inv;
    A[AF_RHO * N + i] = a_rho;
  }
  const double s = block_sum(pG, sh);
  if (threadIdx.x == 0) part[(size_t)blockIdx.x * P_COUNT + P_G] += s;
}

// force^T's gather and moments^T. psi(y) enters F(x) for every link x + c_l = y: sum_l W_l c_l . H(y - c_l);
// a ghost link of a wall plane (x + c_l beyond the wall, its mirror image y) is the same sum over the
// plane's mirror image with H_z negated (33 FP64 additions; 18 dot products with their own loads took
// 166 instructions). 64^3: 65 us against 80. Then lambda_l = (1 - om) lambda*_l + a_rho + c_l . a_j (g: + a_E).
__global__ void __launch_bounds__(kThreads) force_adj_kernel(const double* A, const double* Ln, Geom g, Par p,
                                                             double* L) {
  const Node n = node_of(g);
  wait_for_predecessor();
  if (!n.valid) return;
  const size_t N = (size_t)g.N, plane = (size_t)g.plane, zo = (size_t)n.z * plane, i = zo + n.i;
  const double *Hx = A + AF_HX * N + zo, *Hy = A + AF_HY * N + zo, *Hz = A + AF_HZ * N + zo;
  auto at2 = [&](const double* f, int dx, int dy) { return f[n.xs[1 + dx] + n.ys[1 + dy]]; };
  double s = 2.0 * ((at2(Hx, -1, 0) - at2(Hx, 1, 0)) + (at2(Hy, 0, -1) - at2(Hy, 0, 1)));
  s += ((at2(Hx, -1, -1) + at2(Hy, -1, -1)) - (at2(Hx, 1, 1) + at2(Hy, 1, 1))) +
       ((at2(Hx, -1, 1) - at2(Hy, -1, 1)) - (at2(Hx, 1, -1) - at2(Hy, 1, -1)));
#pragma unroll
  for (int dz = -1; dz <= 1; dz += 2) {
    const bool wall = n.z + dz < 0 || n.z + dz >= g.nz;
    const long long off = wall ? 0 : dz * (long long)plane;
    const double *hx = Hx + off, *hy = Hy + off, *hz = Hz + off;
    s += (at2(hx, -1, 0) - at2(hx, 1, 0)) + (at2(hy, 0, -1) - at2(hy, 0, 1));
    const double t = 2.0 * at2(hz, 0, 0) + ((at2(hz, -1, 0) + at2(hz, 1, 0)) + (at2(hz, 0, -1) + at2(hz, 0, 1)));
    s = ((dz < 0) != wall) ? s + t : s - t;
  }
  const double a_rho = A[AF_RHO * N + i] + A[AF_KP * N + i] * s;
  const double jx = A[AF_JX * N + i], jy = A[AF_JY * N + i], jz = A[AF_JZ * N + i];
  double a[Q];
  if (Ln) adj_pull<false>(a, Ln, g, n);
#pragma unroll
  for (int l = 0; l < Q; ++l) {
    const double c = l == 0 ? a_rho : a_rho + cdot<double>(l, jx, jy, jz);
    L[l * N + i] = Ln ? p.om1 * a[l] + c : c;
  }
  const double aE = A[AF_E * N + i];
  if (Ln) adj_pull<true>(a, Ln + Q * N, g, n);
#pragma unroll
  for (int l = 0; l < Q; ++l) L[(Q + l) * N + i] = Ln ? p.omk1 * a[l] + aE : aE;
}

// dJ/dT0 from lambda_0: x_0 = (f^eq(rho0, 0, T0), g^eq(rho0, T0, 0))
__global__ void init_grad_kernel(const double* __restrict__ L0, const double* __restrict__ M0, Geom g,
                                 double lam, double* __restrict__ out) {
  const size_t N = g.N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.N; i += gridDim.x * blockDim.x) {
    const double rho = M0[MF_RHO * N + i];
    double s = 0.0;
    for (int l = 0; l < Q; ++l) {
      const double k = CSQ(l) - 1, w = WT<double>(l);
      s += L0[l * N + i] * w * rho * 4.5 * k + L0[(Q + l) * N + i] * w * (rho + 4.5 * (lam - rho / 3.0) * k);
    }
    out[i] = s;
  }
}

}  // namespace adj
}  // namespace tlbm

using namespace tlbm;

namespace {

// The step of state n writes the fields that the reverse sweep reads straight into m
// ([MF_COUNT][N]): the three-kernel step keeps its own fields there.
void adj_fields(KArgs& a, double* m) {
  a.adj_m = m;
  if (!a.fd_rho) return;
  const size_t N = (size_t)a.N;
  a.fd_rho = m + MF_RHO * N;
  a.fd_psi = m + MF_PSI * N;
  for (int k = 0; k < 3; ++k) { a.fd_u[k] = m + (MF_UX + k) * N; a.fd_v[k] = m + (MF_VX + k) * N; }
}

struct DevBuf {
  void* p = nullptr;
  ~DevBuf() { if (p) cudaFree(p); }
};

}  // namespace

extern "C" int lb_adjoint_step(lb_ctx* c, long long nsteps, int checkpoint_every, double* J,
                               double* dJ_dTd, double* dJ_dTu, double* dJ_dG, double* dJ_dT0) {
  using namespace tlbm::adj;
  if (!c) return LB_EINVAL;
  if (nsteps < 1 || checkpoint_every < 0) return lb_fail(c, LB_EINVAL, "nsteps must be >= 1 and checkpoint_every >= 0");
  if (dJ_dT0 && (c->step != 0 || !c->from_init))
    return lb_fail(c, LB_EINVAL, "dJ_dT0 needs the state of lb_init (step 0)");
  if (!(c->p.T_d != c->p.T_u)) return lb_fail(c, LB_EINVAL, "T_d == T_u: Nu is undefined");
  if (c->p.forcing != FORCE_SHIFT || c->p.psi_kind != PSI_EXP)
    return lb_fail(c, LB_EUNSUP, "the adjoint transposes the paper's scheme (velocity shift, psi = exp(-1/rho)) only");
  const size_t N = (size_t)c->N;
  const size_t pbytes = (size_t)c->ops->slots * N * c->ops->esize;
  const size_t sbytes = 2 * (size_t)Q * N * sizeof(double);
  const size_t mstate = (size_t)MF_COUNT * N;   // doubles per state's fields
  const int nbp = (c->plane + kThreads - 1) / kThreads;
  const size_t parts = (size_t)nbp * (size_t)c->p.nz;      // CTAs of a reverse kernel
  // device bytes of the call for segment length k (the allocations below)
  auto bytes_for = [&](long long k) -> double {
    const double nck_k = (double)((nsteps + k - 1) / k);
    return nck_k * 2.0 * (double)pbytes + 4.0 * (double)pbytes + 64.0 + 3.0 * (double)sbytes +
           (double)(k + 1) * (double)mstate * 8.0 + (double)AF_COUNT * (double)N * 8.0 +
           (double)parts * P_COUNT * 8.0 + (dJ_dT0 ? (double)N * 8.0 : 0.0);
  };
  long long K = checkpoint_every < nsteps ? checkpoint_every : nsteps;
  if (checkpoint_every == 0) {
    // the longest segment whose buffers fit in 85 % of the free device memory: every state's
    // fields kept (no recomputation with FP64 storage) when they fit
    size_t free_b = 0, total_b = 0;
    LB_CU(c, cudaMemGetInfo(&free_b, &total_b));
    const double budget = 0.85 * (double)free_b;
    const double per_k = (double)mstate * 8.0;
    long long k = std::min<long long>(nsteps, (long long)std::max(1.0, budget / per_k));
    while (k > 1 && bytes_for(k) > budget) --k;
    if (bytes_for(k) > budget) return lb_fail(c, LB_ENOMEM, "adjoint buffers do not fit for any segment length");
    K = k;
  }
  const long long nck = (nsteps + K - 1) / K;
  cudaStream_t st = c->stream;
  const KArgs a0 = make_args(c);
  Geom g{c->p.nx, c->p.ny, c->p.nz, c->plane, c->N, nbp, a0.div_m, a0.div_s};

  // FP64 storage: the step writes the fields of the state it reads (adj_m), so the reverse sweep
  // needs no separate moments, force and divergence passes; other storage recomputes them in
  // FP64 from the FP64 image of each state.
  const bool fields = (c->ops->esize == sizeof(double));
  DevBuf ck, rb, xs, mb, ab, lb, pt, d0;
  if (cudaMalloc(&ck.p, (size_t)nck * 2 * pbytes) != cudaSuccess ||
      cudaMalloc(&rb.p, 4 * pbytes + 64) != cudaSuccess ||
      cudaMalloc(&xs.p, sbytes) != cudaSuccess ||
      cudaMalloc(&mb.p, (size_t)(K + 1) * mstate * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&ab.p, (size_t)AF_COUNT * N * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&lb.p, 2 * sbytes) != cudaSuccess ||
      cudaMalloc(&pt.p, parts * P_COUNT * sizeof(double)) != cudaSuccess ||
      (dJ_dT0 && cudaMalloc(&d0.p, N * sizeof(double)) != cudaSuccess))
    return lb_fail(c, LB_ENOMEM, "adjoint buffers");
  unsigned char* ckp = static_cast<unsigned char*>(ck.p);
  unsigned char* rbp = static_cast<unsigned char*>(rb.p);
  double* X = static_cast<double*>(xs.p);        // FP64 image of one state
  double* Ms = static_cast<double*>(mb.p);       // fields of the segment's states n0..n1
  double* A = static_cast<double*>(ab.p);
  double* Lb[2] = {static_cast<double*>(lb.p), static_cast<double*>(lb.p) + 2 * Q * N};
  double* part = static_cast<double*>(pt.p);
  LB_CU(c, cudaMemsetAsync(part, 0, parts * P_COUNT * sizeof(double), st));
  const int frc = flush_sample(c);    // a Nu sample due for the time average of lb_nusselt
  if (frc) return frc;

  const double dT = c->p.T_d - c->p.T_u;
  Par par;
  std::memset(&par, 0, sizeof(par));
  par.tau = c->p.tau_nu; par.om = 1.0 / c->p.tau_nu; par.omk = 1.0 / c->p.tau_kappa; par.G = c->p.G; par.gz = c->p.g_z;
  par.lam = c->lam; par.cv = c->p.c_v; par.kappa = c->p.kappa; par.Td = c->p.T_d; par.Tu = c->p.T_u;
  par.om1 = 1.0 - par.om; par.omk1 = 1.0 - par.omk;
  const double wc[3] = {1.0 / 3.0, 1.0 / 18.0, 1.0 / 36.0};
  for (int k = 0; k < 3; ++k) { par.w[k] = par.om * wc[k]; par.wg[k] = par.omk * wc[k]; }
  for (int k = 0; k < 2; ++k) {
    par.j3[k] = 3.0 * par.w[k + 1]; par.q9[k] = 9.0 * par.w[k + 1];
    par.j3g[k] = 3.0 * par.wg[k + 1]; par.q9g[k] = 9.0 * par.wg[k + 1];
  }
  par.src = -1.0 / (par.omk * par.cv);
  par.Kc = 1.0 / ((double)nsteps * c->p.kappa * dT * (double)c->p.nx * (double)c->p.ny);
  const int nb = (int)std::min<long long>(1024, ((long long)N + kThreads - 1) / kThreads);   // grid-stride passes
  // fields of a state from its storage image (a.fin, a.gin) by the separate FP64 passes
  auto fields_by_passes = [&](const KArgs& a, double* Mn) -> int {
    LB_CU(c, c->ops->pops(a, X, X + Q * N, st));
    macro_kernel<<<nb, kThreads, 0, st>>>(X, g, Mn);
    force_fwd_kernel<<<nb, kThreads, 0, st>>>(g, par, Mn);
    div_fwd_kernel<<<nb, kThreads, 0, st>>>(g, Mn);
    LB_CU(c, cudaGetLastError());
    return LB_OK;
  };

  // forward: checkpoints every K steps; with FP64 storage the last segment's fields as it goes
  const long long n0_last = (nck - 1) * K;
  for (long long n = 0; n < nsteps; ++n) {
    if (n % K == 0) {
      unsigned char* dst = ckp + (size_t)(n / K) * 2 * pbytes;
      LB_CU(c, cudaMemcpyAsync(dst, c->f[c->cur], pbytes, cudaMemcpyDeviceToDevice, st));
      LB_CU(c, cudaMemcpyAsync(dst + pbytes, c->g[c->cur], pbytes, cudaMemcpyDeviceToDevice, st));
    }
    KArgs a = make_args(c);
    if (fields && n >= n0_last) adj_fields(a, Ms + (size_t)(n - n0_last) * mstate);
    LB_CU(c, launch_step(c, a, MODE_STEP));
    c->cur ^= 1;
    c->step += 1;
  }
  if (fields) {
    const int rc = fields_by_passes(make_args(c), Ms + (size_t)(nsteps - n0_last) * mstate);
    if (rc != LB_OK) return rc;
  }

  int li = 0;   // Lb[li] = lambda_{n+1} (zero before the last state)
  bool have_next = false;
  for (long long s = nck - 1; s >= 0; --s) {
    const long long n0 = s * K;
    const long long n1 = (s == nck - 1) ? nsteps : (s + 1) * K - 1;   // states n0..n1 of this segment
    if (!(fields && s == nck - 1)) {
      // recompute the segment from its checkpoint: the fields of states n0..n1
      unsigned char* src = ckp + (size_t)s * 2 * pbytes;
      LB_CU(c, cudaMemcpyAsync(rbp, src, pbytes, cudaMemcpyDeviceToDevice, st));
      LB_CU(c, cudaMemcpyAsync(rbp + pbytes, src + pbytes, pbytes, cudaMemcpyDeviceToDevice, st));
      int rc = 0;
      for (long long n = n0; n <= n1; ++n) {
        KArgs a = make_args(c);
        a.fin = rbp + (size_t)rc * 2 * pbytes;
        a.gin = rbp + (size_t)rc * 2 * pbytes + pbytes;
        double* Mn = Ms + (size_t)(n - n0) * mstate;
        if (!fields || n == n1) {
          const int frc2 = fields_by_passes(a, Mn);
          if (frc2 != LB_OK) return frc2;
        } else {
          adj_fields(a, Mn);
        }
        if (n < n1) {
          a.fout = rbp + (size_t)(1 - rc) * 2 * pbytes;
          a.gout = rbp + (size_t)(1 - rc) * 2 * pbytes + pbytes;
          LB_CU(c, launch_step(c, a, MODE_STEP));
          rc ^= 1;
        }
      }
    }
    for (long long n = n1; n >= n0; --n) {
      const double* Mn = Ms + (size_t)(n - n0) * mstate;
      par.include_nu = (n >= 1) ? 1 : 0;
      double* Lcur = Lb[1 - li];
      const double* Lnext = have_next ? Lb[li] : nullptr;
      const unsigned pg = (unsigned)parts;
      LB_CU(c, follow(coll_adj_kernel, pg, kThreads, st, Mn, Lnext, g, par, A, part));
      LB_CU(c, follow(vel_adj_kernel, pg, kThreads, st, Mn, g, par, A, part));
      LB_CU(c, follow(force_adj_kernel, pg, kThreads, st, static_cast<const double*>(A), Lnext, g, par, Lcur));
      li = 1 - li;
      have_next = true;
    }
    if (s == 0 && dJ_dT0) {
      init_grad_kernel<<<nb, kThreads, 0, st>>>(Lb[li], Ms, g, c->lam, static_cast<double*>(d0.p));
      LB_CU(c, cudaGetLastError());
    }
  }
  std::vector<double> hp(parts * P_COUNT);
  LB_CU(c, cudaMemcpyAsync(hp.data(), part, hp.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
  if (dJ_dT0) LB_CU(c, cudaMemcpyAsync(dJ_dT0, d0.p, N * sizeof(double), cudaMemcpyDeviceToHost, st));
  LB_CU(c, cudaStreamSynchronize(st));
  double s[P_COUNT] = {0.0, 0.0, 0.0, 0.0};
  for (size_t b = 0; b < parts; ++b)
    for (int k = 0; k < P_COUNT; ++k) s[k] += hp[b * P_COUNT + k];
  // the convective terms sum_x rho U u_z / (T_d - T_u) of Nu depend on the wall temperatures as well
  const double conv = s[P_J] / (par.Td - par.Tu);
  if (J) *J = 1.0 + s[P_J];
  if (dJ_dTd) *dJ_dTd = s[P_TD] - conv;
  if (dJ_dTu) *dJ_dTu = s[P_TU] + conv;
  if (dJ_dG) *dJ_dG = s[P_G];
  return LB_OK;
}
