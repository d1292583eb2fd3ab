// lb_split.cuh -- the time step as three streaming kernels, one node per thread:
//
//   moments   pull f; write rho (FP32 compute: drho; FP64: and 1/rho), j and psi;
//   velocity  gather psi (Eq. (9)); write the physical velocity u = (j + F/2)/rho and, but for 16-bit
//             storage, the equilibrium velocity u' = (j + tau F)/rho (Guo forcing: F in its place);
//   collide   pull f and g, div(u) from six neighbours, collide and write both lattices.
//
// Per node FP32 moves 76 + 20, 20 + 24 and 152 + 28 + 152 bytes in them, at about the rate of a copy (161 x
// 210 x 128: 328 us); FP64 executes 61, 35 and 187 FP64 instructions, each at the rate
// of the FP64 pipe (128^3: 245, 139 and 735 us; the tile march with its pre-pass 1543).
// Nothing is recomputed and nothing waits at a barrier: the form of the FP64 step, which its FP64
// instructions bound, and of the cells too small to fill the GPU with marching CTAs, where the
// latency of one CTA's chain of planes is the time of the step.
#pragma once
#include "lb_kernels.cuh"

namespace tlbm {

// Node of a plane from its in-plane index: column x and row = y nx.
struct NodePos {
  unsigned x, row, i;
  bool valid;
};
__device__ __forceinline__ NodePos node_at(const KArgs& a, unsigned i) {
  NodePos n;
  n.i = i;
  n.valid = i < (unsigned)a.plane;
  n.x = i - (a.div_m ? (__umulhi(i, a.div_m) >> a.div_s) : i) * (unsigned)a.nx;
  n.row = i - n.x;
  return n;
}
// columns x-1, x, x+1 and rows (y-1) nx, y nx, (y+1) nx of a node, periodic
__device__ __forceinline__ void neighbours(unsigned (&xs)[3], unsigned (&ys)[3], const KArgs& a, unsigned x, unsigned row) {
  const unsigned nx = (unsigned)a.nx, last = (unsigned)a.plane - nx;
  xs[0] = x == 0 ? nx - 1 : x - 1; xs[1] = x; xs[2] = x + 1 == nx ? 0u : x + 1;
  ys[0] = row == 0 ? last : row - nx; ys[1] = row; ys[2] = row == last ? 0u : row + nx;
}

// Element i of a plane (the byte offset in a plane fits 32 bits). Plain loads: what a kernel reads here
// the launch before it wrote, and it is up before those writes are complete (wait_for_predecessor), so
// the read-only path, for memory that nobody writes while a kernel is up, is not for it.
template <class T> __device__ __forceinline__ T ld_at(const T* base, unsigned i) {
  return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + (size_t)(i * (unsigned)sizeof(T)));
}
template <class T> __device__ __forceinline__ void st_at(T* base, unsigned i, T v) {
  *reinterpret_cast<T*>(reinterpret_cast<char*>(base) + (size_t)(i * (unsigned)sizeof(T))) = v;
}

__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// c x of a constant c whose FP32 rounding is kept as a second float
__device__ __forceinline__ double mul2(double c, double, double x) { return c * x; }
__device__ __forceinline__ float mul2(float c, float lo, float x) { return fma_rn(c, x, lo * x); }

// 1/x: the division for FP64; for FP32 one step of Newton's iteration, r (2 - y r), on the hardware's
// approximation r of 1/y (relative error at most 2^-23, which the step squares): within 0.501 of the
// last place (every bit pattern is tested). y is x scaled by a power of two, so that neither y nor 1/y
// is subnormal over the whole range of x; 0 and the infinities keep the approximation's own result. No
// branch: __frcp_rn in its place gave the same bits on the timed cells and made the FP16 256^3 cell
// (two nodes per thread) 4.9 % slower, local references 1.4 %, FP32 0.8 %, all against a step that knew
// normal x only; this form 1.4, 0.9 and 0.5 %.
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
__device__ __forceinline__ float recip(float x) {
  const float ax = fabsf(x);
  const float s = ax > 0x1p64f ? 0x1p-64f : (ax < 0x1p-64f ? 0x1p64f : 1.0f);
  const float y = x * s;
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
  const float e = fmaf(-y, r, 1.0f);
  return (fabsf(e) < 0.5f ? fmaf(r, e, r) : r) * s;
}

// The 19 populations pulled at a node of plane z of lattice buf (through a wall the bounce-back
// source), with the local references added.
template <class S, class R>
__device__ __forceinline__ void split_pull(R (&v)[Q], const S* buf, size_t N, size_t plane, int nz,
                                           int z, const unsigned (&xs)[3], const unsigned (&ys)[3]) {
  const unsigned own = xs[1] + ys[1];
  S raw[Q];
#pragma unroll
  for (int l = 0; l < Q; ++l) {
    const bool through = (CZ(l) > 0 && z == 0) || (CZ(l) < 0 && z == nz - 1);
    const S* b = through ? buf + OPP(l) * N + (size_t)z * plane : buf + l * N + (size_t)(z - CZ(l)) * plane;
    raw[l] = ld_at(b, through ? own : xs[1 - CX(l)] + ys[1 - CY(l)]);
  }
#pragma unroll
  for (int l = 0; l < Q; ++l) v[l] = cvt<S, R>(raw[l]);
  if constexpr (IsLoc<S>::v) {
    const S* r1 = buf + (size_t)Q * N;
    const S* r2 = buf + (size_t)(Q + 1) * N;
    const size_t zo = (size_t)z * plane;
    v[0] += 12.0f * (cvt<S, R>(ld_at(r1 + zo, own)) - cvt<S, R>(ld_at(r2 + zo, own)));
#pragma unroll
    for (int l = 1; l < Q; ++l) {
      const bool through = (CZ(l) > 0 && z == 0) || (CZ(l) < 0 && z == nz - 1);
      const size_t zs = through ? zo : (size_t)(z - CZ(l)) * plane;
      v[l] += cvt<S, R>(ld_at((CSQ(l) == 1 ? r1 : r2) + zs, through ? own : xs[1 - CX(l)] + ys[1 - CY(l)]));
    }
  }
}

// Density deviation of a wall node for the thermal wall rule: the sum of its own stored f (with their
// local references), in the order of g_wall_fix.
template <class S, class R>
__device__ __forceinline__ R split_wall_density(const S* fin, size_t N, size_t o) {
  auto at = [&](int l) -> R { return cvt<S, R>(ld_at(fin + l * N + o, 0u)); };
  R ref[3] = {R(0), R(0), R(0)};
  if constexpr (IsLoc<S>::v) {
    ref[1] = at(Q); ref[2] = at(Q + 1);
    ref[0] = R(12) * (ref[1] - ref[2]);
  }
  R dp = IsLoc<S>::v ? at(0) + ref[0] : at(0);
#pragma unroll
  for (int l = 1; l < Q; ++l) dp = dp + (IsLoc<S>::v ? at(l) + ref[CSQ(l)] : at(l));
  return dp;
}

// Density and momentum deviations from the sums and differences of the opposite pairs (39 additions
// instead of 45 term by term; the differences of like numbers come first).
template <class R>
__device__ __forceinline__ void pair_moments(const R (&f)[Q], R& drho, R& jx, R& jy, R& jz) {
  R s[Q / 2], d[Q / 2];
#pragma unroll
  for (int k = 0; k < Q / 2; ++k) { s[k] = f[2 * k + 1] + f[2 * k + 2]; d[k] = f[2 * k + 1] - f[2 * k + 2]; }
  drho = ((f[0] + (s[0] + s[1])) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + (s[7] + s[8])));
  jx = d[0] + ((d[3] + d[4]) + (d[5] + d[6]));
  jy = d[1] + ((d[3] - d[4]) + (d[7] + d[8]));
  jz = d[2] + ((d[5] - d[6]) + (d[7] - d[8]));
}
// 12 sum_l W_l c_l psi(x + c_l) from the nine pair differences d_k = psi(x + c_l) - psi(x - c_l),
// l = 2k + 1: twice the axis pair's plus the diagonal pairs' (W = 1/6, 1/12)
template <class R>
__device__ __forceinline__ void pair_gradient(const R (&d)[Q / 2], R& ax, R& ay, R& az) {
  ax = R(2) * d[0] + ((d[3] + d[4]) + (d[5] + d[6]));
  ay = R(2) * d[1] + ((d[3] - d[4]) + (d[7] + d[8]));
  az = R(2) * d[2] + ((d[5] - d[6]) + (d[7] - d[8]));
}

// psi of a node as the fields keep it. FP32 compute, the paper's psi: e = psi/psi(rho1) - 1 = e^t - 1,
// t = 1/rho1 - 1/rho = drho/(rho rho0) + t1 (sum_l W_l c_l = 0, so the force sum may take e for psi; it
// then adds small numbers). rho1 is the reference density or, where psi(rho0)^2 would leave the range of
// floats, 1/40.
template <class R, bool VDW>
__device__ __forceinline__ R split_psi(R rho, R drho, R inv, const KPar<R>& kp) {
  if constexpr (VDW) return psi_vdw(rho, kp);
  else if constexpr (sizeof(R) == 8) return fexp(-inv);
  else {
    const R x = drho * inv;
    return expm1_dev(fma_rn(x, kp.irho0, fma_rn(x, kp.irho0_lo, kp.t1)));
  }
}
// -G psi / 12 (FP32 compute, the paper's psi: times psi(rho1)) from psi as kept
template <class R, bool VDW>
__device__ __forceinline__ R split_mg(R psi, const KPar<R>& kp) {
  if constexpr (sizeof(R) == 8) return kp.mg * psi;
  else {
    const R p = VDW ? psi : R(1) + psi;
    return mul2(kp.mg, kp.mg_lo, p);
  }
}
// tau F-factor / rho from F-factor / rho
template <class R> __device__ __forceinline__ R split_mv(R mi, const KPar<R>& kp) { return mul2(kp.tau, kp.tau_lo, mi); }

// BGK relaxation of one lattice towards its equilibrium around the velocity v, pair by pair:
//   out_l = om1 in_l + [ev + 9 (c.v)(c.F')] +- [s (c.v) + 3 (c.F')],  ev = q (c.v)^2 + P per class,
// F' = 0 without Guo forcing. in(l) and put(l, value) access the populations. FULL: om1 = 0 (relaxation
// time 1), the populations themselves do not enter.
template <class R, bool GUO, bool FULL = false, class In, class Put>
__device__ __forceinline__ void relax(R om1, const R (&P)[3], const R (&q)[3], const R (&s)[3], R vx, R vy, R vz,
                                      const R (&F)[3], R ks, In in, Put put) {
  put(0, FULL ? P[0] : fma_rn(om1, in(0), P[0]));
#pragma unroll
  for (int l = 1; l < Q; l += 2) {
    const R cv = cdot<R>(l, vx, vy, vz);
    R ev = fma_rn(q[CLS(l)] * cv, cv, P[CLS(l)]);
    if constexpr (GUO) {
      const R cF = (WT<R>(l) * ks) * cdot<R>(l, F[0], F[1], F[2]);
      ev = ev + R(9) * cv * cF;
      const R od = fma_rn(s[CLS(l)], cv, R(3) * cF);
      put(l, fma_rn(om1, in(l), ev) + od);
      put(OPP(l), fma_rn(om1, in(OPP(l)), ev) - od);
    } else {
      put(l, fma_rn(s[CLS(l)], cv, FULL ? ev : fma_rn(om1, in(l), ev)));
      put(OPP(l), fma_rn(-s[CLS(l)], cv, FULL ? ev : fma_rn(om1, in(OPP(l)), ev)));
    }
  }
}
// g towards g^eq(rho, T, u) with the counter term; D2 = 2 div(u). Per class (rest, axis, diagonal)
// P = go [dE - 1.5 E u.u - E div(u)/(c_v omk) + (|c|^2 - 1) tg], tg = 4.5 (lam (T - T0) - dE/3).
template <class R, class In, class Put>
__device__ __forceinline__ void relax_g(const KPar<R>& kp, R E, R dE, R drho, R inv, R D2, R ux, R uy, R uz, In in, Put put) {
  const R uu = ux * ux + uy * uy + uz * uz;
  const R b0 = dE - E * (R(1.5) * uu + D2 * kp.src);
  const R tg = kp.lam45 * ((dE - kp.T0 * drho) * inv) - R(1.5) * dE;
  const R P[3] = {mul2(kp.go[0], kp.go_lo[0], b0 - tg), mul2(kp.go[1], kp.go_lo[1], b0), mul2(kp.go[2], kp.go_lo[2], b0 + tg)};
  const R q[3] = {R(0), kp.gq[1] * E, kp.gq[2] * E};
  const R s[3] = {R(0), mul2(kp.gs[1], kp.gs_lo[1], E), mul2(kp.gs[2], kp.gs_lo[2], E)};
  const R F[3] = {R(0), R(0), R(0)};
  if constexpr (sizeof(R) == 8) {
    // tau_kappa = 1: 18 of the 182 FP64 instructions of a collision less
    if (kp.omk1 == R(0)) {
      relax<R, false, true>(kp.omk1, P, q, s, ux, uy, uz, F, R(0), in, put);
      return;
    }
  }
  relax<R, false>(kp.omk1, P, q, s, ux, uy, uz, F, R(0), in, put);
}
// f towards f^eq(rho, u', T) (w = u'), or with Guo forcing towards f^eq(rho, u, T) plus its source
// (w = F). a0 = drho - 1.5 rho v.v, th = 4.5 (rho (T - 1/3) - rho0 (T0 - 1/3)) = 4.5 (dE - drho/3).
template <class R, bool GUO, class In, class Put>
__device__ __forceinline__ void relax_f(const KPar<R>& kp, R rho, R drho, R dE, R ux, R uy, R uz, const R (&w)[3], In in, Put put) {
  const R vx = GUO ? ux : w[0], vy = GUO ? uy : w[1], vz = GUO ? uz : w[2];
  const R vv = vx * vx + vy * vy + vz * vz;
  const R a0 = drho - (R(1.5) * rho) * vv;
  const R th = R(4.5) * dE - R(1.5) * drho;
  R P[3] = {mul2(kp.fo[0], kp.fo_lo[0], a0 - th), mul2(kp.fo[1], kp.fo_lo[1], a0), mul2(kp.fo[2], kp.fo_lo[2], a0 + th)};
  const R q[3] = {R(0), kp.fq[1] * rho, kp.fq[2] * rho};
  const R s[3] = {R(0), mul2(kp.fs[1], kp.fs_lo[1], rho), mul2(kp.fs[2], kp.fs_lo[2], rho)};
  if constexpr (GUO) {
    // (1 - om/2) w_l [3 (c - u).F + 9 (c.u)(c.F)]: the part -3 u.F of the even terms
    const R uF = R(-3) * kp.ks * (ux * w[0] + uy * w[1] + uz * w[2]);
    P[0] += WT<R>(0) * uF; P[1] += WT<R>(1) * uF; P[2] += WT<R>(7) * uF;
  }
  relax<R, GUO>(kp.om1, P, q, s, vx, vy, vz, w, kp.ks, in, put);
}

// One node's terms of the diagnostics: rho U u_z, T, rho, rho T, minima and the non-finite flag.
// U = c_v T + int_0^rho P_NI/s^2 ds: (G/4) e^{-2/rho}, or -T_v ln(1 - b rho) - a rho (vdW).
template <class R> struct DiagTerms {
  R conv = R(0), T = R(0), rho = R(0), E = R(0), mr = R(sizeof(R) == 8 ? 1e300 : 3.0e38), mT = mr;
  bool bad = false, bad2 = false;
  template <bool VDW>
  __device__ __forceinline__ void take(const KArgs& a, R r, R inv, R t, R e, R ux, R uy, R uz) {
    const KPar<R>& kp = kpar<R>(a);
    R U;
    if constexpr (sizeof(R) == 8)
      U = a.c_v * t + (VDW ? -kp.vT * log(1.0 - kp.vb * r) - kp.va * r : 0.25 * a.G * exp(-2.0 / r));
    else
      U = R(a.c_v) * t + (VDW ? -kp.vT * logf(R(1) - kp.vb * r) - kp.va * r : R(0.25) * kp.G * fexp(R(-2) * inv));
    conv = r * U * uz;
    T = t; rho = r; E = e; mr = r; mT = t;
    bad = !(isfinite(r) && isfinite(t) && isfinite(ux) && isfinite(uy) && isfinite(uz));
  }
  // a second node's terms as well (reduce with PAIR)
  __device__ __forceinline__ void add(const DiagTerms& b) {
    conv += b.conv; T += b.T; rho += b.rho; E += b.E;
    mr = fmin(mr, b.mr); mT = fmin(mT, b.mT);
    bad2 = b.bad;
  }
  // Warp sums in the compute precision into red[7][NW] (column w). The four sums are reduced together,
  // each exchange halving the values a lane carries (6 shuffles instead of 20), the two minima likewise.
  template <int NW, bool PAIR = false> __device__ __forceinline__ void reduce(R (&red)[7][NW], int w, int lane) {
    const bool hi = (lane & 16) != 0, mid = (lane & 8) != 0;
    const R p = (hi ? rho : conv) + __shfl_xor_sync(0xffffffffu, hi ? conv : rho, 16);
    const R q = (hi ? E : T) + __shfl_xor_sync(0xffffffffu, hi ? T : E, 16);
    R s = (mid ? q : p) + __shfl_xor_sync(0xffffffffu, mid ? p : q, 8);
    R m = fmin(hi ? mT : mr, __shfl_xor_sync(0xffffffffu, hi ? mr : mT, 16));
    m = fmin(m, __shfl_xor_sync(0xffffffffu, m, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    int nbad = __popc(__ballot_sync(0xffffffffu, bad));
    if constexpr (PAIR) nbad += __popc(__ballot_sync(0xffffffffu, bad2));
    // lanes 0, 8, 16, 24 hold conv, T, rho, E; lanes 0 and 16 the minima
    if ((lane & 7) == 0) red[lane >> 3][w] = s;
    if ((lane & 15) == 0) red[4 + (lane >> 4)][w] = m;
    if (lane == 0) red[6][w] = R(nbad);
  }
};
// The partials of one CTA's plane piece from its warps', by one warp: eight lanes per quantity, the sums
// in FP64 in a fixed tree (a chain over the warps took twice as long).
template <class R, int NW>
__device__ __forceinline__ void diag_combine(const R (&red)[7][NW], int lane, double* part) {
  static_assert(NW <= 8, "eight lanes per quantity");
  const int k = lane >> 3, w = lane & 7;
  double s = w < NW ? double(red[k][w]) : 0.0;                       // conv, T, rho, E
  const int km = 4 + (k < 2 ? k : 2);                                // min rho, min T, non-finite
  R m = w < NW ? red[km][w] : (km == 6 ? R(0) : R(sizeof(R) == 8 ? 1e300 : 3.0e38));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    const R n = __shfl_xor_sync(0xffffffffu, m, o);
    m = km == 6 ? m + n : fmin(m, n);
  }
  if (w == 0) {
    part[k] = s;
    if (k < 3) part[4 + k] = double(m);
  }
}

// The kernels of one step follow each other closely: each is launched as its predecessor's CTAs end
// (programmatic dependent launch) and waits here, before its first access to memory, until all of the
// predecessor's results are there. (FP32 32^3: 14.7 us a step without, 7.6 us with. Letting the
// successor up earlier, while the predecessor still runs, only crowds its CTAs: FP64 32^3 28 -> 54 us.)
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- kernels: nb CTAs of NT threads per plane ---------------------------------------------------
template <class S, bool VDW, int NT>
__global__ void __launch_bounds__(NT) split_moments_kernel(const KArgs a, int nb) {
  using R = typename Store<S>::R;
  constexpr bool F64 = sizeof(R) == 8;
  const int z = (int)blockIdx.x / nb;
  const NodePos n = node_at(a, (blockIdx.x - (unsigned)(z * nb)) * NT + threadIdx.x);
  wait_for_predecessor();
  if (!n.valid) return;
  unsigned xs[3], ys[3];
  neighbours(xs, ys, a, n.x, n.row);
  R f[Q];
  split_pull<S, R>(f, static_cast<const S*>(a.fin), (size_t)a.N, (size_t)a.plane, a.nz, z, xs, ys);
  R drho, jx, jy, jz;
  pair_moments<R>(f, drho, jx, jy, jz);
  const KPar<R>& kp = kpar<R>(a);
  const R rho = kp.rho0 + drho;
  const R inv = recip(rho);
  const size_t zo = (size_t)z * (size_t)a.plane;
  st_at(static_cast<R*>(a.fd_rho) + zo, n.i, F64 ? rho : drho);
  if constexpr (F64) st_at(static_cast<R*>(a.fd_inv) + zo, n.i, inv);
  st_at(static_cast<R*>(a.fd_j[0]) + zo, n.i, jx);
  st_at(static_cast<R*>(a.fd_j[1]) + zo, n.i, jy);
  st_at(static_cast<R*>(a.fd_j[2]) + zo, n.i, jz);
  st_at(static_cast<R*>(a.fd_psi) + zo, n.i, split_psi<R, VDW>(rho, drho, inv, kp));
}

template <class R, int VAR, int NT>
__global__ void __launch_bounds__(NT) split_velocity_kernel(const KArgs a, int nb) {
  constexpr bool GUO = (VAR & VAR_GUO) != 0, VDW = (VAR & VAR_VDW) != 0, F64 = sizeof(R) == 8;
  const int z = (int)blockIdx.x / nb;
  const NodePos n = node_at(a, (blockIdx.x - (unsigned)(z * nb)) * NT + threadIdx.x);
  wait_for_predecessor();
  if (!n.valid) return;
  unsigned xs[3], ys[3];
  neighbours(xs, ys, a, n.x, n.row);
  const size_t zo = (size_t)z * (size_t)a.plane;
  // radius 1: the mirror image of a plane beyond a wall is the wall plane itself
  const R* p0 = static_cast<const R*>(a.fd_psi) + zo;
  const R* pm = z > 0 ? p0 - a.plane : p0;
  const R* pp = z + 1 < a.nz ? p0 + a.plane : p0;
  R d[Q / 2];
#pragma unroll
  for (int k = 0; k < Q / 2; ++k) {
    const int l = 2 * k + 1;
    const R* hi = CZ(l) == 0 ? p0 : (CZ(l) > 0 ? pp : pm);
    const R* lo = CZ(l) == 0 ? p0 : (CZ(l) > 0 ? pm : pp);
    d[k] = ld_at(hi, xs[1 + CX(l)] + ys[1 + CY(l)]) - ld_at(lo, xs[1 - CX(l)] + ys[1 - CY(l)]);
  }
  R A[3];
  pair_gradient<R>(d, A[0], A[1], A[2]);
  const KPar<R>& kp = kpar<R>(a);
  const R rv = ld_at(static_cast<const R*>(a.fd_rho) + zo, n.i);
  const R j[3] = {ld_at(static_cast<const R*>(a.fd_j[0]) + zo, n.i), ld_at(static_cast<const R*>(a.fd_j[1]) + zo, n.i),
                  ld_at(static_cast<const R*>(a.fd_j[2]) + zo, n.i)};
  const R rho = F64 ? rv : kp.rho0 + rv;
  R inv;
  if constexpr (F64) inv = ld_at(static_cast<const R*>(a.fd_inv) + zo, n.i);
  else inv = recip(rho);
  const R mg = split_mg<R, VDW>(ld_at(p0, n.i), kp);              // F = mg A + rho g_z z
  const R mi = mg * inv;
  const R mu = R(0.5) * mi, mv = split_mv(mi, kp);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const R ji = j[k] * inv;
    st_at(static_cast<R*>(a.fd_u[k]) + zo, n.i, mu * A[k] + (k == 2 ? ji + kp.gz_u : ji));
    if (!F64 && a.fd_v[k] == nullptr) continue;       // 16-bit storage
    if constexpr (GUO) st_at(static_cast<R*>(a.fd_v[k]) + zo, n.i, k == 2 ? mg * A[k] + rho * kp.g_z : mg * A[k]);
    else st_at(static_cast<R*>(a.fd_v[k]) + zo, n.i, mv * A[k] + (k == 2 ? ji + kp.gz_v : ji));
  }
  if constexpr (F64) {
    if (a.adj_m != nullptr) {
#pragma unroll
      for (int k = 0; k < 3; ++k) st_at(a.adj_m + (MF_AX + k) * (size_t)a.N + zo, n.i, A[k] * (1.0 / 12.0));
    }
  }
}

// Resident 256-thread CTAs per SM that the collision's registers allow. FP32: 64 registers (4 CTAs;
// 256^3 boiling cell 0.84 ms against 0.90 with 3 and 0.97 with 2); 16-bit 80 (3); FP64 128 (2).
template <class S, int MODE> constexpr int split_mb() {
  if (MODE == MODE_MOMENTS) return sizeof(S) == 8 ? 3 : 4;    // holds one lattice only
  return sizeof(S) == 4 ? 4 : (sizeof(S) == 2 ? 3 : 2);
}

// whether a moments pass needs the velocities (an exported component or the diagnostics)
__host__ __device__ __forceinline__ bool wants_velocity(const KArgs& a) {
  return a.ux_out || a.uy_out || a.uz_out || a.part;
}

// MODE_MOMENTS: the fields of the state read instead of the collision; DIAG modes: the partials of
// the state read, one set per CTA.
template <class S, int VAR, int MODE, int NT>
__global__ void __launch_bounds__(NT, split_mb<S, MODE>() * 256 / NT) split_collide_kernel(const KArgs a, int nb) {
  using R = typename Store<S>::R;
  constexpr bool GUO = (VAR & VAR_GUO) != 0, VDW = (VAR & VAR_VDW) != 0, F64 = sizeof(R) == 8;
  constexpr bool COLLIDE = MODE != MODE_MOMENTS, DIAG = MODE != MODE_STEP;
  constexpr int NW = NT / 32;
  const int z = (int)blockIdx.x / nb;
  const NodePos n = node_at(a, (blockIdx.x - (unsigned)(z * nb)) * NT + threadIdx.x);
  wait_for_predecessor();
  const size_t N = (size_t)a.N, plane = (size_t)a.plane, zo = (size_t)z * plane;
  const KPar<R>& kp = kpar<R>(a);
  const unsigned o = n.i;
  DiagTerms<R> dt;
  if (n.valid) {
    const S* fin = static_cast<const S*>(a.fin);
    const S* gin = static_cast<const S*>(a.gin);
    R g[Q], f[Q];
    unsigned xs[3], ys[3];
    neighbours(xs, ys, a, n.x, n.row);
    split_pull<S, R>(g, gin, N, plane, a.nz, z, xs, ys);
    if constexpr (COLLIDE) split_pull<S, R>(f, fin, N, plane, a.nz, z, xs, ys);
    const R* pux = static_cast<const R*>(a.fd_u[0]) + zo;
    const R* puy = static_cast<const R*>(a.fd_u[1]) + zo;
    const R* puz = static_cast<const R*>(a.fd_u[2]) + zo;
    const R rv = ld_at(static_cast<const R*>(a.fd_rho) + zo, o);
    // a moments pass that asks for rho and T only has no velocities formed
    const bool need_u = COLLIDE || wants_velocity(a);
    const R ux = need_u ? ld_at(pux, o) : R(0), uy = need_u ? ld_at(puy, o) : R(0), uz = need_u ? ld_at(puz, o) : R(0);
    R inv;
    if constexpr (F64) inv = ld_at(static_cast<const R*>(a.fd_inv) + zo, o);
    if (z == 0 || z == a.nz - 1)
      g_wall_rule<R>(g, split_wall_density<S, R>(fin, N, zo + o), z, a.nz, kp.rho0, kp.T0, kp.T_d, kp.T_u, kp.lam);
    const R rho = F64 ? rv : kp.rho0 + rv;
    const R drho = F64 ? rv - kp.rho0 : rv;
    if constexpr (!F64) inv = recip(rho);
    R dE = g[0];
#pragma unroll
    for (int l = 1; l < Q; ++l) dE = dE + g[l];
    const R E = kp.E0 + dE;
    const R T = E * inv;            // the plain step needs it for the adjoint's fields only
    if constexpr (DIAG) {
      if (a.part != nullptr) dt.template take<VDW>(a, rho, inv, T, E, ux, uy, uz);
    }
    if constexpr (COLLIDE) {
      const R uzp = z + 1 < a.nz ? ld_at(puz + plane, o) : -uz;
      const R uzm = z > 0 ? ld_at(puz - plane, o) : -uz;
      // 2 div(u)
      const R D2 = ((ld_at(pux, xs[2] + ys[1]) - ld_at(pux, xs[0] + ys[1])) +
                    (ld_at(puy, xs[1] + ys[2]) - ld_at(puy, xs[1] + ys[0]))) + (uzp - uzm);
      // u' (Guo forcing: F) as the velocity pass formed it. 16-bit storage: from u = (j + F/2)/rho and j
      // of the pulled f, which saves writing and reading three fields (6 % of a step). That costs
      // 2^-24 |u| of F tau/rho; its populations are rounded to 2^-12, FP32's are not.
      R w[3];
      if constexpr (sizeof(S) != 2) {
#pragma unroll
        for (int k = 0; k < 3; ++k) w[k] = ld_at(static_cast<const R*>(a.fd_v[k]) + zo, o);
      } else {
        R dr, j[3];
        pair_moments<R>(f, dr, j[0], j[1], j[2]);
        const R u[3] = {ux, uy, uz};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const R ji = j[k] * inv;
          w[k] = GUO ? R(2) * (rho * u[k] - j[k]) : ji + split_mv(R(2) * (u[k] - ji), kp);   // u - j/rho = F/(2 rho)
        }
      }
      S* fo = static_cast<S*>(a.fout) + zo;
      S* go = static_cast<S*>(a.gout) + zo;
      R lrf[3] = {R(0), R(0), R(0)}, lrg[3] = {R(0), R(0), R(0)};
      auto put = [&](S* base, int l, R v) {
        Store<S>::st(reinterpret_cast<S*>(reinterpret_cast<char*>(base + l * N) + (size_t)(o * (unsigned)sizeof(S))), v);
      };
      if constexpr (IsLoc<S>::v) {
        float a1, a2, b1, b2;
        loc_refs_of<S>(drho, dE, T - kp.T0, kp.lam, a1, a2, b1, b2);
        lrf[0] = 12.0f * (a1 - a2); lrf[1] = a1; lrf[2] = a2;
        lrg[0] = 12.0f * (b1 - b2); lrg[1] = b1; lrg[2] = b2;
        put(fo, Q, a1); put(fo, Q + 1, a2); put(go, Q, b1); put(go, Q + 1, b2);
      }
      if constexpr (F64) {
        if (a.adj_m != nullptr) {
          st_at(a.adj_m + MF_T * N + zo, o, T);
          st_at(a.adj_m + MF_D * N + zo, o, 0.5 * D2);
        }
      }
      relax_g<R>(kp, E, dE, drho, inv, D2, ux, uy, uz, [&](int l) { return g[l]; },
                 [&](int l, R v) { put(go, l, IsLoc<S>::v ? v - lrg[CSQ(l)] : v); });
      relax_f<R, GUO>(kp, rho, drho, dE, ux, uy, uz, w, [&](int l) { return f[l]; },
                      [&](int l, R v) { put(fo, l, IsLoc<S>::v ? v - lrf[CSQ(l)] : v); });
    } else {
      if (a.rho_out) st_at(a.rho_out + zo, o, double(rho));
      if (a.ux_out) st_at(a.ux_out + zo, o, double(ux));
      if (a.uy_out) st_at(a.uy_out + zo, o, double(uy));
      if (a.uz_out) st_at(a.uz_out + zo, o, double(uz));
      if (a.T_out) st_at(a.T_out + zo, o, double(T));
    }
  }
  if constexpr (DIAG) {
    if (a.part != nullptr) {
      __shared__ R red[7][NW];
      dt.template reduce<NW>(red, threadIdx.x >> 5, threadIdx.x & 31);
      __syncthreads();
      if (threadIdx.x < 32) diag_combine<R, NW>(red, (int)threadIdx.x, a.part + (size_t)blockIdx.x * NPART);
    }
  }
}

}  // namespace tlbm
