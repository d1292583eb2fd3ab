// lb_march2.cuh -- the march of lb_march.cuh for 16-bit deviations with two x-neighbours per thread.
//
// With 2-byte populations the march is bound by its instructions (1133 a node, 70 % of the issue slots),
// half of them addresses, conversions and stores that a pair of neighbours can share: populations
// without an x shift are pulled, kept and stored as 4-byte words, psi and the velocities are read and
// written in pairs, and a 64-wide tile recomputes fewer ring nodes. For even nx (a pair never crosses
// the periodic edge and every word is aligned) and the paper's scheme; everything else takes the one-node
// march. 869 instructions a node; FP16 256^3 boiling cell 722 -> 613 us a step, 512^3 5.58 -> 4.92 ms,
// 128^3 105 -> 86 us.
#pragma once
#include "lb_march.cuh"

namespace tlbm {

template <class S> struct Pair16;   // two 16-bit values in a word
template <> struct Pair16<__half> {
  static __device__ __forceinline__ float one(unsigned short v) { return __half2float(__ushort_as_half(v)); }
  static __device__ __forceinline__ float lo(uint32_t w) { return one((unsigned short)(w & 0xffffu)); }
  static __device__ __forceinline__ float hi(uint32_t w) { return one((unsigned short)(w >> 16)); }
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
};
template <> struct Pair16<__nv_bfloat16> {
  static __device__ __forceinline__ float one(unsigned short v) { return __uint_as_float((uint32_t)v << 16); }
  static __device__ __forceinline__ float lo(uint32_t w) { return __uint_as_float(w << 16); }
  static __device__ __forceinline__ float hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
};

template <int TY> struct March2Geo {
  static constexpr int TX = 64, RX = TX + 4, RY = TY + 4, NP = RX / 2 * RY;      // pairs of the ring
  static constexpr int NM = (NP + 31) / 32 * 32, NC = 32 * TY, NT = NM + NC;     // threads of either group
  static constexpr int NR = RX * RY + 4, NN = TX * TY, DF = 4;                   // ring nodes (padded), tile nodes
  // psi [4][NR], drho, j, 1/rho of a plane until its U [2][5][2 NM], ux, uy [3][2][NR], u', drho, 1/rho
  // [3][5][NN], uz [3][NN], f [DF][Q][NN / 2] words
  static constexpr size_t floats = 4 * NR + 20 * NM + 6 * NR + 15 * NN + 3 * NN;
  static constexpr size_t smem = 4 * floats + 4 * (size_t)(DF * Q * (NN / 2));
};

__device__ __forceinline__ uint32_t ld_here32(const char* p) {
  uint32_t v; asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p)); return v;
}

// What a pair pulls: a word where the source pair is aligned (c_x = 0), else two values
template <class S> struct PairRaw {
  uint32_t w[Q];
  unsigned short a[Q], b[Q];
  // v[dx][dy]: byte offsets of columns x-1, x, x+2 (x even, the pair's first) in rows y-1, y, y+1
  __device__ __forceinline__ void request(const char* const (&src)[Q], const KArgs& ka, int z, const unsigned (&v)[3][3]) {
    if (z > 0 && z < ka.nz - 1) {
#pragma unroll
      for (int l = 0; l < Q; ++l) {
        const int r = 1 - CY(l);
        if (CX(l) == 0) w[l] = ld_here32(src[l] + (size_t)v[1][r]);
        else if (CX(l) > 0) { a[l] = ld_here16(src[l] + (size_t)v[0][r]); b[l] = ld_here16(src[l] + (size_t)v[1][r]); }
        else { a[l] = ld_here16(src[l] + (size_t)v[1][r] + 2); b[l] = ld_here16(src[l] + (size_t)v[2][r]); }
      }
    } else {
      const long long pb = (long long)ka.plane * 2;
#pragma unroll
      for (int l = 0; l < Q; ++l) {
        const int r = 1 - CY(l);
        // through a wall: the bounce-back source, population opp(l) of the node itself
        const bool through = (CZ(l) > 0 && z == 0) || (CZ(l) < 0 && z == ka.nz - 1);
        const char* p = through ? src[OPP(l)] + CZ(OPP(l)) * pb + (size_t)v[1][1] : src[l] + (size_t)v[1][r];
        if (CX(l) == 0) w[l] = ld_here32(p);
        else if (CX(l) > 0) {
          a[l] = ld_here16(through ? p : src[l] + (size_t)v[0][r]);
          b[l] = ld_here16(through ? p + 2 : p);
        } else {
          a[l] = ld_here16(through ? p : p + 2);
          b[l] = ld_here16(through ? p + 2 : src[l] + (size_t)v[2][r]);
        }
      }
    }
  }
  __device__ __forceinline__ uint32_t word(int l) const { return CX(l) == 0 ? w[l] : ((uint32_t)a[l] | ((uint32_t)b[l] << 16)); }
};

__device__ __forceinline__ void pair_offsets(unsigned (&v)[3][3], const KArgs& a, int x, int y, size_t zo) {
  const unsigned nx = (unsigned)a.nx;
  const unsigned xs[3] = {(unsigned)(x == 0 ? nx - 1 : x - 1), (unsigned)x, (unsigned)x + 2 == nx ? 0u : (unsigned)x + 2};
  unsigned dummy[3], ys[3];
  neighbours(dummy, ys, a, 0u, (unsigned)y * nx);
#pragma unroll
  for (int dx = 0; dx < 3; ++dx)
#pragma unroll
    for (int dy = 0; dy < 3; ++dy) v[dx][dy] = (unsigned)((zo + xs[dx] + ys[dy]) * 2u);
}
__device__ __forceinline__ void pair_advance(unsigned (&v)[3][3], unsigned bytes) {
#pragma unroll
  for (int dx = 0; dx < 3; ++dx)
#pragma unroll
    for (int dy = 0; dy < 3; ++dy) v[dx][dy] += bytes;
}

// DIAG: a step that also forms the diagnostics partials of the state it reads. The step itself is the same
// operation for operation, so a sample leaves the populations as they are without it. FP16 256^3: 657 us
// with its finalisation, 612 without a sample (1219 when sampling steps took the one-node march).
template <class S, int TY, bool DIAG>
__global__ void __launch_bounds__(March2Geo<TY>::NT, 1) split_march2_kernel(const KArgs a, const MarchArgs b) {
  using R = float;
  using GE = March2Geo<TY>;
  using P2 = Pair16<S>;
  constexpr int NM = GE::NM, NT = GE::NT, NR = GE::NR, NN = GE::NN, RX = GE::RX, DF = GE::DF;
  constexpr int BAR_M = 1, BAR_R = 2, BAR_D = 4, BAR_C = 6;      // as in split_march_kernel
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R* psi_s = reinterpret_cast<R*>(smem_raw);       // [4][NR], two floats before the first row of a plane
  R* st_s = psi_s + 4 * NR;                        // [2][5][2 NM]: drho, j, 1/rho, by thread
  R* uxy_s = st_s + 20 * NM;                       // [3][2][NR]
  R* w_s = uxy_s + 6 * NR;                         // [3][5][NN]: u', drho, 1/rho
  R* uz_s = w_s + 15 * NN;                         // [3][NN]
  uint32_t* fc_s = reinterpret_cast<uint32_t*>(uz_s + 3 * NN);   // [DF][Q][NN / 2]

  const int x0 = ((int)blockIdx.x % b.tiles_x) * GE::TX, y0 = ((int)blockIdx.x / b.tiles_x) * TY;
  const int nz = a.nz, z0 = (int)blockIdx.y * b.zc, z1 = min(z0 + b.zc, nz);
  const size_t plane = (size_t)a.plane;
  const unsigned step = (unsigned)(plane * sizeof(S));
  const KPar<R>& kp = a.pf;
  const int ps = z0 >= 2 ? z0 - 2 : 0, pe = z1 + 1;
  auto st2 = [](R* p, R x, R y) { *reinterpret_cast<float2*>(p) = make_float2(x, y); };
  auto ld2 = [](const R* p) { return *reinterpret_cast<const float2*>(p); };

  if ((int)threadIdx.x < NM) {
    const int t = (int)threadIdx.x, rx = 2 * (t % (RX / 2)), ry = t / (RX / 2);
    const bool in_r = t < GE::NP;
    const bool in_u = in_r && ry >= 1 && ry <= TY + 2;          // its outermost columns are not read
    const bool in_c = in_r && rx >= 2 && rx <= 65 && ry >= 2 && ry <= TY + 1;
    const int h = 2 + ry * RX + rx;                             // in the ring's planes
    const int ct = (ry - 2) * GE::TX + rx - 2;
    unsigned m[3][3];
    pair_offsets(m, a, wrapi(x0 + rx - 2, a.nx), wrapi(y0 + ry - 2, a.ny), (size_t)ps * plane);
    PairRaw<S> raw;
    raw.request(b.fsrc, a, ps, m);
    int uslot = 2;            // slot of plane p-1 in the rings of three
    for (int p = ps; p <= pe; ++p) {
      if (p >= ps + 2) bar_sync(BAR_D + (p & 1), NT);
      if (p < nz) {
        uint32_t fw[Q];
#pragma unroll
        for (int l = 0; l < Q; ++l) fw[l] = raw.word(l);
        if (in_c) {
          uint32_t* fc = fc_s + (size_t)(p & (DF - 1)) * (Q * NN / 2) + ct / 2;
#pragma unroll
          for (int l = 0; l < Q; ++l) fc[l * (NN / 2)] = fw[l];
        }
        R psi[2], drho[2], j[3][2], inv[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          R f[Q];
#pragma unroll
          for (int l = 0; l < Q; ++l) f[l] = k == 0 ? P2::lo(fw[l]) : P2::hi(fw[l]);
          pair_moments<R>(f, drho[k], j[0][k], j[1][k], j[2][k]);
          const R rho = kp.rho0 + drho[k];
          inv[k] = recip(rho);
          psi[k] = split_psi<R, false>(rho, drho[k], inv[k], kp);
        }
        R* s = st_s + (p & 1) * (10 * NM) + 2 * t;
        st2(s, drho[0], drho[1]); st2(s + 8 * NM, inv[0], inv[1]);
#pragma unroll
        for (int c = 0; c < 3; ++c) st2(s + (2 + 2 * c) * NM, j[c][0], j[c][1]);
        if (in_r) st2(psi_s + (p & 3) * NR + h, psi[0], psi[1]);
        if (p + 1 < nz && p < pe) {
          pair_advance(m, step);
          raw.request(b.fsrc, a, p + 1, m);
        }
      }
      bar_sync(BAR_M, NM);
      const int q = p - 1;
      if (in_u && q >= ps && q < nz && q >= z0 - 1) {
        const R* s0 = psi_s + (q & 3) * NR + h;
        const R* sm = q > 0 ? psi_s + ((q - 1) & 3) * NR + h : s0;
        const R* sp = q + 1 < nz ? psi_s + ((q + 1) & 3) * NR + h : s0;
        // columns x-1 .. x+2 of a row
        auto row = [&](const R* s, int off, R (&c)[4]) {
          c[0] = s[off - 1];
          const float2 v = ld2(s + off);
          c[1] = v.x; c[2] = v.y;
          c[3] = s[off + 2];
        };
        R c0[4], yp[4], ym[4], zp[4], zm[4];
        row(s0, 0, c0); row(s0, RX, yp); row(s0, -RX, ym); row(sp, 0, zp); row(sm, 0, zm);
        const float2 pp = ld2(sp + RX), mm = ld2(sm - RX), mp = ld2(sm + RX), pm = ld2(sp - RX);   // (z, y) signs
        R A[3][2], mi[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const R d[Q / 2] = {c0[k + 2] - c0[k],     yp[k + 1] - ym[k + 1], zp[k + 1] - zm[k + 1],
                              yp[k + 2] - ym[k],     ym[k + 2] - yp[k],     zp[k + 2] - zm[k],
                              zm[k + 2] - zp[k],     (k == 0 ? pp.x - mm.x : pp.y - mm.y),
                              (k == 0 ? mp.x - pm.x : mp.y - pm.y)};
          pair_gradient<R>(d, A[0][k], A[1][k], A[2][k]);
          mi[k] = split_mg<R, false>(c0[k + 1], kp);
        }
        const R* s = st_s + (q & 1) * (10 * NM) + 2 * t;
        const float2 dr = ld2(s), iv = ld2(s + 8 * NM);
        mi[0] *= iv.x; mi[1] *= iv.y;
        R* us = uxy_s + uslot * (2 * NR) + h;
        R* w = w_s + uslot * (5 * NN) + ct;
        const R mv[2] = {split_mv(mi[0], kp), split_mv(mi[1], kp)};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 j = ld2(s + (2 + 2 * c) * NM);
          const R g[2] = {j.x * iv.x, j.y * iv.y};
          const R gu = c == 2 ? kp.gz_u : R(0), gv = c == 2 ? kp.gz_v : R(0);
          const R u0 = (R(0.5) * mi[0]) * A[c][0] + (g[0] + gu), u1 = (R(0.5) * mi[1]) * A[c][1] + (g[1] + gu);
          if (c < 2) st2(us + c * NR, u0, u1);
          if (in_c) {
            if (c == 2) st2(uz_s + uslot * NN + ct, u0, u1);
            st2(w + c * NN, mv[0] * A[c][0] + (g[0] + gv), mv[1] * A[c][1] + (g[1] + gv));
          }
        }
        if (in_c) { st2(w + 3 * NN, dr.x, dr.y); st2(w + 4 * NN, iv.x, iv.y); }
      }
      bar_arrive(BAR_R + (p & 1), NT);
      uslot = uslot == 2 ? 0 : uslot + 1;
    }
  } else {
    __shared__ R red[DIAG ? 2 : 1][7][DIAG ? TY : 1];
    const int t = (int)threadIdx.x - NM, px = t & 31, ty = t >> 5;
    const int x = x0 + 2 * px, y = y0 + ty;
    const bool valid = x < a.nx && y < a.ny;
    const int h = 2 + (ty + 2) * RX + 2 * px + 2, ct = ty * GE::TX + 2 * px;
    unsigned m[3][3];
    pair_offsets(m, a, valid ? x : 0, valid ? y : 0, (size_t)z0 * plane);
    PairRaw<S> raw;
    unsigned own = m[1][1];
    raw.request(b.gsrc, a, z0, m);
    float2 uzm = make_float2(0.0f, 0.0f), uz = uzm, uzp = uzm;
    int uslot = 2;            // slot of plane p-1; plane p-2 has the one before
    for (int p = ps; p <= pe; ++p) {
      bar_sync(BAR_R + (p & 1), NT);
      const int z = p - 2;
      if constexpr (DIAG) {
        // the partials of the plane before are complete
        if (z - 1 >= z0 && ty == 0)
          diag_combine<R, TY>(red[(z - 1) & 1], px, a.part + ((size_t)(z - 1) * gridDim.x + blockIdx.x) * NPART);
      }
      DiagTerms<R> dt[2];
      uzm = uz; uz = uzp;
      if (p >= 1 && p - 1 < nz) uzp = ld2(uz_s + uslot * NN + ct);
      const int zslot = uslot == 0 ? 2 : uslot - 1;
      uslot = uslot == 2 ? 0 : uslot + 1;
      if (z >= z0 && valid) {
        const R* us = uxy_s + zslot * (2 * NR) + h;
        const R* w = w_s + zslot * (5 * NN) + ct;
        uint32_t gw[Q];
#pragma unroll
        for (int l = 0; l < Q; ++l) gw[l] = raw.word(l);
        // wall planes: the thermal wall rule on the populations that come through the wall, with the
        // wall nodes' density deviations (sums of their own stored f)
        const bool wallz = z == 0 || z == nz - 1;
        R dp[2] = {R(0), R(0)};
        if (wallz) {
#pragma unroll 1
          for (int l = 0; l < Q; ++l) {
            const uint32_t v = ld_here32(static_cast<const char*>(a.fin) + (size_t)l * (size_t)a.N * 2u + (size_t)own);
            dp[0] += P2::lo(v); dp[1] += P2::hi(v);
          }
        }
        auto gin = [&](int k, int l, bool wall) -> R {
          const R v = k == 0 ? P2::lo(gw[l]) : P2::hi(gw[l]);
          if (!wall || CZ(l) == 0) return v;
          const R e = CZ(l) > 0 ? (z == 0 ? R(2) * wall_even_dev<R>(l, dp[k], kp.rho0, kp.T0, kp.T_d, kp.lam) - v : v)
                                : (z == nz - 1 ? R(2) * wall_even_dev<R>(l, dp[k], kp.rho0, kp.T0, kp.T_u, kp.lam) - v : v);
          return e;
        };
        const float2 dr = ld2(w + 3 * NN), iv = ld2(w + 4 * NN), ux = ld2(us), uy = ld2(us + NR);
        const float2 yp = ld2(us + NR + RX), ym = ld2(us + NR - RX);
        const R xm = us[-1], xp = us[2];
        const R D2[2] = {((ux.y - xm) + (yp.x - ym.x)) + ((z + 1 < nz ? uzp.x : -uz.x) - (z > 0 ? uzm.x : -uz.x)),
                         ((xp - ux.x) + (yp.y - ym.y)) + ((z + 1 < nz ? uzp.y : -uz.y) - (z > 0 ? uzm.y : -uz.y))};
        const R drho[2] = {dr.x, dr.y}, inv[2] = {iv.x, iv.y};
        const R u[3][2] = {{ux.x, ux.y}, {uy.x, uy.y}, {uz.x, uz.y}};
        R dE[2];
        // the two nodes' relaxations side by side: every population of the pair is one word
        R A[2][3], B[2][3], C[2][3];      // per class: even constant, coefficient of (c.v)^2, of (c.v)
        auto out = [&](char* const (&dst)[Q + 2], R om1, const R (&v)[3][2], auto in) {
          auto put = [&](int l, R s0, R s1) {
            *reinterpret_cast<uint32_t*>(dst[l] + (size_t)own) = P2::pack(s0, s1);
          };
          put(0, fma_rn(om1, in(0, 0), A[0][0]), fma_rn(om1, in(1, 0), A[1][0]));
#pragma unroll
          for (int l = 1; l < Q; l += 2) {
            R s[2][2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const R cv = cdot<R>(l, v[0][k], v[1][k], v[2][k]);
              const R ev = fma_rn(B[k][CLS(l)] * cv, cv, A[k][CLS(l)]);
              s[0][k] = fma_rn(C[k][CLS(l)], cv, fma_rn(om1, in(k, l), ev));
              s[1][k] = fma_rn(-C[k][CLS(l)], cv, fma_rn(om1, in(k, OPP(l)), ev));
            }
            put(l, s[0][0], s[0][1]);
            put(OPP(l), s[1][0], s[1][1]);
          }
        };
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          R e;
          if (wallz) {
            e = gin(k, 0, true);
#pragma unroll
            for (int l = 1; l < Q; ++l) e = e + gin(k, l, true);
          } else {
            e = gin(k, 0, false);
#pragma unroll
            for (int l = 1; l < Q; ++l) e = e + gin(k, l, false);
          }
          dE[k] = e;
          const R E = kp.E0 + e;
          if constexpr (DIAG)
            dt[k].template take<false>(a, kp.rho0 + drho[k], inv[k], E * inv[k], E, u[0][k], u[1][k], u[2][k]);
          const R uu = u[0][k] * u[0][k] + u[1][k] * u[1][k] + u[2][k] * u[2][k];
          const R b0 = e - E * (R(1.5) * uu + D2[k] * kp.src);
          const R tg = kp.lam45 * ((e - kp.T0 * drho[k]) * inv[k]) - R(1.5) * e;
          const R e3[3] = {b0 - tg, b0, b0 + tg};
#pragma unroll
          for (int c = 0; c < 3; ++c) A[k][c] = mul2(kp.go[c], kp.go_lo[c], e3[c]);
#pragma unroll
          for (int c = 1; c < 3; ++c) { B[k][c] = kp.gq[c] * E; C[k][c] = mul2(kp.gs[c], kp.gs_lo[c], E); }
        }
        if (wallz) out(b.gdst, kp.omk1, u, [&](int k, int l) { return gin(k, l, true); });
        else out(b.gdst, kp.omk1, u, [&](int k, int l) { return gin(k, l, false); });
        if (z + 1 < z1) {
          pair_advance(m, step);
          raw.request(b.gsrc, a, z + 1, m);
        }
        const float2 w0 = ld2(w), w1 = ld2(w + NN), w2 = ld2(w + 2 * NN);
        const R v[3][2] = {{w0.x, w0.y}, {w1.x, w1.y}, {w2.x, w2.y}};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const R rho = kp.rho0 + drho[k];
          const R vv = v[0][k] * v[0][k] + v[1][k] * v[1][k] + v[2][k] * v[2][k];
          const R a0 = drho[k] - (R(1.5) * rho) * vv;
          const R th = R(4.5) * dE[k] - R(1.5) * drho[k];
          const R e3[3] = {a0 - th, a0, a0 + th};
#pragma unroll
          for (int c = 0; c < 3; ++c) A[k][c] = mul2(kp.fo[c], kp.fo_lo[c], e3[c]);
#pragma unroll
          for (int c = 1; c < 3; ++c) { B[k][c] = kp.fq[c] * rho; C[k][c] = mul2(kp.fs[c], kp.fs_lo[c], rho); }
        }
        const uint32_t* fc = fc_s + (size_t)(z & (DF - 1)) * (Q * NN / 2) + ct / 2;
        out(b.fdst, kp.om1, v, [&](int k, int l) { return k == 0 ? P2::lo(fc[l * (NN / 2)]) : P2::hi(fc[l * (NN / 2)]); });
        own += step;
      }
      if constexpr (DIAG) {
        if (z >= z0) {
          dt[0].add(dt[1]);
          dt[0].template reduce<TY, true>(red[z & 1], ty, px);
        }
      }
      if (p + 2 <= pe) bar_arrive(BAR_D + (p & 1), NT);
    }
    if constexpr (DIAG) {
      bar_sync(BAR_C, GE::NC);
      if (ty == 0) diag_combine<R, TY>(red[(z1 - 1) & 1], px, a.part + ((size_t)(z1 - 1) * gridDim.x + blockIdx.x) * NPART);
    }
  }
}

}  // namespace tlbm
