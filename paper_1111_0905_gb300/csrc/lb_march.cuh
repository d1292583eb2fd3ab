// lb_march.cuh -- the time step in one launch, for the FP32-compute forms on cells that fill the GPU.
//
// A CTA marches up in z over a 32 x TY tile with two groups of warps. The first has one thread per
// node of the tile's radius-2 ring: it pulls f of plane p (requested one plane ahead into
// registers), writes psi and the tile's f to shared memory (stage M) and, behind a barrier of its
// own, forms u of plane p-1 on the radius-1 ring (U). The second group has one thread per tile node
// and collides plane p-2 (C), its g requested one plane ahead. The groups meet at named barriers
// only and may drift apart by one plane, so M and U of one plane run beside C of another.
// HBM sees the populations once each way; f is pulled once per ring node (no second pull in C).
//
// Why two groups: the tile march (lb_kernels.cuh) runs its stages one after the other in the same 16
// warps, each blocked on its own loads; here every load is requested a plane before its use and the
// stages of different planes overlap. FP32 256^3 boiling cell 1.279 -> 0.944 ms a step, 5.4 TB/s of DRAM
// traffic (81 % of a copy), 512^3 9.88 -> 7.57 ms, 128^3 184 -> 126 us; leaving out any of its loads or
// stores shortens it by the bytes' share: memory traffic bounds it. 16-bit storage: instructions (issue
// slots 59-70 % busy); local references 256^3 1.544 -> 1.19 ms.
#pragma once
#include "lb_split.cuh"

namespace tlbm {

// Where the populations are read and written, as bytes: per population the start of its lattice
// plane -c_lz relative to the node's own plane (pull source) and of its lattice (store). The local
// references are slots 19 and 20 of either lattice, read from fdst's counterparts fref and gref.
struct MarchArgs {
  const char* fsrc[Q]; const char* gsrc[Q];
  char* fdst[Q + 2]; char* gdst[Q + 2];
  const char* fref[2]; const char* gref[2];
  int tiles_x, zc;
};

template <class S, int TY> struct MarchGeo {
  using FC = typename std::conditional<IsLoc<S>::v, float, S>::type;    // the tile's f as kept
  static constexpr int RX = 36, RY = TY + 4, NR = RX * RY, NM = (NR + 31) / 32 * 32, NC = 32 * TY, NT = NM + NC;
  static constexpr int DF = 4;   // planes of f kept: C of plane p-2 may still run when M writes plane p+1
  // psi [4][NM], ux, uy [3][2][NM], u', drho, 1/rho [3][5][NC], uz [3][NC], f [DF][Q][NC]
  static constexpr size_t floats = 4 * NM + 6 * NM + 15 * NC + 3 * NC;
  // local references: windows of four planes of 4-byte words (slot 19 low, slot 20 high half), of f on the ring's
  // neighbourhood (radius 3 of the tile), of g on the tile's (radius 1)
  static constexpr int FWX = 38, FW = FWX * (TY + 6), GWX = 34, GW = GWX * (TY + 2);
  static constexpr size_t smem = 4 * floats + sizeof(FC) * DF * Q * NC + (IsLoc<S>::v ? 16 * (FW + GW) : 0);
  // Ring node of thread t of the first group (the padding threads of its last warp repeat the last node;
  // nobody reads what they form), and the node's word in a plane of f's window. A node reads the words
  // of its eight neighbours in the planes below and above as well.
  static __host__ __device__ constexpr int node(int t) { return t < NR ? t : NR - 1; }
  static __host__ __device__ constexpr int fword(int t) { return (node(t) / RX + 1) * FWX + node(t) % RX + 1; }
  static constexpr bool in_window() {
    for (int t = 0; t < NM; ++t)
      if (fword(t) - FWX - 1 < 0 || fword(t) + FWX + 1 >= FW) return false;
    return true;
  }
};

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// Byte offsets of the nine (dx, dy) neighbours of a node, advanced plane by plane; with them a pull
// is one 32-bit offset on a base that does not change over the march. (With element indices instead FP16
// storage ran 10 % slower.)
template <class S> struct MarchPos {
  unsigned v[3][3];
  __device__ __forceinline__ void set(const unsigned (&xs)[3], const unsigned (&ys)[3], size_t zo) {
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) v[dx][dy] = (unsigned)((zo + xs[dx] + ys[dy]) * sizeof(S));
  }
  __device__ __forceinline__ void advance(unsigned bytes) {
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) v[dx][dy] += bytes;
  }
};

// Loads that stay where they are written: a plane is requested ahead of its use, and the compiler
// would otherwise sink the loads to it.
__device__ __forceinline__ float ld_here(const char* p, float) {
  float v; asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p)); return v;
}
__device__ __forceinline__ unsigned short ld_here16(const char* p) {
  unsigned short v; asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p)); return v;
}
__device__ __forceinline__ __half ld_here(const char* p, __half) { return __ushort_as_half(ld_here16(p)); }
__device__ __forceinline__ __nv_bfloat16 ld_here(const char* p, __nv_bfloat16) { return __ushort_as_bfloat16(ld_here16(p)); }
__device__ __forceinline__ half_loc ld_here(const char* p, half_loc) { half_loc h; h.h = __ushort_as_half(ld_here16(p)); return h; }

// The stored values that a node pulls, in flight or arrived
template <class S> struct MarchRaw {
  S v[Q];
  // request the node at m of plane z
  __device__ __forceinline__ void request(const char* const (&src)[Q], const KArgs& a, int z, const MarchPos<S>& m) {
    if (z > 0 && z < a.nz - 1) {
#pragma unroll
      for (int l = 0; l < Q; ++l) v[l] = ld_here(src[l] + (size_t)m.v[1 - CX(l)][1 - CY(l)], S());
    } else {
      // through a wall: the bounce-back source, population opp(l) of the node itself
      const long long pb = (long long)a.plane * (long long)sizeof(S);
#pragma unroll
      for (int l = 0; l < Q; ++l) {
        const bool through = (CZ(l) > 0 && z == 0) || (CZ(l) < 0 && z == a.nz - 1);
        const char* b = through ? src[OPP(l)] + CZ(OPP(l)) * pb : src[l];
        v[l] = ld_here(b + (size_t)(through ? m.v[1][1] : m.v[1 - CX(l)][1 - CY(l)]), S());
      }
    }
  }
  // the deviations; with local references from the window word i of plane z (rows of WX words)
  template <int WX, int WN>
  __device__ __forceinline__ void decode(float (&f)[Q], const uint32_t* win, int i, int z, int nz) const {
#pragma unroll
    for (int l = 0; l < Q; ++l) f[l] = cvt<S, float>(v[l]);
    if constexpr (IsLoc<S>::v) {
      const uint32_t* w0 = win + (z & 3) * WN + i;
      // a plane beyond a wall: the node's own word (the bounce-back source)
      const bool bot = z == 0, top = z == nz - 1;
      const uint32_t* wm = win + ((z - 1) & 3) * WN + i;
      const uint32_t* wp = win + ((z + 1) & 3) * WN + i;
      auto lo = [](uint32_t w) { return __half2float(__ushort_as_half((unsigned short)(w & 0xffffu))); };
      auto hi = [](uint32_t w) { return __half2float(__ushort_as_half((unsigned short)(w >> 16))); };
      f[0] += 12.0f * (lo(w0[0]) - hi(w0[0]));
#pragma unroll
      for (int l = 1; l < Q; ++l) {
        const int st = -(CY(l) * WX + CX(l));
        uint32_t w;
        if (CZ(l) == 0) w = w0[st];
        else if (CZ(l) > 0) w = bot ? w0[0] : wm[st];
        else w = top ? w0[0] : wp[st];
        f[l] += CSQ(l) == 1 ? lo(w) : hi(w);
      }
    }
  }
};

// Feeds a window of references, WX x WN/WX nodes from (x0, y0), by NTH threads (up to two nodes each):
// the references of a plane are requested an iteration before they are stored.
template <int WX, int WN, int NTH> struct RefFeed {
  unsigned off[2];
  unsigned short a[2], b[2];
  int t;
  __device__ __forceinline__ void set(const KArgs& ka, int thread, int x0, int y0) {
    static_assert(WN <= 2 * NTH, "two words per thread");
    t = thread;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = t + k * NTH;
      off[k] = 2u * ((unsigned)wrapi(y0 + i / WX, ka.ny) * (unsigned)ka.nx + (unsigned)wrapi(x0 + i % WX, ka.nx));
    }
  }
  __device__ __forceinline__ void request(const char* const (&ref)[2], size_t plane_bytes, int z) {
    const char* p0 = ref[0] + (size_t)z * plane_bytes;
    const char* p1 = ref[1] + (size_t)z * plane_bytes;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (t + k * NTH < WN) { a[k] = ld_here16(p0 + off[k]); b[k] = ld_here16(p1 + off[k]); }
    }
  }
  __device__ __forceinline__ void store(uint32_t* win, int z) const {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = t + k * NTH;
      if (i < WN) win[(z & 3) * WN + i] = (uint32_t)a[k] | ((uint32_t)b[k] << 16);
    }
  }
  // planes z-1 .. z+1 at once, and z+2 requested
  __device__ __forceinline__ void start(const char* const (&ref)[2], size_t plane_bytes, uint32_t* win, int z, int nz) {
    for (int q = z - 1; q <= z + 1; ++q) {
      if (q >= 0 && q < nz) { request(ref, plane_bytes, q); store(win, q); }
    }
    if (z + 2 < nz) request(ref, plane_bytes, z + 2);
  }
  // behind the use of planes z-1 .. z+1: plane z+2 into the window, z+3 requested
  __device__ __forceinline__ void next(const char* const (&ref)[2], size_t plane_bytes, uint32_t* win, int z, int nz) {
    if (z + 2 < nz) store(win, z + 2);
    if (z + 3 < nz) request(ref, plane_bytes, z + 3);
  }
};

template <class S, int VAR, int MODE, int TY>
__global__ void __launch_bounds__(MarchGeo<S, TY>::NT, 1) split_march_kernel(const KArgs a, const MarchArgs b) {
  using R = float;
  using GE = MarchGeo<S, TY>;
  using FC = typename GE::FC;
  constexpr bool GUO = (VAR & VAR_GUO) != 0, VDW = (VAR & VAR_VDW) != 0;
  constexpr bool COLLIDE = MODE != MODE_MOMENTS, DIAG = MODE != MODE_STEP;
  constexpr int NM = GE::NM, NC = GE::NC, NT = GE::NT, RX = GE::RX, DF = GE::DF;
  // named barriers: M to U; u of an iteration ready; C of an iteration done (two of each kind in turn)
  constexpr int BAR_M = 1, BAR_R = 2, BAR_D = 4, BAR_C = 6;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R* psi_s = reinterpret_cast<R*>(smem_raw);       // [4][NM]
  R* uxy_s = psi_s + 4 * NM;                       // [3][2][NM]
  R* w_s = uxy_s + 6 * NM;                         // [3][5][NC]: u' (Guo: F), drho, 1/rho
  R* uz_s = w_s + 15 * NC;                         // [3][NC]
  FC* fc_s = reinterpret_cast<FC*>(uz_s + 3 * NC); // [DF][Q][NC]
  uint32_t* fw_s = reinterpret_cast<uint32_t*>(fc_s + DF * Q * NC);   // [4][FW], local references only
  uint32_t* gw_s = fw_s + 4 * GE::FW;                                 // [4][GW]
  const size_t plane_bytes = (size_t)a.plane * sizeof(S);

  const int tile = (int)blockIdx.x;
  const int x0 = (tile % b.tiles_x) * 32, y0 = (tile / b.tiles_x) * TY;
  const int nz = a.nz, z0 = (int)blockIdx.y * b.zc, z1 = min(z0 + b.zc, nz);
  const size_t plane = (size_t)a.plane;
  const unsigned step = (unsigned)(plane * sizeof(S));
  const KPar<R>& kp = a.pf;
  // iteration p: M of plane p, U of p-1, C of p-2 (the planes beyond a wall are its mirror image and
  // not formed)
  const int ps = z0 >= 2 ? z0 - 2 : 0, pe = z1 + 1;

  if ((int)threadIdx.x < NM) {
    static_assert(GE::in_window(), "a word outside the plane of the window belongs to another plane");
    const int t = (int)threadIdx.x, rx = GE::node(t) % RX, ry = GE::node(t) / RX;
    const bool in_u = rx >= 1 && rx <= 34 && ry >= 1 && ry <= TY + 2;
    const bool in_c = rx >= 2 && rx <= 33 && ry >= 2 && ry <= TY + 1;
    const int ct = (ry - 2) * 32 + rx - 2;
    MarchPos<S> m;
    {
      unsigned xs[3], ys[3];
      neighbours(xs, ys, a, (unsigned)wrapi(x0 + rx - 2, a.nx), (unsigned)wrapi(y0 + ry - 2, a.ny) * (unsigned)a.nx);
      m.set(xs, ys, (size_t)ps * plane);
    }
    R inv1 = R(0), drho1 = R(0), jx1 = R(0), jy1 = R(0), jz1 = R(0);     // of the plane before
    MarchRaw<S> raw;
    raw.request(b.fsrc, a, ps, m);
    RefFeed<GE::FWX, GE::FW, NM> feed;
    if constexpr (IsLoc<S>::v) {
      feed.set(a, t, x0 - 3, y0 - 3);
      feed.start(b.fref, plane_bytes, fw_s, ps, nz);
      bar_sync(BAR_M, NM);
    }
    int uslot = 2;            // slot of plane p-1 in the rings of three
    for (int p = ps; p <= pe; ++p) {
      if (p >= ps + 2) bar_sync(BAR_D + (p & 1), NT);        // C of iteration p-2 is done
      R inv = R(0), drho = R(0), jx = R(0), jy = R(0), jz = R(0);
      if (p < nz) {
        R f[Q];
        raw.template decode<GE::FWX, GE::FW>(f, fw_s, GE::fword(t), p, nz);
        if (COLLIDE && in_c) {
          FC* fc = fc_s + (size_t)(p & (DF - 1)) * Q * NC + ct;
#pragma unroll
          for (int l = 0; l < Q; ++l) {
            if constexpr (IsLoc<S>::v) fc[l * NC] = f[l];
            else fc[l * NC] = raw.v[l];
          }
        }
        pair_moments<R>(f, drho, jx, jy, jz);
        const R rho = kp.rho0 + drho;
        inv = recip(rho);
        psi_s[(p & 3) * NM + t] = split_psi<R, VDW>(rho, drho, inv, kp);
        // behind the last use of f, so that its registers take the next request
        if (p + 1 < nz && p < pe) {
          m.advance(step);
          raw.request(b.fsrc, a, p + 1, m);
        }
        if constexpr (IsLoc<S>::v) feed.next(b.fref, plane_bytes, fw_s, p, nz);
      }
      bar_sync(BAR_M, NM);
      const int q = p - 1;
      if (in_u && q >= ps && q < nz && q >= z0 - 1) {
        const R* s0 = psi_s + (q & 3) * NM;
        const R* sm = q > 0 ? psi_s + ((q - 1) & 3) * NM : s0;
        const R* sp = q + 1 < nz ? psi_s + ((q + 1) & 3) * NM : s0;
        R d[Q / 2];
#pragma unroll
        for (int k = 0; k < Q / 2; ++k) {
          const int l = 2 * k + 1;
          const int st = CX(l) + CY(l) * RX;
          const R* hi = CZ(l) == 0 ? s0 : (CZ(l) > 0 ? sp : sm);
          const R* lo = CZ(l) == 0 ? s0 : (CZ(l) > 0 ? sm : sp);
          d[k] = hi[t + st] - lo[t - st];
        }
        R ax, ay, az;
        pair_gradient<R>(d, ax, ay, az);
        const R mg = split_mg<R, VDW>(s0[t], kp);
        const R mi = mg * inv1, mu = R(0.5) * mi, mv = split_mv(mi, kp);
        R* us = uxy_s + uslot * (2 * NM);
        us[t] = mu * ax + jx1 * inv1;
        us[NM + t] = mu * ay + jy1 * inv1;
        if (in_c) {
          R* w = w_s + uslot * (5 * NC) + ct;
          uz_s[uslot * NC + ct] = mu * az + (jz1 * inv1 + kp.gz_u);
          if constexpr (!COLLIDE) {
          } else if constexpr (GUO) {
            w[0] = mg * ax; w[NC] = mg * ay; w[2 * NC] = mg * az + (kp.rho0 + drho1) * kp.g_z;
          } else {
            w[0] = mv * ax + jx1 * inv1; w[NC] = mv * ay + jy1 * inv1; w[2 * NC] = mv * az + (jz1 * inv1 + kp.gz_v);
          }
          w[3 * NC] = drho1; w[4 * NC] = inv1;
        }
      }
      bar_arrive(BAR_R + (p & 1), NT);
      inv1 = inv; drho1 = drho; jx1 = jx; jy1 = jy; jz1 = jz;
      uslot = uslot == 2 ? 0 : uslot + 1;
    }
  } else {
    __shared__ R red[DIAG ? 2 : 1][7][DIAG ? TY : 1];
    const int t = (int)threadIdx.x - NM, tx = t & 31, ty = t >> 5;
    const bool valid = x0 + tx < a.nx && y0 + ty < a.ny;
    const int h = (ty + 2) * RX + tx + 2;
    MarchPos<S> m;
    {
      unsigned xs[3], ys[3];
      neighbours(xs, ys, a, (unsigned)(valid ? x0 + tx : 0), (unsigned)(valid ? y0 + ty : 0) * (unsigned)a.nx);
      m.set(xs, ys, (size_t)z0 * plane);
    }
    MarchRaw<S> raw;
    unsigned own = m.v[1][1];
    raw.request(b.gsrc, a, z0, m);
    RefFeed<GE::GWX, GE::GW, NC> feed;
    if constexpr (IsLoc<S>::v) {
      feed.set(a, t, x0 - 1, y0 - 1);
      feed.start(b.gref, plane_bytes, gw_s, z0, nz);     // the first ready barrier makes it visible
    }
    R uzm = R(0), uz = R(0), uzp = R(0);
    int uslot = 2;            // slot of plane p-1 in the rings of three; plane p-2 has the one before
    for (int p = ps; p <= pe; ++p) {
      bar_sync(BAR_R + (p & 1), NT);                         // u of plane p-1 is there
      const int z = p - 2;
      if constexpr (DIAG) {
        // the partials of the plane before are complete
        if (a.part != nullptr && z - 1 >= z0 && ty == 0)
          diag_combine<R, TY>(red[(z - 1) & 1], tx, a.part + ((size_t)(z - 1) * gridDim.x + tile) * NPART);
      }
      uzm = uz; uz = uzp;
      if (p >= 1 && p - 1 < nz) uzp = uz_s[uslot * NC + t];
      const int zslot = uslot == 0 ? 2 : uslot - 1;
      uslot = uslot == 2 ? 0 : uslot + 1;
      DiagTerms<R> dt;
      if (z >= z0 && valid) {
        const R* us = uxy_s + zslot * (2 * NM);
        const R* w = w_s + zslot * (5 * NC) + t;
        R g[Q];
        raw.template decode<GE::GWX, GE::GW>(g, gw_s, (ty + 1) * GE::GWX + tx + 1, z, nz);
        if (z == 0 || z == nz - 1)
          g_wall_fix<S, R>(g, static_cast<const S*>(a.fin), a.N, (int)(own / (unsigned)sizeof(S)), z, nz, kp.rho0, kp.T0,
                           kp.T_d, kp.T_u, kp.lam);
        const R drho = w[3 * NC], inv = w[4 * NC];
        const R rho = kp.rho0 + drho;
        const R ux = us[h], uy = us[NM + h];
        R dE = g[0];
#pragma unroll
        for (int l = 1; l < Q; ++l) dE = dE + g[l];
        const R E = kp.E0 + dE;
        if constexpr (DIAG) {
          if (a.part != nullptr) dt.template take<VDW>(a, rho, inv, E * inv, E, ux, uy, uz);
        }
        if constexpr (COLLIDE) {
          const R zp = z + 1 < nz ? uzp : -uz, zm = z > 0 ? uzm : -uz;
          // 2 div(u)
          const R D2 = ((us[h + 1] - us[h - 1]) + (us[NM + h + RX] - us[NM + h - RX])) + (zp - zm);
          R lrf[3] = {R(0), R(0), R(0)}, lrg[3] = {R(0), R(0), R(0)};
          auto putf = [&](int l, R v) { Store<S>::st(reinterpret_cast<S*>(b.fdst[l] + (size_t)own), v); };
          auto putg = [&](int l, R v) { Store<S>::st(reinterpret_cast<S*>(b.gdst[l] + (size_t)own), v); };
          if constexpr (IsLoc<S>::v) {
            float a1, a2, b1, b2;
            loc_refs_of<S>(drho, dE, E * inv - kp.T0, kp.lam, a1, a2, b1, b2);
            lrf[0] = 12.0f * (a1 - a2); lrf[1] = a1; lrf[2] = a2;
            lrg[0] = 12.0f * (b1 - b2); lrg[1] = b1; lrg[2] = b2;
            putf(Q, a1); putf(Q + 1, a2); putg(Q, b1); putg(Q + 1, b2);
          }
          relax_g<R>(kp, E, dE, drho, inv, D2, ux, uy, uz, [&](int l) { return g[l]; },
                     [&](int l, R v) { putg(l, IsLoc<S>::v ? v - lrg[CSQ(l)] : v); });
          if (z + 1 < z1) {
            m.advance(step);
            raw.request(b.gsrc, a, z + 1, m);
          }
          const R wf[3] = {w[0], w[NC], w[2 * NC]};
          const FC* fc = fc_s + (size_t)(z & (DF - 1)) * Q * NC + t;
          relax_f<R, GUO>(kp, rho, drho, dE, ux, uy, uz, wf, [&](int l) { return cvt<FC, R>(fc[l * NC]); },
                          [&](int l, R v) { putf(l, IsLoc<S>::v ? v - lrf[CSQ(l)] : v); });
          own += step;
        } else {
          const size_t ob = (size_t)(own / (unsigned)sizeof(S));
          if (a.rho_out) a.rho_out[ob] = double(rho);
          if (a.ux_out) a.ux_out[ob] = double(ux);
          if (a.uy_out) a.uy_out[ob] = double(uy);
          if (a.uz_out) a.uz_out[ob] = double(uz);
          if (a.T_out) a.T_out[ob] = double(E * inv);
          own += step;
          if (z + 1 < z1) {
            m.advance(step);
            raw.request(b.gsrc, a, z + 1, m);
          }
        }
      }
      if constexpr (DIAG) {
        if (a.part != nullptr && z >= z0) dt.template reduce<TY>(red[z & 1], ty, tx);
      }
      if constexpr (IsLoc<S>::v) {
        if (z >= z0) feed.next(b.gref, plane_bytes, gw_s, z, nz);
      }
      if (p + 2 <= pe) bar_arrive(BAR_D + (p & 1), NT);
    }
    if constexpr (DIAG) {
      if (a.part != nullptr) {
        bar_sync(BAR_C, NC);
        if (ty == 0) diag_combine<R, TY>(red[(z1 - 1) & 1], tx, a.part + ((size_t)(z1 - 1) * gridDim.x + tile) * NPART);
      }
    }
  }
}

}  // namespace tlbm
