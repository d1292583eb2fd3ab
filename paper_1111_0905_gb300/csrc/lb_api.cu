// lb_api.cu -- C ABI of the thermal pseudopotential D3Q19 lattice Boltzmann step (include/lb.h).
//
// Host side: parameter validation, device memory of the context (two ping-pong population
// lattices per distribution, diagnostics scratch), launch geometry, checkpoints. Every step of
// the method runs in the kernels of lb_kernels.cuh, lb_split.cuh, lb_march.cuh and lb_march2.cuh; this
// file chooses the form of the step and marshals and orders them.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/lb.h"
#include "lb_launch.cuh"
#include "lb_ctx.h"

namespace tlbm {

// Diagnostics finalisation, in two launches so that the FP64 sums (1/64 of the FP32 rate on
// GB300) spread over the SMs. Every sum has a fixed assignment of terms to threads and a fixed
// combination tree, so the result does not depend on timing. out layout:
// [0, nz) Nu(z) of Eq. (4) (normalised by kappa (T_d - T_u)/nz); nz: Nu_mean; nz+1: min rho;
// nz+2: min T; nz+3: non-finite count; nz+4: sum rho; nz+5: sum rho T;
// [nz+8, 8nz+8) per-plane sums over the tiles, [7][nz] (scratch).
// If acc != null, acc[0] += Nu_mean, acc[1] += 1.

// 1) one CTA (128 threads) per plane: the plane's 7 partials summed (minima taken) over the tiles
__global__ void __launch_bounds__(128) lb_diag_planes(const double* __restrict__ part, int nz, int ntiles,
                                                      double* __restrict__ out) {
  __shared__ double red[7][4];
  const int z = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double v[7] = {0.0, 0.0, 0.0, 0.0, 1e300, 1e300, 0.0};
  for (int k = threadIdx.x; k < ntiles; k += blockDim.x) {
    const double* p = part + ((size_t)z * ntiles + k) * NPART;
#pragma unroll
    for (int q = 0; q < 7; ++q) v[q] = (q == 4 || q == 5) ? fmin(v[q], p[q]) : v[q] + p[q];
  }
#pragma unroll
  for (int q = 0; q < 7; ++q) v[q] = (q == 4 || q == 5) ? warp_min(v[q]) : warp_sum(v[q]);
  if (lane == 0)
    for (int q = 0; q < 7; ++q) red[q][warp] = v[q];
  __syncthreads();
  if (threadIdx.x < 7) {
    const int q = threadIdx.x;
    double a = red[q][0];
    for (int w = 1; w < 4; ++w) a = (q == 4 || q == 5) ? fmin(a, red[q][w]) : a + red[q][w];
    out[nz + 8 + (size_t)q * nz + z] = a;
  }
}

// 2) one CTA: Nu(z) from the plane sums with the wall ghosts, Nu_mean and the global values
__global__ void __launch_bounds__(1024) lb_diag_finalize(int nz, int nxy, double kappa, double T_d,
                                                         double T_u, double* __restrict__ out,
                                                         double* __restrict__ acc) {
  __shared__ double red[6][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const double* ps = out + nz + 8;   // [7][nz]: conv, T, rho, rho T, min rho, min T, non-finite
  const double* sT = ps + nz;
  const double norm = kappa * (T_d - T_u) / nz;
  double s = 0.0, sr = 0.0, sE = 0.0, mr = 1e300, mT = 1e300, bad = 0.0;
  for (int z = threadIdx.x; z < nz; z += blockDim.x) {
    const double Tp = (z + 1 < nz) ? sT[z + 1] : 2.0 * T_u * nxy - sT[nz - 1];
    const double Tm = (z - 1 >= 0) ? sT[z - 1] : 2.0 * T_d * nxy - sT[0];
    const double flux = (ps[z] - kappa * 0.5 * (Tp - Tm)) / nxy;
    const double nu = flux / norm;
    out[z] = nu;
    s += nu;
    sr += ps[2 * nz + z]; sE += ps[3 * nz + z];
    mr = fmin(mr, ps[4 * nz + z]); mT = fmin(mT, ps[5 * nz + z]); bad += ps[6 * nz + z];
  }
  s = warp_sum(s); sr = warp_sum(sr); sE = warp_sum(sE); bad = warp_sum(bad);
  mr = warp_min(mr); mT = warp_min(mT);
  if (lane == 0) {
    red[0][warp] = s; red[1][warp] = sr; red[2][warp] = sE; red[3][warp] = bad;
    red[4][warp] = mr; red[5][warp] = mT;
  }
  __syncthreads();
  if (warp == 0) {
    // the warps' values over the lanes of one warp (a serial chain of 6 x 32 FP64 additions took 15 us)
    const bool on = lane < nwarp;
    const double a0 = warp_sum(on ? red[0][lane] : 0.0), a1 = warp_sum(on ? red[1][lane] : 0.0);
    const double a2 = warp_sum(on ? red[2][lane] : 0.0), a3 = warp_sum(on ? red[3][lane] : 0.0);
    const double a4 = warp_min(on ? red[4][lane] : 1e300), a5 = warp_min(on ? red[5][lane] : 1e300);
    if (lane == 0) {
      const double mean = a0 / nz;
      out[nz] = mean; out[nz + 1] = a4; out[nz + 2] = a5; out[nz + 3] = a3;
      out[nz + 4] = a1; out[nz + 5] = a2;
      if (acc) { acc[0] += mean; acc[1] += 1.0; }
    }
  }
}


// Validation of initial fields: per-block count of bad entries and sums (fixed order).
__global__ void lb_validate_kernel(const double* __restrict__ rho, const double* __restrict__ T,
                                   int N, double rho_lim, double* __restrict__ out /* [gridDim.x][3] */) {
  __shared__ double sh[3][256];
  double bad = 0.0, sr = 0.0, sT = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    const double r = rho[i], t = T[i];
    if (!(r > 0.0) || !(r < rho_lim) || !(t > 0.0) || !isfinite(r) || !isfinite(t)) bad += 1.0;
    sr += r; sT += t;
  }
  sh[0][threadIdx.x] = bad; sh[1][threadIdx.x] = sr; sh[2][threadIdx.x] = sT;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
      for (int k = 0; k < 3; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 3; ++k) out[blockIdx.x * 3 + k] = sh[k][0];
}

}  // namespace tlbm

using namespace tlbm;

namespace {

const char* kNullCtxMsg = "null context";


const PrecOps* ops_for(int prec) {
  switch (prec) {
    case LB_FP64: return &kOpsF64;
    case LB_FP32: return &kOpsF32;
    case LB_BF16_DEV: return &kOpsBF16;
    case LB_FP16_DEV: return &kOpsF16;
    case LB_FP16_LOC: return &kOpsF16Loc;
    default: return nullptr;
  }
}

}  // namespace

KArgs make_args(const lb_ctx* c) {
  KArgs a;
  std::memset(&a, 0, sizeof(a));
  a.fin = c->f[c->cur]; a.gin = c->g[c->cur];
  a.fout = c->f[1 - c->cur]; a.gout = c->g[1 - c->cur];
  a.pre = c->pre;
  if (c->fld) {
    const bool f64 = c->ops->esize == sizeof(double);
    unsigned char* p = static_cast<unsigned char*>(c->fld);
    auto next = [&]() { void* q = p; p += (size_t)c->N * (f64 ? sizeof(double) : sizeof(float)); return q; };
    a.fd_rho = next(); a.fd_psi = next();
    for (int k = 0; k < 3; ++k) a.fd_j[k] = next();
    for (int k = 0; k < 3; ++k) a.fd_u[k] = next();
    // FP32: u' takes the place of j, which its own node has read by then (16-bit storage keeps none)
    for (int k = 0; k < 3; ++k) a.fd_v[k] = f64 ? next() : (c->ops->esize == 4 ? a.fd_j[k] : nullptr);
    if (f64) a.fd_inv = next();
  }
  // i / nx by multiplication, exact for i < 2^31: m = ceil(2^(32+s) / nx), 2^s < nx <= 2^(s+1)
  if (c->p.nx > 1) {
    unsigned s = 0;
    while ((2ull << s) < (unsigned long long)c->p.nx) ++s;
    a.div_s = s;
    a.div_m = (unsigned)(((1ull << (32 + s)) + (unsigned long long)c->p.nx - 1) / (unsigned long long)c->p.nx);
  }
  a.nx = c->p.nx; a.ny = c->p.ny; a.nz = c->p.nz; a.plane = c->plane; a.N = c->N;
  a.tiles_x = c->tiles_x; a.ntiles = c->ntiles; a.zc = c->zc;
  a.forcing = c->p.forcing; a.psi_kind = c->p.psi_kind;
  a.tau_nu = c->p.tau_nu; a.omega_nu = 1.0 / c->p.tau_nu; a.omega_kappa = 1.0 / c->p.tau_kappa;
  a.G = c->p.G; a.g_z = c->p.g_z; a.lam = c->lam; a.inv_cv = 1.0 / c->p.c_v; a.c_v = c->p.c_v;
  a.kappa = c->p.kappa; a.T_d = c->p.T_d; a.T_u = c->p.T_u;
  a.rho0 = c->rho0; a.T0 = c->T0; a.E0 = c->rho0 * c->T0;
  const double vk = c->p.psi_kind == PSI_VDW ? 2.0 / (-c->p.G) : 0.0;
  a.pd = {a.tau_nu, a.omega_nu, a.omega_kappa, a.G, a.g_z, a.lam, a.inv_cv, a.T_d, a.T_u,
          a.rho0, a.T0, a.E0, c->p.vdw_a, c->p.vdw_b, c->p.vdw_T, vk};
  a.pf = {(float)a.tau_nu, (float)a.omega_nu, (float)a.omega_kappa, (float)a.G, (float)a.g_z,
          (float)a.lam, (float)a.inv_cv, (float)a.T_d, (float)a.T_u, (float)a.rho0, (float)a.T0,
          (float)a.E0, (float)c->p.vdw_a, (float)c->p.vdw_b, (float)c->p.vdw_T, (float)vk};
  a.pd.psi0 = std::exp(-1.0 / c->rho0);
  a.pd.irho0 = 1.0 / c->rho0;
  a.pf.psi0 = (float)a.pd.psi0;
  a.pf.irho0 = (float)a.pd.irho0;
  auto split_consts = [&](auto& k) {
    using R = std::decay_t<decltype(k.om1)>;
    constexpr bool F32 = sizeof(R) == 4;
    // x as R and, for FP32, its remainder
    auto two = [](double x, R& hi, R& lo) { hi = (R)x; lo = (R)(x - (double)hi); };
    // the weights of relaxation rate omega; returns the rate that they and om1 add up to
    auto weights = [&](double omega, R& om1, R (&o)[3], R (&o_lo)[3], R (&s3)[3], R (&s3_lo)[3], R (&q)[3]) -> double {
      om1 = (R)(1.0 - omega);
      const double rate = F32 ? 1.0 - (double)om1 : omega, w2 = rate / 36.0;
      const double w[3] = {12.0 * w2, 2.0 * w2, w2};
      for (int c = 0; c < 3; ++c) {
        two(w[c], o[c], o_lo[c]);
        two(3.0 * w[c], s3[c], s3_lo[c]);
        q[c] = (R)(4.5 * w[c]);
      }
      return rate;
    };
    const double en = weights(a.omega_nu, k.om1, k.fo, k.fo_lo, k.fs, k.fs_lo, k.fq);
    const double ek = weights(a.omega_kappa, k.omk1, k.go, k.go_lo, k.gs, k.gs_lo, k.gq);
    const double tau = F32 ? 1.0 / en : a.tau_nu;      // so that a step adds F to j, whole
    const bool dev = F32 && a.psi_kind != PSI_VDW;
    // The reference density of the FP32 forms is the rounded one (their deviations are from it). psi refers
    // to rho1, rho0 unless that is below 1/40: psi(rho1)^2 stays a normal float.
    const double r0 = (double)k.rho0, r1 = std::max(r0, 1.0 / 40.0), p1 = std::exp(-1.0 / r1);
    k.t1 = (R)(1.0 / r1 - 1.0 / r0);
    two(dev ? -a.G * p1 * p1 / 12.0 : -a.G / 12.0, k.mg, k.mg_lo);
    R hi;
    two(1.0 / r0, hi, k.irho0_lo);
    k.irho0 = hi;
    two(tau, k.tau, k.tau_lo);
    k.gz_u = (R)(0.5 * a.g_z); k.gz_v = (R)(tau * a.g_z);
    k.src = (R)(0.5 / (c->p.c_v * ek)); k.lam45 = (R)(4.5 * a.lam);
    k.ks = (R)(1.0 - 0.5 * en);
  };
  split_consts(a.pd);
  split_consts(a.pf);
  // reference equilibria per class (rest, axis, diagonal): f^eq(rho0, 0, T0), g^eq(rho0, T0, 0)
  const double w[3] = {1.0 / 3.0, 1.0 / 18.0, 1.0 / 36.0};
  for (int k = 0; k < 3; ++k) {
    a.fbase[k] = w[k] * c->rho0 * (1.0 + 4.5 * (c->T0 - 1.0 / 3.0) * (k - 1));
    a.gbase[k] = w[k] * (a.E0 + 4.5 * (c->lam * c->T0 - a.E0 / 3.0) * (k - 1));
  }
  for (int l = 0; l < Q; ++l)
    a.loff[l] = (unsigned)((long long)l * c->N - (long long)CZ(l) * c->plane);
  return a;
}

dim3 fused_grid(const lb_ctx* c) { return dim3(c->ntiles, c->nchunks); }

cudaError_t launch_step(const lb_ctx* c, const KArgs& a, int mode) {
  if (c->form == lb_ctx::kThree) return c->ops->split(a, mode, c->three_nt, c->stream);
  if (c->form == lb_ctx::kMarch) return c->ops->march(a, mode, c->march_zc, c->march_zc2, c->stream);
  return c->ops->fused(a, mode, c->by, fused_grid(c), c->stream);
}

namespace {

// The form of the step of a context whose caller left the launch shape to the library.
//
// FP64 takes three kernels: its FP64 instructions bound the step, and the marches recompute ring
// nodes. (256^3: 8.9 ms against 10.7 with the tile march and its pre-pass.)
//
// FP32 compute takes the one-launch march, unless three kernels are expected to be faster. A march
// iteration is one plane of a CTA; a CTA of zc planes takes zc + 4 of them and about two more to
// start, one CTA per SM, in waves: ceil(CTAs / SMs) (zc + 6) iterations. Measured per iteration (128^3,
// 256^3): FP32 1.8 us, 16-bit deviations 1.5 us (two nodes per thread: 2.2 us for a tile of twice the
// width, 7 rows), local references 2.2 us. The three kernels take about
// 7 us and per node 75, 58 and 77 ps (FP32 64^3 28 us and 128^3 172 us, the march 21 and 126 us; 32^3
// 7.4 us against 18; local references 96^3 72 us against 86). The chunk zc is the one of the least cost.
cudaError_t choose_form(lb_ctx* c) {
  c->nblk = c->nblk_step = c->ntiles;
  if (c->p.tile_y != 0 || c->p.z_chunk != 0) { c->form = lb_ctx::kTile; return cudaSuccess; }
  int sms = 0;
  const cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  if (e != cudaSuccess) return e;
  c->form = lb_ctx::kThree;
  if (c->ops->march_ty > 0) {
    const int nz = c->p.nz;
    // the least cost of a march over a number of tiles, and its chunk
    auto chunk = [&](long long tiles, int* best_zc) {
      long long best = -1;
      for (int nch = 1; nch <= nz && nch <= 65535; ++nch) {
        const int zc = (nz + nch - 1) / nch;
        if (zc < 4 && nch > 1) break;
        const long long ctas = tiles * ((nz + zc - 1) / zc);
        const long long cost = ((ctas + sms - 1) / sms) * (zc + 6);
        if (best < 0 || cost < best) { best = cost; *best_zc = zc; }
      }
      return best;
    };
    auto rows = [&](int ty) { return (long long)((c->p.ny + ty - 1) / ty); };
    const long long tiles = (long long)c->tiles_x * rows(c->ops->march_ty);
    const long long best = chunk(tiles, &c->march_zc);
    const bool b16 = c->ops->esize == 2, loc = c->ops->slots > Q;
    const double node = loc ? 77e-12 : (b16 ? 58e-12 : 75e-12);
    double march = (loc ? 2.2e-6 : (b16 ? 1.5e-6 : 1.8e-6)) * (double)best;
    const long long tiles2 = c->ops->march_ty2 > 0 ? (long long)((c->p.nx + 63) / 64) * rows(c->ops->march_ty2) : 0;
    if (tiles2 > 0 && c->p.nx % 2 == 0 && variant_of(c->p.forcing, c->p.psi_kind) == 0) {
      const double two = 2.2e-6 * (double)chunk(tiles2, &c->march_zc2);
      if (two < march) march = two;
      else c->march_zc2 = 0;
    }
    if (march < 7e-6 + node * (double)c->N) {
      c->form = lb_ctx::kMarch;
      c->nblk = (int)tiles;
      c->nblk_step = c->march_zc2 > 0 ? (int)tiles2 : c->nblk;
      return cudaSuccess;
    }
  }
  // Few nodes per SM: CTAs of 64 threads share them out more evenly than 256 (FP64 48^3: 72 us against
  // 76), CTAs of 32 where several run on an SM and the fullest one then has fewer nodes (32^3, 216 nodes
  // per SM on average: 224 instead of 256 on the fullest; 28.4 -> 26.3 us).
  c->three_nt = 256;
  if ((long long)c->N < 4ll * 256 * sms) {
    auto fullest = [&](int nt) { return ((long long)((c->plane + nt - 1) / nt) * c->p.nz + sms - 1) / sms * nt; };
    c->three_nt = fullest(64) > 64 && fullest(32) < fullest(64) ? 32 : 64;
  }
  c->nblk = c->nblk_step = (c->plane + c->three_nt - 1) / c->three_nt;
  return cudaSuccess;
}

void free_all(lb_ctx* c) {
  if (!c) return;
  for (int k = 0; k < 2; ++k) { cudaFree(c->f[k]); cudaFree(c->g[k]); }
  cudaFree(c->part); cudaFree(c->diag); cudaFree(c->nu_acc);
  cudaFree(c->fields); cudaFree(c->pops); cudaFree(c->pre); cudaFree(c->fld);
}

}  // namespace

// Moments pass into the plane partials, then Nu(z) and the global health values into diag;
// Nu_mean is added to acc[0] (and 1 to acc[1]) when acc is not null.
int finalize_diag(lb_ctx* c, double* acc, int nblk) {
  lb_diag_planes<<<c->p.nz, 128, 0, c->stream>>>(c->part, c->p.nz, nblk, c->diag);
  const int ft = std::min(1024, (c->p.nz + 31) / 32 * 32);
  lb_diag_finalize<<<1, ft, 0, c->stream>>>(c->p.nz, c->p.nx * c->p.ny, c->p.kappa, c->p.T_d,
                                               c->p.T_u, c->diag, acc);
  LB_CU(c, cudaGetLastError());
  return LB_OK;
}

int run_diag_acc(lb_ctx* c, double* acc) {
  KArgs a = make_args(c);
  a.part = c->part;
  LB_CU(c, launch_step(c, a, MODE_MOMENTS));
  return finalize_diag(c, acc, c->nblk);
}

int run_diag(lb_ctx* c, bool accumulate) { return run_diag_acc(c, accumulate ? c->nu_acc : nullptr); }

int flush_sample(lb_ctx* c) {
  if (!c->sample_pending) return LB_OK;
  c->sample_pending = false;
  return run_diag(c, true);
}

namespace {

uint64_t fnv1a(uint64_t h, const unsigned char* p, size_t n) {
  for (size_t i = 0; i < n; ++i) { h ^= p[i]; h *= 1099511628211ull; }
  return h;
}

struct CkptHeader {
  char magic[8];
  int32_t version, precision;
  int32_t nx, ny, nz, pad;
  int64_t step;
  double rho0, T0;
  double nu_acc[2];
  lb_params params;
  uint64_t checksum;
};

}  // namespace

extern "C" {

const char* lb_strerror(int code) {
  switch (code) {
    case LB_OK: return "ok";
    case LB_EINVAL: return "invalid argument";
    case LB_ENOMEM: return "out of memory";
    case LB_ECUDA: return "CUDA error";
    case LB_ENONPHYS: return "non-physical state (rho <= 0, T <= 0 or NaN)";
    case LB_EIO: return "checkpoint I/O error";
    case LB_EUNSUP: return "unsupported";
    default: return "unknown error";
  }
}

const char* lb_last_error(const lb_ctx* c) { return c ? c->err.c_str() : kNullCtxMsg; }

long long lb_step_count(const lb_ctx* c) { return c ? c->step : -1; }

int lb_launch_info(lb_ctx* c, int* out) {
  if (!c || !out) return LB_EINVAL;
  int k[4] = {0, 0, 0, 0};
  LB_CU(c, c->ops->info(c->by, variant_of(c->p.forcing, c->p.psi_kind), k));
  const dim3 grid = fused_grid(c);
  out[0] = (int)grid.x; out[1] = (int)grid.y;
  out[2] = k[0]; out[3] = k[1]; out[4] = k[2]; out[5] = k[3];
  return LB_OK;
}

int lb_step_info(lb_ctx* c, int* out) {
  if (!c || !out) return LB_EINVAL;
  const int var = variant_of(c->p.forcing, c->p.psi_kind);
  int k[4] = {0, 0, 0, 0};
  const dim3 grid = fused_grid(c);
  int form = STEP_TILE, gx = (int)grid.x, gy = (int)grid.y;
  if (c->form == lb_ctx::kTile) {
    LB_CU(c, c->ops->info(c->by, var, k));
  } else {
    form = c->form == lb_ctx::kThree ? STEP_THREE : (c->march_zc2 > 0 ? STEP_MARCH2 : STEP_MARCH);
    const int zc = form == STEP_THREE ? 1 : (form == STEP_MARCH2 ? c->march_zc2 : c->march_zc);
    gx = c->nblk_step; gy = (c->p.nz + zc - 1) / zc;
    LB_CU(c, c->ops->step_info(form, c->three_nt, var, k));
  }
  out[0] = form; out[1] = gx; out[2] = gy;
  for (int i = 0; i < 4; ++i) out[3 + i] = k[i];
  return LB_OK;
}

int lb_init(const lb_params* params, const double* rho_init, const double* T_init,
            int init_on_device, void* cuda_stream, lb_ctx** out) {
  if (!out) return LB_EINVAL;
  *out = nullptr;
  if (!params || !rho_init || !T_init) return LB_EINVAL;
  const lb_params& p = *params;
  if (p.nx < 1 || p.ny < 1 || p.nz < 1) return LB_EINVAL;
  const long long N = (long long)p.nx * p.ny * p.nz;
  if (N >= (1ll << 31) || (long long)p.nz * 2 >= (1ll << 30)) return LB_EINVAL;
  if (!(p.tau_nu > 0.5) || !(p.tau_kappa > 0.5) || !(p.kappa > 0.0) || !(p.c_v > 0.0)) return LB_EINVAL;
  if (!std::isfinite(p.G) || !std::isfinite(p.g_z) || !(p.T_d > 0.0) || !(p.T_u > 0.0)) return LB_EINVAL;
  const PrecOps* ops = ops_for(p.precision);
  if (!ops) return LB_EINVAL;
  // default tile height 32 x 8 (measured best on the 128^3/256^3 cells for every form)
  int by = p.tile_y != 0 ? p.tile_y : 8;
  if (by != 4 && by != 8 && by != 16) return LB_EINVAL;
  if (!ops->tile_ok(by)) return LB_EINVAL;
  if ((long long)ops->slots * N >= (1ll << 32)) return LB_EINVAL;   // 32-bit population offsets
  if (p.z_chunk < 0 || p.nu_every < 0 || p.check_every < 0) return LB_EINVAL;
  if (p.forcing != FORCE_SHIFT && p.forcing != FORCE_GUO) return LB_EINVAL;
  if (p.psi_kind != PSI_EXP && p.psi_kind != PSI_VDW) return LB_EINVAL;
  // van der Waals psi: real for rho < (1 - b T_v/a)/b; every initial density must be below it
  double rho_lim = INFINITY;
  if (p.psi_kind == PSI_VDW) {
    if (!(p.G < 0.0) || !(p.vdw_a > 0.0) || !(p.vdw_b > 0.0) || !(p.vdw_T > 0.0) ||
        !(p.vdw_b * p.vdw_T < p.vdw_a))
      return LB_EINVAL;
    rho_lim = (1.0 - p.vdw_b * p.vdw_T / p.vdw_a) / p.vdw_b;
  }

  lb_ctx* c = new (std::nothrow) lb_ctx();
  if (!c) return LB_ENOMEM;
  c->p = p;
  c->ops = ops;
  c->stream = static_cast<cudaStream_t>(cuda_stream);
  c->N = (int)N;
  c->plane = p.nx * p.ny;
  c->by = by;
  c->lam = p.kappa / (p.c_v * (p.tau_kappa - 0.5));
  c->tiles_x = (p.nx + BX - 1) / BX;
  c->tiles_y = (p.ny + by - 1) / by;
  c->ntiles = c->tiles_x * c->tiles_y;

  auto bail = [&](int code) { free_all(c); delete c; return code; };
  if (cudaGetDevice(&c->device) != cudaSuccess) return bail(LB_ECUDA);
  if (ops->prepare() != cudaSuccess) return bail(LB_ECUDA);
  if (p.z_chunk > 0) {
    c->zc = p.z_chunk < p.nz ? p.z_chunk : p.nz;
  } else {
    // Planes per chunk: each chunk adds 4 prologue planes (M stages without collisions) and the
    // CTAs run in waves of (resident CTAs per SM) x SMs, so a launch takes about
    // ceil(CTAs / slots) * (zc + 4) plane-steps. Take the chunk count (zc from 8 to 128, or nz)
    // that minimises it; ties go to the larger chunk.
    int k[4] = {0, 0, 0, 0}, sms = 0;
    if (ops->info(by, variant_of(p.forcing, p.psi_kind), k) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess)
      return bail(LB_ECUDA);
    const long long slots = (long long)(k[2] > 0 ? k[2] : 1) * (sms > 0 ? sms : 1);
    c->zc = p.nz;
    long long best = -1;
    for (int nch = 1; nch <= p.nz; ++nch) {
      const int zc = (p.nz + nch - 1) / nch;
      if (zc > 128) continue;
      if (zc < 8 && nch > 1) break;
      const long long ctas = (long long)c->ntiles * ((p.nz + zc - 1) / zc);
      const long long cost = ((ctas + slots - 1) / slots) * (zc + 4);
      if (best < 0 || cost < best) { best = cost; c->zc = zc; }
    }
  }
  c->nchunks = (p.nz + c->zc - 1) / c->zc;

  // validate the initial fields and form their means on the device (fixed-order sums)
  const double* d_rho = rho_init;
  const double* d_T = T_init;
  double* staging = nullptr;
  const size_t fbytes = (size_t)N * sizeof(double);
  if (!init_on_device) {
    if (cudaMalloc(&staging, 2 * fbytes) != cudaSuccess) return bail(LB_ENOMEM);
    if (cudaMemcpyAsync(staging, rho_init, fbytes, cudaMemcpyHostToDevice, c->stream) != cudaSuccess ||
        cudaMemcpyAsync(staging + N, T_init, fbytes, cudaMemcpyHostToDevice, c->stream) != cudaSuccess) {
      cudaFree(staging);
      return bail(LB_ECUDA);
    }
    d_rho = staging;
    d_T = staging + N;
  }
  const int vblocks = 256;
  double* vpart = nullptr;
  if (cudaMalloc(&vpart, vblocks * 3 * sizeof(double)) != cudaSuccess) { cudaFree(staging); return bail(LB_ENOMEM); }
  lb_validate_kernel<<<vblocks, 256, 0, c->stream>>>(d_rho, d_T, c->N, rho_lim, vpart);
  std::vector<double> hv(vblocks * 3);
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(hv.data(), vpart, hv.size() * sizeof(double), cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
      cudaStreamSynchronize(c->stream) != cudaSuccess) {
    cudaFree(vpart); cudaFree(staging);
    return bail(LB_ECUDA);
  }
  cudaFree(vpart);
  double bad = 0, sr = 0, sT = 0;
  for (int b = 0; b < vblocks; ++b) { bad += hv[b * 3]; sr += hv[b * 3 + 1]; sT += hv[b * 3 + 2]; }
  if (bad > 0) { cudaFree(staging); return bail(LB_EINVAL); }
  c->rho0 = p.rho0 > 0 ? p.rho0 : sr / N;
  c->T0 = p.T0 > 0 ? p.T0 : sT / N;

  // 64 bytes of padding: a word-wide copy of a 16-bit element (stage_word) reads the 4-byte word
  // that contains it
  const size_t pbytes = (size_t)ops->slots * N * ops->esize + 64;
  for (int k = 0; k < 2; ++k) {
    if (cudaMalloc(&c->f[k], pbytes) != cudaSuccess || cudaMalloc(&c->g[k], pbytes) != cudaSuccess) {
      cudaFree(staging);
      return bail(LB_ENOMEM);
    }
  }
  if (choose_form(c) != cudaSuccess) return staging ? (cudaFree(staging), bail(LB_ECUDA)) : bail(LB_ECUDA);
  if (c->form == lb_ctx::kThree) {
    const size_t fb = ops->esize == sizeof(double) ? 12 * sizeof(double) : 8 * sizeof(float);
    if (cudaMalloc(&c->fld, fb * (size_t)N) != cudaSuccess) { cudaFree(staging); return bail(LB_ENOMEM); }
  }
  // FP64: per-node moments and psi that each step kernel's ring reads (lb_fields_kernel)
  if (c->form == lb_ctx::kTile && ops->esize == sizeof(double) && cudaMalloc(&c->pre, 6 * (size_t)N * sizeof(double)) != cudaSuccess) {
    cudaFree(staging);
    return bail(LB_ENOMEM);
  }
  if (cudaMalloc(&c->part, (size_t)p.nz * std::max(c->nblk, c->nblk_step) * NPART * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&c->diag, (size_t)(8 * p.nz + 8) * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&c->nu_acc, 2 * sizeof(double)) != cudaSuccess) {
    cudaFree(staging);
    return bail(LB_ENOMEM);
  }
  if (cudaMemsetAsync(c->nu_acc, 0, 2 * sizeof(double), c->stream) != cudaSuccess) { cudaFree(staging); return bail(LB_ECUDA); }
  c->cur = 0;
  KArgs a = make_args(c);
  a.fout = c->f[0]; a.gout = c->g[0];
  if (ops->init(a, d_rho, d_T, c->stream) != cudaSuccess) { cudaFree(staging); return bail(LB_ECUDA); }
  if (staging) {
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) { cudaFree(staging); return bail(LB_ECUDA); }
    cudaFree(staging);
  }
  c->step = 0;
  *out = c;
  return LB_OK;
}

int lb_step(lb_ctx* c, long long nsteps) {
  if (!c) return LB_EINVAL;
  if (nsteps < 0) return lb_fail(c, LB_EINVAL, "nsteps < 0");
  // a Nu sample of state n is taken by the launch of step n -> n+1 (the paper's scheme; the
  // variants take it with a separate moments pass)
  const bool fuse = variant_of(c->p.forcing, c->p.psi_kind) == 0;
  for (long long s = 0; s < nsteps; ++s) {
    KArgs a = make_args(c);
    if (c->sample_pending && fuse) {
      a.part = c->part;
      LB_CU(c, launch_step(c, a, MODE_STEP_DIAG));
      c->sample_pending = false;
      const int rc = finalize_diag(c, c->nu_acc, c->nblk_step);
      if (rc) return rc;
    } else {
      const int rc = flush_sample(c);
      if (rc) return rc;
      LB_CU(c, launch_step(c, a, MODE_STEP));
    }
    c->cur ^= 1;
    c->step += 1;
    if (c->p.nu_every > 0 && c->step % c->p.nu_every == 0) c->sample_pending = true;
    if (c->p.check_every > 0 && c->step % c->p.check_every == 0) {
      int rc = c->sample_pending ? flush_sample(c) : run_diag(c, false);
      if (rc) return rc;
      double h[4];
      LB_CU(c, cudaMemcpyAsync(h, c->diag + c->p.nz, 4 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
      LB_CU(c, cudaStreamSynchronize(c->stream));
      if (!(h[1] > 0.0) || !(h[2] > 0.0) || h[3] != 0.0)
        return lb_fail(c, LB_ENONPHYS, "health check failed at step " + std::to_string(c->step));
    }
  }
  return LB_OK;
}

int lb_moments(lb_ctx* c, double* rho, double* ux, double* uy, double* uz, double* T, int on_device) {
  if (!c) return LB_EINVAL;
  KArgs a = make_args(c);
  double* outs[5] = {rho, ux, uy, uz, T};
  const size_t N = (size_t)c->N;
  if (!on_device) {
    if (!c->fields && cudaMalloc(&c->fields, 5 * N * sizeof(double)) != cudaSuccess)
      return lb_fail(c, LB_ENOMEM, "moments staging");
    for (int k = 0; k < 5; ++k) if (outs[k]) outs[k] = c->fields + k * N;
  }
  a.rho_out = outs[0]; a.ux_out = outs[1]; a.uy_out = outs[2]; a.uz_out = outs[3]; a.T_out = outs[4];
  a.part = nullptr;
  LB_CU(c, launch_step(c, a, MODE_MOMENTS));
  if (!on_device) {
    double* host[5] = {rho, ux, uy, uz, T};
    for (int k = 0; k < 5; ++k)
      if (host[k])
        LB_CU(c, cudaMemcpyAsync(host[k], c->fields + k * N, N * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    LB_CU(c, cudaStreamSynchronize(c->stream));
  }
  return LB_OK;
}

int lb_nusselt(lb_ctx* c, double* nu_mean, double* nu_z, double* nu_time_avg) {
  if (!c || !nu_mean) return c ? lb_fail(c, LB_EINVAL, "nu_mean is null") : LB_EINVAL;
  int rc = c->sample_pending ? flush_sample(c) : run_diag(c, false);
  if (rc) return rc;
  const int nz = c->p.nz;
  std::vector<double> h(nz + 1);
  double acc[2];
  LB_CU(c, cudaMemcpyAsync(h.data(), c->diag, (nz + 1) * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  LB_CU(c, cudaMemcpyAsync(acc, c->nu_acc, 2 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  LB_CU(c, cudaStreamSynchronize(c->stream));
  *nu_mean = h[nz];
  if (nu_z) std::memcpy(nu_z, h.data(), nz * sizeof(double));
  if (nu_time_avg) *nu_time_avg = acc[1] > 0 ? acc[0] / acc[1] : NAN;
  return LB_OK;
}

int lb_diagnostics(lb_ctx* c, double out[5]) {
  if (!c || !out) return c ? lb_fail(c, LB_EINVAL, "out is null") : LB_EINVAL;
  int rc = c->sample_pending ? flush_sample(c) : run_diag(c, false);
  if (rc) return rc;
  double h[5];
  LB_CU(c, cudaMemcpyAsync(h, c->diag + c->p.nz + 1, 5 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  LB_CU(c, cudaStreamSynchronize(c->stream));
  for (int k = 0; k < 5; ++k) out[k] = h[k];
  return LB_OK;
}

int lb_populations(lb_ctx* c, double* f, double* g, int on_device) {
  if (!c) return LB_EINVAL;
  const size_t n = (size_t)Q * c->N;
  double* df = f;
  double* dg = g;
  if (!on_device) {
    if (!c->pops && cudaMalloc(&c->pops, 2 * n * sizeof(double)) != cudaSuccess)
      return lb_fail(c, LB_ENOMEM, "population staging");
    df = f ? c->pops : nullptr;
    dg = g ? c->pops + n : nullptr;
  }
  KArgs a = make_args(c);
  LB_CU(c, c->ops->pops(a, df, dg, c->stream));
  if (!on_device) {
    if (f) LB_CU(c, cudaMemcpyAsync(f, df, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    if (g) LB_CU(c, cudaMemcpyAsync(g, dg, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    LB_CU(c, cudaStreamSynchronize(c->stream));
  }
  return LB_OK;
}

int lb_set_populations(lb_ctx* c, const double* f, const double* g, int on_device) {
  if (!c) return LB_EINVAL;
  if (!f || !g) return lb_fail(c, LB_EINVAL, "f and g are both required");
  const size_t n = (size_t)Q * c->N;
  const double* df = f;
  const double* dg = g;
  if (!on_device) {
    if (!c->pops && cudaMalloc(&c->pops, 2 * n * sizeof(double)) != cudaSuccess)
      return lb_fail(c, LB_ENOMEM, "population staging");
    LB_CU(c, cudaMemcpyAsync(c->pops, f, n * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    LB_CU(c, cudaMemcpyAsync(c->pops + n, g, n * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    df = c->pops;
    dg = c->pops + n;
  }
  // a Nu sample due for the replaced state is dropped; the buffer written is the current one
  c->sample_pending = false;
  KArgs a = make_args(c);
  a.fout = c->f[c->cur]; a.gout = c->g[c->cur];
  LB_CU(c, c->ops->setpops(a, df, dg, c->stream));
  if (!on_device) LB_CU(c, cudaStreamSynchronize(c->stream));
  c->from_init = false;
  return LB_OK;
}

int lb_save(lb_ctx* c, const char* path) {
  if (!c || !path) return c ? lb_fail(c, LB_EINVAL, "path is null") : LB_EINVAL;
  const int frc = flush_sample(c);    // the saved time average includes every due sample
  if (frc) return frc;
  const size_t pbytes = (size_t)c->ops->slots * c->N * c->ops->esize;
  std::vector<unsigned char> buf(2 * pbytes);
  CkptHeader h;
  std::memset(&h, 0, sizeof(h));
  std::memcpy(h.magic, "TLBMCKP2", 8);
  h.version = 2; h.precision = c->p.precision;
  h.nx = c->p.nx; h.ny = c->p.ny; h.nz = c->p.nz;
  h.step = c->step; h.rho0 = c->rho0; h.T0 = c->T0; h.params = c->p;
  LB_CU(c, cudaMemcpyAsync(buf.data(), c->f[c->cur], pbytes, cudaMemcpyDeviceToHost, c->stream));
  LB_CU(c, cudaMemcpyAsync(buf.data() + pbytes, c->g[c->cur], pbytes, cudaMemcpyDeviceToHost, c->stream));
  LB_CU(c, cudaMemcpyAsync(h.nu_acc, c->nu_acc, 2 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  LB_CU(c, cudaStreamSynchronize(c->stream));
  h.checksum = fnv1a(1469598103934665603ull, buf.data(), buf.size());
  FILE* fp = std::fopen(path, "wb");
  if (!fp) return lb_fail(c, LB_EIO, std::string("cannot open ") + path);
  bool ok = std::fwrite(&h, sizeof(h), 1, fp) == 1 && std::fwrite(buf.data(), 1, buf.size(), fp) == buf.size();
  ok = (std::fclose(fp) == 0) && ok;
  return ok ? LB_OK : lb_fail(c, LB_EIO, std::string("write failed: ") + path);
}

int lb_load(lb_ctx* c, const char* path) {
  if (!c || !path) return c ? lb_fail(c, LB_EINVAL, "path is null") : LB_EINVAL;
  FILE* fp = std::fopen(path, "rb");
  if (!fp) return lb_fail(c, LB_EIO, std::string("cannot open ") + path);
  CkptHeader h;
  const size_t pbytes = (size_t)c->ops->slots * c->N * c->ops->esize;
  std::vector<unsigned char> buf(2 * pbytes);
  bool ok = std::fread(&h, sizeof(h), 1, fp) == 1 && std::fread(buf.data(), 1, buf.size(), fp) == buf.size();
  std::fclose(fp);
  if (!ok) return lb_fail(c, LB_EIO, "short read");
  if (std::memcmp(h.magic, "TLBMCKP2", 8) != 0 || h.version != 2) return lb_fail(c, LB_EIO, "bad magic/version");
  if (h.nx != c->p.nx || h.ny != c->p.ny || h.nz != c->p.nz || h.precision != c->p.precision)
    return lb_fail(c, LB_EIO, "grid or precision mismatch");
  // the physics parameters must be the context's: a state saved under other relaxation times,
  // coupling, conductivity, gravity, wall temperatures or scheme variant is refused (the
  // reference state rho0, T0 of the deviation storage is restored from the file)
  {
    const lb_params& q = h.params;
    const lb_params& p = c->p;
    const bool same = q.tau_nu == p.tau_nu && q.tau_kappa == p.tau_kappa && q.G == p.G &&
                      q.kappa == p.kappa && q.c_v == p.c_v && q.g_z == p.g_z && q.T_d == p.T_d &&
                      q.T_u == p.T_u && q.forcing == p.forcing && q.psi_kind == p.psi_kind &&
                      (p.psi_kind != PSI_VDW ||
                       (q.vdw_a == p.vdw_a && q.vdw_b == p.vdw_b && q.vdw_T == p.vdw_T));
    if (!same) return lb_fail(c, LB_EIO, "checkpoint parameters differ from the context's");
  }
  if (fnv1a(1469598103934665603ull, buf.data(), buf.size()) != h.checksum)
    return lb_fail(c, LB_EIO, "checksum mismatch");
  LB_CU(c, cudaMemcpyAsync(c->f[c->cur], buf.data(), pbytes, cudaMemcpyHostToDevice, c->stream));
  LB_CU(c, cudaMemcpyAsync(c->g[c->cur], buf.data() + pbytes, pbytes, cudaMemcpyHostToDevice, c->stream));
  LB_CU(c, cudaMemcpyAsync(c->nu_acc, h.nu_acc, 2 * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  LB_CU(c, cudaStreamSynchronize(c->stream));
  c->step = h.step;
  c->sample_pending = false;
  c->rho0 = h.rho0;
  c->T0 = h.T0;
  return LB_OK;
}

void lb_free(lb_ctx* c) {
  if (!c) return;
  cudaStreamSynchronize(c->stream);
  free_all(c);
  delete c;
}

}  // extern "C"
