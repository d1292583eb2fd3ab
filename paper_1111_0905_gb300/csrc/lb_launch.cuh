// lb_launch.cuh -- per-precision launch table of the kernels in lb_kernels.cuh, lb_split.cuh, lb_march.cuh
// and lb_march2.cuh.
// Each precision is compiled in its own translation unit (lb_prec_*.cu) that defines one table.
#pragma once
#include "lb_kernels.cuh"
#include "lb_march2.cuh"

namespace tlbm {

// Launch of a kernel that calls wait_for_predecessor first: it comes up as the CTAs of the launch before
// it end (programmatic dependent launch).
template <class... P, class... A>
inline cudaError_t follow(void (*k)(P...), unsigned grid, int nt, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3((unsigned)nt); cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

// forms of the step as lb_step_info reports them
enum { STEP_TILE = 0, STEP_THREE = 1, STEP_MARCH = 2, STEP_MARCH2 = 3 };

struct PrecOps {
  size_t esize;        // bytes per stored population
  int deviation;       // 1 if populations are stored as deviations from w_l * ref
  cudaError_t (*prepare)();   // per-device kernel attributes (call with the device current)
  cudaError_t (*fused)(const KArgs&, int mode, int by, dim3 grid, cudaStream_t);
  cudaError_t (*init)(const KArgs&, const double*, const double*, cudaStream_t);
  cudaError_t (*pops)(const KArgs&, double*, double*, cudaStream_t);
  bool (*tile_ok)(int by);    // whether the tile height's shared-memory window fits a CTA
  // launch description of the step kernel for a tile height and variant: out = {threads per
  // CTA, dynamic shared memory bytes, resident CTAs per SM, registers per thread}
  cudaError_t (*info)(int by, int var, int out[4]);
  // store a given pre-collision state (float64 [19][N] f and g on the device) as the buffer
  cudaError_t (*setpops)(const KArgs&, const double*, const double*, cudaStream_t);
  // the three-kernel step (lb_split.cuh) in mode MODE_* with CTAs of nt threads (32, 64 or 256), and the
  // one-launch march (lb_march.cuh) with chunks of zc planes and its tile height (0: none for FP64)
  cudaError_t (*split)(const KArgs&, int mode, int nt, cudaStream_t);
  cudaError_t (*march)(const KArgs&, int mode, int zc, int zc2, cudaStream_t);
  // the kernel of a plain step (three kernels: the collision) of form STEP_* and variant var, CTAs of nt
  // threads (three kernels only): threads, dynamic shared memory, resident CTAs per SM, registers
  cudaError_t (*step_info)(int form, int nt, int var, int out[4]);
  int march_ty;
  int march_ty2;       // tile height of the march with two nodes per thread (64 wide; chunks of zc2; 0: none)
  int slots;           // stored slots per lattice and node: 19, or 21 with the local references
};

extern const PrecOps kOpsF64, kOpsF32, kOpsBF16, kOpsF16, kOpsF16Loc;

template <class S> struct OpsImpl {
  using R = typename Store<S>::R;

  // dynamic shared memory of a tile height; tile heights whose windows exceed the 227 KB a CTA
  // may use are not available, nor FP64 with BY = 16 (a CTA of 512 threads leaves the FP64
  // collision 128 registers per thread, too few for its 38 double-precision populations)
  static constexpr bool STG = std::is_same<S, float>::value && TLBM_STAGE;
  template <int BY> static constexpr size_t smem() { return Geo<BY>::template smem_bytes<S, R, STG>(); }
  template <int BY> static constexpr bool fits() {
    return smem<BY>() + 1024 <= 227u * 1024u && !(std::is_same<S, double>::value && BY > 8);
  }
  template <int BY, int MODE, int VAR = 0> static cudaError_t attr() {
    if constexpr (!fits<BY>()) {
      return cudaSuccess;
    } else {
      return cudaFuncSetAttribute(lb_fused_kernel<S, BY, MODE, VAR>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem<BY>());
    }
  }
  template <int BY> static cudaError_t attr_by() {
    cudaError_t e;
    if ((e = attr<BY, MODE_STEP, 0>()) != cudaSuccess) return e;
    if ((e = attr<BY, MODE_STEP, VAR_GUO>()) != cudaSuccess) return e;
    if ((e = attr<BY, MODE_STEP, VAR_VDW>()) != cudaSuccess) return e;
    if ((e = attr<BY, MODE_STEP, VAR_GUO | VAR_VDW>()) != cudaSuccess) return e;
    if ((e = attr<BY, MODE_STEP_DIAG, 0>()) != cudaSuccess) return e;
    if ((e = attr<BY, MODE_MOMENTS, 0>()) != cudaSuccess) return e;
    return attr<BY, MODE_MOMENTS, VAR_VDW>();
  }
  static cudaError_t prepare() {
    cudaError_t e;
    if ((e = attr_by<4>()) != cudaSuccess) return e;
    if ((e = attr_by<8>()) != cudaSuccess) return e;
    if ((e = attr_by<16>()) != cudaSuccess) return e;
    return march_prepare();
  }
  template <class K> static cudaError_t kernel_info(K kernel, int nt, size_t dyn, int out[4]) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    int n = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, nt, dyn);
    if (e != cudaSuccess) return e;
    out[0] = nt; out[1] = (int)dyn; out[2] = n; out[3] = fa.numRegs;
    return cudaSuccess;
  }
  template <int BY, int VAR> static cudaError_t info_var(int out[4]) {
    if constexpr (!fits<BY>()) return cudaErrorInvalidConfiguration;
    else return kernel_info(lb_fused_kernel<S, BY, MODE_STEP, VAR>, BX * BY, smem<BY>(), out);
  }
  template <int BY> static cudaError_t info_by(int var, int out[4]) {
    switch (var) {
      case 0: return info_var<BY, 0>(out);
      case VAR_GUO: return info_var<BY, VAR_GUO>(out);
      case VAR_VDW: return info_var<BY, VAR_VDW>(out);
      default: return info_var<BY, VAR_GUO | VAR_VDW>(out);
    }
  }
  static cudaError_t info(int by, int var, int out[4]) {
    if (by == 4) return info_by<4>(var, out);
    if (by == 8) return info_by<8>(var, out);
    if (by == 16) return info_by<16>(var, out);
    return cudaErrorInvalidValue;
  }
  static bool tile_ok(int by) {
    return (by == 4 && fits<4>()) || (by == 8 && fits<8>()) || (by == 16 && fits<16>());
  }
  template <int BY, int MODE, int VAR> static cudaError_t go(const KArgs& a, dim3 grid, cudaStream_t st) {
    if constexpr (!fits<BY>()) {
      return cudaErrorInvalidConfiguration;
    } else {
      lb_fused_kernel<S, BY, MODE, VAR><<<grid, dim3(BX, BY), smem<BY>(), st>>>(a);
      return cudaGetLastError();
    }
  }
  template <int BY> static cudaError_t go_by(const KArgs& a, int mode, dim3 grid, cudaStream_t st) {
    const int var = variant_of(a.forcing, a.psi_kind);
    // the fused step + Nu sample exists for the paper's scheme only (the caller checks)
    if (mode == MODE_STEP_DIAG) return var == 0 ? go<BY, MODE_STEP_DIAG, 0>(a, grid, st) : cudaErrorInvalidValue;
    if (mode == MODE_STEP) {
      switch (var) {
        case 0: return go<BY, MODE_STEP, 0>(a, grid, st);
        case VAR_GUO: return go<BY, MODE_STEP, VAR_GUO>(a, grid, st);
        case VAR_VDW: return go<BY, MODE_STEP, VAR_VDW>(a, grid, st);
        default: return go<BY, MODE_STEP, VAR_GUO | VAR_VDW>(a, grid, st);
      }
    }
    // the moments pass has no collision: only the pseudopotential matters
    if (var & VAR_VDW) return go<BY, MODE_MOMENTS, VAR_VDW>(a, grid, st);
    return go<BY, MODE_MOMENTS, 0>(a, grid, st);
  }
  static cudaError_t fused(const KArgs& a, int mode, int by, dim3 grid, cudaStream_t st) {
    if constexpr (std::is_same<S, double>::value) {
      // FP64: the ring's moments and psi of the state read, once per node, before the step
      if (a.pre == nullptr) return cudaErrorInvalidValue;
      const unsigned blocks = ((unsigned)a.N + 255u) / 256u;
      if (a.psi_kind == PSI_VDW) lb_fields_kernel<true><<<blocks, 256, 0, st>>>(a);
      else lb_fields_kernel<false><<<blocks, 256, 0, st>>>(a);
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    if (by == 4) return go_by<4>(a, mode, grid, st);
    if (by == 8) return go_by<8>(a, mode, grid, st);
    if (by == 16) return go_by<16>(a, mode, grid, st);
    return cudaErrorInvalidValue;
  }
  // The three-kernel step (lb_split.cuh). NT threads per CTA: 256, or fewer for cells of few nodes per
  // SM, which smaller CTAs spread more evenly (the rule stands in lb_api.cu).
  template <int VAR, int NT> static cudaError_t three(const KArgs& a, int mode, cudaStream_t st) {
    const int nb = (a.plane + NT - 1) / NT;
    const unsigned grid = (unsigned)nb * (unsigned)a.nz;
    cudaError_t e;
    if ((e = follow(split_moments_kernel<S, (VAR & VAR_VDW) != 0, NT>, grid, NT, st, a, nb)) != cudaSuccess) return e;
    if (mode != MODE_MOMENTS || wants_velocity(a)) {
      if ((e = follow(split_velocity_kernel<R, VAR, NT>, grid, NT, st, a, nb)) != cudaSuccess) return e;
    }
    if (mode == MODE_STEP) return follow(split_collide_kernel<S, VAR, MODE_STEP, NT>, grid, NT, st, a, nb);
    if (mode == MODE_MOMENTS) return follow(split_collide_kernel<S, VAR & VAR_VDW, MODE_MOMENTS, NT>, grid, NT, st, a, nb);
    // the fused step + Nu sample exists for the paper's scheme only (the caller checks)
    if constexpr (VAR == 0) return follow(split_collide_kernel<S, VAR, MODE_STEP_DIAG, NT>, grid, NT, st, a, nb);
    else return cudaErrorInvalidValue;
  }
  template <int NT> static cudaError_t three_var(const KArgs& a, int mode, cudaStream_t st) {
    switch (variant_of(a.forcing, a.psi_kind)) {
      case 0: return three<0, NT>(a, mode, st);
      case VAR_GUO: return three<VAR_GUO, NT>(a, mode, st);
      case VAR_VDW: return three<VAR_VDW, NT>(a, mode, st);
      default: return three<VAR_GUO | VAR_VDW, NT>(a, mode, st);
    }
  }
  static cudaError_t split(const KArgs& a, int mode, int nt, cudaStream_t st) {
    return nt == 32 ? three_var<32>(a, mode, st) : (nt == 64 ? three_var<64>(a, mode, st) : three_var<256>(a, mode, st));
  }

  // The one-launch step (lb_march.cuh). Tile heights: measured on the 256^3 and 512^3 boiling cells,
  // FP32 7, 8, 9, 10, 12 rows: 0.99, 0.95, 1.03, 1.05, 1.13 ms and 8.0, 7.5, 7.3, 7.9, 8.5 ms; FP16
  // deviations 7, 8, 9, 12 rows: 0.78, 0.72, 0.80, 0.95 ms at 256^3; local references 5, 6, 7, 8 rows:
  // 1.30, 1.34, 1.18, 1.42 ms. Taller tiles recompute fewer ring nodes but leave fewer registers per
  // thread, and a spilled value in flight makes its warp wait for it.
  static constexpr int MTY = IsLoc<S>::v ? 7 : 8;
  // Two nodes per thread (lb_march2.cuh): 16-bit deviations, even nx, steps of the paper's scheme, sampling
  // or not: one form for all steps of a context, so that a sample does not change them.
  // Tile heights 5, 6, 7, 8 on the FP16 256^3 cell: 0.71, 0.67, 0.61, 0.76 ms (8 spills); the one-node
  // march 0.72 ms.
  static constexpr int MTY2 = sizeof(S) == 2 && !IsLoc<S>::v ? 7 : 0;
  static bool pairs(const KArgs& a, int mode, int zc2) {
    return MTY2 > 0 && zc2 > 0 && mode != MODE_MOMENTS && (a.nx & 1) == 0 && variant_of(a.forcing, a.psi_kind) == 0;
  }
  template <int VAR, int MODE> static cudaError_t march_go(const KArgs& a, const MarchArgs& b, dim3 grid, cudaStream_t st) {
    using GE = MarchGeo<S, MTY>;
    split_march_kernel<S, VAR, MODE, MTY><<<grid, GE::NT, GE::smem, st>>>(a, b);
    return cudaGetLastError();
  }
  template <int VAR, int MODE> static cudaError_t march_attr() {
    return cudaFuncSetAttribute(split_march_kernel<S, VAR, MODE, MTY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)MarchGeo<S, MTY>::smem);
  }
  static cudaError_t march_prepare() {
    if constexpr (std::is_same<S, double>::value) {
      return cudaSuccess;
    } else {
      cudaError_t e;
      if constexpr (MTY2 > 0) {
        const int smem2 = (int)March2Geo<MTY2>::smem;
        if ((e = cudaFuncSetAttribute(split_march2_kernel<S, MTY2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      smem2)) != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(split_march2_kernel<S, MTY2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      smem2)) != cudaSuccess) return e;
      }
      if ((e = march_attr<0, MODE_STEP>()) != cudaSuccess) return e;
      if ((e = march_attr<VAR_GUO, MODE_STEP>()) != cudaSuccess) return e;
      if ((e = march_attr<VAR_VDW, MODE_STEP>()) != cudaSuccess) return e;
      if ((e = march_attr<VAR_GUO | VAR_VDW, MODE_STEP>()) != cudaSuccess) return e;
      if ((e = march_attr<0, MODE_STEP_DIAG>()) != cudaSuccess) return e;
      if ((e = march_attr<0, MODE_MOMENTS>()) != cudaSuccess) return e;
      return march_attr<VAR_VDW, MODE_MOMENTS>();
    }
  }
  static cudaError_t march(const KArgs& a, int mode, int zc, int zc2, cudaStream_t st) {
    if constexpr (std::is_same<S, double>::value) {
      return cudaErrorInvalidValue;
    } else {
      MarchArgs b;
      const long long es = (long long)sizeof(S), N = a.N, plane = a.plane;
      for (int l = 0; l < Q + 2; ++l) {
        b.fdst[l] = static_cast<char*>(a.fout) + l * N * es;
        b.gdst[l] = static_cast<char*>(a.gout) + l * N * es;
      }
      for (int l = 0; l < Q; ++l) {
        const long long src = (l * N - CZ(l) * plane) * es;
        b.fsrc[l] = static_cast<const char*>(a.fin) + src;
        b.gsrc[l] = static_cast<const char*>(a.gin) + src;
      }
      for (int k = 0; k < 2; ++k) {
        b.fref[k] = static_cast<const char*>(a.fin) + (Q + k) * N * es;
        b.gref[k] = static_cast<const char*>(a.gin) + (Q + k) * N * es;
      }
      if constexpr (MTY2 > 0) {
        if (pairs(a, mode, zc2)) {
          using GE = March2Geo<MTY2>;
          b.tiles_x = (a.nx + GE::TX - 1) / GE::TX;
          b.zc = zc2;
          const dim3 grid((unsigned)(b.tiles_x * ((a.ny + MTY2 - 1) / MTY2)), (unsigned)((a.nz + zc2 - 1) / zc2));
          if (mode == MODE_STEP) split_march2_kernel<S, MTY2, false><<<grid, GE::NT, GE::smem, st>>>(a, b);
          else split_march2_kernel<S, MTY2, true><<<grid, GE::NT, GE::smem, st>>>(a, b);
          return cudaGetLastError();
        }
      }
      b.tiles_x = (a.nx + BX - 1) / BX;
      b.zc = zc;
      const dim3 grid((unsigned)(b.tiles_x * ((a.ny + MTY - 1) / MTY)), (unsigned)((a.nz + zc - 1) / zc));
      const int var = variant_of(a.forcing, a.psi_kind);
      if (mode == MODE_MOMENTS)
        return (var & VAR_VDW) ? march_go<VAR_VDW, MODE_MOMENTS>(a, b, grid, st) : march_go<0, MODE_MOMENTS>(a, b, grid, st);
      if (mode == MODE_STEP_DIAG)
        return var == 0 ? march_go<0, MODE_STEP_DIAG>(a, b, grid, st) : cudaErrorInvalidValue;
      switch (var) {
        case 0: return march_go<0, MODE_STEP>(a, b, grid, st);
        case VAR_GUO: return march_go<VAR_GUO, MODE_STEP>(a, b, grid, st);
        case VAR_VDW: return march_go<VAR_VDW, MODE_STEP>(a, b, grid, st);
        default: return march_go<VAR_GUO | VAR_VDW, MODE_STEP>(a, b, grid, st);
      }
    }
  }
  template <int VAR> static cudaError_t step_info_var(int form, int nt, int out[4]) {
    if (form == STEP_THREE) {
      if (nt == 32) return kernel_info(split_collide_kernel<S, VAR, MODE_STEP, 32>, 32, 0, out);
      if (nt == 64) return kernel_info(split_collide_kernel<S, VAR, MODE_STEP, 64>, 64, 0, out);
      return kernel_info(split_collide_kernel<S, VAR, MODE_STEP, 256>, 256, 0, out);
    }
    if constexpr (!std::is_same<S, double>::value) {
      using GE = MarchGeo<S, MTY>;
      if (form == STEP_MARCH) return kernel_info(split_march_kernel<S, VAR, MODE_STEP, MTY>, GE::NT, GE::smem, out);
      if constexpr (MTY2 > 0 && VAR == 0) {
        using G2 = March2Geo<MTY2>;
        if (form == STEP_MARCH2) return kernel_info(split_march2_kernel<S, MTY2, false>, G2::NT, G2::smem, out);
      }
    }
    return cudaErrorInvalidValue;
  }
  static cudaError_t step_info(int form, int nt, int var, int out[4]) {
    switch (var) {
      case 0: return step_info_var<0>(form, nt, out);
      case VAR_GUO: return step_info_var<VAR_GUO>(form, nt, out);
      case VAR_VDW: return step_info_var<VAR_VDW>(form, nt, out);
      default: return step_info_var<VAR_GUO | VAR_VDW>(form, nt, out);
    }
  }
  static int blocks_for(int N) {
    long long b = ((long long)N + 255) / 256;
    return (int)(b < 4096 ? (b < 1 ? 1 : b) : 4096);
  }
  static cudaError_t init(const KArgs& a, const double* rho, const double* T, cudaStream_t st) {
    lb_init_kernel<S><<<blocks_for(a.N), 256, 0, st>>>(a, rho, T);
    return cudaGetLastError();
  }
  static cudaError_t setpops(const KArgs& a, const double* f, const double* g, cudaStream_t st) {
    lb_setpops_kernel<S><<<blocks_for(a.N), 256, 0, st>>>(a, f, g);
    return cudaGetLastError();
  }
  static cudaError_t pops(const KArgs& a, double* f, double* g, cudaStream_t st) {
    lb_pops_kernel<S><<<blocks_for(a.N), 256, 0, st>>>(a, f, g);
    return cudaGetLastError();
  }
};

}  // namespace tlbm
