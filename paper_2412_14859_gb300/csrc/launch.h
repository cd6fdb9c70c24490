// launch.h -- host-side launchers of the CUDA kernels (implemented in the .cu files).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace cgevap {

// Tile shapes of the fused step, chosen per lattice by the launch planner / autotuner.
struct TileCfg {
  int tx, ty;
};
constexpr int kNumTiles3D = 5;
constexpr TileCfg kTiles3D[kNumTiles3D] = {{32, 4}, {16, 8}, {16, 16}, {16, 4}, {32, 8}};
constexpr int kNumTiles2D = 2;
constexpr TileCfg kTiles2D[kNumTiles2D] = {{128, 1}, {64, 1}};

inline TileCfg tile_cfg(int q, int variant) {
  return q == 19 ? kTiles3D[variant % kNumTiles3D] : kTiles2D[variant % kNumTiles2D];
}
inline int num_tile_variants(int q) { return q == 19 ? kNumTiles3D : kNumTiles2D; }

// Fused step kernels (step_f64.cu, step_f32.cu, step_dev.cu): the __global__ function of a
// (lattice, storage, tile variant), launched with `threads` threads and one StepArgs argument.
struct KernelRef {
  const void* fn;     // any lattice of that kind
  int threads;
  int smem = 0;       // dynamic shared memory bytes
  int tx = 0, ty = 0; // tile shape (0: take it from tile_cfg)
  int needs_map = 0;  // 1: second kernel argument is the TMA tensor map of the input state
  int shares = 0;               // 1: can divide the tiles' planes evenly (StepArgs::pc = 0)
  int pdl = 0;                  // 1: may be launched ahead of its predecessor's end (it waits itself)
  const void* plain = nullptr;  // the same step without links, site bytes read or a flux field
};
// The instantiation that runs step arguments a.
inline const void* step_fn(const KernelRef& k, const StepArgs& a) {
  return k.plain && !a.g.links && a.ph.rule == 1 && !a.ph.phi_field ? k.plain : k.fn;
}
// Launches a step kernel; a kernel that waits for its predecessor itself is launched ahead of it.
inline cudaError_t launch_step(const KernelRef& k, const StepArgs& a, dim3 grid, void** args, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)k.threads);
  cfg.dynamicSmemBytes = (size_t)k.smem;
  cfg.stream = s;
  cudaLaunchAttribute ahead;
  ahead.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  ahead.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &ahead;
  cfg.numAttrs = k.pdl ? 1u : 0u;
  return cudaLaunchKernelExC(&cfg, step_fn(k, a), args);
}
// How a tiled kernel's planes are divided among `slots` resident CTAs: in chunks of pc planes (the
// time is about waves x (pc + 2) planes, the two extra ones pulled at each chunk's ends), or, pc = 0
// and `shares` CTAs, evenly across tile ends (share + 2 planes per piece of a tile; for_planes).
struct MarchPlan {
  int pc, nchunk, shares;
};
// extra: the weight of the planes pulled in all, which breaks near ties towards fewer extra planes.
// Measured with 0.36 against 0, us a step: FP32 128^3 122.7 (chunks of 32) / 126.5 (15),
// 256 x 256 x 128 with walls 466 (128) / 483 (16), 176^3 315 (88) / 310 (20), eight other sizes the
// same plan; F16RC 128^3 185 / 191; F16DEV 128^3 181 / 176, so the deviation storages plan with 0.
constexpr double kExtraPlanes = 0.36;
inline MarchPlan plan_march(long long tiles, int nm, long long slots, bool can_share, double extra = kExtraPlanes) {
  MarchPlan best{nm, 1, 0};
  double cost = 1e300;
  for (int pc = 1; pc <= nm; ++pc) {
    const long long nchunk = (nm + pc - 1) / pc;
    if (nchunk > 65535) continue;
    const long long waves = (tiles * nchunk + slots - 1) / slots;
    const double c = (double)waves * (pc + 2) + extra * (double)(tiles * nchunk) * (pc + 2) / (double)slots;
    if (c < cost - 1e-9) {
      cost = c;
      best = MarchPlan{pc, (int)nchunk, 0};
    }
  }
  if (can_share && tiles * nm > slots) {
    const long long share = (tiles * nm + slots - 1) / slots;
    const long long pieces = nm % share == 0 ? 1 : (share - 1) / nm + 2;
    // by more than the model's own error
    if ((1.0 + extra) * (double)(share + 2 * pieces) < 0.98 * cost) best = MarchPlan{0, 1, (int)slots};
  }
  return best;
}
KernelRef step_kernel_f64(int q, int variant);
KernelRef step_kernel_f32(int q, int variant);
KernelRef step_kernel_f32x(int q, int variant);  // FP32 pairs, exact colour masses (step_f32.cu)
// D2Q9 step of the pair storages without a march (pair_tile.cuh), for a lattice of that many cells.
KernelRef patch_kernel_f64(long long cells);
KernelRef patch_kernel_f32(int storage, long long cells);  // ST_F32 or ST_F32X
KernelRef step_kernel_dev(int q, int storage, int variant);
// Recolour-on-pull layout (step_rc.cu); pairs_in: the input state holds FP32 pairs (import).
KernelRef step_kernel_rc(int q, int variant, bool pairs_in);
// 16-bit recolour-on-pull layouts (step_rc16.cu); storage is ST_H16RC or ST_B16RC.
KernelRef step_kernel_rc16(int q, int storage, int variant, bool pairs_in);
// TMA-pipelined step (step_tma_f32.cu): FP32 storage; periodic axes need >= 4 cells.
constexpr int kNumTmaVariants3D = 2;
constexpr int kNumTmaVariants2D = 2;
KernelRef step_tma_f32(int q, int variant);
// TMA tensor map (128-byte CUtensorMap written to `map`) of one population buffer: elements of
// elem_bytes, box of box_w x box_h (x, rows) per direction and plane.  Returns 0 on success.
int make_pop_tensor_map(void* map, const void* base, const Geom& g, int q, int elem_bytes,
                        int box_w, int box_h);

// Auxiliary kernels (aux_kernels.cu).
struct AuxArgs {
  Geom g;
  Physics ph;
  int q, storage;
  double rho_r_in, rho_b_in;
};
cudaError_t launch_init_equilibrium(const AuxArgs& a, const double* rhoN0, const void* noise,
                                    int noise_dtype, void* state, cudaStream_t s);
cudaError_t launch_set_populations(const AuxArgs& a, const void* in, int dtype, void* state,
                                   cudaStream_t s);
cudaError_t launch_get_populations(const AuxArgs& a, const void* state, void* out, int dtype,
                                   cudaStream_t s);
cudaError_t launch_macros(const AuxArgs& a, const void* state, double* rho_r, double* rho_b,
                          double* u, double* rhoN, cudaStream_t s);
cudaError_t launch_gradient_sites(const AuxArgs& a, const void* state, double* tmp_rn,
                                  uint8_t* mask, cudaStream_t s);
cudaError_t launch_links(const AuxArgs& a, const uint8_t* solid, uint32_t* links,
                         cudaStream_t s);
cudaError_t launch_zero_solid(const AuxArgs& a, void* state, cudaStream_t s);
cudaError_t launch_health(const AuxArgs& a, const void* state, int* flag, cudaStream_t s);
cudaError_t launch_fill_ghosts(const AuxArgs& a, void* state, cudaStream_t s);
cudaError_t launch_convert_field(const void* in, int in_dtype, void* out, int out_is_double,
                                 long long n, cudaStream_t s);
cudaError_t launch_fill(double* out, double v, long long n, cudaStream_t s);
// Blue pressure outlets (aux_kernels.cu; Sec. III.B.2) on the first / last plane of the march
// axis, prescribed blue density rho_lo / rho_hi (<= 0: wall), written into state before a step.
cudaError_t launch_outlets(const AuxArgs& a, void* state, double rho_lo, double rho_hi, cudaStream_t s);

// Heated-substrate flux field (aux_kernels.cu; Sec. III.C, Eq. heated): every cell of a column
// along the march axis (the wall normal) takes phi_s / (K + h / length), h = the column's summed
// liquid fraction.  `part` holds (heated_plan(g).nchunk + 1) * na * nb doubles; field is double
// (field_double = 1) or float, [N].
struct HeatedPlan {
  int col_blocks = 1, cz = 1, nchunk = 1;
};
HeatedPlan heated_plan(const Geom& g);
cudaError_t launch_heated_flux(const AuxArgs& a, const void* state, double* part, double phi_s,
                               double K, double length, void* field, int field_double, cudaStream_t s);

// Adjoint sweep (adjoint_kernels.cu).  The local kernel (kernel A) takes (StepArgs, AdjointOut)
// and runs on the step's tile grid; F64 / F32 storage only.
// Auxiliary per-cell fields of the sweep, five reals for each of nstore cells (AuxCell): dL/dF_a,
// dL/dF_b, dL/dF_m and d rho^N/d rho_r side by side, then the plane of d rho^N/d rho_b.
constexpr int kAdjAuxPlanes = 5;
struct AdjointOut {
  const void* lam_in;  // the lg part of lambda^{n+1} = dL/df^{n+1}, pushed by the previous
                       // adjoint step (state layout: vec2 per direction and storage index)
  const void* ab;      // the ab part of lambda^{n+1}: nstore vec2 from kernel B1 of that step
  void* lam_g;         // out: the lg part of lambda^n, pushed to where the pull of step n read
  void* aux;           // out: kAdjAuxPlanes planes
};
KernelRef adjoint_local_kernel(int q, int storage);
// Kernel B1: stencil transpose, exchange derivative into dphi (FP64, compact [N]); aux holds
// kAdjAuxPlanes planes of nstore reals; lam_g is kernel A's pushed output (its rest slot of a
// cell is that cell's own lg_0); ab receives nstore vec2.  dLdV may be nullptr.
cudaError_t launch_adjoint_stencil(const AuxArgs& a, const void* aux, const void* lam_g, void* ab,
                                   const uint8_t* mask, double* dphi, double inv_sbar,
                                   const double* dLdV, cudaStream_t s);
// Liquid volume of a state into *out (FP64); part holds kVolumeBlocks doubles, *done starts at 0.
constexpr int kVolumeBlocks = 152 * 16;  // 16 CTAs of 256 threads per SM: loads in flight
cudaError_t launch_volume(const AuxArgs& a, const void* state, double* part, unsigned int* done,
                          double* out, cudaStream_t s);

}  // namespace cgevap
