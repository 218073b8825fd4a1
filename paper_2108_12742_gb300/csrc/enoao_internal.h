// Internal declarations shared by the host runtime and the kernels of the
// ENO-AO library (not part of the public C interface).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace enoao {

constexpr int kMaxNv = 5;

// Device-resident time-stepping state.  Written by the step kernels, read by
// every sweep launch, so alpha and dt never travel to the host inside a step.
struct StepState {
  double alpha[3];          // Lax-Friedrichs alpha per axis of the current step
  double dt;                // current step size
  double t;                 // time at the start of the current step
  double t_end;             // target time of enoao_advance (inf for step counts)
  double cfl;               // CFL number (dt = cfl / sum alpha_d / dx_d)
  double dt_fixed;          // > 0: fixed step size instead of the CFL rule
  long long steps;          // completed steps
  long long max_steps;      // stop after this many steps (<= 0: none)
  int skip;                 // 1: the current step is not taken (done / limit)
  int last;                 // 1: the current step lands on t_end
  int done;                 // 1: t_end reached
  int pending;              // 1: a step was begun and is not yet finalised
  unsigned long long alpha_acc[2][3];  // running max of |u_d| + c (bit patterns);
                                       // step n reads [n % 2], its last stage fills [par]
  int par;                  // alpha_acc slot the current step's last stage fills
  int err;                  // error bits (kErrNonPhys, kErrTimeout, kErrRedoFull)
  long long err_cell;       // first cell (min index) that raised kErrNonPhys
  unsigned long long fallbacks;  // FP32-bulk decisions re-done in FP64
  unsigned long long decisions;  // stencil decisions taken
  unsigned long long tile_next;  // dynamic tile queue of the running sweep launch
  unsigned int blocks_done;      // blocks of the running sweep launch that have left it
  unsigned int redo_n;            // faces listed for FP64 re-decision by the running sweep
  unsigned long long alpha_stage[3];  // per-stage alpha: running max over the
                                      // state stage 0 or 1 writes (bit patterns)
  unsigned int redo_epoch;        // sweeps that listed faces: tags the changed-face marks
  unsigned int redo_done;         // blocks of the running apply pass that have left it
  unsigned int grid_count, grid_gen;  // the grid barrier of the persistent 1D run
  // per-field alpha (Euler): per axis max |u_d - c|, max |u_d|, max |u_d + c|
  double alpha_f[3][3];                   // of the current step
  unsigned long long alpha_acc_f[2][3][3];  // running maxima (bit patterns), as alpha_acc
};


// Ghost cells along the split axis of a sub-domain are layers of the state
// arrays themselves (filled by halo exchange), read as they are.
constexpr int kBcHalo = 2;

constexpr int kErrNonPhys = 1;
constexpr int kErrTimeout = 2;
constexpr int kErrRedoFull = 4;  // re-decision list full (cannot happen: one slot per face)
constexpr int kErrBarrier = 8;   // a block of a persistent 1D run gave up at the grid barrier:
                                 // the pending step is not complete

// Modes of a sweep launch (bit set).
constexpr int kModeRhsStore = 1;   // write this axis' L(u) into rhs
constexpr int kModeRhsAdd = 2;     // add the stored rhs of earlier axes
constexpr int kModeCombine = 4;    // Runge-Kutta combine into u_out
constexpr int kModeAlpha = 8;      // accumulate alpha of u_out: for the next step
                                   // (stage 2) or the next stage (stages 0, 1)
constexpr int kModeFlux = 16;      // write interface fluxes (and choices)

// The arrays of a sweep by component, in sweep order (momentum along the
// swept axis first, tangential momenta cyclic): set_component_pointers.  Kernels
// address a cell as one multiply-add onto these.
struct ComponentPtrs {
  const double* u_in[kMaxNv];
  const double* u0[kMaxNv];
  double* u_out[kMaxNv];
  void* rhs[kMaxNv];
  const float* inc_in[kMaxNv];
  float* inc_out[kMaxNv];
};

// Shapes of a sweep kernel: the axis class and mode it is compiled for (the
// first axis stores L(u), later ones add theirs, the last one combines; 1D
// combines at once).  Sizes, stage, boundary and alpha stay arguments.  One
// kernel for every mode kept the values of all of them live and recomputed
// under the register cap; the compiled shapes issue a fifth fewer instructions.
enum SweepShape {
  kShapeAny = 0,   // everything from the arguments (per-field, TMA staging)
  kShapeXStore,
  kShapeXCombine,
  kShapeYStore,    // y or z, adding to the earlier axes
  kShapeYCombine,
  kShapeFlux       // interface fluxes, any axis
};
inline int sweep_shape(int dir, int mode) {
  if (mode & kModeFlux) return kShapeFlux;
  if (mode == kModeRhsStore) return dir == 0 ? kShapeXStore : kShapeAny;
  if (mode == (kModeRhsStore | kModeRhsAdd)) return dir > 0 ? kShapeYStore : kShapeAny;
  const int m = mode & ~kModeAlpha;
  if (m == kModeCombine) return dir == 0 ? kShapeXCombine : kShapeAny;
  if (m == (kModeCombine | kModeRhsAdd)) return dir > 0 ? kShapeYCombine : kShapeAny;
  return kShapeAny;
}

// How a tile's re-decisions are split over the warps of its block (redecide_tile):
// for the least work in all (batches), ending sooner for little more (sweeps), or
// soonest (launches with no more tiles than SMs).
enum RedoSplit { kSplitDense, kSplitSweep, kSplitAll };

struct SweepArgs {
  ComponentPtrs comp;
  const double* u_in;   // U^(s): stencil source, [nv][N]
  const double* u0;     // U^n for the Runge-Kutta combine
  double* u_out;        // combined state
  void* rhs;            // accumulated L(u) of earlier axes ([nv][N], bulk type)
  const float* inc_in;  // FP32 bulk combine: the FP32 stage increment of the previous
                        // stage ([nv][N], stages 1 and 2: I0 = dt L(U^n), I1 = I0 + dt L(U1))
  float* inc_out;       // FP32 bulk combine: this stage's increment (stages 0 and 1)
  double* fhat;         // kModeFlux: interface fluxes [nv][faces]
  int8_t* idx_out;      // kModeFlux: choices [nv][2][faces] (nullable)
  unsigned long long* redo;  // FP32 bulk, stepping: faces listed for the grid-wide FP64
                        // re-decision pass (face index << 16 | flagged choices, bit
                        // field * 2 + sign), a slot per face of the axis; null: the
                        // sweep re-decides its near-ties itself
  float* redo_dc;       // per listed face: change of its correction C (nv, sweep order)
  unsigned* redo_mark;  // per face of the axis: redo_epoch when its correction changed
  double redo_coef;     // weight of dt L(u) in the stage's combine (1, 1/4, 2/3)
  long long redo_cap;   // slots of redo
  StepState* st;
  long long n[3];       // cells per axis
  long long ncell;      // total cells
  long long nfaces;     // faces of the swept axis, ncell / nd * (nd + 1) (flux output layout)
  long long cstride;    // distance between two conserved components in the state arrays
  long long org;        // array cell of the first interior cell (sub-domains keep ghost
                        // layers in their arrays along the split axis; 0 otherwise)
  int ndim;
  int dir;              // swept axis
  int bc;               // boundary condition along dir (kBcHalo: ghosts stored in the arrays)
  int mode;
  int stage;            // Runge-Kutta stage 0..2
  int ta, ts;           // tile: lines x faces
  int se;               // shared-memory row pitch in cells (sweep_row_pitch)
  int field;            // 1: per-field splitting constants (st->alpha_f), Euler only
  int tma_box;          // TMA: box extent along the swept axis (cells, with alignment slack)
  unsigned tma_bytes;   // TMA: bytes of one box
  int tma_raw_bytes;    // TMA: shared memory reserved for the box (a multiple of 128)
  int redo_split;       // FP32 bulk: how a tile's re-decisions go to its warps (RedoSplit)
  int redo_passes;      // FP32 bulk: bound on the in-sweep re-decision passes of a warp
                        // round; reaching it sets kErrTimeout (64 nv by default)
  long long tiles_s;    // tiles along dir
  long long tiles_a;    // tiles across the line index
  long long tiles_b;    // tiles along the remaining axis (dir != 0)
  long long ntiles;
  double inv_dx;        // 1 / dx along dir
  double dx_all[3];     // dx per axis (alpha accumulation needs none, kept for checks)
  double gamma;
  double adv_speed;
  double delta;
  double tie_rel;
  // gamma - 1 in FP64 and the constants in FP32 (FP32 bulk), set from the
  // fields above by set_derived_constants wherever they are set: kernels read
  // them from the parameter space instead of narrowing them themselves, which
  // the compiler may redo at every use (a conversion on the FP64 unit each).
  double gm1;
  float gm1_f, adv_f, delta_f, tie_rel_f, inv_dx_f;
};

// Derived constants of a SweepArgs (round to nearest, as the device would).
__host__ __device__ inline void set_derived_constants(SweepArgs& a) {
  a.gm1 = a.gamma - 1.0;
  a.gm1_f = (float)a.gm1;
  a.adv_f = (float)a.adv_speed;
  a.delta_f = (float)a.delta;
  a.tie_rel_f = (float)a.tie_rel;
  a.inv_dx_f = (float)a.inv_dx;
}

// Component pointers of a SweepArgs from its arrays, ndim, dir, cstride and the
// bulk precision (fp32: element size of rhs).
__host__ __device__ inline void set_component_pointers(SweepArgs& a, bool fp32) {
  for (int c = 0; c < kMaxNv; ++c) {
    const int k = c >= 1 && c <= a.ndim ? 1 + (a.dir + c - 1) % a.ndim : c;
    const long long off = a.cstride * k;
    a.comp.u_in[c] = a.u_in + off;
    a.comp.u0[c] = a.u0 + off;
    a.comp.u_out[c] = a.u_out + off;
    a.comp.rhs[c] = static_cast<char*>(a.rhs) + off * (fp32 ? 4 : 8);
    a.comp.inc_in[c] = a.inc_in + off;
    a.comp.inc_out[c] = a.inc_out + off;
  }
}

// Host-side interface of the instantiation units.

// The sweep kernel for a system, order, shape and variant, or NULL: FP32 bulk
// re-deciding its near-ties in the sweep, the same with raw tiles staged by
// TMA, FP32 bulk listing them for the grid-wide pass, FP64, and either
// precision with per-field splitting constants (Euler systems).
enum SweepVariant { kSweepFp32, kSweepFp32Tma, kSweepFp32List, kSweepFp64, kSweepFp32Field, kSweepFp64Field };
const void* sweep_kernel_for(int nv, int order, int shape, int variant);
// by instantiation unit
const void* sweep_fp32_o5(int nv, int shape, int variant);
const void* sweep_fp32_o7(int nv, int shape, int variant);
const void* sweep_fp32_list_o5(int nv, int shape);
const void* sweep_fp32_list_o7(int nv, int shape);
const void* sweep_fp64(int nv, int order, int shape);
const void* sweep_fp32_field(int nv, int order);
const void* sweep_fp64_field(int nv, int order);
// the fused 2D stage kernel (both axes in one launch; FP32 bulk, nv 1 or 4)
const void* fused2d_kernel_for(int nv, int order);
cudaError_t redo_launch_fp32(int nv, int order, const SweepArgs& a, int grid, cudaStream_t s);

// tmap: the stencil source as a tensor map for TMA staging, or NULL.
inline cudaError_t sweep_launch(const void* kernel, const SweepArgs& a, int grid, int block,
                                size_t smem, cudaStream_t s, const CUtensorMap* tmap = nullptr) {
  CUtensorMap none{};  // direct loads: the map is not read
  void* args[2] = {const_cast<SweepArgs*>(&a), tmap ? const_cast<CUtensorMap*>(tmap) : &none};
  return cudaLaunchKernel(kernel, dim3(grid), dim3(block), args, smem, s);
}

// Raises a kernel's dynamic shared-memory limit to at least smem, never
// lowers it: the limit belongs to the kernel, not to one launch, and the
// axes and tiles of one kernel (and launches captured earlier into a graph)
// need different sizes.
inline cudaError_t raise_smem_limit(const void* kernel, size_t smem) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  if ((size_t)fa.maxDynamicSharedSizeBytes >= smem) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// Readies a kernel for smem bytes of dynamic shared memory and gives the
// blocks of it that share an SM.
inline cudaError_t sweep_setup(const void* kernel, int block, size_t smem, int* per_sm) {
  if (!kernel) return cudaErrorInvalidValue;
  cudaError_t e = raise_smem_limit(kernel, smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kernel, block, smem);
  return e;
}

// Cell slots of a tile's shared-memory planes: a multiple of four, so that
// every plane starts on a 16-byte boundary.
__host__ __device__ constexpr int tile_cells(int ta, int se) { return (ta * se + 3) & ~3; }

// Row pitch (cells) of a tile's shared-memory rows.  x sweeps read along a
// row (any pitch); y/z sweeps put lines on lanes, so the pitch must spread a
// warp's lanes over distinct banks: odd for 32- and 64-line tiles, for 8-byte
// elements and for FP32 Euler cells (16-byte vectors:
// each quarter-warp access then covers eight distinct 16-byte bank groups),
// 2 (mod 4) for 16-line FP32 tiles kept in planes (a warp spans two cells of 16 lines).
inline int sweep_row_pitch(int nv, int order, int fp32, int dir, int ta, int ts, int field = 0) {
  const int G = order / 2 + 2;
  int se = ts + 2 * G;
  if (dir == 0) return se;
  if (fp32 && ta == 16 && (nv == 1 || (field && nv != 4))) {
    while (se % 4 != 2) ++se;
  } else {
    if (se % 2 == 0) ++se;
  }
  return se;
}

// Dynamic shared memory of one sweep block: per extended cell the split
// differences and the face correction (three vectors), the Roe ingredients
// (Euler equations), in FP32 bulk with one splitting constant the magnitude of
// the pair's differences, and a word of the face list.  The FP32
// vectors of the 1D system are four values wide, the spare ones taking the
// magnitude and two of its Roe ingredients.
inline size_t sweep_smem_bytes(int nv, int fp32, int ta, int se, int field = 0) {
  const size_t cells = (size_t)tile_cells(ta, se);
  const int prims = nv > 1 ? nv : 0;
  if (!fp32) return cells * ((size_t)(3 * nv + prims) * 8 + 4);
  if (field) return cells * (size_t)(4 * nv + 1) * 4;
  return cells * (size_t)(nv == 3 ? 14 : 3 * nv + prims + 2) * 4;
}

}  // namespace enoao
