// Host-side launch entry points of the batched kernels (one translation unit
// per spinor precision instantiates them).
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "batch.cuh"

namespace lqcd {

// Link storage precision paired with a spinor precision.
inline int link_prec_for(int sp) { return (sp == P_F64 || sp == P_F32 || sp == P_DF64) ? sp : P_F16; }

// grid <= 0: persistent grid of the autotuned CTAs per SM (else the occupancy limit);
// form < 0: the autotuned Dslash form (else the default), 0 site, 1 colour split,
// 3 site at the second register budget (FP32 only; other precisions take form 0).
cudaError_t launch_dslash(int sp, int nr, bool dag, int epi, const Launch& L, int grid,
                          cudaStream_t s, int form = -1);
// tp: precision of the FP64-class operand of the mixed ops (P_F64 or P_DF64)
cudaError_t launch_blas(int sp, int op, const Launch& L, int grid, cudaStream_t s, int tp = P_F64);
// k_finish for a launch whose slots reduce or finish (finish.cu); launch_dslash and
// launch_blas issue it themselves when L.finish is set
cudaError_t launch_finish(const Launch& L, cudaStream_t s);

// per precision
#define LQCD_DECL(SFX)                                                                     \
  cudaError_t launch_dslash_##SFX(int nr, bool dag, int epi, const Launch& L, int grid,   \
                                  cudaStream_t s, int form);                               \
  int dslash_occupancy_##SFX(int nr, int form);                                            \
  cudaError_t launch_blas_##SFX(int op, int tp, const Launch& L, int grid, cudaStream_t s);
LQCD_DECL(f64)
LQCD_DECL(f32)
LQCD_DECL(f16)
LQCD_DECL(bf16)
LQCD_DECL(df64)
#undef LQCD_DECL

// Launches of the batched kernels, with programmatic stream serialization where enabled:
// the kernel may then be launched before the previous kernel on the stream completes, and
// waits for it itself (pdl_wait in batch.cuh). Enabled for operator launches and for the
// step chains of small solves; disabled while a PdlSolverScope(true) is alive on the calling
// thread, which the solvers open when their launches hold more than PDL_SOLVER_MAX_TILES
// tiles; LQCD_PDL=1 / 0 forces it on / off everywhere.
bool pdl_enabled();
struct PdlSolverScope {
  explicit PdlSolverScope(bool off);
  ~PdlSolverScope();
  PdlSolverScope(const PdlSolverScope&) = delete;
  PdlSolverScope& operator=(const PdlSolverScope&) = delete;
  bool off_;
};
// Measured on GB300: in solver step chains of up to about two tiles per resident CTA (8^4 to
// 16^3x32 one slot at a time, the 16^3x32 HMC) the programmatic launch hides launch latency
// (one-by-one small solves 9% faster, HMC 2%); in larger ones it costs up to 10% (the
// 32^3x64 double-float CG, the 64-lattice engine 6%).
constexpr long long PDL_SOLVER_MAX_TILES = 2048;
inline bool pdl_solver_off(long long tiles) { return tiles > PDL_SOLVER_MAX_TILES; }
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t dyn_smem, cudaStream_t s,
                     Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = dyn_smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// The next launch of this thread is an ordinary one (true): programmatic dependence is
// between kernels, and what it follows in a captured graph is another kind of node.
void pdl_skip_next(bool skip);

// Bytes of the link copy that fields of precision sp (FP32, FP16, BF16) read
inline size_t link_copy_bytes(int sp, int nr, int Vh) { return (size_t)2 * 4 * nr * Vh * (sp == P_F32 ? 4 : 2); }

// Launch::stream_links (single-slot launches: the rule itself): the links are read past L1, by
// slots of `gauges` different gauge fields with link_bytes of links in all. Measured on GB300,
// past L1 against through it, us a call:
//  - Up to 58 MiB, which L2 still holds beside the spinors, L1 saves L2 traffic: M-hat FP32-18
//    16^3x32 16.9 / 15.2, 18^3x36 (58 MiB) 30.2 / 27.2, FP16-12 16^3x64 28.0 / 23.4, 24^3x36
//    (46 MiB) 42.1 / 41.1.
//  - Above it L1 finds nothing again: FP32-12 20^3x40 (59 MiB) 35.0 / 36.6, 24^3x48 68.5 / 74.3
//    (its CG 22.5 / 23.5 ms), FP16-12 24^3x48 (61 MiB) 51.2 / 53.9, FP16-18 there 50.8 / 56.0,
//    BF16-18 64.9 / 70.5, five to ten 16^3x32 FP16 fields in a batch 1-7% less.
//  - Above 256 MiB, twice L2, HBM bounds both, and rows that start off a sector boundary gain by
//    L1: FP32-18 28^3x56 158.5 / 155.1, FP16-18 32^3x64 157.1 / 156.3.
//  - Slots that share a gauge field find each other's links in L1 at every size: 24^3x48 with 12
//    sources, FP16-12 258 / 247, FP32-12 280 / 245.
//  - FP32 batches over several gauge fields take no upper bound (ten 16^3x32, 18 reals, 81.0 /
//    81.8), and go past L1 also where some slots share one.
inline bool stream_links(int sp, int slots, int gauges, size_t link_bytes) {
  constexpr size_t MIB = (size_t)1 << 20;
  if (sp != P_F32 && sp != P_F16 && sp != P_BF16) return false;
  if (sp == P_F32 && gauges > 1) return link_bytes > 64 * MIB;
  return gauges == slots && link_bytes > 58 * MIB && link_bytes <= 256 * MIB;
}

// Counts changes of what decides a launch's shape (tuner table, grid caps, kernel form): a
// captured graph is good for as long as it stands.
unsigned launch_config_epoch();
void launch_config_changed();

// Number of SMs of the current device and the persistent-grid multiplier.
int device_sm_count();
void set_grid_multiplier(int kernel_family, int mult);  // 0 = occupancy limit
// ctas_per_sm > 0 caps the grid below the occupancy limit (autotuned choice)
int grid_for(const void* kernel_fn, int ntiles, int family, int block, int ctas_per_sm = 0);
int kernel_occupancy(const void* kernel_fn, int block);
// resident CTAs per SM of the Dslash of this precision, link reals and form (0 if no such
// form): 0 one thread per site, 1 colour split (double-float), 2 shared-link multi-RHS,
// 3 one thread per site at 8 CTAs per SM (FP32)
int dslash_occupancy(int sp, int nr, int form);

// Autotuner table (tune.cu): the launch choice for Dslash launches of this precision and
// link reals whose tile count has the same floor(log2) as a tuned launch.
struct TuneChoice {
  int ctas_per_sm;  // 0: occupancy limit
  int form;         // 0 site, 1 colour split, 3 site at the second register budget
};
TuneChoice tune_choice(int sp, int nr, int ntiles);
// Shared-link choice for nrhs slots on one gauge field of `blocks` site blocks: the tuned
// slots per group (0: every slot loads its own links), with *ctas_per_sm the tuned grid
// (0: occupancy limit); -1 when nothing was tuned for the key.
int tune_shared_links(int sp, int nr, int nrhs, int blocks, int* ctas_per_sm);

// Whether the Dslash of spinor precision prec uses the colour-split form (double-float
// only; a runtime switch for measurement).
bool dslash_colour_split(int prec);
void set_dslash_colour_split(int prec, bool on);

// The Dslash form without a tuned choice (for FP32 a rule of waves: tune.cu)
int default_dslash_form(int prec, int nr, int ntiles);

// layout kernels (layout.cu)
// (the AoS arrays need the alignment of their FP64 reals only)
cudaError_t links_from_aos(const double* d_aos, const Geom& g, double2* d_U, cudaStream_t s);
cudaError_t links_to_aos(const double2* d_U, const Geom& g, double2* d_aos, cudaStream_t s);
cudaError_t master_from_df(double2* d_U, const float4* d_Ud, const Geom& g, cudaStream_t s);
cudaError_t gauge_convert(const void* d_f64_18, const Geom& g, int prec, int nr, void* d_out,
                          cudaStream_t s);
cudaError_t spinor_from_aos(const double* d_aos, const Geom& g, int prec, void* d_even,
                            void* d_odd, cudaStream_t s);
cudaError_t spinor_to_aos(const void* d_even, const void* d_odd, const Geom& g, int prec,
                          double* d_aos, cudaStream_t s);
cudaError_t spinor_convert(const void* d_in, int pin, void* d_out, int pout, int Vh, double scale,
                           cudaStream_t s);

}  // namespace lqcd
