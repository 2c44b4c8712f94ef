// Host-side launch functions shared between translation units of libscatter.
#pragma once

#include "plan.h"

namespace scatter {

// A call's choice on the device: kernels that stand by for crystals past a plan's
// assumed radius return at once while this call's extent squared (rmax2, float
// bits, per instance) is within lim2; those of a node set also where it is not
// within the set's own (only2, one instance).
struct CallGate {
  const unsigned* rmax2;  // null: no gate
  const float* lim2;      // null: nothing smaller serves
  int n;                  // instances
  const float* only2;     // null: no bound of its own
};
#ifdef __CUDACC__
__device__ __forceinline__ bool within(const CallGate& g, int inst) {
  if (!g.rmax2) return false;
  const float r2 = __uint_as_float(g.rmax2[inst]);
  return (g.lim2 && r2 <= g.lim2[inst]) || (g.only2 && !(r2 <= g.only2[inst]));
}
#endif

// Per-call position preparation (all instances): integer centring t of each
// instance (rint of its bounding-box centre), split r - t = n + delta,
// c = frac(H . delta), fp32 slots.  Enqueued on `st`.
scatter_status launch_prep(scatter_plan_t p, const double* xyz, const float* occ, cudaStream_t st,
                           const CallGate& gate = CallGate{});

// Bounding boxes of `batch` instances (ordered-int min / max xyz, atom ranges
// atom_off [batch+1] in device memory) into `bbox` [batch][6], which must hold
// the empty-box values (min slots ~0, max slots 0) beforehand; non-finite
// coordinates set kStatusNonFinite.  For callers that own their buffers.
scatter_status launch_bbox_raw(const double* xyz, const int64_t* atom_off, int batch, int64_t max_atoms,
                               unsigned long long* bbox, unsigned* status, cudaStream_t st);

// A(S) (and/or |A|^2) of every point with the generic FP32/MUFU kernel;
// positions must have been prepared by launch_prep on the same stream.
scatter_status launch_generic(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st,
                              const CallGate& gate = CallGate{});

// Ordered sum of n_chunks partials [chunk][M] (p->d.partial) with the
// translation phase, into the outputs (GenericArgs reduction of forward.cu).
scatter_status launch_generic_reduce(scatter_plan_t p, int n_chunks, float2* amp_out, float* int_out,
                                     cudaStream_t st);

// Clustered S lists (cluster.cu).  Direct kernels skip an instance whose largest
// |x'|^2 of the call (rmax2) is within lim2.
struct ClArgs {
  const ClInst* inst;
  const unsigned* rmax2;
  const float* rho;
  const int32_t* exps;
  const float* cen;
  int64_t n_rows;
  const float4* pt;
  const int64_t* pt_out;
  const ClItem* items;
  const ClTabBlock* tab_blocks;
  const ClRedBlock* red_blocks;
  const ClEvalBlock* eval_blocks;
  float* tab;
  float2* partial;
  float2* M;
  const float4* atom4;
  const float* atom_w;
  const float* coef;
  const float2* ftab;
  int n_species;
  float inv4a2;
  const float* s_hi;
  const double* S64;
  int64_t n_s;
  const double* inst_shift;
  unsigned* status;
  float2* out_amp;
  float* out_int;
};
scatter_status prepare_clusters(scatter_plan_s* p, const double* s_list, double radius_hint);
scatter_status launch_clusters(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st);
void release_clusters(scatter_plan_s* p);
ClArgs cluster_args(scatter_plan_s* p);
// Of one term, for crystals within `radius`: the neglected columns, and the roundings of
// the columns' powers and sums.
void cluster_error(const scatter_plan_s* p, double radius, double* truncation, double* rounding);
// Their adjoint (cluster_adjoint.cu): Sum_S S Im(gF e) per slot into
// [split][n_slots][3] from gF [species][M].
scatter_status prepare_cluster_adjoint(scatter_plan_s* p);
scatter_status launch_cluster_adjoint(scatter_plan_t p, const float2* gf, float* partial, cudaStream_t st);
void release_cluster_adjoint(ClAdjState& s);
inline CallGate cluster_gate(const scatter_plan_s* p) {
  return p->cl.active ? CallGate{p->cl.rmax2, p->cl.lim2, p->batch, nullptr} : CallGate{};
}

// FP32 adjoint on grids as rows times columns (grid_adjoint.cu): prepared where it
// is the cheaper form; partial sums in p->ga.partial.
scatter_status prepare_grid_adjoint(scatter_plan_s* p);
scatter_status launch_grid_adjoint(scatter_plan_t p, const float2* gf, cudaStream_t st, const CallGate& gate);
void release_grid_adjoint(GridAdjState& g);
double grid_adjoint_ops(const scatter_plan_s* p);

// Maps sampled far finer than the crystal's extent asks for (coarse.cu): the sum
// at the Chebyshev nodes of each axis, interpolated to the map.
scatter_status prepare_coarse(scatter_plan_s* p, const scatter_problem* pr, const scatter_options* op);
scatter_status launch_coarse(scatter_plan_t p, const double* xyz, const float* occ, float2* amp_out, float* int_out,
                             cudaStream_t st);
void release_coarse(scatter_plan_s* p);
// Of one term, for crystals within `radius`: the interpolation's own error, its
// roundings, and the factor by which it can amplify errors at the nodes.
void coarse_error(const scatter_plan_s* p, double radius, double* truncation, double* rounding, double* amplify);
// The adjoint from the weights gF [species][M] contracted to the nodes.
scatter_status prepare_coarse_adjoint(scatter_plan_s* p);
scatter_status launch_coarse_adjoint(scatter_plan_t p, const float2* gf, float* grad, cudaStream_t st);
// Tensor-core intensities keep the direct sum: |A|^2 doubles the difference
// between the two (up to 2.5e-5 of the map, amplitudes 1.6e-5).
inline bool coarse_serves(const scatter_plan_s* p, const void* amp_out) {
  return p->coarse_levels > 0 && (amp_out || p->path != SCATTER_PATH_SEPARABLE);
}
// Of the first `levels` node sets: crystals that one of them resolves.
inline CallGate coarse_gate(const scatter_plan_s* p, int levels) {
  return levels > 0 ? CallGate{p->coarse_rmax2, p->coarse[levels - 1].lim2, 1, nullptr} : CallGate{};
}
// Set l itself: crystals that it resolves and no smaller one does.
inline CallGate level_gate(const scatter_plan_s* p, int l) {
  return CallGate{p->coarse_rmax2, l > 0 ? p->coarse[l - 1].lim2 : nullptr, 1, p->coarse[l].lim2};
}
// Positions prepared for the first `levels` node sets, each where no smaller one serves.
scatter_status launch_coarse_prep(scatter_plan_t p, int levels, const double* xyz, const float* occ, cudaStream_t st);
// scatter_plan without a coarse grid of its own, around H, its tensor-core
// accumulation groups at least `group` steps (0: its own choice).
scatter_status plan_nodes(const scatter_problem* pr, const scatter_options* op, const double (&H)[3], double group,
                          scatter_plan_t* out);

// Factorised FP32 sum on single GRID plans (gridsum.cu).
constexpr int kGridSumMaxSplit = 2048;  // chunks that a tuned plan may ask for
bool gridsum_preferred(const scatter_plan_s* p);
scatter_status prepare_gridsum(scatter_plan_s* p, int split_override);
void release_gridsum(scatter_plan_s* p);
scatter_status launch_gridsum(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st,
                              const CallGate& gate = CallGate{});

// Middle of an axis that is symmetric about it: |v_i + v_{n-1-i} - 2 mid| below
// 2e-13 of its largest value (a phase error under 1e-8 cycles for crystals of
// 1e5 cells at |S| = 1; evenly spaced axes miss by a few ulp).
bool axis_symmetric(const std::vector<double>& v, double* mid);

// Atom-parallel form of the generic sum for short S lists (atompar.cu).
bool atompar_applicable(const scatter_plan_s* p);
bool atompar_preferred(const scatter_plan_s* p, const Tiling& s_parallel);
int atompar_choose_k(const scatter_plan_s* p);
scatter_status prepare_atompar(scatter_plan_s* p, int K);
scatter_status launch_atompar(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st);

// Plain FP64 kernel (no prep needed).
scatter_status launch_f64(scatter_plan_t p, const double* xyz, const float* occ, float2* amp_out,
                          float* int_out, cudaStream_t st);

// Loss L (loss_out), and/or gradient dL/dr (grad, caller order) from either
// (A, I_obs) [misfit] or an upstream gradient G [vjp].  Runs prep itself.
scatter_status launch_backward(scatter_plan_t p, const double* xyz, const float* occ, const float2* A,
                               const float* I_obs, const float2* G, double* loss_out, float* grad,
                               cudaStream_t st);

// Tensor-core adjoint on grids of SEPARABLE plans (adjoint_sep.cu).
bool adjoint_sep_applicable(const scatter_plan_s* p);
scatter_status prepare_adjoint_sep(scatter_plan_s* p);
// Mean steps of the accumulation group that a step lies in, of the direct or
// (where the plan folds) the folded form.
double adjoint_sep_group(const scatter_plan_s* p, bool fold);
scatter_status launch_adjoint_sep(scatter_plan_t p, float* grad, cudaStream_t st,
                                  const CallGate& gate = CallGate{});
// FP32 adjoint from the plan's weight table, or from gF where it runs as rows times
// columns (adjoint.cu).
scatter_status launch_adjoint_rows(scatter_plan_t p, const float2* gf, float* grad, cudaStream_t st,
                                   const CallGate& gate = CallGate{});
scatter_status launch_adjoint_tiles(scatter_plan_t p, float* grad, cudaStream_t st,
                                    const CallGate& gate = CallGate{});
scatter_status prepare_adjoint(scatter_plan_s* p);

// Grazing-incidence (DWBA) path: plan tables, split choice, launches.
scatter_status prepare_gid(scatter_plan_s* p);
int dwba_best_split(const scatter_plan_s* p);
scatter_status launch_dwba(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st);
scatter_status launch_gid_combine(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st,
                                  const CallGate& gate = CallGate{});
scatter_status launch_f64_gid(scatter_plan_t p, const double* xyz, const float* occ, float2* amp_out,
                              float* int_out, cudaStream_t st);

// Separable tensor-core path (GRID plans): tables, tiling, launches, and its
// error model (relative L2 of a map with uncorrelated per-term errors).
double separable_error_model(const scatter_plan_s* p, double radius, int split, double* per_pair);
scatter_status prepare_separable(scatter_plan_s* p, int split_override);
scatter_status launch_separable(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st,
                                const CallGate& gate = CallGate{});
double sep_direct_group(const scatter_plan_s* p);

// Batched persistent path (batch > 1): work list, launches (graph-captured).
scatter_status prepare_batch(scatter_plan_s* p);
scatter_status launch_batch(scatter_plan_t p, const double* xyz, const float* occ, float2* amp, float* inten,
                            cudaStream_t st);
scatter_status enqueue_batch_kernels(scatter_plan_t p, float2* amp, float* inten, cudaStream_t st);
int batch_blocks_per_sm(int R, int threads);

// Opt-in event timing around the main kernel of a call.
inline void timing_begin(scatter_plan_s* p, cudaStream_t st) {
  if (p->timing) cudaEventRecord(p->ev_begin, st);
}
inline void timing_end(scatter_plan_s* p, cudaStream_t st) {
  if (p->timing) {
    cudaEventRecord(p->ev_end, st);
    p->timed_call = true;
  }
}

// Occupancy-based residency of the generic kernel for a tiling.
int generic_blocks_per_sm(const scatter_plan_s* p, const Tiling& t);
bool generic_tiling_supported(const Tiling& t);
int64_t generic_num_tiles(const scatter_plan_s* p, const Tiling& t);

}  // namespace scatter
