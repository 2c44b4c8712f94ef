// Internal plan object of libscatter (not part of the public ABI).
//
// Device data layout (all owned by the plan, reused by every call):
//   atoms  : species-sorted, per-instance "slots", each segment of one
//            (instance, species) padded to a multiple of kSlotAlign with
//            zero-weight slots so every tile is full and 16-byte aligned.
//            slot_src[slot]  caller's atom index (or -1 for padding)
//            atom4[slot]     (x', y', z', c) fp32: x' = r - t (lattice units,
//                            t the per-call integer centring of the instance),
//                            c = frac(H . delta) with delta = r - t - rint(r - t)
//            atom_lo[slot]   (x, y, z) - fp32(x', y', z'), 0: the positions as
//                            double-floats for the exact-product phases
//            atom_w[slot]    occupancy (0 for padding)
//   S      : LIST  -> s_hi[3][M] fp32 (s = S - H), s_lo[3][M] its rounding
//                     error, S64[M][3] fp64 (epilogue)
//            GRID  -> axis_s[d][n_d] fp32, axis_lo[d][n_d] its rounding
//                     error, axis64[d][n_d] fp64
//   chunks : split-K partition of each instance's slots into contiguous
//            pieces; a chunk is a list of segments (slot range, species).
#pragma once

#include <cstdint>
#include <vector>
#include "scatter_internal.h"

struct scatter_plan_s;

namespace scatter {

constexpr int kSlotAlign = 32;     // padding granularity of species segments
constexpr int kNCoef = 12;         // a0..a3 b0..b3 c f' f'' B_dw
constexpr int kMaxSpecies = 64;
constexpr int kPrepParts = 256;    // partial bounding boxes of a call (single instances)
constexpr int kPrepSmall = 4096;   // atoms up to which every CTA of the preparation takes the box itself
constexpr int kLossParts = 1024;   // per-block partial sums of the misfit

// Status bits written by kernels into plan->d_status.
enum : unsigned {
  kStatusNonFinite = 1u,
  kStatusTimeout = 2u,
};

struct Segment {
  int64_t begin;    // first slot
  int64_t end;      // one past last slot (multiple of kSlotAlign - begin aligned)
  int32_t species;
  int32_t instance;
};

struct Instance {
  int64_t atom_begin, atom_end;  // caller's atom indices
  int64_t slot_begin, slot_end;  // device slots
  int64_t s_begin, s_end;        // output points
  double H[3];                   // reference reflection (integers)
};

// Atom block of the adjoint kernel (slots of one species segment).
struct AdjBlock {
  int64_t begin;
  int32_t count;
  int32_t species;
};

// Instance and work item of the persistent batched kernel.
struct BatchInst {
  int64_t s_begin, s_end;
  int64_t part_off;  // float2 offset of this instance's partials (split > 1)
  int32_t split;
  int32_t chunk0;
  float H[3];
  float pad;
};

struct BatchItem {
  int64_t p0;        // first S point of the tile
  int32_t inst;
  int32_t chunk;     // chunk index within the instance
};

// Launch shape of the generic kernel.
struct Tiling {
  int threads = 256;
  int R = 8;          // S points per thread
  int split_k = 1;    // atom chunks per S tile
  int atom_k = 0;     // > 0: atom-parallel form, atoms per thread (atompar.cu)
};

// row ranges of a separable map reduced and copied out one after another by
// scatter_amplitude_host (at most one per 32-row block of partials): the
// more ranges, the less of the map's copy is left after the last reduction
constexpr int kHostPieces = 16;

// Clustered S lists (cluster.cu).
struct ClInst {
  int64_t slot_begin, n_slots;
  float R[9];         // frame: xh = R x' (rows: the points' principal axes over X)
  float lim2;         // X^2; -1: the instance is not clustered
  int K, col0;        // columns, the first in exps and rho
  int rows;           // clusters
  int64_t row0;       // the first in cen
  int64_t tab_off;    // floats into tab: [column tile][slot][16]
  int64_t part_off;   // float2 into partial: [chunk][column][cluster]
  int64_t m_off;      // float2 into M: [species][column][cluster]
  uint64_t species;   // bit s: atoms of species s
  float H[3];
  double H64[3];
};
struct ClItem {
  int32_t inst, row0, col_tile, species;
  int64_t begin, end;  // slots within the instance
  int64_t part;        // float2 offset of the chunk's partials
};
struct ClTabBlock {
  int32_t inst;
  int64_t slot;
};
struct ClRedBlock {
  int32_t inst, species, c0, c1;  // chunks of the species
  int64_t elem;                   // first of 32 (column, cluster) elements
};
struct ClEvalBlock {
  int32_t inst, n;
  int64_t p0;
};
struct ClGBlock {
  int32_t row, n;  // points of one cluster
  int64_t p0;
};
// Adjoint over the clusters (cluster_adjoint.cu), single instances.
struct ClAdjState {
  bool active = false;
  AdjBlock* blocks = nullptr;       // atom blocks of one species
  ClGBlock* g_blocks = nullptr;     // <= 256 points of one cluster
  int32_t* row_blk = nullptr;       // [rows + 1] the first g_block of each cluster
  short4* up = nullptr;             // per column: columns of a + e_d, -1: none
  short4* down = nullptr;           //             columns of a - e_d
  float* rho = nullptr;             // per column: the relative radius from which it or its derivative matters
  float2* g_part = nullptr;         // [g_block][species][column]
  float* g8 = nullptr;              // [species][cluster][column][8]
  int n_blocks = 0, n_g = 0, split = 1, rows_per_chunk = 0, smem = 0;
  int emax[3] = {0, 0, 0};
};
// A clustered instance's radius and its clusters' largest corner phases, for the
// error bound.
struct ClExtent {
  double X, th[3];
};
struct ClState {
  bool active = false;
  ClAdjState adj;
  std::vector<ClExtent> extents;
  ClInst first;                     // the only instance, with its columns and its clusters' points
  std::vector<int32_t> h_exps;
  std::vector<int64_t> h_row;
  ClInst* inst = nullptr;           // [batch]
  float* lim2 = nullptr;            // [batch] X^2, -1: not clustered
  unsigned* rmax2 = nullptr;        // [batch] this call's largest |x'|^2 (float bits)
  float* rho = nullptr;             // per column: the relative radius from which it matters
  int32_t* exps = nullptr;          // per column: exponents (4 bits each), |a| mod 4 at bit 12
  float* cen = nullptr;             // [3][n_rows] cluster centres - H
  float4* pt = nullptr;             // points by cluster: 2 pi X (s - centre) in the frame, cluster
  int64_t* pt_out = nullptr;        // their output indices
  ClItem* items = nullptr;
  ClTabBlock* tab_blocks = nullptr;
  ClRedBlock* red_blocks = nullptr;
  ClEvalBlock* eval_blocks = nullptr;
  float* tab = nullptr;
  float2* partial = nullptr;
  float2* M = nullptr;
  int64_t n_rows = 0;
  int n_items = 0, n_tab = 0, n_red = 0, n_eval = 0;
};

// FP32 adjoint on grids, rows times columns (grid_adjoint.cu).
struct GridAdjState {
  bool active = false;
  int q = 2, np = 0, chunks = 1, pairs = 0;  // column axis, pairs per CTA, chunks of them, pairs in all
  bool mirror = false;
  double mid = 0.0;                 // middle of a symmetric column axis - H
  int64_t rows_per_split = 0;
  int split = 1, n_blocks = 0;
  AdjBlock* blocks = nullptr;
  float* d = nullptr;               // column offsets, and rounding errors
  float* dlo = nullptr;
  float* table = nullptr;           // [species][chunk][row][np][16]
  float* partial = nullptr;         // [split][chunk][slot][3]
  float2* gf = nullptr;             // [species][M]
};

// Oversampled maps (coarse.cu).
struct CoarseStage {
  int axis = 0;
  int64_t n_in = 0, n_out = 0;      // nodes, points of the axis
  int64_t outer = 0, inner = 0;     // of the array at that stage
  float* W = nullptr;               // [n_in][n_out], then its rounding errors
  float* Wt = nullptr;              // the adjoint's: [n_out][n_in], then its rounding errors
  std::vector<float> h_W;           // W on the host
};
constexpr int kCoarseLevels = 2;
struct CoarseState {
  scatter_plan_s* sub = nullptr;    // the sum at the nodes, without the translation phase
  double X = 0.0;                   // |x'_d| that they resolve
  CoarseStage stage[3];
  int n_stages = 0;
  float2* map = nullptr;            // at the nodes
  float2* tmp[2] = {nullptr, nullptr};
  float* lim2 = nullptr;            // X^2
  float2* adj_tmp[2] = {nullptr, nullptr};
  float2* adj_gf = nullptr;         // weights at the nodes (FP32 sums)
};

// The factorised FP32 grid sum (gridsum.cu).
struct GridSum {
  bool active = false;
  int q = 2, R = 1, threads = 256;  // column axis, columns and rows per thread block
  bool mirror = false;              // the columns of a symmetric axis: half of them, each with its mirror
  int64_t n_cols = 0, row_tiles = 0, col_tiles = 0;
  int split = 1, n_chunks = 0;      // chunks asked for, chunks (one species each)
  int64_t bytes = 0;                // its device memory (in tiling_bytes)
  double mid = 0.0;                 // mirror: the axis' middle - H
  Segment* chunks = nullptr;        // device
  float* d = nullptr;               // device: column offsets and their rounding errors
  float* dlo = nullptr;
  bool tab = false;                 // records and column factors tabulated per call (device below)
  float4* rec = nullptr;
  float2* rec_lo = nullptr;
  float2* ztab = nullptr;
};

// One form of the separable contraction: its tiles, atom chunks and launch
// choices.  The A table and the partials are the plan's, sized for the larger.
struct SepForm {
  bool fold = false, fold_h = false;  // folded over the (k, l) axes' middles, over h's too (sep_common.cuh)
  int64_t mt = 0, nt = 0, steps = 0;  // M tiles, N tiles, K steps
  int64_t cols = 0;                   // columns of the partials
  int64_t lanes = 0, pairs = 0;       // fold: h values with rows of their own, mirror pairs of (k, l) points
  int split = 1;
  int32_t n_chunks = 0;
  Segment* chunks = nullptr;          // device: atom chunks, one species each, step-aligned slots
  int flush = 0;                      // steps between TMEM flushes
  bool form_a = false;                // A formed inside the CTA-pair kernel, no A table
  float smax[2] = {0.f, 0.f};         // max offset of the b and c axes
};

struct DeviceBuffers {
  int32_t* slot_src = nullptr;      // [n_slots]
  int32_t* slot_inst = nullptr;     // [n_slots]
  float4* atom4 = nullptr;          // [n_slots]
  float4* atom_lo = nullptr;        // [n_slots] FP32 rounding errors of (x', y', z'), 0
  float* atom_w = nullptr;          // [n_slots]
  int32_t* atom_species = nullptr;  // [n_atoms] caller order (FP64 kernel)
  Segment* segs = nullptr;          // [n_segs] (chunked)
  int32_t* chunk_seg_off = nullptr; // [n_chunks+1]
  float* coef = nullptr;            // [n_species][12] fp32
  double* coef64 = nullptr;         // [n_species][12] fp64
  int64_t* atom_off = nullptr;      // [batch+1] caller atom ranges
  int64_t* inst_slot_begin = nullptr; // [batch]
  double* inst_H = nullptr;         // [batch][3]
  double* inst_shift = nullptr;     // [batch][3] integer centring t (per call)
  unsigned long long* box_part = nullptr;   // [kPrepParts][6] partial boxes (single instances)
  unsigned long long* inst_bbox = nullptr;  // [batch][6] ordered-int min/max
  // S
  float* s_hi = nullptr;            // LIST: [3][M]
  float* s_lo = nullptr;            // LIST: [3][M] s - s_hi (double-float s of the exact-product phases)
  double* S64 = nullptr;            // LIST: [M][3]
  int32_t* s_inst = nullptr;        // LIST batch: instance of each point (or null)
  float* axis_s = nullptr;          // GRID: concatenated axes (s = axis - H)
  float* axis_lo = nullptr;         // GRID: s - axis_s
  double* axis64 = nullptr;         // GRID: concatenated axes (full S)
  // workspace
  float2* partial = nullptr;        // [split_k][M] split-K partials
  float2* amp = nullptr;            // [M] amplitude scratch (intensity, backward)
  double* loss_part = nullptr;      // per-block loss partials
  float2* gS = nullptr;             // [M] adjoint weights g(S)
  unsigned* status = nullptr;       // [1]
  // grazing incidence (GID grids)
  float* gid_sz = nullptr;          // [2][n_af] Sz1, Sz2 r.l.u.
  float* gid_sz_lo = nullptr;       // [2][n_af] their FP32 rounding errors
  float* gid_sz_im = nullptr;       // [2][n_af] Im of a buried object's S_z (0 on the substrate)
  float* gid_szf = nullptr;         // [4][n_af] S_z of each beam's form factor (vacuum)
  double* gid_szf64 = nullptr;      // [4][n_af]
  double* gid_sz64_im = nullptr;    // [n_af] Im sigma of a buried object's beam (0 on the substrate)
  double* gid_sz64 = nullptr;       // [2][n_af]
  float2* gid_w = nullptr;          // [4][n_af] beam weights
  double2* gid_w64 = nullptr;       // [4][n_af]
  float4* ztab = nullptr;           // [n_afb][n_slots][32] Z1, Z2 per call
  // separable path
  void* sep_A = nullptr;            // A operand blocks (f16 hi/lo)
  float* sep_partial = nullptr;     // [chunk][2][sep_ns] planar
  Segment* ap_blocks = nullptr;     // atom-parallel blocks: one species each, <= 256 K slots
  float2* ftab = nullptr;           // Eq. 4 factor table [n_species][M], or null (form factors)
  double* ftab64 = nullptr;         // the same in FP64 (re, im) for the FP64 kernel
  float* sep_axis_s = nullptr;      // separable grid axes, s = axis - H (virtual for GID)
  float* sep_axis_lo = nullptr;     // their FP32 rounding errors
  float* sep_axis_d = nullptr;      // folded forward: offsets from the axes' middles [n0 | n1 | n2]
  float* sep_axis_dlo = nullptr;    // their FP32 rounding errors
  float4* sep_rec = nullptr;        // folded forward: (x', its rounding error, Re W, Im W) per slot (written by prep)
  float2* sep_virt = nullptr;       // GID: map over the virtual (h, k, 4 beams x alpha_f) grid
  // batches
  BatchInst* batch_inst = nullptr;
  BatchItem* batch_items = nullptr;
  int* counter = nullptr;
  // adjoint workspace (allocated on first backward)
  AdjBlock* adj_blocks = nullptr;
  float4* adj_table = nullptr;      // [n_species][M][2], or [n_species][M] in line mode
  float* adj_partial = nullptr;     // [split][n_slots][3]
  // tensor-core adjoint on grids (adjoint_sep.cu)
  float2* adj_gf = nullptr;         // [n_species][M] gF_s
  int* adj_sexp = nullptr;          // [n_species][3][n0] row scale exponents
  void* adj_sepA = nullptr;         // A blocks [species][M-tile pair][point step][2][hi|lo]
  float* adj_sep_partial = nullptr; // [chunk][Re, Im][3 n0][n_slots]
  float4* adj_rec = nullptr;        // point records (0, s_b, s_c, 0), 16 per step
  Segment* adj_ntiles = nullptr;    // 256-slot atom tiles of one species
  Segment* adj_kchunks = nullptr;   // point-step chunks (split over K)
  // scatter_amplitude_host: device copies of the caller's host buffers
  double* host_xyz = nullptr;       // [n_atoms][3]
  float* host_occ = nullptr;        // [n_atoms]
  float2* host_amp = nullptr;       // [n_s]
  // separable path of a buried object: per virtual l column
  float* sep_att = nullptr;         // 2 pi Im(sigma): the formed rows carry exp(-sep_att z')
  float* sep_szf = nullptr;         // S_z of the column's form factor (the vacuum beam S_1)
};

}  // namespace scatter

struct scatter_plan_s {
  int device = 0;
  int n_sm = 0;
  scatter_path path = SCATTER_PATH_GENERIC;
  scatter_s_kind s_kind = SCATTER_S_LIST;
  int64_t n_atoms = 0;
  int64_t n_slots = 0;
  int64_t n_s = 0;
  int32_t n_species = 1;
  int32_t batch = 1;
  double lattice_a = 1.0;
  int64_t n_axis[3] = {0, 0, 0};
  std::vector<double> axis_host[3];
  std::vector<double> coef_host;                 // [n_species][12]
  std::vector<scatter::Instance> inst;
  std::vector<scatter::Segment> all_segs;        // (instance, species) segments
  std::vector<scatter::Segment> segs;            // chunk-major
  std::vector<int32_t> chunk_seg_off;            // [n_chunks+1]
  std::vector<int64_t> chunk_slots;              // slots per chunk (cost)
  scatter::Tiling tiling;
  double wavelength = 0, alpha_i = 0, delta = 0, beta = 0;
  int gid_mode = 0;                              // 0: on the substrate (four beams), 1: buried (one beam)
  scatter::DeviceBuffers d;
  scatter::GridSum gs;
  scatter::ClState cl;
  scatter::GridAdjState ga;
  scatter::CoarseState coarse[scatter::kCoarseLevels];  // by growing radius
  int coarse_levels = 0;
  int coarse_adj_levels = 0;                     // the first ones, with an adjoint
  unsigned* coarse_rmax2 = nullptr;              // this call's largest |x'_d|^2 (float bits)
  double* coarse_shift = nullptr;                // [3] the nodes' out_shift
  unsigned* extent2 = nullptr;                   // the sum at the nodes of another plan: prep writes the largest |x'_d|^2
  double* out_shift = nullptr;                   //   its reductions' shift in place of the call's: 0 on the interpolated
                                                 //   axes (grazing incidence: prep writes the call's t_z)
  double sep_group = 0.0;                        //   accumulation groups of at least this many steps
  int64_t base_bytes = 0;                        // tables and backward workspace
  int64_t tiling_bytes = 0;                      // chunk tables and split-K partials
  double s_max[3] = {0, 0, 0};                   // max |S - H| per axis (error model)
  bool use_graph = true;
  bool timing = false;
  cudaEvent_t ev_begin = nullptr, ev_end = nullptr;
  bool timed_call = false;
  int32_t last_launches = 0;
  // batches: work list and captured graph
  int32_t batch_items = 0;
  int batch_ctas = 0;
  bool batch_has_split = false;
  cudaGraphExec_t graph_exec = nullptr;
  const void* graph_key[4] = {nullptr, nullptr, nullptr, nullptr};
  cudaStream_t graph_stream = nullptr;
  cudaEvent_t graph_in = nullptr, graph_out = nullptr;
  int32_t graph_launches = 0;
  int64_t sep_n[3] = {0, 0, 0};                  // separable grid shape (GID: n_h, n_k, 4 n_af)
  int64_t sep_ns = 0;
  scatter::SepForm sep_direct, sep_folded;       // sep_folded.fold: the folded form exists (amplitude calls)
  double sep_mid[3] = {0, 0, 0};                 // the folded axes' middles - H
  int32_t ap_n_blocks = 0;
  int32_t ap_tile = 0;               // reflections per atom-parallel CTA (<= kApPts)
  std::vector<double> gid_sz_host;               // [2][n_af] Sz1, Sz2 (r.l.u.)
  std::vector<double> gid_sz_im_host;            // [n_af] Im sigma of a buried object's beam
  std::vector<double> gid_szf_host;              // [4][n_af] S_z of each beam's form factor
  int32_t sep_beams = 4;                         // beams stacked on the separable l axis (buried: 1)
  bool adj_ready = false;
  int adj_split = 1;
  int adj_blocks = 0;
  int64_t adj_s_per_chunk = 0;
  bool adj_line = false;            // uniform-l grid: k_adjoint_line (phase recurrence)
  float adj_ds = 0.f;               // its l step
  int64_t adj_lines_per_chunk = 0;
  bool adj_sep = false;             // SEPARABLE grid plan: the adjoint runs on k_sep
  bool adj_no_fold = false;         // asked for: the direct form
  bool adj_sep_fold = false;        // its points folded over the middle of the (k, l) plane
  int64_t adj_sep_k = 0;            // points (mirror pairs) of a plane
  double adj_sep_mid[2] = {0, 0};   // the middles of the k and l axes - H
  int64_t adj_sep_ksteps = 0, adj_sep_mt = 0;
  int32_t adj_sep_ntiles = 0, adj_sep_chunks = 0;
  float adj_sep_smax[2] = {0.f, 0.f};
  // scatter_amplitude_host on a separable grid: the reduction runs in
  // kHostPieces row ranges and each range's copy to the host (destination
  // host_out) starts on copy_stream as soon as the range is reduced
  void* host_out = nullptr;
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t copy_ev[scatter::kHostPieces + 1] = {};
  // separable contractions with an odd M-tile pair count of 3 or more: the
  // last pair's one-CTA kernel runs on side_stream beside the CTA-pair kernel
  cudaStream_t side_stream = nullptr;
  cudaEvent_t side_fork = nullptr, side_join = nullptr;
};
