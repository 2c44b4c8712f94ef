// Separable tensor-core path for axis-aligned S grids (tcgen05, sm_103a).
//
// On a grid S = H + (s_a, s_b, s_c) the phase of Eq. 2 separates,
//   w_j exp(2 i pi (c_j + s_a x'_j + s_b y'_j + s_c z'_j)) = Xw[a,j] B[(b,c),j]
// with Xw = w e^{2 pi i s_a x'} and B = e^{2 pi i (s_b y' + s_c z' + c)},
// so the per-species sum is a complex matrix product over the atoms:
//   T_s[a, (b,c)] = sum_{j in s} Xw[a,j] B[(b,c), j].
// It runs as a real GEMM D = A B^T on the 5th-generation tensor cores:
//   A  (M = 2 n_a rows: Re/Im of each a) x (K = 2 per atom: Re/Im):
//      rows 2a: [Xwr, -Xwi], rows 2a+1: [Xwi, Xwr]  -> D[2a] = Re T, D[2a+1] = Im T
//   B  (N = (b,c) points) x (K): [Br, Bi]
// Both operands are split into f16 hi + lo parts and three products
// (hi.hi + hi.lo + lo.hi) accumulate in FP32 in tensor memory (TMEM), which
// keeps the result near FP32 accuracy (the lo.lo term is below 2^-22).
//
// Per call: k_sep_tab_a writes the A operand (hi/lo, already in the
// canonical no-swizzle K-major shared-memory layout, one 16 KB block per
// (M tile, 16-atom step), the two tiles of a pair adjacent).
// k_sep: CTA = a pair of 128-row M tiles (two 128 x 256 FP32
// accumulators filling the 512 TMEM columns) x one 256-point N tile x one
// atom chunk; per 16-atom step the TMA engine copies the pair's A blocks
// and the step's 16 atom records (y', z', c), two threads per point compute its
// row of B from them (FP32 phase, exact reduction mod 1, MUFU
// sincos, f16 split) into shared memory once for both tiles, and one
// thread issues 12 tcgen05.mma (2 tiles x 2 K16 sub-steps x 3 products,
// M=128 N=256).  Warp roles: sixteen warps form B (and read the accumulators
// out), one warp issues the MMAs, one warp issues the copies (a 32 KB bulk
// copy holds its issuing thread for ~1000 cycles, so it must not be the MMA
// thread).  A ring for the A blocks (four stages, eight where the CTA has one
// M tile), an eight-stage ring for the
// atom records and a two-stage ring for the B blocks, each stage with a
// full and an empty mbarrier, keep the formation of step k+1 and the copies
// of later steps overlapped with the MMAs of step k.  The MMAs read ~96 B/clk of shared memory on their own;
// computing B from the atom records, instead of loading tabulated factors
// through L1, keeps the rest of the shared-memory traffic to the A copies
// and the B stores.
// Atom chunks (grid y) hold one species each.  Every kSepFlush steps (folded:
// the form's own interval) and at the
// end of the chunk the accumulator is read from TMEM (tcgen05.ld) and added
// into FP32 partials owned by the CTA, in the accumulator's 32 x 32 blocks
// (sep_part_off; shorter groups keep the
// tensor core's FP32 accumulation error down); k_sep_reduce sums the chunks
// in order, each times its species' f_s(|S|), and applies the translation
// phase.
// The same kernel, with the roles of the operands swapped, runs the adjoint
// on grids (adjoint_sep.cu); the arguments in sep_common.cuh cover both.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>
#include "launch.h"
#include "sep_common.cuh"
#include "tuner.h"

namespace scatter {

// -------------------------------------------------------------------------
// tables
// -------------------------------------------------------------------------

struct SepTabArgs {
  const float4* atom4;
  const float4* atom_lo;  // position rounding errors
  const float* atom_w;
  const float* axis_s;  // [n0 | n1 | n2] s values
  const float* axis_lo; // their FP32 rounding errors (s as a double-float)
  int64_t n0, n1, n2;
  int64_t n_slots, n_steps, n_mt;
  uint4* A;             // [n_mt/2][n_steps][2 tiles][hi|lo][4 kb][16 mg][8 rows] of 16 B
  CallGate gate;
};

// One thread per 16-byte row of a core matrix of the A operand (4 atoms x
// Re/Im of one row m), hi and lo parts; the weight w_j is folded in here.
__global__ void k_sep_tab_a(const SepTabArgs t) {
  if (within(t.gate, 0)) return;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = t.n_mt * t.n_steps * 4 * kSepM;
  // total is a multiple of 512: whole warps leave here, the shuffles below
  // always see all 32 lanes
  if (i >= total) return;
  const int r = (int)(i % 8), mg = (int)((i / 8) % 16), kb = (int)((i / 128) % 4);
  const int64_t ks = (i / 512) % t.n_steps, mt = i / (512 * t.n_steps);
  const int64_t m = mt * kSepM + mg * 8 + r;
  const int64_t a = m >> 1;
  const int ri = (int)(m & 1);
  const bool ok = a < t.n0;
  const float sa = ok ? t.axis_s[a] : 0.f, sal = ok ? t.axis_lo[a] : 0.f;
  float x[2] = {0.f, 0.f}, xl[2] = {0.f, 0.f}, w[2] = {0.f, 0.f};
  if (ok) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t slot = ks * kSepStep + kb * 4 + 2 * ri + u;
      x[u] = t.atom4[slot].x;
      xl[u] = t.atom_lo[slot].x;
      w[u] = t.atom_w[slot];
    }
  }
  uint4 hi, lo;
  sep_a_row(sa, sal, ok, ri, x, xl, w, hi, lo);
  uint4* blk = t.A + (((mt >> 1) * t.n_steps + ks) * kSepPair + (mt & 1)) * (kSepABytes / 16);
  const int64_t off = (int64_t)(kb * 16 + mg) * 8 + r;
  blk[off] = hi;
  blk[512 + off] = lo;
}

// The folded A operand (sep_common.cuh): one thread per (M tile, step, K block
// of 8 atoms, lane), the lane's four rows; a warp is the 32 lanes of one K
// block, so the records are broadcast loads and each of the eight stores
// covers 512 contiguous bytes.  Bound by the table's write: 275 MB in 42 us on the
// strained sphere (the direct form's k_sep_tab_a: 549 MB in 116 us).
template <bool FOLD_H>
__global__ void __launch_bounds__(256) k_sep_tab_fold(const float4* __restrict__ rec_a, const float* __restrict__ axis_d,
                                                      const float* __restrict__ axis_dlo, int64_t n0, int64_t n_lanes,
                                                      int64_t n_steps, int64_t n_mt, uint4* __restrict__ A,
                                                      const CallGate gate) {
  if (within(gate, 0)) return;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_mt * n_steps * 128) return;  // whole warps
  const int lane = (int)(i & 31), kb = (int)((i >> 5) & 3);
  const int64_t ks = (i >> 7) % n_steps, mt = (i >> 7) / n_steps;
  float d[2], dl[2];
  bool ok[2];
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const int64_t ah = sep_fold_a(mt, lane, w, FOLD_H, n0);
    ok[w] = FOLD_H ? 32 * mt + lane < n_lanes : ah < n_lanes;
    d[w] = ok[w] ? axis_d[ah] : 0.f;
    dl[w] = ok[w] ? axis_dlo[ah] : 0.f;
  }
  uint4 hi[4], lo[4];
  sep_a_fold<FOLD_H>(d, dl, ok, rec_a + ks * kSepFoldStep + kb * 8, hi, lo);
  uint4* blk = A + (((mt >> 1) * n_steps + ks) * kSepPair + (mt & 1)) * (kSepABytes / 16) + kb * 128 + lane;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    blk[32 * r] = hi[r];
    blk[512 + 32 * r] = lo[r];
  }
}

// -------------------------------------------------------------------------
// main kernel
// -------------------------------------------------------------------------


// Warp roles: 16 formation warps form the B rows (two threads per point) and read
// the accumulators out at every group end; the next warp (one lane) issues the
// MMAs; the last (one lane) issues the TMA copies.  Hand-offs go through
// mbarriers only:
//   bar_full[a]   A block of a step arrived            (TMA, 1 arrival + bytes)
//   bar_done[a]   MMAs of the step done (one commit per step); frees the A
//                 stage of that step and the B stage it read
//   bar_atom[t]   atom records of a step arrived       (TMA)
//   bar_tempty[t] atom records read by the formation   (formation warps)
//   bar_bfull[b]  B block of a step formed             (formation warps)
//   bar_tfree     accumulators read out after a group end (formation warps)
// FOLD: the folded forward (sep_common.cuh): 32 atoms per step, the 256 columns
// are the cos and sin columns of 128 mirror pairs of points; thread (p, kb)
// forms both columns of pair p over one of the four K blocks.  The formation binds
// a step of one M tile; 16 warps against 8: 43 x 43 x 31 nodes of a 127,560-atom
// island 1.15 against 1.33 ms per call, folded 64 x 64 x 24 nodes of 134,009 atoms
// 1.0 against 1.1 us a step; two M tiles are bound by the MMAs either way.
template <bool FOLD>
__global__ void __maxnreg__(112) k_sep(const SepArgs a) {
  if (within(a.gate, 0)) return;  // before any barrier or allocation
  constexpr int kRec = FOLD ? kSepFoldStep : kSepStep;  // records per step
  constexpr int kForm = kSepOneWarps;
  constexpr int kSpan = kSepN / (kForm / 4);  // columns that a formation warp reads out
  // a B stage is freed by the done barrier of the step that read it: the A
  // ring (and with it the done ring) must be at least as deep as the B ring
  static_assert(kSepBStages <= kSepAStages, "B-stage reuse is tracked on the done ring");
  extern __shared__ __align__(1024) unsigned char sep_smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[2 * kSepAStages];
  __shared__ __align__(8) uint64_t bar_done[2 * kSepAStages];
  __shared__ __align__(8) uint64_t bar_atom[kSepTStages];
  __shared__ __align__(8) uint64_t bar_tempty[kSepTStages];
  __shared__ __align__(8) uint64_t bar_bfull[kSepBStages];
  __shared__ __align__(8) uint64_t bar_tfree;
  __shared__ __align__(16) float4 ring_atom[kSepTStages][kRec];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(sep_smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* ringA = smem;
  unsigned char* ringB = smem + kSepAStages * kSepPair * kSepABytes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool mma_warp = warp == kForm, copy_warp = warp == kForm + 1;
  const int64_t n_mp = a.mp_count > 0 ? a.mp_count : (a.n_mt + 1) / 2;  // pairs of this launch
  const int64_t mp = a.mp_first + blockIdx.x % n_mp, nt = blockIdx.x / n_mp;
  const int ntp = 2 * mp + 1 < a.n_mt ? 2 : 1;  // M tiles of this CTA with rows
  // one M tile: twice the A stages, of half the bytes (127,560-atom island, 43 x 43 x
  // 31 nodes: 1.26 ms per call with three stages, 1.148 with four, 1.134 with eight;
  // the bytes in two more B stages instead: 1.20)
  const int la = ntp == 1 ? kSepALog + 1 : kSepALog, n_a = 1 << la;
  const int chunk = blockIdx.y;
  const int64_t nbc = a.n1 * a.n2;
  // up to 64 mirror pairs in all: 128 columns are contracted
  const bool narrow = FOLD && a.n_pairs <= kSepFoldPairs / 2;
  // this CTA's columns [col_base, col_end) and the species of its A table
  int64_t col_base = nt * kSepN, col_end = FOLD ? sep_fold_cols(a.n_pairs) : nbc;
  int a_species = 0;
  if (!FOLD && a.ntiles) {
    const Segment t = a.ntiles[nt];
    col_base = t.begin;
    col_end = t.end;
    a_species = t.species;
  }

  if (mma_warp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dev::smem_addr(&tmem_slot)),
                 "r"(kSepTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int s = 0; s < n_a; ++s) {
      dev::mbar_init(&bar_full[s], 1);
      dev::mbar_init(&bar_done[s], 1);
    }
    for (int s = 0; s < kSepTStages; ++s) {
      dev::mbar_init(&bar_atom[s], 1);
      dev::mbar_init(&bar_tempty[s], kForm);
    }
    for (int s = 0; s < kSepBStages; ++s) {
      dev::mbar_init(&bar_bfull[s], kForm);
    }
    dev::mbar_init(&bar_tfree, kForm);
    s_abort = 0;
    dev::mbar_fence_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  // the chunk's steps (record bounds on step edges)
  const int64_t ks_begin = a.chunks[chunk].begin / kRec, ks_end = a.chunks[chunk].end / kRec;
  SepGroups grp{ks_end, ks_begin, FOLD ? a.flush : kSepFlush};
  bool ok = true;
  // copies issued and MMA steps committed (steps), for the drain on abort
  int64_t a_issued = 0, t_issued = 0, g_committed = 0;

  if (copy_warp) {
    if (lane == 0) {
      // A block and K records of every step, in step order; a stage is
      // refilled once its previous contents were consumed
      const uint4* Ablk = a.A + a_species * a.a_sp_stride + mp * a.n_steps * (kSepPair * kSepABytes / 16);
      const uint32_t a_bytes = (uint32_t)ntp * kSepABytes;
      int64_t g = 0;
      for (int64_t ks = ks_begin; ks < ks_end; ++ks, ++g) {
        if (s_abort) {
          ok = false;
          break;
        }
        const int tst = (int)(g % kSepTStages), ast = (int)(g & (n_a - 1));
        if (g >= kSepTStages &&
            !dev::mbar_wait_bounded(&bar_tempty[tst], (uint32_t)(((g - kSepTStages) / kSepTStages) & 1))) {
          ok = false;
          break;
        }
        dev::mbar_arrive_expect_tx(&bar_atom[tst], kRec * sizeof(float4));
        dev::bulk_g2s(&ring_atom[tst][0], a.rec + ks * kRec, kRec * sizeof(float4), &bar_atom[tst]);
        t_issued = g + 1;
        if (g >= n_a && !dev::mbar_wait_bounded(&bar_done[ast], (uint32_t)(((g - n_a) >> la) & 1))) {
          ok = false;
          break;
        }
        dev::mbar_arrive_expect_tx(&bar_full[ast], a_bytes);
        dev::bulk_g2s(ringA + ast * ntp * kSepABytes, Ablk + ks * (kSepPair * kSepABytes / 16), a_bytes,
                      &bar_full[ast]);
        a_issued = g + 1;
      }
    }
  } else if (mma_warp) {
    if (lane == 0) {
      // descriptors of A stage 0 tile 0 and B stage 0 (hi and lo of the two
      // K16 halves); other stages and tiles add their byte offset / 16 to the
      // address field (every shared-memory address here is below 2^18)
      const uint32_t a0 = dev::smem_addr(ringA), b0 = dev::smem_addr(ringB);
      const uint64_t dah[2] = {smem_desc(a0, 2048, 128), smem_desc(a0 + 4096, 2048, 128)};
      const uint64_t dal[2] = {smem_desc(a0 + 8192, 2048, 128), smem_desc(a0 + 8192 + 4096, 2048, 128)};
      const uint64_t dbh[2] = {smem_desc(b0, 4096, 128), smem_desc(b0 + 8192, 4096, 128)};
      const uint64_t dbl[2] = {smem_desc(b0 + 16384, 4096, 128), smem_desc(b0 + 16384 + 8192, 4096, 128)};
      const uint32_t idesc = narrow ? kSepIdescHalf : kSepIdesc;
      int64_t flushes = 0;  // groups read out before the current one
      int64_t g = 0;
      for (int64_t ks = ks_begin; ks < ks_end; ++ks, ++g) {
        if ((g & 15) == 0 && s_abort) {  // waits are bounded; a prompt exit is a bonus
          ok = false;
          break;
        }
        if (ks == grp.grp_start && flushes > 0 &&
            !dev::mbar_wait_bounded(&bar_tfree, (uint32_t)((flushes - 1) & 1))) {
          ok = false;
          break;
        }
        const int ast = (int)(g & (n_a - 1)), bst = (int)(g % kSepBStages);
        if (!dev::mbar_wait_bounded(&bar_full[ast], (uint32_t)((g >> la) & 1)) ||
            !dev::mbar_wait_bounded(&bar_bfull[bst], (uint32_t)((g / kSepBStages) & 1))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t offB = (uint64_t)((bst * kSepBBytes) >> 4);
        for (int tp = 0; tp < ntp; ++tp) {
          const uint64_t offA = (uint64_t)(((ast * ntp + tp) * kSepABytes) >> 4);
          const uint32_t d = tmem + (uint32_t)(tp * kSepN);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const uint32_t acc0 = (ks > grp.grp_start || u > 0) ? 1u : 0u;
            mma_f16(d, dah[u] + offA, dbh[u] + offB, acc0, idesc);
            mma_f16(d, dah[u] + offA, dbl[u] + offB, 1u, idesc);
            mma_f16(d, dal[u] + offA, dbh[u] + offB, 1u, idesc);
          }
        }
        mma_commit(&bar_done[ast]);
        g_committed = g + 1;
        if (grp.ends_at(ks)) {
          grp.advance(ks);
          ++flushes;
        }
      }
    }
  } else {
    // ---- formation warps ---------------------------------------------------
    // this thread's B row (column col of D): forward the point (b, c) with
    // offsets (s_b, s_c) from H, adjoint the atom's (y', z')
    // (folded: the first point of the thread's mirror pair)
    const int p_loc = tid & (narrow ? kSepFoldPairs / 2 - 1 : kSepFoldPairs - 1);
    const int64_t col = FOLD ? nt * kSepFoldPairs + p_loc : col_base + (tid & (kSepN - 1));
    const bool row_ok = col < (FOLD ? a.n_pairs : col_end);
    float sb, sc, sbl = 0.f, scl = 0.f;  // sbl, scl: low parts of a double-float s (forward)
    float att = 0.f;                     // buried object: 2 pi Im(sigma) of the column's beam
    bool att_over = false;               // an attenuation exponent passed kSepAttMax
    if (!FOLD && a.ntiles) {
      const float4 at = row_ok ? a.atom4[col] : make_float4(0.f, 0.f, 0.f, 0.f);
      sb = at.y;
      sc = at.z;
    } else {
      const int64_t rb = row_ok ? col / a.n2 : 0, rc = row_ok ? col % a.n2 : 0;
      sb = a.axis_s[a.n0 + rb];
      sc = a.axis_s[a.n0 + a.n1 + rc];
      if (!FOLD && a.axis_att) att = a.axis_att[rc];
      if (a.axis_lo) {
        sbl = a.axis_lo[a.n0 + rb];
        scl = a.axis_lo[a.n0 + a.n1 + rc];
      }
    }
    const int b_row = FOLD ? (p_loc >> 6) * 128 + (p_loc & 63) : tid & (kSepN - 1);  // folded: the cos column, the sin column 64 on
    const uint32_t b_row_off = (uint32_t)((b_row >> 3) * 128 + (b_row & 7) * 16);
    // |s_b y' + s_c z' + c| of every B element of this call stays below
    // kSepPhaseLim cycles when the centred extent is small: the exact mod-1
    // reduction is then skipped (MUFU sin/cos of an argument of L cycles errs
    // by ~L 2^-24 cycles, 6e-6 rad at the limit, below this path's 1e-4)
    // (and above dev::kPhaseExactLim cycles, crystals hundreds of cells long,
    // each product is taken with its rounding error restored)
    bool reduce = true, exact = false;
    {
      const unsigned long long ylo = a.bbox[1], zlo = a.bbox[2], yhi = a.bbox[4], zhi = a.bbox[5];
      if (ylo != ~0ULL && zlo != ~0ULL && yhi != 0ULL && zhi != 0ULL) {
        const double ey = fmax(fabs(dev::unordered(ylo) - a.shift[1]), fabs(dev::unordered(yhi) - a.shift[1]));
        const double ez = fmax(fabs(dev::unordered(zlo) - a.shift[2]), fabs(dev::unordered(zhi) - a.shift[2]));
        const double bound = (double)a.smax_b * (ey + 1.0) + (double)a.smax_c * (ez + 1.0) + 0.5;
        reduce = bound > kSepPhaseLim;
        exact = bound > dev::kPhaseExactLim;
      }
    }
    float* part = a.partial + (int64_t)chunk * a.chunk_floats;
    bool first_flush = true;
    int64_t g = 0;
    for (int64_t ks = ks_begin; ks < ks_end; ++ks, ++g) {
      const int bst = (int)(g % kSepBStages), tst = (int)(g % kSepTStages);
      // B stage bst is free once the MMAs of step g - kSepBStages completed;
      // every lane waits, the warp agrees on the outcome
      bool w = !s_abort;
      if (w && g >= kSepBStages)
        w = dev::mbar_wait_bounded(&bar_done[(g - kSepBStages) & (n_a - 1)], (uint32_t)(((g - kSepBStages) >> la) & 1));
      if (w) w = dev::mbar_wait_bounded(&bar_atom[tst], (uint32_t)((g / kSepTStages) & 1));
      if (!__all_sync(0xffffffffu, w)) {
        ok = false;
        break;
      }
      // B[col, k] = e^{2 pi i (s_b y' + s_c z' + c)}, zero past the last column
      unsigned char* sB = ringB + bst * kSepBBytes;
      const float4* at = ring_atom[tst];
      if constexpr (FOLD) {
        const int kb = tid / (narrow ? kSepFoldPairs / 2 : kSepFoldPairs);
        if (kb < 4) {  // narrow: half of the warps
          uint4 hi[2], lo[2];
          hi[0] = hi[1] = lo[0] = lo[1] = make_uint4(0u, 0u, 0u, 0u);
          if (row_ok) {
            if (exact)
              sep_b_fold<2>(sb, sc, sbl, scl, at + kb * 8, hi, lo);
            else if (reduce)
              sep_b_fold<1>(sb, sc, sbl, scl, at + kb * 8, hi, lo);
            else
              sep_b_fold<0>(sb, sc, sbl, scl, at + kb * 8, hi, lo);
          }
          unsigned char* q = sB + kb * 4096 + b_row_off;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            *reinterpret_cast<uint4*>(q + u * 1024) = hi[u];
            *reinterpret_cast<uint4*>(q + 16384 + u * 1024) = lo[u];
          }
        }
      } else {
      // mode 0: raw phase, 1: reduced mod 1, 2: exact products, reduced
      // kAtt: a buried object's rows carry exp(-att z')
      auto form = [&](auto mode_tag, auto att_tag) {
        constexpr int kMode = decltype(mode_tag)::value;
        constexpr bool kAtt = decltype(att_tag)::value;
#pragma unroll
        for (int kq = 0; kq < 2; ++kq) {
          const int kb = 2 * (tid / kSepN) + kq;  // two threads per column
          uint32_t hi[4] = {0u, 0u, 0u, 0u}, lo[4] = {0u, 0u, 0u, 0u};
          if (row_ok) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float4 v = at[kb * 4 + q];
              const float ph =
                  kMode == 2 ? dev::frac_rn(dev::frac_product2_plus(sb, sbl, v.y,
                                                                    dev::frac_product2_plus(sc, scl, v.z, v.w)))
                  : kMode == 1 ? dev::frac_rn(fmaf(sb, v.y, fmaf(sc, v.z, v.w)))
                               : fmaf(sb, v.y, fmaf(sc, v.z, v.w));
              float sn, cs;
              dev::sincos_cycles_mufu(ph, &sn, &cs);
              if (kAtt) {
                float ex = -att * v.z;
                if (ex > kSepAttMax) {
                  ex = kSepAttMax;
                  att_over = true;
                }
                const float gz = __expf(ex);
                sn *= gz;
                cs *= gz;
              }
              split2(cs, sn, hi[q], lo[q]);
            }
          }
          *reinterpret_cast<uint4*>(sB + kb * 4096 + b_row_off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(sB + 16384 + kb * 4096 + b_row_off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      };
      auto form_all = [&](auto att_tag) {
        if (exact)
          form(std::integral_constant<int, 2>{}, att_tag);
        else if (reduce)
          form(std::integral_constant<int, 1>{}, att_tag);
        else
          form(std::integral_constant<int, 0>{}, att_tag);
      };
      if (a.axis_att)
        form_all(std::true_type{});
      else
        form_all(std::false_type{});
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&bar_bfull[bst]);
        mbar_arrive(&bar_tempty[tst]);
      }
      if (!grp.ends_at(ks)) continue;

      // ---- group end: TMEM -> blocked partials -------------------------------
      // the commit of step g covers every earlier MMA of the group
      w = dev::mbar_wait_bounded(&bar_done[g & (n_a - 1)], (uint32_t)((g >> la) & 1));
      if (!__all_sync(0xffffffffu, w)) {
        ok = false;
        break;
      }
      tc_fence_after();
      // TMEM lane = row (2 pa + ri) of this CTA's tile: one 32 x 32 block of
      // the partials per load; padding rows and columns are written too
      const int sub = warp & 3;
      const int col0 = (warp >> 2) * kSpan;
      for (int tp = 0; tp < ntp; ++tp) {
        const int64_t m0 = (2 * mp + tp) * kSepM + sub * 32;
#pragma unroll 1
        for (int cc = 0; cc < kSpan; cc += 32) {
          const int64_t bc0 = col_base + col0 + cc;
          if (bc0 >= col_end) break;
          float4* blk = reinterpret_cast<float4*>(part + sep_part_off(m0, bc0, a.n_cb)) + lane;
          float v[32];
          tmem_ld32(tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)(tp * kSepN + col0 + cc), v);
          // the first read-out stores, later ones add in L2 (reductions, no
          // load round trip); every element belongs to this CTA and its
          // updates come from this thread in program order, so the sum is
          // deterministic
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float4 x = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            if (first_flush)
              blk[q * 32] = x;
            else
              atomicAdd(blk + q * 32, x);
          }
        }
      }
      first_flush = false;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_tfree);
      grp.advance(ks);
    }
    if (att_over) dev::set_status(a.status, kStatusNonFinite);
    if (ok && first_flush) {
      // empty chunk: its partials are zero
      const int sub = warp & 3;
      const int col0 = (warp >> 2) * kSpan;
      for (int tp = 0; tp < ntp; ++tp) {
        const int64_t m0 = (2 * mp + tp) * kSepM + sub * 32;
        for (int cc = 0; cc < kSpan && col_base + col0 + cc < col_end; cc += 32) {
          float4* blk = reinterpret_cast<float4*>(part + sep_part_off(m0, col_base + col0 + cc, a.n_cb)) + lane;
          for (int q = 0; q < 8; ++q) blk[q * 32] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
  }
  if (!ok) {
    s_abort = 1;
    dev::set_status(a.status, kStatusTimeout);
  }
  __syncthreads();
  // on abort, wait (bounded) for MMAs and copies still in flight before
  // releasing TMEM and shared memory; phases already complete return at once
  if (mma_warp && lane == 0 && s_abort && g_committed > 0) {
    const int64_t gl = g_committed - 1;
    dev::mbar_wait_bounded(&bar_done[gl & (n_a - 1)], (uint32_t)((gl >> la) & 1), 1LL << 28);
  }
  if (copy_warp && lane == 0 && s_abort) {
    for (int64_t s = a_issued > n_a ? a_issued - n_a : 0; s < a_issued; ++s)
      dev::mbar_wait_bounded(&bar_full[s & (n_a - 1)], (uint32_t)((s >> la) & 1), 1LL << 28);
    for (int64_t s = t_issued > kSepTStages ? t_issued - kSepTStages : 0; s < t_issued; ++s)
      dev::mbar_wait_bounded(&bar_atom[s % kSepTStages], (uint32_t)((s / kSepTStages) & 1), 1LL << 28);
  }
  tc_fence_before();
  __syncthreads();
  if (mma_warp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSepTmemCols));
}

// Sum over the chunks in order of f_s(|S|) x T_chunk (Eq. 2: each chunk holds
// one species s), translation phase, outputs.
// Sum of the chunks' partials with f_s(|S|) per chunk's species, the
// centring phase and |A|^2.  One CTA per 32 x 32 block of the blocked
// partials (16 h values x 32 (k, l) columns, 512 points): each chunk's block
// is 4 KB contiguous and is read as one float4 per thread, thread t holding
// D row t % 32 (Re of h row (t % 32) / 2 for even t % 32, Im for odd) of the
// columns 4 (t / 32) .. +3.  One exchange between the two lanes of a row
// pair gives lane 2i columns 4q, 4q+1 and lane 2i+1 columns 4q+2, 4q+3 (two
// points each).  The sum over chunks runs in chunk order, eight chunks' loads
// in flight.
__global__ void __launch_bounds__(256) k_sep_reduce(const float* __restrict__ partial, int64_t chunk_floats,
                                                    int64_t n_cb, const Segment* __restrict__ chunks, int n_chunks,
                                                    const float* __restrict__ coef, const float2* __restrict__ ftab,
                                                    float inv4a2, const float* __restrict__ axis_s,
                                                    const float* __restrict__ axis_lo, int64_t n0, int64_t n1,
                                                    int64_t n2, float3 H, const double* __restrict__ shift,
                                                    const float* __restrict__ att, const float* __restrict__ szf,
                                                    int64_t bm_base, float2* out_amp, float* out_int,
                                                    const CallGate gate) {
  if (within(gate, 0)) return;
  // the centring shift of the call (integers), once per block
  __shared__ float sh_t[3];
  __shared__ int sh_shifted;
  if (threadIdx.x == 0) {
    sh_t[0] = (float)shift[0];
    sh_t[1] = (float)shift[1];
    sh_t[2] = (float)shift[2];
    sh_shifted = shift[0] != 0.0 || shift[1] != 0.0 || shift[2] != 0.0;
  }
  __syncthreads();
  const int t = threadIdx.x, lane = t & 31, odd = lane & 1;
  const int64_t bm = bm_base + blockIdx.y, bc = blockIdx.x;
  const int64_t ncols = n1 * n2, n_s = n0 * ncols;
  const int64_t i0 = bm * 16 + (lane >> 1);
  const int64_t col0 = bc * 32 + (t >> 5) * 4 + odd * 2;  // the thread's two columns
  // per point: double-float offsets s, |S|^2 / (4 a^2) in FP32 (S = H + s)
  float s_hi[2][3], s_lo[2][3], s2[2];
  bool ok[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int64_t col = col0 + u;
    ok[u] = i0 < n0 && col < ncols;
    const int64_t ia[3] = {ok[u] ? i0 : 0, n0 + (ok[u] ? col / n2 : 0), n0 + n1 + (ok[u] ? col % n2 : 0)};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      s_hi[u][d] = axis_s[ia[d]];
      s_lo[u][d] = axis_lo[ia[d]];
    }
    // (a buried object's form factor is taken at the vacuum beam's S_z)
    const int64_t il = ia[2] - n0 - n1;
    const float S0 = H.x + (s_hi[u][0] + s_lo[u][0]), S1 = H.y + (s_hi[u][1] + s_lo[u][1]),
                S2 = szf ? szf[il] : H.z + (s_hi[u][2] + s_lo[u][2]);
    s2[u] = (S0 * S0 + S1 * S1 + S2 * S2) * inv4a2;
  }
  const int64_t m0 = i0 * ncols + col0;
  const float* blk = partial + (bm * n_cb + bc) * 1024 + 4 * t;
  float2 v[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, F[2] = {v[0], v[1]};
  int cur = -1;
  constexpr int kU = 8;
  for (int c0 = 0; c0 < n_chunks; c0 += kU) {
    float4 x[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      x[u] = c0 + u < n_chunks ? __ldcs(reinterpret_cast<const float4*>(blk + (int64_t)(c0 + u) * chunk_floats))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      if (c0 + u >= n_chunks) break;  // uniform over the block
      // even lane: Re of columns 4q..4q+3, needs Im of 4q, 4q+1; odd lane:
      // Im, needs Re of 4q+2, 4q+3
      const float sx = odd ? x[u].x : x[u].z, sy = odd ? x[u].y : x[u].w;
      const float rx = __shfl_xor_sync(0xffffffffu, sx, 1), ry = __shfl_xor_sync(0xffffffffu, sy, 1);
      const float re[2] = {odd ? rx : x[u].x, odd ? ry : x[u].y};
      const float im[2] = {odd ? x[u].z : rx, odd ? x[u].w : ry};
      const int sp = chunks[c0 + u].species;
      if (sp != cur) {
#pragma unroll
        for (int w = 0; w < 2; ++w)
          F[w] = ftab ? (ok[w] ? ftab[(int64_t)sp * n_s + m0 + w] : make_float2(0.f, 0.f))
                      : dev::form_factor(coef + kNCoef * sp, s2[w]);
        cur = sp;
      }
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        v[w].x += F[w].x * re[w] - F[w].y * im[w];
        v[w].y += F[w].x * im[w] + F[w].y * re[w];
      }
    }
  }
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    if (!ok[w]) continue;
    float2 a = v[w];
    if (sh_shifted) a = dev::cmul(dev::shift_phase2(s_hi[w], s_lo[w], sh_t), a);
    if (att) {
      // a buried object's attenuation over the centring shift t_z (the rows
      // carried exp(-2 pi Im(sigma) z') of the centred z')
      const float g = __expf(-att[(col0 + w) % n2] * sh_t[2]);
      a.x *= g;
      a.y *= g;
    }
    if (out_amp) out_amp[m0 + w] = a;
    if (out_int) out_int[m0 + w] = a.x * a.x + a.y * a.y;
  }
}

struct SepFoldReduceArgs {
  const float* partial;
  int64_t chunk_floats, n_cb;
  const Segment* chunks;
  int n_chunks;
  const float* coef;
  const float2* ftab;
  float inv4a2;
  const float* axis_s;   // [n0 | n1 | n2] s = axis - H, and rounding errors
  const float* axis_lo;
  int64_t n0, n1, n2, n_pairs, n_lanes;
  int fold_h;
  float H[3];
  const double* shift;
  int64_t l8_base;       // first block of 8 lanes of this launch
  float2* out_amp;
  float* out_int;
  CallGate gate;
};

// The reduction of the folded forward: per species run of the chunks the
// eight real sums of every (lane, pair), then their four points (two h values,
// a point and its mirror) with f_s at each point's own |S|, and at the end the
// centring phase and |A|^2.  A thread holds one lane's rows and four pairs:
// rows l % 8 and quad l / 8 of pairs, so a read covers 128 contiguous bytes
// per quad, and the four row blocks and the two columns of a pair (blocks of
// the partials that the same thread reads) combine with no exchange.  GROUPS
// threads share a quadruple's chunks on small maps and meet in shared memory in a
// fixed order (64 CTAs of seven chunks: 21.5 us with one thread per quadruple,
// 12.7 us with four; 51 x 51 nodes of 150 chunks: 35 us with eight,
// 19 us with 32).
template <int GROUPS>
__global__ void __launch_bounds__(256) k_sep_reduce_fold(const SepFoldReduceArgs a) {
  if (within(a.gate, 0)) return;
  constexpr int kCols = 256 / GROUPS;  // threads over (alpha, quad)
  __shared__ float sh_t[3];
  __shared__ int sh_shifted;
  __shared__ float sh_v[GROUPS > 1 ? GROUPS - 1 : 1][GROUPS > 1 ? 32 : 1][GROUPS > 1 ? kCols : 1];
  if (threadIdx.x == 0) {
    sh_t[0] = (float)a.shift[0];
    sh_t[1] = (float)a.shift[1];
    sh_t[2] = (float)a.shift[2];
    sh_shifted = a.shift[0] != 0.0 || a.shift[1] != 0.0 || a.shift[2] != 0.0;
  }
  const int t = threadIdx.x % kCols, grp = threadIdx.x / kCols;
  const int64_t lg = (a.l8_base + blockIdx.y) * 8 + (t & 7);  // lane of the map: 32 per M tile
  const int64_t p0 = ((int64_t)blockIdx.x * (kCols / 8) + (t >> 3)) * 4;
  const int64_t ncols = a.n1 * a.n2, n_s = a.n0 * ncols;
  int64_t ia[2];
  bool a_ok[2];
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    ia[w] = sep_fold_a(lg >> 5, (int)(lg & 31), w, a.fold_h, a.n0);
    a_ok[w] = a.fold_h ? lg < a.n_lanes && (w == 0 || ia[1] != ia[0]) : ia[w] < a.n_lanes;
    if (!a_ok[w]) ia[w] = 0;
  }
  const bool l_ok = a_ok[0] || a_ok[1];
  // |S|^2 parts in FP32 (S = H + s): of the two h values, of the points p and p'
  float h2[2], q2[4][2];
  auto s_of = [&](int64_t i, int d) { return a.H[d] + (a.axis_s[i] + a.axis_lo[i]); };
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const float x = s_of(ia[u], 0);
    h2[u] = x * x;
  }
  bool p_ok[4];
  int64_t pt[4][2];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    p_ok[j] = l_ok && p0 + j < a.n_pairs;
    pt[j][0] = p_ok[j] ? p0 + j : 0;
    pt[j][1] = ncols - 1 - pt[j][0];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float y = s_of(a.n0 + pt[j][u] / a.n2, 1), z = s_of(a.n0 + a.n1 + pt[j][u] % a.n2, 2);
      q2[j][u] = y * y + z * z;
    }
  }
  // block (row block r, cos | sin) of this thread's lane and pairs: the M tile
  // lg / 32 has four consecutive 32-row blocks, the pair group p0 / 64 its cos
  // and sin columns in two pairs of 32-column blocks
  const int64_t c = (p0 >> 6) * 128 + (p0 & 63);
  const bool in = l_ok && p0 < (a.n_pairs + 63) / 64 * 64;
  const float* base = a.partial + sep_part_off((lg >> 5) * 128 + (lg & 31), c, a.n_cb);
  const int64_t r_off = a.n_cb * 1024, s_off = 2 * 1024;
  float2 v[4][4];  // [pair][first h value: p, p' | second: p, p']
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int k = 0; k < 4; ++k) v[j][k] = make_float2(0.f, 0.f);
  float4 z[4][2];
  auto zero = [&]() {
#pragma unroll
    for (int r = 0; r < 4; ++r) z[r][0] = z[r][1] = make_float4(0.f, 0.f, 0.f, 0.f);
  };
  zero();
  const int per = (a.n_chunks + GROUPS - 1) / GROUPS;
  const int c_lo = grp * per, c_hi = min(a.n_chunks, c_lo + per);
  for (int ch = c_lo; ch < c_hi; ++ch) {
    const int sp = a.chunks[ch].species;
    if (in) {
      const float* q = base + (int64_t)ch * a.chunk_floats;
      float4 x[4][2];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int y = 0; y < 2; ++y) x[r][y] = __ldcs(reinterpret_cast<const float4*>(q + r * r_off + y * s_off));
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          z[r][y].x += x[r][y].x;
          z[r][y].y += x[r][y].y;
          z[r][y].z += x[r][y].z;
          z[r][y].w += x[r][y].w;
        }
    }
    if (ch + 1 < c_hi && a.chunks[ch + 1].species == sp) continue;  // uniform over the group
    const float* cf = a.coef + kNCoef * sp;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      auto e = [&](const float4& f) { return j == 0 ? f.x : j == 1 ? f.y : j == 2 ? f.z : f.w; };
      // C and S of the two h values
      float cr[2], ci[2], sr[2], si[2];
      const float c0 = e(z[0][0]), c1 = e(z[1][0]), c2 = e(z[2][0]), c3 = e(z[3][0]);
      const float s0 = e(z[0][1]), s1 = e(z[1][1]), s2 = e(z[2][1]), s3 = e(z[3][1]);
      cr[0] = a.fold_h ? c0 - c3 : c0;
      ci[0] = a.fold_h ? c1 + c2 : c1;
      cr[1] = a.fold_h ? c0 + c3 : c2;
      ci[1] = a.fold_h ? c1 - c2 : c3;
      sr[0] = a.fold_h ? s0 - s3 : s0;
      si[0] = a.fold_h ? s1 + s2 : s1;
      sr[1] = a.fold_h ? s0 + s3 : s2;
      si[1] = a.fold_h ? s1 - s2 : s3;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        // p runs over the first half of the points, whose offsets are the formed ones: C + i S, its mirror C - i S
        const int w = k >> 1;
        const float re = k & 1 ? cr[w] + si[w] : cr[w] - si[w];
        const float im = k & 1 ? ci[w] - sr[w] : ci[w] + sr[w];
        const float2 F = a.ftab ? (p_ok[j] ? a.ftab[(int64_t)sp * n_s + ia[k >> 1] * ncols + pt[j][k & 1]]
                                           : make_float2(0.f, 0.f))
                                : dev::form_factor(cf, (h2[k >> 1] + q2[j][k & 1]) * a.inv4a2);
        v[j][k].x += F.x * re - F.y * im;
        v[j][k].y += F.x * im + F.y * re;
      }
    }
    zero();
  }
  __syncthreads();  // sh_t; and before the groups' exchange
  if constexpr (GROUPS > 1) {
    if (grp > 0) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          sh_v[grp - 1][8 * j + 2 * k][t] = v[j][k].x;
          sh_v[grp - 1][8 * j + 2 * k + 1][t] = v[j][k].y;
        }
    }
    __syncthreads();
    if (grp > 0) return;
    for (int g = 0; g < GROUPS - 1; ++g)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          v[j][k].x += sh_v[g][8 * j + 2 * k][t];
          v[j][k].y += sh_v[g][8 * j + 2 * k + 1][t];
        }
  }
  if (!l_ok) return;
  if (sh_shifted) {
    // e^{2 pi i s.t}: the products' fractional parts per axis value
    float fh[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) fh[u] = dev::frac_of_product2(a.axis_s[ia[u]], a.axis_lo[ia[u]], sh_t[0]);
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int64_t iy = a.n0 + pt[j][u] / a.n2, iz = a.n0 + a.n1 + pt[j][u] % a.n2;
        const float fy = dev::frac_of_product2(a.axis_s[iy], a.axis_lo[iy], sh_t[1]);
        const float fz = dev::frac_of_product2(a.axis_s[iz], a.axis_lo[iz], sh_t[2]);
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          float sn, cs;
          sincospif(2.0f * dev::frac_rn(fh[w] + fy + fz), &sn, &cs);
          v[j][2 * w + u] = dev::cmul(make_float2(cs, sn), v[j][2 * w + u]);
        }
      }
  }
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    if (!a_ok[w]) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (!p_ok[j] || (u == 1 && pt[j][1] == pt[j][0])) continue;  // the middle point of an odd plane
        const int64_t m = ia[w] * ncols + pt[j][u];
        const float2 x = v[j][2 * w + u];
        if (a.out_amp) a.out_amp[m] = x;
        if (a.out_int) a.out_int[m] = x.x * x.x + x.y * x.y;
      }
  }
}

// -------------------------------------------------------------------------
// host side
// -------------------------------------------------------------------------

bool sep_axis_middle(const std::vector<double>& v, double H, double* mid) {
  if (!axis_symmetric(v, mid)) return false;
  return v.size() == 1 || std::fabs(*mid - H) <= 0.125 * std::fabs(v.back() - v.front()) + 1e-12;
}

cudaError_t sep_prepare_kernel() {
  static_assert(kSepSmem + 8192 <= 227 * 1024, "dynamic + static shared memory of k_sep");
  cudaError_t e = cudaFuncSetAttribute(k_sep<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSepSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_sep<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSepSmem);
  return e != cudaSuccess ? e : sep_pair_prepare_kernel();
}

// grid: x = M-tile pairs x N tiles, y = chunks.  The CTA-pair kernel
// (sep_pair.cu) covers the same tiles with two M-tile pairs per cluster.  An
// odd last pair runs on the one-CTA kernel (a pair cluster with one
// accumulator tile would form all of its B columns for half the MMA work),
// on the side stream where one is given, so that its CTAs take the SMs the
// pair kernel's last clusters leave idle.
static void launch_one_cta(const SepArgs& a, dim3 grid, cudaStream_t st) {
  if (a.fold)
    k_sep<true><<<grid, 32 * (kSepOneWarps + 2), kSepSmem, st>>>(a);
  else
    k_sep<false><<<grid, 32 * (kSepOneWarps + 2), kSepSmem, st>>>(a);
}

cudaError_t sep_launch_core(const SepArgs& a, dim3 grid, cudaStream_t st, cudaStream_t side, cudaEvent_t fork,
                            cudaEvent_t join) {
  const int64_t n_mp = (a.n_mt + 1) / 2;
  const int64_t n_nt = (int64_t)grid.x / n_mp;
  const int64_t n_even = n_mp & ~int64_t(1);
  if (!sep_pair_enabled() || n_even == 0) {
    launch_one_cta(a, grid, st);
    return cudaGetLastError();
  }
  SepArgs pa = a;
  pa.mp_first = 0;
  pa.mp_count = n_even;
  SepArgs sa = a;
  sa.mp_first = n_even;
  sa.mp_count = 1;
  const bool split = n_even < n_mp;
  const bool beside = split && side && fork && join;
  cudaError_t e = cudaSuccess;
  if (beside && ((e = cudaEventRecord(fork, st)) != cudaSuccess || (e = cudaStreamWaitEvent(side, fork, 0)) != cudaSuccess))
    return e;
  e = sep_pair_launch_core(pa, n_nt, (int)grid.y, st);
  if (split) {
    if (e == cudaSuccess) {
      launch_one_cta(sa, dim3((unsigned)n_nt, grid.y), beside ? side : st);
      e = cudaGetLastError();
    }
    if (beside) {  // join even after a failed launch: a capture needs the side stream back
      const cudaError_t ej = cudaEventRecord(join, side);
      const cudaError_t ew = ej == cudaSuccess ? cudaStreamWaitEvent(st, join, 0) : ej;
      if (e == cudaSuccess) e = ew;
    }
  }
  return e;
}

scatter_status sep_prepare_side(scatter_plan_s* p, int64_t n_mt) {
  if (sep_core_launches(n_mt) < 2 || p->side_stream) return SCATTER_OK;
  cudaError_t e;
  if ((e = cudaStreamCreateWithFlags(&p->side_stream, cudaStreamNonBlocking)) != cudaSuccess)
    return cuda_status(e, "side stream");
  if ((e = cudaEventCreateWithFlags(&p->side_fork, cudaEventDisableTiming)) != cudaSuccess ||
      (e = cudaEventCreateWithFlags(&p->side_join, cudaEventDisableTiming)) != cudaSuccess)
    return cuda_status(e, "side stream events");
  return SCATTER_OK;
}

int sep_core_launches(int64_t n_mt) {
  const int64_t n_mp = (n_mt + 1) / 2;
  return (sep_pair_enabled() && n_mp >= 2 && n_mp % 2 == 1) ? 2 : 1;
}

namespace {

// Smallest crystal (atom slots) whose map is folded: AUTO's own line below
// which a grid is not sent to the tensor cores, a few hundred steps of atoms
// bound by fixed costs that the fold does not change.
constexpr int64_t kSepFoldMinSlots = 4096;

// Atom chunks: every species segment split into step-aligned pieces, about
// `split` pieces in all, so that each chunk carries a single form factor.
std::vector<Segment> sep_chunks(const scatter_plan_s* p, int split, int step) {
  std::vector<Segment> chunks;
  int64_t total_steps = 0;
  for (const Segment& sg : p->all_segs)
    if (sg.instance == 0 && sg.end > sg.begin) total_steps += (sg.end - sg.begin) / step;
  for (const Segment& sg : p->all_segs) {
    if (sg.instance != 0 || sg.end <= sg.begin) continue;
    const int64_t steps = (sg.end - sg.begin) / step;
    const int64_t k = std::max<int64_t>(1, std::llround((double)split * (double)steps / (double)total_steps));
    const int64_t per = (steps + k - 1) / k;
    for (int64_t b = 0; b < steps; b += per)
      chunks.push_back(Segment{sg.begin + b * step, sg.begin + std::min(steps, b + per) * step, sg.species, 0});
  }
  return chunks;
}

// Mean steps of the accumulation group that a step lies in, for chunks flushed
// every `flush` steps: the truncation error of a map grows with it.
double sep_mean_group(const std::vector<Segment>& chunks, int step, int64_t flush) {
  double sq = 0.0, all = 0.0;
  for (const Segment& c : chunks) {
    const int64_t n = (c.end - c.begin) / step, full = n / flush, rest = n % flush;
    sq += (double)full * (double)flush * (double)flush + (double)rest * (double)rest;
    all += (double)n;
  }
  return all > 0.0 ? sq / all : 0.0;
}

}  // namespace

double sep_direct_group(const scatter_plan_s* p) {
  return sep_mean_group(sep_chunks(p, p->sep_direct.split, kSepStep), kSepStep, kSepFlush);
}

namespace {

// Atom chunks (split over K) of `steps` steps in all that minimise the waves
// of CTAs x steps per CTA, each chunk at least min_steps long; *cost_out in
// steps.
int sep_best_split(const scatter_plan_s* p, int64_t tiles, int64_t n_steps, double min_steps, double* cost_out) {
  const double cap = (double)p->n_sm;  // one CTA per SM (TMEM + shared memory)
  const double steps = (double)std::max<int64_t>(n_steps, 1);
  double best = 1e300;
  int best_k = 1;
  // up to two chunks per SM: a grid of one N tile and one M quad (a few
  // columns, a long atom list) needs ~n_sm / 2 chunks to give every SM a CTA
  for (int k = 1; k <= 2 * p->n_sm; ++k) {
    if (k > 1 && steps / k < min_steps) break;
    // one step ~1 us of MMA; an extra chunk costs one partial of the
    // map (8 B per point written once, read once by the reduction)
    const double part_steps = 16.0 * (double)p->sep_ns / 6.0e12 / 1.0e-6;
    const double cost = std::ceil((double)tiles * k / cap) * (steps / k + 40.0) + (k > 1 ? k * part_steps : 0.0);
    if (cost < best * 0.995) {
      best = cost;
      best_k = k;
    }
  }
  *cost_out = best;
  return best_k;
}

}  // namespace

// The separable grid: the plan's own axes, or for a grazing-incidence plan
// the virtual grid (h, k, l) whose l axis stacks the four beams' Sz values
// [Sz1 | Sz2 | -Sz2 | -Sz1] over alpha_f, so each beam is a plain grid sum.
// A buried object has one beam, l = Re(sigma) per alpha_f; its formed rows
// carry the attenuation exp(-2 pi Im(sigma) z') and its form factor is taken
// at the vacuum beam S_1 (the per-column tables sep_att and sep_szf).
scatter_status prepare_separable(scatter_plan_s* p, int split_override) {
  const bool gid = p->s_kind == SCATTER_S_GID_GRID;
  if ((p->s_kind != SCATTER_S_GRID && !gid) || p->batch != 1)
    return fail(SCATTER_ERR_UNSUPPORTED, "the separable path needs a single axis-aligned grid");
  if (p->n_slots % kSepStep) return fail(SCATTER_ERR_UNSUPPORTED, "slot padding is not a multiple of 16");
  std::vector<double> ax64[3];
  for (int d = 0; d < 2; ++d) ax64[d] = p->axis_host[d];
  const bool buried = gid && p->gid_mode == 1;
  std::vector<float> att, szf;
  p->sep_beams = buried ? 1 : 4;
  if (buried) {
    const int64_t n_af = p->n_axis[2];
    ax64[2].assign(p->gid_sz_host.begin(), p->gid_sz_host.begin() + n_af);
    for (int64_t i = 0; i < n_af; ++i) {
      att.push_back((float)(6.283185307179586 * p->gid_sz_im_host[i]));
      szf.push_back((float)p->gid_szf_host[i]);
    }
  } else if (gid) {
    const int64_t n_af = p->n_axis[2];
    ax64[2].resize(4 * n_af);
    for (int64_t i = 0; i < n_af; ++i) {
      const double z1 = p->gid_sz_host[i], z2 = p->gid_sz_host[n_af + i];
      ax64[2][i] = z1;
      ax64[2][n_af + i] = z2;
      ax64[2][2 * n_af + i] = -z2;
      ax64[2][3 * n_af + i] = -z1;
    }
  } else {
    ax64[2] = p->axis_host[2];
  }
  std::vector<float> alls, alls_lo;
  for (int d = 0; d < 3; ++d) {
    p->sep_n[d] = (int64_t)ax64[d].size();
    for (double v : ax64[d]) {
      const double sv = v - p->inst[0].H[d];
      alls.push_back((float)sv);
      alls_lo.push_back((float)(sv - (double)(float)sv));
    }
  }
  p->sep_ns = p->sep_n[0] * p->sep_n[1] * p->sep_n[2];
  const int64_t nbc = p->sep_n[1] * p->sep_n[2];
  // The direct form
  SepForm& fd = p->sep_direct;
  fd.mt = (2 * p->sep_n[0] + kSepM - 1) / kSepM;
  fd.cols = nbc;
  fd.nt = (fd.cols + kSepN - 1) / kSepN;
  fd.steps = p->n_slots / kSepStep;
  fd.flush = kSepFlush;
  double cost_d = 0.0, cost_f = 0.0;
  fd.split = split_override > 0 ? split_override
                                : sep_best_split(p, (fd.mt + 1) / 2 * fd.nt, fd.steps, std::max(64.0, p->sep_group), &cost_d);
  // The folded form, where the (k, l) axes are symmetric (evenly spaced axes)
  // and the crystal has at least kSepFoldMinSlots slots, for amplitude calls.
  // Not on grazing incidence: near the critical angle the four beams nearly
  // cancel, and the errors of a point and its mirror (opposite beams), one
  // sum's in the fold, no longer cancel with them (2-3 times the direct form's
  // scatter on some maps).  The accumulators' truncation grows with the steps
  // of a group, so the fold takes chunks that allow 0.95 of the direct form's mean
  // group, where that leaves it the cheaper form by the cost model, and flushes
  // them at 0.65 of it: a strong point leaves its error on its mirror, and at 0.95
  // maps of coherent crystals were up to 1.53 times as far from FP64 as the direct
  // form's (26 drawn maps, 0.71-1.53; at 0.75 0.58-1.22, at 0.65 0.51-1.05, up to
  // 3 % of the time).  Sums at nodes keep 0.95 of theirs: they are below it.
  // Intensities keep the direct form: |A|^2 doubles the forms' difference.
  SepForm& ff = p->sep_folded;
  double mid[3] = {0, 0, 0};
  ff.fold = !gid && p->n_slots >= kSepFoldMinSlots && p->n_slots % kSepFoldStep == 0 &&
            sep_axis_middle(ax64[1], p->inst[0].H[1], &mid[1]) && sep_axis_middle(ax64[2], p->inst[0].H[2], &mid[2]);
  if (ff.fold) {
    ff.fold_h = sep_axis_middle(ax64[0], p->inst[0].H[0], &mid[0]);
    ff.lanes = ff.fold_h ? (p->sep_n[0] + 1) / 2 : p->sep_n[0];
    ff.pairs = (nbc + 1) / 2;
    ff.mt = ff.fold_h ? (ff.lanes + 31) / 32 : (ff.lanes + kSepFoldRows - 1) / kSepFoldRows;
    ff.cols = sep_fold_cols(ff.pairs);
    ff.nt = (ff.cols + kSepN - 1) / kSepN;
    ff.steps = p->n_slots / kSepFoldStep;
    const double group = 0.95 * (p->sep_group > 0.0 ? p->sep_group : sep_direct_group(p));
    ff.split = fd.split;
    if (split_override <= 0) {
      ff.split = sep_best_split(p, (ff.mt + 1) / 2 * ff.nt, ff.steps, group, &cost_f);
      ff.fold = cost_f < 0.95 * cost_d && (double)ff.steps >= 0.9 * group;
    }
    const std::vector<Segment> cf = sep_chunks(p, ff.split, kSepFoldStep);
    const double flush_group = p->sep_group > 0.0 ? group : group * (0.65 / 0.95);
    double off = 1e300;
    for (int f = 1; f <= kSepFlush + kSepFlush / 2; ++f) {
      const double d = std::fabs(sep_mean_group(cf, kSepFoldStep, f) - flush_group);
      if (d < off) {
        off = d;
        ff.flush = f;
      }
    }
  }
  std::vector<float> dvals, dvals_lo;
  if (ff.fold) {
    for (int d = 0; d < 3; ++d) {
      const bool fold_d = d > 0 || ff.fold_h;
      if (!fold_d) mid[d] = p->inst[0].H[d];  // an h axis that is not folded: offsets from H
      p->sep_mid[d] = mid[d] - p->inst[0].H[d];
      const size_t n = ax64[d].size();
      for (size_t i = 0; i < n; ++i) {
        const double dv = fold_d ? 0.5 * (ax64[d][i] - ax64[d][n - 1 - i]) : ax64[d][i] - mid[d];
        dvals.push_back((float)dv);
        dvals_lo.push_back((float)(dv - (double)(float)dv));
      }
    }
  }
  Tiling t;
  t.threads = 256;
  t.R = 8;
  t.split_k = fd.split;
  // chunk tables (segments) as for the generic path; the partial buffer is blocked
  scatter_status st = apply_tiling(p, t);
  if (st != SCATTER_OK) return st;
  if (p->d.partial) {  // the generic path's partials are not used here
    cudaFree(p->d.partial);
    p->d.partial = nullptr;
  }
  cudaError_t e;
  size_t bytes = 0;
  auto alloc = [&](auto** dst, size_t size) {
    bytes += size;
    return injected_alloc_failure() ? cudaErrorMemoryAllocation : cudaMalloc((void**)dst, size);
  };
  auto put = [&](auto** dst, const auto& v) {
    const size_t size = v.size() * sizeof(v[0]);
    const cudaError_t r = alloc(dst, size);
    return r != cudaSuccess ? r : cudaMemcpy(*dst, v.data(), size, cudaMemcpyHostToDevice);
  };
  // Chunk tables, A table, partials and offsets of the direct form, and of the folded one
  auto make = [&](bool fold) {
    cudaError_t r = cudaSuccess;
    size_t a_bytes = 0, part_bytes = 0;
    for (SepForm* f : {&fd, &ff}) {
      if (f == &ff && !fold) break;
      const std::vector<float>& off = f->fold ? dvals : alls;  // offsets that the kernels form phases from
      for (int64_t i = 0; i < p->sep_n[1]; ++i) f->smax[0] = std::max(f->smax[0], std::fabs(off[p->sep_n[0] + i]));
      for (int64_t i = 0; i < p->sep_n[2]; ++i)
        f->smax[1] = std::max(f->smax[1], std::fabs(off[p->sep_n[0] + p->sep_n[1] + i]));
      // With one N tile every A tile is read by one cluster only: the CTA pair
      // then forms its A tiles itself from the atom records (the same arithmetic
      // as k_sep_tab_a), and the table, written and read once, is not kept.
      // With several N tiles that formation would repeat per tile, so the table
      // stays; an odd pair count runs its last pair on the one-CTA kernel, which
      // reads the table.
      const int64_t n_mp = (f->mt + 1) / 2;
      f->form_a = sep_pair_enabled() && n_mp % 2 == 0 && f->nt == 1;
      if (!f->form_a)
        a_bytes = std::max(a_bytes, (size_t)(2 * n_mp) * (size_t)std::max<int64_t>(f->steps, 1) * kSepABytes);
      std::vector<Segment> chunks = sep_chunks(p, f->split, f->fold ? kSepFoldStep : kSepStep);
      if (chunks.empty()) chunks.push_back(Segment{0, 0, 0, 0});  // no atoms: one empty chunk, zero partials
      f->n_chunks = (int32_t)chunks.size();
      part_bytes = std::max(part_bytes, (size_t)f->n_chunks * (size_t)sep_part_floats(f->mt, f->cols) * sizeof(float));
      if ((r = put(&f->chunks, chunks)) != cudaSuccess) return r;
    }
    if (a_bytes) {
      // tiles past the last row are never written by the table kernel (the
      // CTA-pair kernel streams the second tile of a pair always; its rows are
      // never read): zero them once
      if ((r = alloc(&p->d.sep_A, a_bytes)) != cudaSuccess) return r;
      if ((r = cudaMemset(p->d.sep_A, 0, a_bytes)) != cudaSuccess) return r;
    }
    if ((r = alloc(&p->d.sep_partial, part_bytes)) != cudaSuccess) return r;
    if (!fold) return cudaSuccess;
    if ((r = alloc(&p->d.sep_rec, (size_t)p->n_slots * sizeof(float4))) != cudaSuccess) return r;
    if ((r = put(&p->d.sep_axis_d, dvals)) != cudaSuccess) return r;
    return put(&p->d.sep_axis_dlo, dvals_lo);
  };
  e = make(ff.fold);
  if (e == cudaErrorMemoryAllocation && ff.fold) {  // no room: the direct form may have no table, or a smaller one
    cudaGetLastError();
    for (void* b : {(void*)fd.chunks, (void*)ff.chunks, (void*)p->d.sep_A, (void*)p->d.sep_partial, (void*)p->d.sep_rec,
                    (void*)p->d.sep_axis_d, (void*)p->d.sep_axis_dlo})
      if (b) cudaFree(b);
    ff = SepForm{};
    fd.chunks = nullptr;
    p->d.sep_A = nullptr;
    p->d.sep_partial = p->d.sep_axis_d = p->d.sep_axis_dlo = nullptr;
    p->d.sep_rec = nullptr;
    for (double& m : p->sep_mid) m = 0.0;
    bytes = 0;
    e = make(false);
  }
  if (e != cudaSuccess) return cuda_status(e, "separable tables");
  if ((e = put(&p->d.sep_axis_s, alls)) != cudaSuccess || (e = put(&p->d.sep_axis_lo, alls_lo)) != cudaSuccess)
    return cuda_status(e, "separable axes");
  size_t virt_bytes = 0;
  if (gid) {
    virt_bytes = (size_t)p->sep_ns * sizeof(float2);
    if ((e = cudaMalloc(&p->d.sep_virt, virt_bytes)) != cudaSuccess) return cuda_status(e, "cudaMalloc virtual map");
  }
  if (buried) {
    const size_t tb = att.size() * sizeof(float);
    if ((e = cudaMalloc(&p->d.sep_att, tb)) != cudaSuccess) return cuda_status(e, "attenuation table");
    if ((e = cudaMalloc(&p->d.sep_szf, tb)) != cudaSuccess) return cuda_status(e, "form-factor Sz table");
    cudaMemcpy(p->d.sep_att, att.data(), tb, cudaMemcpyHostToDevice);
    cudaMemcpy(p->d.sep_szf, szf.data(), tb, cudaMemcpyHostToDevice);
    virt_bytes += 2 * tb;
  }
  p->base_bytes += (int64_t)(bytes + virt_bytes);
  if ((e = sep_prepare_kernel()) != cudaSuccess) return cuda_status(e, "separable shared memory attribute");
  st = sep_prepare_side(p, fd.mt);
  return st == SCATTER_OK && ff.fold ? sep_prepare_side(p, ff.mt) : st;
}

scatter_status launch_separable(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st,
                                const CallGate& gate) {
  const double* out_shift = p->out_shift ? p->out_shift : p->d.inst_shift;
  const SepForm& fm = p->sep_folded.fold && amp_out ? p->sep_folded : p->sep_direct;
  SepTabArgs t{};
  t.atom4 = p->d.atom4;
  t.atom_lo = p->d.atom_lo;
  t.atom_w = p->d.atom_w;
  t.axis_s = p->d.sep_axis_s;
  t.axis_lo = p->d.sep_axis_lo;
  t.n0 = p->sep_n[0];
  t.n1 = p->sep_n[1];
  t.n2 = p->sep_n[2];
  t.n_slots = p->n_slots;
  t.n_steps = fm.steps;
  t.n_mt = fm.mt;
  t.A = static_cast<uint4*>(p->d.sep_A);
  t.gate = gate;
  const int n_chunks = fm.n_chunks;
  if (fm.fold && !fm.form_a) {
    const int64_t na = fm.mt * fm.steps * 128;
    const auto kernel = fm.fold_h ? k_sep_tab_fold<true> : k_sep_tab_fold<false>;
    kernel<<<(unsigned)((na + 255) / 256), 256, 0, st>>>(p->d.sep_rec, p->d.sep_axis_d, p->d.sep_axis_dlo, p->sep_n[0],
                                                         fm.lanes, fm.steps, fm.mt, t.A, gate);
    p->last_launches += 1;
  } else if (p->n_slots > 0 && !fm.form_a) {
    const int64_t na = fm.mt * fm.steps * 4 * kSepM;  // real tiles; a padding tile is never read
    k_sep_tab_a<<<(unsigned)((na + 255) / 256), 256, 0, st>>>(t);
    p->last_launches += 1;
  }
  SepArgs a{};
  a.A = static_cast<const uint4*>(p->d.sep_A);
  a.a_sp_stride = 0;
  a.rec = p->d.atom4;
  a.chunks = fm.chunks;
  a.ntiles = nullptr;
  a.bbox = p->d.inst_bbox;
  a.shift = p->d.inst_shift;
  a.smax_b = fm.smax[0];
  a.smax_c = fm.smax[1];
  a.axis_s = fm.fold ? p->d.sep_axis_d : p->d.sep_axis_s;
  a.axis_lo = fm.fold ? p->d.sep_axis_dlo : p->d.sep_axis_lo;
  a.n0 = p->sep_n[0];
  a.n1 = p->sep_n[1];
  a.n2 = p->sep_n[2];
  a.n_cb = (fm.cols + 31) / 32;
  a.chunk_floats = sep_part_floats(fm.mt, fm.cols);
  a.fold = fm.fold ? 1 : 0;
  a.n_pairs = fm.pairs;
  a.n_lanes = fm.lanes;
  a.fold_h = fm.fold_h ? 1 : 0;
  a.flush = fm.flush;
  a.rec_a = p->d.sep_rec;
  a.n_steps = fm.steps;
  a.n_mt = fm.mt;
  a.partial = p->d.sep_partial;
  a.status = p->d.status;
  a.axis_att = p->d.sep_att;
  a.form_a = fm.form_a ? 1 : 0;
  a.rec_lo = p->d.atom_lo;
  a.rec_w = p->d.atom_w;
  a.gate = gate;
  dim3 grid((unsigned)(((fm.mt + 1) / 2) * fm.nt), (unsigned)n_chunks);
  if (!gate.rmax2) timing_begin(p, st);
  const cudaError_t le = sep_launch_core(a, grid, st, p->side_stream, p->side_fork, p->side_join);
  timing_end(p, st);
  if (le != cudaSuccess) return cuda_status(le, "separable kernel launch");
  p->last_launches += sep_core_launches(fm.mt);
  const bool gid = p->s_kind == SCATTER_S_GID_GRID;
  const int64_t n_cb = a.n_cb, ncols = p->sep_n[1] * p->sep_n[2];
  // row blocks of the reduction: 16 h values (32 partial rows); folded 8 lanes, 32 per
  // M tile: the h values of a tile's second half (or their mirrors) with those of its first
  const int64_t n_bm = !fm.fold ? (2 * p->sep_n[0] + 31) / 32
                       : fm.fold_h ? (fm.lanes + 7) / 8 : 4 * fm.mt;
  // a host call copies each row range to the host while the next is reduced
  const bool pieces = p->host_out && !gid;
  // (folded: four; 2 to 16 ranges measured the same 3.59 ms on the strained
  // sphere, and fewer leave each reduction more CTAs)
  const int max_pieces = (int)std::min<int64_t>(fm.fold ? 4 : kHostPieces, n_bm);
  const int n_pieces = pieces ? max_pieces : 1;
  float2* amp_dst = gid ? p->d.sep_virt : amp_out;
  float* int_dst = gid ? nullptr : int_out;
  for (int k = 0; k < n_pieces; ++k) {
    const int64_t b0 = n_bm * k / n_pieces, b1 = n_bm * (k + 1) / n_pieces;
    if (fm.fold) {
      SepFoldReduceArgs r{};
      r.partial = p->d.sep_partial;
      r.chunk_floats = a.chunk_floats;
      r.n_cb = n_cb;
      r.chunks = fm.chunks;
      r.n_chunks = n_chunks;
      r.coef = p->d.coef;
      r.ftab = p->d.ftab;
      r.inv4a2 = (float)(1.0 / (4.0 * p->lattice_a * p->lattice_a));
      r.axis_s = p->d.sep_axis_s;
      r.axis_lo = p->d.sep_axis_lo;
      r.n0 = p->sep_n[0];
      r.n1 = p->sep_n[1];
      r.n2 = p->sep_n[2];
      r.n_pairs = fm.pairs;
      r.n_lanes = fm.lanes;
      r.fold_h = fm.fold_h ? 1 : 0;
      for (int d = 0; d < 3; ++d) r.H[d] = (float)p->inst[0].H[d];
      r.shift = out_shift;
      r.gate = gate;
      r.l8_base = b0;
      r.out_amp = amp_dst;
      r.out_int = int_dst;
      // small maps: several threads share each quadruple's chunks until a row
      // range's launch has a CTA per SM (the same choice with and without
      // ranges: a host call's map equals the device call's bit for bit)
      const int64_t quads = (fm.pairs + 3) / 4, range = (n_bm + max_pieces - 1) / max_pieces;
      int groups = 1;
      while (groups < 32 && 2 * groups <= n_chunks && (quads + 31) / 32 * range * groups < p->n_sm) groups *= 2;
      const auto kernel = groups == 1    ? k_sep_reduce_fold<1>
                          : groups == 2  ? k_sep_reduce_fold<2>
                          : groups == 4  ? k_sep_reduce_fold<4>
                          : groups == 8  ? k_sep_reduce_fold<8>
                          : groups == 16 ? k_sep_reduce_fold<16>
                                         : k_sep_reduce_fold<32>;
      const int64_t per_cta = 32 / groups;  // quads per CTA
      kernel<<<dim3((unsigned)((quads + per_cta - 1) / per_cta), (unsigned)(b1 - b0)), 256, 0, st>>>(r);
    } else {
      const dim3 rgrid((unsigned)n_cb, (unsigned)(b1 - b0));
      k_sep_reduce<<<rgrid, 256, 0, st>>>(
          p->d.sep_partial, a.chunk_floats, n_cb, fm.chunks, n_chunks, p->d.coef, p->d.ftab,
          (float)(1.0 / (4.0 * p->lattice_a * p->lattice_a)), p->d.sep_axis_s, p->d.sep_axis_lo, p->sep_n[0],
          p->sep_n[1], p->sep_n[2],
          make_float3((float)p->inst[0].H[0], (float)p->inst[0].H[1], (float)p->inst[0].H[2]), out_shift,
          p->d.sep_att, p->d.sep_szf, b0, amp_dst, int_dst, gate);
    }
    p->last_launches += 1;
    if (pieces) {
      const int64_t n0 = p->sep_n[0];
      cudaError_t e = cudaEventRecord(p->copy_ev[k], st);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(p->copy_stream, p->copy_ev[k], 0);
      auto copy_rows = [&](int64_t r0, int64_t r1) {
        r1 = std::min(r1, n0);
        if (e == cudaSuccess && r1 > r0)
          e = cudaMemcpyAsync(static_cast<float2*>(p->host_out) + r0 * ncols, amp_out + r0 * ncols,
                              (size_t)((r1 - r0) * ncols) * sizeof(float2), cudaMemcpyDeviceToHost, p->copy_stream);
      };
      if (!fm.fold) {
        copy_rows(16 * b0, 16 * b1);
      } else if (fm.fold_h) {
        // h rows 8 b0 .. 8 b1 of the axis' first half and their mirror rows
        const int64_t i0 = std::min(8 * b0, fm.lanes), i1 = std::min(8 * b1, fm.lanes);
        copy_rows(i0, i1);
        copy_rows(std::max(i1, n0 - i1), n0 - i0);
      } else {
        // per block of 8 lanes, the rows of the tile's first and second 32 h values
        for (int64_t b = b0; b < b1; ++b)
          for (int w = 0; w < 2; ++w) copy_rows(64 * (b / 4) + 32 * w + 8 * (b % 4), 64 * (b / 4) + 32 * w + 8 * (b % 4) + 8);
      }
      if (e != cudaSuccess) return cuda_status(e, "map range to the host");
    }
  }
  if (pieces) {
    // the caller's stream resumes once the last range is on the host
    cudaError_t e = cudaEventRecord(p->copy_ev[kHostPieces], p->copy_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, p->copy_ev[kHostPieces], 0);
    if (e != cudaSuccess) return cuda_status(e, "host copy completion");
  }
  if (gid) {
    scatter_status s2 = launch_gid_combine(p, amp_out, int_out, st, gate);
    if (s2 != SCATTER_OK) return s2;
  }
  return cuda_status(cudaGetLastError(), "separable launch");
}

}  // namespace scatter
