// Generic forward path of the direct scattering sum (Eq. 2) on sm_103a.
//
//   prep     per call: integer centring t of each instance (rint of the
//            bounding-box centre of its atoms), split r - t = n + delta with
//            n = rint(r - t), and the per-atom phase c = frac(H . delta) in
//            FP64, stored as fp32 slots (x', y', z', c) with x' = r - t.
//            Because H . n is an integer, for S = H + s
//              S . r = S . t + H . delta + s . (r - t)  (mod 1)
//            so only the small quantities c and s . x' reach FP32.
//   generic  CTA = a tile of S points, THREADS x R points in registers; atom
//            tiles (20 B/atom) staged in shared memory by the TMA engine
//            (cp.async.bulk, double buffered on mbarriers, bounded waits).
//            Per pair: phase = c + s . x' (FFMA), reduction mod 1 (FADD),
//            sin/cos of 2 pi phase on MUFU, two FFMA into tile-blocked FP32
//            accumulators.  Species segments fold f_s(|S|) in-kernel
//            (Section 4.2: f factors out of the sum over atoms of a species).
//   reduce   split-K partials summed in a fixed order (deterministic), then
//            the translation phase e^{2 pi i s.t} and |A|^2 if requested.
#include <cuda_runtime.h>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include "device_common.cuh"
#include "generic_impl.cuh"
#include "launch.h"

namespace scatter {


// ---------------------------------------------------------------------------
// prep
// ---------------------------------------------------------------------------

using dev::ordered;
using dev::unordered;

__global__ void k_bbox_init(unsigned long long* bbox, int batch, unsigned* rmax2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (rmax2 && i < batch) rmax2[i] = 0u;
  if (i < batch * 6) bbox[i] = (i % 6) < 3 ? ~0ULL : 0ULL;  // min slots: max value; max slots: 0
}

// Bounding box as ordered integers: min xyz, max xyz.  GB300 issues FP64 (its
// comparisons too) at ~2 operations per SM and clock, so the coordinates are
// compared as order-preserving 64-bit integers and tested for Inf / NaN by
// their exponent bits.
struct Box {
  unsigned long long v[6] = {~0ULL, ~0ULL, ~0ULL, 0ULL, 0ULL, 0ULL};
  __device__ __forceinline__ void add(const double* p, bool& bad) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double x = p[d];
      if ((__double2hiint(x) & 0x7ff00000) == 0x7ff00000) {
        bad = true;
        continue;
      }
      const unsigned long long u = ordered(x);
      v[d] = min(v[d], u);
      v[3 + d] = max(v[3 + d], u);
    }
  }
  __device__ __forceinline__ void join(const unsigned long long* o) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      v[d] = min(v[d], o[d]);
      v[3 + d] = max(v[3 + d], o[3 + d]);
    }
  }
  // the block's box in thread d < 6 (value d), 256 threads
  __device__ __forceinline__ unsigned long long reduce(unsigned long long (*sh)[8]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 0; d < 6; ++d) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long q = __shfl_xor_sync(0xffffffffu, v[d], o);
        v[d] = d < 3 ? min(v[d], q) : max(v[d], q);
      }
      if (lane == 0) sh[d][warp] = v[d];
    }
    __syncthreads();
    unsigned long long r = 0;
    if (threadIdx.x < 6) {
      r = sh[threadIdx.x][0];
#pragma unroll
      for (int w = 1; w < 8; ++w) r = threadIdx.x < 3 ? min(r, sh[threadIdx.x][w]) : max(r, sh[threadIdx.x][w]);
    }
    return r;
  }
};

// One grid row per instance; each CTA reduces a strided share of the
// instance's atoms and merges with order-independent atomic min/max.
__global__ void __launch_bounds__(256) k_bbox(const double* __restrict__ xyz, const int64_t* __restrict__ atom_off,
                                              unsigned long long* bbox, unsigned* status) {
  __shared__ unsigned long long sh[6][8];
  const int inst = blockIdx.y;
  const int64_t b = atom_off[inst], e = atom_off[inst + 1];
  Box box;
  bool bad = false;
  for (int64_t j = b + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < e; j += (int64_t)gridDim.x * blockDim.x)
    box.add(xyz + 3 * j, bad);
  if (bad) dev::set_status(status, kStatusNonFinite);
  const unsigned long long r = box.reduce(sh);
  if (threadIdx.x < 3 && r != ~0ULL) atomicMin(&bbox[6 * inst + threadIdx.x], r);
  if (threadIdx.x >= 3 && threadIdx.x < 6 && r != 0ULL) atomicMax(&bbox[6 * inst + threadIdx.x], r);
}

// One instance: the box of each CTA's share of the atoms, joined by k_prep_one.
__global__ void __launch_bounds__(256) k_box_part(const double* __restrict__ xyz, int64_t n_atoms,
                                                  unsigned long long* __restrict__ part, unsigned* status,
                                                  unsigned* rmax2, const CallGate gate) {
  __shared__ unsigned long long sh[6][8];
  if (within(gate, 0)) return;
  if (rmax2 && blockIdx.x == 0 && threadIdx.x == 0) *rmax2 = 0u;
  Box box;
  bool bad = false;
#pragma unroll 4
  for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < n_atoms; j += (int64_t)gridDim.x * 256)
    box.add(xyz + 3 * j, bad);
  if (bad) dev::set_status(status, kStatusNonFinite);
  const unsigned long long r = box.reduce(sh);
  if (threadIdx.x < 6) part[6 * (int64_t)blockIdx.x + threadIdx.x] = r;
}

struct PrepArgs {
  const double* xyz;
  const float* occ;
  const int32_t* slot_src;
  const double* inst_H;   // [batch][3]
  float4* atom4;
  float4* atom_lo;
  float* atom_w;
  unsigned* status;
  float4* rec_a;          // the folded separable forward's A records, or null
  float mid[3], mid_lo[3];  // middles of its axes - H
  unsigned* rmax2;        // [batch] largest |x'|^2 (float bits, zeroed before), or null
  int per_axis;           // rmax2 of the largest |x'_d| of this many axes instead
  double* z_shift;        // [3] third element: t_z, or null
  int wide;               // |S| past kPrepFixedS: the split in FP64 throughout
  CallGate gate;          // one instance
};

// Positions in 2^-42 fixed point err by up to 2^-43 cells, a phase by |S| times as
// much: 2^-31 cycles at |S| = 2^12, a 64th of the rounding of c itself.  Longer S go
// with coordinates that are small numbers (crystals in metres: S of 1e10, positions of
// 1e-8, of which fixed point keeps four digits) and take FP64.
constexpr double kPrepFixedS = 4096.0;

// a + b with its rounding error
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

// One coordinate: r = x - t as a double-float x0 + lo and its distance
// delta = r - rint(r) as dh + dl.  Below 2^19 cells in 64-bit fixed point
// (2^-42 cells: what FP64 holds at 2^10 cells, four decades below what the
// double-float keeps of a centred position), with integer and FP32
// operations only; beyond, in FP64.
__device__ __forceinline__ void prep_coord(double x, double t, float& x0, float& lo, float& dh, float& dl) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  if (e < 1023 + 19 && fabsf((float)t) < 524288.0f) {
    const unsigned long long m =
        ((unsigned long long)__double_as_longlong(x) & 0xfffffffffffffULL) | (e ? 0x10000000000000ULL : 0ULL);
    const int sh = e - (1075 - 42);  // x = m 2^(e - 1075)
    unsigned long long mag = 0ULL;
    if (sh >= 0)
      mag = m << sh;
    else if (sh > -64)
      mag = ((m >> (-sh - 1)) + 1ULL) >> 1;
    const long long r = (hi < 0 ? -(long long)mag : (long long)mag) - ((long long)(int)t << 42);
    const int n = (int)((r + (1LL << 41)) >> 42);
    const long long d = r - ((long long)n << 42);  // [-2^41, 2^41)
    // 24 bits of 2^-24 and 18 of 2^-42, joined to the nearest float and the rest: a
    // small coordinate keeps its digits
    dh = two_sum((float)(int)(d >> 18) * 5.9604644775390625e-08f, (float)(int)(d & 0x3ffffLL) * 2.2737367544323206e-13f, dl);
    float err;
    x0 = two_sum((float)n, dh, err);
    lo = err + dl;
  } else {
    const double r = x - t, d = r - rint(r);
    x0 = (float)r;
    lo = (float)(r - (double)x0);
    dh = (float)d;
    dl = (float)(d - (double)dh);
  }
}

// The slot's records from its atom centred on t: (x', y', z', c), rounding
// errors, occupancy; c = frac(H . delta) from exact products and TwoSums, one
// rounding at the end as in FP64.
// H: the instance's reflection, h the same in FP32.  Returns |x'|^2.
__device__ __forceinline__ float prep_slot(const PrepArgs& a, int64_t slot, const double (&t)[3], const double* H,
                                          const float (&h)[3]) {
  const int32_t src = a.slot_src[slot];
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  bool ok = src >= 0;
  double x[3] = {0.0, 0.0, 0.0};
  float w = 0.f;
  if (ok) {
    const double* p = a.xyz + 3 * (int64_t)src;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      x[d] = p[d];
      ok = ok && (__double2hiint(x[d]) & 0x7ff00000) != 0x7ff00000;
    }
    w = a.occ ? a.occ[src] : 1.0f;
    ok = ok && isfinite(w);
    if (!ok) dev::set_status(a.status, kStatusNonFinite);
  }
  if (!ok) {
    a.atom4[slot] = zero;
    a.atom_lo[slot] = zero;
    a.atom_w[slot] = 0.f;
    if (a.rec_a) a.rec_a[slot] = zero;
    return 0.f;
  }
  float x0[3], lo[3], cr, ce = 0.f, err;
  if (a.wide) {
    double c = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double r = x[d] - t[d];
      x0[d] = (float)r;
      lo[d] = (float)(r - (double)x0[d]);
      c = fma(H[d], r - rint(r), c);
    }
    c -= rint(c);
    cr = (float)c;
    ce = (float)(c - (double)cr);
  } else {
    float c = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float dh, dl;
      prep_coord(x[d], t[d], x0[d], lo[d], dh, dl);
      const float pr = __fmul_rn(h[d], dh);
      c = two_sum(c, __fsub_rn(pr, rintf(pr)), err);
      ce += err + (fmaf(h[d], dh, -pr) + h[d] * dl);
    }
    cr = c - rintf(c);  // exact
  }
  const float c = cr + ce;
  a.atom4[slot] = make_float4(x0[0], x0[1], x0[2], c);
  a.atom_lo[slot] = make_float4(lo[0], lo[1], lo[2], 0.f);
  a.atom_w[slot] = w;
  if (a.rec_a) {
    // the folded forward's A record: x' as a double-float and W = w e^{2 pi i (c + (mid - H).x')}
    float ph = cr, pe = ce;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float pr = __fmul_rn(a.mid[d], x0[d]);
      ph = two_sum(ph, pr - rintf(pr), err);
      pe += err + (fmaf(a.mid[d], x0[d], -pr) + fmaf(a.mid_lo[d], x0[d], a.mid[d] * lo[d]));
    }
    float sn, cs;
    sincospif(2.0f * ((ph - rintf(ph)) + pe), &sn, &cs);
    a.rec_a[slot] = make_float4(x0[0], lo[0], w * cs, w * sn);
  }
  const float q[3] = {x0[0] * x0[0], x0[1] * x0[1], x0[2] * x0[2]};
  // a NaN stays one: its bits are the largest
  if (a.per_axis)
    return __uint_as_float(max(max(__float_as_uint(q[0]), __float_as_uint(q[1])), a.per_axis > 2 ? __float_as_uint(q[2]) : 0u));
  return q[0] + q[1] + q[2];
}

__device__ __forceinline__ double centre(unsigned long long ulo, unsigned long long uhi) {
  return (ulo == ~0ULL || uhi == 0ULL) ? 0.0 : rint(0.5 * (unordered(ulo) + unordered(uhi)));
}

// Batches: one thread per slot, each instance's box in `bbox`.
__global__ void __launch_bounds__(256) k_prep(const PrepArgs a, const int32_t* __restrict__ slot_inst,
                                              const int64_t* __restrict__ inst_slot_begin,
                                              const unsigned long long* __restrict__ bbox, double* inst_shift,
                                              int64_t n_slots) {
  const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (slot >= n_slots) return;
  const int inst = slot_inst[slot];
  double t[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) t[d] = centre(bbox[6 * inst + d], bbox[6 * inst + 3 + d]);
  if (slot == inst_slot_begin[inst]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) inst_shift[3 * inst + d] = t[d];
  }
  const double* H = a.inst_H + 3 * inst;
  const float h[3] = {(float)H[0], (float)H[1], (float)H[2]};
  const unsigned r2 = __float_as_uint(prep_slot(a, slot, t, H, h));
  if (a.rmax2) {  // n_slots is a multiple of 32: whole warps are here
    if (__all_sync(0xffffffffu, inst == __shfl_sync(0xffffffffu, inst, 0))) {
      const unsigned m = __reduce_max_sync(0xffffffffu, r2);
      if ((threadIdx.x & 31) == 0) atomicMax(&a.rmax2[inst], m);
    } else {
      atomicMax(&a.rmax2[inst], r2);
    }
  }
}

// One instance, one launch after the boxes: every CTA joins the n_part partial
// boxes (n_part = 0: takes the box of all the atoms itself, for small
// crystals), then prepares its share of the slots.  1e6 atoms: 9.6 us for
// the boxes and ~20 us here, from 63 + 76 us and an initialising launch when
// the comparisons and the split ran in FP64; 4 CTAs per SM, each joining 256
// boxes, measured 5 us less than 8 joining 512.
__global__ void __launch_bounds__(256) k_prep_one(const PrepArgs a, int64_t n_atoms, int64_t n_slots,
                                                  const unsigned long long* __restrict__ part, int n_part,
                                                  unsigned long long* bbox, double* inst_shift) {
  if (within(a.gate, 0)) return;
  __shared__ unsigned long long sh[6][8];
  __shared__ unsigned long long sh_box[6];
  __shared__ double sh_t[3];
  __shared__ float sh_h[3];
  Box box;
  if (n_part > 0) {
    for (int i = threadIdx.x; i < n_part; i += 256) box.join(part + 6 * (int64_t)i);
  } else {
    bool bad = false;
#pragma unroll 4
    for (int64_t j = threadIdx.x; j < n_atoms; j += 256) box.add(a.xyz + 3 * j, bad);
    if (bad && blockIdx.x == 0) dev::set_status(a.status, kStatusNonFinite);
  }
  const unsigned long long r = box.reduce(sh);
  if (threadIdx.x < 6) {
    sh_box[threadIdx.x] = r;
    if (blockIdx.x == 0) bbox[threadIdx.x] = r;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    const double t = centre(sh_box[threadIdx.x], sh_box[3 + threadIdx.x]);
    sh_t[threadIdx.x] = t;
    sh_h[threadIdx.x] = (float)a.inst_H[threadIdx.x];
    if (blockIdx.x == 0) inst_shift[threadIdx.x] = t;
    if (blockIdx.x == 0 && threadIdx.x == 2 && a.z_shift) a.z_shift[2] = t;
  }
  __syncthreads();
  const double t[3] = {sh_t[0], sh_t[1], sh_t[2]};
  const float h[3] = {sh_h[0], sh_h[1], sh_h[2]};
  unsigned r2 = 0u;  // |x'|^2 >= 0 orders as its bits
  for (int64_t slot = (int64_t)blockIdx.x * 256 + threadIdx.x; slot < n_slots; slot += (int64_t)gridDim.x * 256)
    r2 = max(r2, __float_as_uint(prep_slot(a, slot, t, a.inst_H, h)));
  if (a.rmax2) {
    r2 = __reduce_max_sync(0xffffffffu, r2);
    if ((threadIdx.x & 31) == 0) atomicMax(a.rmax2, r2);
  }
}

// ---------------------------------------------------------------------------
// generic kernel
// ---------------------------------------------------------------------------

template <int MODE, int R, int THREADS>
__global__ void __launch_bounds__(THREADS) k_generic(const GenericArgs a) {
  __shared__ __align__(128) float4 sh_atom[2][kTile];
  __shared__ __align__(128) float4 sh_lo[2][kTile];  // position rounding errors (exact-product phases)
  __shared__ __align__(128) float sh_w[2][kTile];
  __shared__ __align__(8) uint64_t sh_bar[2];

  if (within(a.gate, 0)) return;
  const int tid = threadIdx.x;
  const int chunk = blockIdx.y;

  // ---- S points of this thread -------------------------------------------
  float sx[R], sy[R], sz[R];
  int64_t idx0 = 0;      // GRID: output index of point 0; LIST: tile base
  int nvalid = 0;        // GRID: number of valid points (prefix)
  bool valid[R];
  if (MODE == kModeGrid) {
    const int64_t q = (a.n2 + R - 1) / R;
    const int64_t g = (int64_t)blockIdx.x * THREADS + tid;
    const bool active = g < a.n0 * a.n1 * q;
    const int64_t line = active ? g / q : 0, blk = active ? g % q : 0;
    const int64_t i0 = line / a.n1, i1 = line % a.n1, i2 = blk * R;
    const float x = a.axis_s[i0], y = a.axis_s[a.n0 + i1];
    nvalid = active ? (int)dev::min64(R, a.n2 - i2) : 0;
    idx0 = line * a.n2 + i2;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      sx[r] = x;
      sy[r] = y;
      sz[r] = a.axis_s[a.n0 + a.n1 + dev::min64(i2 + r, a.n2 - 1)];
      valid[r] = r < nvalid;
    }
  } else {
    idx0 = (int64_t)blockIdx.x * THREADS * R;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t m = idx0 + (int64_t)r * THREADS + tid;
      valid[r] = m < a.n_s;
      const int64_t mm = valid[r] ? m : 0;
      sx[r] = a.s_hi[mm];
      sy[r] = a.s_hi[a.n_s + mm];
      sz[r] = a.s_hi[2 * a.n_s + mm];
    }
  }

  if (tid == 0) {
    dev::mbar_init(&sh_bar[0], 1);
    dev::mbar_init(&sh_bar[1], 1);
    dev::mbar_fence_init();
  }
  __syncthreads();
  // output index of point r: pbase + r pstride (for a factor table)
  const int64_t pbase = MODE == kModeGrid ? idx0 : idx0 + tid;
  const int64_t pstride = MODE == kModeGrid ? 1 : THREADS;
  float2 tot[R];
  int k = 0;
  // one decision per call (every CTA computes the same): phases that can
  // pass kPhaseExactLim cycles take the exact-product route, with s as a
  // double-float
  bool ok;
  if (dev::phase_needs_exact(a.bbox, a.shift, a.smax_dev ? a.smax_dev : a.smax)) {
    int64_t i0 = 0, i1 = 0, i2 = 0;
    if (MODE == kModeGrid) {
      const int64_t q = (a.n2 + R - 1) / R;
      const int64_t g = (int64_t)blockIdx.x * THREADS + tid;
      const int64_t line = g < a.n0 * a.n1 * q ? g / q : 0;
      i0 = line / a.n1;
      i1 = line % a.n1;
      i2 = idx0 - line * a.n2;
    }
    auto lo = [&](int r, float& x, float& y, float& z) {
      if (MODE == kModeGrid) {
        x = a.axis_lo[i0];
        y = a.axis_lo[a.n0 + i1];
        z = a.axis_lo[a.n0 + a.n1 + dev::min64(i2 + r, a.n2 - 1)];
      } else {
        const int64_t m = valid[r] ? idx0 + (int64_t)r * THREADS + tid : 0;
        x = a.s_lo[m];
        y = a.s_lo[a.n_s + m];
        z = a.s_lo[2 * a.n_s + m];
      }
    };
    ok = chunk_sum_exact_halves<MODE, R>(a.atom4, a.atom_lo, a.atom_w, a.segs, a.chunk_seg_off[chunk],
                                         a.chunk_seg_off[chunk + 1], a.coef, a.H, a.inv4a2, sx, sy, sz, lo, sh_atom,
                                         sh_lo, sh_w, sh_bar, k, tot, a.status, a.ftab, a.n_s, pbase, pstride);
  } else {
    ok = chunk_sum<MODE, R, false>(a.atom4, a.atom_lo, a.atom_w, a.segs, a.chunk_seg_off[chunk],
                                   a.chunk_seg_off[chunk + 1], a.coef, a.H, a.inv4a2, sx, sy, sz, sx, sy, sz, sh_atom,
                                   sh_lo, sh_w, sh_bar, k, tot, a.status, a.ftab, a.n_s, pbase, pstride);
  }
  if (!ok) return;

  // ---- epilogue -----------------------------------------------------------------
  if (a.partial) {
    float2* out = a.partial + (int64_t)chunk * a.n_s;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!valid[r]) continue;
      const int64_t m = MODE == kModeGrid ? idx0 + r : idx0 + (int64_t)r * THREADS + tid;
      out[m] = tot[r];
    }
    return;
  }
  const double* t = a.shift;
  const bool shifted = t[0] != 0.0 || t[1] != 0.0 || t[2] != 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (!valid[r]) continue;
    int64_t m;
    float2 v = tot[r];
    if (MODE == kModeGrid) {
      m = idx0 + r;
      if (shifted) {
        const int64_t i2 = m % a.n2, line = m / a.n2, i1 = line % a.n1, i0 = line / a.n1;
        v = dev::cmul(dev::shift_phase(a.axis64[i0] - a.H64[0], a.axis64[a.n0 + i1] - a.H64[1],
                                       a.axis64[a.n0 + a.n1 + i2] - a.H64[2], t),
                      v);
      }
    } else {
      m = idx0 + (int64_t)r * THREADS + tid;
      if (shifted)
        v = dev::cmul(dev::shift_phase(a.S64[3 * m] - a.H64[0], a.S64[3 * m + 1] - a.H64[1],
                                       a.S64[3 * m + 2] - a.H64[2], t),
                      v);
    }
    if (a.out_amp) a.out_amp[m] = v;
    if (a.out_int) a.out_int[m] = v.x * v.x + v.y * v.y;
  }
}

// Sum of split-K partials, translation phase, outputs.  GROUPS threads per
// point, each over a contiguous share of the chunks in order, joined in order:
// a short list with many chunks (atom-parallel blocks) fills the SMs and keeps
// eight loads in flight per thread (1000 points x 245 blocks: 38 us with one
// thread per point, 10.5 us with eight).
template <int GROUPS>
__global__ void __launch_bounds__(256) k_reduce(GenericArgs a, int split_k, int grid_mode) {
  constexpr int kPts = 256 / GROUPS;
  __shared__ float2 sh[GROUPS > 1 ? GROUPS - 1 : 1][kPts];
  if (within(a.gate, 0)) return;
  const int pt = threadIdx.x % kPts, grp = threadIdx.x / kPts;
  const int64_t m = (int64_t)blockIdx.x * kPts + pt;
  float2 v = make_float2(0.f, 0.f);
  if (m < a.n_s) {
    const int per = (split_k + GROUPS - 1) / GROUPS, c1 = min(split_k, (grp + 1) * per);
#pragma unroll 8
    for (int c = grp * per; c < c1; ++c) {
      const float2 p = a.partial[(int64_t)c * a.n_s + m];
      v.x += p.x;
      v.y += p.y;
    }
  }
  if constexpr (GROUPS > 1) {
    if (grp > 0) sh[grp - 1][pt] = v;
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int g = 0; g < GROUPS - 1; ++g) {
      v.x += sh[g][pt].x;
      v.y += sh[g][pt].y;
    }
  }
  if (m >= a.n_s) return;
  const double* t = a.shift;
  if (t[0] != 0.0 || t[1] != 0.0 || t[2] != 0.0) {
    if (grid_mode) {
      const int64_t i2 = m % a.n2, line = m / a.n2, i1 = line % a.n1, i0 = line / a.n1;
      v = dev::cmul(dev::shift_phase(a.axis64[i0] - a.H64[0], a.axis64[a.n0 + i1] - a.H64[1],
                                     a.axis64[a.n0 + a.n1 + i2] - a.H64[2], t),
                    v);
    } else {
      v = dev::cmul(dev::shift_phase(a.S64[3 * m] - a.H64[0], a.S64[3 * m + 1] - a.H64[1],
                                     a.S64[3 * m + 2] - a.H64[2], t),
                    v);
    }
  }
  if (a.out_amp) a.out_amp[m] = v;
  if (a.out_int) a.out_int[m] = v.x * v.x + v.y * v.y;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

namespace {

template <int MODE, int R, int THREADS>
void* generic_fn() {
  return (void*)&k_generic<MODE, R, THREADS>;
}

void* pick_generic(int mode, int R, int threads) {
#define SCATTER_CASE(M, RR, TT) \
  if (mode == M && R == RR && threads == TT) return generic_fn<M, RR, TT>();
  SCATTER_CASE(kModeList, 4, 128) SCATTER_CASE(kModeList, 4, 256)
  SCATTER_CASE(kModeList, 8, 128) SCATTER_CASE(kModeList, 8, 256)
  SCATTER_CASE(kModeList, 16, 128) SCATTER_CASE(kModeList, 16, 256)
  SCATTER_CASE(kModeGrid, 4, 128) SCATTER_CASE(kModeGrid, 4, 256)
  SCATTER_CASE(kModeGrid, 8, 128) SCATTER_CASE(kModeGrid, 8, 256)
  SCATTER_CASE(kModeGrid, 16, 128) SCATTER_CASE(kModeGrid, 16, 256)
#undef SCATTER_CASE
  return nullptr;
}

int mode_of(const scatter_plan_s* p) { return p->s_kind == SCATTER_S_GRID ? kModeGrid : kModeList; }

GenericArgs make_args(scatter_plan_t p) {
  GenericArgs a{};
  a.atom4 = p->d.atom4;
  a.atom_lo = p->d.atom_lo;
  a.atom_w = p->d.atom_w;
  a.segs = p->d.segs;
  a.chunk_seg_off = p->d.chunk_seg_off;
  a.coef = p->d.coef;
  a.n_s = p->n_s;
  a.s_hi = p->d.s_hi;
  a.s_lo = p->d.s_lo;
  a.S64 = p->d.S64;
  a.axis_s = p->d.axis_s;
  a.axis_lo = p->d.axis_lo;
  a.axis64 = p->d.axis64;
  a.n0 = p->n_axis[0];
  a.n1 = p->n_axis[1];
  a.n2 = p->n_axis[2];
  for (int d = 0; d < 3; ++d) {
    a.H[d] = (float)p->inst[0].H[d];
    a.H64[d] = p->inst[0].H[d];
  }
  a.inv4a2 = (float)(1.0 / (4.0 * p->lattice_a * p->lattice_a));
  a.shift = p->d.inst_shift;
  a.bbox = p->d.inst_bbox;
  for (int d = 0; d < 3; ++d) a.smax[d] = (float)p->s_max[d];
  a.ftab = p->d.ftab;
  a.status = p->d.status;
  a.gate = cluster_gate(p);
  return a;
}

}  // namespace

namespace {

void launch_reduce(const GenericArgs& a, int n_chunks, int grid_mode, cudaStream_t st) {
  if (n_chunks >= 16 && a.n_s <= 65536)
    k_reduce<8><<<(unsigned)((a.n_s + 31) / 32), 256, 0, st>>>(a, n_chunks, grid_mode);
  else
    k_reduce<1><<<(unsigned)((a.n_s + 255) / 256), 256, 0, st>>>(a, n_chunks, grid_mode);
}

}  // namespace

bool generic_tiling_supported(const Tiling& t) {
  return pick_generic(kModeList, t.R, t.threads) != nullptr && t.split_k >= 1;
}

int64_t generic_num_tiles(const scatter_plan_s* p, const Tiling& t) {
  if (mode_of(p) == kModeGrid) {
    const int64_t q = (p->n_axis[2] + t.R - 1) / t.R;
    return (p->n_axis[0] * p->n_axis[1] * q + t.threads - 1) / t.threads;
  }
  const int64_t per = (int64_t)t.threads * t.R;
  return (p->n_s + per - 1) / per;
}

int generic_blocks_per_sm(const scatter_plan_s* p, const Tiling& t) {
  void* fn = pick_generic(mode_of(p), t.R, t.threads);
  if (!fn) return 0;
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, t.threads, 0) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return nb > 0 ? nb : 1;
}

scatter_status launch_prep(scatter_plan_t p, const double* xyz, const float* occ, cudaStream_t st,
                           const CallGate& gate) {
  const int batch = p->batch;
  PrepArgs a{};
  a.xyz = xyz;
  a.occ = occ;
  a.slot_src = p->d.slot_src;
  a.inst_H = p->d.inst_H;
  a.atom4 = p->d.atom4;
  a.atom_lo = p->d.atom_lo;
  a.atom_w = p->d.atom_w;
  a.status = p->d.status;
  a.rec_a = p->d.sep_rec;
  a.rmax2 = p->cl.active ? p->cl.rmax2 : p->extent2;
  const bool gid = p->s_kind == SCATTER_S_GID_GRID;
  a.per_axis = p->extent2 ? (gid ? 2 : 3) : 0;
  a.z_shift = gid ? p->out_shift : nullptr;
  for (const Instance& in : p->inst)
    for (int d = 0; d < 3; ++d) a.wide |= std::fabs(in.H[d]) + p->s_max[d] > kPrepFixedS;
  a.gate = gate;
  for (int d = 0; d < 3; ++d) {
    a.mid[d] = (float)p->sep_mid[d];
    a.mid_lo[d] = (float)(p->sep_mid[d] - (double)a.mid[d]);
  }
  if (batch == 1) {
    // up to kPrepSmall atoms every CTA takes the box of all of them itself: one launch
    int n_part = 0;
    if (p->n_atoms > kPrepSmall || a.rmax2) {
      n_part = (int)std::min<int64_t>(kPrepParts, (p->n_atoms + 511) / 512);
      k_box_part<<<n_part, 256, 0, st>>>(xyz, p->n_atoms, p->d.box_part, p->d.status, a.rmax2, gate);
      p->last_launches += 1;
    }
    const int64_t nb = std::min<int64_t>(std::max<int64_t>((p->n_slots + 255) / 256, 1), 4 * (int64_t)p->n_sm);
    k_prep_one<<<(unsigned)nb, 256, 0, st>>>(a, p->n_atoms, p->n_slots, p->d.box_part, n_part, p->d.inst_bbox,
                                             p->d.inst_shift);
    p->last_launches += 1;
    return cuda_status(cudaGetLastError(), "prep launch");
  }
  k_bbox_init<<<(batch * 6 + 255) / 256, 256, 0, st>>>(p->d.inst_bbox, batch, a.rmax2);
  p->last_launches += 2;
  int64_t max_atoms = 0;
  for (const auto& in : p->inst) max_atoms = std::max<int64_t>(max_atoms, in.atom_end - in.atom_begin);
  const int bx = (int)dev::min64(std::max<int64_t>((max_atoms + 1023) / 1024, 1), 64);
  k_bbox<<<dim3(bx, batch), 256, 0, st>>>(xyz, p->d.atom_off, p->d.inst_bbox, p->d.status);
  if (p->n_slots > 0) {
    const int64_t nb = (p->n_slots + 255) / 256;
    k_prep<<<(unsigned)nb, 256, 0, st>>>(a, p->d.slot_inst, p->d.inst_slot_begin, p->d.inst_bbox, p->d.inst_shift,
                                         p->n_slots);
    p->last_launches += 1;
  }
  return cuda_status(cudaGetLastError(), "prep launch");
}

scatter_status launch_bbox_raw(const double* xyz, const int64_t* atom_off, int batch, int64_t max_atoms,
                               unsigned long long* bbox, unsigned* status, cudaStream_t st) {
  const int bx = (int)dev::min64(std::max<int64_t>((max_atoms + 255) / 256, 1), 64);
  k_bbox<<<dim3(bx, batch), 256, 0, st>>>(xyz, atom_off, bbox, status);
  return cuda_status(cudaGetLastError(), "bounding-box launch");
}

scatter_status launch_generic_reduce(scatter_plan_t p, int n_chunks, float2* amp_out, float* int_out,
                                     cudaStream_t st) {
  GenericArgs a = make_args(p);
  a.partial = p->d.partial;
  a.out_amp = amp_out;
  a.out_int = int_out;
  if (p->n_s > 0) {
    launch_reduce(a, n_chunks, mode_of(p) == kModeGrid, st);
    p->last_launches += 1;
  }
  return cuda_status(cudaGetLastError(), "generic reduction launch");
}

scatter_status launch_generic(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st, const CallGate& gate) {
  if (p->gs.active) return launch_gridsum(p, amp_out, int_out, st, gate);
  if (p->cl.active) {
    const scatter_status cs = launch_clusters(p, amp_out, int_out, st);
    if (cs != SCATTER_OK) return cs;
  }
  if (p->tiling.atom_k > 0) return launch_atompar(p, amp_out, int_out, st);
  const Tiling& t = p->tiling;
  void* fn = pick_generic(mode_of(p), t.R, t.threads);
  if (!fn) return fail(SCATTER_ERR_UNSUPPORTED, "no generic kernel for R=%d threads=%d", t.R, t.threads);
  GenericArgs a = make_args(p);
  const int n_chunks = (int)p->chunk_seg_off.size() - 1;
  if (n_chunks > 1) {
    a.partial = p->d.partial;
  } else {
    a.out_amp = amp_out;
    a.out_int = int_out;
  }
  const int64_t tiles = generic_num_tiles(p, t);
  if (tiles > 0 && n_chunks > 0) {
    dim3 grid((unsigned)tiles, (unsigned)n_chunks);
    void* args[] = {&a};
    if (!p->cl.active) timing_begin(p, st);
    cudaError_t e = cudaLaunchKernel(fn, grid, dim3(t.threads), args, 0, st);
    timing_end(p, st);
    if (e != cudaSuccess) return cuda_status(e, "generic kernel launch");
    p->last_launches += 1;
  }
  if (n_chunks > 1) {
    a.partial = p->d.partial;
    a.out_amp = amp_out;
    a.out_int = int_out;
    launch_reduce(a, n_chunks, mode_of(p) == kModeGrid, st);
    p->last_launches += 1;
  }
  return cuda_status(cudaGetLastError(), "generic launch");
}

// Launches the LIST-mode generic kernel (and the split-K reduction) on fully
// prepared arguments; used by callers that own their buffers.
scatter_status launch_generic_args(GenericArgs a, int R, int threads, int n_chunks, cudaStream_t st) {
  void* fn = pick_generic(kModeList, R, threads);
  if (!fn) return fail(SCATTER_ERR_UNSUPPORTED, "no generic kernel for R=%d threads=%d", R, threads);
  float2* out_amp = a.out_amp;
  float* out_int = a.out_int;
  float2* partial = a.partial;
  if (n_chunks > 1) {
    a.out_amp = nullptr;
    a.out_int = nullptr;
  } else {
    a.partial = nullptr;
  }
  const int64_t per = (int64_t)threads * R;
  const int64_t tiles = (a.n_s + per - 1) / per;
  if (tiles > 0 && n_chunks > 0) {
    void* args[] = {&a};
    cudaError_t e = cudaLaunchKernel(fn, dim3((unsigned)tiles, (unsigned)n_chunks), dim3(threads), args, 0, st);
    if (e != cudaSuccess) return cuda_status(e, "generic kernel launch");
  }
  if (n_chunks > 1 && a.n_s > 0) {
    a.partial = partial;
    a.out_amp = out_amp;
    a.out_int = out_int;
    launch_reduce(a, n_chunks, 0, st);
  }
  return cuda_status(cudaGetLastError(), "generic launch");
}

}  // namespace scatter
