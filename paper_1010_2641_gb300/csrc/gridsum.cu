// FP32 sum on axis-aligned grids: rows of two axes times a table of the third.
//
// On a grid S = H + s the phase of Eq. 2 separates, so with one axis q chosen
// as the columns and the other two as the rows
//   w_j e^{2 i pi (c_j + s.x'_j)} = E[row, j] Z[col, j],
//   E = e^{2 i pi (c_j + s_u u_j + s_v v_j)}        one MUFU sincos per (row, atom)
//   Z = w_j e^{2 i pi s_q q_j}                      a table in shared memory
// and a point costs four FP32 multiply-adds instead of a phase, its reduction
// and a sincos.  The products run as packed pairs, (P, R) += Er (Zr, Zi) and
// (T, Q) += Ei (Zr, Zi), with E Z = (P - Q, R + T) and E conj(Z) = (P + Q,
// T - R): where the column axis is symmetric about its middle the same four
// sums give a column and its mirror (the middle's phase joins c_j), two
// multiply-adds per point.  All in FP32 like the sincos form (forward.cu), the
// table's entries to ~1 ulp, the sums blocked by 128 atoms.
//
// CTA: up to 256 rows (one per thread) x R columns (in registers) x one chunk
// of atoms of one species.  A tile of 128 atoms is staged in shared memory:
// the rows' records (u, v, phase) and the R table entries per atom, read as
// broadcasts; two stages, one barrier per tile.  On small sums the CTA forms
// them itself from the atoms (128 R sincospif per tile and CTA: a sixth of the
// instructions with 64 rows per CTA); on larger ones (TAB) a kernel writes them
// once per call and the TMA engine copies them in.  Bound by issue (R = 6:
// 33 instructions per row and atom for 12 points, 3.3 per clock).  The loop
// is unrolled over 16 atoms: with 8 warps per SM the sincos latency is hidden
// inside a warp (1.33 ms with 4 atoms, 1.19 ms with 16).
// Strained sphere (134,009 atoms) x 61 x 47 x 33: 1.19 ms per call against 6.69 ms in
// the sincos form (1.73 ms with 64 rows per CTA forming their own tables);
// 1000 atoms x 32^3: 33 against 67 us.
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>
#include "device_common.cuh"
#include "launch.h"

namespace scatter {

namespace {

constexpr int kGsTile = 128;   // atoms per stage
constexpr int kGsMaxR = 8;     // columns per thread
constexpr int kGsChunk = 32;   // chunk granularity (slots)
constexpr int64_t kGsMaxTiles = 65535;  // column tiles and chunks: y and z of the launch grid

struct GridSumArgs {
  const float4* atom4;
  const float4* atom_lo;
  const float* atom_w;
  const Segment* chunks;       // one species each
  const float* axis_s;         // [n0 | n1 | n2] s = axis - H, and rounding errors
  const float* axis_lo;
  const float* col_d;          // column offsets (from H, or from the middle of a symmetric axis)
  const float* col_dlo;
  float mid, mid_lo;           // that middle - H, else 0
  int iu, iv, iq;              // coordinate of the slow and fast row axis, of the columns
  int64_t off_u, off_v;        // their axes in axis_s
  int64_t n_u, n_v;            // row axis lengths
  int64_t n_cols, n_q;         // columns summed, columns of the axis (mirror: n_cols = (n_q + 1) / 2)
  int mirror;
  int64_t st_u, st_v, st_q;    // output strides
  int64_t n_s;
  const unsigned long long* bbox;
  const double* shift;
  float smax[3];               // max |s| per axis, 0 for the columns' (their products are exact)
  float2* partial;             // [chunk][M], without f_s
  // TAB: the tiles' contents, written by k_gridsum_tab
  float4* rec;                 // [slot] (u, v, phase, 0)
  float2* rec_lo;              // [slot] rounding errors of u, v
  float2* ztab;                // [column tile][slot][RS]
  int64_t n_slots;
  unsigned* status;
  CallGate gate;
};

__device__ __forceinline__ float comp(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : v.z; }

// The record and the table entry of a slot (shared by the table kernel and the
// CTAs that form their own tiles: the two routes agree bit for bit).
__device__ __forceinline__ void gs_record(const GridSumArgs& a, int64_t slot, float4& rec, float2& lo2) {
  const float4 at = a.atom4[slot], lo = a.atom_lo[slot];
  const float q = comp(at, a.iq);
  const float ph = dev::frac_of_product2(a.mid, a.mid_lo, q) + a.mid * comp(lo, a.iq);
  rec = make_float4(comp(at, a.iu), comp(at, a.iv), dev::frac_rn(at.w + ph), 0.f);
  lo2 = make_float2(comp(lo, a.iu), comp(lo, a.iv));
}
__device__ __forceinline__ float2 gs_entry(const GridSumArgs& a, int64_t slot, float d, float dl) {
  const float q = comp(a.atom4[slot], a.iq), ql = comp(a.atom_lo[slot], a.iq), w = a.atom_w[slot];
  float sn, cs;
  sincospif(2.0f * (dev::frac_of_product2(d, dl, q) + d * ql), &sn, &cs);
  return make_float2(w * cs, w * sn);
}

// One thread per table entry (column tile, slot, column).
__global__ void __launch_bounds__(256) k_gridsum_tab(const GridSumArgs a, int R, int RS, int64_t total) {
  if (within(a.gate, 0)) return;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int r = (int)(i % RS);
  const int64_t slot = (i / RS) % a.n_slots, ct = i / RS / a.n_slots;
  const int64_t c = dev::min64(ct * R + r, a.n_cols - 1);
  a.ztab[i] = r < R ? gs_entry(a, slot, a.col_d[c], a.col_dlo[c]) : make_float2(0.f, 0.f);
  if (ct == 0 && r == 0) gs_record(a, slot, a.rec[slot], a.rec_lo[slot]);
}

template <int R, bool TAB>
__global__ void __launch_bounds__(256, 2) k_gridsum(const GridSumArgs a) {
  if (within(a.gate, 0)) return;
  constexpr int RS = R + (R & 1);  // table row stride: 16-byte aligned
  __shared__ __align__(16) float4 sh_rec[2][kGsTile];     // (u, v, phase, 0)
  __shared__ __align__(16) float2 sh_lo[2][kGsTile];      // rounding errors of u, v (exact phases)
  __shared__ __align__(16) float2 sh_z[2][kGsTile][RS];
  __shared__ float2 sh_d[R];
  __shared__ __align__(8) uint64_t sh_bar[2];
  using u64 = unsigned long long;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int64_t row = (int64_t)blockIdx.x * nt + tid, n_rows = a.n_u * a.n_v;
  const bool row_ok = row < n_rows;
  const int64_t iu = row_ok ? row / a.n_v : 0, iv = row_ok ? row % a.n_v : 0;
  const int64_t col0 = (int64_t)blockIdx.y * R;
  const Segment ck = a.chunks[blockIdx.z];
  const float su = a.axis_s[a.off_u + iu], sv = a.axis_s[a.off_v + iv];
  if (tid < R) {
    const int64_t c = dev::min64(col0 + tid, a.n_cols - 1);
    sh_d[tid] = make_float2(a.col_d[c], a.col_dlo[c]);
  }
  const bool exact = dev::phase_needs_exact(a.bbox, a.shift, a.smax);
  const float sul = a.axis_lo[a.off_u + iu], svl = a.axis_lo[a.off_v + iv];
  if (TAB && tid == 0) {
    dev::mbar_init(&sh_bar[0], 1);
    dev::mbar_init(&sh_bar[1], 1);
    dev::mbar_fence_init();
  }
  __syncthreads();

  // fills a stage with the tile at slot b (TAB: thread 0 starts the copies)
  auto form = [&](int64_t b, int st) {
    if (b >= ck.end) return;
    const int cnt = (int)dev::min64(kGsTile, ck.end - b);
    if constexpr (TAB) {
      if (tid != 0) return;
      const uint32_t zb = (uint32_t)cnt * RS * (uint32_t)sizeof(float2);
      dev::mbar_arrive_expect_tx(&sh_bar[st], zb + (uint32_t)cnt * (exact ? 24u : 16u));
      dev::bulk_g2s(&sh_z[st][0][0], a.ztab + ((int64_t)blockIdx.y * a.n_slots + b) * RS, zb, &sh_bar[st]);
      dev::bulk_g2s(&sh_rec[st][0], a.rec + b, (uint32_t)cnt * 16u, &sh_bar[st]);
      if (exact) dev::bulk_g2s(&sh_lo[st][0], a.rec_lo + b, (uint32_t)cnt * 8u, &sh_bar[st]);
    } else {
      for (int i = tid; i < cnt; i += nt) gs_record(a, b + i, sh_rec[st][i], sh_lo[st][i]);
      for (int i = tid; i < cnt * R; i += nt) {
        const int j = i / R, r = i % R;
        sh_z[st][j][r] = gs_entry(a, b + j, sh_d[r].x, sh_d[r].y);
      }
    }
  };

  float tot[R][4];
#pragma unroll
  for (int r = 0; r < R; ++r) tot[r][0] = tot[r][1] = tot[r][2] = tot[r][3] = 0.f;
  form(ck.begin, 0);
  if (TAB) form(ck.begin + kGsTile, 1);
  if (!TAB) __syncthreads();
  int st = 0, k = 0;
  for (int64_t b = ck.begin; b < ck.end; b += kGsTile, st ^= 1, ++k) {
    const int cnt = (int)dev::min64(kGsTile, ck.end - b);
    const bool ok = !TAB || dev::mbar_wait_bounded(&sh_bar[st], (uint32_t)((k >> 1) & 1));
    u64 pk[R][2];  // (P, R), (T, Q) of the tile
#pragma unroll
    for (int r = 0; r < R; ++r) pk[r][0] = pk[r][1] = 0ull;
    auto tile = [&](auto exact_tag) {
      constexpr bool kExact = decltype(exact_tag)::value;
      const float4* rec = sh_rec[st];
      const float2* rlo = sh_lo[st];
      auto add = [&](float er, float ei, const float2* z) {
        const u64 er2 = dev::pack2(er, er), ei2 = dev::pack2(ei, ei);
#pragma unroll
        for (int r = 0; r + 1 < RS; r += 2) {
          const float4 zz = *reinterpret_cast<const float4*>(z + r);
          const u64 z0 = dev::pack2(zz.x, zz.y), z1 = dev::pack2(zz.z, zz.w);
          dev::ffma2(pk[r][0], er2, z0);
          dev::ffma2(pk[r][1], ei2, z0);
          if (r + 1 < R) {
            dev::ffma2(pk[r + 1 < R ? r + 1 : r][0], er2, z1);
            dev::ffma2(pk[r + 1 < R ? r + 1 : r][1], ei2, z1);
          }
        }
      };
      if (kExact) {
#pragma unroll 2
        for (int j = 0; j < cnt; ++j) {
          const float4 at = rec[j];
          const float2 e = rlo[j];
          const float f = dev::frac_rn(dev::frac_product2_plus(
              su, sul, at.x, dev::frac_product2_plus(sv, svl, at.y, fmaf(su, e.x, fmaf(sv, e.y, at.z)))));
          float er, ei;
          dev::sincos_cycles_mufu(f, &ei, &er);
          add(er, ei, sh_z[st][j]);
        }
      } else {
        // two atoms' phases per packed pair (tiles hold multiples of 32 atoms)
        const u64 su2 = dev::pack2(su, su), sv2 = dev::pack2(sv, sv);
        const u64 magic2 = dev::pack2(12582912.0f, 12582912.0f);  // 1.5 * 2^23: rint by addition
        const u64 twopi2 = dev::pack2(6.28318530717958647692f, 6.28318530717958647692f);
#pragma unroll 8
        for (int j = 0; j < cnt; j += 2) {
          const float4 p0 = rec[j], p1 = rec[j + 1];
          const u64 ph = dev::fma2(sv2, dev::pack2(p0.y, p1.y),
                                   dev::fma2(su2, dev::pack2(p0.x, p1.x), dev::pack2(p0.z, p1.z)));
          const u64 f = dev::sub2(ph, dev::sub2(dev::add2(ph, magic2), magic2));  // ph - rint(ph)
          float t0, t1;
          dev::unpack2(dev::mul2(f, twopi2), t0, t1);
          add(__cosf(t0), __sinf(t0), sh_z[st][j]);
          add(__cosf(t1), __sinf(t1), sh_z[st][j + 1]);
        }
      }
    };
    if (ok) {
      if (exact)
        tile(std::true_type{});
      else
        tile(std::false_type{});
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float P, Rr, T, Q;
      dev::unpack2(pk[r][0], P, Rr);
      dev::unpack2(pk[r][1], T, Q);
      tot[r][0] += P - Q;  // E Z
      tot[r][1] += Rr + T;
      tot[r][2] += P + Q;  // E conj(Z)
      tot[r][3] += T - Rr;
    }
    if constexpr (TAB) {
      if (__syncthreads_or(!ok)) {
        if (tid == 0) {
          dev::set_status(a.status, kStatusTimeout);
          // drain the copies still in flight (bounded): this stage's and the next one's
          dev::mbar_wait_bounded(&sh_bar[st], (uint32_t)((k >> 1) & 1), 1LL << 28);
          if (b + kGsTile < ck.end) dev::mbar_wait_bounded(&sh_bar[st ^ 1], (uint32_t)(((k + 1) >> 1) & 1), 1LL << 28);
        }
        return;
      }
      form(b + 2 * kGsTile, st);
    } else {
      form(b + kGsTile, st ^ 1);
      __syncthreads();
    }
  }
  if (!row_ok) return;
  float2* out = a.partial + (int64_t)blockIdx.z * a.n_s + iu * a.st_u + iv * a.st_v;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t c = col0 + r;
    if (c >= a.n_cols) break;
    out[c * a.st_q] = make_float2(tot[r][0], tot[r][1]);
    const int64_t m = a.n_q - 1 - c;
    if (a.mirror && m != c) out[m * a.st_q] = make_float2(tot[r][2], tot[r][3]);
  }
}

struct GridSumReduce {
  const float2* partial;
  const Segment* chunks;
  int n_chunks;
  const float* coef;
  const float2* ftab;
  float inv4a2;
  const float* axis_s;
  const double* axis64;
  int64_t n0, n1, n2, n_s;
  float H[3];
  double H64[3];
  const double* shift;
  float2* out_amp;
  float* out_int;
  CallGate gate;
};

// Ordered sum of the chunks with f_s(|S|) per species run, translation phase,
// outputs; one thread per point, eight chunks' loads in flight.
__global__ void __launch_bounds__(128) k_gridsum_reduce(const GridSumReduce a) {
  const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= a.n_s || within(a.gate, 0)) return;
  const int64_t i2 = m % a.n2, line = m / a.n2, i1 = line % a.n1, i0 = line / a.n1;
  const float Sx = a.H[0] + a.axis_s[i0], Sy = a.H[1] + a.axis_s[a.n0 + i1], Sz = a.H[2] + a.axis_s[a.n0 + a.n1 + i2];
  const float s2 = (Sx * Sx + Sy * Sy + Sz * Sz) * a.inv4a2;
  float2 v = make_float2(0.f, 0.f), T = v;
  constexpr int kU = 8;
  for (int c0 = 0; c0 < a.n_chunks; c0 += kU) {
    float2 x[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      x[u] = c0 + u < a.n_chunks ? a.partial[(int64_t)(c0 + u) * a.n_s + m] : make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int c = c0 + u;
      if (c >= a.n_chunks) break;
      T.x += x[u].x;
      T.y += x[u].y;
      const int sp = a.chunks[c].species;
      if (c + 1 < a.n_chunks && a.chunks[c + 1].species == sp) continue;
      const float2 F = a.ftab ? a.ftab[(int64_t)sp * a.n_s + m] : dev::form_factor(a.coef + kNCoef * sp, s2);
      const float2 p = dev::cmul(F, T);
      v.x += p.x;
      v.y += p.y;
      T = make_float2(0.f, 0.f);
    }
  }
  const double* t = a.shift;
  if (t[0] != 0.0 || t[1] != 0.0 || t[2] != 0.0)
    v = dev::cmul(dev::shift_phase(a.axis64[i0] - a.H64[0], a.axis64[a.n0 + i1] - a.H64[1],
                                   a.axis64[a.n0 + a.n1 + i2] - a.H64[2], t),
                  v);
  if (a.out_amp) a.out_amp[m] = v;
  if (a.out_int) a.out_int[m] = v.x * v.x + v.y * v.y;
}

using GridSumFn = void (*)(const GridSumArgs);
template <int R>
GridSumFn pick(int r, bool tab) {
  if constexpr (R == 0)
    return nullptr;
  else
    return r != R ? pick<R - 1>(r, tab) : tab ? (GridSumFn)k_gridsum<R, true> : (GridSumFn)k_gridsum<R, false>;
}

// SM clocks per warp and atom with R columns, measured on the strained sphere's
// 61 x 47 x 33 map (8 to 16 warps per SM): R = 6 is the cheapest per column, at
// 33 instructions in 10 clocks; more columns leave too few registers for the
// unrolled loop, fewer repeat the row's sincos, odd ones split a 16-byte read.
double warp_cost(int R) {
  static const double c[kGsMaxR + 1] = {0.0, 5.2, 6.4, 7.9, 8.0, 9.0, 10.0, 11.4, 14.1};
  return c[R];
}

struct Shape {
  int q = 2, R = 1, threads = 256;
  bool mirror = false;
  double cost = 1e300;  // SM clocks per atom over the whole grid
};

Shape best_shape(const scatter_plan_s* p) {
  Shape best;
  for (int q = 0; q < 3; ++q) {
    const int64_t n = p->n_axis[q];
    double mid;
    const bool mirror = axis_symmetric(p->axis_host[q], &mid);
    const int64_t cols = mirror ? (n + 1) / 2 : n, rows = p->n_s / n;
    for (int R = 1; R <= kGsMaxR; ++R) {
      if ((cols + R - 1) / R > kGsMaxTiles) continue;  // a long axis: more columns per thread, or rows
      for (int th : {64, 128, 256}) {
        const double warps = std::ceil((double)rows / th) * (th / 32);
        const double c = warps * std::ceil((double)cols / R) * warp_cost(R);
        if (c < best.cost * 0.999) best = Shape{q, R, th, mirror, c};
      }
    }
  }
  return best;
}

}  // namespace

bool axis_symmetric(const std::vector<double>& v, double* mid) {
  if (v.empty()) return false;
  double top = 1.0;
  for (double x : v) top = std::max(top, std::fabs(x));
  const size_t n = v.size();
  *mid = 0.5 * (v.front() + v.back());
  for (size_t i = 0; i < n; ++i)
    if (std::fabs(v[i] + v[n - 1 - i] - 2.0 * *mid) > 2e-13 * top) return false;
  return true;
}

// The sincos forms spend 4 SM clocks per 32 (atom, point) pairs on the MUFU pipe;
// the factorised form is taken where its clocks, rows and columns padded, are
// at most 7/8 of that: everything but a handful of points, or single lines
// shorter than a warp.
bool gridsum_preferred(const scatter_plan_s* p) {
  if (p->s_kind != SCATTER_S_GRID || p->batch != 1 || p->n_s <= 0) return false;
  return best_shape(p).cost < 0.875 * 4.0 * std::ceil((double)p->n_s / 32.0);
}

void release_gridsum(scatter_plan_s* p) {
  GridSum& g = p->gs;
  for (void* b : {(void*)g.chunks, (void*)g.d, (void*)g.dlo, (void*)g.rec, (void*)g.rec_lo, (void*)g.ztab,
                  (void*)p->d.partial})
    if (b) cudaFree(b);
  p->d.partial = nullptr;
  p->tiling_bytes -= g.bytes;
  g = GridSum{};
}

scatter_status prepare_gridsum(scatter_plan_s* p, int split_override) {
  const Shape sh = best_shape(p);
  release_gridsum(p);  // of an earlier split (autotuning)
  GridSum& g = p->gs;
  g.q = sh.q;
  g.R = sh.R;
  g.threads = sh.threads;
  g.mirror = sh.mirror;
  const int64_t n = p->n_axis[sh.q], rows = p->n_s / n;
  g.n_cols = sh.mirror ? (n + 1) / 2 : n;
  g.row_tiles = (rows + sh.threads - 1) / sh.threads;
  g.col_tiles = (g.n_cols + sh.R - 1) / sh.R;
  // The table where forming the tiles in every CTA (~45 instructions per entry)
  // would cost more than its launch, a few us, and it stays below 2 GiB.
  const double all_s = sh.cost * (double)p->n_slots / (2.0e9 * p->n_sm);
  const double form = 14.0 * sh.R / (sh.threads * warp_cost(sh.R));  // of that, 45 instructions at ~3.3 per clock
  const int RS = sh.R + (sh.R & 1);
  const size_t zb = (size_t)g.col_tiles * (size_t)p->n_slots * RS * sizeof(float2);
  g.tab = all_s * form > 8.0e-6 && zb <= (size_t)2 << 30;
  GridSumFn fn = pick<kGsMaxR>(sh.R, g.tab);
  int per_sm = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, sh.threads, 0) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  // atom chunks: the split that minimises waves x atoms per CTA, with ~1.5 us of
  // fixed cost per CTA and the partials' write and read
  const double cap = (double)p->n_sm * per_sm, tiles = (double)(g.row_tiles * g.col_tiles);
  const double clk = 2.0e9, warps = sh.threads / 32.0;
  int64_t total = 0;
  for (const Segment& sg : p->all_segs) total += (sg.end - sg.begin) / kGsChunk;
  // steps per chunk and chunks of a species segment of `steps` steps for a split k
  auto pieces = [&](int64_t steps, int k, int64_t& per) {
    const int64_t n = std::max<int64_t>(1, std::llround((double)k * (double)steps / (double)total));
    per = (steps + n - 1) / n;
    return (steps + per - 1) / per;
  };
  auto cost = [&](int k) {
    int64_t n = 0, longest = 1;
    for (const Segment& sg : p->all_segs) {
      int64_t per = 0;
      n += pieces((sg.end - sg.begin) / kGsChunk, k, per);
      longest = std::max(longest, per);
    }
    const double ctas = tiles * (double)n, waves = std::ceil(ctas / cap);
    const double resident = std::min(per_sm * 1.0, std::max(1.0, ctas / p->n_sm));
    // latency-bound with few warps: full rate from 16 per SM on (1.43 ms with 12,
    // 1.19 ms with 16 on that map); the reduction reads eight chunks at a time
    const double rate = std::min(1.0, warps * resident / 16.0);
    const double atom = warp_cost(sh.R) * warps * resident / rate / clk;
    return waves * ((double)(longest * kGsChunk) * atom + 1.5e-6) +
           (double)n * ((double)p->n_s * 16.0 / 3.0e12 + 3.0e-7);
  };
  int split = 1;
  if (split_override > 0) {
    split = split_override;
  } else {
    const int most = (int)std::min<int64_t>(1024, std::max<int64_t>(1, p->n_slots / kGsChunk));
    double best = 1e300;
    for (int k = 1; k <= most; ++k)
      if (const double c = cost(k); c < best * 0.995) {
        best = c;
        split = k;
      }
  }
  std::vector<Segment> chunks;
  for (const Segment& sg : p->all_segs) {
    const int64_t steps = (sg.end - sg.begin) / kGsChunk;
    if (steps <= 0) continue;
    int64_t per = 0;
    pieces(steps, split, per);
    for (int64_t b = 0; b < steps; b += per)
      chunks.push_back(Segment{sg.begin + b * kGsChunk, sg.begin + std::min(steps, b + per) * kGsChunk, sg.species, 0});
  }
  if (chunks.empty()) chunks.push_back(Segment{0, 0, 0, 0});  // no atoms: one empty chunk, zero partials
  if ((int64_t)chunks.size() > kGsMaxTiles || g.col_tiles > kGsMaxTiles)
    return fail(SCATTER_ERR_UNSUPPORTED, "grid sum: %zu chunks or %lld column tiles exceed the launch grid",
                chunks.size(), (long long)g.col_tiles);
  g.n_chunks = (int)chunks.size();
  // column offsets: from the middle of a symmetric axis (first half), else from H
  const std::vector<double>& ax = p->axis_host[sh.q];
  const double H = p->inst[0].H[sh.q];
  double mid = H;
  if (sh.mirror) axis_symmetric(ax, &mid);
  g.mid = mid - H;
  std::vector<float> d, dl;
  for (int64_t i = 0; i < g.n_cols; ++i) {
    const double v = sh.mirror ? 0.5 * (ax[i] - ax[n - 1 - i]) : ax[i] - H;
    d.push_back((float)v);
    dl.push_back((float)(v - (double)(float)v));
  }
  cudaError_t e;
  const size_t db = d.size() * sizeof(float), cb = chunks.size() * sizeof(Segment);
  const size_t pb = chunks.size() * (size_t)p->n_s * sizeof(float2);
  auto alloc = [](auto** dst, size_t size) {
    return injected_alloc_failure() ? cudaErrorMemoryAllocation : cudaMalloc((void**)dst, size);
  };
  if ((e = alloc(&g.d, db)) != cudaSuccess || (e = alloc(&g.dlo, db)) != cudaSuccess ||
      (e = alloc(&g.chunks, cb)) != cudaSuccess || (e = alloc(&p->d.partial, pb)) != cudaSuccess)
    return cuda_status(e, "cudaMalloc grid sum");
  if ((e = cudaMemcpy(g.d, d.data(), db, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemcpy(g.dlo, dl.data(), db, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemcpy(g.chunks, chunks.data(), cb, cudaMemcpyHostToDevice)) != cudaSuccess)
    return cuda_status(e, "grid sum tables");
  size_t tb = 0;
  if (g.tab) {
    const size_t n4 = (size_t)p->n_slots * sizeof(float4), n2 = (size_t)p->n_slots * sizeof(float2);
    if ((e = alloc(&g.rec, n4)) != cudaSuccess || (e = alloc(&g.rec_lo, n2)) != cudaSuccess ||
        (e = alloc(&g.ztab, zb)) != cudaSuccess)
      return cuda_status(e, "cudaMalloc grid sum table");
    tb = n4 + n2 + zb;
  }
  g.bytes = (int64_t)(2 * db + cb + pb + tb);
  p->tiling_bytes += g.bytes;
  g.split = split;
  p->tiling.threads = sh.threads;
  p->tiling.R = sh.R * (sh.mirror ? 2 : 1);
  p->tiling.split_k = g.n_chunks;
  g.active = true;
  return SCATTER_OK;
}

scatter_status launch_gridsum(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st, const CallGate& gate) {
  const GridSum& g = p->gs;
  const int64_t n[3] = {p->n_axis[0], p->n_axis[1], p->n_axis[2]};
  const int64_t off[3] = {0, n[0], n[0] + n[1]}, stride[3] = {n[1] * n[2], n[2], 1};
  const int u = g.q == 0 ? 1 : 0, v = g.q == 2 ? 1 : 2;
  GridSumArgs a{};
  a.atom4 = p->d.atom4;
  a.atom_lo = p->d.atom_lo;
  a.atom_w = p->d.atom_w;
  a.chunks = g.chunks;
  a.axis_s = p->d.axis_s;
  a.axis_lo = p->d.axis_lo;
  a.col_d = g.d;
  a.col_dlo = g.dlo;
  a.mid = (float)g.mid;
  a.mid_lo = (float)(g.mid - (double)a.mid);
  a.iu = u;
  a.iv = v;
  a.iq = g.q;
  a.off_u = off[u];
  a.off_v = off[v];
  a.n_u = n[u];
  a.n_v = n[v];
  a.n_cols = g.n_cols;
  a.n_q = n[g.q];
  a.mirror = g.mirror;
  a.st_u = stride[u];
  a.st_v = stride[v];
  a.st_q = stride[g.q];
  a.n_s = p->n_s;
  a.bbox = p->d.inst_bbox;
  a.shift = p->d.inst_shift;
  for (int d = 0; d < 3; ++d) a.smax[d] = d == g.q ? 0.f : (float)p->s_max[d];
  a.partial = p->d.partial;
  a.rec = g.rec;
  a.rec_lo = g.rec_lo;
  a.ztab = g.ztab;
  a.n_slots = p->n_slots;
  a.status = p->d.status;
  a.gate = gate;
  if (g.tab) {
    const int RS = g.R + (g.R & 1);
    const int64_t total = g.col_tiles * p->n_slots * RS;
    k_gridsum_tab<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(a, g.R, RS, total);
    p->last_launches += 1;
  }
  if (!gate.rmax2) timing_begin(p, st);
  pick<kGsMaxR>(g.R, g.tab)<<<dim3((unsigned)g.row_tiles, (unsigned)g.col_tiles, (unsigned)g.n_chunks), g.threads, 0, st>>>(a);
  timing_end(p, st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "grid sum launch");
  GridSumReduce r{};
  r.partial = p->d.partial;
  r.chunks = g.chunks;
  r.n_chunks = g.n_chunks;
  r.coef = p->d.coef;
  r.ftab = p->d.ftab;
  r.inv4a2 = (float)(1.0 / (4.0 * p->lattice_a * p->lattice_a));
  r.axis_s = p->d.axis_s;
  r.axis64 = p->d.axis64;
  r.n0 = n[0];
  r.n1 = n[1];
  r.n2 = n[2];
  r.n_s = p->n_s;
  for (int d = 0; d < 3; ++d) {
    r.H[d] = (float)p->inst[0].H[d];
    r.H64[d] = p->inst[0].H[d];
  }
  r.shift = p->out_shift ? p->out_shift : p->d.inst_shift;
  r.gate = gate;
  r.out_amp = amp_out;
  r.out_int = int_out;
  k_gridsum_reduce<<<(unsigned)((p->n_s + 127) / 128), 128, 0, st>>>(r);
  p->last_launches += 2;
  return cuda_status(cudaGetLastError(), "grid sum reduction");
}

}  // namespace scatter
