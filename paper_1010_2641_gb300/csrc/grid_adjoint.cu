// FP32 adjoint on axis-aligned grids: rows of two axes times a table of the
// third, as the forward's factorised sum (gridsum.cu).
//
// With one axis q as the columns (offsets d from H, or from the middle of a
// symmetric axis) and the other two as the rows, an atom's sums over the points
//   sum gF e^{2 pi i s.x'}            = sum_rows E_row U0,   U0 = sum_q gF Z_q,
//   the same weighted with d          = sum_rows E_row U1,   U1 = sum_q d gF Z_q,
//   E_row = e^{2 pi i (c + s_u u + s_v v)},  Z_q = e^{2 pi i d_q q} = C + i S,
// and the gradient is H sum Im(E U0) + (sum s_u Im(E U0), sum s_v Im(E U0),
// sum Im(E U1)).  A column and its mirror -d share C and S:
//   gF Z + gF' conj(Z) = (gF + gF') C + i (gF - gF') S,
// so a pair of points costs eight multiply-adds (a single point on an axis
// without a middle as well), and a row of a thread's columns one sincos.
//
//   k_grid_adj_tab  per (species, row, pair): the eight coefficients of C and S in
//                   U0 and U1, each twice (two atoms per packed operation)
//   k_grid_adj      256 atoms of one species (two per thread, their C and S of NP
//                   pairs in registers) x a range of rows; rows staged by bulk
//                   copies, 16 per stage; FP32 sums per stage, double-float across
//                   (the sums over all points nearly cancel)
// Bound by the FMA pipe and the broadcast loads together (four 16-byte loads for
// eight packed multiply-adds).  27,040 atoms x 24,948 nodes: 0.17 ms against 0.35 ms
// of a sincos per pair (adjoint.cu); 76,664 atoms x 85 x 23 x 42 points, 1.04 ms per
// call against 2.10 ms of the line recurrence.  Chunks of up to 12, 10 or 8 pairs
// instead of 16: 0.30, 0.29 and 0.29 ms per call at the nodes against 0.26.
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <vector>
#include "device_common.cuh"
#include "launch.h"

namespace scatter {

namespace {

constexpr int kGaThreads = 128;
constexpr int kGaAtoms = 2 * kGaThreads;
constexpr int kGaRows = 16;   // rows per stage
constexpr int kGaMaxNP = 16;  // pairs per CTA
constexpr int kGaMaxY = 65535;  // row ranges x chunks of pairs: y of the launch grid

struct GridAdjArgs {
  const float4* atom4;
  const float4* atom_lo;
  const AdjBlock* blocks;
  const float* table;      // [species][chunk][row][NP][16]
  const float2* gf;        // [species][M]
  const float* axis_s;     // [n0 | n1 | n2] s = axis - H
  const float* col_d;      // column offsets and rounding errors
  const float* col_dlo;
  int64_t off_u, off_v, n_v, n_rows, rows_per_split;
  int64_t st_u, st_v, st_q, n_q, n_s;
  int iu, iv, iq, n_pairs, n_chunks, np, mirror;
  float mid, mid_lo;
  float h[3], h_lo[3];     // H (columns: + middle) and rounding errors
  float* partial;          // [split][n_slots][3]
  int64_t n_slots;
  unsigned* status;
  CallGate gate;
};

__device__ __forceinline__ float ga_comp(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : v.z; }

__global__ void __launch_bounds__(256) k_grid_adj_tab(const GridAdjArgs a, float* __restrict__ table, int64_t total) {
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= total || within(a.gate, 0)) return;
  const int64_t slots = (int64_t)a.n_chunks * a.np;
  // neighbouring threads: neighbouring pairs of a chunk's row
  const int p = (int)(e % a.np);
  const int64_t row = (e / a.np) % a.n_rows, ch = e / (a.np * a.n_rows) % a.n_chunks, sp = e / (slots * a.n_rows);
  const int64_t q = ch * a.np + p;
  float2 g = make_float2(0.f, 0.f), m = g;
  float d = 0.f;
  if (q < a.n_pairs) {
    const float2* gf = a.gf + sp * a.n_s + (row / a.n_v) * a.st_u + (row % a.n_v) * a.st_v;
    g = gf[q * a.st_q];
    if (a.mirror && q != a.n_q - 1 - q) m = gf[(a.n_q - 1 - q) * a.st_q];
    d = a.col_d[q];
  }
  const float2 P = make_float2(g.x + m.x, g.y + m.y), D = make_float2(g.x - m.x, g.y - m.y);
  float4* out = reinterpret_cast<float4*>(table + e * 16);
  out[0] = make_float4(P.x, P.x, P.y, P.y);
  out[1] = make_float4(-D.y, -D.y, D.x, D.x);
  out[2] = make_float4(d * D.x, d * D.x, d * D.y, d * D.y);
  out[3] = make_float4(-d * P.y, -d * P.y, d * P.x, d * P.x);
}

template <int NP>
__global__ void __launch_bounds__(kGaThreads) k_grid_adj(const GridAdjArgs a) {
  using u64 = unsigned long long;
  __shared__ __align__(128) float sh_t[2][kGaRows][NP * 16];
  __shared__ float2 sh_s[2][kGaRows];
  __shared__ __align__(8) uint64_t sh_bar[2];
  if (within(a.gate, 0)) return;
  const int t = threadIdx.x;
  const AdjBlock blk = a.blocks[blockIdx.x];
  const int ch = blockIdx.y % a.n_chunks;
  const int64_t r0 = (int64_t)(blockIdx.y / a.n_chunks) * a.rows_per_split, r1 = dev::min64(a.n_rows, r0 + a.rows_per_split);
  const float* tab = a.table + ((int64_t)(blk.species * a.n_chunks + ch) * a.n_rows) * (NP * 16);
  if (t == 0) {
    dev::mbar_init(&sh_bar[0], 1);
    dev::mbar_init(&sh_bar[1], 1);
    dev::mbar_fence_init();
  }
  float u[2], v[2], c[2];
  u64 C[NP], S[NP];
  {
    float cs[2][NP], sn[2][NP];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int i = r * kGaThreads + t;
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 at = i < blk.count ? a.atom4[blk.begin + i] : zero, lo = i < blk.count ? a.atom_lo[blk.begin + i] : zero;
      const float q = ga_comp(at, a.iq), ql = ga_comp(lo, a.iq);
      u[r] = ga_comp(at, a.iu);
      v[r] = ga_comp(at, a.iv);
      c[r] = dev::frac_rn(at.w + dev::frac_of_product2(a.mid, a.mid_lo, q) + a.mid * ql);
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const int64_t k = ch * NP + p;
        const float d = k < a.n_pairs ? a.col_d[k] : 0.f, dl = k < a.n_pairs ? a.col_dlo[k] : 0.f;
        sincospif(2.0f * (dev::frac_of_product2(d, dl, q) + d * ql), &sn[r][p], &cs[r][p]);
      }
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      C[p] = dev::pack2(cs[0][p], cs[1][p]);
      S[p] = dev::pack2(sn[0][p], sn[1][p]);
    }
  }
  const int64_t n_tiles = r1 > r0 ? (r1 - r0 + kGaRows - 1) / kGaRows : 0;
  auto issue = [&](int64_t k) {
    if (k >= n_tiles) return;
    const int64_t b = r0 + k * kGaRows;
    const int st = (int)(k & 1);
    const uint32_t bytes = (uint32_t)dev::min64(kGaRows, r1 - b) * NP * 64u;
    if (t == 0) {
      dev::mbar_arrive_expect_tx(&sh_bar[st], bytes);
      dev::bulk_g2s(&sh_t[st][0][0], tab + b * (NP * 16), bytes, &sh_bar[st]);
    }
    if (t < kGaRows && b + t < r1)  // read two barriers on
      sh_s[st][t] = make_float2(a.axis_s[a.off_u + (b + t) / a.n_v], a.axis_s[a.off_v + (b + t) % a.n_v]);
  };
  __syncthreads();
  issue(0);
  issue(1);
  __syncthreads();
  dev::DFloatSum gv[2], gu[2], gw[2], gq[2];
  bool aborted = false;
  for (int64_t k = 0; k < n_tiles; ++k) {
    const int st = (int)(k & 1);
    const int cnt = (int)dev::min64(kGaRows, r1 - (r0 + k * kGaRows));
    const bool ok = dev::mbar_wait_bounded(&sh_bar[st], (uint32_t)((k >> 1) & 1));
    u64 av = 0ull, au = 0ull, aw = 0ull, aq = 0ull;
    if (ok) {
#pragma unroll 1
      for (int j = 0; j < cnt; ++j) {
        const float2 s = sh_s[st][j];
        float er[2], ei[2];
#pragma unroll
        for (int r = 0; r < 2; ++r)
          dev::sincos_cycles_mufu(dev::frac_rn(dev::frac_product_plus(s.x, u[r], dev::frac_product_plus(s.y, v[r], c[r]))),
                                  &ei[r], &er[r]);
        u64 u0r = 0ull, u0i = 0ull, u1r = 0ull, u1i = 0ull;
        const ulonglong2* g = reinterpret_cast<const ulonglong2*>(&sh_t[st][j][0]);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const ulonglong2 g0 = g[4 * p], g1 = g[4 * p + 1], g2 = g[4 * p + 2], g3 = g[4 * p + 3];
          dev::ffma2(u0r, g0.x, C[p]);
          dev::ffma2(u0i, g0.y, C[p]);
          dev::ffma2(u1r, g2.x, C[p]);
          dev::ffma2(u1i, g2.y, C[p]);
          dev::ffma2(u0r, g1.x, S[p]);
          dev::ffma2(u0i, g1.y, S[p]);
          dev::ffma2(u1r, g3.x, S[p]);
          dev::ffma2(u1i, g3.y, S[p]);
        }
        const u64 er2 = dev::pack2(er[0], er[1]), ei2 = dev::pack2(ei[0], ei[1]);
        const u64 im = dev::fma2(ei2, u0r, dev::mul2(er2, u0i));
        av = dev::add2(av, im);
        au = dev::fma2(dev::pack2(s.x, s.x), im, au);
        aw = dev::fma2(dev::pack2(s.y, s.y), im, aw);
        aq = dev::fma2(ei2, u1r, dev::fma2(er2, u1i, aq));
      }
    }
    float x0, x1;
    dev::unpack2(av, x0, x1), gv[0].add(x0), gv[1].add(x1);
    dev::unpack2(au, x0, x1), gu[0].add(x0), gu[1].add(x1);
    dev::unpack2(aw, x0, x1), gw[0].add(x0), gw[1].add(x1);
    dev::unpack2(aq, x0, x1), gq[0].add(x0), gq[1].add(x1);
    if (__syncthreads_or(!ok)) {
      aborted = true;
      if (t == 0) {
        dev::set_status(a.status, kStatusTimeout);
        for (int64_t kk = k; kk < dev::min64(k + 2, n_tiles); ++kk)
          dev::mbar_wait_bounded(&sh_bar[kk & 1], (uint32_t)((kk >> 1) & 1), 1LL << 28);
      }
      break;
    }
    issue(k + 2);
  }
  if (aborted) return;
  float* out = a.partial + (int64_t)blockIdx.y * a.n_slots * 3;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int i = r * kGaThreads + t;
    if (i >= blk.count) continue;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const dev::DFloatSum& own = d == a.iu ? gu[r] : d == a.iv ? gw[r] : gq[r];
      dev::DFloatSum s;
      s.hi = __fmul_rn(a.h[d], gv[r].hi);
      s.lo = __fmaf_rn(a.h[d], gv[r].hi, -s.hi) + fmaf(a.h[d], gv[r].lo, a.h_lo[d] * gv[r].hi);
      s.add(own.hi);
      s.lo += own.lo;
      out[3 * (blk.begin + i) + d] = s.value();
    }
  }
}

template <int NP>
const void* ga_kernel(int np) {
  if (np == NP) return (const void*)k_grid_adj<NP>;
  if constexpr (NP > 2) return ga_kernel<NP - 2>(np);
  return nullptr;
}

// Columns on axis q, pairs per CTA and chunks of them; lane operations per atom.
struct GaShape {
  int q = -1, np = 0, chunks = 0, pairs = 0;
  bool mirror = false;
  double mid = 0.0, cost = 1e300;
};
GaShape ga_shape(const scatter_plan_s* p) {
  GaShape best;
  for (int q = 0; q < 3; ++q) {
    GaShape s;
    s.q = q;
    s.mirror = axis_symmetric(p->axis_host[q], &s.mid);
    const int64_t n = p->n_axis[q], pairs = s.mirror ? (n + 1) / 2 : n;
    if (pairs > (int64_t)kGaMaxNP * kGaMaxY) continue;
    s.pairs = (int)pairs;
    s.chunks = (s.pairs + kGaMaxNP - 1) / kGaMaxNP;
    s.np = 2 * ((s.pairs + 2 * s.chunks - 1) / (2 * s.chunks));
    // eight multiply-adds per pair, some 45 operations per row
    s.cost = (double)(p->n_s / n) * s.chunks * (8.0 * s.np + 45.0) / 0.7;
    if (!s.mirror) s.mid = 0.0;
    if (s.cost < best.cost) best = s;
  }
  return best;
}

bool uniform_l(const scatter_plan_s* p) {
  const std::vector<double>& l = p->axis_host[2];
  const int64_t n = (int64_t)l.size();
  const double ds = n > 1 ? (l[n - 1] - l[0]) / (double)(n - 1) : 0.0;
  for (int64_t i = 0; i < n; ++i)
    if (std::fabs(l[i] - (l[0] + (double)i * ds)) > 1e-9 * std::max(1.0, std::fabs(l[i]))) return false;
  return true;
}

}  // namespace

// Lane operations per atom and point of the FP32 adjoint's best form: the line
// recurrence 8 at 0.74 of the FMA pipe, the tiles 16 (eight pairs per clock) at 0.8,
// this one as above.
double grid_adjoint_ops(const scatter_plan_s* p) {
  const double other = (double)p->n_s * (uniform_l(p) ? 10.8 : 20.0);
  return std::min(other, ga_shape(p).cost) / (double)p->n_s;
}

scatter_status prepare_grid_adjoint(scatter_plan_s* p) {
  GridAdjState& g = p->ga;
  if (p->s_kind != SCATTER_S_GRID || p->batch != 1 || p->n_s <= 0 || p->n_slots <= 0 || g.active) return SCATTER_OK;
  const GaShape s = ga_shape(p);
  if (s.q < 0 || s.cost > 0.9 * (double)p->n_s * (uniform_l(p) ? 10.8 : 20.0)) return SCATTER_OK;
  const int64_t n_rows = p->n_s / p->n_axis[s.q];
  const size_t tab = (size_t)p->n_species * (size_t)s.chunks * (size_t)n_rows * (size_t)s.np * 64;
  if (tab > ((size_t)16 << 30)) return SCATTER_OK;
  std::vector<AdjBlock> blocks;
  for (const Segment& sg : p->all_segs)
    for (int64_t b = sg.begin; b < sg.end; b += kGaAtoms)
      blocks.push_back(AdjBlock{b, (int32_t)std::min<int64_t>(kGaAtoms, sg.end - b), sg.species});
  const void* kernel = ga_kernel<kGaMaxNP>(s.np);
  int bps = 0;
  if (!kernel || blocks.empty() ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kernel, kGaThreads, 0) != cudaSuccess || bps < 1) {
    cudaGetLastError();
    return SCATTER_OK;
  }
  // rows per CTA: waves x (rows + some 20 rows' worth of table and output)
  double best = 1e300;
  const double cap = (double)p->n_sm * bps, base = (double)blocks.size() * s.chunks;
  for (int64_t split = 1; split <= std::min<int64_t>(n_rows, 4096) && split * s.chunks <= kGaMaxY; ++split) {
    const int64_t per = (n_rows + split - 1) / split, n = (n_rows + per - 1) / per;
    const double cost = std::ceil(base * (double)n / cap) * ((double)per + 20.0) + 0.02 * (double)n;
    if (cost < best * 0.999) {
      best = cost;
      g.rows_per_split = per;
      g.split = (int)n;
    }
    if (base * (double)split > 64.0 * cap) break;
  }
  std::vector<float> d, dlo;
  for (int k = 0; k < s.pairs; ++k) {
    const double v = p->axis_host[s.q][k] - (s.mirror ? s.mid : p->inst[0].H[s.q]);
    d.push_back((float)v);
    dlo.push_back((float)(v - (double)(float)v));
  }
  const size_t part = (size_t)g.split * s.chunks * (size_t)p->n_slots * 3 * sizeof(float);
  const size_t gf = (size_t)p->n_species * (size_t)p->n_s * sizeof(float2);
  auto put = [](auto** dst, const auto& v) {
    return cudaMalloc((void**)dst, v.size() * sizeof(v[0])) == cudaSuccess &&
           cudaMemcpy(*dst, v.data(), v.size() * sizeof(v[0]), cudaMemcpyHostToDevice) == cudaSuccess;
  };
  const bool ok = put(&g.blocks, blocks) && put(&g.d, d) && put(&g.dlo, dlo) &&
                  cudaMalloc((void**)&g.table, tab) == cudaSuccess && cudaMalloc((void**)&g.partial, part) == cudaSuccess &&
                  cudaMalloc((void**)&g.gf, gf) == cudaSuccess;
  if (!ok) {  // no room: the line or tile form needs less
    cudaGetLastError();
    release_grid_adjoint(g);
    return SCATTER_OK;
  }
  g.q = s.q;
  g.np = s.np;
  g.chunks = s.chunks;
  g.pairs = s.pairs;
  g.mirror = s.mirror;
  g.mid = s.mirror ? s.mid - p->inst[0].H[s.q] : 0.0;
  g.n_blocks = (int)blocks.size();
  p->adj_line = uniform_l(p);  // the form that is reported
  p->base_bytes += (int64_t)(tab + part + gf + blocks.size() * sizeof(AdjBlock) + 8 * d.size());
  g.active = true;
  return SCATTER_OK;
}

scatter_status launch_grid_adjoint(scatter_plan_t p, const float2* gf, cudaStream_t st, const CallGate& gate) {
  const GridAdjState& g = p->ga;
  const int64_t n[3] = {p->n_axis[0], p->n_axis[1], p->n_axis[2]};
  const int64_t off[3] = {0, n[0], n[0] + n[1]}, stride[3] = {n[1] * n[2], n[2], 1};
  const int u = g.q == 0 ? 1 : 0, v = g.q == 2 ? 1 : 2;
  GridAdjArgs a{};
  a.atom4 = p->d.atom4;
  a.atom_lo = p->d.atom_lo;
  a.blocks = g.blocks;
  a.table = g.table;
  a.gf = gf;
  a.axis_s = p->d.axis_s;
  a.col_d = g.d;
  a.col_dlo = g.dlo;
  a.off_u = off[u];
  a.off_v = off[v];
  a.n_v = n[v];
  a.n_rows = n[u] * n[v];
  a.rows_per_split = g.rows_per_split;
  a.st_u = stride[u];
  a.st_v = stride[v];
  a.st_q = stride[g.q];
  a.n_q = n[g.q];
  a.n_s = p->n_s;
  a.iu = u;
  a.iv = v;
  a.iq = g.q;
  a.n_pairs = g.pairs;
  a.n_chunks = g.chunks;
  a.np = g.np;
  a.mirror = g.mirror;
  a.mid = (float)g.mid;
  a.mid_lo = (float)(g.mid - (double)a.mid);
  for (int d = 0; d < 3; ++d) {
    const double h = p->inst[0].H[d] + (d == g.q ? g.mid : 0.0);
    a.h[d] = (float)h;
    a.h_lo[d] = (float)(h - (double)a.h[d]);
  }
  a.partial = g.partial;
  a.n_slots = p->n_slots;
  a.status = p->d.status;
  a.gate = gate;
  const int64_t total = (int64_t)p->n_species * g.chunks * a.n_rows * g.np;
  k_grid_adj_tab<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(a, g.table, total);
  if (!gate.rmax2) timing_begin(p, st);
  void* args[] = {&a};
  const cudaError_t e = cudaLaunchKernel(ga_kernel<kGaMaxNP>(g.np), dim3((unsigned)g.n_blocks, (unsigned)(g.split * g.chunks)),
                                         dim3(kGaThreads), args, 0, st);
  timing_end(p, st);
  if (e != cudaSuccess) return cuda_status(e, "grid adjoint launch");
  p->last_launches += 2;
  return cuda_status(cudaGetLastError(), "grid adjoint launch");
}

void release_grid_adjoint(GridAdjState& g) {
  for (void* b : {(void*)g.blocks, (void*)g.d, (void*)g.dlo, (void*)g.table, (void*)g.partial, (void*)g.gf})
    if (b) cudaFree(b);
  g = GridAdjState{};
}

}  // namespace scatter
