// Maps sampled far finer than the crystal's extent asks for: the sum at the
// Chebyshev nodes of each axis, interpolated to the map.
//
// After centring, F(s) = sum_s f_s sum_j w_j e^{2 pi i (c_j + s.x'_j)} is a sum of
// waves with |x'_d| <= X along each axis.  On an axis of half-width L the
// polynomial through n Chebyshev nodes reproduces such a wave to
//   4 sum_{k >= n} |J_k(c)|,   c = 2 pi X L
// (the tail of its Chebyshev series), which falls below 1e-6 some 20 nodes
// past c, whatever the map's step: 256 x 256 x 64 points around a reflection of a
// 20-cell sphere are resolved by 64 x 64 x 24.  The form factors vary slowly; the
// node counts are checked against them, in FP64, along lines of the map.
//
// The plan at the nodes is an ordinary one (tensor-core or factorised FP32 sum,
// as the map's own path), its accumulation groups as long as the map's own would
// be, so that its rounding is that of the direct sum.  It leaves out the
// translation phase e^{2 pi i s.t}, which would add |t| to the bandwidth; the
// last interpolation stage applies it.
//
// X is chosen at plan time: the caller's radius hint, or up to two node sets for
// 1.1 (a sphere, a cube, a slab) and 1.3 (a simple cubic cube) of a compact crystal's radius at
// four atoms per cell.  A call measures its largest |x'_d|; the smallest set that
// holds it serves, and a crystal past them is left to the direct kernels.  The
// others' launches return at once (CallGate).
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>
#include "device_common.cuh"
#include "launch.h"

namespace scatter {

namespace {

// interpolation error of one wave at |x'_d| = X (it falls a hundredfold by 0.9 X):
// FP32 sums, tensor-core sums (3e-5 by themselves)
constexpr double kCoarseEps = 5e-8, kCoarseEpsSep = 1e-6;
// Truncation in the tensor cores' accumulators shrinks a gradient by up to 1.3e-7
// per step of a group, on coherent maps.  The nodes' planes have fewer steps than
// the map's; they are taken where that moves a gradient by less than the tensor-core
// path's own scatter, 1.8e-5.
constexpr double kCoarseAdjSteps = 135.0;  // 1.8e-5 / 1.3e-7
constexpr double kCoarseMaxWeights = 1.6e7;  // nodes x points of an axis (128 MB, 0.1 s of planning)
constexpr int kIpK = 16;  // nodes per stage of the interpolation

struct InterpArgs {
  const float2* in;
  float2* out;
  const float* W;             // [n_in][n_out], and its rounding errors
  const float* W_lo;
  int64_t n_in, n_out;
  int64_t outer, inner;       // the array is [outer][n_in][inner]; a column is an (outer, inner)
  // last stage: translation phase and outputs
  int last, axis;
  const float* axis_s;        // the map's axes - H, and rounding errors
  const float* axis_lo;
  const double* axis64;       // exact64: FP64 phases, from these and H64
  double H64[3];
  int exact64;
  int planar;                 // the last axis is not interpolated: its t is in the nodes' sum
  int64_t n0, n1, n2;
  const double* shift;
  float2* out_amp;
  float* out_int;
  CallGate gate;
};

// out[o, i, b] = sum_k W[k, i] in[o, k, b], 16 T values of i x 16 T columns (o, b)
// per CTA, T x T per thread: the largest T that gives every SM two CTAs (61 x 47 x 33
// points from 39 x 34 x 27 nodes: 16, 9 and 6 us a stage with T = 4, 2 and 1).  ROWS:
// the last axis (inner = 1).  Lanes run along the
// contiguous index of the output.  Sums of 16 joined one by one in FP32; WIDE (maps
// of FP32 sums): weights and sums as double-floats, eleven operations per term
// instead of one, which leaves a map's error to its nodes (61 x 47 x 33 points
// of a 20-cell sphere against FP64: 2.8e-7, plain 3.9e-7, summed directly 3.4e-7).
template <bool ROWS, bool WIDE, int T>
__global__ void __launch_bounds__(256) k_interp(const InterpArgs a) {
  constexpr int kIpTile = 16 * T;
  __shared__ float sh_w[kIpK][kIpTile];
  __shared__ float sh_wl[WIDE ? kIpK : 1][WIDE ? kIpTile : 1];
  __shared__ float2 sh_in[kIpK][kIpTile + (ROWS ? 1 : 0)];
  using u64 = unsigned long long;
  static_assert(T == 1 || T == 2 || T == 4, "outputs and columns per thread");
  if (within(a.gate, 0)) return;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int64_t b0 = (int64_t)blockIdx.x * kIpTile, i0 = (int64_t)blockIdx.y * kIpTile;
  const int64_t cols = a.outer * a.inner;
  // loads: T weights and inputs per thread and stage of 16 nodes, the next
  // stage's on their way while this one's are used
  constexpr int kLoads = kIpK * kIpTile / 256;
  const int li = t & (kIpTile - 1), lk = t / kIpTile;         // weights; inputs unless ROWS
  const int rk = t & (kIpK - 1), rb = t / kIpK;               // inputs if ROWS
  const int64_t col = b0 + li;
  const float2* src = ROWS ? a.in + (b0 + rb) * a.n_in + rk
                           : a.in + (col / a.inner) * a.n_in * a.inner + col % a.inner + lk * a.inner;
  float w_next[kLoads], wl_next[kLoads];
  float2 in_next[kLoads];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int64_t k = k0 + lk + u * (256 / kIpTile);
      const bool ok = k < a.n_in && i0 + li < a.n_out;
      w_next[u] = ok ? a.W[k * a.n_out + i0 + li] : 0.f;
      if (WIDE) wl_next[u] = ok ? a.W_lo[k * a.n_out + i0 + li] : 0.f;
      if (ROWS)
        in_next[u] = k0 + rk < a.n_in && b0 + rb + u * (256 / kIpK) < cols ? src[u * (256 / kIpK) * a.n_in + k0]
                                                                           : make_float2(0.f, 0.f);
      else
        in_next[u] = k < a.n_in && col < cols ? src[(k - lk) * a.inner] : make_float2(0.f, 0.f);
    }
  };
  u64 sum[T][T], sum_lo[T][T];  // [contiguous][other]
#pragma unroll
  for (int p = 0; p < T; ++p)
#pragma unroll
    for (int q = 0; q < T; ++q) sum[p][q] = sum_lo[p][q] = 0ull;
  load(0);
  for (int64_t k0 = 0; k0 < a.n_in; k0 += kIpK) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      sh_w[lk + u * (256 / kIpTile)][li] = w_next[u];
      if (WIDE) sh_wl[lk + u * (256 / kIpTile)][li] = wl_next[u];
      if (ROWS)
        sh_in[rk][rb + u * (256 / kIpK)] = in_next[u];
      else
        sh_in[lk + u * (256 / kIpTile)][li] = in_next[u];
    }
    __syncthreads();
    if (k0 + kIpK < a.n_in) load(k0 + kIpK);
    u64 acc[T][T];
    if (!WIDE) {
#pragma unroll
      for (int p = 0; p < T; ++p)
#pragma unroll
        for (int q = 0; q < T; ++q) acc[p][q] = 0ull;
    }
#pragma unroll(WIDE ? 4 : kIpK)
    for (int k = 0; k < kIpK; ++k) {
      u64 w[T], wl[T], wn[T], x[T];
#pragma unroll
      for (int p = 0; p < T; ++p) {
        const float wv = sh_w[k][(ROWS ? tx : ty) + 16 * p];
        const float2 xv = sh_in[k][(ROWS ? ty : tx) + 16 * p];
        w[p] = dev::pack2(wv, wv);
        x[p] = dev::pack2(xv.x, xv.y);
        if (WIDE) {
          const float wlo = sh_wl[k][(ROWS ? tx : ty) + 16 * p];
          wl[p] = dev::pack2(wlo, wlo);
          wn[p] = dev::pack2(-wv, -wv);
        }
      }
#pragma unroll
      for (int p = 0; p < T; ++p)
#pragma unroll
        for (int q = 0; q < T; ++q) {
          const int i = ROWS ? p : q, b = ROWS ? q : p;
          if (WIDE) {
            // TwoSum of the sum and the product, both rounding errors kept
            const u64 n = dev::mul2(wn[i], x[b]), h = sum[p][q];
            const u64 e = dev::fma2(wl[i], x[b], dev::fma2(w[i], x[b], n));
            const u64 s = dev::sub2(h, n), v = dev::sub2(s, h);
            const u64 err = dev::sub2(dev::sub2(h, dev::sub2(s, v)), dev::add2(n, v));
            sum[p][q] = s;
            sum_lo[p][q] = dev::add2(sum_lo[p][q], dev::add2(err, e));
          } else {
            dev::ffma2(acc[p][q], w[i], x[b]);
          }
        }
    }
    if (!WIDE) {
#pragma unroll
      for (int p = 0; p < T; ++p)
#pragma unroll
        for (int q = 0; q < T; ++q) sum[p][q] = dev::add2(sum[p][q], acc[p][q]);
    }
  }
  if (WIDE) {
#pragma unroll
    for (int p = 0; p < T; ++p)
#pragma unroll
      for (int q = 0; q < T; ++q) sum[p][q] = dev::add2(sum[p][q], sum_lo[p][q]);
  }
  const bool shifted = a.last && (a.shift[0] != 0.0 || a.shift[1] != 0.0 || a.shift[2] != 0.0);
  const float ts[3] = {shifted ? (float)a.shift[0] : 0.f, shifted ? (float)a.shift[1] : 0.f,
                       shifted && !a.planar ? (float)a.shift[2] : 0.f};
#pragma unroll
  for (int c = 0; c < T; ++c) {  // this thread's columns
    const int64_t b = b0 + (ROWS ? ty : tx) + 16 * c;
    if (b >= cols) continue;
    const int64_t o = ROWS ? b : b / a.inner, r = ROWS ? 0 : b % a.inner;
    // the column's place in the map, its axis' own index left out
    int64_t at[3] = {0, 0, 0};
    if (shifted) {
      at[0] = a.axis == 0 ? 0 : a.axis == 1 ? o : o / a.n1;
      at[1] = a.axis == 0 ? r / a.n2 : a.axis == 1 ? 0 : o % a.n1;
      at[2] = a.axis == 0 ? r % a.n2 : r;
    }
#pragma unroll
    for (int e = 0; e < T; ++e) {  // its outputs
      const int64_t i = i0 + (ROWS ? tx : ty) + 16 * e;
      if (i >= a.n_out) continue;
      const int64_t m = (o * a.n_out + i) * a.inner + r;
      float2 v;
      dev::unpack2(ROWS ? sum[e][c] : sum[c][e], v.x, v.y);
      if (!a.last) {
        a.out[m] = v;
        continue;
      }
      if (shifted) {
        const int64_t x0 = at[0] + (a.axis == 0 ? i : 0), x1 = a.n0 + at[1] + (a.axis == 1 ? i : 0),
                      x2 = a.n0 + a.n1 + at[2] + (a.axis == 2 ? i : 0);
        float2 ph;
        if (a.exact64) {
          ph = dev::shift_phase(a.axis64[x0] - a.H64[0], a.axis64[x1] - a.H64[1], a.axis64[x2] - a.H64[2], a.shift);
        } else {
          const float hi[3] = {a.axis_s[x0], a.axis_s[x1], a.axis_s[x2]};
          const float lo[3] = {a.axis_lo[x0], a.axis_lo[x1], a.axis_lo[x2]};
          ph = dev::shift_phase2(hi, lo, ts);
        }
        v = dev::cmul(ph, v);
      }
      if (a.out_amp) a.out_amp[m] = v;
      if (a.out_int) a.out_int[m] = v.x * v.x + v.y * v.y;
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

// 4 sum_{k >= n} |J_k(c)| for every n <= n_max (Miller's downward recurrence,
// normalised by J_0 + 2 (J_2 + J_4 + ...) = 1).
std::vector<double> chebyshev_tails(double c, int n_max) {
  const int top = 2 * ((int)std::max((double)n_max, c) / 2 + 40 + (int)std::cbrt(40000.0 * (c + 1.0)) / 2);
  std::vector<double> J(top + 2, 0.0);
  J[top] = 1e-250;
  double norm = 0.0;
  for (int k = top; k > 0; --k) {
    J[k - 1] = 2.0 * k / std::max(c, 1e-12) * J[k] - J[k + 1];
    if (std::fabs(J[k - 1]) > 1e200) {
      for (int i = k - 1; i <= top; ++i) J[i] *= 1e-250;
      norm *= 1e-250;
    }
    if ((k - 1) % 2 == 0) norm += (k - 1 ? 2.0 : 1.0) * J[k - 1];
  }
  std::vector<double> tail(n_max + 1);
  double s = 0.0;
  for (int k = top; k >= 0; --k) {
    s += 4.0 * std::fabs(J[k] / norm);
    if (k <= n_max) tail[k] = s;
  }
  return tail;
}

struct Nodes {
  std::vector<double> x, w;  // ascending nodes, barycentric weights
};
Nodes chebyshev_nodes(double lo, double hi, int n) {
  const double pi = 3.14159265358979323846, mid = 0.5 * (lo + hi), half = 0.5 * (hi - lo);
  Nodes r;
  for (int i = 0; i < n; ++i) {
    const double th = (i + 0.5) * pi / n;
    // symmetric about the middle to the last place: sin of the angle from it
    r.x.push_back(mid + half * std::sin(0.5 * pi * (2.0 * i + 1.0 - n) / n));
    r.w.push_back((i % 2 ? -1.0 : 1.0) * std::sin(th));
  }
  return r;
}

// Interpolation weights of the nodes at x.
void weights_at(const Nodes& nd, double x, double* w) {
  const int n = (int)nd.x.size();
  double sum = 0.0;
  for (int k = 0; k < n; ++k) {
    const double d = x - nd.x[k];
    if (d == 0.0) {
      for (int j = 0; j < n; ++j) w[j] = j == k ? 1.0 : 0.0;
      return;
    }
    sum += w[k] = nd.w[k] / d;
  }
  for (int k = 0; k < n; ++k) w[k] /= sum;
}

double form_modulus(const double* cf, double s2) {
  double f0 = cf[8];
  for (int i = 0; i < 4; ++i) f0 += cf[i] * std::exp(-cf[4 + i] * s2);
  return (f0 + cf[9]) * std::exp(-cf[11] * s2);
}

// Largest error of interpolating f_s(|S|) e^{i c u} along axis d at up to 48 of
// its points, against the largest |f_s| there, over the map's middle and ends
// of the other axes and every species.
double form_error(const scatter_plan_s* p, int d, const Nodes& nd, double X) {
  const double inv4a2 = 1.0 / (4.0 * p->lattice_a * p->lattice_a), two_pi = 6.283185307179586;
  const std::vector<double>& ax = p->axis_host[d];
  const int n = (int)nd.x.size(), o1 = (d + 1) % 3, o2 = (d + 2) % 3;
  const int64_t step = std::max<int64_t>(1, (int64_t)ax.size() / 48);
  auto pick = [&](int axis, int which) {
    const std::vector<double>& v = p->axis_host[axis];
    if (p->s_kind == SCATTER_S_GID_GRID && axis == 2) return 0.0;  // small S_z
    return which == 0 ? v.front() : which == 1 ? v[v.size() / 2] : v.back();
  };
  std::vector<double> w(n);
  double worst = 0.0;
  for (int s = 0; s < p->n_species; ++s) {
    const double* cf = p->coef_host.data() + kNCoef * s;
    for (int q = 0; q < 9; ++q) {
      const double a = pick(o1, q / 3), b = pick(o2, q % 3), rest = a * a + b * b;
      double top = 0.0, err = 0.0;
      std::vector<double> re(n), im(n);
      for (int k = 0; k < n; ++k) {
        const double f = form_modulus(cf, (nd.x[k] * nd.x[k] + rest) * inv4a2), ph = two_pi * X * (nd.x[k] - nd.x[0]);
        re[k] = f * std::cos(ph);
        im[k] = f * std::sin(ph);
        top = std::max(top, std::fabs(f));
      }
      for (int64_t i = 0; i < (int64_t)ax.size(); i += step) {
        weights_at(nd, ax[i], w.data());
        const double f = form_modulus(cf, (ax[i] * ax[i] + rest) * inv4a2), ph = two_pi * X * (ax[i] - nd.x[0]);
        double dr = -f * std::cos(ph), di = -f * std::sin(ph);
        for (int k = 0; k < n; ++k) {
          dr += w[k] * re[k];
          di += w[k] * im[k];
        }
        err = std::max(err, std::hypot(dr, di));
      }
      if (top > 0.0) worst = std::max(worst, err / top);
    }
  }
  return worst;
}

}  // namespace

namespace {

void launch_stage(scatter_plan_t p, const InterpArgs& a, cudaStream_t st) {
  auto tiles = [&](int64_t tile) {
    return dim3((unsigned)((a.outer * a.inner + tile - 1) / tile), (unsigned)((a.n_out + tile - 1) / tile));
  };
  // the largest tiles that still give every SM two CTAs
  int T = 4;
  while (T > 1 && (int64_t)tiles(16 * T).x * tiles(16 * T).y < 2 * p->n_sm) T /= 2;
  const dim3 grid = tiles(16 * T);
  const bool wide = p->path != SCATTER_PATH_SEPARABLE, rows = a.inner == 1 && a.axis == 2;
  auto pick = [&](auto t) {
    constexpr int kT = decltype(t)::value;
    return wide ? (rows ? k_interp<true, true, kT> : k_interp<false, true, kT>)
                : (rows ? k_interp<true, false, kT> : k_interp<false, false, kT>);
  };
  const auto kernel = T == 4   ? pick(std::integral_constant<int, 4>{})
                      : T == 2 ? pick(std::integral_constant<int, 2>{})
                               : pick(std::integral_constant<int, 1>{});
  kernel<<<grid, 256, 0, st>>>(a);
}

// The nodes' weight table of the FP32 adjoint: rows {s, gF.re | S, gF.im}, for the
// line form (s_z, S_z, gF).
__global__ void __launch_bounds__(256) k_node_table(const float2* __restrict__ gf, const float* __restrict__ axis_s,
                                                    int64_t n0, int64_t n1, int64_t n2, float3 H, int64_t total,
                                                    int line_form, float4* __restrict__ table, const CallGate gate) {
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= total || within(gate, 0)) return;
  const int64_t m = e % (n0 * n1 * n2), i2 = m % n2, line = m / n2;
  const float sx = axis_s[line / n1], sy = axis_s[n0 + line % n1], sz = axis_s[n0 + n1 + i2];
  const float2 g = gf[e];
  if (line_form) {
    table[e] = make_float4(sz, H.z + sz, g.x, g.y);
    return;
  }
  table[2 * e] = make_float4(sx, sy, sz, g.x);
  table[2 * e + 1] = make_float4(H.x + sx, H.y + sy, H.z + sz, g.y);
}

}  // namespace

namespace {

// Nodes that resolve crystals with |x'_d| <= X on the map's axes.
struct NodeSet {
  double X = 0.0, seconds = 1e300;  // by the model
  std::vector<double> axis[3];      // nodes, or the axis' own points
  Nodes nd[3];
};

// Time of a sum at n0 x n12 points on the plan's path.  FP32: pairs per second.
// Tensor cores: 1 us (up to 64 mirror pairs 0.75 us) per step of 32 atoms and tile
// of 64 lanes x 128 mirror pairs, in chunks of at least some 200 steps.
double sum_seconds(const scatter_plan_s* p, double n0, double n12) {
  const double N = (double)p->n_slots;
  if (p->path != SCATTER_PATH_SEPARABLE) return N * n0 * n12 / 1.0e13;
  double tiles = std::ceil(n0 / 128.0) * std::ceil(n12 / 256.0), steps = N / 32.0;
  if (p->s_kind == SCATTER_S_GID_GRID) {  // four beams, the direct form: 16 atoms, 128 values x 256 columns
    tiles = std::ceil(n0 / 128.0) * std::ceil(4.0 * n12 / 256.0);
    steps = N / 16.0;
  }
  double best = 1e300;
  for (double k = 1.0; k <= std::max(1.0, steps / 200.0); k += 1.0)
    best = std::min(best, std::ceil(tiles * k / p->n_sm) * (steps / k + 40.0) * (n12 <= 128.0 ? 0.75e-6 : 1e-6));
  return best;
}

NodeSet choose_nodes(const scatter_plan_s* p, double X) {
  NodeSet r;
  r.X = X;
  const bool sep = p->path == SCATTER_PATH_SEPARABLE;
  const double eps = sep ? kCoarseEpsSep : kCoarseEps;
  bool any = false;
  double M = 1.0;
  const bool gid = p->s_kind == SCATTER_S_GID_GRID;
  for (int d = 0; d < 3; ++d) {
    const std::vector<double>& ax = p->axis_host[d];
    if (gid && d == 2) {  // exit angles: four beams each, not a wave per atom
      r.axis[d] = ax;
      M *= (double)ax.size();
      continue;
    }
    const double lo = *std::min_element(ax.begin(), ax.end()), hi = *std::max_element(ax.begin(), ax.end());
    const int most = (int)std::min<int64_t>(4096, (int64_t)(0.9 * (double)ax.size()));
    int n = 0;
    if (hi > lo && most >= 8) {
      const double c = 3.14159265358979323846 * X * (hi - lo);
      if (c < (double)most) {
        const std::vector<double> tail = chebyshev_tails(c, most);
        for (n = 4; n <= most && tail[n] > eps;) ++n;
        for (; n <= most; n += 2)
          if (form_error(p, d, r.nd[d] = chebyshev_nodes(lo, hi, n), X) < 2.0 * eps) break;
        if (n > most || (double)n * (double)ax.size() > kCoarseMaxWeights) n = 0;
      }
    }
    any = any || n > 0;
    r.axis[d] = n > 0 ? r.nd[d].x : ax;
    M *= (double)ax.size();
  }
  const double sum = sum_seconds(p, r.axis[0].size(), (double)r.axis[1].size() * (double)r.axis[2].size());
  if (any) r.seconds = sum + 60e-6 + M * 30.0 / 4.0e12;
  return r;
}

bool build_level(scatter_plan_s* p, const scatter_problem* pr, const scatter_options* op, const NodeSet& set);
void release_level(scatter_plan_s* p, CoarseState& c);

}  // namespace

scatter_status prepare_coarse(scatter_plan_s* p, const scatter_problem* pr, const scatter_options* op) {
  const bool sep = p->path == SCATTER_PATH_SEPARABLE, gid = p->s_kind == SCATTER_S_GID_GRID;
  if (!(p->s_kind == SCATTER_S_GRID || (gid && sep && p->gid_mode == 0)) || p->batch != 1 || pr->factor_table ||
      p->n_atoms <= 0 || p->n_s <= 0)
    return SCATTER_OK;
  if (!sep && !(p->path == SCATTER_PATH_GENERIC && p->gs.active)) return SCATTER_OK;
  if (op && (op->threads || op->points_per_thread || op->split_k || op->atoms_per_thread > 0)) return SCATTER_OK;
  for (int d = 0; d < 3; ++d)
    if (p->n_axis[d] > 4000000) return SCATTER_OK;
  // taken where the time saved by the model is worth the extra launches; two sets
  // where the tighter one saves some more (20 us of launches that return at once:
  // 35,802 against 24,600 nodes of 61 x 47 x 33 points: 567 against 436 us)
  const double fine = sum_seconds(p, (double)p->n_axis[0], (double)p->n_axis[1] * (double)p->n_axis[2]);
  const double compact = std::cbrt(3.0 * (double)p->n_atoms / (16.0 * 3.14159265358979323846));
  std::vector<NodeSet> sets;
  if (op && op->radius_hint > 0.0) {
    sets.push_back(choose_nodes(p, op->radius_hint));
  } else {
    // (flat islands reach further sideways: 1.6 and 2.3)
    sets.push_back(choose_nodes(p, (gid ? 1.6 : 1.1) * compact + 1.0));
    sets.push_back(choose_nodes(p, (gid ? 2.3 : 1.3) * compact + 1.0));
    if (sets[1].seconds <= 0.75 * fine && sets[0].seconds + 40e-6 > sets[1].seconds) sets.erase(sets.begin());
  }
  for (const NodeSet& set : sets)
    if (set.seconds <= 0.75 * fine && !build_level(p, pr, op, set)) break;
  return SCATTER_OK;
}

namespace {

bool build_level(scatter_plan_s* p, const scatter_problem* pr, const scatter_options* op, const NodeSet& set) {
  const bool sep = p->path == SCATTER_PATH_SEPARABLE;
  const std::vector<double>* nodes = set.axis;
  const Nodes* nd = set.nd;
  scatter_problem q = *pr;
  scatter_options o{};
  if (op) o = *op;
  o.path = p->path;
  o.autotune = 0;
  o.tune_cache = nullptr;
  o.timing = 0;
  o.use_graph = -1;
  for (int d = 0; d < 3; ++d) {
    q.axis[d] = nodes[d].data();
    q.n_axis[d] = (int64_t)nodes[d].size();
  }
  CoarseState& c = p->coarse[p->coarse_levels];
  const double H[3] = {p->inst[0].H[0], p->inst[0].H[1], p->inst[0].H[2]};
  bool ok = plan_nodes(&q, &o, H, sep ? 0.9 * sep_direct_group(p) : 0.0, &c.sub) == SCATTER_OK && (sep || c.sub->gs.active);
  // stages in the order that costs the least
  int order[3] = {0, 1, 2}, best[3] = {0, 1, 2};
  double best_cost = 1e300;
  do {
    double n[3] = {(double)nodes[0].size(), (double)nodes[1].size(), (double)nodes[2].size()}, cost = 0.0;
    for (int d : order) {
      const double in = n[d];
      n[d] = (double)p->n_axis[d];
      if (!nd[d].x.empty() && in != n[d]) cost += n[0] * n[1] * n[2] * (in + 24.0);
    }
    if (cost < best_cost) {
      best_cost = cost;
      std::copy(order, order + 3, best);
    }
  } while (std::next_permutation(order, order + 3));
  int64_t n[3] = {(int64_t)nodes[0].size(), (int64_t)nodes[1].size(), (int64_t)nodes[2].size()};
  int64_t tmp[2] = {0, 0}, bytes = 0;
  auto alloc = [&](void* ptr, size_t size) {
    bytes += (int64_t)size;
    return cudaMalloc(static_cast<void**>(ptr), std::max<size_t>(size, 16)) == cudaSuccess;
  };
  for (int d : best) {
    if (nodes[d].size() == (size_t)p->n_axis[d] || !ok) continue;
    CoarseStage& s = c.stage[c.n_stages];
    s.axis = d;
    s.n_in = n[d];
    s.n_out = p->n_axis[d];
    s.outer = d == 0 ? 1 : d == 1 ? n[0] : n[0] * n[1];
    s.inner = d == 0 ? n[1] * n[2] : d == 1 ? n[2] : 1;
    n[d] = s.n_out;
    if (c.n_stages < 2) tmp[c.n_stages] = n[0] * n[1] * n[2];
    std::vector<double> w(s.n_in);
    std::vector<float> W(2 * (size_t)(s.n_in * s.n_out));  // and rounding errors
    for (int64_t i = 0; i < s.n_out; ++i) {
      weights_at(nd[d], p->axis_host[d][i], w.data());
      for (int64_t k = 0; k < s.n_in; ++k) {
        const float h = (float)w[k];
        W[(size_t)(k * s.n_out + i)] = h;
        W[(size_t)((s.n_in + k) * s.n_out + i)] = (float)(w[k] - (double)h);
      }
    }
    ok = alloc(&s.W, W.size() * sizeof(float)) &&
         cudaMemcpy(s.W, W.data(), W.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
    s.h_W = std::move(W);
    ++c.n_stages;
  }
  const float lim2 = (float)(set.X * set.X);
  ok = ok && alloc(&c.map, (size_t)c.sub->n_s * sizeof(float2)) && alloc(&c.lim2, sizeof(float)) &&
       (p->coarse_rmax2 || (alloc(&p->coarse_rmax2, sizeof(unsigned)) && alloc(&p->coarse_shift, 3 * sizeof(double)) &&
                            cudaMemset(p->coarse_rmax2, 0, sizeof(unsigned)) == cudaSuccess &&
                            cudaMemset(p->coarse_shift, 0, 3 * sizeof(double)) == cudaSuccess)) &&
       cudaMemcpy(c.lim2, &lim2, sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
  for (int i = 0; i < c.n_stages - 1; ++i) ok = ok && alloc(&c.tmp[i], (size_t)tmp[i] * sizeof(float2));
  if (!ok) {  // no room: the direct kernels need none of it
    cudaGetLastError();
    release_level(p, c);
    return false;
  }
  // the call's status word and shift are the map's own
  cudaFree(c.sub->d.status);
  cudaFree(c.sub->d.inst_shift);
  c.sub->d.status = p->d.status;
  c.sub->d.inst_shift = p->d.inst_shift;
  c.sub->extent2 = p->coarse_levels == 0 ? p->coarse_rmax2 : nullptr;  // measured once
  c.sub->out_shift = p->coarse_shift;
  c.X = set.X;
  p->base_bytes += bytes + c.sub->base_bytes + c.sub->tiling_bytes;
  ++p->coarse_levels;
  return true;
}

}  // namespace

void coarse_error(const scatter_plan_s* p, double radius, double* truncation, double* rounding, double* amplify) {
  *truncation = *rounding = 0.0;
  *amplify = 1.0;
  const double u = std::ldexp(1.0, -24);
  for (int l = 0; l < p->coarse_levels; ++l) {
    const CoarseState& c = p->coarse[l];
    const double X = std::min(radius, c.X);
    // Lebesgue constants: 2/pi ln n + 1 bounds those of n Chebyshev nodes
    double product = 1.0;
    auto lebesgue = [](double n) { return 0.63661977236758134 * std::log(n) + 1.0; };
    for (int i = 0; i < c.n_stages; ++i) product *= lebesgue((double)c.stage[i].n_in);
    // A wave has |x'| <= X in all: past 0.9 X along one axis it stays within 0.44 X along
    // the others, whose tails are then nothing.
    double one = 0.0, near = 0.0, round = 0.0;
    for (int i = 0; i < c.n_stages; ++i) {
      const CoarseStage& s = c.stage[i];
      const std::vector<double>& ax = p->axis_host[s.axis];
      const double lo = *std::min_element(ax.begin(), ax.end()), hi = *std::max_element(ax.begin(), ax.end());
      const int n = (int)s.n_in;
      const double others = product / lebesgue((double)n), c1 = 3.14159265358979323846 * X * (hi - lo);
      // waves, and waves times form factors
      const double form = form_error(p, s.axis, chebyshev_nodes(lo, hi, n), X);
      one = std::max(one, others * (chebyshev_tails(c1, n)[n] + form));
      near += others * (chebyshev_tails(0.9 * c1, n)[n] + form);
      // WIDE: double-float weights and sums; else n products in sums of 16
      round += product * u * (p->path == SCATTER_PATH_SEPARABLE ? 18.0 + (double)n / 16.0 : 1.0);
    }
    *truncation = std::max(*truncation, one + near);
    *rounding = std::max(*rounding, round);
    *amplify = std::max(*amplify, product);
  }
}

scatter_status launch_coarse_prep(scatter_plan_t p, int levels, const double* xyz, const float* occ, cudaStream_t st) {
  for (int l = 0; l < levels; ++l) {
    scatter_plan_s* sub = p->coarse[l].sub;
    sub->last_launches = 0;
    if (const scatter_status s = launch_prep(sub, xyz, occ, st, coarse_gate(p, l)); s != SCATTER_OK) return s;
    p->last_launches += sub->last_launches;
  }
  return SCATTER_OK;
}

scatter_status launch_coarse(scatter_plan_t p, const double* xyz, const float* occ, float2* amp_out, float* int_out,
                             cudaStream_t st) {
  timing_begin(p, st);  // to the end of the direct kernel, which may do the work instead
  scatter_status s = launch_coarse_prep(p, p->coarse_levels, xyz, occ, st);
  for (int l = 0; l < p->coarse_levels && s == SCATTER_OK; ++l) {
    const CoarseState& c = p->coarse[l];
    const CallGate gate = level_gate(p, l);
    c.sub->last_launches = 0;
    s = p->path == SCATTER_PATH_SEPARABLE ? launch_separable(c.sub, c.map, nullptr, st, gate)
                                          : launch_generic(c.sub, c.map, nullptr, st, gate);
    p->last_launches += c.sub->last_launches;
    InterpArgs a{};
    a.axis_s = p->d.axis_s;
    a.axis_lo = p->d.axis_lo;
    a.axis64 = p->d.axis64;
    for (int d = 0; d < 3; ++d) a.H64[d] = p->inst[0].H[d];
    a.exact64 = p->path != SCATTER_PATH_SEPARABLE;
    a.planar = p->s_kind == SCATTER_S_GID_GRID;
    a.n0 = p->n_axis[0];
    a.n1 = p->n_axis[1];
    a.n2 = p->n_axis[2];
    a.shift = p->d.inst_shift;
    a.out_amp = amp_out;
    a.out_int = int_out;
    a.gate = gate;
    const float2* in = c.map;
    for (int i = 0; i < c.n_stages; ++i) {
      const CoarseStage& g = c.stage[i];
      a.in = in;
      a.last = i + 1 == c.n_stages;
      a.out = a.last ? nullptr : c.tmp[i];
      a.W = g.W;
      a.W_lo = g.W + g.n_in * g.n_out;
      a.n_in = g.n_in;
      a.n_out = g.n_out;
      a.outer = g.outer;
      a.inner = g.inner;
      a.axis = g.axis;
      launch_stage(p, a, st);
      in = a.out;
      p->last_launches += 1;
    }
  }
  return s != SCATTER_OK ? s : cuda_status(cudaGetLastError(), "interpolation launch");
}

// S_d e^{2 pi i S.r} is interpolated from the nodes as the wave itself is, so the
// gradient is the nodes' own adjoint with the weights sum_S l_node(S) gF(S): the
// interpolation's transpose, stage by stage in reverse.
scatter_status prepare_coarse_adjoint(scatter_plan_s* p) {
  const bool sep = p->adj_sep;
  const int l = p->coarse_adj_levels;
  if (l >= p->coarse_levels) return SCATTER_OK;
  CoarseState& c = p->coarse[l];
  if (!sep && p->path == SCATTER_PATH_SEPARABLE) return SCATTER_OK;
  // pairs per second: tensor cores 5e13 (fewer points 4e13), FP32 lanes at 2 GHz
  const double lanes = 128.0 * p->n_sm * 2.0e9;
  const double pairs = (double)p->n_slots;
  const double fine = pairs * (double)p->n_s / (sep ? 5.0e13 : lanes / grid_adjoint_ops(p));
  bool fold = true;
  if (sep) {
    const double least = adjoint_sep_group(p, false) - kCoarseAdjSteps;
    fold = adjoint_sep_group(c.sub, true) >= least;
    if (!fold && adjoint_sep_group(c.sub, false) < least) return SCATTER_OK;
  }
  const double few = pairs * (double)c.sub->n_s / (!sep ? lanes / grid_adjoint_ops(c.sub) : fold ? 4.0e13 : 2.0e13) + 60e-6 +
                     (double)p->n_s * p->n_species * 30.0 / 4.0e12;
  if (few > 0.75 * fine) return SCATTER_OK;  // nor any larger set
  c.sub->adj_no_fold = !fold;
  const int64_t before = c.sub->base_bytes;
  if (prepare_adjoint(c.sub) != SCATTER_OK || c.sub->adj_sep != sep) return SCATTER_OK;
  int64_t bytes = c.sub->base_bytes - before;
  auto alloc = [&](void* ptr, size_t size) {
    bytes += (int64_t)size;
    return cudaMalloc(static_cast<void**>(ptr), std::max<size_t>(size, 16)) == cudaSuccess;
  };
  bool ok = true;
  for (int i = 0; i < c.n_stages && ok; ++i) {
    CoarseStage& s = c.stage[i];
    std::vector<float> T(s.h_W.size());
    const size_t n = (size_t)(s.n_in * s.n_out);
    for (int part = 0; part < 2; ++part)
      for (int64_t k = 0; k < s.n_in; ++k)
        for (int64_t j = 0; j < s.n_out; ++j) T[part * n + j * s.n_in + k] = s.h_W[part * n + k * s.n_out + j];
    ok = alloc(&s.Wt, T.size() * sizeof(float)) &&
         cudaMemcpy(s.Wt, T.data(), T.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
    // stage i leaves the input of the forward's stage i
    const size_t out = (size_t)p->n_species * (size_t)(s.outer * s.n_in * s.inner) * sizeof(float2);
    if (i > 0 && ok) ok = alloc(&c.adj_tmp[i - 1], out);
    if (i == 0 && ok && !sep) ok = alloc(&c.adj_gf, out);
  }
  if (!ok) {
    cudaGetLastError();
    return SCATTER_OK;  // what was allocated goes with the plan
  }
  p->base_bytes += bytes;
  ++p->coarse_adj_levels;
  return prepare_coarse_adjoint(p);  // the next set
}

namespace {

scatter_status level_adjoint(scatter_plan_t p, int l, const float2* gf, float* grad, cudaStream_t st) {
  const CoarseState& c = p->coarse[l];
  scatter_plan_s* sub = c.sub;
  InterpArgs a{};
  a.gate = level_gate(p, l);
  a.shift = p->d.inst_shift;
  const float2* in = gf;
  for (int i = c.n_stages - 1; i >= 0; --i) {
    const CoarseStage& g = c.stage[i];
    a.in = in;
    a.out = i > 0 ? c.adj_tmp[i - 1] : p->adj_sep ? sub->d.adj_gf : c.adj_gf;
    a.W = g.Wt;
    a.W_lo = g.Wt + g.n_in * g.n_out;
    a.n_in = g.n_out;
    a.n_out = g.n_in;
    a.outer = p->n_species * g.outer;
    a.inner = g.inner;
    a.axis = g.axis;
    launch_stage(p, a, st);
    in = a.out;
    p->last_launches += 1;
  }
  sub->last_launches = 0;
  scatter_status s;
  if (p->adj_sep) {
    s = launch_adjoint_sep(sub, grad, st, a.gate);
  } else if (sub->ga.active) {
    s = launch_adjoint_rows(sub, in, grad, st, a.gate);
  } else {
    const int64_t total = (int64_t)p->n_species * sub->n_s;
    k_node_table<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(
        in, sub->d.axis_s, sub->n_axis[0], sub->n_axis[1], sub->n_axis[2],
        make_float3((float)p->inst[0].H[0], (float)p->inst[0].H[1], (float)p->inst[0].H[2]), total, sub->adj_line,
        sub->d.adj_table, a.gate);
    p->last_launches += 1;
    s = launch_adjoint_tiles(sub, grad, st, a.gate);
  }
  p->last_launches += sub->last_launches;
  return s;
}

}  // namespace

scatter_status launch_coarse_adjoint(scatter_plan_t p, const float2* gf, float* grad, cudaStream_t st) {
  scatter_status s = SCATTER_OK;
  for (int l = 0; l < p->coarse_adj_levels && s == SCATTER_OK; ++l) s = level_adjoint(p, l, gf, grad, st);
  return s;
}

namespace {

void release_level(scatter_plan_s* p, CoarseState& c) {
  if (c.sub) {
    if (c.sub->d.status == p->d.status) c.sub->d.status = nullptr;
    if (c.sub->d.inst_shift == p->d.inst_shift) c.sub->d.inst_shift = nullptr;
    scatter_plan_destroy(c.sub);
  }
  for (CoarseStage& s : c.stage)
    for (float* w : {s.W, s.Wt})
      if (w) cudaFree(w);
  for (void* b : {(void*)c.adj_tmp[0], (void*)c.adj_tmp[1], (void*)c.adj_gf, (void*)c.map, (void*)c.tmp[0], (void*)c.tmp[1], (void*)c.lim2})
    if (b) cudaFree(b);
  c = CoarseState{};
}

}  // namespace

void release_coarse(scatter_plan_s* p) {
  for (CoarseState& c : p->coarse) release_level(p, c);
  for (void* b : {(void*)p->coarse_rmax2, (void*)p->coarse_shift})
    if (b) cudaFree(b);
  p->coarse_rmax2 = nullptr;
  p->coarse_shift = nullptr;
  p->coarse_levels = p->coarse_adj_levels = 0;
}

}  // namespace scatter
