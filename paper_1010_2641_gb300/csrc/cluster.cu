// S lists whose points lie close together (detector patches, Ewald-sphere
// slices): the sum over the atoms once per cluster of points, not per point.
//
// The points of an instance are grouped at plan time into clusters with
// centres s_k and offsets d_m = s_m - s_k.  With x'_j = X xh_j, |xh_j| <= 1,
// and th_m = 2 pi X d_m (a radian or two at the cluster's corners)
//   e^{2 pi i s_m.x'_j} = e^{2 pi i s_k.x'_j} sum_a i^|a| th_m^a (xh_j^a / a!)
// over multi-indices a in a frame of the points' principal axes (a patch is
// flat: the third axis needs one or two orders).  So
//   M_s[k, a] = sum_{j in s} w_j e^{2 pi i (c_j + s_k.x'_j)} xh_j^a / a!    (moments)
//   T_s(S_m)  = sum_a i^|a| th_m^a M_s[k, a]                                 (evaluation)
// and a (cluster, atom) costs one sincos and two multiply-adds per column a
// instead of a phase, a sincos and two multiply-adds per (point, atom).  The
// columns are those whose largest term over the ball |xh| <= 1 exceeds
// kClEps; the neglected ones come to ~4e-8 of a map (rounding: 2e-7), to 1.2e-5 of a
// term at the ball's surface and a cluster's corner.
//
// X is chosen at plan time, 1.45 of a compact crystal's radius (a cube's
// corners) or the caller's radius hint.  A call measures its atoms' largest
// |x'|: columns that a smaller crystal does not need are skipped (they are
// sorted by the radius from which they matter), and a larger crystal is left
// to the direct kernels, whose launches otherwise return at once (CallGate).
//
//   k_cl_tab     per slot: w xh^a / a! for every column
//   k_cl_moments 64 clusters x 16 columns x one chunk of atoms of one species
//   k_cl_reduce  chunks summed in order per species, times i^|a|
//   k_cl_eval    per point: the columns' sum, f_s(|S|), translation phase
// FP32 throughout, sums blocked by chunks of at most 256 atoms.
// 134,009 atoms x 60,001 points of a detector patch (128 clusters, 97 of 147
// columns in use): 0.25-0.27 ms per call, by how the patch falls into clusters, against
// 3.72 ms; relative error against FP64 1.9e-7 against 2.0e-7.
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>
#include "cluster_common.cuh"
#include "device_common.cuh"
#include "launch.h"

namespace scatter {

constexpr int kClCols = 16;       // columns per thread of the moments kernel
constexpr int kClRows = 64;       // clusters per CTA (one per thread)
constexpr int kClTile = 64;       // atoms per stage
constexpr int kClEval = 64;       // points per CTA of the evaluation
constexpr int64_t kClMaxBytes = 4LL << 30;  // workspace of a plan's clusters

namespace {

// w xh^a / a! of every column of 128 slots: a thread per slot takes the powers of its
// three coordinates, then a thread per four columns of a slot writes 16 bytes
// next to its neighbour's (a thread per slot and all its columns wrote 64-byte
// strides: 25 us on the 134,009-atom sphere, 17 us so).
__global__ void __launch_bounds__(128) k_cl_tab(const ClArgs a) {
  __shared__ float sh_p[3][kClMaxExp + 1][128 + 4];
  __shared__ int sh_e[kClMaxK];
  const ClTabBlock b = a.tab_blocks[blockIdx.x];
  const ClInst in = a.inst[b.inst];
  const int K = cl_columns(a, in, b.inst);
  const int t = threadIdx.x;
  if (K == 0) return;
  const int n = (int)dev::min64(128, in.n_slots - b.slot);
  for (int c = t; c < K; c += 128) sh_e[c] = a.exps[in.col0 + c];
  if (t < n) {
    const float4 at = a.atom4[in.slot_begin + b.slot + t];
    const float w = a.atom_w[in.slot_begin + b.slot + t];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float x = in.R[3 * d] * at.x + in.R[3 * d + 1] * at.y + in.R[3 * d + 2] * at.z;
      float p = d == 0 ? w : 1.f;
#pragma unroll
      for (int e = 0; e <= kClMaxExp; ++e) {
        sh_p[d][e][t] = p;  // x^e / e!
        p *= x * (1.0f / (float)(e + 1));
      }
    }
  }
  __syncthreads();
  constexpr int kQ = kClCols / 4;
  for (int i = t; i < n * kQ; i += 128) {
    const int s = i / kQ, q = i % kQ;
    float4* out = reinterpret_cast<float4*>(a.tab + in.tab_off + (b.slot + s) * kClCols) + q;
    for (int c0 = 0; c0 < K; c0 += kClCols, out += in.n_slots * kQ) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + 4 * q + u;
        const int e = sh_e[min(c, K - 1)];
        v[u] = c < K ? sh_p[0][e & 15][s] * (sh_p[1][(e >> 4) & 15][s] * sh_p[2][(e >> 8) & 15][s]) : 0.f;
      }
      *out = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

// Moments of 64 clusters (one per thread) x 16 columns over one chunk: the
// chunk's atoms and table rows come in by bulk copies, two stages; E =
// e^{2 pi i (c + s_k.x')} once per (cluster, atom), the columns in packed pairs
// (re of two columns, im of two columns).  Bound by issue: 14 clocks of an SM per
// (warp of clusters, atom).  32 columns per thread share the sincos among more,
// but leave half of the warps and more idle columns: 0.43 ms against 0.35 ms on
// the patch above at 296 clusters of 90 columns.
__global__ void __launch_bounds__(kClRows) k_cl_moments(const ClArgs a) {
  __shared__ __align__(128) float4 sh_at[2][kClTile];
  __shared__ __align__(128) float sh_m[2][kClTile][kClCols];
  __shared__ __align__(8) uint64_t sh_bar[2];
  using u64 = unsigned long long;
  const ClItem it = a.items[blockIdx.x];
  const ClInst in = a.inst[it.inst];
  const int K = cl_columns(a, in, it.inst);
  if (it.col_tile * kClCols >= K) return;
  const int tid = threadIdx.x;
  const int row = it.row0 + tid;
  const bool ok_row = row < in.rows;
  const int64_t rg = in.row0 + (ok_row ? row : 0);
  const float sx = a.cen[rg], sy = a.cen[a.n_rows + rg], sz = a.cen[2 * a.n_rows + rg];
  if (tid == 0) {
    dev::mbar_init(&sh_bar[0], 1);
    dev::mbar_init(&sh_bar[1], 1);
    dev::mbar_fence_init();
  }
  __syncthreads();
  const float* tab = a.tab + in.tab_off + (int64_t)it.col_tile * in.n_slots * kClCols;
  auto issue = [&](int64_t b, int st) {
    if (b >= it.end) return;
    const uint32_t cnt = (uint32_t)dev::min64(kClTile, it.end - b);
    dev::mbar_arrive_expect_tx(&sh_bar[st], cnt * (16u + 4u * kClCols));
    dev::bulk_g2s(&sh_at[st][0], a.atom4 + in.slot_begin + b, cnt * 16u, &sh_bar[st]);
    dev::bulk_g2s(&sh_m[st][0][0], tab + b * kClCols, cnt * 4u * kClCols, &sh_bar[st]);
  };
  if (tid == 0) {
    issue(it.begin, 0);
    issue(it.begin + kClTile, 1);
  }
  u64 re[kClCols / 2], im[kClCols / 2];
#pragma unroll
  for (int c = 0; c < kClCols / 2; ++c) re[c] = im[c] = 0ull;
  const u64 sx2 = dev::pack2(sx, sx), sy2 = dev::pack2(sy, sy), sz2 = dev::pack2(sz, sz);
  const u64 magic2 = dev::pack2(12582912.0f, 12582912.0f);  // 1.5 * 2^23: rint by addition
  const u64 twopi2 = dev::pack2(6.28318530717958647692f, 6.28318530717958647692f);
  int st = 0, k = 0;
  for (int64_t b = it.begin; b < it.end; b += kClTile, st ^= 1, ++k) {
    const int cnt = (int)dev::min64(kClTile, it.end - b);
    const bool ok = dev::mbar_wait_bounded(&sh_bar[st], (uint32_t)((k >> 1) & 1));
    if (ok) {
      auto add = [&](float er, float ei, const float* m) {
        const u64 er2 = dev::pack2(er, er), ei2 = dev::pack2(ei, ei);
#pragma unroll
        for (int q = 0; q < kClCols / 4; ++q) {
          const float4 v = *reinterpret_cast<const float4*>(m + 4 * q);
          const u64 m0 = dev::pack2(v.x, v.y), m1 = dev::pack2(v.z, v.w);
          dev::ffma2(re[2 * q], er2, m0);
          dev::ffma2(im[2 * q], ei2, m0);
          dev::ffma2(re[2 * q + 1], er2, m1);
          dev::ffma2(im[2 * q + 1], ei2, m1);
        }
      };
#pragma unroll 4
      for (int j = 0; j < cnt; j += 2) {  // tiles hold multiples of 32 atoms
        const float4 p0 = sh_at[st][j], p1 = sh_at[st][j + 1];
        const u64 ph = dev::fma2(sz2, dev::pack2(p0.z, p1.z),
                                 dev::fma2(sy2, dev::pack2(p0.y, p1.y),
                                           dev::fma2(sx2, dev::pack2(p0.x, p1.x), dev::pack2(p0.w, p1.w))));
        const u64 f = dev::sub2(ph, dev::sub2(dev::add2(ph, magic2), magic2));  // ph - rint(ph)
        float t0, t1;
        dev::unpack2(dev::mul2(f, twopi2), t0, t1);
        add(__cosf(t0), __sinf(t0), &sh_m[st][j][0]);
        add(__cosf(t1), __sinf(t1), &sh_m[st][j + 1][0]);
      }
    }
    if (__syncthreads_or(!ok)) {
      if (tid == 0) {
        dev::set_status(a.status, kStatusTimeout);
        // drain the copies still in flight (bounded): this stage's and the next one's
        dev::mbar_wait_bounded(&sh_bar[st], (uint32_t)((k >> 1) & 1), 1LL << 28);
        if (b + kClTile < it.end) dev::mbar_wait_bounded(&sh_bar[st ^ 1], (uint32_t)(((k + 1) >> 1) & 1), 1LL << 28);
      }
      return;
    }
    if (tid == 0) issue(b + 2 * kClTile, st);
  }
  if (!ok_row) return;
  float2* out = a.partial + it.part + row;
#pragma unroll
  for (int c = 0; c < kClCols / 2; ++c) {
    float r0, r1, i0, i1;
    dev::unpack2(re[c], r0, r1);
    dev::unpack2(im[c], i0, i1);
    const int col = it.col_tile * kClCols + 2 * c;
    if (col < K) out[(int64_t)col * in.rows] = make_float2(r0, i0);
    if (col + 1 < K) out[(int64_t)(col + 1) * in.rows] = make_float2(r1, i1);
  }
}

// M[species][column][cluster] = i^|a| times the chunks' partials in order; 32 elements x 8
// contiguous shares of the chunks per CTA, joined in order.
__global__ void __launch_bounds__(256) k_cl_reduce(const ClArgs a) {
  __shared__ float2 sh[7][32];
  const ClRedBlock b = a.red_blocks[blockIdx.x];
  const ClInst in = a.inst[b.inst];
  const int K = cl_columns(a, in, b.inst);
  const int e = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int64_t i = b.elem + e;  // column * rows + cluster
  if (b.elem >= (int64_t)K * in.rows) return;
  const bool ok = i < (int64_t)K * in.rows;
  float2 v = make_float2(0.f, 0.f);
  if (ok) {
    const int per = (b.c1 - b.c0 + 7) / 8, lo = b.c0 + grp * per, hi = min(b.c1, lo + per);
    const float2* p = a.partial + in.part_off + i;
    const int64_t stride = (int64_t)in.K * in.rows;
#pragma unroll 8
    for (int c = lo; c < hi; ++c) {
      const float2 x = p[c * stride];
      v.x += x.x;
      v.y += x.y;
    }
  }
  if (grp > 0) sh[grp - 1][e] = v;
  __syncthreads();
  if (grp > 0 || !ok) return;
#pragma unroll
  for (int g = 0; g < 7; ++g) {
    v.x += sh[g][e].x;
    v.y += sh[g][e].y;
  }
  switch (a.exps[in.col0 + i / in.rows] >> 12) {  // i^|a|
    case 1: v = make_float2(-v.y, v.x); break;
    case 2: v = make_float2(-v.x, -v.y); break;
    case 3: v = make_float2(v.y, -v.x); break;
  }
  a.M[in.m_off + (int64_t)b.species * in.K * in.rows + i] = v;
}

// One thread per point, the points of a cluster next to each other: their loads
// of M are one broadcast.  32 us of the patch above; two species per pass over
// the columns share the powers but took 10 us more.
__global__ void __launch_bounds__(kClEval) k_cl_eval(const ClArgs a) {
  __shared__ float sh_p[3][kClMaxExp + 1][kClEval];
  __shared__ uchar4 sh_e[kClMaxK];
  const ClEvalBlock b = a.eval_blocks[blockIdx.x];
  const ClInst in = a.inst[b.inst];
  const int K = cl_columns(a, in, b.inst);
  const int t = threadIdx.x;
  if (K == 0) return;
  for (int c = t; c < K; c += kClEval) {
    const int e = a.exps[in.col0 + c];
    sh_e[c] = make_uchar4(e & 15, (e >> 4) & 15, (e >> 8) & 15, 0);
  }
  __syncthreads();
  if (t >= b.n) return;
  const float4 th = a.pt[b.p0 + t];  // 2 pi X d in the frame, cluster
  const int64_t m = a.pt_out[b.p0 + t];
  const int row = __float_as_int(th.w);
  const float thd[3] = {th.x, th.y, th.z};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    float p = 1.f;
#pragma unroll
    for (int e = 0; e <= kClMaxExp; ++e) {
      sh_p[d][e][t] = p;
      p *= thd[d];
    }
  }
  const float Sx = in.H[0] + a.s_hi[m], Sy = in.H[1] + a.s_hi[a.n_s + m], Sz = in.H[2] + a.s_hi[2 * a.n_s + m];
  const float s2 = (Sx * Sx + Sy * Sy + Sz * Sz) * a.inv4a2;
  float2 v = make_float2(0.f, 0.f);
  for (int sp = 0; sp < a.n_species; ++sp) {
    if (!((in.species >> sp) & 1ULL)) continue;  // no atoms of it in this instance
    const float2* M = a.M + in.m_off + (int64_t)sp * in.K * in.rows + row;
    // the last, smallest columns first: their rounding errors stay small
    float2 T = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int c = K - 1; c >= 0; --c) {
      const uchar4 e = sh_e[c];
      const float q = sh_p[0][e.x][t] * (sh_p[1][e.y][t] * sh_p[2][e.z][t]);
      const float2 x = M[(int64_t)c * in.rows];
      T.x = fmaf(q, x.x, T.x);
      T.y = fmaf(q, x.y, T.y);
    }
    const float2 F = a.ftab ? a.ftab[(int64_t)sp * a.n_s + m] : dev::form_factor(a.coef + kNCoef * sp, s2);
    const float2 f = dev::cmul(F, T);
    v.x += f.x;
    v.y += f.y;
  }
  const double* sh = a.inst_shift + 3 * b.inst;
  if (sh[0] != 0.0 || sh[1] != 0.0 || sh[2] != 0.0)
    v = dev::cmul(dev::shift_phase(a.S64[3 * m] - in.H64[0], a.S64[3 * m + 1] - in.H64[1], a.S64[3 * m + 2] - in.H64[2],
                                   sh),
                  v);
  if (a.out_amp) a.out_amp[m] = v;
  if (a.out_int) a.out_int[m] = v.x * v.x + v.y * v.y;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

// Eigenvectors (rows of R, by falling eigenvalue) of a symmetric 3 x 3 matrix:
// cyclic Jacobi rotations.
void principal_axes(double (&m)[3][3], double (&R)[3][3]) {
  double V[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
  for (int sweep = 0; sweep < 32; ++sweep)
    for (int p = 0; p < 2; ++p)
      for (int q = p + 1; q < 3; ++q) {
        if (std::fabs(m[p][q]) < 1e-300) continue;
        const double th = 0.5 * std::atan2(2.0 * m[p][q], m[q][q] - m[p][p]);
        const double c = std::cos(th), s = std::sin(th);
        for (int k = 0; k < 3; ++k) {
          const double a = m[k][p], b = m[k][q];
          m[k][p] = c * a - s * b;
          m[k][q] = s * a + c * b;
        }
        for (int k = 0; k < 3; ++k) {
          const double a = m[p][k], b = m[q][k];
          m[p][k] = c * a - s * b;
          m[q][k] = s * a + c * b;
        }
        for (int k = 0; k < 3; ++k) {
          const double a = V[k][p], b = V[k][q];
          V[k][p] = c * a - s * b;
          V[k][q] = s * a + c * b;
        }
      }
  int o[3] = {0, 1, 2};
  std::sort(o, o + 3, [&](int x, int y) { return m[x][x] > m[y][y]; });
  for (int d = 0; d < 3; ++d)
    for (int k = 0; k < 3; ++k) R[d][k] = V[k][o[d]];
}

struct Column {
  int e[3];
  int n;
  double rho;  // the relative radius of the crystal from which its term exceeds kClEps
};

// Columns whose largest term over |xh| <= 1, |th_d| <= th[d] exceeds kClEps:
// prod th_d^e_d / e_d! times the maximum prod e_d^(e_d / 2) / n^(n / 2) of the
// monomial over the unit ball.
std::vector<Column> columns_for(const double (&th)[3]) {
  std::vector<Column> cols;
  double ax[3][kClMaxExp + 1], nn[3 * kClMaxExp + 1], lf = 0.0;
  for (int e = 0; e <= kClMaxExp; ++e) {
    if (e) lf += std::log((double)e);
    for (int d = 0; d < 3; ++d)
      ax[d][e] = e ? e * (std::log(std::max(th[d], 1e-12)) + 0.5 * std::log((double)e)) - lf : 0.0;
  }
  for (int n = 0; n <= 3 * kClMaxExp; ++n) nn[n] = n ? 0.5 * n * std::log((double)n) : 0.0;
  const double eps = std::log(kClEps);
  // exponents that can matter: th^e / e! times the other axes' largest such
  // factors (the monomials stay below 1)
  double top[3] = {0, 0, 0}, fac[3][kClMaxExp + 1];
  int last[3] = {0, 0, 0};
  lf = 0.0;
  for (int e = 0; e <= kClMaxExp; ++e) {
    if (e) lf += std::log((double)e);
    for (int d = 0; d < 3; ++d) {
      fac[d][e] = e * std::log(std::max(th[d], 1e-12)) - lf;
      top[d] = std::max(top[d], fac[d][e]);
    }
  }
  for (int d = 0; d < 3; ++d)
    for (int e = 0; e <= kClMaxExp; ++e)
      if (fac[d][e] + top[(d + 1) % 3] + top[(d + 2) % 3] > eps) last[d] = e;
  for (int a = 0; a <= last[0]; ++a)
    for (int b = 0; b <= last[1]; ++b)
      for (int c = 0; c <= last[2]; ++c) {
        const int n = a + b + c;
        const double t = ax[0][a] + ax[1][b] + ax[2][c] - nn[n];
        if (t <= eps) continue;
        if (a == kClMaxExp || b == kClMaxExp || c == kClMaxExp) return {};  // exponents run out: too wide a cluster
        cols.push_back(Column{{a, b, c}, n, n ? std::exp((eps - t) / n) : 0.0});
      }
  return cols;
}

template <class T>
bool up(T** dst, const std::vector<T>& v, int64_t* bytes) {
  *bytes += (int64_t)(v.size() * sizeof(T));
  return cudaMalloc((void**)dst, std::max<size_t>(v.size(), 1) * sizeof(T)) == cudaSuccess &&
         (v.empty() || cudaMemcpy(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) == cudaSuccess);
}

}  // namespace

// Clusters of a LIST plan's instances, where the model finds them cheaper than
// the direct kernels (leaves p->cl.active false, and allocates nothing, where
// no instance is).  s_list: the caller's points (host, r.l.u.).
scatter_status prepare_clusters(scatter_plan_s* p, const double* s_list, double radius_hint) {
  if (p->s_kind != SCATTER_S_LIST || p->n_s <= 0 || p->n_slots <= 0 || p->n_species > kMaxSpecies) return SCATTER_OK;
  ClState& cl = p->cl;
  const double two_pi = 6.283185307179586;
  const int B = p->batch;
  std::vector<ClInst> insts(B);
  std::vector<float> lim(B, -1.0f), rho;
  std::vector<int32_t> exps;
  std::vector<float> cen[3];
  std::vector<float4> pt;
  std::vector<int64_t> pt_out;
  std::vector<ClItem> items;
  std::vector<ClTabBlock> tab_blocks;
  std::vector<ClRedBlock> red_blocks;
  std::vector<ClEvalBlock> eval_blocks;
  std::vector<ClExtent> extents;
  std::vector<int64_t> row_begin;  // of the last clustered instance: its clusters' points
  int64_t tab_floats = 0, part_floats = 0, m_floats = 0;
  double gain = 0.0;
  struct Framed {
    double q[3];
  };
  std::vector<Framed> fr;  // an instance's points in its frame
  for (int b = 0; b < B; ++b) {
    const Instance& in = p->inst[b];
    ClInst& ci = insts[b];
    ci = ClInst{};
    ci.lim2 = -1.0f;
    const int64_t M = in.s_end - in.s_begin, N = in.atom_end - in.atom_begin, slots = in.slot_end - in.slot_begin;
    if (M < 256 || N < 256) continue;
    // frame: principal axes of the points (moments about the first one)
    const double* S = s_list + 3 * in.s_begin;
    double mean[3] = {0, 0, 0}, cov[3][3] = {{0}}, R[3][3];
    for (int64_t i = 0; i < M; ++i) {
      const double q[3] = {S[3 * i] - S[0], S[3 * i + 1] - S[1], S[3 * i + 2] - S[2]};
      for (int d = 0; d < 3; ++d) {
        mean[d] += q[d];
        for (int e = d; e < 3; ++e) cov[d][e] += q[d] * q[e];
      }
    }
    for (int d = 0; d < 3; ++d) mean[d] /= (double)M;
    for (int d = 0; d < 3; ++d)
      for (int e = d; e < 3; ++e) cov[d][e] = cov[e][d] = cov[d][e] - (double)M * mean[d] * mean[e];
    for (int d = 0; d < 3; ++d) mean[d] += S[d] - in.H[d];
    principal_axes(cov, R);
    // the points in it, about their mean
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
    fr.resize((size_t)M);
    for (int64_t i = 0; i < M; ++i) {
      const double s[3] = {S[3 * i] - in.H[0] - mean[0], S[3 * i + 1] - in.H[1] - mean[1], S[3 * i + 2] - in.H[2] - mean[2]};
      for (int d = 0; d < 3; ++d) {
        const double q = R[d][0] * s[0] + R[d][1] * s[1] + R[d][2] * s[2];
        fr[i].q[d] = q;
        lo[d] = std::min(lo[d], q);
        hi[d] = std::max(hi[d], q);
      }
    }
    const double compact = std::cbrt(3.0 * (double)N / (16.0 * 3.14159265358979323846));
    const double X = radius_hint > 0.0 ? radius_hint : 1.45 * compact + 1.0;
    // a hint whose square is no float: a crystal of one point would be within it, and no
    // column matter
    if (!((float)(X * X) > 0.0f)) continue;
    // phases s.x' below the bound past which the direct kernels take exact products
    if (0.5 + (p->s_max[0] + p->s_max[1] + p->s_max[2]) * (X + 1.0) > 100.0) continue;
    // candidates for the cell side (corner phase th0) by the model, in clocks of
    // the SMs: measured 14 per (32 clusters, 16 columns, atom) and 4.3 per (32
    // points, atom) of the direct kernels.  Wide cells need more columns, narrow
    // ones more clusters: the patch of 60,001 points takes 0.32 ms at 296
    // clusters x 90 columns, 0.24 ms at 128 x 147, 0.29 ms at 100 x 177.  A flat
    // patch's third axis only tilts within a cell
    const double use = std::min(1.0, (compact + 0.5) / X), direct = std::ceil((double)M / 32.0) * (double)slots * 4.3;
    auto cost_of = [&](double cells, const double (&th)[3]) {
      const double th_use[3] = {th[0] * use, th[1] * use, th[2] * use};
      const size_t K = columns_for(th).size(), Ku = columns_for(th_use).size();
      if (K == 0 || K > (size_t)kClMaxK) return 1e300;
      const double tiles = std::ceil((double)Ku / kClCols);
      return std::ceil(cells / kClRows) * (kClRows / 32) * tiles * 14.0 * (double)slots +
             (double)M / 32.0 * (double)Ku * p->n_species * 6.0 + (double)slots / 32.0 * (double)Ku * 4.0;
    };
    struct Cand {
      double cost, h, th[3];
    };
    std::vector<Cand> cand;
    for (double th0 = 0.6; th0 < 3.2; th0 *= 1.1) {
      const double h = 1.41421356 * th0 / (two_pi * X);
      double cells = 1.0, nbd[3], th[3];
      for (int d = 0; d < 3; ++d) {
        nbd[d] = std::max(1.0, std::ceil((hi[d] - lo[d]) / h));
        cells *= nbd[d];
        th[d] = two_pi * X * 0.5 * (hi[d] - lo[d]) / nbd[d];
      }
      if (nbd[2] == 1.0 && nbd[0] > 2.0) th[2] *= 2.0 / nbd[0];
      if (cells > (double)M / 3.0 || cells > 4.0e6) continue;
      if (const double c = cost_of(cells, th); c < direct) cand.push_back({c, h, {th[0], th[1], th[2]}});
    }
    std::sort(cand.begin(), cand.end(), [](const Cand& x, const Cand& y) { return x.cost < y.cost; });
    // clusters: the cells that hold points
    int rows = 0;
    std::vector<int32_t> cell(cand.empty() ? 0 : M), row_of;
    std::vector<int64_t> first;
    auto build = [&](double h) {
      int64_t nb[3];
      double inv[3];
      for (int d = 0; d < 3; ++d) {
        nb[d] = std::max<int64_t>(1, (int64_t)std::ceil((hi[d] - lo[d]) / h));
        inv[d] = hi[d] > lo[d] ? (double)nb[d] / (hi[d] - lo[d]) : 0.0;
      }
      first.assign(nb[0] * nb[1] * nb[2], 0);
      for (int64_t i = 0; i < M; ++i) {
        int64_t id = 0;
        for (int d = 0; d < 3; ++d)
          id = id * nb[d] +
               std::max<int64_t>(0, std::min<int64_t>(nb[d] - 1, (int64_t)((fr[i].q[d] - lo[d]) * inv[d])));
        cell[i] = (int32_t)id;
        ++first[id];
      }
      row_of.assign(first.size(), -1);
      rows = 0;
      int64_t at = 0;
      for (size_t k = 0; k < row_of.size(); ++k)
        if (first[k]) {
          row_of[k] = rows;
          const int64_t n = first[k];
          first[rows++] = at;
          at += n;
        }
    };
    // the cells as they come out: a disc leaves corners empty, and rows come in 64s
    double best = 0.7 * direct, best_h = 0.0, last_h = 0.0;
    for (size_t t = 0; t < std::min<size_t>(cand.size(), 6); ++t) {
      build(last_h = cand[t].h);
      if (const double c = cost_of((double)rows, cand[t].th); c < best) best = c, best_h = last_h;
    }
    if (best_h == 0.0) continue;
    if (best_h != last_h) build(best_h);
    // clusters centred on their points
    std::vector<double> mn(3 * (size_t)rows, 1e300), mx(3 * (size_t)rows, -1e300);
    for (int64_t i = 0; i < M; ++i) {
      const int r = cell[i] = row_of[cell[i]];
      for (int d = 0; d < 3; ++d) {
        mn[3 * r + d] = std::min(mn[3 * r + d], fr[i].q[d]);
        mx[3 * r + d] = std::max(mx[3 * r + d], fr[i].q[d]);
      }
    }
    double th[3] = {0, 0, 0};
    for (int r = 0; r < rows; ++r)
      for (int d = 0; d < 3; ++d) th[d] = std::max(th[d], two_pi * X * 0.5 * (mx[3 * r + d] - mn[3 * r + d]));
    std::vector<Column> cols = columns_for(th);
    if (cols.empty() || cols.size() > (size_t)kClMaxK) continue;
    std::sort(cols.begin(), cols.end(), [](const Column& x, const Column& y) {
      return x.rho != y.rho ? x.rho < y.rho : std::lexicographical_compare(x.e, x.e + 3, y.e, y.e + 3);
    });
    // chunks of one species: at most 256 atoms, fewer where the SMs would idle
    const int row_tiles = (rows + kClRows - 1) / kClRows, col_tiles = ((int)cols.size() + kClCols - 1) / kClCols;
    int64_t len = 256;
    while (len > 64 && (double)row_tiles * std::max(1, col_tiles * 2 / 3) * std::ceil((double)slots / (double)len) * B <
                           24.0 * p->n_sm)
      len /= 2;
    int64_t n_chunks = 0;
    for (const Segment& sg : p->all_segs)
      if (sg.instance == b && sg.end > sg.begin) n_chunks += (sg.end - sg.begin + len - 1) / len;
    const int64_t more_tab = (int64_t)col_tiles * slots * kClCols, more_part = n_chunks * (int64_t)cols.size() * rows;
    if ((tab_floats + more_tab) * 4 + (part_floats + more_part) * 8 > kClMaxBytes) continue;
    // tables of the instance
    ci.slot_begin = in.slot_begin;
    ci.n_slots = slots;
    ci.lim2 = (float)(X * X);
    ci.K = (int)cols.size();
    ci.col0 = (int)exps.size();
    ci.rows = rows;
    ci.row0 = (int64_t)cen[0].size();
    ci.tab_off = tab_floats;
    ci.m_off = m_floats;
    ci.part_off = part_floats;
    for (int d = 0; d < 3; ++d) {
      ci.H[d] = (float)in.H[d];
      ci.H64[d] = in.H[d];
      for (int k = 0; k < 3; ++k) ci.R[3 * d + k] = (float)(R[d][k] / X);
    }
    for (const Column& c : cols) {
      exps.push_back(c.e[0] | c.e[1] << 4 | c.e[2] << 8 | (c.n & 3) << 12);
      rho.push_back(c.n ? (float)c.rho : -1.0f);
    }
    for (int r = 0; r < rows; ++r) {
      double q[3], s[3];
      for (int d = 0; d < 3; ++d) q[d] = 0.5 * (mn[3 * r + d] + mx[3 * r + d]);
      for (int k = 0; k < 3; ++k) {
        s[k] = R[0][k] * q[0] + R[1][k] * q[1] + R[2][k] * q[2] + mean[k];
        cen[k].push_back((float)s[k]);
      }
      // the centre that the kernels use is the rounded one: offsets from it
      for (int d = 0; d < 3; ++d) {
        q[d] = 0.0;
        for (int k = 0; k < 3; ++k) q[d] += R[d][k] * ((double)(float)s[k] - mean[k]);
        mn[3 * r + d] = q[d];
      }
    }
    const size_t p_base = pt.size();
    pt.resize(p_base + M);
    pt_out.resize(p_base + M);
    for (int64_t i = 0; i < M; ++i) {
      const double* q = fr[i].q;
      const int r = cell[i];
      const size_t o = p_base + (size_t)first[r]++;
      float4 v;
      v.x = (float)(two_pi * X * (q[0] - mn[3 * r]));
      v.y = (float)(two_pi * X * (q[1] - mn[3 * r + 1]));
      v.z = (float)(two_pi * X * (q[2] - mn[3 * r + 2]));
      const int32_t rr = r;
      std::memcpy(&v.w, &rr, sizeof(float));
      pt[o] = v;
      pt_out[o] = in.s_begin + i;
    }
    row_begin.assign(1, 0);  // first[r] is now the cluster's end
    row_begin.insert(row_begin.end(), first.begin(), first.begin() + rows);
    for (int64_t o = 0; o < M; o += kClEval)
      eval_blocks.push_back(ClEvalBlock{b, (int32_t)std::min<int64_t>(kClEval, M - o), (int64_t)p_base + o});
    for (int64_t s = 0; s < slots; s += 128) tab_blocks.push_back(ClTabBlock{b, s});
    int chunk = 0;
    for (const Segment& sg : p->all_segs) {
      if (sg.instance != b || sg.end <= sg.begin) continue;
      ci.species |= 1ULL << sg.species;
      const int c0 = chunk;
      for (int64_t x = sg.begin; x < sg.end; x += len, ++chunk)
        for (int ct = 0; ct < col_tiles; ++ct)
          for (int rt = 0; rt < row_tiles; ++rt)
            items.push_back(ClItem{b, rt * kClRows, ct, sg.species, x - in.slot_begin, std::min(sg.end, x + len) - in.slot_begin,
                                   part_floats + (int64_t)chunk * ci.K * rows});
      for (int64_t e = 0; e < (int64_t)ci.K * rows; e += 32) red_blocks.push_back(ClRedBlock{b, sg.species, c0, chunk, e});
    }
    tab_floats += more_tab;
    part_floats += more_part;
    m_floats += (int64_t)p->n_species * ci.K * rows;
    lim[b] = ci.lim2;
    extents.push_back(ClExtent{X, {th[0], th[1], th[2]}});
    gain += direct - best;
  }
  // worth the extra launches (~30 us)
  if (items.empty() || gain < 30e-6 * 2.0e9 * p->n_sm) return SCATTER_OK;
  int64_t bytes = 0;
  std::vector<float> centres;
  for (int d = 0; d < 3; ++d) centres.insert(centres.end(), cen[d].begin(), cen[d].end());
  const bool ok = up(&cl.inst, insts, &bytes) && up(&cl.lim2, lim, &bytes) && up(&cl.rho, rho, &bytes) &&
                  up(&cl.exps, exps, &bytes) && up(&cl.cen, centres, &bytes) && up(&cl.pt, pt, &bytes) &&
                  up(&cl.pt_out, pt_out, &bytes) && up(&cl.items, items, &bytes) &&
                  up(&cl.tab_blocks, tab_blocks, &bytes) && up(&cl.red_blocks, red_blocks, &bytes) &&
                  up(&cl.eval_blocks, eval_blocks, &bytes) && up(&cl.rmax2, std::vector<unsigned>(B, 0u), &bytes) &&
                  cudaMalloc(&cl.tab, (size_t)tab_floats * sizeof(float)) == cudaSuccess &&
                  cudaMalloc(&cl.partial, (size_t)part_floats * sizeof(float2)) == cudaSuccess &&
                  cudaMalloc(&cl.M, (size_t)m_floats * sizeof(float2)) == cudaSuccess;
  if (!ok) {  // no room: the direct kernels need none of it
    cudaGetLastError();
    release_clusters(p);
    return SCATTER_OK;
  }
  bytes += tab_floats * 4 + (part_floats + m_floats) * 8;
  cl.n_rows = (int64_t)cen[0].size();
  cl.n_items = (int)items.size();
  cl.n_tab = (int)tab_blocks.size();
  cl.n_red = (int)red_blocks.size();
  cl.n_eval = (int)eval_blocks.size();
  p->base_bytes += bytes;
  if (B == 1) {  // backward prepares its own tables from these
    cl.first = insts[0];
    cl.h_exps = exps;
    cl.h_row = row_begin;
  }
  cl.extents = std::move(extents);
  cl.active = true;
  return SCATTER_OK;
}

void cluster_error(const scatter_plan_s* p, double radius, double* truncation, double* rounding) {
  *truncation = *rounding = 0.0;
  for (const ClExtent& e : p->cl.extents) {
    const double r = std::min(1.0, radius / e.X), u = std::ldexp(1.0, -24);
    if (!(r > 0.0)) continue;
    // Every term above 1e-12 with the relative radius from which it is a column (past 1
    // never).  A crystal of relative radius q leaves out those past q: of degree n at most
    // their largest values over the ball, and at most all terms' (|th| q)^n / n!.
    // The sum is largest just before a column joins, or at r.
    constexpr int kTop = 40;
    struct Term {
      double value, rho;  // over the whole ball
      int n;
    };
    std::vector<Term> terms;
    double ax[3][kTop + 1], lf = 0.0;
    for (int i = 0; i <= kTop; ++i) {
      if (i) lf += std::log((double)i);
      for (int d = 0; d < 3; ++d)
        ax[d][i] = i ? i * (std::log(std::max(e.th[d], 1e-12)) + 0.5 * std::log((double)i)) - lf : 0.0;
    }
    for (int a = 0; a <= kTop; ++a)
      for (int b = 0; a + b <= kTop; ++b)
        for (int c = 0; a + b + c <= kTop; ++c) {
          const int n = a + b + c;
          if (n == 0) continue;
          const double t = ax[0][a] + ax[1][b] + ax[2][c] - 0.5 * n * std::log((double)n);
          if (t > -27.6) terms.push_back({std::exp(t), std::exp((std::log(kClEps) - t) / n), n});
        }
    const double len = std::sqrt(e.th[0] * e.th[0] + e.th[1] * e.th[1] + e.th[2] * e.th[2]);
    auto neglected = [&](double q) {
      double by[kTop + 1] = {0.0}, sum = 0.0, all = 1.0, power = 1.0;
      for (const Term& m : terms)
        if (m.rho >= q) by[m.n] += m.value;
      for (int n = 1; n <= kTop; ++n) {
        all *= len * q / n;
        power *= q;
        sum += std::min(by[n] * power, all);
      }
      return sum;
    };
    double worst = neglected(r);
    for (const Term& m : terms)
      if (m.rho < r) worst = std::max(worst, neglected(m.rho));
    *truncation = std::max(*truncation, worst);
    // a column of degree n carries 4 n + 5 roundings; the columns' absolute sum is below e^(|th| r)
    *rounding = std::max(*rounding, u * std::exp(len * r) * (4.0 * len * r + 5.0));
  }
}

ClArgs cluster_args(scatter_plan_s* p) {
  const ClState& cl = p->cl;
  ClArgs a{};
  a.inst = cl.inst;
  a.rmax2 = cl.rmax2;
  a.rho = cl.rho;
  a.exps = cl.exps;
  a.cen = cl.cen;
  a.n_rows = cl.n_rows;
  a.pt = cl.pt;
  a.pt_out = cl.pt_out;
  a.items = cl.items;
  a.tab_blocks = cl.tab_blocks;
  a.red_blocks = cl.red_blocks;
  a.eval_blocks = cl.eval_blocks;
  a.tab = cl.tab;
  a.partial = cl.partial;
  a.M = cl.M;
  a.atom4 = p->d.atom4;
  a.atom_w = p->d.atom_w;
  a.coef = p->d.coef;
  a.ftab = p->d.ftab;
  a.n_species = p->n_species;
  a.inv4a2 = (float)(1.0 / (4.0 * p->lattice_a * p->lattice_a));
  a.s_hi = p->d.s_hi;
  a.S64 = p->d.S64;
  a.n_s = p->n_s;
  a.inst_shift = p->d.inst_shift;
  a.status = p->d.status;
  return a;
}

// The clustered instances' points, on prepared positions (launch_prep writes
// rmax2); the direct kernels do the others.
scatter_status launch_clusters(scatter_plan_t p, float2* amp_out, float* int_out, cudaStream_t st) {
  const ClState& cl = p->cl;
  ClArgs a = cluster_args(p);
  a.out_amp = amp_out;
  a.out_int = int_out;
  k_cl_tab<<<cl.n_tab, 128, 0, st>>>(a);
  if (p->batch == 1) timing_begin(p, st);  // to the end of the direct kernel, which may do the work instead
  k_cl_moments<<<cl.n_items, kClRows, 0, st>>>(a);
  k_cl_reduce<<<cl.n_red, 256, 0, st>>>(a);
  k_cl_eval<<<cl.n_eval, kClEval, 0, st>>>(a);
  p->last_launches += 4;
  return cuda_status(cudaGetLastError(), "cluster launch");
}

void release_clusters(scatter_plan_s* p) {
  ClState& cl = p->cl;
  for (void* b : {(void*)cl.inst, (void*)cl.lim2, (void*)cl.rho, (void*)cl.exps, (void*)cl.cen, (void*)cl.pt,
                  (void*)cl.pt_out, (void*)cl.items, (void*)cl.tab_blocks, (void*)cl.red_blocks, (void*)cl.eval_blocks,
                  (void*)cl.rmax2, (void*)cl.tab, (void*)cl.partial, (void*)cl.M})
    if (b) cudaFree(b);
  release_cluster_adjoint(cl.adj);
  cl = ClState{};
}

}  // namespace scatter
