// Adjoint of the clustered S lists (cluster.cu): the sum over the points once
// per cluster, not per atom.
//
// With cluster centres s_k, th_m = 2 pi X (s_m - s_k) in the clusters' frame and
// x'_j = X xh_j there,
//   sum_{m in k} gF_m e^{2 pi i (c_j + s_m.x'_j)} = E_jk P_k(xh_j),
//   E_jk = e^{2 pi i (c_j + s_k.x'_j)},  P_k(xh) = sum_a G_k[a] xh^a / a!,
//   G_k[a] = i^|a| sum_{m in k} gF_m th_m^a,
// and the same sum weighted by th_m,d is -i E_jk dP_k/dxh_d, whose coefficients
// are G_k[a + e_d].  With S_m = H + s_k + (s_m - s_k) an (atom, cluster) pair
// costs one sincos and eight multiply-adds per column, and gives
//   v = Im(E P)          sum_k v and sum_k s_k v,
//   u_d = -Re(E dP_d)    sum_k u_d, turned back from the frame at the end.
// The clusters hold hundreds of points each.  The large sum over k of v, which
// nearly cancels, is a double-float one as in adjoint.cu; s_k and th are some
// hundredths of H.
//
//   k_cl_gsum  per 256 points of a cluster: sum gF th^a, every column and species
//   k_cl_gfin  per cluster and species: their ordered double-float sums, times
//              i^|a|, into the rows of eight that k_cl_adj reads
//   k_cl_adj   256 atoms x a range of clusters, four clusters at a time
// A crystal past the clusters' radius is left to k_adjoint, whose launch
// otherwise returns at once.
// 28,953 atoms x 100,003 points of a detector patch (64 clusters): 0.13-0.16 ms per
// call against 1.47 ms; relative error against FP64 1.8e-7 against 2.6e-7.
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <vector>
#include "cluster_common.cuh"
#include "device_common.cuh"
#include "launch.h"

namespace scatter {

namespace {

constexpr int kGThreads = 128;
constexpr int kGTile = 64;                                         // points per stage
constexpr int kGPoints = 256;                                      // points per CTA
constexpr int kGCols = (kClMaxK + kGThreads - 1) / kGThreads;      // columns per thread
constexpr int kGPow = 3 * (kClMaxExp + 1) + 1;                     // powers of a point, odd stride
constexpr int kAtThreads = 128;
constexpr int kAtRA = 2;                                           // atoms per thread
constexpr int kAtRows = 4;                                         // clusters at a time

struct ClAdjArgs {
  ClArgs c;
  const float2* gf;        // [species][M]
  const ClGBlock* g_blocks;
  const int32_t* row_blk;
  const short4* up;
  const short4* down;
  float2* g_part;
  float* g8;
  const AdjBlock* blocks;
  int rows_per_chunk;
  int emax[3];
  float* partial;          // [split][n_slots][3]
  int64_t n_slots;
};

// A thread per column (a few where there are more than 128): the points' powers
// are staged per point, so the lanes read at most 48 neighbouring words.
__global__ void __launch_bounds__(kGThreads) k_cl_gsum(const ClAdjArgs a) {
  __shared__ float sh_p[kGTile][kGPow];
  __shared__ float4 sh_g[kGTile];  // gF of two species
  const ClGBlock b = a.g_blocks[blockIdx.x];
  const ClInst in = a.c.inst[0];
  const int K = cl_columns(a.c, in, 0);
  const int t = threadIdx.x;
  if (K == 0) return;
  const int s0 = 2 * blockIdx.y, n_sp = a.c.n_species;
  float4 acc[kGCols];
  uint32_t off[kGCols];
#pragma unroll
  for (int i = 0; i < kGCols; ++i) {
    const int c = i * kGThreads + t;
    const int e = c < K ? a.c.exps[in.col0 + c] : 0;
    off[i] = (uint32_t)(e & 15) | (uint32_t)(((e >> 4) & 15) + 16) << 8 | (uint32_t)(((e >> 8) & 15) + 32) << 16;
    acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  for (int p0 = 0; p0 < b.n; p0 += kGTile) {
    const int n = min(kGTile, b.n - p0);
    const int pt = t & (kGTile - 1);
    __syncthreads();
    if (pt < n) {
      const int64_t i = b.p0 + p0 + pt;
      const float4 th = a.c.pt[i];
      const int64_t m = a.c.pt_out[i];
      auto powers = [&](int d, float x) {
        float p = 1.f;
#pragma unroll
        for (int e = 0; e <= kClMaxExp; ++e) {
          sh_p[pt][16 * d + e] = p;
          p *= x;
        }
      };
      if (t < kGTile) {
        powers(0, th.x);
        const float2 g0 = a.gf[(int64_t)s0 * a.c.n_s + m];
        const float2 g1 = s0 + 1 < n_sp ? a.gf[(int64_t)(s0 + 1) * a.c.n_s + m] : make_float2(0.f, 0.f);
        sh_g[pt] = make_float4(g0.x, g0.y, g1.x, g1.y);
      } else {
        powers(1, th.y);
        powers(2, th.z);
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kGCols; ++i) {
      if (i * kGThreads + t >= K) break;
      const float* p = sh_p[0];
      const float *px = p + (off[i] & 255), *py = p + ((off[i] >> 8) & 255), *pz = p + (off[i] >> 16);
#pragma unroll 4
      for (int j = 0; j < n; ++j) {
        const float q = px[j * kGPow] * (py[j * kGPow] * pz[j * kGPow]);
        const float4 g = sh_g[j];
        acc[i].x = fmaf(q, g.x, acc[i].x);
        acc[i].y = fmaf(q, g.y, acc[i].y);
        acc[i].z = fmaf(q, g.z, acc[i].z);
        acc[i].w = fmaf(q, g.w, acc[i].w);
      }
    }
  }
  float2* out = a.g_part + ((int64_t)blockIdx.x * n_sp + s0) * in.K;
#pragma unroll
  for (int i = 0; i < kGCols; ++i) {
    const int c = i * kGThreads + t;
    if (c >= K) break;
    out[c] = make_float2(acc[i].x, acc[i].y);
    if (s0 + 1 < n_sp) out[in.K + c] = make_float2(acc[i].z, acc[i].w);
  }
}

// Row of eight of column b: G[b], G[b + e_0], G[b + e_1], G[b + e_2]; columns
// without a raised one keep 0 there.
__global__ void __launch_bounds__(kGThreads) k_cl_gfin(const ClAdjArgs a) {
  const ClInst in = a.c.inst[0];
  const int K = cl_columns(a.c, in, 0);
  const int row = blockIdx.x, sp = blockIdx.y;
  const int b0 = a.row_blk[row], b1 = a.row_blk[row + 1];
  float2* g8 = reinterpret_cast<float2*>(a.g8) + ((int64_t)sp * in.rows + row) * in.K * 4;
  for (int c = threadIdx.x; c < K; c += kGThreads) {
    const float2* p = a.g_part + ((int64_t)b0 * a.c.n_species + sp) * in.K + c;
    const int64_t stride = (int64_t)a.c.n_species * in.K;
    dev::DFloatSum re, im;
#pragma unroll 4
    for (int b = b0; b < b1; ++b, p += stride) {
      const float2 v = *p;
      re.add(v.x);
      im.add(v.y);
    }
    float2 v = make_float2(re.value(), im.value());
    switch (a.c.exps[in.col0 + c] >> 12) {  // i^|a|
      case 1: v = make_float2(-v.y, v.x); break;
      case 2: v = make_float2(-v.x, -v.y); break;
      case 3: v = make_float2(v.y, -v.x); break;
    }
    const short4 up = a.up[c], dn = a.down[c];
    const int u[3] = {up.x, up.y, up.z}, d[3] = {dn.x, dn.y, dn.z};
    g8[4 * c] = v;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (u[k] < 0 || u[k] >= K) g8[4 * c + 1 + k] = make_float2(0.f, 0.f);
      if (d[k] >= 0 && d[k] < K) g8[4 * d[k] + 1 + k] = v;
    }
  }
}

// 256 atoms of one species per CTA, two per thread, against four clusters at a
// time: 64 accumulators; per column two monomials from the atoms' powers and
// eight broadcast 16-byte loads feed 32 packed multiply-adds.  Bound by the FMA
// pipe and the loads' latency: 75 us on the patch above, 94 us with two columns
// in flight instead of eight; 2 atoms x 2 clusters 97 us, 4 x 2 79 us, 1 x 8 107 us.
__global__ void __launch_bounds__(kAtThreads) k_cl_adj(const ClAdjArgs a) {
  using u64 = unsigned long long;
  constexpr int kAtoms = kAtThreads * kAtRA;
  extern __shared__ __align__(16) float sh[];
  __shared__ uchar4 sh_e[kClMaxK];
  const ClInst in = a.c.inst[0];
  const int K = cl_columns(a.c, in, 0);
  if (K == 0) return;
  const AdjBlock blk = a.blocks[blockIdx.x];
  const int t = threadIdx.x;
  const int o1 = a.emax[0] + 1, o2 = o1 + a.emax[1] + 1;
  float4* sh_g = reinterpret_cast<float4*>(sh);                      // [kAtRows][K][2]
  float* sh_p = sh + (int64_t)kAtRows * in.K * 8;                    // [powers][atoms]
  for (int c = t; c < K; c += kAtThreads) {
    const int e = a.c.exps[in.col0 + c];
    sh_e[c] = make_uchar4(e & 15, o1 + ((e >> 4) & 15), o2 + ((e >> 8) & 15), 0);
  }
  float4 at[kAtRA];
#pragma unroll
  for (int r = 0; r < kAtRA; ++r) {
    const int i = r * kAtThreads + t;
    at[r] = i < blk.count ? a.c.atom4[blk.begin + i] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float x = in.R[3 * d] * at[r].x + in.R[3 * d + 1] * at[r].y + in.R[3 * d + 2] * at[r].z;
      float* o = sh_p + (int64_t)(d == 0 ? 0 : d == 1 ? o1 : o2) * kAtoms + i;
      float p = 1.f;
      for (int e = 0; e <= a.emax[d]; ++e) {
        o[e * kAtoms] = p;  // xh^e / e!
        p *= x / (float)(e + 1);
      }
    }
  }
  dev::DFloatSum sv[kAtRA];
  float ss[kAtRA][3], su[kAtRA][3];
#pragma unroll
  for (int r = 0; r < kAtRA; ++r)
#pragma unroll
    for (int d = 0; d < 3; ++d) ss[r][d] = su[r][d] = 0.f;
  const int r0 = blockIdx.y * a.rows_per_chunk, r1 = min(in.rows, r0 + a.rows_per_chunk);
  const float4* g8 = reinterpret_cast<const float4*>(a.g8) + (int64_t)blk.species * in.rows * in.K * 2;
  for (int row = r0; row < r1; row += kAtRows) {
    __syncthreads();
    for (int k = 0; k < kAtRows; ++k) {
      const float4* src = g8 + (int64_t)(row + k) * in.K * 2;
      for (int i = t; i < 2 * K; i += kAtThreads)
        sh_g[2 * K * k + i] = row + k < r1 ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    u64 acc[kAtRA][kAtRows][4];
#pragma unroll
    for (int r = 0; r < kAtRA; ++r)
#pragma unroll
      for (int k = 0; k < kAtRows; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][k][q] = 0ull;
#pragma unroll 8
    for (int c = K - 1; c >= 0; --c) {
      const uchar4 e = sh_e[c];
      u64 q[kAtRA];
#pragma unroll
      for (int r = 0; r < kAtRA; ++r) {
        const float* p = sh_p + r * kAtThreads + t;
        const float m = p[e.x * kAtoms] * (p[e.y * kAtoms] * p[e.z * kAtoms]);
        q[r] = dev::pack2(m, m);
      }
#pragma unroll
      for (int k = 0; k < kAtRows; ++k) {
        const float4* g = sh_g + 2 * (K * k + c);
        const float4 g0 = g[0], g1 = g[1];
        const u64 w[4] = {dev::pack2(g0.x, g0.y), dev::pack2(g0.z, g0.w), dev::pack2(g1.x, g1.y),
                          dev::pack2(g1.z, g1.w)};
#pragma unroll
        for (int r = 0; r < kAtRA; ++r)
#pragma unroll
          for (int i = 0; i < 4; ++i) dev::ffma2(acc[r][k][i], q[r], w[i]);
      }
    }
#pragma unroll
    for (int k = 0; k < kAtRows; ++k) {
      const int64_t rg = in.row0 + min(row + k, in.rows - 1);  // past r1: the coefficients are 0
      const float s[3] = {a.c.cen[rg], a.c.cen[a.c.n_rows + rg], a.c.cen[2 * a.c.n_rows + rg]};
#pragma unroll
      for (int r = 0; r < kAtRA; ++r) {
        // one exponential for hundreds of points: its products with their
        // rounding errors, sin and cos to the last place
        const float f = dev::frac_product_plus(
            s[2], at[r].z, dev::frac_product_plus(s[1], at[r].y, dev::frac_product_plus(s[0], at[r].x, at[r].w)));
        float es, ec, x, y;
        sincospif(2.0f * dev::frac_rn(f), &es, &ec);
        dev::unpack2(acc[r][k][0], x, y);
        const float v = fmaf(es, x, ec * y);
        sv[r].add(v);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          ss[r][d] = fmaf(s[d], v, ss[r][d]);
          dev::unpack2(acc[r][k][1 + d], x, y);
          su[r][d] += fmaf(es, y, -ec * x);
        }
      }
    }
  }
  float* out = a.partial + (int64_t)blockIdx.y * a.n_slots * 3;
#pragma unroll
  for (int r = 0; r < kAtRA; ++r) {
    const int i = r * kAtThreads + t;
    if (i >= blk.count) continue;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      // H sum v (H as a double-float) + sum s_k v + the frame's part
      const float h = in.H[d], hl = (float)(in.H64[d] - (double)h);
      const float p = __fmul_rn(h, sv[r].hi);
      const float e = __fmaf_rn(h, sv[r].hi, -p) + fmaf(h, sv[r].lo, hl * sv[r].hi);
      const float u = in.R[d] * su[r][0] + in.R[3 + d] * su[r][1] + in.R[6 + d] * su[r][2];
      dev::DFloatSum g;
      g.hi = p;
      g.add(ss[r][d]);
      g.lo += e + 0.159154943091895335769f * u;
      out[3 * (blk.begin + i) + d] = g.value();
    }
  }
}

template <class T>
bool up_host(T** dst, const std::vector<T>& v) {
  return cudaMalloc((void**)dst, std::max<size_t>(v.size(), 1) * sizeof(T)) == cudaSuccess &&
         (v.empty() || cudaMemcpy(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) == cudaSuccess);
}

}  // namespace

scatter_status prepare_cluster_adjoint(scatter_plan_s* p) {
  ClState& cl = p->cl;
  if (!cl.active || p->batch != 1 || cl.first.K == 0 || cl.adj.active) return SCATTER_OK;
  const ClInst& in = cl.first;
  const int K = in.K, rows = in.rows;
  // lanes x clocks per atom: eight multiply-adds per column and cluster (and as
  // much again for loads and monomials) against the direct kernel's measured 19
  // per point
  if ((double)rows * (8.0 * 2.0 * K + 100.0) > 0.7 * 19.0 * (double)p->n_s) return SCATTER_OK;
  ClAdjState& s = cl.adj;
  for (int d = 0; d < 3; ++d) s.emax[d] = 0;
  std::vector<int> index(1 << 12, -1);
  for (int c = 0; c < K; ++c) {
    index[cl.h_exps[c] & 0xfff] = c;
    for (int d = 0; d < 3; ++d) s.emax[d] = std::max(s.emax[d], (cl.h_exps[c] >> (4 * d)) & 15);
  }
  std::vector<short4> upv(K), dnv(K);
  for (int c = 0; c < K; ++c) {
    const int e = cl.h_exps[c] & 0xfff;
    short u[3], v[3];
    for (int d = 0; d < 3; ++d) {
      const int x = (e >> (4 * d)) & 15;
      u[d] = x < 15 ? (short)index[e + (1 << (4 * d))] : (short)-1;
      v[d] = x > 0 ? (short)index[e - (1 << (4 * d))] : (short)-1;
    }
    upv[c] = make_short4(u[0], u[1], u[2], 0);
    dnv[c] = make_short4(v[0], v[1], v[2], 0);
  }
  // A column of degree n and largest term t counts for the sum from the radius at which
  // t r^n passes kClEps, and for a derivative from n t r^(n - 1) = kClEps of the whole
  // phase gradient, 2 pi X |H| and the corner's own: of a crystal that is a point the first
  // degree is left (dropped, the gradient kept |S| at the clusters' centres: 3e-2 off).
  // The columns in use are the first ones, so each takes the least radius behind it.
  const ClExtent& ext = cl.extents[0];
  const double* H = p->inst[0].H;
  const double corner = std::sqrt(ext.th[0] * ext.th[0] + ext.th[1] * ext.th[1] + ext.th[2] * ext.th[2]);
  const double scale = std::max(corner, 6.283185307179586 * ext.X * std::sqrt(H[0] * H[0] + H[1] * H[1] + H[2] * H[2]));
  std::vector<float> rho(K);
  for (int c = K - 1; c >= 0; --c) {
    int n = 0;
    double t = 0.0;
    for (int d = 0; d < 3; ++d) {
      const int x = (cl.h_exps[c] >> (4 * d)) & 15;
      n += x;
      if (x) t += x * (std::log(std::max(ext.th[d], 1e-12)) + 0.5 * std::log((double)x)) - std::lgamma(x + 1.0);
    }
    double r = -1.0;
    if (n > 0) {
      t -= 0.5 * n * std::log((double)n);
      const double own = (std::log(kClEps) - t) / n, der = std::log(kClEps * scale / n) - t;
      r = std::exp(n > 1 ? std::min(own, der / (n - 1)) : own);
      if (n == 1 && der < 0.0) r = -1.0;
    }
    rho[c] = (float)r;
    if (c + 1 < K) rho[c] = std::min(rho[c], rho[c + 1]);
  }
  std::vector<ClGBlock> gb;
  std::vector<int32_t> row_blk(rows + 1);
  for (int r = 0; r < rows; ++r) {
    row_blk[r] = (int32_t)gb.size();
    for (int64_t o = cl.h_row[r]; o < cl.h_row[r + 1]; o += kGPoints)
      gb.push_back(ClGBlock{r, (int32_t)std::min<int64_t>(kGPoints, cl.h_row[r + 1] - o), o});
  }
  row_blk[rows] = (int32_t)gb.size();
  std::vector<AdjBlock> blocks;
  const int per = kAtThreads * kAtRA;
  for (const Segment& sg : p->all_segs)
    for (int64_t b = sg.begin; b < sg.end; b += per)
      blocks.push_back(AdjBlock{b, (int32_t)std::min<int64_t>(per, sg.end - b), sg.species});
  const int64_t part = (int64_t)gb.size() * p->n_species * K, g8 = (int64_t)p->n_species * rows * K * 8;
  s.smem = (int)((kAtRows * K * 8 + (s.emax[0] + s.emax[1] + s.emax[2] + 3) * per) * sizeof(float));
  int bps = 0, most = 0;
  if (cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device) != cudaSuccess) most = 0;
  if (blocks.empty() || part * 8 + g8 * 4 > (4LL << 30) || s.smem + 4096 > most ||
      cudaFuncSetAttribute(k_cl_adj, cudaFuncAttributeMaxDynamicSharedMemorySize, most - 4096) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_cl_adj, kAtThreads, s.smem) != cudaSuccess || bps < 1) {
    cudaGetLastError();
    return SCATTER_OK;
  }
  // clusters per CTA: the fewest waves x (clusters + 8 clusters' worth of powers and output)
  double best = 1e300;
  for (int n = kAtRows; n < rows + kAtRows; n += kAtRows) {
    const int split = (rows + n - 1) / n;
    const double cost = std::ceil((double)blocks.size() * split / ((double)p->n_sm * bps)) * (n + 8.0);
    if (cost < best * 0.999) {
      best = cost;
      s.rows_per_chunk = n;
      s.split = split;
    }
  }
  const bool ok = up_host(&s.up, upv) && up_host(&s.down, dnv) && up_host(&s.g_blocks, gb) &&
                  up_host(&s.row_blk, row_blk) && up_host(&s.blocks, blocks) && up_host(&s.rho, rho) &&
                  cudaMalloc(&s.g_part, (size_t)part * sizeof(float2)) == cudaSuccess &&
                  cudaMalloc(&s.g8, (size_t)g8 * sizeof(float)) == cudaSuccess;
  if (!ok) {  // no room: the direct kernel needs none of it
    cudaGetLastError();
    release_cluster_adjoint(s);
    return SCATTER_OK;
  }
  s.n_blocks = (int)blocks.size();
  s.n_g = (int)gb.size();
  p->base_bytes += part * 8 + g8 * 4 + (int64_t)(K * 20 + gb.size() * sizeof(ClGBlock) + rows * 4 + blocks.size() * sizeof(AdjBlock));
  s.active = true;
  return SCATTER_OK;
}

scatter_status launch_cluster_adjoint(scatter_plan_t p, const float2* gf, float* partial, cudaStream_t st) {
  const ClAdjState& s = p->cl.adj;
  ClAdjArgs a{};
  a.c = cluster_args(p);
  a.c.rho = s.rho;
  a.gf = gf;
  a.g_blocks = s.g_blocks;
  a.row_blk = s.row_blk;
  a.up = s.up;
  a.down = s.down;
  a.g_part = s.g_part;
  a.g8 = s.g8;
  a.blocks = s.blocks;
  a.rows_per_chunk = s.rows_per_chunk;
  for (int d = 0; d < 3; ++d) a.emax[d] = s.emax[d];
  a.partial = partial;
  a.n_slots = p->n_slots;
  timing_begin(p, st);  // to the end of the direct kernel, which may do the work instead
  k_cl_gsum<<<dim3((unsigned)s.n_g, (unsigned)((p->n_species + 1) / 2)), kGThreads, 0, st>>>(a);
  k_cl_gfin<<<dim3((unsigned)p->cl.first.rows, (unsigned)p->n_species), kGThreads, 0, st>>>(a);
  k_cl_adj<<<dim3((unsigned)s.n_blocks, (unsigned)s.split), kAtThreads, s.smem, st>>>(a);
  p->last_launches += 3;
  return cuda_status(cudaGetLastError(), "cluster adjoint launch");
}

void release_cluster_adjoint(ClAdjState& s) {
  for (void* b : {(void*)s.blocks, (void*)s.g_blocks, (void*)s.row_blk, (void*)s.up, (void*)s.down, (void*)s.rho,
                  (void*)s.g_part, (void*)s.g8})
    if (b) cudaFree(b);
  s = ClAdjState{};
}

}  // namespace scatter
