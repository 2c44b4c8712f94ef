// Adjoint of Eq. 2 on axis-aligned grids, on the tensor cores.
//
// With gF_s(S) = g(S) f_s(|S|) e^{2 i pi s.t} (k_loss_weights) the gradient is
//   dL/dr_j = -2 pi w_j sum_S S Im( gF_s(S) e^{2 i pi (c_j + s.x'_j)} ).
// On a grid s = (s_a, s_b, s_c) the exponential separates as in the forward.
// Define, for the weights omega_0 = 1, omega_1 = s_b, omega_2 = s_c,
//   U_w[a, j] = sum_{(b,c)} gF_s[a,b,c] omega_w(b,c) e^{2 i pi (s_b y'_j + s_c z'_j)}
// a complex matrix product of (a, w) rows by atom columns over the n1 n2
// points of each a-plane.  Every sum the gradient needs is then a short sum
// over a with E[a, j] = e^{2 i pi s_a x'_j}:
//   V = sum_a E U_0,  W_a = sum_a s_a E U_0,  W_b = sum_a E U_1,  W_c = sum_a E U_2
//   dL/dr_j,d = -2 pi w_j Im( e^{2 i pi c_j} (H_d V + W_d) ).
// The product runs on k_sep with the operands' roles swapped: A holds gF
// omega (f16 hi/lo, rows 2 pa + {Re, Im} for pa = w n0 + a, K = points),
// B is formed per step from the columns' atoms (y', z') and the step's 16
// point records (s_b, s_c).  gF spans many decades across a map, so every
// A row is scaled by a power of two that puts its largest element near
// 2^14 (f16 keeps 22 bits of it in hi + lo down to 2^-17 of the row's
// maximum); the epilogue undoes the scale exactly.
//
// Where the (k, l) axes are symmetric about their middles (offsets +-d of a
// point p and its mirror p', phases +-phi_p around the middle's) the products
// of the two share their cos and sin:
//   U_w e^{-2 pi i (mid - H).r'} = sum over half the points of P cos phi + i M sin phi,
//   P, M = omega(p) gF(p) +- omega(p') gF(p'),  omega_1 = d_b, omega_2 = d_c
// (odd, so their sums take the other sign): the same rows over half the K, half
// the MMAs, formation and A table.  The epilogue turns the result by the
// middle's phase and adds the middle to H.
//
// k_adj_sep_scale  per (species, a): the exponents of the three rows' scales
// k_adj_sep_tab    A blocks of every species in the tcgen05 no-swizzle layout
// k_sep            U for every (M-tile pair, 256-atom tile, point chunk)
// k_adj_sep_final  per atom: the sum over a and the chunks, gradient
#include <algorithm>
#include <cmath>
#include <vector>
#include "launch.h"
#include "sep_common.cuh"

namespace scatter {

constexpr int kAdjSepRowMax = 14;  // binary exponent of a row's largest |element| after scaling

// P and M of a point (fold: of the pair p, p'; else P = M = omega gF), for the
// weight row w; gp, gm: gF at p and p', om: omega_w(p).
struct AdjPair {
  float2 P, M;
};
__device__ __forceinline__ AdjPair adj_pair(float2 gp, float2 gm, float om, int w, bool fold, bool self) {
  AdjPair r;
  if (!fold) {
    r.P = r.M = make_float2(gp.x * om, gp.y * om);
  } else if (self) {  // the middle point: phase 0, offsets 0
    r.P = w == 0 ? gp : make_float2(0.f, 0.f);
    r.M = make_float2(0.f, 0.f);
  } else {
    const float2 sum = make_float2(gp.x + gm.x, gp.y + gm.y), dif = make_float2(gp.x - gm.x, gp.y - gm.y);
    r.P = w == 0 ? sum : make_float2(om * dif.x, om * dif.y);
    r.M = w == 0 ? dif : make_float2(om * sum.x, om * sum.y);
  }
  return r;
}

// x 2^k in two exact steps (k beyond a float's exponents; a subnormal result
// may round twice): ldexpf without its branches
__device__ __forceinline__ float scale2(float x, int k) {
  const int k1 = k / 2;
  return x * __int_as_float((k1 + 127) << 23) * __int_as_float((k - k1 + 127) << 23);
}

// One CTA per (species, a): the largest |Re|, |Im| of the three weights' P and
// M over the plane's points, as the exponent e of 2^e >= max (frexp), stored
// as the shift k = e - kAdjSepRowMax of the row's scale 2^k.  Latency-bound
// (128 planes of 131 KB on the 128^3 cube): 1024 threads keep the loads in
// flight, 37.7 us with 256, 7.3 us with 1024.
__global__ void __launch_bounds__(1024) k_adj_sep_scale(const float2* __restrict__ gf, const float4* __restrict__ rec,
                                                        int64_t n0, int64_t nbc, int64_t n_k, int fold, int64_t n_s,
                                                        int* __restrict__ sexp, const CallGate gate) {
  if (within(gate, 0)) return;
  const int64_t sp = blockIdx.x / n0, a = blockIdx.x % n0;
  const float2* row = gf + sp * n_s + a * nbc;
  float m[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
  for (int64_t p = threadIdx.x; p < n_k; p += blockDim.x) {
    const float2 gp = row[p], gm = fold ? row[nbc - 1 - p] : gp;
    const float4 r = rec[p];
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      const AdjPair q = adj_pair(gp, gm, w == 0 ? 1.f : w == 1 ? r.y : r.z, w, fold, 2 * p + 1 == nbc);
      m[w] = fmaxf(m[w], fmaxf(fmaxf(fabsf(q.P.x), fabsf(q.P.y)), fmaxf(fabsf(q.M.x), fabsf(q.M.y))));
    }
  }
  __shared__ float sh[3][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int w = 0; w < 3; ++w) {
    for (int o = 16; o > 0; o >>= 1) m[w] = fmaxf(m[w], __shfl_xor_sync(0xffffffffu, m[w], o));
    if (lane == 0) sh[w][warp] = m[w];
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    float v = 0.f;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) v = fmaxf(v, sh[threadIdx.x][q]);
    int e = 0;
    if (v > 0.f && v <= 3.0e38f) frexpf(v, &e);  // zero or non-finite rows: scale 2^-14
    sexp[(sp * 3 + threadIdx.x) * n0 + a] = e - kAdjSepRowMax;
  }
}

struct AdjSepTabArgs {
  const float2* gf;     // [n_species][M] gF_s, M = n0 n1 n2 row-major
  const float4* rec;    // point records (0, omega_1, omega_2, 0)
  const int* sexp;      // [n_species][3][n0] row scale exponents
  int64_t n0, nbc, n_k, n_s;  // n_k: points (fold: mirror pairs) of a plane
  int fold;
  int64_t n_ksteps, n_mt, n_mp;
  int64_t total;        // threads: n_species x n_mt x n_ksteps x 512
  uint4* A;             // [species][n_mp][n_ksteps][2 tiles][hi|lo][4 kb][16 mg][8 rows] of 16 B
  CallGate gate;
};

// One thread per 16-byte row of a core matrix (4 points x Re/Im of one A row).
// Row 2 pa: (Pr, -Mi); row 2 pa + 1: (Pi, Mr) with P, M scaled by 2^-k.
__global__ void k_adj_sep_tab(const AdjSepTabArgs t) {
  if (within(t.gate, 0)) return;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= t.total) return;
  const int r = (int)(i % 8), mg = (int)((i / 8) % 16), kb = (int)((i / 128) % 4);
  const int64_t ks = (i / 512) % t.n_ksteps, mt = (i / (512 * t.n_ksteps)) % t.n_mt;
  const int64_t sp = i / (512 * t.n_ksteps * t.n_mt);
  const int64_t m = mt * kSepM + mg * 8 + r;
  const int64_t pa = m >> 1;
  const int ri = (int)(m & 1);
  const bool in_row = pa < 3 * t.n0;
  const int w = in_row ? (int)(pa / t.n0) : 0;
  const int64_t a = in_row ? pa % t.n0 : 0;
  const int k = in_row ? t.sexp[(sp * 3 + w) * t.n0 + a] : 0;
  const float2* row = t.gf + sp * t.n_s + a * t.nbc;
  float v[8];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int64_t p = ks * kSepStep + kb * 4 + q;
    float c0 = 0.f, c1 = 0.f;
    if (in_row && p < t.n_k) {
      const float2 gp = row[p], gm = t.fold ? row[t.nbc - 1 - p] : gp;
      const float4 rc = t.rec[p];
      const AdjPair g = adj_pair(gp, gm, w == 0 ? 1.f : w == 1 ? rc.y : rc.z, w, t.fold, 2 * p + 1 == t.nbc);
      c0 = scale2(ri ? g.P.y : g.P.x, -k);
      c1 = scale2(ri ? g.M.x : -g.M.y, -k);
    }
    v[2 * q] = c0;
    v[2 * q + 1] = c1;
  }
  uint4 hi, lo;
  split2(v[0], v[1], hi.x, lo.x);
  split2(v[2], v[3], hi.y, lo.y);
  split2(v[4], v[5], hi.z, lo.z);
  split2(v[6], v[7], hi.w, lo.w);
  uint4* blk = t.A + (((sp * t.n_mp + (mt >> 1)) * t.n_ksteps + ks) * kSepPair + (mt & 1)) * (kSepABytes / 16);
  const int64_t off = (int64_t)(kb * 16 + mg) * 8 + r;
  blk[off] = hi;
  blk[512 + off] = lo;
}

struct AdjSepFinalArgs {
  const float* partial;    // [chunk] blocked as sep_part_off: rows 2 (w n0 + a) + {Re, Im}, columns slots
  int64_t chunk_floats, n_cb;
  int n_chunks;
  const Segment* ntiles;
  const int* sexp;
  const float4* atom4;
  const float4* atom_lo;
  const float* atom_w;
  const int32_t* slot_src;
  const float* axis_s;
  int64_t n0, n_slots;
  float H[3], H_lo[3];     // as double-floats; fold: k and l at the middles of their axes
  float mid[2], mid_lo[2]; // fold: those middles - H as double-floats, else 0
  float* grad;             // [n_atoms][3] caller order
  CallGate gate;
};

// One warp per four atom slots: lane 2 i + ri holds row (Re or Im) of a = a0 + i
// of a block of 16 values, so a read of one weight's rows is 512 contiguous
// bytes (the partials keep four columns of a 32-row block together).  One
// exchange gives the even lane (Re, Im) of the first two slots and the odd
// lane of the last two.  The sum over a (and over the point chunks) runs with
// FP32 products and double-float (TwoSum) FP32 sums (FP64 runs at ~1/75 of
// the FP32 rate here; the 3 n0 terms are already contracted values whose own
// error is ~1e-6).  Only Im(e^{2 pi i theta} X) is wanted, so the atom's phase
// c + (mid - H).r' joins the row factor's (exactly reduced, MUFU sin/cos,
// |error| < 4e-7) and four imaginary sums are enough; the 16 lanes' sums meet
// in a fixed order.  116 us on the 102,400-atom cube x 128^3 (315 MB of
// partials, 47 us at the copy rate; 217 us with one thread per slot, whose
// reads were 16-byte pieces).
constexpr int kAdjFinalWarps = 8;
__global__ void __launch_bounds__(32 * kAdjFinalWarps) k_adj_sep_final(const AdjSepFinalArgs f) {
  if (within(f.gate, 0)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = lane >> 1, ri = lane & 1;
  const Segment t = f.ntiles[blockIdx.x];
  const int64_t slot0 = t.begin + 4 * ((int64_t)blockIdx.y * kAdjFinalWarps + warp);
  if (slot0 >= t.end) return;  // segments are multiples of 32 slots
  const int64_t slot = slot0 + 2 * ri;  // this lane's two slots
  const int64_t rows = 3 * f.n0;
  const int* se = f.sexp + (int64_t)t.species * rows;
  float x[2], th[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const float4 at = f.atom4[slot + u], lo = f.atom_lo[slot + u];
    x[u] = at.x;
    const float py = dev::frac_of_product2(f.mid[0], f.mid_lo[0], at.y) + f.mid[0] * lo.y;
    const float pz = dev::frac_of_product2(f.mid[1], f.mid_lo[1], at.z) + f.mid[1] * lo.z;
    th[u] = dev::frac_rn(at.w + (py + pz));
  }
  // sums of Im P_0, s_a Im P_0, Im P_1, Im P_2
  dev::DFloatSum sum[2][4];
  const float* base = f.partial + sep_part_off(0, slot0, f.n_cb);
  const int64_t row_block = f.n_cb << 10;  // floats per 32-row block
  for (int64_t a0 = 0; a0 < f.n0; a0 += 16) {
    const int64_t a = a0 + i;
    const bool ok = a < f.n0;
    float4 U[3];
    int k[3];
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      U[w] = make_float4(0.f, 0.f, 0.f, 0.f);
      k[w] = 0;
      if (ok) {
        const int64_t m = 2 * (w * f.n0 + a) + ri;
        const float* pc = base + (m >> 5) * row_block + ((m & 31) << 2);
        U[w] = __ldcs(reinterpret_cast<const float4*>(pc));
        for (int c = 1; c < f.n_chunks; ++c) {
          const float4 v = __ldcs(reinterpret_cast<const float4*>(pc + c * f.chunk_floats));
          U[w].x += v.x;
          U[w].y += v.y;
          U[w].z += v.z;
          U[w].w += v.w;
        }
        k[w] = se[w * f.n0 + a];
      }
    }
    const float sa = ok ? f.axis_s[a] : 0.f;
    float sn[2], cs[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) dev::sincos_cycles_mufu(dev::frac_rn(dev::frac_of_product(sa, x[u]) + th[u]), &sn[u], &cs[u]);
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      const float rx = __shfl_xor_sync(0xffffffffu, ri ? U[w].x : U[w].z, 1);
      const float ry = __shfl_xor_sync(0xffffffffu, ri ? U[w].y : U[w].w, 1);
      const float re[2] = {ri ? rx : U[w].x, ri ? ry : U[w].y}, im[2] = {ri ? U[w].z : rx, ri ? U[w].w : ry};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float v = scale2(fmaf(cs[u], im[u], sn[u] * re[u]), k[w]);
        sum[u][w == 0 ? 0 : w + 1].add(v);
        if (w == 0) sum[u][1].add(sa * v);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int o = 2; o < 32; o <<= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, sum[u][q].hi, o), l = __shfl_xor_sync(0xffffffffu, sum[u][q].lo, o);
        sum[u][q].add(h);
        sum[u][q].lo = __fadd_rn(sum[u][q].lo, l);
      }
  if (i > 0) return;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int32_t src = f.slot_src[slot + u];
    if (src < 0) continue;
    // -2 pi w (H_d V + W_d) in double-floats (an FP64 operation of two lanes
    // costs the whole warp's 19 cycles here), H_d exact in two floats
    const float w = f.atom_w[slot + u];
    const dev::DFloatSum v = sum[u][0];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      dev::DFloatSum g = sum[u][d + 1];
      g.add_product(f.H[d], v.hi);
      g.lo = __fadd_rn(g.lo, fmaf(f.H[d], v.lo, f.H_lo[d] * v.hi));
      f.grad[3 * (int64_t)src + d] = g.times_minus_two_pi(w);
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

namespace {

constexpr size_t kAdjSepMaxBytes = (size_t)32 << 30;  // A tables + partials; larger maps use the FP32 adjoint

// Point chunks (split over K) that minimise waves x steps per CTA plus the
// cost of one more set of partials (written once, read once).
// A folded plane has half the steps: its chunks may be half as long, which
// keeps the points per chunk and with them the accumulators' truncation no
// larger than the direct form's.
int adj_sep_split(const scatter_plan_s* p, int64_t tiles, int64_t n_ksteps, size_t part_bytes, bool fold) {
  const double cap = (double)p->n_sm;
  const double part_steps = 2.0 * (double)part_bytes / 6.0e12 / 1.0e-6;  // ~1 us per step
  double best = 1e300;
  int best_k = 1;
  for (int k = 1; k <= 64; ++k) {
    if (k > 1 && (double)n_ksteps / k < (fold ? 32 : 64)) break;
    const double cost = std::ceil((double)tiles * k / cap) * ((double)n_ksteps / k + 40.0) + (k - 1) * part_steps;
    if (cost < best * 0.995) {
      best = cost;
      best_k = k;
    }
  }
  return best_k;
}

}  // namespace

bool adjoint_sep_applicable(const scatter_plan_s* p) {
  return p->path == SCATTER_PATH_SEPARABLE && p->s_kind == SCATTER_S_GRID && p->batch == 1 &&
         p->n_s > 0 && p->n_slots % kSepStep == 0;
}

namespace {

// The (k, l) plane folds over its middle where both axes are symmetric.
bool adj_folds(const scatter_plan_s* p, double (&mid)[2]) {
  return !p->adj_no_fold && sep_axis_middle(p->axis_host[1], p->inst[0].H[1], &mid[0]) &&
         sep_axis_middle(p->axis_host[2], p->inst[0].H[2], &mid[1]);
}

}  // namespace

double adjoint_sep_group(const scatter_plan_s* p, bool fold) {
  double mid[2];
  fold = fold && adj_folds(p, mid);
  const int64_t nbc = p->n_axis[1] * p->n_axis[2], n_k = fold ? (nbc + 1) / 2 : nbc;
  const int64_t n_ksteps = (n_k + kSepStep - 1) / kSepStep;
  const int64_t n_mt = (2 * 3 * p->n_axis[0] + kSepM - 1) / kSepM;
  int64_t tiles = 0;
  for (const Segment& sg : p->all_segs) tiles += (sg.end - sg.begin + kSepN - 1) / kSepN;
  const int split = adj_sep_split(p, (n_mt + 1) / 2 * tiles, n_ksteps,
                                  (size_t)sep_part_floats(n_mt, p->n_slots) * sizeof(float), fold);
  const int64_t per = (n_ksteps + split - 1) / split, full = per / kSepFlush, rest = per % kSepFlush;
  return (double)(full * kSepFlush * kSepFlush + rest * rest) / (double)per;
}

// Tables and tiling of the tensor-core adjoint; leaves p->adj_sep false (and
// allocates nothing) when the map is too large for its workspace.
scatter_status prepare_adjoint_sep(scatter_plan_s* p) {
  p->adj_sep = false;
  if (!adjoint_sep_applicable(p)) return SCATTER_OK;
  const int64_t n0 = p->n_axis[0], n1 = p->n_axis[1], n2 = p->n_axis[2];
  const int64_t nbc = n1 * n2;
  double mid[2] = {0, 0};
  const bool fold = adj_folds(p, mid);
  const int64_t n_k = fold ? (nbc + 1) / 2 : nbc;
  const int64_t n_ksteps = (n_k + kSepStep - 1) / kSepStep;
  const int64_t n_mt = (2 * 3 * n0 + kSepM - 1) / kSepM;
  const int64_t n_mp = (n_mt + 1) / 2;
  // N tiles: 256 slots of one species
  std::vector<Segment> ntiles;
  for (const Segment& sg : p->all_segs) {
    if (sg.instance != 0) continue;
    for (int64_t b = sg.begin; b < sg.end; b += kSepN)
      ntiles.push_back(Segment{b, std::min(sg.end, b + (int64_t)kSepN), sg.species, 0});
  }
  if (ntiles.empty()) return SCATTER_OK;  // no atoms: the FP32 path writes the empty gradient
  const size_t a_bytes = (size_t)p->n_species * (size_t)n_mp * (size_t)n_ksteps * kSepPair * kSepABytes;
  const size_t part1 = (size_t)sep_part_floats(n_mt, p->n_slots) * sizeof(float);
  const int split = adj_sep_split(p, n_mp * (int64_t)ntiles.size(), n_ksteps, part1, fold);
  std::vector<Segment> chunks;
  const int64_t per = (n_ksteps + split - 1) / split;
  for (int64_t b = 0; b < n_ksteps; b += per)
    chunks.push_back(Segment{b * kSepStep, std::min(n_ksteps, b + per) * kSepStep, 0, 0});
  const size_t part_bytes = chunks.size() * part1;
  if (a_bytes + part_bytes > kAdjSepMaxBytes) return SCATTER_OK;
  if (ntiles.size() * (size_t)n_mp > 0x7fffffffULL || chunks.size() > 65535) return SCATTER_OK;
  // point records (0, s_b, s_c, 0), folded (0, d_b, d_c, 0), zero past the last point
  std::vector<float4> rec((size_t)n_ksteps * kSepStep, make_float4(0.f, 0.f, 0.f, 0.f));
  float smax_b = 0.f, smax_c = 0.f;
  const std::vector<double>&k64 = p->axis_host[1], &l64 = p->axis_host[2];
  for (int64_t q = 0; q < n_k; ++q) {
    const int64_t b = q / n2, c = q % n2;
    const float sb = (float)(fold ? 0.5 * (k64[b] - k64[n1 - 1 - b]) : k64[b] - p->inst[0].H[1]);
    const float sc = (float)(fold ? 0.5 * (l64[c] - l64[n2 - 1 - c]) : l64[c] - p->inst[0].H[2]);
    rec[q] = make_float4(0.f, sb, sc, 0.f);
    smax_b = std::max(smax_b, std::fabs(sb));
    smax_c = std::max(smax_c, std::fabs(sc));
  }
  const size_t gf_bytes = (size_t)p->n_species * (size_t)p->n_s * sizeof(float2);
  const size_t sexp_bytes = (size_t)p->n_species * 3 * (size_t)n0 * sizeof(int);
  cudaError_t e;
  if ((e = cudaMalloc(&p->d.adj_gf, gf_bytes)) != cudaSuccess) return cuda_status(e, "cudaMalloc adjoint gF");
  if ((e = cudaMalloc(&p->d.adj_sexp, sexp_bytes)) != cudaSuccess) return cuda_status(e, "cudaMalloc row scales");
  if ((e = cudaMalloc(&p->d.adj_sepA, a_bytes)) != cudaSuccess) return cuda_status(e, "cudaMalloc adjoint A");
  if ((e = cudaMemset(p->d.adj_sepA, 0, a_bytes)) != cudaSuccess) return cuda_status(e, "memset adjoint A");
  if ((e = cudaMalloc(&p->d.adj_sep_partial, part_bytes)) != cudaSuccess)
    return cuda_status(e, "cudaMalloc adjoint partials");
  if ((e = cudaMalloc(&p->d.adj_rec, rec.size() * sizeof(float4))) != cudaSuccess)
    return cuda_status(e, "cudaMalloc point records");
  if ((e = cudaMalloc(&p->d.adj_ntiles, ntiles.size() * sizeof(Segment))) != cudaSuccess)
    return cuda_status(e, "cudaMalloc atom tiles");
  if ((e = cudaMalloc(&p->d.adj_kchunks, chunks.size() * sizeof(Segment))) != cudaSuccess)
    return cuda_status(e, "cudaMalloc point chunks");
  if ((e = cudaMemcpy(p->d.adj_rec, rec.data(), rec.size() * sizeof(float4), cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemcpy(p->d.adj_ntiles, ntiles.data(), ntiles.size() * sizeof(Segment), cudaMemcpyHostToDevice)) !=
          cudaSuccess ||
      (e = cudaMemcpy(p->d.adj_kchunks, chunks.data(), chunks.size() * sizeof(Segment), cudaMemcpyHostToDevice)) !=
          cudaSuccess)
    return cuda_status(e, "adjoint tables upload");
  if ((e = sep_prepare_kernel()) != cudaSuccess) return cuda_status(e, "separable shared memory attribute");
  if (const scatter_status ss = sep_prepare_side(p, n_mt); ss != SCATTER_OK) return ss;
  p->base_bytes += (int64_t)(gf_bytes + sexp_bytes + a_bytes + part_bytes + rec.size() * sizeof(float4) +
                             (ntiles.size() + chunks.size()) * sizeof(Segment));
  p->adj_sep_fold = fold;
  p->adj_sep_k = n_k;
  for (int d = 0; d < 2; ++d) p->adj_sep_mid[d] = fold ? mid[d] - p->inst[0].H[d + 1] : 0.0;
  p->adj_sep_ksteps = n_ksteps;
  p->adj_sep_mt = n_mt;
  p->adj_sep_ntiles = (int32_t)ntiles.size();
  p->adj_sep_chunks = (int32_t)chunks.size();
  p->adj_sep_smax[0] = smax_b;
  p->adj_sep_smax[1] = smax_c;
  p->adj_sep = true;
  return SCATTER_OK;
}

// After k_loss_weights wrote gF (p->d.adj_gf): scales, A tables, the
// contraction and the per-atom epilogue, all on `st`.
scatter_status launch_adjoint_sep(scatter_plan_t p, float* grad, cudaStream_t st, const CallGate& gate) {
  const int64_t n0 = p->n_axis[0], n1 = p->n_axis[1], n2 = p->n_axis[2];
  const int64_t n_mp = (p->adj_sep_mt + 1) / 2;
  k_adj_sep_scale<<<(unsigned)(p->n_species * n0), 1024, 0, st>>>(p->d.adj_gf, p->d.adj_rec, n0, n1 * n2, p->adj_sep_k,
                                                                   p->adj_sep_fold, p->n_s, p->d.adj_sexp, gate);
  AdjSepTabArgs t{};
  t.gf = p->d.adj_gf;
  t.rec = p->d.adj_rec;
  t.sexp = p->d.adj_sexp;
  t.n0 = n0;
  t.nbc = n1 * n2;
  t.n_k = p->adj_sep_k;
  t.fold = p->adj_sep_fold;
  t.n_s = p->n_s;
  t.n_ksteps = p->adj_sep_ksteps;
  t.n_mt = p->adj_sep_mt;
  t.n_mp = n_mp;
  t.total = (int64_t)p->n_species * p->adj_sep_mt * p->adj_sep_ksteps * 512;
  t.A = static_cast<uint4*>(p->d.adj_sepA);
  t.gate = gate;
  k_adj_sep_tab<<<(unsigned)((t.total + 255) / 256), 256, 0, st>>>(t);
  SepArgs a{};
  a.A = static_cast<const uint4*>(p->d.adj_sepA);
  a.a_sp_stride = n_mp * p->adj_sep_ksteps * (int64_t)(kSepPair * kSepABytes / 16);
  a.rec = p->d.adj_rec;
  a.chunks = p->d.adj_kchunks;
  a.ntiles = p->d.adj_ntiles;
  a.atom4 = p->d.atom4;
  a.axis_s = p->d.axis_s;
  a.bbox = p->d.inst_bbox;
  a.shift = p->d.inst_shift;
  a.smax_b = p->adj_sep_smax[0];
  a.smax_c = p->adj_sep_smax[1];
  a.n0 = n0;
  a.n1 = n1;
  a.n2 = n2;
  a.n_cb = (p->n_slots + 31) / 32;
  a.chunk_floats = sep_part_floats(p->adj_sep_mt, p->n_slots);
  a.n_steps = p->adj_sep_ksteps;
  a.n_mt = p->adj_sep_mt;
  a.partial = p->d.adj_sep_partial;
  a.status = p->d.status;
  a.gate = gate;
  dim3 grid((unsigned)(n_mp * p->adj_sep_ntiles), (unsigned)p->adj_sep_chunks);
  if (!gate.rmax2) timing_begin(p, st);
  const cudaError_t le = sep_launch_core(a, grid, st, p->side_stream, p->side_fork, p->side_join);
  timing_end(p, st);
  if (le != cudaSuccess) return cuda_status(le, "adjoint contraction launch");
  AdjSepFinalArgs f{};
  f.partial = p->d.adj_sep_partial;
  f.chunk_floats = sep_part_floats(p->adj_sep_mt, p->n_slots);
  f.n_cb = (p->n_slots + 31) / 32;
  f.n_chunks = p->adj_sep_chunks;
  f.ntiles = p->d.adj_ntiles;
  f.sexp = p->d.adj_sexp;
  f.atom4 = p->d.atom4;
  f.atom_lo = p->d.atom_lo;
  f.atom_w = p->d.atom_w;
  f.slot_src = p->d.slot_src;
  f.axis_s = p->d.axis_s;
  f.n0 = n0;
  f.n_slots = p->n_slots;
  for (int d = 0; d < 3; ++d) {
    const double h = p->inst[0].H[d] + (d > 0 ? p->adj_sep_mid[d - 1] : 0.0);
    f.H[d] = (float)h;
    f.H_lo[d] = (float)(h - (double)f.H[d]);
  }
  for (int d = 0; d < 2; ++d) {
    f.mid[d] = (float)p->adj_sep_mid[d];
    f.mid_lo[d] = (float)(p->adj_sep_mid[d] - (double)f.mid[d]);
  }
  f.grad = grad;
  f.gate = gate;
  k_adj_sep_final<<<dim3((unsigned)p->adj_sep_ntiles, kSepN / (4 * kAdjFinalWarps)), 32 * kAdjFinalWarps, 0, st>>>(f);
  p->last_launches += 3 + sep_core_launches(p->adj_sep_mt);
  return cuda_status(cudaGetLastError(), "adjoint launch");
}

}  // namespace scatter
