// The (n, n+1) IIM operator w = L_Omega u (+ L_Gamma u_Gamma), paper Sec. 2.3, Eq. 12.
//
// Two kernels:
//   k_ho_ghost    eight lanes per control point: u_c (Dirichlet data, Neumann elimination
//                 Eqs. 5-6, or the interface closure Eqs. 9-11) and the w ghost values
//                 p_c(x_g) = s_c u_c + sum s_a u_a of Eq. 4;
//   k_ho_apply    every node: beta_sigma/h^2 sum_axes sum_j a_j u_{i+j e}.  Plain nodes (no
//                 control point and no box face within w nodes along any axis) read only u
//                 and one class byte.  Affected nodes are left to other blocks of the same
//                 launch: a lane per direction, neighbours outside phase sigma (or outside
//                 the box) contributing 0, plus a_j p_c(x_{i+j e}) for every out-of-phase
//                 offset past the first control point of each walk, and the outer-box ghosts.
// k_ho_apply is launched as a programmatic dependent of k_ho_ghost: its plain blocks need
// nothing from it and run beside it, its affected blocks wait for it and are spread over
// the rest of the grid, so that neither the ghost values nor the corrections add to the time of
// the plain nodes.  Three kernels, the ghosts on a second stream between two events and the
// corrections after both, took 17.2 us for a 64^2 circle and 57.5 us for the order-6 star at
// 1024^2; the two take 9.4 to 12.5 and 38.8.
// The plain nodes are FP64 and bound by the FP64 pipe on GB300 (2 FMA/clk/SM), so they are
// written to use the fewest FP64 operations: neighbours at equal |j| are summed first, then
// one FMA per |j| with beta/h^2 folded into the coefficients.  Large 3D grids sum in fixed point
// instead (k_ho_tiles, op_tile.cuh).
#include <mutex>
#include <string>

#include "engine.cuh"

namespace iim {

#include "op_tile.cuh"

template <int D, int W>
__device__ __forceinline__ void ho_stencil_node(const GridView& g, const StencilCoef& C, int interface_,
                                                const double* __restrict__ u, const uint8_t* __restrict__ phase,
                                                double* __restrict__ w, int64_t i) {
  const int n = g.n;
  const uint8_t ph = phase[i];
  if (!interface_ && !ph) { w[i] = 0.0; return; }
  int m[3];
  m[0] = (int)(i % n);
  int64_t r = i / n;
  m[1] = (int)(r % n);
  m[2] = D > 2 ? (int)(r / n) : 0;
  const int sig = ph ? 1 : 0;
  double acc = C.c0[sig] * u[i];
#pragma unroll
  for (int j = 1; j <= W; ++j) {
    double v[2 * D];
#pragma unroll
    for (int ax = 0; ax < D; ++ax) {
      const int64_t st = ax == 0 ? 1 : (ax == 1 ? (int64_t)n : (int64_t)n * n);
      v[2 * ax] = 0.0;
      v[2 * ax + 1] = 0.0;
      if (m[ax] - j >= 0) {
        int64_t nb = i - j * st;
        double t = u[nb];
        v[2 * ax] = phase[nb] == ph ? t : 0.0;
      }
      if (m[ax] + j < n) {
        int64_t nb = i + j * st;
        double t = u[nb];
        v[2 * ax + 1] = phase[nb] == ph ? t : 0.0;
      }
    }
    double s = v[0];
#pragma unroll
    for (int k = 1; k < 2 * D; ++k) s += v[k];
    acc = fma(C.cj[sig][j - 1], s, acc);
  }
  w[i] = acc;
}

// Eight lanes per control point: each lane accumulates an eighth of the X_c terms
// of every row (sequential FMAs, no per-term reduction), then two shuffle steps
// combine the quarters.  Boundary problems: rows 0..w-1 of fit c.  Interface
// problems: rows 0..w of fits 2c (+) and 2c+1 (-), then the closure of Eqs. 9-11.
constexpr int kGhostLanes = 8, kGhostThreads = 64;

__device__ inline double quad_sum(double v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4, kGhostLanes);
  v += __shfl_xor_sync(0xffffffffu, v, 2, kGhostLanes);
  v += __shfl_xor_sync(0xffffffffu, v, 1, kGhostLanes);
  return v;
}

template <int W>
__device__ __forceinline__ void ho_ghost_body(const GhostParams& P, const double* __restrict__ u, int gid) {
  const int c = gid / kGhostLanes, q = gid % kGhostLanes;
  const int K = *P.K;
  const bool live = c < K;                       // every lane takes part in the shuffles
  const int rows = W + 1;
  const int nsides = P.interface_ ? 2 : 1;
  double acc[2][W + 1];
#pragma unroll
  for (int sd = 0; sd < 2; ++sd)
#pragma unroll
    for (int k = 0; k <= W; ++k) acc[sd][k] = 0.0;
#pragma unroll
  for (int sd = 0; sd < 2; ++sd) {
    if (sd >= nsides || !live) continue;
    const int f = P.interface_ ? 2 * c + sd : c;
    const int R = P.fit_R[f];
    const int32_t* nodes = P.fit_nodes + (size_t)f * P.rcap;
    const double* coef = P.fit_coef + (size_t)f * rows * P.rcap;
    const int nr = P.interface_ ? W + 1 : W;
    if (!u) continue;                            // u = 0: the data alone
#pragma unroll 4
    for (int a = q; a < R; a += kGhostLanes) {
      const double ua = u[nodes[a]];
#pragma unroll
      for (int k = 0; k <= W; ++k)
        if (k < nr) acc[sd][k] = fma(coef[(size_t)k * P.rcap + a], ua, acc[sd][k]);
    }
  }
  // the rows' sums over the lanes, transposed (FP64 additions hold a scheduler for 64 clocks: 3 for the two
  // rows of a 3D boundary point instead of 9, 7 instead of 24 for an order-6 interface point), then an
  // output per lane: 61 -> 55 us at 256^3 (98 k points), 24 -> 20.6 at 96^3, 16.5 -> 14.4 at 64^3 (interface)
  __shared__ double sums[kGhostThreads / kGhostLanes][2 * (W + 1)];
  double* sum = sums[threadIdx.x / kGhostLanes];
  if (P.interface_) lane_sums<kGhostLanes, 2 * (W + 1)>(&acc[0][0], q, sum);
  else lane_sums<kGhostLanes, W>(&acc[0][0], q, sum);
  __syncwarp();
  if (!live) return;
  if (!P.interface_) {
    const double data = P.with_data ? P.g[c] : 0.0;
    if (q < W) P.G[(size_t)c * W + q] = sum[q] + P.fit_cdat[(size_t)c * rows + q] * data;
    return;
  }
  if (q >= 2 * W) return;
  // Eqs. 9-11: S = b+ s+_c - b- s-_c ; ubar = -(b+ D+ - b- D-)/S
  const double *cp = P.fit_cdat + (size_t)(2 * c) * rows, *cm = P.fit_cdat + (size_t)(2 * c + 1) * rows;
  const double bp = P.beta_p, bm = P.beta_m;
  const double Sden = bp * cp[W] - bm * cm[W];
  double us = -(bp * sum[W] - bm * sum[2 * W + 1]) / Sden;         // this lane's side of it
  if (P.with_data) us += (P.j1[c] - (q < W ? bm * cm[W] : bp * cp[W]) * P.j0[c]) / Sden;
  const int k = q < W ? q : q - W;
  P.G[(size_t)(2 * c + (q < W ? 0 : 1)) * W + k] = sum[q < W ? k : W + 1 + k] + (q < W ? cp : cm)[k] * us;
}

template <int W>
__global__ void __launch_bounds__(kGhostThreads) k_ho_ghost(GhostParams P, const double* __restrict__ u) {
  pdl_trigger();                                 // k_ho_apply's plain blocks start beside this kernel
  ho_ghost_body<W>(P, u, blockIdx.x * blockDim.x + threadIdx.x);
}


// Ghost contribution of one direction (axis ax, side sd) at affected node t (node i, indices m, phase
// ph): a_j p_c(x_{i+j e}) over the out-of-phase offsets past the first control point, or the outer box.
// u = nullptr: the data's part alone (u = 0).
// coef.at(j, s): the stencil's coefficient at offset j s; coef.box(v, s): P.box_c's sum v on side s.
template <class Coef>
__device__ __forceinline__ double ho_direction(const CorrectParams& P, Coef coef, const double* __restrict__ u, int t,
                                               int64_t i, const int* m, uint8_t ph, int ax, int sd) {
  const GridView& g = P.g;
  const int n = g.n, d = g.dim, W = P.w;
  const int64_t st = ax == 0 ? 1 : (ax == 1 ? (int64_t)n : (int64_t)n * n);
  const int s = sd ? 1 : -1;
  const int fit = P.aff_fit[t * 2 * d + 2 * ax + sd];
  const int js = P.aff_j[t * 2 * d + 2 * ax + sd];
  double acc = 0.0;
  if (fit == -1 || fit >= P.nfit_cap) return acc;
  if (fit >= 0) {
    for (int j = js; j <= W; ++j) {
      const int pos = m[ax] + j * s;
      if (pos >= 0 && pos < n && P.phase[i + j * s * st] == ph) continue;   // back in phase: uses u
      acc = fma(coef.at(j, s), P.G[(size_t)fit * W + (j - js)], acc);
    }
    return acc;
  }
  // outer box: ghosts js .. w from the degree-q line polynomial through the face value and the nodes
  // 2..q+1 counted from the face, their weights summed beforehand (q + 1 operations for all of them)
  double face = 0.0;
  if (P.with_data) {
    int64_t off = 0, mul = 1;
    for (int k = 0; k < d; ++k) {
      if (k == ax) continue;
      off += m[k] * mul;
      mul *= n;
    }
    off += (int64_t)(2 * ax + sd) * mul;
    face = P.box[off];
  }
  acc = P.box_c[js - 1][0] * face;
  if (u)
    for (int mm = 2; mm <= P.q + 1; ++mm) {
      const int pos = s > 0 ? n - mm : mm - 1;
      acc = fma(P.box_c[js - 1][mm - 1], u[i + (int64_t)(pos - m[ax]) * st], acc);
    }
  return coef.box(acc, s);
}

// the operator's coefficients (even)
struct OpCoef {
  const CorrectParams& P;
  __device__ __forceinline__ double at(int j, int) const { return P.a[P.w + j]; }
  __device__ __forceinline__ double box(double v, int) const { return v; }
};

__device__ __forceinline__ void node_indices(int n, int d, int64_t i, int* m) {
  m[0] = (int)(i % n);
  const int64_t r = i / n;
  m[1] = (int)(r % n);
  m[2] = d > 2 ? (int)(r / n) : 0;
}

// the corrections alone, added to w (batched engine): one thread per affected node
__device__ __forceinline__ void ho_correct_body(const CorrectParams& P, const double* __restrict__ u,
                                                double* __restrict__ w, int t) {
  if (t >= *P.n_aff || t >= P.n_aff_cap) return;
  const int64_t i = P.aff_node[t];
  int m[3];
  node_indices(P.g.n, P.g.dim, i, m);
  const uint8_t ph = P.phase[i];
  double acc = 0.0;
  for (int k = 0; k < 2 * P.g.dim; ++k) acc += ho_direction(P, OpCoef{P}, u, t, i, m, ph, k >> 1, k & 1);
  w[i] = fma(P.scale[ph ? 1 : 0], acc, w[i]);
}

// Blocks of a launch over plain and affected nodes: after the first `first` plain blocks (by then the
// ghost kernel is done), every `every`-th block takes affected nodes until `aff` have, so that their
// chains of loads run beside plain blocks that keep the FP64 pipe busy (FP64 sums at 256^3, exterior:
// affected blocks in one piece 522 us, spread 518).
struct AffSplit {
  int plain, first, every, aff;
  // this block's index among the plain (>= 0) or affected (~index < 0) ones
  __device__ __forceinline__ int index(int b) const {
    const int r = b - first;
    if (r < 0) return b;
    const int k = r / every;
    if (k < aff && r - k * every == every - 1) return ~k;
    return b - min(k, aff);
  }
};

// The affected nodes: four lanes per node in 2D, one per direction (axis k / 2, side k & 1), because
// there are few of them and their chains of dependent loads are what a small application waits for;
// one thread per node in 3D, where the box faces alone have 6 w n^2 and the lanes' repeated FP64 sums
// would cost more than the plain nodes (256^3: 423 us
// against 83).
template <int D>
constexpr int aff_lanes() { return D == 2 ? 4 : 1; }

// Sums over the directions in their order (the separate corrections kernel's order): of w neighbour
// values at each offset, and of the ghost contributions.  v and part hold this thread's directions.
template <int D>
__device__ __forceinline__ double dir_sum(const double (&v)[2 * D / aff_lanes<D>()]) {
  double s;
  if constexpr (aff_lanes<D>() == 1) {
    s = v[0];
#pragma unroll
    for (int k = 1; k < 2 * D; ++k) s += v[k];
  } else {
    s = __shfl_sync(0xffffffffu, v[0], 0, 4);
#pragma unroll
    for (int k = 1; k < 2 * D; ++k) s += __shfl_sync(0xffffffffu, v[0], k, 4);
  }
  return s;
}

// Node of this thread among the affected ones, its neighbours in phase (v[j][direction], else 0) and
// its directions' ghost contributions.
template <int D, int W, int NT, class Coef>
struct Affected {
  static constexpr int LG = aff_lanes<D>(), ND = 2 * D / LG;
  int64_t i = 0;
  uint8_t ph = 0;
  int k0;                                // first of this thread's directions
  bool live;
  double v[W][ND], part[ND];
  __device__ __forceinline__ Affected(const CorrectParams& P, Coef coef, const double* __restrict__ u, int block) {
    const int t = (block * NT + (int)threadIdx.x) / LG, n = P.g.n;
    k0 = LG == 1 ? 0 : threadIdx.x % LG;
    live = t < min(*P.n_aff, P.n_aff_cap);
#pragma unroll
    for (int q = 0; q < ND; ++q) {
      part[q] = 0.0;
#pragma unroll
      for (int j = 0; j < W; ++j) v[j][q] = 0.0;
    }
    if (!live) return;
    i = P.aff_node[t];
    int m[3];
    node_indices(n, D, i, m);
    ph = P.phase[i];
#pragma unroll
    for (int q = 0; q < ND; ++q) {
      const int k = k0 + q, ax = k >> 1, s = k & 1 ? 1 : -1, ma = ax == 0 ? m[0] : (ax == 1 ? m[1] : m[2]);
      const int64_t st = ax == 0 ? 1 : (ax == 1 ? (int64_t)n : (int64_t)n * n);
      if (u)
#pragma unroll
        for (int j = 1; j <= W; ++j) {
          const int pos = ma + j * s;
          if (pos >= 0 && pos < n && P.phase[i + j * s * st] == ph) v[j - 1][q] = u[i + j * s * st];
        }
      part[q] = ho_direction(P, coef, u, t, i, m, ph, ax, k & 1);
    }
  }
};
template <int D, int W, int NT, class Coef>
__device__ __forceinline__ Affected<D, W, NT, Coef> affected(const CorrectParams& P, Coef coef,
                                                             const double* __restrict__ u, int block) {
  return Affected<D, W, NT, Coef>(P, coef, u, block);
}

template <int D, int W, int NT>
__device__ __forceinline__ void ho_affected(const CorrectParams& P, const StencilCoef& C, const double* __restrict__ u,
                                            double* __restrict__ w, int block) {
  const auto A = affected<D, W, NT>(P, OpCoef{P}, u, block);
  const bool plus = A.ph != 0;
  double acc = (plus ? C.c0[1] : C.c0[0]) * (A.live ? u[A.i] : 0.0);
#pragma unroll
  for (int j = 0; j < W; ++j) acc = fma(plus ? C.cj[1][j] : C.cj[0][j], dir_sum<D>(A.v[j]), acc);
  const double corr = dir_sum<D>(A.part);
  if (A.live && A.k0 == 0) w[A.i] = fma(plus ? P.scale[1] : P.scale[0], corr, acc);
}

// parts: 1 plain nodes, 2 affected nodes (both in an application; one alone for timing)
template <int D, int W>
__global__ void __launch_bounds__(256) k_ho_apply(CorrectParams P, StencilCoef C, const uint8_t* __restrict__ kind,
                                                  const double* __restrict__ u, double* __restrict__ w, AffSplit S) {
  const int b = S.index(blockIdx.x);
  if (b < 0) {
    pdl_wait();                            // the ghost values
    ho_affected<D, W, 256>(P, C, u, w, ~b);
    return;
  }
  const int64_t i = (int64_t)b * 256 + threadIdx.x;
  if (i >= P.g.N) return;
  const uint8_t kd = kind[i];
  if (kd & kKindAffected) return;
  if (!(kd & kKindUnknown)) {
    w[i] = 0.0;
    return;
  }
  w[i] = ho_plain_node<D, W>(P.g.n, C, (kd & kKindPlus) != 0, u, i);
}

// the same with the plain nodes in fixed-point tiles (op_tiled)
template <int W>
__global__ void __launch_bounds__(OpTile<W>::NT, 2)
    k_ho_tiles(CorrectParams P, StencilCoef C, const uint8_t* __restrict__ kind, const uint8_t* __restrict__ tiles,
               const double* __restrict__ u, double* __restrict__ w, AffSplit S) {
  const int b = S.index(blockIdx.x);
  if (b < 0) {
    pdl_wait();                            // the ghost values
    ho_affected<3, W, OpTile<W>::NT>(P, C, u, w, ~b);
    return;
  }
  __shared__ OpTile<W> sm;
  op_tile<W, false>(sm, P.g, C, kind, tiles, u, w, b, [](int64_t) {});
}

// b = f - L_Gamma u_Gamma (f at plain nodes; the data's ghosts at affected ones), from the ghost
// values of u = 0
template <int D>
__global__ void __launch_bounds__(256) k_ho_rhs(CorrectParams P, const uint8_t* __restrict__ kind,
                                                const double* __restrict__ f, double* __restrict__ b, AffSplit S) {
  const int blk = S.index(blockIdx.x);
  if (blk < 0) {
    pdl_wait();
    const auto A = affected<D, 1, 256>(P, OpCoef{P}, nullptr, ~blk);
    const double corr = dir_sum<D>(A.part);
    if (A.live && A.k0 == 0) b[A.i] = f[A.i] - (A.ph ? P.scale[1] : P.scale[0]) * corr;
    return;
  }
  const int64_t i = (int64_t)blk * 256 + threadIdx.x;
  if (i >= P.g.N) return;
  const uint8_t kd = kind[i];
  if (kd & kKindAffected) return;
  b[i] = kd & kKindUnknown ? f[i] : 0.0;
}

static StencilCoef stencil_coef(const Problem& P) {
  StencilCoef C;
  const double h2 = P.g.h * P.g.h;
  const double beta[2] = {P.desc.beta_minus, P.desc.beta_plus};
  for (int s = 0; s < 2; ++s) {
    C.c0[s] = P.g.dim * P.a[P.w] * beta[s] / h2;
    for (int j = 1; j <= kMaxW; ++j) C.cj[s][j - 1] = j <= P.w ? P.a[P.w + j] * beta[s] / h2 : 0.0;
  }
  return C;
}

void ho_ghost(Problem& P, const double* u, bool with_data, double* G, cudaStream_t s) {
  StencilCoef C;
  GhostParams GP;
  CorrectParams CP;
  eng_operator_params(P, &C, &GP, &CP);
  GP.with_data = with_data;
  GP.G = G;
  if (P.K_cap > 0) {
    // small blocks: a few thousand control points must still spread over all 152 SMs
    const int grid = ceil_div((int64_t)P.K_cap * kGhostLanes, kGhostThreads);
    if (P.w == 2) IIM_LAUNCH(k_ho_ghost<2>, grid, kGhostThreads, 0, s, GP, u);
    else IIM_LAUNCH(k_ho_ghost<3>, grid, kGhostThreads, 0, s, GP, u);
  }
}

// plain: blocks of plain nodes; threads: of a block
static AffSplit aff_split(const Problem& P, int parts, int plain, int threads) {
  AffSplit S;
  const int lanes = P.g.dim == 2 ? aff_lanes<2>() : aff_lanes<3>();
  S.plain = parts & 1 ? plain : 0;
  S.aff = parts & 2 ? ceil_div((int64_t)P.aff_cap * lanes, threads) : 0;
  S.first = S.plain / 3;
  S.every = S.aff > 0 ? (S.plain - S.first) / S.aff + 1 : 1;
  return S;
}

void ho_nodes(Problem& P, const double* u, double* w, bool with_data, const double* G, int parts, cudaStream_t s) {
  StencilCoef C;
  GhostParams GP;
  CorrectParams CP;
  eng_operator_params(P, &C, &GP, &CP);
  CP.with_data = with_data;
  CP.G = G;
  // (with no control point there is no ghost kernel to run beside: an ordinary launch)
#define IIM_APPLY(kernel_, nblk_, nthr_, ...)                                                     \
  do {                                                                                             \
    const AffSplit S = aff_split(P, parts, nblk_, nthr_);                                        \
    if (S.plain + S.aff == 0) return;                                                              \
    if (P.K_cap > 0) IIM_LAUNCH_PDL(kernel_, S.plain + S.aff, nthr_, 0, s, CP, C, __VA_ARGS__, S); \
    else IIM_LAUNCH(kernel_, S.plain + S.aff, nthr_, 0, s, CP, C, __VA_ARGS__, S);                \
  } while (0)
#define IIM_NODES(D, W) IIM_APPLY((k_ho_apply<D, W>), ceil_div(P.g.N, 256), 256, (const uint8_t*)P.kind, u, w)
  if (P.g.dim == 2) {
    if (P.w == 2) IIM_NODES(2, 2);
    else IIM_NODES(2, 3);
  } else if (op_tiled(P.g, P.w)) {
    IIM_APPLY(k_ho_tiles<2>, OpTile<2>::count(P.g.n), OpTile<2>::NT, (const uint8_t*)P.kind, (const uint8_t*)P.tile_kind, u, w);
  } else {
    if (P.w == 2) IIM_NODES(3, 2);
    else IIM_NODES(3, 3);
  }
#undef IIM_NODES
#undef IIM_APPLY
}

int op_tile_count(const Problem& P) { return op_tiled(P.g, P.w) ? OpTile<2>::count(P.g.n) : 0; }

void op_tile_kinds(Problem& P, cudaStream_t s) {
  const int count = op_tile_count(P);
  if (count > 0) IIM_LAUNCH(k_tile_kinds<2>, count, OpTile<2>::NT, 0, s, P.g.n, P.kind, P.tile_kind);
}

void ho_apply(Problem& P, const double* u, double* w, bool with_data, cudaStream_t s) {
  ho_ghost(P, u, with_data, P.G, s);
  ho_nodes(P, u, w, with_data, P.G, 3, s);
}

// b = f - L_Gamma u_Gamma: the operator of u = 0 with the data switched on, subtracted from f
void compute_rhs(Problem& P, const double* f, cudaStream_t s) {
  ho_ghost(P, nullptr, true, P.G, s);
  StencilCoef C;
  GhostParams GP;
  CorrectParams CP;
  eng_operator_params(P, &C, &GP, &CP);
  CP.with_data = 1;
  const AffSplit S = aff_split(P, 3, ceil_div(P.g.N, 256), 256);
  const int grid = S.plain + S.aff;
#define IIM_RHS(D)                                                                                        \
  do {                                                                                                    \
    if (P.K_cap > 0) IIM_LAUNCH_PDL(k_ho_rhs<D>, grid, 256, 0, s, CP, (const uint8_t*)P.kind, f, P.b, S); \
    else IIM_LAUNCH(k_ho_rhs<D>, grid, 256, 0, s, CP, (const uint8_t*)P.kind, f, P.b, S); \
  } while (0)
  if (P.g.dim == 2) IIM_RHS(2);
  else IIM_RHS(3);
#undef IIM_RHS
}


// ---------------------------------------------------------------------------- no-allocation apply
// The same kernels as ho_apply, but the ghost values go to a file-scope
// device array instead of the problem's workspace.  kNoAllocGhostMax doubles
// (2 MiB) are reserved on every device that loads the library, for the life of
// the process.  All calls share the array, so calls that overlap on the device
// (other streams, other threads, other problems) race on it.  Each call writes
// every ghost value before it reads it, so nothing in the array has to be cleared.
namespace {
constexpr int64_t kNoAllocGhostMax = 1 << 18;
__device__ __align__(256) double g_noalloc_ghost[kNoAllocGhostMax];
constexpr int kNoAllocMaxDevices = 64;
double* g_noalloc_addr[kNoAllocMaxDevices] = {nullptr};
std::mutex g_noalloc_mu;
}  // namespace

iim_status ho_apply_noalloc(Problem& P, const double* u, double* w, bool with_data, cudaStream_t s) {
  const int64_t need = (int64_t)P.nfit_cap * P.w;
  if (need > kNoAllocGhostMax) {
    set_error("iim_apply_noalloc: the problem needs " + std::to_string(need) + " ghost values, more than the " +
              std::to_string(kNoAllocGhostMax) + " the static scratch holds");
    return IIM_ERR_CAPACITY;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) {
    cudaGetLastError();
    set_error("iim_apply_noalloc: no usable current device");
    return IIM_ERR_CUDA;
  }
  double* G = nullptr;
  {
    // first call on this device: look up the device address of the array (the host
    // symbol is only a stand-in), with this device current
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
      void* ptr = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_ghost);
      if (e != cudaSuccess) {
        cudaGetLastError();
        set_error(std::string("iim_apply_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        return IIM_ERR_CUDA;
      }
      g_noalloc_addr[dev] = (double*)ptr;
    }
    G = g_noalloc_addr[dev];
  }
  ho_ghost(P, u, with_data, G, s);
  ho_nodes(P, u, w, with_data, G, 3, s);
  return IIM_OK;
}


// ---------------------------------------------------------------------------- batched engine
// Three kernels, each over all slots: the sums of every node in phase, the ghosts, the corrections of
// affected nodes, in the arithmetic of the two launches above.  A stencil item is 1024 nodes; ghost
// and correction items are one block each.
template <int D, int W>
__global__ void __launch_bounds__(kEngThreads) k_eng_stencil(EngArgs A) {
  eng_for_items(A, kListStencil + (D - 2) * 2 + (W - 2), [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role == kRoleIdle) return;
    const double* u;
    double* w;
    eng_apply_io(s, u, w);
    const int64_t base = (int64_t)item * (4 * kEngThreads) + threadIdx.x;
    const int64_t N = s.g.N;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t i = base + k * kEngThreads;
      if (i < N) ho_stencil_node<D, W>(s.g, s.C, s.iface, u, s.phase, w, i);
    }
  });
}

// items of problems with fixed-point tiles: one tile each (affected nodes as in k_eng_stencil)
template <int W>
__global__ void __launch_bounds__(OpTile<W>::NT, 2) k_eng_tiles(EngArgs A) {
  __shared__ OpTile<W> sm;
  eng_for_items(A, kListTile, [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role == kRoleIdle) return;
    const double* u;
    double* w;
    eng_apply_io(s, u, w);
    op_tile<W, true>(sm, s.g, s.C, s.kind, s.tile_kind, u, w, item,
                        [&](int64_t i) { ho_stencil_node<3, W>(s.g, s.C, s.iface, u, s.phase, w, i); });
  });
}

template <int W>
__global__ void __launch_bounds__(64) k_eng_ghost(EngArgs A) {
  eng_for_items(A, kListGhost + (W - 2), [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role == kRoleIdle) return;
    const double* u;
    double* w;
    eng_apply_io(s, u, w);
    ho_ghost_body<W>(s.GP, u, item * 64 + threadIdx.x);
  });
}

__global__ void __launch_bounds__(64) k_eng_correct(EngArgs A) {
  eng_for_items(A, kListCorrect, [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role == kRoleIdle) return;
    const double* u;
    double* w;
    eng_apply_io(s, u, w);
    ho_correct_body(s.CP, u, w, item * 64 + threadIdx.x);
  });
}

void eng_launch_apply(const EngArgs& A, const unsigned char* present, cudaStream_t s) {
#define IIM_ENG_ST(D, W)                                                                                       \
  if (present[kListStencil + (D - 2) * 2 + (W - 2)])                                                          \
    IIM_LAUNCH((k_eng_stencil<D, W>), eng_grid((const void*)k_eng_stencil<D, W>, kEngThreads, 0), kEngThreads, 0, s, A);
  IIM_ENG_ST(2, 2) IIM_ENG_ST(2, 3) IIM_ENG_ST(3, 2) IIM_ENG_ST(3, 3)
#undef IIM_ENG_ST
  if (present[kListTile])
    IIM_LAUNCH(k_eng_tiles<2>, eng_grid((const void*)k_eng_tiles<2>, OpTile<2>::NT, 0), OpTile<2>::NT, 0, s, A);
  if (present[kListGhost + 0]) IIM_LAUNCH(k_eng_ghost<2>, eng_grid((const void*)k_eng_ghost<2>, 64, 0), 64, 0, s, A);
  if (present[kListGhost + 1]) IIM_LAUNCH(k_eng_ghost<3>, eng_grid((const void*)k_eng_ghost<3>, 64, 0), 64, 0, s, A);
  if (present[kListCorrect]) IIM_LAUNCH(k_eng_correct, eng_grid((const void*)k_eng_correct, 64, 0), 64, 0, s, A);
}

// Q.box_c for a stencil with coefficient coef(j) at offset j on the + side
template <class F>
static void box_sums(const Problem& P, CorrectParams& Q, F coef) {
  for (int js = 1; js <= kMaxW; ++js)
    for (int m = 0; m < 8; ++m) {
      double v = 0.0;
      for (int j = js; j <= P.w; ++j) v += coef(j) * P.box_w[j - js][m];
      Q.box_c[js - 1][m] = v;
    }
}

// the operator's per-problem parameters (homogeneous: the data enter through b)
void eng_operator_params(Problem& P, StencilCoef* C, GhostParams* GP, CorrectParams* CP) {
  *C = stencil_coef(P);
  GhostParams& G = *GP;
  G.nfit = P.nfit_cap;
  G.w = P.w;
  G.rcap = P.rcap;
  G.bc = P.desc.bc;
  G.interface_ = P.desc.bc == IIM_BC_INTERFACE;
  G.with_data = 0;
  G.beta_p = P.desc.beta_plus;
  G.beta_m = P.desc.beta_minus;
  G.K = P.d_counts + 0;
  G.fit_R = P.fit_R;
  G.fit_nodes = P.fit_nodes;
  G.fit_coef = P.fit_coef;
  G.fit_cdat = P.fit_cdat;
  G.g = P.d_g;
  G.j0 = P.d_j0;
  G.j1 = P.d_j1;
  G.G = P.G;
  CorrectParams& Q = *CP;
  Q.g = P.g;
  Q.w = P.w;
  Q.q = P.q;
  Q.with_data = 0;
  Q.n_aff_cap = P.aff_cap;
  Q.nfit_cap = P.nfit_cap;
  Q.n_aff = P.d_counts + 1;
  Q.aff_node = P.aff_node;
  Q.aff_fit = P.aff_fit;
  Q.aff_j = P.aff_j;
  Q.G = P.G;
  Q.phase = P.phase;
  Q.box = P.d_box;
  for (int k = 0; k < 2 * kMaxW + 1; ++k) Q.a[k] = k < 2 * P.w + 1 ? P.a[k] : 0.0;
  const double h2 = P.g.h * P.g.h;
  Q.scale[0] = P.desc.beta_minus / h2;
  Q.scale[1] = P.desc.beta_plus / h2;
  box_sums(P, Q, [&](int j) { return P.a[P.w + j]; });
}


// ---------------------------------------------------------------------------- boundary quantities, gradient
// Sec. 2.4: the boundary quantity the data do not prescribe, from row w of each fit:
// Dirichlet -> n . grad u(x_c) (derivative row, n out of Omega+), Neumann -> u(x_c)
// (Eq. 6, stored as coefficients over X_c plus 1/D_c times qbar).  Eight lanes per
// control point.
__global__ void __launch_bounds__(64) k_boundary_values(GhostParams P, const double* __restrict__ u,
                                                        double* __restrict__ out) {
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  const int c = gid / kGhostLanes, q = gid % kGhostLanes;
  const int K = *P.K;
  const bool live = c < K;
  double acc = 0.0;
  if (live) {
    const int R = P.fit_R[c];
    const int32_t* nodes = P.fit_nodes + (size_t)c * P.rcap;
    const double* row = P.fit_coef + ((size_t)c * (P.w + 1) + P.w) * P.rcap;
    for (int a = q; a < R; a += kGhostLanes) acc = fma(row[a], u[nodes[a]], acc);
  }
  acc = quad_sum(acc);
  if (live && q == 0) out[c] = acc + P.fit_cdat[(size_t)c * (P.w + 1) + P.w] * P.g[c];
}

// centred first-derivative stencil b_{-w..w} of order 2w (odd, b_0 = 0): the unique
// stencil exact for polynomials of degree <= 2w (2/3, -1/12 for w = 2; 3/4, -3/20,
// 1/60 for w = 3)
struct GradCoef {
  double b[2 * kMaxW + 1];
  double ih;                             // 1 / h
};

static GradCoef grad_coef(int w, double h) {
  GradCoef B;
  B.ih = 1.0 / h;
  const double h2[2] = {2.0 / 3.0, -1.0 / 12.0};
  const double h3[3] = {3.0 / 4.0, -3.0 / 20.0, 1.0 / 60.0};
  for (int k = 0; k < 2 * kMaxW + 1; ++k) B.b[k] = 0.0;
  for (int j = 1; j <= w; ++j) {
    const double v = w == 2 ? h2[j - 1] : h3[j - 1];
    B.b[w + j] = v;
    B.b[w - j] = -v;
  }
  return B;
}

// its coefficients as ho_direction takes them (odd)
template <int W>
struct GradFunctor {
  const GradCoef& B;
  __device__ __forceinline__ double at(int j, int s) const { return s > 0 ? B.b[W + j] : -B.b[W + j]; }
  __device__ __forceinline__ double box(double v, int s) const { return s > 0 ? v : -v; }
};

// Direction k (axis k / 2, side k & 1) at affected node t: the neighbours in phase (v[j], else 0) and,
// returned, the ghost contribution
template <int W, class Coef>
__device__ __forceinline__ double aff_direction(const CorrectParams& P, Coef coef, const double* __restrict__ u, int t,
                                                int64_t i, const int* m, uint8_t ph, int k, double (&v)[W]) {
  const int n = P.g.n, ax = k >> 1, s = k & 1 ? 1 : -1, ma = ax == 0 ? m[0] : (ax == 1 ? m[1] : m[2]);
  const int64_t st = ax == 0 ? 1 : (ax == 1 ? (int64_t)n : (int64_t)n * n);
#pragma unroll
  for (int j = 1; j <= W; ++j) {
    const int pos = ma + j * s;
    v[j - 1] = u && pos >= 0 && pos < n && P.phase[i + j * s * st] == ph ? u[i + j * s * st] : 0.0;
  }
  return ho_direction(P, coef, u, t, i, m, ph, ax, k & 1);
}

// grad u by the centred first-derivative stencil b of the scheme's order, in one launch beside the
// ghost kernel like k_ho_apply.  out is [dim][N]; zero at nodes that are not unknowns.
// Plain nodes per thread: four in 3D, where most of an interior problem's nodes only store zeros and a
// thread each left too few stores in flight (gradient and boundary values, 192^3 interior 141 -> 111 us,
// three separate kernels 134; exterior 277 -> 284, 364); one in 2D, whose grids have fewer blocks.
template <int D>
__host__ __device__ constexpr int grad_nodes() { return D == 3 ? 4 : 1; }

template <int D, int W>
__global__ void __launch_bounds__(256, 6) k_grad_apply(CorrectParams P, GradCoef B, const uint8_t* __restrict__ kind,
                                                    const double* __restrict__ u, double* __restrict__ out, AffSplit S) {
  const int blk = S.index(blockIdx.x), n = P.g.n;
  if (blk < 0) {
    pdl_wait();                            // the ghost values
    // direction 2 ax + 1 is the + side, 2 ax the - side
    if constexpr (aff_lanes<D>() == 1) {
      const int t = ~blk * 256 + (int)threadIdx.x;
      if (t >= min(*P.n_aff, P.n_aff_cap)) return;
      const int64_t i = P.aff_node[t];
      int m[3];
      node_indices(n, D, i, m);
      const uint8_t ph = P.phase[i];
#pragma unroll 1
      for (int ax = 0; ax < D; ++ax) {   // an axis at a time: few registers, so that the plain blocks' stores overlap
        double lo[W], hi[W], acc = 0.0;
        const double pl = aff_direction<W>(P, GradFunctor<W>{B}, u, t, i, m, ph, 2 * ax, lo);
        const double pr = aff_direction<W>(P, GradFunctor<W>{B}, u, t, i, m, ph, 2 * ax + 1, hi);
#pragma unroll
        for (int j = 0; j < W; ++j) acc = fma(B.b[W + j + 1], hi[j] - lo[j], acc);
        out[(size_t)ax * P.g.N + i] = fma(pr + pl, B.ih, acc * B.ih);
      }
    } else {
      const auto A = affected<D, W, 256>(P, GradFunctor<W>{B}, u, ~blk);
      double acc = 0.0;
#pragma unroll
      for (int j = 0; j < W; ++j) acc = fma(B.b[W + j + 1], A.v[j][0] - __shfl_xor_sync(0xffffffffu, A.v[j][0], 1), acc);
      const double corr = A.part[0] + __shfl_xor_sync(0xffffffffu, A.part[0], 1);
      if (A.live && (A.k0 & 1)) out[(size_t)(A.k0 >> 1) * P.g.N + A.i] = fma(corr, B.ih, acc * B.ih);
    }
    return;
  }
  constexpr int R = grad_nodes<D>();
  uint8_t kd[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t i = ((int64_t)blk * R + r) * 256 + threadIdx.x;
    kd[r] = i < P.g.N ? kind[i] : kKindAffected;
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t i = ((int64_t)blk * R + r) * 256 + threadIdx.x;
    if (kd[r] & kKindAffected) continue;
#pragma unroll
    for (int ax = 0; ax < D; ++ax) {
      const int64_t st = ax == 0 ? 1 : (ax == 1 ? (int64_t)n : (int64_t)n * n);
      double v = 0.0;
      if (kd[r] & kKindUnknown) {
        double acc = 0.0;
#pragma unroll
        for (int j = 1; j <= W; ++j) acc = fma(B.b[W + j], u[i + j * st] - u[i - j * st], acc);
        v = acc * B.ih;
      }
      out[(size_t)ax * P.g.N + i] = v;
    }
  }
}

iim_status boundary_values(Problem& P, const double* u, double* out, cudaStream_t s) {
  if (P.desc.bc == IIM_BC_INTERFACE) {
    set_error("boundary values are defined for boundary problems");
    return IIM_ERR_INVALID_ARG;
  }
  StencilCoef C;
  GhostParams GP;
  CorrectParams CP;
  eng_operator_params(P, &C, &GP, &CP);
  if (P.K_cap > 0)
    IIM_LAUNCH(k_boundary_values, ceil_div((int64_t)P.K_cap * kGhostLanes, 64), 64, 0, s, GP, u, out);
  return IIM_OK;
}

iim_status gradient(Problem& P, const double* u, double* grad, cudaStream_t s) {
  const GradCoef B = grad_coef(P.w, P.g.h);
  ho_ghost(P, u, true, P.G, s);                     // ghost values with the problem's data
  StencilCoef C;
  GhostParams GP;
  CorrectParams CP;
  eng_operator_params(P, &C, &GP, &CP);
  CP.with_data = 1;
  box_sums(P, CP, [&](int j) { return B.b[P.w + j]; });
  const AffSplit S = aff_split(P, 3, ceil_div(P.g.N, 256 * (P.g.dim == 3 ? grad_nodes<3>() : grad_nodes<2>())), 256);
  const int grid = S.plain + S.aff;
#define IIM_GRAD(D, W)                                                                                              \
  do {                                                                                                              \
    if (P.K_cap > 0)                                                                                                \
      IIM_LAUNCH_PDL((k_grad_apply<D, W>), grid, 256, 0, s, CP, B, (const uint8_t*)P.kind, u, grad, S); \
    else                                                                                                            \
      IIM_LAUNCH((k_grad_apply<D, W>), grid, 256, 0, s, CP, B, (const uint8_t*)P.kind, u, grad, S); \
  } while (0)
  if (P.g.dim == 2) {
    if (P.w == 2) IIM_GRAD(2, 2);
    else IIM_GRAD(2, 3);
  } else {
    if (P.w == 2) IIM_GRAD(3, 2);
    else IIM_GRAD(3, 3);
  }
#undef IIM_GRAD
  return IIM_OK;
}

}  // namespace iim
