// Right-preconditioned flexible GMRES(m) with device-side control (paper Sec. 4.1).
//
// Per iteration j (all on the device, no host round trip):
//   z_j = M(v_j)                 one SW multigrid V-cycle      (multigrid.cu)
//   w   = L z_j                  the IIM operator              (operator.cu)
//   h   = V^T w, |w|^2           one fused pass over v_0..v_j  (k_multidot)
//   w  -= V h, |w|^2             one fused pass                (k_update)
//   optional second pass when |w| dropped below 1e-3 |w_old|   (classical
//   Gram-Schmidt with re-orthogonalisation on severe cancellation)
//   Givens rotation, Arnoldi residual estimate, flags         (last block of k_update)
// v_{j+1} is kept unnormalised; 1/|v_{j+1}| is applied inside the kernels that
// read it.  Reductions are deterministic: per-block partials in a fixed grid,
// summed in block order by the last block to finish.  Convergence is decided on
// the true residual |b - A x| / |b| at every restart (x += Z y).
// The whole solve is one CUDA graph: WHILE(not done) { IF(active) iteration 0;
// ...; IF(active) iteration m-1; restart }, with the conditions set by kernels.
//
// Left-preconditioned GMRES(m) (Sec. 3.2) shares the Arnoldi kernels: its basis is
// built from w = M(L v_j), x += V y, and the residual it tests and restarts from is
// the preconditioned one, M (b - L x), relative to |M b|.
#include <algorithm>

#include "engine.cuh"

namespace iim {



constexpr int kRedThreads = 256;

// Reductions run over a virtual grid of nvb blocks (the launch grid of a single
// solve, or the work items of one solve inside a batched launch): block vb stores
// its partial sums, and the last of the nvb blocks to finish combines them.
template <int NV>
__device__ inline void block_reduce_store(double (&acc)[NV], double* partial, int stride, int vb, int nv = NV) {
  __shared__ double red[kRedThreads / 32][NV > 0 ? NV : 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  lane_sums<32, NV>(acc, lane, red[wid]);
  __syncthreads();
  if (threadIdx.x < nv) {
    double s = 0;
    for (int w = 0; w < kRedThreads / 32; ++w) s += red[w][threadIdx.x];
    partial[(size_t)vb * stride + threadIdx.x] = s;
  }
}

// true in exactly one of the nvb blocks: the last one to finish (all partials visible)
__device__ inline bool last_block(unsigned int* counter, int nvb) {
  __shared__ bool is_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int t = atomicAdd(counter, 1u);
    is_last = (t == (unsigned int)nvb - 1);
  }
  __syncthreads();
  if (is_last) __threadfence();
  return is_last;
}

// Sum the per-block partials in the last block: thread t adds blocks t, t+256, ... of
// every component, then a fixed-order tree over the threads (deterministic).
template <int NV>
__device__ inline void sum_partials(const double* partial, int nblocks, int stride, int nv, double* out) {
  __shared__ double red[kRedThreads / 32][NV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double s[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) s[k] = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (k < nv) s[k] += partial[(size_t)b * stride + k];
  lane_sums<32, NV>(s, lane, red[wid]);
  __syncthreads();
  if (threadIdx.x < nv) {
    double t = 0;
    for (int w = 0; w < kRedThreads / 32; ++w) t += red[w][threadIdx.x];
    out[threadIdx.x] = t;
  }
  __syncthreads();
}

__device__ inline void set_cond(SolverScalars* S, cudaGraphConditionalHandle h, int v) {
  if (S->graph_mode) cudaGraphSetConditional(h, v ? 1u : 0u);
}

// restart / start: V0 = b - Ax (Ax in ax), |V0|^2, |b|^2.  With b == nullptr V0 already
// holds the residual (left preconditioning: M (b - A x)) and is only measured.
// first: 0 restart, 1 start, 2 only store |V0| as the norm of b (left preconditioning:
// V0 = M b), 3 start with that norm already stored.
__device__ inline void residual_body(const double* __restrict__ b, const double* __restrict__ ax,
                                     double* __restrict__ v0, int64_t N, double* partial, unsigned int* counter,
                                     SolverScalars* S, int first, int* status, int vb, int nvb) {
  double acc[2] = {0.0, 0.0};
  for (int64_t i = (int64_t)vb * blockDim.x + threadIdx.x; i < N; i += (int64_t)nvb * blockDim.x) {
    double bi, r;
    if (b) {
      bi = b[i];
      r = bi - ax[i];
      v0[i] = r;
    } else {
      r = v0[i];
      bi = r;
    }
    acc[0] = fma(r, r, acc[0]);
    acc[1] = fma(bi, bi, acc[1]);
  }
  block_reduce_store<2>(acc, partial, 4, vb);
  if (!last_block(counter, nvb)) return;
  __shared__ double tot[4];
  sum_partials<2>(partial, nvb, 4, 2, tot);
  if (threadIdx.x == 0) {
    *counter = 0;
    if (first == 2) {
      S->bnorm = sqrt(tot[1]);
      return;
    }
    double rn = sqrt(tot[0]);
    if (first) {
      if (first == 1) S->bnorm = sqrt(tot[1]);
      S->iters = 0;
      S->restarts = 0;
      S->done = 0;
      S->converged = 0;
      S->breakdown = 0;
      S->first = 0;
    } else {
      S->restarts += 1;
    }
    double bn = S->bnorm;
    double rel = bn > 0 ? rn / bn : 0.0;
    S->relres = rel;
    bool bad = !(rn == rn) || isinf(rn);
    if (bad) {
      set_status(status, IIM_ERR_BREAKDOWN);
      S->done = 1;
    } else if (bn == 0.0 || rel <= S->tol) {
      S->done = 1;
      S->converged = 1;
    } else if (S->iters >= S->max_iter) {
      S->done = 1;
    }
    S->g[0] = rn;
    for (int k = 1; k <= kMaxRestart; ++k) S->g[k] = 0.0;
    S->inv_norm[0] = rn > 0 ? 1.0 / rn : 0.0;
    S->k = 0;
    S->active = !S->done;
    set_cond(S, S->h_while, !S->done);
    for (int k = 0; k < S->m; ++k) set_cond(S, S->h_if[k], k == 0 ? S->active : 0);
  }
}

__global__ void __launch_bounds__(kRedThreads) k_residual(const double* __restrict__ b, const double* __restrict__ ax,
                                                          double* __restrict__ v0, int64_t N, double* partial,
                                                          unsigned int* counter, SolverScalars* S, int first,
                                                          int* status) {
  residual_body(b, ax, v0, N, partial, counter, S, first, status, blockIdx.x, gridDim.x);
}

// One pass over w and the vectors before it: f(element, w, v(k)) for the pairs first, first + step, ...
// STAGED: every vector's pair of several elements is loaded before the first is used.  The grid has two
// blocks of 256 threads per SM, so a thread needs six and more 16-byte loads in flight to keep the
// memory busy; left to itself the compiler went from 64 to 48 registers with a change elsewhere in the
// kernel and took 286 us for 220 (256^3, ten vectors).
template <int NV, bool STAGED, class F>
__device__ __forceinline__ void orth_elements(const double* __restrict__ V, int64_t Np, const double2* w2, int64_t first,
                                              int64_t step, int64_t N2, F f) {
  int64_t e = first;
  if constexpr (STAGED) {
    constexpr int U = NV <= 2 ? 6 : (NV <= 3 ? 4 : (NV <= 6 ? 2 : 1));
    for (; e + (U - 1) * step < N2; e += U * step) {
      double2 wv[U], vv[U][NV];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        wv[u] = w2[e + u * step];
#pragma unroll
        for (int k = 0; k < NV; ++k) vv[u][k] = reinterpret_cast<const double2*>(V + (size_t)k * Np)[e + u * step];
      }
#pragma unroll
      for (int u = 0; u < U; ++u) f(e + u * step, wv[u], [&](int k) { return vv[u][k]; });
    }
  }
  for (; e < N2; e += step)
    f(e, w2[e], [&](int k) { return reinterpret_cast<const double2*>(V + (size_t)k * Np)[e]; });
}

// h_i = inv_norm_i <V_i, w> (i < nv = j + 1), |w|^2 ; w = V[j+1].  NVMAX bounds nv at
// compile time (a single solve instantiates NVMAX = nv; the batched engine 16).
template <int NVMAX, bool STAGED>
__device__ inline void multidot_body(const double* __restrict__ V, int64_t Np, int j, int nv, double* partial,
                                     unsigned int* counter, SolverScalars* S, int second, int vb, int nvb) {
  if (second && !S->reorth_needed) return;
  const double* w = V + (size_t)(j + 1) * Np;
  double acc[NVMAX + 1];
#pragma unroll
  for (int k = 0; k <= NVMAX; ++k) acc[k] = 0.0;
  const int64_t N2 = Np / 2;
  const double2* w2 = reinterpret_cast<const double2*>(w);
  const int64_t first = (int64_t)vb * blockDim.x + threadIdx.x, step = (int64_t)nvb * blockDim.x;
  auto take = [&](double2 wv, auto vv) {
#pragma unroll
    for (int k = 0; k < NVMAX; ++k) {
      if (k >= nv) break;
      const double2 v = vv(k);
      acc[k] = fma(v.x, wv.x, acc[k]);
      acc[k] = fma(v.y, wv.y, acc[k]);
    }
    acc[NVMAX] = fma(wv.x, wv.x, acc[NVMAX]);
    acc[NVMAX] = fma(wv.y, wv.y, acc[NVMAX]);
  };
  orth_elements<NVMAX, STAGED>(V, Np, w2, first, step, N2, [&](int64_t, double2 wv, auto vv) { take(wv, vv); });
  pdl_trigger();                       // the next kernel's launch overlaps the reduction
  {
    // partials [h_0 .. h_j, |w|^2]: component nv is acc[NVMAX] (static register indices)
    __shared__ double red[kRedThreads / 32][NVMAX + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    lane_sums<32, NVMAX + 1>(acc, lane, red[wid]);
    __syncthreads();
    if (threadIdx.x <= nv) {
      const int k = threadIdx.x < nv ? threadIdx.x : NVMAX;
      double s = 0;
      for (int w = 0; w < kRedThreads / 32; ++w) s += red[w][k];
      partial[(size_t)vb * (kMaxRestart + 4) + threadIdx.x] = s;
    }
  }
  if (!last_block(counter, nvb)) return;
  __shared__ double tot[kMaxRestart + 4];
  sum_partials<NVMAX + 1>(partial, nvb, kMaxRestart + 4, nv + 1, tot);
  if (threadIdx.x == 0) {
    *counter = 0;
    if (!second) {
      for (int k = 0; k < nv; ++k) S->hcol[k] = tot[k] * S->inv_norm[k];
      S->w2_old = tot[nv];
    } else {
      // second pass: store the correction in y[] temporarily
      for (int k = 0; k < nv; ++k) S->y[k] = tot[k] * S->inv_norm[k];
    }
  }
}

template <int NV>
__global__ void __launch_bounds__(kRedThreads, 2) k_multidot(const double* __restrict__ V, int64_t Np, int j,
                                                          double* partial, unsigned int* counter, SolverScalars* S,
                                                          int second) {
  pdl_wait();
  multidot_body<NV, true>(V, Np, j, NV, partial, counter, S, second, blockIdx.x, gridDim.x);
}

// The kernels of an iteration are chained as dependent launches; each lets the next one be launched when
// its blocks are through with the vectors, not before, so that no waiting block takes an SM's room from
// a running one.  With the sums across a warp transposed (common.cuh), the Givens step in the last block
// of the update and the coefficients of x in the blocks that use them, a pass takes (multi-dot / update
// with six vectors) 26.7 -> 18.0 / 18.5 -> 16.8 us at 96^3, 210 -> 204 / 220 -> 209 us at 256^3, and the
// launches of one thread (9 us per iteration, 10 per restart) are gone: the 64^2 circle's solve
// 1463 -> 1260 us, the 1024^2 star's step 7.31 -> 6.93 ms.
//
// Givens rotations on column j, estimate, flags, by one block: the column and the rotations so far are
// read by as many threads, threads of other warps take the
// norms' roots and reciprocals, one thread rotates.
__device__ inline void arnoldi_block(SolverScalars* S, int j, int* status) {
  __shared__ double h[kMaxRestart + 1], cs[kMaxRestart], sn[kMaxRestart], s_w2, s_hn, s_inv, s_ib;
  const int t = threadIdx.x, L = kMaxRestart + 1;
  double* H = S->H;
  if (t <= j) h[t] = S->hcol[t];
  if (t < j) {
    cs[t] = S->cs[t];
    sn[t] = S->sn[t];
  }
  if (t == (blockDim.x > 32 ? 32 : 0)) {
    s_w2 = S->w2;
    s_hn = sqrt(s_w2);
    s_inv = s_hn > 0 ? 1.0 / s_hn : 0.0;
  }
  if (t == (blockDim.x > 64 ? 64 : 0)) s_ib = S->bnorm > 0 ? 1.0 / S->bnorm : 0.0;
  double g = 0, tol = 0;
  int iters = 0, max_iter = 0, m = 0;
  if (t == 0) {
    g = S->g[j];
    tol = S->tol;
    iters = S->iters;
    max_iter = S->max_iter;
    m = S->m;
  }
  __syncthreads();
  if (t == 0) {
    for (int i = 0; i < j; ++i) {
      const double a = h[i], b = h[i + 1];
      h[i] = cs[i] * a + sn[i] * b;
      h[i + 1] = -sn[i] * a + cs[i] * b;
    }
    const double hn = s_hn;
    const double a = h[j], b = hn;
    // the square of b = |w| is what was summed: one reciprocal root gives the radius and the rotation
    const double q = fma(a, a, s_w2);
    double den, c, s;
    if (q > 1e-280 && q < 1e280) {
      const double r = rsqrt(q);
      den = q * r;
      c = a * r;
      s = b * r;
    } else {
      den = hypot(a, b);
      c = den > 0 ? a / den : 1.0;
      s = den > 0 ? b / den : 0.0;
    }
    h[j] = den;
    S->inv_norm[j + 1] = s_inv;
    S->cs[j] = c;
    S->sn[j] = s;
    const double gn = -s * g;
    S->g[j + 1] = gn;
    S->g[j] = c * g;
    S->iters = iters + 1;
    S->k = j + 1;
    const double est = fabs(gn) * s_ib;
    S->est = est;
    const bool bad = !(est == est) || !(hn == hn) || isinf(hn);
    if (bad) {
      set_status(status, IIM_ERR_BREAKDOWN);
      S->breakdown = 1;
    }
    const bool stop = bad || hn == 0.0 || est <= tol || iters + 1 >= max_iter || j + 1 >= m;
    S->active = !stop;
    if (j + 1 < m) set_cond(S, S->h_if[j + 1], !stop);
  }
  __syncthreads();
  if (t <= j) H[t + L * j] = h[t];
  if (t == j + 1) H[t + L * j] = 0.0;
}

// w -= sum_i c_i V_i with c_i = h_i inv_norm_i (i < nv) ; |w|^2.  With arnoldi, the last block also
// closes the iteration (arnoldi_block) unless a second pass is due.
template <int NVMAX, bool STAGED>
__device__ inline void update_body(double* __restrict__ V, int64_t Np, int j, int nv, double* partial,
                                   unsigned int* counter, SolverScalars* S, int second, int vb, int nvb, bool arnoldi,
                                   int* status) {
  if (second && !S->reorth_needed) return;
  __shared__ double c[NVMAX];
  if (threadIdx.x < nv) c[threadIdx.x] = (second ? S->y[threadIdx.x] : S->hcol[threadIdx.x]) * S->inv_norm[threadIdx.x];
  __syncthreads();
  double* w = V + (size_t)(j + 1) * Np;
  double acc[1] = {0.0};
  const int64_t N2 = Np / 2;
  double2* w2 = reinterpret_cast<double2*>(w);
  const int64_t first = (int64_t)vb * blockDim.x + threadIdx.x, step = (int64_t)nvb * blockDim.x;
  orth_elements<NVMAX, STAGED>(V, Np, w2, first, step, N2, [&](int64_t e, double2 wv, auto vv) {
#pragma unroll
    for (int k = 0; k < NVMAX; ++k) {
      if (k >= nv) break;
      const double2 v = vv(k);
      wv.x = fma(-c[k], v.x, wv.x);
      wv.y = fma(-c[k], v.y, wv.y);
    }
    w2[e] = wv;
    acc[0] = fma(wv.x, wv.x, acc[0]);
    acc[0] = fma(wv.y, wv.y, acc[0]);
  });
  pdl_trigger();                       // the next kernel's launch overlaps the reduction
  block_reduce_store<1>(acc, partial, kMaxRestart + 4, vb);
  if (!last_block(counter, nvb)) return;
  __shared__ double tot[kMaxRestart + 4];
  __shared__ int close;
  sum_partials<1>(partial, nvb, kMaxRestart + 4, 1, tot);
  if (threadIdx.x == 0) {
    *counter = 0;
    S->w2 = tot[0];
    if (!second) {
      // second pass only on severe cancellation, |w| < 1e-3 |w_old| (a DGKS test with a small eta:
      // with the multigrid preconditioner |w| drops below |w_old|/sqrt(2) at every iteration,
      // yet one pass gives the same iterates' quality and iteration counts)
      const int again = S->reorth && (tot[0] < 1e-6 * S->w2_old);
      S->reorth_needed = again;
      close = arnoldi && !again;
    } else {
      for (int k = 0; k < nv; ++k) S->hcol[k] += S->y[k];
      S->reorth_needed = 0;
      close = arnoldi;
    }
  }
  __syncthreads();
  if (close) arnoldi_block(S, j, status);
}

template <int NV>
__global__ void __launch_bounds__(kRedThreads, 2) k_update(double* __restrict__ V, int64_t Np, int j, double* partial,
                                                        unsigned int* counter, SolverScalars* S, int second, int arnoldi,
                                                        int* status) {
  pdl_wait();
  update_body<NV, true>(V, Np, j, NV, partial, counter, S, second, blockIdx.x, gridDim.x, arnoldi != 0, status);
}

// y = H^-1 g (k x k upper triangular) by one warp: lane r holds g_r, each y_i leaves its column from
// the rows above at once
__device__ inline void solve_y_warp(const SolverScalars* S, double* y) {
  const int L = kMaxRestart + 1, k = S->k, r = threadIdx.x & 31;
  const double d = r < k ? S->H[r + L * r] : 0.0;
  const double inv = d != 0.0 ? 1.0 / d : 0.0;
  double g = r < k ? S->g[r] : 0.0;
  double h[kMaxRestart];
#pragma unroll
  for (int c = 0; c < kMaxRestart; ++c) h[c] = r < c && c < k ? S->H[r + L * c] : 0.0;
#pragma unroll
  for (int i = kMaxRestart - 1; i >= 0; --i) {
    if (i >= k) continue;
    const double yi = __shfl_sync(0xffffffffu, g * inv, i);
    if (r == i) g = yi;
    else g = fma(-h[i], yi, g);
  }
  if (r < kMaxRestart) y[r] = r < k ? g : 0.0;
}

// x += sum_{i<k} y_i Z_i (right preconditioning), or x += sum_{i<k} y_i V_i / |V_i| with
// Z = V (left preconditioning: the basis is stored unnormalised).  Every block solves for the coefficients
// itself, which costs less than a launch of one warp before this one.
__device__ inline void xupdate_body(double* __restrict__ x, const double* __restrict__ Z, int64_t Np, int64_t N,
                                    const SolverScalars* S, int vb, int nvb,
                                    bool unnormalised = false) {
  __shared__ double y[kMaxRestart];
  if (threadIdx.x < 32) {
    solve_y_warp(S, y);
    __syncwarp();
    if (unnormalised && threadIdx.x < kMaxRestart) y[threadIdx.x] *= S->inv_norm[threadIdx.x];
  }
  const int k = S->k;
  __syncthreads();
  for (int64_t i = (int64_t)vb * blockDim.x + threadIdx.x; i < N; i += (int64_t)nvb * blockDim.x) {
    double acc = x[i];
    for (int c = 0; c < k; ++c) acc = fma(y[c], Z[(size_t)c * Np + i], acc);
    x[i] = acc;
  }
}

__global__ void __launch_bounds__(256) k_xupdate(double* __restrict__ x, const double* __restrict__ Z, int64_t Np,
                                                 int64_t N, const SolverScalars* S, int unnormalised) {
  xupdate_body(x, Z, Np, N, S, blockIdx.x, gridDim.x, unnormalised != 0);
}

// r = b - ax
__global__ void __launch_bounds__(256) k_sub(const double* __restrict__ b, const double* __restrict__ ax,
                                             double* __restrict__ r, int64_t N) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
    r[i] = b[i] - ax[i];
}

__global__ void k_init_scalars(SolverScalars* S, int m, int max_iter, double tol, int graph_mode, int reorth) {
  S->m = m;
  S->max_iter = max_iter;
  S->tol = tol;
  S->graph_mode = graph_mode;
  S->reorth = reorth;
  S->reorth_needed = 0;
  S->k = 0;
  S->first = 1;
  S->active = 0;
  S->done = 0;
}

// the solve graph's condition handles, passed by value (no staging buffer: building a
// graph allocates and frees nothing, so it does not synchronise the device)
struct GraphHandles {
  cudaGraphConditionalHandle h_while;
  cudaGraphConditionalHandle h_if[kMaxRestart];
  int m;
};

__global__ void k_set_handles(SolverScalars* S, GraphHandles H) {
  S->h_while = H.h_while;
  for (int k = 0; k < H.m; ++k) S->h_if[k] = H.h_if[k];
}

// ---------------------------------------------------------------------------- host side
iim_status krylov_alloc(Problem& P) {
  P.Npad = ((P.g.N + P.aug + 63) / 64) * 64;   // augmented: entry N holds the shift alpha
  const int m = P.opt.restart;
  // right preconditioning keeps the m preconditioned vectors; left needs one scratch vector
  const int mz = P.opt.krylov == IIM_KRYLOV_GMRES_LEFT ? 1 : m;
  P.V = (double*)dev_alloc(P, sizeof(double) * (size_t)(m + 1) * P.Npad);
  P.Z = (double*)dev_alloc(P, sizeof(double) * (size_t)mz * P.Npad);
  P.x = (double*)dev_alloc(P, sizeof(double) * P.Npad);
  P.tmp = (double*)dev_alloc(P, sizeof(double) * P.Npad);
  P.sc = (SolverScalars*)dev_alloc(P, sizeof(SolverScalars));
  // reduction blocks: two per SM for large vectors, fewer for small ones (every thread
  // takes at least four double2 pairs); the sums depend only on this count
  const int64_t pairs_per_block = (int64_t)kRedThreads * 4;
  P.red_blocks = (int)std::min<int64_t>(2 * kNumSMs, std::max<int64_t>(1, (P.Npad / 2 + pairs_per_block - 1) / pairs_per_block));
  P.partial = (double*)dev_alloc(P, sizeof(double) * (size_t)P.red_blocks * (kMaxRestart + 4));
  P.counter = (unsigned int*)dev_alloc(P, sizeof(unsigned int) * 4);
  if (!P.V || !P.Z || !P.x || !P.tmp || !P.sc || !P.partial || !P.counter) return IIM_ERR_BUDGET;
  cudaMemsetAsync(P.V, 0, sizeof(double) * (size_t)(m + 1) * P.Npad, P.stream);
  cudaMemsetAsync(P.Z, 0, sizeof(double) * (size_t)mz * P.Npad, P.stream);
  cudaMemsetAsync(P.x, 0, sizeof(double) * P.Npad, P.stream);
  cudaMemsetAsync(P.tmp, 0, sizeof(double) * P.Npad, P.stream);
  cudaMemsetAsync(P.counter, 0, sizeof(unsigned int) * 4, P.stream);
  return IIM_OK;
}

// one multidot (which = 0) or update (which = 1) pass over v_0..v_j; close: the update ends the iteration
static void orth_pass(Problem& P, int j, int which, int second, int close, cudaStream_t s) {
  switch (j + 1) {
#define IIM_CASE(k)                                                                                                 \
  case k:                                                                                                           \
    if (which == 0)                                                                                                 \
      IIM_LAUNCH_PDL(k_multidot<k>, P.red_blocks, kRedThreads, 0, s, (const double*)P.V, P.Npad, j, P.partial, P.counter, P.sc, second); \
    else                                                                                                            \
      IIM_LAUNCH_PDL(k_update<k>, P.red_blocks, kRedThreads, 0, s, P.V, P.Npad, j, P.partial, P.counter, P.sc, second, close,   \
                     P.d_status + 1);                                                                               \
    break;
    IIM_CASE(1) IIM_CASE(2) IIM_CASE(3) IIM_CASE(4) IIM_CASE(5) IIM_CASE(6) IIM_CASE(7) IIM_CASE(8)
    IIM_CASE(9) IIM_CASE(10) IIM_CASE(11) IIM_CASE(12) IIM_CASE(13) IIM_CASE(14) IIM_CASE(15) IIM_CASE(16)
#undef IIM_CASE
  }
}

void krylov_orth_pass(Problem& P, int j, int which, cudaStream_t s) { orth_pass(P, j, which, 0, 0, s); }

// Augmented system (pure Neumann, Sec. 2.3): w = L u + alpha 1 on the unknowns, w_N = 1^T u.
// The sum is deterministic: block partials in a fixed grid, summed by the last block to finish (a
// launch of one thread for that took 18 us).
__global__ void __launch_bounds__(256) k_aug_apply(const double* __restrict__ u, double* __restrict__ w,
                                                   const uint8_t* __restrict__ phase, int64_t N, double* partial,
                                                   unsigned int* counter) {
  const double alpha = u[N];
  double acc[1] = {0.0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
    if (phase[i]) {
      w[i] += alpha;
      acc[0] += u[i];
    }
  block_reduce_store<1>(acc, partial, 1, blockIdx.x);
  if (!last_block(counter, gridDim.x)) return;
  __shared__ double tot[1];
  sum_partials<1>(partial, gridDim.x, 1, 1, tot);
  if (threadIdx.x == 0) {
    *counter = 0;
    w[N] = tot[0];
  }
}

// z_N = v_N (scaled like the rest of v): the preconditioner is the identity on alpha
__global__ void k_aug_pass(const double* __restrict__ v, const double* __restrict__ vscale, double* __restrict__ z,
                           int64_t N) {
  if (threadIdx.x == 0 && blockIdx.x == 0) z[N] = v[N] * (vscale ? *vscale : 1.0);
}

// the operator of the Krylov iteration
static void krylov_apply(Problem& P, const double* u, double* w, cudaStream_t s) {
  ho_apply(P, u, w, false, s);
  if (!P.aug) return;
  IIM_LAUNCH(k_aug_apply, P.red_blocks, kRedThreads, 0, s, u, w, P.phase, P.g.N, P.partial, P.counter);
}

// the preconditioner of the Krylov iteration: z = M(v * vscale) (identity on alpha)
static void krylov_precondition(Problem& P, const double* v, const double* vscale, double* z, cudaStream_t s) {
  mg_precondition(P, v, vscale, z, s);
  if (P.aug) IIM_LAUNCH(k_aug_pass, 1, 32, 0, s, v, vscale, z, P.g.N);
}

static bool left_prec(const Problem& P) { return P.opt.krylov == IIM_KRYLOV_GMRES_LEFT; }

static void enqueue_iteration(Problem& P, int j, cudaStream_t s) {
  double* vj = P.V + (size_t)j * P.Npad;
  double* w = P.V + (size_t)(j + 1) * P.Npad;
  if (left_prec(P)) {
    krylov_apply(P, vj, P.tmp, s);                                  // L v_j (v_j unnormalised)
    krylov_precondition(P, P.tmp, &P.sc->inv_norm[j], w, s);       // w = M L v_j / |v_j|
  } else {
    double* zj = P.Z + (size_t)j * P.Npad;
    krylov_precondition(P, vj, &P.sc->inv_norm[j], zj, s);
    krylov_apply(P, zj, w, s);
  }
  for (int pass = 0; pass < (P.opt.reorth ? 2 : 1); ++pass) {
    orth_pass(P, j, 0, pass, 0, s);
    orth_pass(P, j, 1, pass, 1, s);
  }
}

// left preconditioning: V0 = M (b - L x), measured (first: 0 restart, 3 start)
static void enqueue_left_residual(Problem& P, cudaStream_t s, int first) {
  const int64_t n = P.g.N + P.aug;
  double* r = P.Z;   // scratch
  krylov_apply(P, P.x, P.tmp, s);
  IIM_LAUNCH(k_sub, 4 * kNumSMs, 256, 0, s, P.b, P.tmp, r, n);
  krylov_precondition(P, r, nullptr, P.V, s);
  IIM_LAUNCH(k_residual, P.red_blocks, kRedThreads, 0, s, nullptr, nullptr, P.V, n, P.partial, P.counter, P.sc,
             first, P.d_status + 1);
}

static void enqueue_restart(Problem& P, cudaStream_t s) {
  if (left_prec(P)) {
    IIM_LAUNCH(k_xupdate, 4 * kNumSMs, 256, 0, s, P.x, P.V, P.Npad, P.g.N + P.aug, P.sc, 1);
    enqueue_left_residual(P, s, 0);
    return;
  }
  IIM_LAUNCH(k_xupdate, 4 * kNumSMs, 256, 0, s, P.x, P.Z, P.Npad, P.g.N + P.aug, P.sc, 0);
  krylov_apply(P, P.x, P.tmp, s);
  IIM_LAUNCH(k_residual, P.red_blocks, kRedThreads, 0, s, P.b, P.tmp, P.V, P.g.N + P.aug, P.partial, P.counter, P.sc,
             0, P.d_status + 1);
}

static void enqueue_start(Problem& P, cudaStream_t s, int graph_mode) {
  IIM_LAUNCH(k_init_scalars, 1, 1, 0, s, P.sc, P.opt.restart, P.opt.max_iter, P.opt.tol, graph_mode, P.opt.reorth);
  if (left_prec(P)) {
    // |M b| first (the reference of the stopping test), then the preconditioned residual
    krylov_precondition(P, P.b, nullptr, P.V, s);
    IIM_LAUNCH(k_residual, P.red_blocks, kRedThreads, 0, s, nullptr, nullptr, P.V, P.g.N + P.aug, P.partial,
               P.counter, P.sc, 2, P.d_status + 1);
    enqueue_left_residual(P, s, 3);
    return;
  }
  krylov_apply(P, P.x, P.tmp, s);
  IIM_LAUNCH(k_residual, P.red_blocks, kRedThreads, 0, s, P.b, P.tmp, P.V, P.g.N + P.aug, P.partial, P.counter, P.sc,
             1, P.d_status + 1);
}

static int64_t launches_now() { return iim_launch_count(); }

// host-driven loop (one synchronisation per iteration); used when graphs are off
void krylov_enqueue_solve(Problem& P, double* x, bool graph_mode) {
  cudaStream_t s = P.stream;
  (void)x;
  enqueue_start(P, s, 0);
  SolverScalars h;
  for (;;) {
    cudaMemcpyAsync(&h, P.sc, sizeof(SolverScalars), cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    if (h.done) break;
    for (int j = 0; j < P.opt.restart; ++j) {
      enqueue_iteration(P, j, s);
      cudaMemcpyAsync(&h, P.sc, sizeof(SolverScalars), cudaMemcpyDeviceToHost, s);
      cudaStreamSynchronize(s);
      if (!h.active) break;
    }
    enqueue_restart(P, s);
  }
}

// Add a conditional node after the capture's current dependencies and make it the
// only dependency of what follows; *body receives the node's body graph.
static cudaError_t add_conditional(cudaGraph_t g, cudaStream_t s, cudaGraphConditionalHandle h,
                                   cudaGraphConditionalNodeType type, cudaGraph_t* body) {
  const cudaGraphNode_t* deps = nullptr;
  size_t ndeps = 0;
  cudaStreamCaptureStatus st;
  cudaError_t e = cudaStreamGetCaptureInfo(s, &st, nullptr, nullptr, &deps, nullptr, &ndeps);
  if (e != cudaSuccess) return e;
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = h;
  cp.conditional.type = type;
  cp.conditional.size = 1;
  cudaGraphNode_t node;
  e = cudaGraphAddNode(&node, g, deps, nullptr, ndeps, &cp);
  if (e != cudaSuccess) return e;
  e = cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
  if (e != cudaSuccess) return e;
  *body = cp.conditional.phGraph_out[0];
  return cudaSuccess;
}

// Build the solve graph once per problem.  The solve reads and writes P.x.
// Every graph and capture call is checked; on a failure the capture is ended, the
// graph and the stream are destroyed and the error names the call.
iim_status krylov_build_graph(Problem& P, double* x) {
  (void)x;
  cudaStream_t s;
  cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error(std::string("solve graph: cudaStreamCreateWithFlags: ") + cudaGetErrorString(e));
    return IIM_ERR_CUDA;
  }
  cudaGraph_t g = nullptr;
  const char* failed = nullptr;
  auto ok = [&](cudaError_t r, const char* what) {
    if (r != cudaSuccess && !failed) {
      failed = what;
      e = r;
    }
    return failed == nullptr;
  };
  auto fail = [&]() -> iim_status {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
      cudaGraph_t captured = nullptr;     // the graph captured into: g or one of its bodies
      cudaStreamEndCapture(s, &captured);
    }
    cudaGetLastError();
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(s);
    set_error(std::string("solve graph: ") + failed + ": " + cudaGetErrorString(e));
    return IIM_ERR_CUDA;
  };
  // capture into an existing graph: end the capture and check that the stream's work
  // recorded without error
  auto end_capture = [&](const char* what) {
    cudaGraph_t captured = nullptr;
    if (!ok(cudaStreamEndCapture(s, &captured), what)) return false;
    return ok(cudaGetLastError(), what);
  };
  const int m = P.opt.restart;
  cudaGraphConditionalHandle hw;
  if (!ok(cudaGraphCreate(&g, 0), "cudaGraphCreate")) return fail();
  if (!ok(cudaGraphConditionalHandleCreate(&hw, g, 0, 0), "cudaGraphConditionalHandleCreate")) return fail();
  if (!ok(cudaStreamBeginCaptureToGraph(s, g, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed),
          "cudaStreamBeginCaptureToGraph (start)"))
    return fail();
  int64_t c0 = launches_now();
  enqueue_start(P, s, 1);
  P.kern_start = launches_now() - c0;
  cudaGraph_t body = nullptr;
  if (!ok(add_conditional(g, s, hw, cudaGraphCondTypeWhile, &body), "conditional WHILE node")) return fail();
  if (!end_capture("cudaStreamEndCapture (start)")) return fail();
  std::vector<cudaGraphConditionalHandle> hif(m);
  for (int j = 0; j < m; ++j)
    if (!ok(cudaGraphConditionalHandleCreate(&hif[j], body, 0, 0), "cudaGraphConditionalHandleCreate (IF)"))
      return fail();
  if (!ok(cudaStreamBeginCaptureToGraph(s, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed),
          "cudaStreamBeginCaptureToGraph (restart)"))
    return fail();
  std::vector<cudaGraph_t> ibody(m);
  for (int j = 0; j < m; ++j)
    if (!ok(add_conditional(body, s, hif[j], cudaGraphCondTypeIf, &ibody[j]), "conditional IF node")) return fail();
  c0 = launches_now();
  enqueue_restart(P, s);
  P.kern_restart = launches_now() - c0;
  if (!end_capture("cudaStreamEndCapture (restart)")) return fail();
  for (int j = 0; j < m; ++j) {
    if (!ok(cudaStreamBeginCaptureToGraph(s, ibody[j], nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed),
            "cudaStreamBeginCaptureToGraph (iteration)"))
      return fail();
    c0 = launches_now();
    enqueue_iteration(P, j, s);
    P.kern_iter[j] = launches_now() - c0;
    if (!end_capture("cudaStreamEndCapture (iteration)")) return fail();
  }
  // the handles live in the solver scalars so that kernels can set them
  GraphHandles H = {};
  H.h_while = hw;
  H.m = m;
  for (int j = 0; j < m; ++j) H.h_if[j] = hif[j];
  k_set_handles<<<1, 1, 0, s>>>(P.sc, H);
  note_launch();
  if (!ok(cudaGetLastError(), "k_set_handles launch")) return fail();
  if (!ok(cudaStreamSynchronize(s), "cudaStreamSynchronize")) return fail();
  cudaGraphExec_t ge = nullptr;
  if (!ok(cudaGraphInstantiate(&ge, g, 0), "cudaGraphInstantiate")) return fail();
  cudaStreamDestroy(s);
  P.graph_exec = ge;
  P.graph = g;
  return IIM_OK;
}

void krylov_read_info(Problem& P, iim_solve_info* info) {
  SolverScalars h;
  cudaMemcpy(&h, P.sc, sizeof(SolverScalars), cudaMemcpyDeviceToHost);
  if (!info) return;
  // kernels executed by the graph: start + restarts x restart body + iterations
  // (iterations of a cycle are consecutive from j = 0)
  int64_t kern = P.kern_start + (int64_t)h.restarts * P.kern_restart;
  {
    int left = h.iters, m = P.opt.restart;
    while (left > 0) {
      int take = left < m ? left : m;
      for (int j = 0; j < take; ++j) kern += P.kern_iter[j];
      left -= take;
    }
  }
  info->kernels = kern;
  info->iters = h.iters;
  info->restarts = h.restarts;
  info->converged = h.converged;
  info->relres = h.relres;
}


// ---------------------------------------------------------------------------- batched engine
// Plan of a tick (one block per per-tick list).  The role of a slot follows from its
// FGMRES state (or is ITER for every slot with force_iter, for the autotuner); block 0
// writes roles and iteration indices into the slot descriptors, and block k copies
// static list k keeping the slots whose role uses it, with their item prefix sums.
__global__ void __launch_bounds__(1024) k_eng_plan(EngArgs A, int* dyn, int force_iter) {
  const int b = blockIdx.x;
  auto role_of = [&](int si) -> int {
    if (force_iter) return kRoleIter;
    const SolverScalars* S = A.slots[si].sc;
    return S->done ? kRoleIdle : (S->active ? kRoleIter : kRoleRestart);
  };
  if (b == 0) {
    const int* L = A.slist(kListAll);
    const int count = L[0];
    const int* slot = L + 2 + A.cap;
    for (int e = threadIdx.x; e < count; e += blockDim.x) {
      SlotDev& sd = A.slots[slot[e]];
      sd.role = role_of(slot[e]);
      sd.j = force_iter ? 0 : sd.sc->k;
    }
  }
  const int mask = eng_list_mask(b);
  const int* L = A.slist(eng_list_source(b));
  const int count = L[0];
  const int* pre = L + 1;
  const int* slot = L + 2 + A.cap;
  int* D = dyn + (size_t)b * (2 * A.cap + 2);
  int* dpre = D + 1;
  int* dslot = D + 2 + A.cap;
  __shared__ int wn[32], wi[32];
  __shared__ int base_n, base_i, tot_n, tot_i;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if (threadIdx.x == 0) { base_n = 0; base_i = 0; }
  __syncthreads();
  for (int c0 = 0; c0 < count; c0 += blockDim.x) {
    const int e = c0 + threadIdx.x;
    int keep = 0, items = 0, si = 0;
    if (e < count) {
      si = slot[e];
      items = pre[e + 1] - pre[e];
      keep = ((mask >> role_of(si)) & 1) && items > 0;
      if (!keep) items = 0;
    }
    // block-wide exclusive scans of keep and items
    int in = keep, ii = items;
    for (int o = 1; o < 32; o <<= 1) {
      const int yn = __shfl_up_sync(0xffffffffu, in, o), yi = __shfl_up_sync(0xffffffffu, ii, o);
      if (lane >= o) { in += yn; ii += yi; }
    }
    if (lane == 31) { wn[wid] = in; wi[wid] = ii; }
    __syncthreads();
    if (wid == 0) {
      int vn = lane < nw ? wn[lane] : 0, vi = lane < nw ? wi[lane] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        const int yn = __shfl_up_sync(0xffffffffu, vn, o), yi = __shfl_up_sync(0xffffffffu, vi, o);
        if (lane >= o) { vn += yn; vi += yi; }
      }
      if (lane < nw) { wn[lane] = vn; wi[lane] = vi; }
      if (lane == nw - 1) { tot_n = vn; tot_i = vi; }
    }
    __syncthreads();
    const int xn = in - keep + (wid > 0 ? wn[wid - 1] : 0);
    const int xi = ii - items + (wid > 0 ? wi[wid - 1] : 0);
    if (keep) {
      dslot[base_n + xn] = si;
      dpre[base_n + xn] = base_i + xi;
    }
    __syncthreads();
    if (threadIdx.x == 0) { base_n += tot_n; base_i += tot_i; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    D[0] = base_n;
    dpre[base_n] = base_i;
  }
}

__global__ void __launch_bounds__(256) k_eng_xupdate(EngArgs A) {
  eng_for_items(A, kListXup, [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role != kRoleRestart) return;
    xupdate_body(s.x, s.Z, s.Npad, s.g.N, s.sc, item, s.xup_blocks);
  });
}

__global__ void __launch_bounds__(kRedThreads) k_eng_multidot(EngArgs A, int second) {
  eng_for_items(A, kListRed, [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role != kRoleIter) return;
    multidot_body<kMaxRestart, false>(s.V, s.Npad, s.j, s.j + 1, s.partial, s.counter, s.sc, second, item, s.red_blocks);
  });
}

__global__ void __launch_bounds__(kRedThreads) k_eng_update(EngArgs A, int second) {
  eng_for_items(A, kListRed, [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role != kRoleIter) return;
    update_body<kMaxRestart, false>(s.V, s.Npad, s.j, s.j + 1, s.partial, s.counter, s.sc, second, item, s.red_blocks, true,
                             s.status);
  });
}

__global__ void __launch_bounds__(kRedThreads) k_eng_residual(EngArgs A) {
  eng_for_items(A, kDynRedRestart, [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role != kRoleRestart) return;
    residual_body(s.b, s.tmp, s.V, s.g.N, s.partial, s.counter, s.sc, s.sc->first, s.status, item, s.red_blocks);
  });
}

// End of a tick: done flags per slot, the number of unfinished slots, the tick budget
// and the loop condition of the run graph (one block)
__global__ void __launch_bounds__(256) k_eng_tick_end(EngArgs A, int* live, int* done_flags, int* ticks_left,
                                                      cudaGraphConditionalHandle h, int use_cond) {
  const int* L = A.slist(kListAll);
  const int count = L[0];
  const int* slot = L + 2 + A.cap;
  int mine = 0;
  for (int e = threadIdx.x; e < count; e += blockDim.x) {
    const int si = slot[e];
    const int d = A.slots[si].sc->done;
    done_flags[si] = d;
    mine += !d;
  }
  __shared__ int red[256 / 32];
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    int n = 0;
    for (int k = 0; k < 256 / 32; ++k) n += red[k];
    *live = n;
    const int t = *ticks_left - 1;
    *ticks_left = t;
    if (use_cond) cudaGraphSetConditional(h, (n > 0 && t > 0) ? 1u : 0u);
  }
}

void eng_launch_plan(const EngArgs& A, int* dyn, int force_iter, cudaStream_t s) {
  IIM_LAUNCH(k_eng_plan, kDynCount, 1024, 0, s, A, dyn, force_iter);
}

void eng_launch_krylov_head(const EngArgs& A, int* dyn, cudaStream_t s) {
  eng_launch_plan(A, dyn, 0, s);
  IIM_LAUNCH(k_eng_xupdate, eng_grid((const void*)k_eng_xupdate, 256, 0), 256, 0, s, A);
}

// ctl: [0] unfinished slots, [1] tick budget, [2 + slot] done flag of each slot
void eng_launch_krylov_tail(const EngArgs& A, int* ctl, cudaGraphConditionalHandle h, int use_cond, cudaStream_t s) {
  const int gr = eng_grid((const void*)k_eng_multidot, kRedThreads, 0);
  const int gu = eng_grid((const void*)k_eng_update, kRedThreads, 0);
  IIM_LAUNCH(k_eng_multidot, gr, kRedThreads, 0, s, A, 0);
  IIM_LAUNCH(k_eng_update, gu, kRedThreads, 0, s, A, 0);
  IIM_LAUNCH(k_eng_multidot, gr, kRedThreads, 0, s, A, 1);
  IIM_LAUNCH(k_eng_update, gu, kRedThreads, 0, s, A, 1);
  IIM_LAUNCH(k_eng_residual, eng_grid((const void*)k_eng_residual, kRedThreads, 0), kRedThreads, 0, s, A);
  IIM_LAUNCH(k_eng_tick_end, 1, 256, 0, s, A, ctl, ctl + 2, ctl + 1, h, use_cond);
}

void eng_init_scalars(Problem& P, cudaStream_t s) {
  IIM_LAUNCH(k_init_scalars, 1, 1, 0, s, P.sc, P.opt.restart, P.opt.max_iter, P.opt.tol, 0, P.opt.reorth);
}

}  // namespace iim
