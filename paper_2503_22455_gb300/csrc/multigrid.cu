// Shortley-Weller geometric multigrid V-cycle (paper Sec. 3.3), FP32 or FP64.
//
// Cell-centred levels n, n/2, ...; red-black Gauss-Seidel (red = even index
// sum, red first); residual + restriction as the mean of the 2^d children with
// zeros outside the domain; bi/trilinear interpolation with zeros outside the
// domain (Dirichlet, interface) or the mean of the in-domain coarse neighbours
// (Neumann, Sec. 3.3); a dense direct solve on the coarsest level.  Interface
// problems run on lap(u) = f/beta per phase (Sec. 3.3): the FP64 Krylov vector
// is divided by beta_sigma when it enters the FP32 hierarchy.
#include <algorithm>
#include <type_traits>
#include <utility>

#include "engine.cuh"
#include "mg_rb.cuh"
#include "mg_3d.cuh"

namespace iim {

template <typename T>
struct LevelView {
  GridView g;
  const int32_t* aux;
  const T* tab;
};

template <typename T>
__device__ inline T tabv(const LevelView<T>& L, int r, int k) {
  return L.tab[(size_t)r * sw_row(L.g.dim) + k];
}

__device__ inline void idx3(const GridView& g, int64_t i, int* m) {
  m[0] = (int)(i % g.n);
  int64_t r = i / g.n;
  m[1] = (int)(r % g.n);
  m[2] = g.dim > 2 ? (int)(r / g.n) : 0;
}

// the neighbours' values (-x, +x, -y, +y, -z, +z), zero beyond the grid
template <typename T>
__device__ inline void neighbours(const GridView& g, int64_t i, const int* m, const T* __restrict__ u, T (&v)[6]) {
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const int64_t st = ax == 0 ? 1 : (ax == 1 ? (int64_t)g.n : (int64_t)g.n * g.n);
    v[2 * ax] = ax < g.dim && m[ax] > 0 ? u[i - st] : (T)0;
    v[2 * ax + 1] = ax < g.dim && m[ax] < g.n - 1 ? u[i + st] : (T)0;
  }
}

// Gauss-Seidel value and residual of a node (aux code a) in the arithmetic of the fused kernels.  3D:
// every node is a row of weights (ih2 in a regular one) with the diagonal's reciprocal.
template <typename T>
__device__ inline T off_residual_node(const LevelView<T>& L, T ih2, int a, T f, const T (&v)[6]) {
  if (a == -1) return off_residual3(f, ih2, ih2, ih2, ih2, ih2, ih2, v[0], v[1], v[2], v[3], v[4], v[5]);
  return off_residual3(f, tabv(L, a, 1), tabv(L, a, 2), tabv(L, a, 3), tabv(L, a, 4), tabv(L, a, 5), tabv(L, a, 6), v[0],
                       v[1], v[2], v[3], v[4], v[5]);
}
template <typename T>
__device__ inline T irregular_sum2(const LevelView<T>& L, int a, const T (&v)[6]) {
  return irr_offdiag(tabv(L, a, 1), tabv(L, a, 2), tabv(L, a, 3), tabv(L, a, 4), v[0], v[1], v[2], v[3]);
}
template <typename T>
__device__ inline T gs_node(const LevelView<T>& L, T ih2, T inv_dreg, int a, T f, const T (&v)[6]) {
  if (L.g.dim > 2) return mul_rn(off_residual_node(L, ih2, a, f, v), a == -1 ? inv_dreg : tabv(L, a, 7));
  if (a == -1) return gs_regular(f, (v[0] + v[1]) + (v[2] + v[3]), ih2, inv_dreg);
  const T dg = tabv(L, a, 0);
  return dg != (T)0 ? (f - irregular_sum2(L, a, v)) / dg : (T)0;
}
template <typename T>
__device__ inline T residual_node(const LevelView<T>& L, T ih2, T dreg, int a, T f, T u, const T (&v)[6]) {
  if (L.g.dim > 2) return fma(-(a == -1 ? dreg : tabv(L, a, 0)), u, off_residual_node(L, ih2, a, f, v));
  if (a != -1) return f - fma(tabv(L, a, 0), u, irregular_sum2(L, a, v));
  return res_regular(f, u, (v[0] + v[1]) + (v[2] + v[3]), dreg, ih2);
}

template <typename T>
__device__ inline T diag_of(const LevelView<T>& L, T dreg, int a) {
  if (a == -1) return dreg;
  return tabv(L, a, 0);
}

template <typename T>
__device__ __forceinline__ void smooth_body(const LevelView<T>& L, T ih2, T inv_dreg, T* __restrict__ u,
                                            const T* __restrict__ f, int f_bf16, int colour, int64_t t) {
  // one thread per node of the colour: node = 2 * t + parity fix-up along x
  const GridView& g = L.g;
  int64_t rows = g.N / g.n;
  int64_t half = (g.n + 1) / 2;
  if (t >= rows * half) return;
  int64_t row = t / half;
  int xi = (int)(t - row * half) * 2;
  int ry = (int)(row % g.n), rz = g.dim > 2 ? (int)(row / g.n) : 0;
  if (((xi + ry + rz) & 1) != colour) xi += 1;
  if (xi >= g.n) return;
  int64_t i = row * g.n + xi;
  int a = L.aux[i];
  if (a == -2) return;
  int m[3] = {xi, ry, rz};
  T v[6];
  neighbours(g, i, m, u, v);
  u[i] = gs_node(L, ih2, inv_dreg, a, load_f(f, i, f_bf16), v);
}

template <typename T>
__global__ void __launch_bounds__(256) k_smooth(LevelView<T> L, T ih2, T inv_dreg, T* __restrict__ u,
                                                const T* __restrict__ f, int f_bf16, int colour) {
  smooth_body<T>(L, ih2, inv_dreg, u, f, f_bf16, colour, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// coarse f = mean over the 2^d children of r = f - L u (zero at non-unknowns)
template <typename T>
__device__ __forceinline__ void resid_restrict_body(const LevelView<T>& F, T ih2, T dreg, const T* __restrict__ u,
                                                    const T* __restrict__ f, int f_in_bf16, const GridView& gc,
                                                    const int32_t* __restrict__ aux_c, T* __restrict__ fc, int64_t I,
                                                    int f_bf16) {
  if (I >= gc.N) return;
  if (aux_c[I] == -2) { store_f(fc, I, (T)0, f_bf16); return; }
  int mc[3];
  idx3(gc, I, mc);
  const GridView& g = F.g;
  // rows first, then the two rows of a plane, then the planes
  T r[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    r[c] = (T)0;
    if (c >= (1 << g.dim)) continue;
    int m[3] = {2 * mc[0] + (c & 1), 2 * mc[1] + ((c >> 1) & 1), g.dim > 2 ? 2 * mc[2] + ((c >> 2) & 1) : 0};
    int64_t i = m[0] + (int64_t)g.n * m[1] + (int64_t)g.n * g.n * m[2];
    int a = F.aux[i];
    if (a == -2) continue;
    T v[6];
    neighbours(g, i, m, u, v);
    r[c] = residual_node(F, ih2, dreg, a, load_f(f, i, f_in_bf16), u[i], v);
  }
  const T lo = (r[0] + r[1]) + (r[2] + r[3]);
  store_f(fc, I, g.dim > 2 ? (lo + ((r[4] + r[5]) + (r[6] + r[7]))) * (T)0.125 : lo * (T)0.25, f_bf16);
}

template <typename T>
__global__ void __launch_bounds__(256) k_resid_restrict(LevelView<T> F, T ih2, T dreg, const T* __restrict__ u,
                                                        const T* __restrict__ f, int f_in_bf16, GridView gc,
                                                        const int32_t* __restrict__ aux_c, T* __restrict__ fc,
                                                        int f_bf16) {
  resid_restrict_body<T>(F, ih2, dreg, u, f, f_in_bf16, gc, aux_c, fc, (int64_t)blockIdx.x * blockDim.x + threadIdx.x,
                         f_bf16);
}

// u_fine += P e_coarse at fine unknowns
template <typename T>
__device__ __forceinline__ void prolong_body(const GridView& gf, const int32_t* __restrict__ aux_f, T* __restrict__ uf,
                                             const GridView& gc, const int32_t* __restrict__ aux_c,
                                             const T* __restrict__ ec, int neumann, int64_t i) {
  if (i >= gf.N) return;
  if (aux_f[i] == -2) return;
  int m[3];
  idx3(gf, i, m);
  int I[3] = {m[0] >> 1, m[1] >> 1, m[2] >> 1};
  int sg[3] = {(m[0] & 1) ? 1 : -1, (m[1] & 1) ? 1 : -1, (m[2] & 1) ? 1 : -1};
  T ev[8];
  unsigned ok = 0;
#pragma unroll
  for (int sel = 0; sel < 8; ++sel) {
    ev[sel] = (T)0;
    if (sel >= (1 << gf.dim)) continue;
    int c[3];
    bool inb = true;
    for (int k = 0; k < 3; ++k) {
      c[k] = k < gf.dim ? I[k] + ((sel >> k) & 1) * sg[k] : 0;
      if (k < gf.dim && (c[k] < 0 || c[k] >= gc.n)) inb = false;
    }
    if (!inb) continue;
    int64_t ci = c[0] + (int64_t)gc.n * c[1] + (int64_t)gc.n * gc.n * c[2];
    if (aux_c[ci] == -2) continue;
    ev[sel] = ec[ci];
    ok |= 1u << sel;
  }
  uf[i] += neumann ? prolong_mean8(ev, ok)
                   : (gf.dim > 2 ? prolong_trilinear(ev) : prolong_bilinear(ev[0], ev[1], ev[2], ev[3]));
}

template <typename T>
__global__ void __launch_bounds__(256) k_prolong(GridView gf, const int32_t* __restrict__ aux_f, T* __restrict__ uf,
                                                 GridView gc, const int32_t* __restrict__ aux_c,
                                                 const T* __restrict__ ec, int neumann) {
  prolong_body<T>(gf, aux_f, uf, gc, aux_c, ec, neumann, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// f_fine = v * scale / beta_sigma at unknowns (FP64 -> level precision)
template <typename T>
__device__ __forceinline__ void bridge_in_body(const GridView& g, const double* __restrict__ v,
                                               const double* __restrict__ scale, const uint8_t* __restrict__ phase,
                                               const int32_t* __restrict__ aux, double inv_bp, double inv_bm,
                                               T* __restrict__ f, int64_t i) {
  if (i >= g.N) return;
  if (aux[i] == -2) { f[i] = (T)0; return; }
  f[i] = mul_rn((T)v[i], mul_rn((T)(scale ? *scale : 1.0), (T)(phase[i] ? inv_bp : inv_bm)));
}

template <typename T>
__global__ void k_bridge_in(GridView g, const double* __restrict__ v, const double* __restrict__ scale,
                            const uint8_t* __restrict__ phase, const int32_t* __restrict__ aux, double inv_bp,
                            double inv_bm, T* __restrict__ f) {
  bridge_in_body<T>(g, v, scale, phase, aux, inv_bp, inv_bm, f, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename T>
__global__ void k_zero(T* __restrict__ u, int64_t N) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) u[i] = (T)0;
}

template <typename T>
__global__ void k_bridge_out(GridView g, const T* __restrict__ u, double* __restrict__ z) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  z[i] = (double)u[i];
}

// ---------------------------------------------------------------------------- coarsest level
// The coarse system has n = nu + aug unknowns, nu counted on the device (a later set-up with
// other geometry keeps the arrays, of fixed stride ld >= n).  Its dense inverse is formed by
// blocked Gauss-Jordan elimination with row pivoting: per block of kGJ (32) columns one CTA
// factors the panel and inverts its pivot block (k_gj_panel), then a grid of 32 x 32 tiles
// carries the step to the whole matrix (k_gj_update).  A step reads one of the two n x n
// buffers and writes the other, so no tile waits for another; the first buffer is chosen so
// that the last step ends in buffer 0, from which k_gj_finish writes the inverse of the matrix
// with its original row order to buffer 1.
// The panel is bound by its chain of pivots (two barriers each, about 0.5 us); the rest of the
// chip is idle meanwhile, but the chain is n long instead of the n^3 / 1024 of one CTA that
// works on the matrix in global memory.  Measured: set-up of a 736^2 exterior star (coarsest
// level 23^2) 82.5 -> 2.8 ms, of a 80^3 sphere interface 43.6 -> 5.5 ms with the fits.
constexpr int kGJ = 32;

struct GJView {                         // sizes of the current set-up's system
  int n, steps;
  __device__ GJView(const int* nu_dev, int aug, int ld, int b) {
    const int nu = *nu_dev;
    n = nu < 0 || nu + aug > ld ? 0 : nu + aug;        // out of range: reported by k_coarse_assemble
    steps = (n + b - 1) / b;
  }
  // buffer (0 or 1) that step k reads
  __device__ int src(int k) const { return (steps + k) & 1; }
};

// rows of the dense matrix (zeroed beforehand): row r < nu the SW operator of unknown r;
// augmented (pure Neumann, Sec. 2.3): a last column and row of ones over the unknowns
template <typename T>
__global__ void k_coarse_assemble(LevelView<double> L, const int32_t* __restrict__ map, const int* __restrict__ nu_dev,
                                  int ld, const int32_t* __restrict__ inv, T* __restrict__ buf, int aug, int b,
                                  int* status) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int nu = *nu_dev;
  if (nu < 0 || nu + aug > ld) {       // more unknowns than the system has room for
    if (r == 0) set_status(status, IIM_ERR_CAPACITY);
    return;
  }
  if (r >= nu) return;
  const GJView V(nu_dev, aug, ld, b);
  T* A = buf + (size_t)V.src(0) * ld * ld;
  if (aug) {
    A[(size_t)r * ld + nu] = (T)1;
    A[(size_t)nu * ld + r] = (T)1;
  }
  int64_t i = map[r];
  int a = L.aux[i];
  int m[3];
  idx3(L.g, i, m);
  A[(size_t)r * ld + r] = (T)diag_of(L, -2.0 * L.g.dim / (L.g.h * L.g.h), a);
  const GridView& g = L.g;
  for (int ax = 0; ax < g.dim; ++ax) {
    int64_t st = ax == 0 ? 1 : (ax == 1 ? (int64_t)g.n : (int64_t)g.n * g.n);
    for (int s = -1; s <= 1; s += 2) {
      int pos = m[ax] + s;
      if (pos < 0 || pos >= g.n) continue;
      double cf = a == -1 ? 1.0 / (g.h * g.h) : tabv(L, a, (s < 0 ? 1 : 2) + 2 * ax);
      if (cf == 0.0) continue;
      int col = inv[i + s * st];
      if (col >= 0) A[(size_t)r * ld + col] = (T)cf;
    }
  }
}

__global__ void k_coarse_map(GridView g, const int32_t* __restrict__ aux, const int32_t* __restrict__ idx,
                             int32_t* __restrict__ map, int32_t* __restrict__ inv) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  if (aux[i] == -2) { inv[i] = -1; return; }
  int k = idx[i];
  map[k] = (int32_t)i;
  inv[i] = k;
}

__global__ void k_unknown_flag(GridView g, const int32_t* __restrict__ aux, int32_t* __restrict__ flag) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < g.N) flag[i] = aux[i] != -2;
}

// Panel of one block step: rows k0 .. n - 1 of columns k0 .. k0 + bb - 1, in shared memory column
// by column; LU with partial pivoting (ties: the lowest row).  Writes the inverse of the pivot
// block, the row each row of the step comes from and the row order so far.
template <typename T>
__global__ void __launch_bounds__(1024) k_gj_panel(const T* __restrict__ buf, int ld, const int* __restrict__ nu_dev,
                                                   int aug, int step, int b, int* __restrict__ order,
                                                   int* __restrict__ from, T* __restrict__ D, int* status) {
  extern __shared__ unsigned char smraw[];
  __shared__ T s_best[2][32];
  __shared__ int s_row[2][32];
  const GJView V(nu_dev, aug, ld, b);
  const int n = V.n, k0 = step * b;
  if (k0 >= n) return;
  const int bb = min(b, n - k0), h = n - k0;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  T* P = (T*)smraw;                      // [bb][h]
  int* rows = (int*)(P + (size_t)bb * h);
  const T* src = buf + (size_t)V.src(step) * ld * ld;
  for (int e = tid; e < h * bb; e += 1024) {
    const int r = e / bb, c = e - r * bb;
    P[(size_t)c * h + r] = src[(size_t)(k0 + r) * ld + k0 + c];
  }
  for (int r = tid; r < h; r += 1024) rows[r] = k0 + r;
  __syncthreads();
  T best = -1;
  int row = h;
  for (int r = tid; r < h; r += 1024) {
    const T v = fabs(P[r]);
    if (v > best) { best = v; row = r; }
  }
  for (int j = 0; j < bb; ++j) {
    for (int o = 16; o > 0; o >>= 1) {
      const T ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int orow = __shfl_xor_sync(0xffffffffu, row, o);
      if (ob > best || (ob == best && orow < row)) { best = ob; row = orow; }
    }
    if (lane == 0) { s_best[j & 1][wid] = best; s_row[j & 1][wid] = row; }
    __syncthreads();
    best = s_best[j & 1][lane];          // every warp reduces the warps' candidates
    row = s_row[j & 1][lane];
    for (int o = 16; o > 0; o >>= 1) {
      const T ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int orow = __shfl_xor_sync(0xffffffffu, row, o);
      if (ob > best || (ob == best && orow < row)) { best = ob; row = orow; }
    }
    if (tid == 0 && !(best > 0)) set_status(status, IIM_ERR_SINGULAR);
    const int p = best >= 0 ? row : j;   // NaN entries only: no candidate
    if (p != j) {
      if (tid < bb) {
        const T t = P[(size_t)tid * h + j];
        P[(size_t)tid * h + j] = P[(size_t)tid * h + p];
        P[(size_t)tid * h + p] = t;
      } else if (tid == 32) {
        const int t = rows[j];
        rows[j] = rows[p];
        rows[p] = t;
      }
    }
    __syncthreads();
    const T d = P[(size_t)j * h + j];
    best = -1;
    row = h;
    for (int r = j + 1 + tid; r < h; r += 1024) {
      const T l = P[(size_t)j * h + r] / d;
      P[(size_t)j * h + r] = l;
      for (int c = j + 1; c < bb; ++c) {
        const T v = P[(size_t)c * h + r] - l * P[(size_t)c * h + j];
        P[(size_t)c * h + r] = v;
        if (c == j + 1 && fabs(v) > best) { best = fabs(v); row = r; }
      }
    }
  }
  __syncthreads();
  if (wid < bb) {
    // column wid of (L U)^-1, rows over the lanes
    T x = lane == wid ? (T)1 : (T)0;
    for (int i = 0; i < bb; ++i) {
      const T xi = __shfl_sync(0xffffffffu, x, i);
      if (lane > i && lane < bb) x -= P[(size_t)i * h + lane] * xi;
    }
    for (int i = bb - 1; i >= 0; --i) {
      const T xi = __shfl_sync(0xffffffffu, x, i) / P[(size_t)i * h + i];
      if (lane == i) x = xi;
      else if (lane < i) x -= P[(size_t)i * h + lane] * xi;
    }
    if (lane < bb) D[lane * kGJ + wid] = x;
  }
  for (int r = tid; r < h; r += 1024) from[k0 + r] = rows[r];
  int old[4];                            // n <= 4096 + 1: at most five rows per thread
  int last = 0;
  for (int r = tid, q = 0; r < h; r += 1024, ++q) {
    const int v = step == 0 ? rows[r] : order[rows[r]];
    if (q < 4) old[q] = v;
    else last = v;
  }
  __syncthreads();
  for (int r = tid, q = 0; r < h; r += 1024, ++q) order[k0 + r] = q < 4 ? old[q] : last;
}

// One 32 x 32 tile of a block step.  With A the matrix in the step's row order and K the pivot
// columns (rows): T = A_KK^-1 A_K: (the inverse itself in the columns K); rows K become T, the
// others A - A_:K T (minus A_:K T in the columns K).
template <typename T>
__global__ void __launch_bounds__(256) k_gj_update(T* __restrict__ buf, int ld, const int* __restrict__ nu_dev, int aug,
                                                   int step, int b, const int* __restrict__ from,
                                                   const T* __restrict__ D) {
  __shared__ T sD[kGJ][kGJ + 1], sK[kGJ][kGJ], sT[kGJ][kGJ], sA[32][kGJ + 1];
  const GJView V(nu_dev, aug, ld, b);
  const int n = V.n, k0 = step * b;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  if (k0 >= n || r0 >= n || c0 >= n) return;
  const int bb = min(b, n - k0);
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const T* src = buf + (size_t)V.src(step) * ld * ld;
  T* dst = buf + (size_t)(1 - V.src(step)) * ld * ld;
  const int c = c0 + tx;
  const bool cK = c >= k0 && c < k0 + bb;
  T a[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int j = ty + 8 * q, r = r0 + j;
    const int fr = r < n ? (r < k0 ? r : from[r]) : 0;
    sD[j][tx] = j < bb && tx < bb ? D[j * kGJ + tx] : (T)0;
    sK[j][tx] = j < bb && c < n ? src[(size_t)from[k0 + j] * ld + c] : (T)0;
    sA[j][tx] = r < n && tx < bb ? src[(size_t)fr * ld + k0 + tx] : (T)0;
    a[q] = r < n && c < n && !cK ? src[(size_t)fr * ld + c] : (T)0;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int j = ty + 8 * q;
    T s = 0;
    if (cK) s = sD[j][c - k0];
    else
      for (int i = 0; i < bb; ++i) s = fma(sD[j][i], sK[i][tx], s);
    sT[j][tx] = s;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int j = ty + 8 * q, r = r0 + j;
    if (r >= n || c >= n) continue;
    T s = a[q];
    if (r >= k0 && r < k0 + bb) s = sT[r - k0][tx];
    else
      for (int i = 0; i < bb; ++i) s = fma(-sA[j][i], sT[i][tx], s);
    dst[(size_t)r * ld + c] = s;
  }
}

// buffer 0 holds the inverse of the matrix with its rows in the order `order`: its columns go
// back to the original rows' places
template <typename T>
__global__ void __launch_bounds__(256) k_gj_finish(T* __restrict__ buf, int ld, const int* __restrict__ nu_dev, int aug,
                                                   int b, const int* __restrict__ order) {
  const GJView V(nu_dev, aug, ld, b);
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c >= V.n) return;
  const int oc = order[c];
  for (int r = blockIdx.y; r < V.n; r += gridDim.y) buf[((size_t)ld + r) * ld + oc] = buf[(size_t)r * ld + c];
}

// ---------------------------------------------------------------------------- host side
template <typename T>
static LevelView<T> view(const Level& L) {
  LevelView<T> v;
  v.g = L.g;
  v.aux = L.aux;
  v.tab = (const T*)(sizeof(T) == 8 ? (const void*)L.tab64 : (const void*)L.tab32);
  return v;
}

// first level handled by the single-CTA tail: the first with at most kTailNodes nodes
static size_t tail_start(const Problem& P) {
  size_t l = 0;
  while (l + 1 < P.lv.size() && P.lv[l].g.N > kTailNodes) ++l;
  return l;
}
size_t mg_tail_start(const Problem& P) { return tail_start(P); }

// Parameters of the single-CTA tail over levels l0 .. end; *smem gets its shared
// memory bytes.  FP32: the irregular-row tables are staged in shared memory when the
// total stays within smem_limit (staging changes where they are read, not the result).
// FP64 always stages them, for its sweeps take rows of a form of their own (tail_row64) and a row
// for the regular nodes that the table does not have.  They always fit: the tail's levels hold up to
// 4/3 kTailNodes nodes, and 5/4 as many rows with 65 more for each level.
static_assert((2 * sizeof(double) + 2 * sizeof(int)) * (4 * kTailNodes / 3) + sizeof(double) * kTailNodes +
                  sizeof(double) * tail_row64(3) * (5 * kTailNodes / 3 + 65 * kTailMaxLevels) <= 227 * 1024,
              "the FP64 tail's rows must fit in shared memory");
template <typename T>
TailParams<T> make_tail_params(Problem& P, size_t l0, T* u_out, size_t smem_limit, size_t* smem) {
  TailParams<T> tp;
  tp.u_out = u_out ? u_out : (T*)P.lv[l0].u;
  tp.nlev = (int)(P.lv.size() - l0);
  int off = 0;
  for (int k = 0; k < tp.nlev; ++k) {
    tp.L[k] = levk<T>(P.lv[l0 + k]);
    tp.off[k] = off;
    off += (int)P.lv[l0 + k].g.N;
  }
  tp.off[tp.nlev] = off;
  int toff = 0;
  for (int k = 0; k < tp.nlev; ++k) {
    const Level& L = P.lv[l0 + k];
    tp.toff[k] = toff;
    tp.tcount[k] = P.d_counts + 2 + (int)(l0 + k);
    tp.tcap[k] = L.irr_cap;
    // (the coarsest level's matrix is used in the dense inverse only; FP64: one more row, regular nodes)
    if (k + 1 < tp.nlev) toff += (L.irr_cap + (sizeof(T) == 8 ? 1 : 0)) * tail_row<T>(L.g.dim);
  }
  tp.toff[tp.nlev] = toff;
  // u, f, aux, node coordinates; FP64: residuals of the largest level
  const size_t base = (sizeof(T) * 2 + 2 * sizeof(int)) * (size_t)off +
                      (sizeof(T) == 8 && tp.nlev > 1 ? sizeof(T) * (size_t)tp.off[1] : 0);
  tp.stage_tables = sizeof(T) == 8 || base + sizeof(T) * (size_t)toff <= smem_limit;
  if (!tp.stage_tables) {
    toff = 0;
    for (int k = 0; k <= tp.nlev; ++k) tp.toff[k] = 0;
  }
  tp.nu1 = P.opt.nu1;
  tp.nu2 = P.opt.nu2;
  tp.gamma = P.opt.cycle;
  tp.top_visits = 1;
  tp.neumann = P.desc.bc == IIM_BC_NEUMANN;
  tp.ld = P.coarse_n;
  tp.nu_dev = P.d_counts + kCountCoarse;
  tp.aug = P.aug;
  tp.map = P.coarse_map;
  tp.status = P.d_status + 1;
  const T* inv = (const T*)(sizeof(T) == 8 ? (void*)P.coarse_lu64 : (void*)P.coarse_lu32);
  tp.inv = inv + (size_t)P.coarse_n * P.coarse_n;
  tp.v = nullptr;
  tp.vscale = nullptr;
  tp.phase = P.phase;
  tp.inv_bp = (T)(1.0 / P.desc.beta_plus);
  tp.inv_bm = (T)(1.0 / P.desc.beta_minus);
  tp.z = nullptr;
  *smem = base + sizeof(T) * (size_t)toff;
  return tp;
}
template TailParams<float> make_tail_params<float>(Problem&, size_t, float*, size_t, size_t*);

// The tail entered from a finer level runs all gamma visits of its first level (they
// follow one another with the same right-hand side); from the finest level, one.
template <typename T>
static void launch_tail(Problem& P, size_t l0, const double* v, const double* vscale, double* z, cudaStream_t s,
                        T* u_out = nullptr) {
  size_t smem = 0;
  TailParams<T> tp = make_tail_params<T>(P, l0, u_out, 200 * 1024, &smem);
  tp.top_visits = l0 == 0 ? 1 : P.opt.cycle;
  tp.v = v;
  tp.vscale = vscale;
  tp.z = z;
  // A dense inverse too large for one SM to read or (FP64) to multiply in a few us is split over a
  // cluster of eight, whose two barriers cost 1.5 us.  Tail alone / in a cluster, us, by the coarsest
  // level's nodes: FP32 64: 14.4 / 15.5, 100: 8.9 / 9.4, 144: 10.9 / 11.0, 169: 11.1 / 11.0, 196: 12.0 /
  // 11.4, 225: 12.1 / 11.5, 289: 8.2 / 5.1, 529: 12.8 / 6.2, 3D 125: 15.2 / 15.4, 216: 6.6 / 4.7; FP64
  // 64: 23.7 / 23.9, 100: 13.5 / 12.1, 121: 17.9 / 13.7, 289: 27.8 / 7.7, 529: 59.3 / 12.5.  (FP32
  // sizes between 144 and the line of 200 would gain 0.2 to 0.6 us; a batched engine's tail is always alone.)
  const bool cluster = P.coarse_n >= (sizeof(T) == 8 ? 100 : 200);
  if (cluster) smem += sizeof(T) * (size_t)P.coarse_n;
  auto run = [&](auto kernel) {
    if (smem > 48 * 1024) smem_optin((const void*)kernel);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster ? kTailCluster : 1);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = kTailCluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kernel, tp);
    note_launch();
  };
  if (P.g.dim == 2) {
    if (cluster) run(k_vcycle_tail<T, 2, true>);
    else run(k_vcycle_tail<T, 2, false>);
  } else {
    if (cluster) run(k_vcycle_tail<T, 3, true>);
    else run(k_vcycle_tail<T, 3, false>);
  }
}

template <typename T, int TX, int TY>
static void launch_fine2d(Problem& P, size_t l, int mode, const double* v, const double* vscale, double* z,
                          const T* u_in, T* u_out, const T* uc, cudaStream_t s) {
  Fine2DParams<T> fp;
  fp.L = levk<T>(P.lv[l]);
  fp.u_in = u_in;
  fp.u_out = u_out;
  fp.uc = uc;
  if (l + 1 < P.lv.size()) fp.C = levk<T>(P.lv[l + 1]);
  fp.neumann = P.desc.bc == IIM_BC_NEUMANN;
  fp.v = v;
  fp.vscale = vscale;
  fp.phase = P.phase;
  fp.inv_bp = (T)(1.0 / P.desc.beta_plus);
  fp.inv_bm = (T)(1.0 / P.desc.beta_minus);
  fp.z = z;
  const int n = P.lv[l].g.n;
  dim3 grid(ceil_div(n, TX), ceil_div(n, TY));
  switch (mode) {
    case 0: IIM_LAUNCH((k_mg2d<T, TX, TY, 0>), grid, 256, 0, s, fp); break;
    case 1: IIM_LAUNCH((k_mg2d<T, TX, TY, 1>), grid, 256, 0, s, fp); break;
    case 2: IIM_LAUNCH((k_mg2d<T, TX, TY, 2>), grid, 256, 0, s, fp); break;
    case 3: IIM_LAUNCH((k_mg2d<T, TX, TY, 3>), grid, 256, 0, s, fp); break;
    case 5: IIM_LAUNCH((k_mg2d<T, TX, TY, 5>), grid, 256, 0, s, fp); break;
    case 6: IIM_LAUNCH((k_mg2d<T, TX, TY, 6>), grid, 256, 0, s, fp); break;
    case 7: IIM_LAUNCH((k_mg2d<T, TX, TY, 7>), grid, 256, 0, s, fp); break;
    default: IIM_LAUNCH((k_mg2d<T, TX, TY, 4>), grid, 256, 0, s, fp); break;
  }
}

// The red-black tile kernels (mg_rb.cuh) for the first visit's down (MODE 5) and up
// (MODE 6) steps of levels with at least kRbMinN cells per axis: NW warps of RW rows each.
constexpr int kRbMinN = 64;

template <typename T, int NW, int RW>
static void launch_rb(Problem& P, size_t l, int mode, const double* v, const double* vscale, double* z,
                      const T* u_in, T* u_out, const T* uc, cudaStream_t s) {
  const Level& L = P.lv[l];
  const Level& C = P.lv[l + 1];
  const LevelK<T> K = levk<T>(L);
  Rb2DParams<T> rp;
  rp.n = L.g.n;
  rp.nc = C.g.n;
  rp.ih2 = K.ih2;
  rp.inv_dreg = K.inv_dreg;
  rp.dreg = K.dreg;
  rp.cls = L.cls;
  rp.aux = L.aux;
  rp.tab = K.tab;
  rp.f_in = (const T*)L.f;
  rp.f_bf16 = L.f_bf16;
  rp.f_out = (T*)L.f;
  rp.v = mode == 5 ? v : nullptr;
  rp.vscale = vscale;
  rp.inv_bp = (T)(1.0 / P.desc.beta_plus);
  rp.inv_bm = (T)(1.0 / P.desc.beta_minus);
  rp.u_in = u_in;
  rp.u_out = u_out;
  rp.z = mode == 6 ? z : nullptr;
  rp.uc = uc;
  rp.cls_c = C.cls;
  rp.fc = (T*)C.f;
  rp.fc_bf16 = C.f_bf16;
  rp.neumann = P.desc.bc == IIM_BC_NEUMANN;
  constexpr int SY = NW * RW, TY = SY - 2 * kRbHalo;
  const dim3 grid(ceil_div(L.g.n, kRbTX), ceil_div(L.g.n, TY));
  if (mode == 5) {
    constexpr size_t sm = rb_smem_bytes<T, NW, RW, false>();
    if (sm > 48 * 1024) smem_optin((const void*)k_mg2d_rb<T, NW, RW, false>);
    IIM_LAUNCH_PDL((k_mg2d_rb<T, NW, RW, false>), grid, NW * 32, sm, s, rp);
  } else {
    constexpr size_t sm = rb_smem_bytes<T, NW, RW, true>();
    if (sm > 48 * 1024) smem_optin((const void*)k_mg2d_rb<T, NW, RW, true>);
    IIM_LAUNCH_PDL((k_mg2d_rb<T, NW, RW, true>), grid, NW * 32, sm, s, rp);
  }
}

template <typename T>
static void fine2d(Problem& P, size_t l, int mode, const double* v, const double* vscale, double* z, const T* u_in,
                   T* u_out, const T* uc, cudaStream_t s) {
  const int n = P.lv[l].g.n;
  if ((mode == 5 || mode == 6) && n >= kRbMinN) {
    // window heights measured best on GB300 (V-cycles of the 1024^2 and 2048^2 star problems):
    // 64 rows (512 threads) from 2048, 32 rows (512 threads) from 512, 16 rows (256 threads) below
    if (n >= 2048) launch_rb<T, 16, 4>(P, l, mode, v, vscale, z, u_in, u_out, uc, s);
    else if (n >= 512) launch_rb<T, 16, 2>(P, l, mode, v, vscale, z, u_in, u_out, uc, s);
    else launch_rb<T, 8, 2>(P, l, mode, v, vscale, z, u_in, u_out, uc, s);
    return;
  }
  if (n >= 512) launch_fine2d<T, 64, 16>(P, l, mode, v, vscale, z, u_in, u_out, uc, s);
  else launch_fine2d<T, 32, 8>(P, l, mode, v, vscale, z, u_in, u_out, uc, s);
}

// 2D: fused kernels per fine level (MODE 0, [4...], 1 down; 2, [4...], 3 up), ping-ponging
// between the level's two u buffers.  u0 is the level's starting u (the previous visit's
// result in a W-cycle; nullptr: zero).  Returns the buffer that holds the level's result.
template <typename T>
static T* vcycle2d(Problem& P, size_t l, size_t lt, const double* v, const double* vscale, double* z,
                   cudaStream_t s, const T* u0 = nullptr) {
  T* A = (T*)P.lv[l].u;
  T* B = (T*)P.lv[l].u2;
  if (l == lt) {
    launch_tail<T>(P, l, l == 0 ? v : nullptr, l == 0 ? vscale : nullptr, l == 0 ? z : nullptr, s, A);
    return A;
  }
  // gamma visits of the next level (one launch of the tail runs all of its own)
  auto coarser = [&]() -> const T* {
    if (l + 1 == lt) return vcycle2d<T>(P, l + 1, lt, nullptr, nullptr, nullptr, s);
    const T* uc = nullptr;
    for (int g = 0; g < P.opt.cycle; ++g) uc = vcycle2d<T>(P, l + 1, lt, nullptr, nullptr, nullptr, s, uc);
    return uc;
  };
  if (P.opt.nu1 == 2 && P.opt.nu2 == 2) {
    // two fused kernels per level: both pre-smoothing sweeps + restriction, then the
    // correction + both post-smoothing sweeps.  The result is in B, so a later visit
    // reads B and writes A.
    if (u0) fine2d<T>(P, l, 7, nullptr, nullptr, nullptr, u0, A, nullptr, s);
    else fine2d<T>(P, l, 5, l == 0 ? v : nullptr, vscale, nullptr, nullptr, A, nullptr, s);
    const T* uc = coarser();
    fine2d<T>(P, l, 6, nullptr, nullptr, l == 0 ? z : nullptr, A, B, uc, s);
    return B;
  }
  if (u0) fine2d<T>(P, l, 4, nullptr, nullptr, nullptr, u0, A, nullptr, s);
  else fine2d<T>(P, l, 0, l == 0 ? v : nullptr, vscale, nullptr, nullptr, A, nullptr, s);
  for (int it = 1; it < P.opt.nu1 - 1; ++it) {
    fine2d<T>(P, l, 4, nullptr, nullptr, nullptr, A, B, nullptr, s);
    std::swap(A, B);
  }
  fine2d<T>(P, l, 1, nullptr, nullptr, nullptr, A, B, nullptr, s);
  std::swap(A, B);
  const T* uc = coarser();
  fine2d<T>(P, l, 2, nullptr, nullptr, nullptr, A, B, uc, s);
  std::swap(A, B);
  for (int it = 1; it < P.opt.nu2 - 1; ++it) {
    fine2d<T>(P, l, 4, nullptr, nullptr, nullptr, A, B, nullptr, s);
    std::swap(A, B);
  }
  fine2d<T>(P, l, 3, nullptr, nullptr, l == 0 ? z : nullptr, A, B, nullptr, s);
  return B;
}

template <typename T>
static Grid3D<T> grid3d(const Level& L) {
  const LevelK<T> K = levk<T>(L);
  Grid3D<T> G;
  G.n = L.g.n;
  G.ih2 = K.ih2;
  G.inv_dreg = K.inv_dreg;
  G.dreg = K.dreg;
  // rows of nodes at box faces, as k_sw_fill computes them (a face half a cell away: psi = 1/2)
  const double h2 = L.g.h * L.g.h;
  G.wall = (T)(2.0 / (1.0 * (0.5 + 1.0)) / h2);
  for (int k = 0; k < 4; ++k) {
    double d = 0;
    for (int ax = 0; ax < 3; ++ax) d += ax < k ? -2.0 / (0.5 * 1.0) / h2 : -2.0 / (1.0 * 1.0) / h2;
    G.wdiag[k] = (T)d;
    G.winv[k] = (T)(1.0 / d);
  }
  G.cls = L.cls;
  G.aux = L.aux;
  G.tab = K.tab;
  return G;
}

// One half sweep of a 3D level.  FP32 levels from 204^3, whose u and f take more than half of L2, go
// through 4 planes per thread, two pairs at a time; smaller ones, and FP64, a plane per thread.  V-cycle
// in us, runs / planes: FP32 exterior 320^3 1244 / 1564, 256^3 701 / 863, 208^3 456 / 505, 192^3 336 /
// 362 (but interior 249 / 240), 128^3 171 / 158, 96^3 128 / 101, where the loop only adds latency; FP64
// exterior 256^3 3192 / 2924, 208^3 1977 / 1758, 176^3 1268 / 1080.  Longer runs (FP32, 256^3): 8 planes
// 699 against 689, 16 planes 765, a pair and 16 planes 777.
constexpr int kSmooth3dRun = 4;
template <typename T>
static void smooth3d(const Grid3D<T>& G, T* u, const T* f, int f_bf16, int colour, double* z, cudaStream_t s) {
  const int n = G.n;
  if constexpr (sizeof(T) == 4) {
    if ((int64_t)n * n * n * 8 > (64 << 20) && n % 4 == 0) {
      const dim3 grid(ceil_div((int64_t)n * (n / 4), 256), ceil_div(n, kSmooth3dRun));
      if (z) IIM_LAUNCH_PDL(k_smooth3d_run<true>, grid, 256, 0, s, G, u, f, f_bf16, colour, kSmooth3dRun, z);
      else IIM_LAUNCH_PDL(k_smooth3d_run<false>, grid, 256, 0, s, G, u, f, f_bf16, colour, kSmooth3dRun, z);
      return;
    }
  }
  const dim3 grid(ceil_div((int64_t)n * (n / 2), 256), n);
  if (z) IIM_LAUNCH_PDL((k_smooth3d<T, true>), grid, 256, 0, s, G, u, f, f_bf16, colour, z);
  else IIM_LAUNCH_PDL((k_smooth3d<T, false>), grid, 256, 0, s, G, u, f, f_bf16, colour, z);
}

// 3D: u of every level is updated in place (stored by colour above the tail) and starts from zero unless this is a later visit of a
// W-cycle.  The level's right-hand side is v scale / beta on the finest level (v set), else L.f; the
// finest level's result leaves through z.
template <typename T>
static void vcycle3d(Problem& P, size_t l, size_t lt, const double* v, const double* vscale, double* z, cudaStream_t s,
                     bool from_zero = true) {
  Level& L = P.lv[l];
  T* u = (T*)L.u;
  T* f = (T*)L.f;
  if (l == lt) {
    launch_tail<T>(P, l, nullptr, nullptr, nullptr, s);
    return;
  }
  const int Tn = 256, n = L.g.n;
  const Grid3D<T> G = grid3d<T>(L);
  const dim3 grid(ceil_div(n * (n / 2), Tn), n);
  auto sweep = [&](int colour, bool out) {
    smooth3d<T>(G, u, (const T*)f, L.f_bf16, colour, out ? z : nullptr, s);
  };
  if (from_zero)
    IIM_LAUNCH_PDL(k_first3d<T>, grid, Tn, 0, s, G, v, vscale, (T)(1.0 / P.desc.beta_plus), (T)(1.0 / P.desc.beta_minus),
                   f, L.f_bf16, u);
  for (int it = 0; it < P.opt.nu1; ++it)
    for (int c = 0; c < 2; ++c)
      if (!(from_zero && it == 0 && c == 0)) sweep(c, false);
  Level& C = P.lv[l + 1];
  const int nc = C.g.n;
  const bool split = l + 1 < lt;         // the tail's levels keep the natural order
  auto transfers = [&](auto split_, auto rows_, bool down) {
    constexpr int SPLIT = decltype(split_)::value, ROWS = decltype(rows_)::value;
    const dim3 grid_c(ceil_div(4 / ROWS * nc * nc, Tn), nc);
    if (down)
      IIM_LAUNCH_PDL((k_restrict3d<T, SPLIT, ROWS>), grid_c, Tn, 0, s, G, (const T*)u, (const T*)f, L.f_bf16, nc,
                     (const uint8_t*)C.cls, (T*)C.f, C.f_bf16);
    else
      IIM_LAUNCH_PDL((k_prolong3d<T, SPLIT, ROWS>), grid_c, Tn, 0, s, n, (const uint8_t*)L.cls, u, nc, (const uint8_t*)C.cls,
                     (const T*)C.u, (int)(P.desc.bc == IIM_BC_NEUMANN));
  };
  auto transfer = [&](bool down) {
    using std::integral_constant;
    if (!split) transfers(integral_constant<int, 0>(), integral_constant<int, 1>(), down);
    else if (n < 128) transfers(integral_constant<int, 1>(), integral_constant<int, 1>(), down);
    else transfers(integral_constant<int, 1>(), integral_constant<int, 4>(), down);
  };
  transfer(true);
  if (l + 1 == lt) vcycle3d<T>(P, l + 1, lt, nullptr, nullptr, nullptr, s);
  else
    for (int g = 0; g < P.opt.cycle; ++g) vcycle3d<T>(P, l + 1, lt, nullptr, nullptr, nullptr, s, g == 0);
  transfer(false);
  for (int it = 0; it < P.opt.nu2; ++it)
    for (int c = 0; c < 2; ++c) sweep(c, z != nullptr && it == P.opt.nu2 - 1 && c == 1);
}

// generic path (2D with fewer than two sweeps): one kernel per half sweep, transfers separate; u is
// updated in place and starts from zero unless this is a later visit of a W-cycle
template <typename T>
static void vcycle(Problem& P, size_t l, size_t lt, cudaStream_t s, bool from_zero = true) {
  const int Tn = 256;
  Level& L = P.lv[l];
  T* u = (T*)L.u;
  T* f = (T*)L.f;
  if (l == lt) {
    launch_tail<T>(P, l, nullptr, nullptr, nullptr, s);
    return;
  }
  LevelView<T> V = view<T>(L);
  LevelK<T> K = levk<T>(L);
  const int64_t ncol = (L.g.N / L.g.n) * ((L.g.n + 1) / 2);
  if (from_zero) IIM_LAUNCH(k_zero<T>, ceil_div(L.g.N, Tn), Tn, 0, s, u, L.g.N);
  for (int it = 0; it < P.opt.nu1; ++it)
    for (int c = 0; c < 2; ++c)
      IIM_LAUNCH(k_smooth<T>, ceil_div(ncol, Tn), Tn, 0, s, V, K.ih2, K.inv_dreg, u, f, L.f_bf16, c);
  Level& C = P.lv[l + 1];
  IIM_LAUNCH(k_resid_restrict<T>, ceil_div(C.g.N, Tn), Tn, 0, s, V, K.ih2, K.dreg, u, f, L.f_bf16, C.g, C.aux,
             (T*)C.f, C.f_bf16);
  if (l + 1 == lt) vcycle<T>(P, l + 1, lt, s);
  else
    for (int g = 0; g < P.opt.cycle; ++g) vcycle<T>(P, l + 1, lt, s, g == 0);
  IIM_LAUNCH(k_prolong<T>, ceil_div(L.g.N, Tn), Tn, 0, s, L.g, L.aux, u, C.g, C.aux, (const T*)C.u,
             P.desc.bc == IIM_BC_NEUMANN);
  for (int it = 0; it < P.opt.nu2; ++it)
    for (int c = 0; c < 2; ++c)
      IIM_LAUNCH(k_smooth<T>, ceil_div(ncol, Tn), Tn, 0, s, V, K.ih2, K.inv_dreg, u, f, L.f_bf16, c);
}

template <typename T>
static void precondition_t(Problem& P, const double* v, const double* vscale, double* z, cudaStream_t s) {
  Level& L = P.lv[0];
  const int Tn = 256;
  const size_t lt = tail_start(P);
  if (lt == 0) {
    launch_tail<T>(P, 0, v, vscale, z, s);
    return;
  }
  if (P.g.dim == 2 && P.opt.nu1 >= 2 && P.opt.nu2 >= 2) {
    vcycle2d<T>(P, 0, lt, v, vscale, z, s);
    return;
  }
  if (P.g.dim == 3 && P.opt.nu1 >= 1 && P.opt.nu2 >= 1) {
    vcycle3d<T>(P, 0, lt, v, vscale, z, s);
    return;
  }
  IIM_LAUNCH(k_bridge_in<T>, ceil_div(L.g.N, Tn), Tn, 0, s, L.g, v, vscale, P.phase, L.aux,
             1.0 / P.desc.beta_plus, 1.0 / P.desc.beta_minus, (T*)L.f);
  vcycle<T>(P, 0, lt, s);
  IIM_LAUNCH(k_bridge_out<T>, ceil_div(L.g.N, Tn), Tn, 0, s, L.g, (const T*)L.u, z);
}

template <typename T>
static void smooth_fine_t(Problem& P, int colour, cudaStream_t s) {
  Level& L = P.lv[0];
  if (P.g.dim == 3 && tail_start(P) > 0) {
    smooth3d<T>(grid3d<T>(L), (T*)L.u, (const T*)L.f, L.f_bf16, colour, nullptr, s);
    return;
  }
  LevelView<T> V = view<T>(L);
  LevelK<T> K = levk<T>(L);
  const int64_t ncol = (L.g.N / L.g.n) * ((L.g.n + 1) / 2);
  IIM_LAUNCH(k_smooth<T>, ceil_div(ncol, 256), 256, 0, s, V, K.ih2, K.inv_dreg, (T*)L.u, (const T*)L.f, L.f_bf16, colour);
}

// one red or black half sweep on the finest level (kernel timing)
void mg_smooth_fine(Problem& P, int colour, cudaStream_t s) {
  if (P.opt.mg_precision == IIM_MG_FP64) smooth_fine_t<double>(P, colour, s);
  else smooth_fine_t<float>(P, colour, s);
}

void mg_precondition(Problem& P, const double* v, const double* vscale, double* z, cudaStream_t s) {
  if (P.opt.mg_precision == IIM_MG_FP64) precondition_t<double>(P, v, vscale, z, s);
  else precondition_t<float>(P, v, vscale, z, s);
}

// The first level runs the fused down / up kernels (2D, V(2,2), above the tail)
bool mg_has_fused_first(const Problem& P) {
  return P.g.dim == 2 && tail_start(P) > 0 && P.opt.nu1 == 2 && P.opt.nu2 == 2;
}

// One kernel of the V-cycle alone (profiling): which 0 = the first level's down kernel,
// 1 = its up kernel (both need mg_has_fused_first), 2 = the coarse tail.
template <typename T>
static bool mg_one_kernel_t(Problem& P, int which, const double* v, double* z, cudaStream_t s) {
  const size_t lt = tail_start(P);
  if (which == 2) {
    launch_tail<T>(P, lt, lt == 0 ? v : nullptr, nullptr, lt == 0 ? z : nullptr, s);
    return true;
  }
  if (!mg_has_fused_first(P)) return false;
  T* A = (T*)P.lv[0].u;
  T* B = (T*)P.lv[0].u2;
  if (which == 0) fine2d<T>(P, 0, 5, v, nullptr, nullptr, nullptr, A, nullptr, s);
  else fine2d<T>(P, 0, 6, nullptr, nullptr, z, A, B, (const T*)P.lv[1].u, s);
  return true;
}

bool mg_one_kernel(Problem& P, int which, const double* v, double* z, cudaStream_t s) {
  if (P.opt.mg_precision == IIM_MG_FP64) return mg_one_kernel_t<double>(P, which, v, z, s);
  return mg_one_kernel_t<float>(P, which, v, z, s);
}

// columns per block step: the panel's columns must fit in shared memory
template <typename T>
static int gj_block(int cn) {
  int b = kGJ;
  while (b > 1 && (sizeof(T) * b + sizeof(int)) * (size_t)cn > 220 * 1024) b /= 2;
  return b;
}

// dense matrix and inverse of the coarsest level: buf holds two cn x cn buffers and one pivot block
template <typename T>
static void coarse_invert(Problem& P, const LevelView<double>& L, const int* nu, const int32_t* node_row, T* buf,
                          cudaStream_t s) {
  const int cn = P.coarse_n, b = gj_block<T>(cn);
  T* D = buf + 2 * (size_t)cn * cn;
  int* order = P.coarse_piv;
  int* from = P.coarse_piv + cn;
  cudaMemsetAsync(buf, 0, sizeof(T) * 2 * (size_t)cn * cn, s);
  IIM_LAUNCH(k_coarse_assemble<T>, ceil_div(cn, 64), 64, 0, s, L, P.coarse_map, nu, cn, node_row, buf, P.aug, b,
             P.d_status);
  smem_optin((const void*)k_gj_panel<T>);
  const dim3 tiles(ceil_div(cn, 32), ceil_div(cn, 32));
  for (int k = 0; k * b < cn; ++k) {
    const size_t sm = (sizeof(T) * b + sizeof(int)) * (size_t)(cn - k * b);
    IIM_LAUNCH(k_gj_panel<T>, 1, 1024, sm, s, buf, cn, nu, P.aug, k, b, order, from, D, P.d_status);
    IIM_LAUNCH(k_gj_update<T>, tiles, 256, 0, s, buf, cn, nu, P.aug, k, b, from, D);
  }
  IIM_LAUNCH(k_gj_finish<T>, dim3(ceil_div(cn, 256), std::min(cn, 256)), 256, 0, s, buf, cn, nu, P.aug, b, order);
}

// coarse matrix and inverse; coarse_lu{64,32} hold [scratch (cn*cn) | inverse (cn*cn) | pivot block], cn the
// fixed size of the padded system (a re-run set-up with another geometry changes only the
// device-side unknown count)
void mg_coarse_factor(Problem& P, cudaStream_t s) {
  Level& C = P.lv.back();
  const int cn = P.coarse_n;
  if (cn <= 0) return;
  const int Tn = 256;
  IIM_LAUNCH(k_unknown_flag, ceil_div(C.g.N, Tn), Tn, 0, s, C.g, C.aux, C.flag);
  scan_exclusive(C.flag, C.idx, C.g.N, P.d_counts + kCountCoarse, P.scan_scratch, s);
  int32_t* inv = C.flag;            // reuse: node -> unknown index
  cudaMemsetAsync(P.coarse_map, 0xff, sizeof(int32_t) * (size_t)cn, s);    // -1: a slot no unknown uses
  IIM_LAUNCH(k_coarse_map, ceil_div(C.g.N, Tn), Tn, 0, s, C.g, C.aux, C.idx, P.coarse_map, inv);
  LevelView<double> V = view<double>(C);
  const int* nu = P.d_counts + kCountCoarse;
  if (P.opt.mg_precision == IIM_MG_FP64) coarse_invert(P, V, nu, inv, P.coarse_lu64, s);
  else coarse_invert(P, V, nu, inv, P.coarse_lu32, s);
}


// ---------------------------------------------------------------------------- batched engine
// Grouped forms of the V-cycle kernels: each item is one block of the single-problem
// launch (a tile of the 2D fused kernels, 256 nodes of the 3D kernels, the whole
// tail), so a slot's V-cycle is the one its own solve would run.

__device__ __forceinline__ const double* eng_vj(const SlotDev& s) { return s.V + (size_t)s.j * s.Npad; }
__device__ __forceinline__ double* eng_zj(const SlotDev& s) { return s.Z + (size_t)s.j * s.Npad; }

template <int TX, int TY, int MODE>
__global__ void __launch_bounds__(256, 4) k_eng_mg2d(EngArgs A, int list, int d, int in_sel, int out_sel, int res_sel) {
  eng_for_items(A, list, [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role != kRoleIter) return;
    Fine2DParams<float> fp;
    fp.L = s.lev[d];
    fp.C = s.lev[d + 1 < s.nlev ? d + 1 : d];
    float* b0 = s.lev[d].u;
    float* b1 = s.u2[d];
    constexpr bool DOWN_FIRST = MODE == 0 || MODE == 5, UP_FIRST = MODE == 2 || MODE == 6;
    constexpr bool UP_LAST = MODE == 3 || MODE == 6;
    fp.u_in = DOWN_FIRST ? nullptr : (in_sel ? b1 : b0);
    fp.u_out = out_sel ? b1 : b0;
    fp.uc = nullptr;
    if (UP_FIRST) fp.uc = (d + 1 < s.nfine && res_sel) ? s.u2[d + 1] : s.lev[d + 1].u;
    fp.neumann = s.neumann;
    fp.v = (DOWN_FIRST && d == 0) ? eng_vj(s) : nullptr;
    fp.vscale = &s.sc->inv_norm[s.j];
    fp.phase = s.phase;
    fp.inv_bp = s.inv_bp;
    fp.inv_bm = s.inv_bm;
    fp.z = (UP_LAST && d == 0) ? eng_zj(s) : nullptr;
    const int gx = (s.lev[d].n + TX - 1) / TX;
    mg2d_tile<float, TX, TY, MODE>(fp, item % gx, item / gx);
  });
}

__global__ void __launch_bounds__(kTailThreads) k_eng_tail(EngArgs A) {
  eng_for_items(A, kListTail, [&](int si, int) {
    const SlotDev& s = A.slots[si];
    if (s.role != kRoleIter) return;
    const bool top = s.nfine == 0;
    if (s.dim == 2)
      vcycle_tail_body<float, 2>(s.tail, top ? eng_vj(s) : nullptr, top ? &s.sc->inv_norm[s.j] : nullptr,
                            top ? eng_zj(s) : nullptr);
    else
      vcycle_tail_body<float, 3>(s.tail, top ? eng_vj(s) : nullptr, top ? &s.sc->inv_norm[s.j] : nullptr,
                            top ? eng_zj(s) : nullptr);
  });
}

__device__ __forceinline__ LevelView<float> eng_view(const SlotDev& s, int d) {
  LevelView<float> v;
  v.g.dim = s.lev[d].dim;
  v.g.n = s.lev[d].n;
  v.g.N = s.lev[d].N;
  v.g.h = 2.0 / s.lev[d].n;
  v.aux = s.lev[d].aux;
  v.tab = s.lev[d].tab;
  return v;
}

// 3D kernels, kind: 0 bridge in, 1 zero, 2 smooth, 3 residual + restriction, 4 prolongation, 5 bridge out
template <int KIND>
__global__ void __launch_bounds__(256) k_eng_mg3d(EngArgs A, int list, int d, int colour) {
  eng_for_items(A, list, [&](int si, int item) {
    const SlotDev& s = A.slots[si];
    if (s.role != kRoleIter) return;
    const int64_t i = (int64_t)item * 256 + threadIdx.x;
    const LevelK<float>& K = s.lev[d];
    const LevelView<float> V = eng_view(s, d);
    if (KIND == 0) {
      bridge_in_body<float>(V.g, eng_vj(s), &s.sc->inv_norm[s.j], s.phase, K.aux, 1.0 / s.GP.beta_p,
                            1.0 / s.GP.beta_m, K.f, i);
    } else if (KIND == 1) {
      if (i < K.N) K.u[i] = 0.f;
    } else if (KIND == 2) {
      smooth_body<float>(V, K.ih2, K.inv_dreg, K.u, K.f, K.f_bf16, colour, i);
    } else if (KIND == 3) {
      const LevelView<float> C = eng_view(s, d + 1);
      resid_restrict_body<float>(V, K.ih2, K.dreg, K.u, K.f, K.f_bf16, C.g, C.aux, s.lev[d + 1].f, i,
                                 s.lev[d + 1].f_bf16);
    } else if (KIND == 4) {
      const LevelView<float> C = eng_view(s, d + 1);
      prolong_body<float>(V.g, K.aux, K.u, C.g, C.aux, s.lev[d + 1].u, s.neumann, i);
    } else {
      if (i < K.N) eng_zj(s)[i] = (double)K.u[i];
    }
  });
}

void eng_mg2d_tile_items(int n, int shape, int* gx, int* gy) {
  *gx = ceil_div(n, kShapeTX[shape]);
  *gy = ceil_div(n, kShapeTY[shape]);
}

template <int TX, int TY>
static void launch_eng_mg2d(const EngArgs& A, const EngMgStep& st, cudaStream_t s) {
  const int list = kListMg2d + st.depth * kEngShapes + st.shape;
#define IIM_ENG_MG2D(MODE)                                                                                     \
  IIM_LAUNCH((k_eng_mg2d<TX, TY, MODE>), eng_grid((const void*)k_eng_mg2d<TX, TY, MODE>, 256, 0), 256, 0, s, A, \
             list, st.depth, st.in_sel, st.out_sel, st.res_sel)
  switch (st.mode) {
    case 0: IIM_ENG_MG2D(0); break;
    case 1: IIM_ENG_MG2D(1); break;
    case 2: IIM_ENG_MG2D(2); break;
    case 3: IIM_ENG_MG2D(3); break;
    case 5: IIM_ENG_MG2D(5); break;
    case 6: IIM_ENG_MG2D(6); break;
    default: IIM_ENG_MG2D(4); break;
  }
#undef IIM_ENG_MG2D
}

void eng_launch_mg(const EngArgs& A, const EngMgStep& st, size_t tail_smem, cudaStream_t s) {
  if (st.kind == 0) {
    switch (st.shape) {
      case 0: launch_eng_mg2d<32, 8>(A, st, s); break;
      case 1: launch_eng_mg2d<64, 8>(A, st, s); break;
      case 2: launch_eng_mg2d<32, 16>(A, st, s); break;
      default: launch_eng_mg2d<64, 16>(A, st, s); break;
    }
    return;
  }
  if (st.kind == 1) {
    smem_optin((const void*)k_eng_tail);
    IIM_LAUNCH(k_eng_tail, eng_grid((const void*)k_eng_tail, kTailThreads, tail_smem), kTailThreads, tail_smem, s, A);
    return;
  }
  const int k3 = st.kind - 2;
  const int d = st.depth;
#define IIM_ENG_MG3D(KIND, LIST)                                                                             \
  IIM_LAUNCH(k_eng_mg3d<KIND>, eng_grid((const void*)k_eng_mg3d<KIND>, 256, 0), 256, 0, s, A, LIST, d, st.colour)
  switch (k3) {
    case 0: IIM_ENG_MG3D(0, kList3dN + 0); break;
    case 1: IIM_ENG_MG3D(1, kList3dN + d); break;
    case 2: IIM_ENG_MG3D(2, kList3dCol + d); break;
    case 3: IIM_ENG_MG3D(3, kList3dCoarse + d); break;
    case 4: IIM_ENG_MG3D(4, kList3dN + d); break;
    default: IIM_ENG_MG3D(5, kList3dN + 0); break;
  }
#undef IIM_ENG_MG3D
}

}  // namespace iim
