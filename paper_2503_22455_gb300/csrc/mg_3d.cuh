// Kernels of the 3D levels above the coarse tail (paper Sec. 3.3), included by multigrid.cu: one
// kernel per half sweep and transfer, in the arithmetic of multigrid.cu's node functions (the
// batched engine runs those; both give the same bits).
//
// What bounds them: bytes on the levels that exceed L2, launches on the others, hence programmatic
// dependent launches.  To stay near that,
//   - u and f of these levels are stored by colour: all red cells, then all black ones, the cell of
//     pair k (x = 2 k, 2 k + 1) of row (y, z) at place (z n + y) n / 2 + k of its colour.  A half sweep
//     then reads the other colour's u, its own f and class and writes its own u, all in whole
//     sectors: 7 bytes per node of the level instead of 13.  The y and z neighbours of a cell have
//     its place k in their rows, the x neighbours k and k - 1 or k + 1;
//   - a thread finds its cell by 32-bit arithmetic and takes a path without any table for regular
//     cells and for cells at a box face alone, whose weights follow from the position;
//   - the first half sweep from u = 0 is a product and comes with the entry of f, the last one with
//     the exit of z;
//   - on the levels that exceed L2 a half sweep in FP32 goes through several planes per thread, two
//     pairs at a time, so that a plane crosses L2 once per run instead of three times.
// Not kept: all four half sweeps in one kernel that streams planes through registers (1.5 ms per
// cycle at 256^3: 500 dependent instructions per warp and plane), and the natural order of u and f
// (0.80 ms).
//
// Measured (V-cycle, FP32, against one kernel per half sweep in natural order with 64-bit index
// divisions and 4-byte row codes): 256^3 exterior ellipsoid 2.28 -> 0.69 ms, 96^3 perturbed sphere
// 0.27 -> 0.10 ms; 128^3 in FP64 0.52 ms.
#pragma once

namespace iim {

// constants of one level
template <typename T>
struct Grid3D {
  int n;
  T ih2, inv_dreg, dreg;
  T wall;                    // weight of the neighbour opposite a box face
  T wdiag[4], winv[4];       // diagonal and its reciprocal by the number of axes with a face
  const uint8_t* cls;
  const int32_t* aux;
  const T* tab;              // irregular rows, 8 entries: diag, -x, +x, -y, +y, -z, +z, 1 / diag
};

// weights, diagonal and its reciprocal of an irregular cell (class w): by position, or the table row
template <typename T>
__device__ __forceinline__ void irregular_row(const Grid3D<T>& G, int i, int x, int y, int z, uint8_t w, T (&c)[8]) {
  if (w & kClsBox) {
    const int m[3] = {x, y, z};
    int faces = 0;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const bool lo = m[ax] == 0, hi = m[ax] == G.n - 1;
      c[1 + 2 * ax] = lo ? (T)0 : (hi ? G.wall : G.ih2);
      c[2 + 2 * ax] = hi ? (T)0 : (lo ? G.wall : G.ih2);
      faces += lo || hi ? 1 : 0;
    }
    c[0] = faces == 1 ? G.wdiag[1] : (faces == 2 ? G.wdiag[2] : G.wdiag[3]);
    c[7] = faces == 1 ? G.winv[1] : (faces == 2 ? G.winv[2] : G.winv[3]);
  } else {
    const T* t = G.tab + (size_t)__ldg(G.aux + i) * 8;
#pragma unroll
    for (int k = 0; k < 8; ++k) c[k] = __ldg(t + k);
  }
}

// f - (off-diagonal part) of cell (x, y, z) of class w from its neighbours' values (-x, +x, ...; any
// finite value beyond the grid), and the row's diagonal and reciprocal
template <typename T>
__device__ __forceinline__ T row_minus(const Grid3D<T>& G, int x, int y, int z, uint8_t w, T f, const T (&v)[6], T& diag,
                                       T& inv) {
  if (!(w & kClsIrregular)) {
    diag = G.dreg;
    inv = G.inv_dreg;
    return off_residual3(f, G.ih2, G.ih2, G.ih2, G.ih2, G.ih2, G.ih2, v[0], v[1], v[2], v[3], v[4], v[5]);
  }
  T c[8];
  irregular_row(G, (z * G.n + y) * G.n + x, x, y, z, w, c);
  diag = c[0];
  inv = c[7];
  return off_residual3(f, c[1], c[2], c[3], c[4], c[5], c[6], v[0], v[1], v[2], v[3], v[4], v[5]);
}

// pair t of plane z = blockIdx.y: row y, cells 2 k and 2 k + 1, place p in either colour
struct Pair3D {
  int y, z, k, p;
  __device__ Pair3D(int n) {
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x, h = n / 2;
    z = blockIdx.y;
    y = (int)(t / h);
    k = (int)(t - (unsigned)y * h);
    p = z * n * (int)h + (int)t;
  }
};

// entry and first red half sweep from u = 0: f = v scale / beta (finest level) or as stored
template <typename T>
__global__ void __launch_bounds__(256) k_first3d(Grid3D<T> G, const double* __restrict__ v,
                                                 const double* __restrict__ vscale, T inv_bp, T inv_bm,
                                                 T* __restrict__ f, int f_bf16, T* __restrict__ u) {
  const Pair3D q(G.n);
  const bool in = q.y < G.n;
  const int e = (q.y + q.z) & 1, half = G.n * G.n * (G.n / 2);   // e: the red cell of the pair
  const uchar2 w = in ? __ldg((const uchar2*)(G.cls + 2 * q.p)) : make_uchar2(0, 0);
  pdl_trigger();
  pdl_wait();
  if (!in) return;
  T fr;
  if (v) {
    const double2 vv = *(const double2*)(v + 2 * q.p);
    const T vs = (T)(vscale ? *vscale : 1.0);
    const T f0 = w.x & kClsUnknown ? mul_rn((T)vv.x, mul_rn(vs, w.x & kClsPlus ? inv_bp : inv_bm)) : (T)0;
    const T f1 = w.y & kClsUnknown ? mul_rn((T)vv.y, mul_rn(vs, w.y & kClsPlus ? inv_bp : inv_bm)) : (T)0;
    fr = e ? f1 : f0;
    f[q.p] = fr;
    f[half + q.p] = e ? f0 : f1;
  } else {
    fr = load_f(f, q.p, f_bf16);
  }
  const uint8_t c = e ? w.y : w.x;
  T r = 0;
  if (c & kClsUnknown) {
    T inv = G.inv_dreg;
    if (c & kClsIrregular) {
      T row[8];
      irregular_row(G, 2 * q.p + e, 2 * q.k + e, q.y, q.z, c, row);
      inv = row[7];
    }
    r = mul_rn(fr, inv);
  }
  u[q.p] = r;
}

// One half sweep in place (cells that are no unknowns get 0), a thread per pair; OUT: the level's result
// leaves as FP64 (finest level, last half sweep).
template <typename T, bool OUT>
__global__ void __launch_bounds__(256) k_smooth3d(Grid3D<T> G, T* __restrict__ u, const T* __restrict__ f, int f_bf16,
                                                  int colour, double* __restrict__ zout) {
  const Pair3D q(G.n);
  const int n = G.n, h = n / 2, hn = h * n, half = n * hn, p = q.p;
  const T* o = u + (colour ? 0 : half);
  T* own = u + (colour ? half : 0);
  const int e = (q.y + q.z + colour) & 1;
  const bool in = q.y < n;
  const uint8_t w = in ? __ldg(G.cls + 2 * p + e) : 0;
  pdl_trigger();
  pdl_wait();
  if (!in) return;
  T val = 0;
  const T oc = o[p];
  if (w & kClsUnknown) {
    const T side = e ? (q.k < h - 1 ? o[p + 1] : (T)0) : (q.k > 0 ? o[p - 1] : (T)0);
    const T v[6] = {e ? oc : side, e ? side : oc, q.y > 0 ? o[p - h] : (T)0, q.y < n - 1 ? o[p + h] : (T)0,
                    q.z > 0 ? o[p - hn] : (T)0, q.z < n - 1 ? o[p + hn] : (T)0};
    T diag, inv;
    const T r = row_minus(G, 2 * q.k + e, q.y, q.z, w, load_f(f, (colour ? half : 0) + p, f_bf16), v, diag, inv);
    val = mul_rn(r, inv);
  }
  if (OUT) {
    double2 st;
    st.x = (double)(e ? oc : val);
    st.y = (double)(e ? val : oc);
    *(double2*)(zout + 2 * p) = st;
  } else {
    own[p] = val;
  }
}

// The same in FP32 for levels that exceed L2 (n a multiple of 4): a thread takes two neighbouring pairs through
// `run` planes.  The other colour's values at its places in the next plane become the x neighbours there
// and the z neighbours one plane on, so a plane of u crosses L2 once per run instead of three times; the
// pairs share a vector load per neighbour row, the x neighbour between them and the index arithmetic,
// which bounded the single pairs (99 instructions per cell, 67 % of the issue slots): 41.4 -> 30.1 us per
// half sweep at 256^3 (17 us for its bytes), V-cycle 777 -> 689 us.
template <bool OUT>
__global__ void __launch_bounds__(256) k_smooth3d_run(Grid3D<float> G, float* __restrict__ u, const float* __restrict__ f,
                                                      int f_bf16, int colour, int run, double* __restrict__ zout) {
  const int n = G.n, h = n / 2, hn = h * n, half = n * hn;
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = (int)(t / (unsigned)(h / 2)), k = 2 * (int)(t - (unsigned)y * (unsigned)(h / 2));
  const int z0 = blockIdx.y * run, z1 = min(n, z0 + run);
  const float* o = u + (colour ? 0 : half);
  float* own = u + (colour ? half : 0);
  const int fofs = colour ? half : 0;
  const bool in = y < n;
  int p = z0 * hn + y * h + k;
  // classes of the four cells of both pairs
  unsigned w = in ? __ldg((const unsigned*)(G.cls + 2 * p)) : 0;
  pdl_trigger();
  pdl_wait();
  if (!in) return;
  auto two = [](const float* p) { return *reinterpret_cast<const float2*>(p); };
  const float2 zero = make_float2(0.f, 0.f);
  float2 om = z0 > 0 ? two(o + p - hn) : zero, oc = two(o + p);
  for (int z = z0; z < z1; ++z, p += hn) {
    const int e = (y + z + colour) & 1;
    const float2 op = z < n - 1 ? two(o + p + hn) : zero;
    const unsigned wn = z + 1 < z1 ? __ldg((const unsigned*)(G.cls + 2 * (p + hn))) : 0;
    const unsigned wa = (w >> (8 * e)) & 255, wb = (w >> (16 + 8 * e)) & 255;
    float va = 0, vb = 0;
    if ((wa | wb) & kClsUnknown) {
      const float side = e ? (k + 2 < h ? o[p + 2] : 0.f) : (k > 0 ? o[p - 1] : 0.f);
      const float2 ym = y > 0 ? two(o + p - h) : zero, yp = y < n - 1 ? two(o + p + h) : zero;
      const float2 ff = load_f2(f, fofs + p, f_bf16);
      const float a[6] = {e ? oc.x : side, e ? oc.y : oc.x, ym.x, yp.x, om.x, op.x};
      const float b[6] = {e ? oc.y : oc.x, e ? side : oc.y, ym.y, yp.y, om.y, op.y};
      if ((wa & wb & kClsUnknown) && !((wa | wb) & kClsIrregular)) {
        va = mul_rn(off_residual3(ff.x, G.ih2, G.ih2, G.ih2, G.ih2, G.ih2, G.ih2, a[0], a[1], a[2], a[3], a[4], a[5]), G.inv_dreg);
        vb = mul_rn(off_residual3(ff.y, G.ih2, G.ih2, G.ih2, G.ih2, G.ih2, G.ih2, b[0], b[1], b[2], b[3], b[4], b[5]), G.inv_dreg);
      } else {
        float diag, inv;
        if (wa & kClsUnknown) {
          const float r = row_minus(G, 2 * k + e, y, z, (uint8_t)wa, ff.x, a, diag, inv);
          va = mul_rn(r, inv);
        }
        if (wb & kClsUnknown) {
          const float r = row_minus(G, 2 * k + 2 + e, y, z, (uint8_t)wb, ff.y, b, diag, inv);
          vb = mul_rn(r, inv);
        }
      }
    }
    if (OUT) {
      *(double2*)(zout + 2 * p) = make_double2((double)(e ? oc.x : va), (double)(e ? va : oc.x));
      *(double2*)(zout + 2 * p + 2) = make_double2((double)(e ? oc.y : vb), (double)(e ? vb : oc.y));
    } else {
      *reinterpret_cast<float2*>(own + p) = make_float2(va, vb);
    }
    om = oc;
    oc = op;
    w = wn;
  }
}

// place of coarse cell (X, Y, Z): by colour, or natural (SPLIT = 0, the tail's first level)
template <int SPLIT>
__device__ __forceinline__ int coarse_place(int X, int Y, int Z, int nc) {
  const int r = Z * nc + Y;
  if (!SPLIT) return r * nc + X;
  return ((X + Y + Z) & 1 ? nc * nc * (nc / 2) : 0) + r * (nc / 2) + (X >> 1);
}

// Residual and restriction.  ROWS rows of children per thread: 1 (four lanes per coarse cell, lane q
// the row y + (q & 1), z + (q >> 1); small levels, where a row next to the boundary costs two
// dependent loads per child) or 4 (a thread per coarse cell, which reads every value its children
// share once; the levels from n = 128).
template <typename T, int SPLIT, int ROWS>
__global__ void __launch_bounds__(256) k_restrict3d(Grid3D<T> G, const T* __restrict__ u, const T* __restrict__ f,
                                                    int f_in_bf16, int nc, const uint8_t* __restrict__ cls_c,
                                                    T* __restrict__ fc, int f_bf16) {
  const unsigned tt = blockIdx.x * blockDim.x + threadIdx.x, t = ROWS == 1 ? tt >> 2 : tt;
  const int Z = blockIdx.y, Y = (int)(t / (unsigned)nc), X = (int)(t - (unsigned)Y * (unsigned)nc);
  const bool in = Y < nc;
  const int n = G.n, h = n / 2, hn = h * n, half = n * hn, q0 = ROWS == 1 ? (int)(threadIdx.x & 3) : 0;
  const int p00 = (2 * Z * n + 2 * Y) * h + X;         // the first row's place
  const uint8_t wc = in ? __ldg(cls_c + (Z * nc + Y) * nc + X) : 0;
  uchar2 w[ROWS];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int q = q0 + r;
    w[r] = in ? __ldg((const uchar2*)(G.cls + 2 * (p00 + (q & 1) * h + (q >> 1) * hn))) : make_uchar2(0, 0);
  }
  pdl_trigger();
  pdl_wait();
  T sum[ROWS];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) sum[r] = (T)0;
  if (wc & kClsUnknown) {
    // value of cell (e, row q) with its colour's half: c = (e + y + z) & 1, y and z of row 0 being even
    T c[ROWS][2], ff[ROWS][2];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int q = q0 + r, p = p00 + (q & 1) * h + (q >> 1) * hn;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int own = p + (((e + (q & 1) + (q >> 1)) & 1) ? half : 0);
        c[r][e] = u[own];
        ff[r][e] = load_f(f, own, f_in_bf16);
      }
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int q = q0 + r, y = 2 * Y + (q & 1), z = 2 * Z + (q >> 1), p = p00 + (q & 1) * h + (q >> 1) * hn;
      T res[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint8_t we = e ? w[r].y : w[r].x;
        const T* o = u + (((e + (q & 1) + (q >> 1)) & 1) ? 0 : half);   // the other colour
        res[e] = (T)0;
        if (!(we & kClsUnknown)) continue;
        const T side = e ? (X < h - 1 ? o[p + 1] : (T)0) : (X > 0 ? o[p - 1] : (T)0);
        T v[6] = {e ? c[r][0] : side, e ? side : c[r][1], (T)0, (T)0, (T)0, (T)0};
        if constexpr (ROWS == 4) {       // the children's own neighbours are in registers
          const T yn = (r & 1) ? (y < n - 1 ? o[p + h] : (T)0) : (y > 0 ? o[p - h] : (T)0);
          const T zn = (r >> 1) ? (z < n - 1 ? o[p + hn] : (T)0) : (z > 0 ? o[p - hn] : (T)0);
          v[2] = (r & 1) ? c[r ^ 1][e] : yn;
          v[3] = (r & 1) ? yn : c[r ^ 1][e];
          v[4] = (r >> 1) ? c[r ^ 2][e] : zn;
          v[5] = (r >> 1) ? zn : c[r ^ 2][e];
        } else {
          v[2] = y > 0 ? o[p - h] : (T)0;
          v[3] = y < n - 1 ? o[p + h] : (T)0;
          v[4] = z > 0 ? o[p - hn] : (T)0;
          v[5] = z < n - 1 ? o[p + hn] : (T)0;
        }
        T diag, inv;
        const T off = row_minus(G, 2 * X + e, y, z, we, ff[r][e], v, diag, inv);
        res[e] = fma(-diag, c[r][e], off);
      }
      sum[r] = res[0] + res[1];
    }
  }
  // the two rows of a plane, then the planes
  T s;
  if constexpr (ROWS == 4) {
    s = (sum[0] + sum[1]) + (sum[2] + sum[3]);
  } else {
    s = sum[0];
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
  }
  if (in && q0 == 0) store_f(fc, coarse_place<SPLIT>(X, Y, Z, nc), s * (T)0.125, f_bf16);
}

// u += P e, ROWS rows of children per thread as in k_restrict3d
template <typename T, int SPLIT, int ROWS>
__global__ void __launch_bounds__(256) k_prolong3d(int n, const uint8_t* __restrict__ cls, T* __restrict__ u, int nc,
                                                   const uint8_t* __restrict__ cls_c, const T* __restrict__ ec,
                                                   int neumann) {
  const unsigned tt = blockIdx.x * blockDim.x + threadIdx.x, t = ROWS == 1 ? tt >> 2 : tt;
  const int Z = blockIdx.y, Y = (int)(t / (unsigned)nc), X = (int)(t - (unsigned)Y * (unsigned)nc);
  const bool in = Y < nc;
  const int h = n / 2, hn = h * n, half = n * hn, q0 = ROWS == 1 ? (int)(threadIdx.x & 3) : 0;
  const int p00 = (2 * Z * n + 2 * Y) * h + X;
  // parents: x offset k % 3 - 1; rows and planes: all three (ROWS = 4), or the own one and the one on
  // this row's side
  constexpr int NY = ROWS == 4 ? 3 : 2, NP = 3 * NY * NY;
  const int sy = (q0 & 1) ? 1 : -1, sz = (q0 >> 1) ? 1 : -1;
  uchar2 w[ROWS];
  unsigned any = 0, ok = 0;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int q = q0 + r;
    w[r] = in ? __ldg((const uchar2*)(cls + 2 * (p00 + (q & 1) * h + (q >> 1) * hn))) : make_uchar2(0, 0);
    any |= (unsigned)(w[r].x | w[r].y) & kClsUnknown;
  }
  auto parent = [&](int k, int& x, int& y, int& z) {
    const int ry = k / 3 % NY, rz = k / 3 / NY;
    x = X + k % 3 - 1;
    y = Y + (ROWS == 4 ? ry - 1 : (ry ? sy : 0));
    z = Z + (ROWS == 4 ? rz - 1 : (rz ? sz : 0));
    return x >= 0 && x < nc && y >= 0 && y < nc && z >= 0 && z < nc;
  };
  if (neumann && any) {
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      int x, y, z;
      if (parent(k, x, y, z)) ok |= (unsigned)(__ldg(cls_c + (z * nc + y) * nc + x) & kClsUnknown) << k;
    }
  }
  pdl_trigger();
  pdl_wait();
  if (!any) return;
  T e[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    int x, y, z;
    e[k] = parent(k, x, y, z) ? ec[coarse_place<SPLIT>(x, y, z, nc)] : (T)0;   // zero at cells that are no unknowns
  }
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int q = q0 + r, p = p00 + (q & 1) * h + (q >> 1) * hn;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (!((s ? w[r].y : w[r].x) & kClsUnknown)) continue;
      T ev[8];
      unsigned o = 0;
#pragma unroll
      for (int sel = 0; sel < 8; ++sel) {
        const int dx = (sel & 1) ? (s ? 1 : -1) : 0;
        int ry = (sel >> 1) & 1, rz = sel >> 2;
        if (ROWS == 4) {
          ry = 1 + (ry ? ((r & 1) ? 1 : -1) : 0);
          rz = 1 + (rz ? ((r >> 1) ? 1 : -1) : 0);
        }
        const int k = (1 + dx) + 3 * (ry + NY * rz);
        ev[sel] = e[k];
        o |= ((ok >> k) & 1u) << sel;
      }
      T* up = u + p + (((s + (q & 1) + (q >> 1)) & 1) ? half : 0);
      *up += neumann ? prolong_mean8(ev, o) : prolong_trilinear(ev);
    }
  }
}

}  // namespace iim
