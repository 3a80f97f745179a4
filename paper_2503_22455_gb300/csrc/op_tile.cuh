// The 3D operator (order 4) at plain nodes of large grids, in fixed point; included by operator.cu.
//
// A plain node takes 13 FP64 operations, and GB300 issues two per clock and SM: 357 us at 256^3, where
// reading u and writing w takes 40 us.  Integers are 32 to 64 times faster, so a tile's values are
// turned once into 60-bit integers k = u 2^(59-e), |u| < 2^e over the tile, and a node's sum becomes
// integer additions: with D_j = sum over the axes of (k_{i+je} + k_{i-je}) - 6 k_i,
//     L u = beta a_1 / h^2  (D_1 - D_2 / 16)  2^(e-59)          (a_2 = -a_1 / 16, a_0 = -2 sum a_j)
// where only the conversion of the bracket and one product are left to FP64.  Everything up to the
// conversion is exact but for the cut of u at 2^(e-59) and of D_2 / 16 to whole units, while FP64 rounds
// each partial sum at 2^-53 of its size: as long as one of the node's values is above 2^(e-6), the
// integers lose less.  Every k carries in its lowest bit whether its value is above 2^(e-5); a node that
// sees no such value is left to the FP64 sum, and so is a tile whose exponents leave the range in which
// the product is sure to be normal (NaN, infinities).  RMS error against the exact sum, relative to
// max |u| beta / h^2, at 128^3 (96^3 the same): smooth u 3e-19 (FP64 sums: 3.6e-16), a product of sines
// 4e-18 (3.0e-16), a peak 1e-18 (5.7e-17), normal random u 1.44e-16 (1.53e-16).
//
// Tiles of 32 x 16 columns of 8 planes, one thread each; the column and its 2 w halo planes stay in the
// thread's registers, neighbours across come from shared memory (46 KB, two CTAs per SM).  Two thirds
// of an exterior problem's tiles are whole and plain (noted at set-up) and read without a bound or a
// class.  One application at 256^3 (Neumann, exterior of an ellipsoid), ghosts and affected nodes
// included: 518 us with a thread per node, 281 with the tiles; at 96^3 (interior) 38 and 37.
template <int W>
struct OpTile {
  static constexpr int TX = 32, TY = 16, TZ = 8, NT = TX * TY;
  static constexpr int HX = TX + 2 * W, HY = TY + 2 * W;
  long long k[TZ][HY][HX];
  unsigned red[NT / 32];
  static __host__ __device__ int tiles(int n, int axis) {
    const int t = axis == 0 ? TX : (axis == 1 ? TY : TZ);
    return (n + t - 1) / t;
  }
  static __host__ __device__ int count(int n) {
    return tiles(n, 0) * tiles(n, 1) * tiles(n, 2);
  }
};

// k = u 2^(59-e) cut to a whole number, its lowest bit replaced by the flag |u| >= 2^(e-5); ebits: the
// tile's largest exponent field
__device__ __forceinline__ long long op_fixed(double u, int ebits) {
  const int hi = __double2hiint(u), lo = __double2loint(u);
  const int sh = min(ebits - ((hi >> 20) & 0x7ff), 63);
  unsigned long long m = ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)lo) << 6;
  m >>= sh;
  const long long s = (long long)hi >> 31;
  const long long k = ((long long)m ^ s) - s;
  return (k & ~1ll) | (sh <= 4 ? 1 : 0);
}

// the FP64 sum of a plain node (all neighbours in phase)
template <int D, int W>
__device__ __forceinline__ double ho_plain_node(int n, const StencilCoef& C, bool plus, const double* __restrict__ u,
                                                int64_t i) {
  double acc = (plus ? C.c0[1] : C.c0[0]) * u[i];
#pragma unroll
  for (int j = 1; j <= W; ++j) {
    double s = u[i - j];
    s += u[i + j];
    s += u[i - (int64_t)j * n];
    s += u[i + (int64_t)j * n];
    if (D > 2) {
      const int64_t nn = (int64_t)n * n;
      s += u[i - j * nn];
      s += u[i + j * nn];
    }
    acc = fma(plus ? C.cj[1][j - 1] : C.cj[0][j - 1], s, acc);
  }
  return acc;
}

// What the set-up notes of a tile: it has plain nodes; every value it reads is an unknown's and inside
// the grid; all its own nodes are plain (and then of one phase)
constexpr uint8_t kTileWork = 1, kTileWhole = 2, kTilePlain = 4;

// tile's first node, and the number of its values that e = 0 .. counts: columns with their halo planes,
// then the halo columns
template <int W>
struct TileWalk {
  using T = OpTile<W>;
  static constexpr int NP = T::TZ + 2 * W;
  static constexpr int XH = 2 * W * T::TY * T::TZ, YH = 2 * W * T::TX * T::TZ;
  int n, bx, by, bz;
  __device__ __forceinline__ TileWalk(int n_, int tile) : n(n_) {
    const int tx = T::tiles(n, 0), ty = T::tiles(n, 1), br = tile / tx;
    bx = tile % tx * T::TX;
    by = br % ty * T::TY;
    bz = br / ty * T::TZ;
  }
  // halo entry e of the columns across x / y: its place relative to the tile
  static __device__ __forceinline__ void x_halo(int e, int& px, int& py, int& pz) {
    const int h = e % (2 * W), r = e / (2 * W);
    px = h < W ? h - W : T::TX + h - W;
    py = r % T::TY;
    pz = r / T::TY;
  }
  static __device__ __forceinline__ void y_halo(int e, int& px, int& py, int& pz) {
    const int r = e / T::TX, h = r % (2 * W);
    px = e % T::TX;
    py = h < W ? h - W : T::TY + h - W;
    pz = r / (2 * W);
  }
  __device__ __forceinline__ bool inside(int px, int py, int pz) const {
    return bx + px >= 0 && bx + px < n && by + py >= 0 && by + py < n && bz + pz >= 0 && bz + pz < n;
  }
  // node of a place; outside the grid, the nearest one inside (no plain node reads it)
  __device__ __forceinline__ int64_t node(int px, int py, int pz) const {
    const int x = min(max(bx + px, 0), n - 1), y = min(max(by + py, 0), n - 1), z = min(max(bz + pz, 0), n - 1);
    return x + (int64_t)n * (y + (int64_t)n * z);
  }
};

// the tiles' notes (set-up): one block per tile
template <int W>
__global__ void __launch_bounds__(OpTile<W>::NT) k_tile_kinds(int n, const uint8_t* __restrict__ kind,
                                                                 uint8_t* __restrict__ tiles) {
  using T = OpTile<W>;
  using K = TileWalk<W>;
  const K t(n, blockIdx.x);
  const int tid = threadIdx.x, x = tid % T::TX, y = tid / T::TX;
  bool work = false, whole = true, plain = true;
  int px, py, pz;
  auto at = [&](int ax, int ay, int az, bool own) {
    const bool in = t.inside(ax, ay, az);
    const uint8_t kd = in ? kind[t.node(ax, ay, az)] : 0;
    whole = whole && (kd & kKindUnknown);
    if (!own) return;
    const bool p = (kd & kKindUnknown) && !(kd & kKindAffected);
    work = work || p;
    plain = plain && p;
  };
  for (int p = 0; p < K::NP; ++p) at(x, y, p - W, p >= W && p < W + T::TZ);
  for (int e = tid; e < K::XH; e += T::NT) {
    K::x_halo(e, px, py, pz);
    at(px, py, pz, false);
  }
  for (int e = tid; e < K::YH; e += T::NT) {
    K::y_halo(e, px, py, pz);
    at(px, py, pz, false);
  }
  work = __syncthreads_or(work);
  whole = __syncthreads_and(whole);
  plain = __syncthreads_and(plain);
  if (tid == 0) tiles[blockIdx.x] = (work ? kTileWork : 0) | (whole ? kTileWhole : 0) | (plain ? kTilePlain : 0);
}

// One tile, FAST: both kTileWhole and kTilePlain hold.  Values at nodes that are no unknowns read as 0
// (no plain node needs them).  AFF: affected(i) is called for every affected node (else another
// kernel's).
template <int W, bool FAST, bool AFF, class Aff>
__device__ __forceinline__ void op_tile_body(OpTile<W>& S, const GridView& g, const StencilCoef& C, bool whole,
                                             const uint8_t* __restrict__ kind, const double* __restrict__ u,
                                             double* __restrict__ w, int tile, Aff affected) {
  static_assert(W == 2, "the sum below has a_2 = -a_1 / 16 and 60 bits for two offsets");
  using T = OpTile<W>;
  using K = TileWalk<W>;
  constexpr int TX = T::TX, TZ = T::TZ, NT = T::NT, NP = K::NP, XH = K::XH, YH = K::YH;
  constexpr int NXH = (XH + NT - 1) / NT, NYH = (YH + NT - 1) / NT;
  const int n = g.n, tid = threadIdx.x, x = tid % TX, y = tid / TX;
  const K tw(n, tile);
  const int64_t i0 = tw.bx + x + (int64_t)n * (tw.by + y + (int64_t)n * tw.bz), st = (int64_t)n * n;
  auto value = [&](int px, int py, int pz) -> double {
    const int64_t i = FAST ? tw.bx + px + (int64_t)n * (tw.by + py + (int64_t)n * (tw.bz + pz)) : tw.node(px, py, pz);
    return FAST || whole || (kind[i] & kKindUnknown) ? u[i] : 0.0;
  };
  double v[NP], vx[NXH], vy[NYH];
#pragma unroll
  for (int p = 0; p < NP; ++p) v[p] = FAST ? u[i0 + (p - W) * st] : value(x, y, p - W);
#pragma unroll
  for (int q = 0; q < NXH; ++q) {
    int px, py, pz;
    K::x_halo(tid + q * NT, px, py, pz);
    vx[q] = XH % NT == 0 || tid + q * NT < XH ? value(px, py, pz) : 0.0;
  }
#pragma unroll
  for (int q = 0; q < NYH; ++q) {
    int px, py, pz;
    K::y_halo(tid + q * NT, px, py, pz);
    vy[q] = YH % NT == 0 || tid + q * NT < YH ? value(px, py, pz) : 0.0;
  }
  unsigned top = 0;
  auto raise = [&](double d) { top = max(top, ((unsigned)__double2hiint(d) & 0x7fffffffu) | (__double2loint(d) != 0)); };
#pragma unroll
  for (int p = 0; p < NP; ++p) raise(v[p]);
#pragma unroll
  for (int q = 0; q < NXH; ++q) raise(vx[q]);
#pragma unroll
  for (int q = 0; q < NYH; ++q) raise(vy[q]);
  top = __reduce_max_sync(0xffffffffu, top);
  if ((tid & 31) == 0) S.red[tid >> 5] = top;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NT / 32; ++k) top = max(top, S.red[k]);
  const bool zero = top == 0;
  const int eb = zero ? 200 : (int)(top >> 20);
  const bool fixed = eb >= 200 && eb <= 1800;
  long long k[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    k[p] = op_fixed(v[p], eb);
    if (p >= W && p < W + TZ) S.k[p - W][y + W][x + W] = k[p];
  }
#pragma unroll
  for (int q = 0; q < NXH; ++q) {
    int px, py, pz;
    K::x_halo(tid + q * NT, px, py, pz);
    if (XH % NT == 0 || tid + q * NT < XH) S.k[pz][py + W][px + W] = op_fixed(vx[q], eb);
  }
#pragma unroll
  for (int q = 0; q < NYH; ++q) {
    int px, py, pz;
    K::y_halo(tid + q * NT, px, py, pz);
    if (YH % NT == 0 || tid + q * NT < YH) S.k[pz][py + W][px + W] = op_fixed(vy[q], eb);
  }
  __syncthreads();
  if (!FAST && (tw.bx + x >= n || tw.by + y >= n)) return;
  // the product's factor: beta a_1 / h^2 2^(e-59), 2^e = 2^(eb-1022)
  const double unit = __hiloint2double((eb - 58) << 20, 0);
  const double f0 = C.cj[0][0] * unit, f1 = C.cj[1][0] * unit;
  uint8_t kd = FAST ? kind[i0] : 0;
  unsigned todo = 0;
#pragma unroll
  for (int z = 0; z < TZ; ++z) {
    const int64_t i = i0 + z * st;
    if (!FAST) {
      if (tw.bz + z >= n) break;
      kd = kind[i];
      if (kd & kKindAffected) {
        if (AFF) todo |= 1u << z;
        continue;
      }
      if (!(kd & kKindUnknown)) {
        w[i] = 0.0;
        continue;
      }
    }
    const long long kc = k[z + W];
    unsigned seen = (unsigned)kc;
    long long t = 0;
#pragma unroll
    for (int j = 1; j <= W; ++j) {
      const long long xa = S.k[z][y + W][x + W - j], xb = S.k[z][y + W][x + W + j], za = k[z + W - j], zb = k[z + W + j];
      const long long ya = S.k[z][y + W - j][x + W], yb = S.k[z][y + W + j][x + W];
      seen |= (unsigned)xa | (unsigned)xb | (unsigned)ya | (unsigned)yb | (unsigned)za | (unsigned)zb;
      const long long s = (xa + xb) + (ya + yb) + (za + zb) - 6 * kc;
      t = j == 1 ? s : t - (s >> 4);       // a_2 / a_1 = -1/16
    }
    if (fixed && ((seen & 1) || zero)) w[i] = (double)t * (kd & kKindPlus ? f1 : f0);
    else todo |= 1u << z;
  }
  while (todo) {
    const int z = __ffs(todo) - 1;
    todo &= todo - 1;
    const int64_t i = i0 + z * st;
    if (!FAST) kd = kind[i];
    if (AFF && (kd & kKindAffected)) affected(i);
    else w[i] = ho_plain_node<3, W>(n, C, (kd & kKindPlus) != 0, u, i);
  }
}

template <int W, bool AFF, class Aff>
__device__ __forceinline__ void op_tile(OpTile<W>& S, const GridView& g, const StencilCoef& C,
                                        const uint8_t* __restrict__ kind, const uint8_t* __restrict__ tiles,
                                        const double* __restrict__ u, double* __restrict__ w, int tile, Aff affected) {
  const uint8_t note = tiles[tile];
  if ((note & kTileWhole) && (note & kTilePlain)) {
    op_tile_body<W, true, AFF>(S, g, C, true, kind, u, w, tile, affected);
  } else if (note & kTileWork) {
    op_tile_body<W, false, AFF>(S, g, C, (note & kTileWhole) != 0, kind, u, w, tile, affected);
  } else {                                 // only affected nodes and nodes that are no unknowns
    using T = OpTile<W>;
    const TileWalk<W> t(g.n, tile);
    const int x = threadIdx.x % T::TX, y = threadIdx.x / T::TX;
    for (int z = 0; z < T::TZ; ++z) {
      if (!t.inside(x, y, z)) break;
      const int64_t i = t.node(x, y, z);
      const uint8_t kd = kind[i];
      if (!(kd & kKindUnknown)) w[i] = 0.0;
      else if (AFF) affected(i);
    }
  }
}
