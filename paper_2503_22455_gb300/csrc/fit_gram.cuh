// Least-squares fits (paper Sec. 2.1-2.2) of the common case, included by setup.cu.
//
// Each fit needs the rows s_t = V (V^T V)^-1 c_t of its w + 1 targets c_t (w ghosts and the
// normal derivative): one FP64 problem of M monomials and about 93 (3D, degree 4) or 44 (2D,
// degree 6) rows.  A GB300 SM takes one FP64 warp instruction per 16 clocks, so the method is
// the one with the fewest of them: corrected semi-normal equations (Bjoerck 1987).
//   1. V^T V from the moments of the nodes: its M^2 / 2 entries are sums of x^a y^b z^c of
//      degree <= 2 q, 165 different ones for M = 35 (91 for M = 28);
//   2. L D L^T of it, in registers;
//   3. s = V z with V^T V z = c; the residual r = c - V^T s in the same arithmetic;
//      s += V dz with V^T V dz = r.
// Semi-normal equations square the condition number, so the monomials are taken around the
// middle of the half-ellipsoid and scaled (xi' = (xi - x_mid) / 4): s does not depend on the
// basis, and cond(V) falls from 2e3-4e3 (3D) and 1e6 (2D, degree 6) to 3e2-5e2 and 1e3.
// Against extended precision the rows are then good to 6e-16 of their size (3D) and 4e-15 (2D,
// degree 6); Householder QR of the monomials around x_c gives 2e-14 and 4e-13.
//
// The rank test of k_fit is on |R_kk| of the monomials around x_c.  Shifting the centre does
// not change them (the shifted monomials are the old ones plus terms of lower degree, which
// come earlier), so |R_kk|^2 = D_k 16^deg(k) here.  Only fits with min |R_kk| >= 1e-3 max |R_kk|
// are taken (the test asks for 1e-8; 0.2 and 0.014 are seen); the others, and those with too few or
// too many rows for this layout, are listed for k_fit, which decides by QR.
//
// Layout: LANES lanes per fit (32 in 3D, 16 in 2D), rows over the lanes in three slots (a fourth
// for fits of more than 3 LANES rows in 3D).  Sums over the rows are transposed butterflies:
// P sums over the lanes cost about P additions.  The 14^3 (2D: 18^2) window is scanned in FP32
// with a margin of 1e-4 (its rounding error stays below 1e-5); only nodes inside the margin are
// decided in FP64, by the expression k_fit uses, so both kernels select the same nodes.
//
// Measured on a GB300 (against Householder QR kernels of the same fits, one warp per fit in 3D
// and four fits per warp in 2D): set-up of the 192^3 ellipsoid (36.9 k fits) 96.1 -> 11.3 ms,
// fits of the 1024^2 star interface (degree 6, 5.3 k fits) 1.40 -> 0.68 ms; the FP64 pipe is 86 %
// (3D) and 83 % (2D) busy.  A Householder QR with two fits per warp, rows over 16 lanes, took
// 23 ms for the 192^3 fits: 33 KB of shared memory per fit left three warps per SM.
#pragma once

namespace iim {

template <int DIM, int Q, int LANES_, int SLOTS_>
struct GramShape {
  static constexpr int dim = DIM, q = Q, LANES = LANES_, SLOTS = SLOTS_;
  static constexpr int W = Q / 2, NT = W + 1;
  static constexpr int M = DIM == 2 ? (Q + 1) * (Q + 2) / 2 : (Q + 1) * (Q + 2) * (Q + 3) / 6;
  static constexpr int D2 = 2 * Q;
  static constexpr int NMOM = DIM == 2 ? (D2 + 1) * (D2 + 2) / 2 : (D2 + 1) * (D2 + 2) * (D2 + 3) / 6;
  static constexpr int CMAX = DIM == 3 ? Q : 0;        // largest z exponent of a monomial
  static constexpr int CMOM = DIM == 3 ? D2 : 0;       // ... of a moment
  static constexpr int NPAIR = M * (M + 1) / 2;
  static constexpr int NG = (NPAIR + LANES - 1) / LANES;   // matrix entries per lane
  static constexpr int NZ = (M + LANES - 1) / LANES;       // unknowns per lane
  static constexpr int ROWS = LANES * SLOTS;
  static constexpr int WIN = 2 * (Q + 2) + 2;          // window nodes per axis: ceil(q + 1) + 1 each side
  static constexpr int LD = M | 1;                     // odd stride: columns hit distinct banks

  // position of x^a y^b z^c among the monomials (graded, then decreasing a, then b)
  static constexpr int mono(int a, int b, int c) {
    const int deg = a + b + c;
    if (DIM == 2) return deg * (deg + 1) / 2 + (deg - a);
    return deg * (deg + 1) * (deg + 2) / 6 + (deg - a) * (deg - a + 1) / 2 + (deg - a - b);
  }
  // position of the moment x^a y^b z^c: by c, then a, then b
  static constexpr int mom(int a, int b, int c) {
    int o = 0;
    for (int cc = 0; cc < c; ++cc) o += (D2 - cc + 1) * (D2 - cc + 2) / 2;
    for (int aa = 0; aa < a; ++aa) o += D2 - c - aa + 1;
    return o + b;
  }
};

// Entries of the lower triangle, columns from the last to the first (so that the entries a step
// still updates are a prefix): row, column and the moment each entry is.
template <typename S>
struct GramTable {
  int32_t e[S::NG * S::LANES];           // row | column << 6 | moment << 12
  int8_t ex[S::M][3];                    // exponents of each monomial
  constexpr GramTable() : e(), ex() {
    int k = 0;
    for (int deg = 0; deg <= S::q; ++deg)
      for (int a = deg; a >= 0; --a)
        for (int b = S::dim == 2 ? deg - a : deg - a; b >= (S::dim == 2 ? deg - a : 0); --b) {
          ex[k][0] = (int8_t)a;
          ex[k][1] = (int8_t)b;
          ex[k][2] = (int8_t)(deg - a - b);
          ++k;
        }
    int p = 0;
    for (int j = S::M - 1; j >= 0; --j)
      for (int i = j; i < S::M; ++i)
        e[p++] = i | (j << 6) | (S::mom(ex[i][0] + ex[j][0], ex[i][1] + ex[j][1], ex[i][2] + ex[j][2]) << 12);
    for (; p < S::NG * S::LANES; ++p) e[p] = 0;
  }
};

template <typename S>
__device__ constexpr GramTable<S> kGramTable = GramTable<S>();

template <typename S>
struct GramSmem {                        // one fit
  double mom[S::NMOM > S::NT * S::M ? S::NMOM : S::NT * S::M];   // moments, then V^T s
  double L[S::M * S::LD];                // column k: l_ik (i > k), unscaled
  double C[S::M + 1];                    // the current column before its scaling
  double rd[S::M + 1];                   // 1 / D_k
  double z[S::NT][S::M];                 // solutions, residuals (targets' order of the monomials)
  double xi[S::dim][S::WIN];             // (node - x_c) / h along each axis of the window
  int code[S::ROWS];                     // window position of each row's node, i0 | i1 << 5 | i2 << 10
};

// moments with x exponents A0 .. A1 and z exponents C0 .. C1
template <typename S, int A0, int A1, int C0, int C1>
__device__ __forceinline__ void gram_moments(const double (&x)[S::SLOTS], const double (&y)[S::SLOTS],
                                             const double (&z)[S::SLOTS], const double (&w)[S::SLOTS], int ns, int hl,
                                             double* out) {
  constexpr int N = [] {
    int n = 0;
    for (int c = C0; c <= C1; ++c)
      for (int a = A0; a <= A1 && a <= S::D2 - c; ++a) n += S::D2 - c - a + 1;
    return n;
  }();
  constexpr int B = S::D2 - C0 - A0;
  double acc[N];
#pragma unroll
  for (int k = 0; k < N; ++k) acc[k] = 0.0;
#pragma unroll
  for (int s = 0; s < S::SLOTS; ++s) {
    if (s >= ns) break;
    double py[B + 1];
    py[0] = 1.0;
#pragma unroll
    for (int b = 1; b <= B; ++b) py[b] = py[b - 1] * y[s];
    double wc = w[s];
#pragma unroll
    for (int c = 0; c < C0; ++c) wc *= z[s];
    int k = 0;
#pragma unroll
    for (int c = C0; c <= C1; ++c) {
      double t = wc;
#pragma unroll
      for (int a = 0; a < A0; ++a) t *= x[s];
#pragma unroll
      for (int a = A0; a <= A1; ++a) {
        if (a > S::D2 - c) break;
#pragma unroll
        for (int b = 0; b <= B; ++b) {
          if (b > S::D2 - c - a) break;
          acc[k] = b == 0 ? acc[k] + t : fma(t, py[b], acc[k]);
          ++k;
        }
        t *= x[s];
      }
      wc *= z[s];
    }
  }
  lane_sums<S::LANES, N>(acc, hl, out + S::mom(A0, 0, C0));
}

// reciprocal by Newton's iteration from the FP32 one: relative error 2^-23 -> 2^-46 -> 2^-53
__device__ __forceinline__ double gram_rcp(double d) {
  double r = (double)(1.0f / (float)d);
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}

// polynomials with the coefficients sm.z at this lane's rows, by nested Horner: s (+)= P(x, y, z)
template <typename S, bool ADD>
__device__ __forceinline__ void gram_rows(const GramSmem<S>& sm, const double (&x)[S::SLOTS], const double (&y)[S::SLOTS],
                                          const double (&z)[S::SLOTS], int m, int hl, int ns,
                                          double (&s)[S::NT][S::SLOTS]) {
#pragma unroll
  for (int t = 0; t < S::NT; ++t) {
    double pc[S::SLOTS];
#pragma unroll
    for (int c = S::CMAX; c >= 0; --c) {
      double pb[S::SLOTS];
#pragma unroll
      for (int b = S::q - c; b >= 0; --b) {
        double pa[S::SLOTS];
#pragma unroll
        for (int a = S::q - c - b; a >= 0; --a) {
          const double cf = sm.z[t][S::mono(a, b, c)];
#pragma unroll
          for (int k = 0; k < S::SLOTS; ++k) {
            if (k >= ns) break;
            pa[k] = a == S::q - c - b ? cf : fma(pa[k], x[k], cf);
          }
        }
#pragma unroll
        for (int k = 0; k < S::SLOTS; ++k) {
          if (k >= ns) break;
          pb[k] = b == S::q - c ? pa[k] : fma(pb[k], y[k], pa[k]);
        }
      }
#pragma unroll
      for (int k = 0; k < S::SLOTS; ++k) {
        if (k >= ns) break;
        pc[k] = c == S::CMAX ? pb[k] : fma(pc[k], z[k], pb[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < S::SLOTS; ++k) {
      if (k >= ns) break;
      const double v = hl + S::LANES * k < m ? pc[k] : 0.0;
      s[t][k] = ADD ? s[t][k] + v : v;
    }
  }
}

// sums over the rows of the monomials with z exponent C times each target's s: V^T s
template <typename S, int C>
__device__ __forceinline__ void gram_project(const double (&x)[S::SLOTS], const double (&y)[S::SLOTS],
                                             const double (&z)[S::SLOTS], const double (&s)[S::NT][S::SLOTS], int ns, int hl,
                                             double* out) {
  constexpr int NXY = (S::q - C + 1) * (S::q - C + 2) / 2;
  // in 2D the targets go one after the other (28 sums each), in 3D all three together
  constexpr int TG = S::dim == 2 ? 1 : S::NT;
#pragma unroll
  for (int t0 = 0; t0 < S::NT; t0 += TG) {
    double acc[NXY * TG];
#pragma unroll
    for (int k = 0; k < NXY * TG; ++k) acc[k] = 0.0;
#pragma unroll
    for (int k = 0; k < S::SLOTS; ++k) {
      if (k >= ns) break;
      double py[S::q - C + 1], sc[TG];
      py[0] = 1.0;
#pragma unroll
      for (int b = 1; b <= S::q - C; ++b) py[b] = py[b - 1] * y[k];
#pragma unroll
      for (int t = 0; t < TG; ++t) {
        sc[t] = s[t0 + t][k];
#pragma unroll
        for (int c = 0; c < C; ++c) sc[t] *= z[k];
      }
      int n = 0;
      double xa = 1.0;
#pragma unroll
      for (int a = 0; a <= S::q - C; ++a) {
#pragma unroll
        for (int b = 0; b <= S::q - C; ++b) {
          if (b > S::q - C - a) break;
          const double xy = a == 0 ? py[b] : (b == 0 ? xa : xa * py[b]);
#pragma unroll
          for (int t = 0; t < TG; ++t) acc[n * TG + t] = fma(xy, sc[t], acc[n * TG + t]);
          ++n;
        }
        xa *= x[k];
      }
    }
    lane_sums<S::LANES, NXY * TG>(acc, hl, out + t0 * NXY);
  }
}

// z <- (L D L^T)^-1 z for every target; lane hl holds unknowns hl, hl + LANES, ...
template <typename S>
__device__ __forceinline__ void gram_solve(const GramSmem<S>& sm, double (&z)[S::NT][S::NZ], int hl, int base) {
  constexpr int LN = S::LANES, M = S::M, NT = S::NT;
  // With a few unknowns more than lanes (3D: 35), the lanes that hold two are done with their
  // first after EX steps; from then on each lane has one unknown left.
  constexpr int EX = M - LN;
  constexpr bool WRAP = S::NZ == 2 && EX <= LN / 4;
  constexpr int K1 = WRAP ? EX : M - 1;
#pragma unroll 1
  for (int k = 0; k < K1; ++k) {                       // z_i -= l_ik z_k, i > k
    double zk[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      double v = z[t][0];
#pragma unroll
      for (int s = 1; s < S::NZ; ++s) v = k >= LN * s ? z[t][s] : v;
      zk[t] = __shfl_sync(0xffffffffu, v, base + k % LN);
    }
#pragma unroll
    for (int s = 0; s < S::NZ; ++s) {
      if (LN * (s + 1) - 1 <= k) continue;
      const int i = hl + LN * s;
      const double l = i > k && i < M ? sm.L[k * S::LD + i] : 0.0;
#pragma unroll
      for (int t = 0; t < NT; ++t) z[t][s] = fma(-l, zk[t], z[t][s]);
    }
  }
  if constexpr (WRAP) {
    const bool sec = hl < EX;
    const int i = sec ? hl + LN : hl;
    double cur[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) cur[t] = sec ? z[t][1] : z[t][0];
#pragma unroll 1
    for (int k = EX; k < M - 1; ++k) {
      const double l = i > k ? sm.L[k * S::LD + i] : 0.0;
#pragma unroll
      for (int t = 0; t < NT; ++t) cur[t] = fma(-l, __shfl_sync(0xffffffffu, cur[t], k % LN), cur[t]);
    }
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      z[t][0] = sec ? z[t][0] : cur[t];
      z[t][1] = sec ? cur[t] : 0.0;
    }
  }
#pragma unroll
  for (int s = 0; s < S::NZ; ++s) {
    const int i = hl + LN * s;
    const double r = i < M ? sm.rd[i] : 0.0;
#pragma unroll
    for (int t = 0; t < NT; ++t) z[t][s] *= r;
  }
#pragma unroll 1
  for (int k = M - 1; k > 0; --k) {                    // z_i -= l_ki z_k, i < k
    double zk[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      double v = z[t][0];
#pragma unroll
      for (int s = 1; s < S::NZ; ++s) v = k >= LN * s ? z[t][s] : v;
      zk[t] = __shfl_sync(0xffffffffu, v, base + k % LN);
    }
#pragma unroll
    for (int s = 0; s < S::NZ; ++s) {
      if (LN * s >= k) continue;
      const int i = hl + LN * s;
      const double l = i < k ? sm.L[i * S::LD + k] : 0.0;
#pragma unroll
      for (int t = 0; t < NT; ++t) z[t][s] = fma(-l, zk[t], z[t][s]);
    }
  }
}

__device__ __forceinline__ void fit_append(int* list, int f) { list[1 + atomicAdd(list, 1)] = f; }

template <typename S>
__global__ void __launch_bounds__(32) k_fit_gram(FitParams P, int* __restrict__ later) {
  extern __shared__ __align__(16) unsigned char smg[];
  constexpr int LN = S::LANES, FW = 32 / LN, DIM = S::dim, M = S::M, NT = S::NT, NZ = S::NZ;
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x, hl = lane % LN, base = lane - hl;
  GramSmem<S>& sm = reinterpret_cast<GramSmem<S>*>(smg)[lane / LN];
  const GramTable<S>& tab = kGramTable<S>;
  const GridView& g = P.g;
  const int n = g.n;
  const int nfit_here = P.interface_ ? 2 * (*P.K) : *P.K;
  if ((int)blockIdx.x * FW >= nfit_here) return;
  const int f = blockIdx.x * FW + lane / LN;
  bool active = f < nfit_here;
  const int c = active ? (P.interface_ ? (f >> 1) : f) : 0;
  const bool sig_plus = P.interface_ ? ((f & 1) == 0) : true;
  double xc[DIM], nrm[DIM], ns_[DIM];
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    xc[k] = P.cr_x[c * DIM + k];
    nrm[k] = P.cr_n[c * DIM + k];
    ns_[k] = sig_plus ? -nrm[k] : nrm[k];              // points into phase sigma
  }
  const int ax = P.cr_axis[c];
  const int lo = P.cr_lo[c];
  const bool lo_sig = (P.cr_loplus[c] != 0) == sig_plus;
  const double tq = P.cr_t[c];
  // the phase-sigma node nearest to x_c is the sigma end of the cut edge, every other node being at
  // least h away, unless x_c sits on the other end (below)
  const int st_ax = ax == 0 ? 1 : (ax == 1 ? n : n * n);
  int nearest = lo_sig ? lo : lo + st_ax;
  const bool on_end = active && !((lo_sig ? tq : 1.0 - tq) < 1.0 - 1e-9);
  // ---- window coordinates
  int w0[DIM];
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    w0[k] = (int)floor((xc[k] + 1.0) / g.h - 0.5) - (S::q + 2);
    for (int i = hl; i < S::WIN; i += LN) sm.xi[k][i] = (node_x(g, w0[k] + i) - xc[k]) / g.h;
  }
  __syncwarp();
  if (on_end) {
    // then that end's other neighbours may be as near: the least distance, the smallest index among
    // equals, by the expressions of k_fit.  Left to k_fit, the 1.6 k such fits of a flat-sided interface took
    // 0.57 ms at 1024^2 (order 4), 6.5 k 4.6 ms at 4096^2 (order 6), 16 of 36 ms of set-up at 128^3.
    const int e = lo_sig ? lo + st_ax : lo, ei[3] = {e % n, (e / n) % n, DIM == 2 ? 0 : e / n / n};
    double bd = 1e300;
    nearest = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < 2 * DIM; ++j) {
      const int pos = ei[j >> 1] + (j & 1 ? 1 : -1);
      if (pos < 0 || pos >= n) continue;
      const int fl = e + (j & 1 ? 1 : -1) * (j < 2 ? 1 : (j < 4 ? n : n * n));
      if ((P.phase[fl] != 0) != sig_plus) continue;
      double d2 = 0;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        const double rr = sm.xi[k][(k == j >> 1 ? pos : ei[k]) - w0[k]];
        d2 = fma(rr, rr, d2);
      }
      better(bd, nearest, d2, fl);
    }
  }
  // ---- rows of X_c, in the order of the flat index
  const double an = S::q + 1.0, at = S::q / 2 + 1.0;
  int R = 0;
  {
    float fn[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) fn[k] = (float)ns_[k];
    constexpr float ian2 = 1.0f / ((S::q + 1) * (S::q + 1)), iat2 = 1.0f / ((S::q / 2 + 1) * (S::q / 2 + 1));
    constexpr int TOTAL = DIM == 2 ? S::WIN * S::WIN : S::WIN * S::WIN * S::WIN;
    constexpr int LB = 4;              // phase loads in flight together
#pragma unroll 1
    for (int p0 = 0; p0 < TOTAL; p0 += LB * LN) {
      int code[LB], fl[LB];
      uint8_t ph[LB];
      bool cand[LB];
#pragma unroll
      for (int l = 0; l < LB; ++l) {
        const int p = p0 + l * LN + hl;
        const int i0 = p % S::WIN, r = p / S::WIN, i1 = DIM == 2 ? r : r % S::WIN, i2 = DIM == 2 ? 0 : r / S::WIN;
        const int m0 = w0[0] + i0, m1 = w0[1] + i1, m2 = DIM == 2 ? 0 : w0[DIM - 1] + i2;
        bool ok = active && p < TOTAL && m0 >= 0 && m0 < n && m1 >= 0 && m1 < n && m2 >= 0 && m2 < n;
        ph[l] = 0;
        code[l] = i0 | (i1 << 5) | (i2 << 10);
        fl[l] = m0 + n * (m1 + n * m2);
        if (ok) {
          const float x = (float)sm.xi[0][i0], y = (float)sm.xi[1][i1], z = DIM == 2 ? 0.f : (float)sm.xi[DIM - 1][i2];
          const float t = x * fn[0] + y * fn[1] + (DIM == 2 ? 0.f : z * fn[DIM - 1]), d2 = x * x + y * y + z * z;
          const float val = fmaxf(d2 - t * t, 0.f) * iat2 + t * t * ian2;
          ok = t > -1e-4f && val < 1.f + 1e-4f;
          if (ok && !(t > 1e-4f && val < 1.f - 1e-4f)) {
            // too close to call in FP32
            const int ii[3] = {i0, i1, i2};
            double e2 = 0, td = 0;
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
              const double rr = sm.xi[k][ii[k]];
              e2 += rr * rr;
              td += rr * ns_[k];
            }
            const double ta2 = fmax(e2 - td * td, 0.0);
            ok = td >= 0.0 && ta2 / (at * at) + td * td / (an * an) <= 1.0;
          }
        }
        cand[l] = ok;
        if (ok) ph[l] = P.phase[fl[l]];
      }
#pragma unroll
      for (int l = 0; l < LB; ++l) {
        const bool sel = cand[l] && (ph[l] != 0) == sig_plus && fl[l] != nearest;
        unsigned mk = __ballot_sync(FULL, sel) >> base;
        if (LN < 32) mk &= (1u << (LN & 31)) - 1u;
        const int o = R + __popc(mk & ((1u << hl) - 1u));
        if (sel && o < S::ROWS - 1) sm.code[o] = code[l];
        R += __popc(mk);
      }
    }
  }
  if (active && (R + 1 > S::ROWS || R + 1 < M)) {
    if (hl == 0) fit_append(later, f);
    active = false;
  }
  const int m = active ? R + 1 : 0;
  int mmax = m;
#pragma unroll
  for (int o = LN; o < 32; o <<= 1) mmax = max(mmax, __shfl_xor_sync(FULL, mmax, o));
  if (mmax == 0) return;
  const int nsl = mmax > LN * (S::SLOTS - 1) ? S::SLOTS : S::SLOTS - 1;   // row slots in use
  __syncwarp();
  // ---- this lane's rows (row 0: the control point), coordinates around the middle of the set
  constexpr double SC = 0.25;
  double mid[DIM];
#pragma unroll
  for (int k = 0; k < DIM; ++k) mid[k] = 0.4 * an * ns_[k];
  double x[S::SLOTS], y[S::SLOTS], z[S::SLOTS], w[S::SLOTS];
#pragma unroll
  for (int s = 0; s < S::SLOTS; ++s) {
    const int row = hl + LN * s;
    const bool in = row < m;
    const int code = in && row > 0 ? sm.code[row - 1] : 0;
    const bool node = in && row > 0;
    x[s] = in ? ((node ? sm.xi[0][code & 31] : 0.0) - mid[0]) * SC : 0.0;
    y[s] = in ? ((node ? sm.xi[1][(code >> 5) & 31] : 0.0) - mid[1]) * SC : 0.0;
    z[s] = DIM == 3 && in ? ((node ? sm.xi[DIM - 1][code >> 10] : 0.0) - mid[DIM - 1]) * SC : 0.0;
    w[s] = in ? 1.0 : 0.0;
  }
  // ---- moments
  if constexpr (DIM == 3) {
    static_assert(DIM == 2 || S::q == 4, "groups of moments");
    gram_moments<S, 0, 8, 0, 0>(x, y, z, w, nsl, hl, sm.mom);
    gram_moments<S, 0, 8, 1, 1>(x, y, z, w, nsl, hl, sm.mom);
    gram_moments<S, 0, 8, 2, 2>(x, y, z, w, nsl, hl, sm.mom);
    gram_moments<S, 0, 8, 3, 4>(x, y, z, w, nsl, hl, sm.mom);
    gram_moments<S, 0, 8, 5, 8>(x, y, z, w, nsl, hl, sm.mom);
  } else {
    gram_moments<S, 0, 3, 0, 0>(x, y, z, w, nsl, hl, sm.mom);
    gram_moments<S, 4, S::D2, 0, 0>(x, y, z, w, nsl, hl, sm.mom);
  }
  __syncwarp();
  // ---- L D L^T, the matrix in registers: a step updates the entries of later columns
  bool good = true;
  {
    double ge[S::NG];
    int ij[S::NG];
#pragma unroll
    for (int q = 0; q < S::NG; ++q) {
      const int e = __ldg(&tab.e[q * LN + hl]);
      ij[q] = e & 4095;
      ge[q] = sm.mom[e >> 12];
    }
    float mx = 0.f, mn = 3e38f;          // FP32 is enough for a bound a thousand times below what is seen
#pragma unroll 1
    for (int k = 0; k < M; ++k) {
      const int t = M - 1 - k, cnt = t * (t + 1) / 2;   // entries of the columns after k
#pragma unroll
      for (int q = 0; q < S::NG; ++q) {
        if (q * LN > cnt + t || q * LN + LN <= cnt) continue;
        const int e = q * LN + hl;
        if (e >= cnt && e <= cnt + t) sm.C[k + e - cnt] = ge[q];
      }
      __syncwarp();
      const double d = sm.C[k], rd = gram_rcp(d);
      const int8_t* ex = tab.ex[k];
      const float dr = (float)d * (float)(1 << (4 * (ex[0] + ex[1] + ex[2])));   // |R_kk|^2 around x_c
      mx = fmaxf(mx, dr);
      mn = fminf(mn, dr);
      good = good && dr > 0.f;
      if (hl == 0) sm.rd[k] = rd;
      for (int i = k + 1 + hl; i < M; i += LN) sm.L[k * S::LD + i] = sm.C[i] * rd;
      __syncwarp();
#pragma unroll
      for (int q = 0; q < S::NG; ++q) {
        if (q * LN >= cnt) continue;
        if (q * LN + hl < cnt) ge[q] = fma(-sm.L[k * S::LD + (ij[q] & 63)], sm.C[ij[q] >> 6], ge[q]);
      }
      __syncwarp();
    }
    good = good && mn >= 1e-6f * mx && mx < 1e38f;
  }
  if (active && !good) {
    if (hl == 0) fit_append(later, f);
    active = false;
  }
  if (!__any_sync(FULL, active)) return;
  // ---- targets: w ghosts and the normal derivative (n out of Omega+) at x_c
  double cz[NT][NZ];
  {
    int gm[3] = {lo % n, (lo / n) % n, DIM == 2 ? 0 : lo / n / n};
    const int step = lo_sig ? 1 : -1;
#pragma unroll
    for (int s = 0; s < NZ; ++s) {
      const int i = hl + LN * s;
      const bool in = i < M;
      int ex[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) ex[k] = in ? tab.ex[i][k] : 0;
#pragma unroll
      for (int t = 0; t < S::W; ++t) {
        double v = in ? 1.0 : 0.0;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          // the ghosts lie at most w nodes from the cell of x_c, well inside the window
          const int pos = gm[k] + (k == ax ? (lo_sig ? 1 : 0) + t * step : 0);
          const double xg = (sm.xi[k][pos - w0[k]] - mid[k]) * SC;
#pragma unroll
          for (int p = 0; p < S::q; ++p) v = p < ex[k] ? v * xg : v;
        }
        cz[t][s] = v;
      }
      double dn = 0.0;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        double v = in ? nrm[k] * (double)ex[k] : 0.0;
#pragma unroll
        for (int kk = 0; kk < DIM; ++kk) {
          const double x0 = -mid[kk] * SC;
#pragma unroll
          for (int p = 0; p < S::q; ++p) v = p < ex[kk] - (kk == k ? 1 : 0) ? v * x0 : v;
        }
        dn += v;
      }
      cz[S::W][s] = dn * (SC / g.h);
    }
  }
  // ---- s = V z, then one correction from the residual c - V^T s
  double zz[NT][NZ], sr[NT][S::SLOTS];
#pragma unroll
  for (int t = 0; t < NT; ++t)
#pragma unroll
    for (int s = 0; s < NZ; ++s) zz[t][s] = cz[t][s];
  auto put = [&]() {
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int s = 0; s < NZ; ++s)
        if (hl + LN * s < M) sm.z[t][hl + LN * s] = zz[t][s];
    __syncwarp();
  };
  gram_solve<S>(sm, zz, hl, base);
  put();
  gram_rows<S, false>(sm, x, y, z, m, hl, nsl, sr);
  __syncwarp();
  {
    // V^T s by z exponent: groups of (x, y) monomials [a][b], the targets inside (3D) or outside (2D)
    double* out = sm.mom;
    if constexpr (DIM == 3) {
      gram_project<S, 0>(x, y, z, sr, nsl, hl, out);
      gram_project<S, 1>(x, y, z, sr, nsl, hl, out + 45);
      gram_project<S, 2>(x, y, z, sr, nsl, hl, out + 75);
      gram_project<S, 3>(x, y, z, sr, nsl, hl, out + 93);
      gram_project<S, 4>(x, y, z, sr, nsl, hl, out + 102);
    } else {
      gram_project<S, 0>(x, y, z, sr, nsl, hl, out);
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < NZ; ++s) {
      const int i = hl + LN * s;
      if (i >= M) continue;
      const int a = tab.ex[i][0], b = tab.ex[i][1], cc = tab.ex[i][2];
      const int q1 = S::q - (DIM == 3 ? cc : 0) + 1;   // group cc: q1 (q1 + 1) / 2 pairs (a, b)
      const int off = DIM == 2 || cc == 0 ? 0 : (cc == 1 ? 45 : (cc == 2 ? 75 : (cc == 3 ? 93 : 102)));
      const int xy = a * q1 - a * (a - 1) / 2 + b;
#pragma unroll
      for (int t = 0; t < NT; ++t) zz[t][s] = cz[t][s] - (DIM == 3 ? out[off + xy * NT + t] : out[t * M + xy]);
    }
  }
  __syncwarp();
  gram_solve<S>(sm, zz, hl, base);
  put();
  gram_rows<S, true>(sm, x, y, z, m, hl, nsl, sr);
  // ---- outputs (same folding as k_fit)
  double* coef = P.fit_coef + (size_t)f * NT * P.rcap;
  double* cdat = P.fit_cdat + (size_t)f * NT;
  double s0[NT];                         // the control point's own coefficient of each row
#pragma unroll
  for (int t = 0; t < NT; ++t) s0[t] = __shfl_sync(FULL, sr[t][0], base);
  if (P.bc == IIM_BC_NEUMANN) {
    // u_c = (qbar - sum D_i u_i) / D_c with D = beta+ x derivative row (Eqs. 5-6)
    double s2 = 0.0;
#pragma unroll
    for (int s = 0; s < S::SLOTS; ++s) {
      if (s >= nsl) break;
      sr[S::W][s] *= P.beta_p;
      s2 = fma(sr[S::W][s], sr[S::W][s], s2);
    }
#pragma unroll
    for (int o = LN / 2; o > 0; o >>= 1) s2 += __shfl_xor_sync(FULL, s2, o);
    const double Dc = P.beta_p * s0[S::W];
    if (active && !(fabs(Dc) >= 1e-12 * sqrt(s2))) {
      if (hl == 0) set_status(P.status, IIM_ERR_SINGULAR);
      active = false;
    }
    if (!active) return;
    const double iDc = 1.0 / Dc;
#pragma unroll
    for (int s = 0; s < S::SLOTS; ++s) {
      if (s >= nsl) break;
      const double e = sr[S::W][s] * iDc;
#pragma unroll
      for (int t = 0; t < S::W; ++t) sr[t][s] = fma(-s0[t], e, sr[t][s]);
      sr[S::W][s] = -e;
    }
#pragma unroll
    for (int t = 0; t < S::W; ++t) s0[t] *= iDc;
    s0[S::W] = iDc;
  }
  if (!active) return;
#pragma unroll
  for (int s = 0; s < S::SLOTS; ++s) {
    const int al = LN * s + hl - 1;
    if (s >= nsl || al < 0 || al >= R) continue;
    const int code = sm.code[al];
#pragma unroll
    for (int t = 0; t < NT; ++t) coef[(size_t)t * P.rcap + al] = sr[t][s];
    P.fit_nodes[(size_t)f * P.rcap + al] =
        (w0[0] + (code & 31)) + n * ((w0[1] + ((code >> 5) & 31)) + (DIM == 2 ? 0 : n * (w0[DIM - 1] + (code >> 10))));
  }
  if (hl == 0) {
#pragma unroll
    for (int t = 0; t < NT; ++t) cdat[t] = s0[t];
    P.fit_R[f] = R;
  }
}

}  // namespace iim
