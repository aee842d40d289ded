// Matrix-free SIPG / BR2 operator y = A x on square meshes (Section 2, Eq.
// fe-problem; BR2 stabilisation of Section 4.4), FP64.
//
// As on cubes (apply3_kernel.cuh) the operator works in the orthonormal
// Legendre modes of each element, where mass and the face terms of same-size
// neighbours are diagonal and a larger side enters a hanging sub-face through
// one triangular restriction R.  Two kernels per apply:
//  modal2  x^ of every element, the traces u and a grad u . n of its four
//          sides in modes and, for every sub-face smaller than its side, both
//          traces restricted to it;
//  apply2  side residuals: same-size neighbours and the boundary mode by mode,
//          sub-faces of larger sides mode by mode on the sub-face and back
//          through R^T (BR2: the lifting R R^T J of the larger side, which its
//          smaller neighbour forms too); then along y and x the stiffness of
//          every line of modes plus the lift of its two side residuals, and the
//          transposed transform along x and y.
// An FP64 warp instruction takes its SM 19 cycles whatever its active lanes, so
// a tile is at most 32 lines of modes (32 / (p+1) elements of degree p), all of
// them taken by one warp, and at most 128 points on sides, one per thread of
// the CTA; the other three warps share the loads, the sides and the sub-faces.
// (A tile per warp, four to a CTA, was slower than the nodal kernel: 35 against
// 25 us on 98k unknowns, one warp working through all of a tile's sub-faces.)
// Records, items and tables are fetched before the wait for the preceding
// kernel: no kernel writes them.  Tiles come heaviest first.
// For large meshes (modal2_pays, which has both sides of its line); on smaller
// ones the chain of phases before the traces costs more than the operations that
// the modes save.  Measured (GB300), whole apply and mixed PCG iteration, nodal
// kernels / these: SIPG, degrees up to 8, 648k unknowns 102.8 / 72.7 and 285 /
// 255 us, 297k 53.1 / 43.8 and 162 / 153; degrees up to 6, 150k 29.5 / 24.6 and
// 89.9 / 89.8, 104k (nodal by the rule) 24.6 / 24.2; degrees up to 3, 176k 35.1 /
// 26.7 and 74.5 / 69.8; BR2, degrees up to 8, 648k 122.1 / 102.7 and 306 / 291.
// Every sub-face is evaluated from both of its sides and every sum has a fixed
// order: applies are bit-reproducible.
#pragma once

#include "modal.cuh"

namespace dg {

// shared doubles: work space (the sub-face items of a round: J, the residual and
// their two results; then the tile's residual in modes) and the kernels' totals
constexpr int kWork2 = 4 * kThreads3;
constexpr int modal2_doubles() {   // tables, modes, side traces
  int mx = 0;
  for (int p = 1; p <= kMaxP; ++p) {
    const int np = p + 1, e = apply2_epb(p), n = modal_table_doubles(p) + e * np * np + 8 * e * np;
    mx = n > mx ? n : mx;
  }
  return mx;
}
constexpr int apply2_doubles() {   // tables, modes, work space, side residuals r and c2
  int mx = 0;
  for (int p = 1; p <= kMaxP; ++p) {
    const int np = p + 1, e = apply2_epb(p), n = modal_table_doubles(p) + e * np * np + kWork2 + 8 * e * np;
    mx = n > mx ? n : mx;
  }
  return mx;
}
constexpr bool tile2_fits() {
  for (int p = 1; p <= kMaxP; ++p) {
    const int lines = apply2_epb(p) * (p + 1);
    if (lines > 32 || 4 * lines > kThreads3 || lines * (p + 1) > kWork2) return false;
  }
  return true;
}
static_assert(tile2_fits(), "a line per lane of a warp, a side point per thread, the residual in the work space");

// the start of modal2's shared memory: side traces, modes, then the tables
template <int P>
__device__ __forceinline__ double* modal2_table(double* sm) {
  return sm + 8 * apply2_epb(P) * (P + 1) + apply2_epb(P) * (P + 1) * (P + 1);
}
template <int P>
__device__ __forceinline__ void modal2_tables(const ApplyArgs& A, double* sm) {
  double* tab = modal2_table<P>(sm);
  for (int i = threadIdx.x; i < ModalTab<P>::SIZE; i += kThreads3) tab[i] = __ldg(A.tab + A.moff3[P] + i);
}

// Modes, side traces and restricted traces of one tile.  UPDATE (inside PCG):
// x is p, formed here as z + beta p (first: z) and stored.
template <int P, bool UPDATE>
__device__ __forceinline__ void modal2_tile(const ApplyArgs& A, const ApplyTile& T, const int4 hang, double* tb,
                                            double* p, const double* z, double beta, bool first) {
  using B = ModalTab<P>;
  constexpr int NP = P + 1, N2 = NP * NP;
  double2* st = reinterpret_cast<double2*>(tb);        // [cnt][4][NP] side traces
  double* sx = tb + 8 * apply2_epb(P) * NP;
  const double* tab = modal2_table<P>(tb);
  const double *E = tab, *O = tab + B::oO, *S = tab + B::oS, *Q = tab + B::oQ;
  const int tid = (int)threadIdx.x, cnt = T.count;
  const ElemRec3* er = A.erec3 + T.first;
  for (int t = tid; t < cnt * N2; t += kThreads3) {
    const int e = t / N2;
    const int64_t i = er[e].off + (t - e * N2);
    double v;
    if (UPDATE) {
      v = first ? z[i] : fma(beta, p[i], z[i]);
      p[i] = v;
    } else {
      v = __ldg(A.x + i);
    }
    sx[t] = v;
  }
  __syncthreads();
  const bool on = tid < cnt * NP;
  const int e = tid / NP, r = tid - e * NP;
  double v[NP];
  double2 lo, hi;
  if (on) {   // along y
    double* c = sx + e * N2 + r;
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = c[q * NP];
    line_to_modes<NP>(v, E, O);
#pragma unroll
    for (int q = 0; q < NP; ++q) c[q * NP] = v[q];
  }
  __syncthreads();
  if (on) {   // along x, with the traces of sides 0 and 1
    double* c = sx + e * N2 + r * NP;
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = c[q];
    line_to_modes<NP>(v, E, O);
#pragma unroll
    for (int q = 0; q < NP; ++q) c[q] = v[q];
    line_ends<NP>(v, S, Q, er[e].aih, lo, hi);
    st[4 * e * NP + r] = lo;
    st[(4 * e + 1) * NP + r] = hi;
  }
  __syncthreads();
  if (on) {   // sides 2 and 3
    const double* c = sx + e * N2 + r;
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = c[q * NP];
    line_ends<NP>(v, S, Q, er[e].aih, lo, hi);
    st[(4 * e + 2) * NP + r] = lo;
    st[(4 * e + 3) * NP + r] = hi;
  }
  __syncthreads();
  double2* tr = reinterpret_cast<double2*>(A.tr);
  if (tid < cnt * 4 * NP) {
    const int k = tid / (4 * NP);
    tr[er[k].toff + (tid - k * 4 * NP)] = st[tid];
  }
  for (int t = tid; t < cnt * N2; t += kThreads3) {
    const int k = t / N2;
    A.xm[er[k].off + (t - k * N2)] = sx[t];
  }
  for (int t = tid; t < hang.y * NP; t += kThreads3) {   // restricted to the sub-faces of larger sides
    const int it = t / NP, k = t - it * NP;
    const int2 hi2 = __ldg(A.hang2 + hang.x + it);
    const SubFaceModal2& f = A.sfm2[hi2.x];
    const double* R = A.tab + f.tab_r + k * kMaxN;
    const double2* src = st + hi2.y * NP;
    double u = 0.0, d = 0.0;
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      const double w = __ldg(R + m);   // zero for m < k
      u = fma(w, src[m].x, u);
      d = fma(w, src[m].y, d);
    }
    tr[f.own_off + k] = make_double2(u, d);
  }
}

// What a thread needs of its side point and of its item of the first round:
// fetched before the wait for the preceding kernel.
struct Side2 {
  int2 sd;           // as in side2; kSideSmaller without a point
  SubFaceModal2 f;   // whole sides
  int2 item;
  SubFaceModal2 g;   // the item's record
};
template <int P, bool BR2>
__device__ __forceinline__ void side2_fetch(const ApplyArgs& A, const ApplyTile& T, const int4 hang, Side2& s) {
  constexpr int NP = P + 1;
  const int W = BR2 ? hang.w : NP;
  const int tid = (int)threadIdx.x;
  s.sd = make_int2(0, kSideSmaller);
  if (tid < T.count * 4 * NP) s.sd = __ldg(A.side2 + (int64_t)T.first * 4 + tid / NP);
  if (s.sd.y == kSideWhole) s.f = A.sfm2[s.sd.x];
  if (tid / W < min(kThreads3 / W, BR2 ? hang.z : hang.y)) {
    s.item = __ldg(A.hang2 + hang.x + tid / W);
    s.g = A.sfm2[s.item.x];
  }
}

// r = cz (u- - u+) + cf F, the two traces multiplied one after the other: with
// the jump formed first the operator's rounding errors are antisymmetric
// between the two sides, and CG's counts drift from those of the assembled
// matrix where they depend on rounding (4,990 unknowns, eta = 10^4 without the
// block solves, forced into modes: 4,385 iterations against 4,648 nodal, 4,601
// this way).  The terms that need J itself - BR2's liftings - and the cubes' form
// it first: there the counts stay within 2.5% of the nodal operator's.
__device__ __forceinline__ double side_residual(double cz, double cf, double o, double n, double F) {
  return fma(-cz, n, fma(cz, o, cf * F));
}

// One tile; returns this thread's part of x . y.
template <int P, bool BR2>
__device__ __forceinline__ double apply2_tile(const ApplyArgs& A, const ApplyTile& T, const int4 hang, double* tab,
                                              const Side2& first) {
  using B = ModalTab<P>;
  constexpr int NP = P + 1, N2 = NP * NP, EPB = apply2_epb(P);
  const double *E = tab, *O = tab + B::oO, *K = tab + B::oK, *S = tab + B::oS, *Q = tab + B::oQ;
  double* sx = tab + B::SIZE;
  double* sg = sx + EPB * N2;
  double* sr = sg + kWork2;             // [cnt][4][NP] side residuals over a
  double* sc = sr + 4 * EPB * NP;       // [cnt][4][NP] normal-derivative coefficients over a
  const int tid = (int)threadIdx.x, cnt = T.count;
  const ElemRec3* er = A.erec3 + T.first;
  const double2* tr = reinterpret_cast<const double2*>(A.tr);
  for (int t = tid; t < cnt * N2; t += kThreads3) {
    const int e = t / N2;
    sx[t] = __ldg(A.xm + er[e].off + (t - e * N2));
  }
  // ---- same-size neighbours and the boundary: diagonal in modes
  const int sq = tid % NP;
  double rs = 0.0, cs = 0.0;
  if (first.sd.y == kSideWhole) {
    const SubFaceModal2& f = first.f;
    const double2 o = __ldg(tr + f.own_off + sq);
    const bool in = sq < f.nn;   // boundary: nn = 0
    const double2 n = in ? __ldg(tr + f.nbr_off + sq) : make_double2(0.0, 0.0);
    rs = side_residual(BR2 && in ? f.cx : f.cz, f.cf, o.x, n.x, o.y - n.y);   // n.y: the neighbour's outward dn
    cs = f.cc * (o.x - n.x);
  }
  // ---- sub-faces between a larger and a smaller side, in rounds.  SIPG: those
  // of larger sides (to a smaller side they are diagonal, above); BR2: then
  // those of smaller sides, which need the neighbour's lifting
  const int W = BR2 ? hang.w : NP;      // modes of J: BR2 takes the neighbour's too
  const int ROUND = kThreads3 / W;      // one mode per thread
  double *sJ = sg, *sF = sJ + kThreads3, *s1 = sF + kThreads3, *s2 = s1 + kThreads3;
  const int n_hang = BR2 ? hang.z : hang.y;
  for (int h0 = 0; h0 < n_hang; h0 += ROUND) {
    const int n = min(ROUND, n_hang - h0);
    const int it = tid / W, q = tid - it * W;
    const bool has = it < n, big = h0 + it < hang.y;
    int2 item = first.item;
    SubFaceModal2 f = first.g;
    if (has && h0 > 0) {
      item = __ldg(A.hang2 + hang.x + h0 + it);
      f = A.sfm2[item.x];
    }
    double J = 0.0, R0 = 0.0;
    if (has) {
      double2 o = make_double2(0.0, 0.0), v = o;
      if (q < NP) o = __ldg(tr + f.own_off + q);
      const bool in = q < f.nn;
      if (in) v = __ldg(tr + f.nbr_off + q);
      J = o.x - v.x;
      // the diagonal part; BR2: all but the larger side's lifting
      if (BR2 && big) R0 = in ? fma(f.cx, J, f.cf * (o.y - v.y)) : f.cf * (o.y - v.y);
      else R0 = side_residual(f.cz, f.cf, o.x, v.x, o.y - v.y);
      sJ[tid] = J;
      sF[tid] = R0;
    }
    __syncthreads();
    const double* R = A.tab + f.tab_r;
    double a = 0.0, b = 0.0;
    if (BR2) {   // t = R^T J, J in the modes the larger side has
      const int nr = big ? NP : f.nn;
      if (has && q < nr)
        for (int k = 0; k <= q; ++k) b = fma(__ldg(R + k * kMaxN + q), sJ[it * W + k], b);
      if (has) s2[tid] = b;
      __syncthreads();
      if (has && q < NP) {   // the lifting R t
        double l = 0.0;
        for (int m = q; m < nr; ++m) l = fma(__ldg(R + q * kMaxN + m), s2[it * W + m], l);
        R0 = fma(big ? f.cz : f.cx, l, R0);
        sF[tid] = R0;
      }
      __syncthreads();
    }
    if (BR2 && has && !big) {   // a smaller side: its only sub-face
      if (q < NP) {
        sr[item.y * NP + q] = R0;
        sc[item.y * NP + q] = f.cc * J;
      }
    } else if (has && q < NP) {   // back to the side's modes
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const double w = __ldg(R + k * kMaxN + q);   // zero for k > q
        a = fma(w, sF[it * W + k], a);
        if (!BR2) b = fma(w, sJ[it * W + k], b);
      }
      s1[tid] = a;
      s2[tid] = f.cc * b;
    }
    __syncthreads();
    if (first.sd.y > 0) {   // larger sides: their sub-faces in order
      const int g1 = min(first.sd.x + first.sd.y, h0 + n);
      for (int g = max(first.sd.x, h0); g < g1; ++g) {
        rs += s1[(g - h0) * W + sq];
        cs += s2[(g - h0) * W + sq];
      }
    }
    __syncthreads();
  }
  if (first.sd.y != kSideSmaller) {
    sr[tid] = rs;
    sc[tid] = cs;
  }
  __syncthreads();
  // ---- volume and lift, one lane of a warp per line of modes
  const bool on = tid < cnt * NP;
  const int e = tid / NP, r = tid - e * NP;
  double v[NP], g[NP], part = 0.0;
  if (tid >= 32) return 0.0;   // one warp from here on
  if (on) {   // along y
    const double* c = sx + e * N2 + r;
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = c[q * NP];
    line_stiffness<NP, false>(v, g, K);
    const int f = (4 * e + 2) * NP + r;
    line_lift<NP>(g, S, Q, sr[f], sr[f + NP], sc[f], sc[f + NP]);
#pragma unroll
    for (int q = 0; q < NP; ++q) sg[e * N2 + r + q * NP] = g[q];
  }
  __syncwarp();
  if (on) {   // along x: x . y, then back to nodes
    const double* c = sx + e * N2 + r * NP;
    double* d = sg + e * N2 + r * NP;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      v[q] = c[q];
      g[q] = d[q];
    }
    line_stiffness<NP, true>(v, g, K);
    const int f = 4 * e * NP + r;
    line_lift<NP>(g, S, Q, sr[f], sr[f + NP], sc[f], sc[f + NP]);
    if (A.dot_partial) {
      double dot = v[0] * g[0];
#pragma unroll
      for (int q = 1; q < NP; ++q) dot = fma(v[q], g[q], dot);
      part = er[e].ah * dot;
    }
    line_to_nodes<NP>(g, E, O);
#pragma unroll
    for (int q = 0; q < NP; ++q) d[q] = g[q];
  }
  __syncwarp();
  if (on) {   // along y
    const double* d = sg + e * N2 + r;
#pragma unroll
    for (int q = 0; q < NP; ++q) g[q] = d[q * NP];
    line_to_nodes<NP>(g, E, O);
    double* y = A.y + er[e].off + r;
    const double ah = er[e].ah;
#pragma unroll
    for (int q = 0; q < NP; ++q) y[q * NP] = ah * g[q];
  }
  return part;
}

}  // namespace dg
