// Matrix-free SIPG / BR2 operator y = A x on cube meshes (the method of
// Section 2 on hexahedra; BR2 stabilisation of Section 4.4), FP64.
//
// The part issues one FP64 warp instruction per SM every 19 cycles (1.06
// TFLOP/s measured), so FP64 operations are what an apply costs and loads,
// barriers and index arithmetic are nearly free beside them.  The operator
// therefore works in the element's orthonormal Legendre basis phi_k =
// sqrt(2k+1) P_k on [0, 1] per direction (x = V x^, the transform exact up to
// rounding), where
//   - the 1D mass matrix is the identity and the 1D stiffness couples modes
//     of one parity only;
//   - two touching whole faces share their basis: the face-mass matrices and
//     the BR2 lifting products are diagonal, whatever the two degrees;
//   - on a hanging sub-face the larger side's trace enters through the
//     restriction R of its modes to the sub-interval, one triangular matrix
//     per position whatever the degree;
//   - the nodes' mirror symmetry and the modes' parity halve the transforms
//     and the traces of opposite faces (sums and differences of node pairs).
// Two kernels per apply:
//  modal3  x^ of every element, the traces u and a grad u . n of its six sides
//          in modes and, on the sides with smaller neighbours, their
//          restriction to every sub-face (formed once for both sides' use);
//  apply3  one CTA per tile of elements of one degree P:
//    faces   whole sides point by point in modes; a side with smaller
//            neighbours per sub-face (J = jump, F = flux in the sub-face's
//            modes, back through R^T; BR2's own lifting through S = R R^T);
//            BR2's neighbour lifting on sub-faces of a larger neighbour
//            through its S;
//    volume  per line of modes K x^ plus the lift of the two side residuals,
//            along z, y, x; then the transposed transform along x, y, z.
// On the 16^3 hp-random workload (1.7M unknowns, BR2) FP64 operations per
// apply fell from 219 M to 128 M FMA-sized ones against the nodal form
// with its face-mass products.
// Each sub-face is evaluated from both of its sides (no atomics): applies are
// bit-reproducible.
#pragma once

#include "apply_kernel.cuh"

namespace dg {

// One line of NP values between nodes and modes.  E: even modes x (sums of
// mirrored nodes, then the middle node), O: odd modes x differences.
template <int NP>
__device__ __forceinline__ void line_to_modes(double (&v)[NP], const double* E, const double* O) {
  constexpr int H = NP / 2, HC = (NP + 1) / 2;
  double s[HC], d[H];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    s[i] = v[i] + v[NP - 1 - i];
    d[i] = v[i] - v[NP - 1 - i];
  }
  if (NP & 1) s[HC - 1] = v[H];
#pragma unroll
  for (int a = 0; a < HC; ++a) {
    double t = E[a * HC] * s[0];
#pragma unroll
    for (int i = 1; i < HC; ++i) t = fma(E[a * HC + i], s[i], t);
    v[2 * a] = t;
  }
#pragma unroll
  for (int a = 0; a < H; ++a) {
    double t = O[a * H] * d[0];
#pragma unroll
    for (int i = 1; i < H; ++i) t = fma(O[a * H + i], d[i], t);
    v[2 * a + 1] = t;
  }
}
// the transposed transform: node values of the residual from its modes
template <int NP>
__device__ __forceinline__ void line_to_nodes(double (&v)[NP], const double* E, const double* O) {
  constexpr int H = NP / 2, HC = (NP + 1) / 2;
  double ev[HC], od[H];
#pragma unroll
  for (int i = 0; i < HC; ++i) {
    ev[i] = E[i] * v[0];
#pragma unroll
    for (int a = 1; a < HC; ++a) ev[i] = fma(E[a * HC + i], v[2 * a], ev[i]);
  }
#pragma unroll
  for (int i = 0; i < H; ++i) {
    od[i] = O[i] * v[1];
#pragma unroll
    for (int a = 1; a < H; ++a) od[i] = fma(O[a * H + i], v[2 * a + 1], od[i]);
  }
#pragma unroll
  for (int i = 0; i < H; ++i) {
    v[i] = ev[i] + od[i];
    v[NP - 1 - i] = ev[i] - od[i];
  }
  if (NP & 1) v[H] = ev[HC - 1];
}
// values and outward normal derivatives (times h / a) at both ends of a line
template <int NP>
__device__ __forceinline__ void line_ends(const double (&v)[NP], const double* s, const double* q, double aih,
                                          double2& lo, double2& hi) {
  double ev = v[0], od = s[1] * v[1], de = 0.0, dodd = q[1] * v[1];   // phi_0 = 1
#pragma unroll
  for (int k = 2; k < NP; ++k) {
    if (k & 1) {
      od = fma(s[k], v[k], od);
      dodd = fma(q[k], v[k], dodd);
    } else {
      ev = fma(s[k], v[k], ev);
      de = k == 2 ? q[k] * v[k] : fma(q[k], v[k], de);
    }
  }
  hi = make_double2(ev + od, NP > 2 ? aih * (de + dodd) : aih * dodd);
  lo = make_double2(ev - od, NP > 2 ? aih * (de - dodd) : -aih * dodd);
}
// g += K v (same-parity modes, K_0m = 0)
template <int NP, bool ADD>
__device__ __forceinline__ void line_stiffness(const double (&v)[NP], double (&g)[NP], const double* K) {
  if (!ADD) g[0] = 0.0;
#pragma unroll
  for (int k = 1; k < NP; ++k) {
    double t = ADD ? g[k] : 0.0;
#pragma unroll
    for (int m = 2 - (k & 1); m < NP; m += 2) t = (!ADD && m <= 2) ? K[k * NP + m] * v[m] : fma(K[k * NP + m], v[m], t);
    g[k] = t;
  }
}
// g += value and normal-derivative test functions times the residuals of the
// two end faces
template <int NP>
__device__ __forceinline__ void line_lift(double (&g)[NP], const double* s, const double* q, double r0, double r1,
                                          double c0, double c1) {
  const double rp = r1 + r0, rm = r1 - r0, cp = c1 + c0, cm = c1 - c0;
  g[0] += rp;
#pragma unroll
  for (int k = 1; k < NP; ++k)
    g[k] = (k & 1) ? fma(s[k], rm, fma(q[k], cm, g[k])) : fma(s[k], rp, fma(q[k], cp, g[k]));
}

// shared copy of a degree's modal tables
template <int P>
struct Modal3 {
  static constexpr int NP = P + 1, H = NP / 2, HC = (NP + 1) / 2;
  static constexpr int oO = HC * HC, oK = oO + H * H, oS = oK + NP * NP, oQ = oS + NP;
  static constexpr int SIZE = oQ + NP;
};

// Modes and traces of one tile.  UPDATE (inside PCG): x is p, formed here as
// z + beta p (first: z) and stored.
template <int P, bool UPDATE>
__device__ __forceinline__ void modal3_tile(const ApplyArgs& A, const ApplyTile& T, double* sm, double* p,
                                            const double* z, double beta, bool first) {
  using B = Modal3<P>;
  constexpr int NP = P + 1, N2 = NP * NP, N3 = N2 * NP;
  double* tb = sm;
  double* sx = tb + B::SIZE;
  double* sy = sx + T.count * N3;   // [cap_c][2][N2]: half-restricted traces
  const double *E = tb, *O = tb + B::oO, *S = tb + B::oS, *Q = tb + B::oQ;
  const int tid = threadIdx.x, nl = T.count * N2;
  for (int i = tid; i < B::SIZE; i += kThreads3) tb[i] = __ldg(A.tab + A.moff3[P] + i);
  const ElemRec3* er = A.erec3 + T.first;
  for (int t = tid; t < T.count * N3; t += kThreads3) {
    const int e = t / N3;
    const int64_t i = er[e].off + (t - e * N3);
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
  double v[NP];
  auto along = [&](int base, int st) {
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = sx[base + q * st];
    line_to_modes<NP>(v, E, O);
#pragma unroll
    for (int q = 0; q < NP; ++q) sx[base + q * st] = v[q];
  };
  for (int l = tid; l < nl; l += kThreads3) {
    const int e = l / N2, r = l - e * N2;
    along(e * N3 + r, N2);
  }
  __syncthreads();
  for (int l = tid; l < nl; l += kThreads3) {
    const int e = l / N2, r = l - e * N2;
    along(e * N3 + (r / NP) * N2 + r % NP, NP);
  }
  __syncthreads();
  double2* tr = reinterpret_cast<double2*>(A.tr);
  for (int l = tid; l < nl; l += kThreads3) {   // along x, with the traces of sides 0 and 1
    const int e = l / N2, r = l - e * N2;
    along(e * N3 + r * NP, 1);
    double2 lo, hi;
    line_ends<NP>(v, S, Q, er[e].aih, lo, hi);
    double2* te = tr + er[e].toff + r;
    te[0] = lo;
    te[N2] = hi;
  }
  __syncthreads();
  for (int l = tid; l < 2 * nl; l += kThreads3) {   // sides 2..5; node = the two tangential modes
    const int ax = l < nl ? 0 : 1, m = l - ax * nl;
    const int e = m / N2, r = m - e * N2;
    const int base = ax == 0 ? e * N3 + (r / NP) * N2 + r % NP : e * N3 + r, st = ax == 0 ? NP : N2;
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = sx[base + q * st];
    double2 lo, hi;
    line_ends<NP>(v, S, Q, er[e].aih, lo, hi);
    double2* te = tr + er[e].toff + (2 + 2 * ax) * N2 + r;
    te[0] = lo;
    te[N2] = hi;
  }
  for (int t = tid; t < T.count * N3; t += kThreads3) {
    const int e = t / N3;
    A.xm[er[e].off + (t - e * N3)] = sx[t];
  }
  // sides with smaller neighbours: u and dn restricted to each sub-face,
  // R_a (x) R_b, one thread per line of one of the two quantities
  const int2* hang = A.hang3 + T.hang;
  for (int c0 = 0; c0 < T.n_c; c0 += T.cap_c) {
    const int nc = min(T.cap_c, T.n_c - c0);
    __syncthreads();   // the traces above (and the last round's scratch)
    for (int t = tid; t < nc * 2 * NP; t += kThreads3) {
      const int it = t / (2 * NP), rem = t - it * 2 * NP;
      const int w = rem / NP, n = rem - w * NP;
      const int2 hg = hang[c0 + it];
      const SubFaceModal3& f = A.sfm3[hg.x];
      const int e = hg.y / 6, s = hg.y - e * 6;
      const double* src = reinterpret_cast<const double*>(tr + er[e].toff + s * N2 + n * NP) + w;
#pragma unroll
      for (int q = 0; q < NP; ++q) v[q] = src[2 * q];
      const double* R = A.tab + f.tab_ra;
      double* dst = sy + (it * 2 + w) * N2 + n * NP;
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        double a = __ldg(R + k * kMaxN + k) * v[k];
#pragma unroll
        for (int m = k + 1; m < NP; ++m) a = fma(__ldg(R + k * kMaxN + m), v[m], a);
        dst[k] = a;
      }
    }
    __syncthreads();
    for (int t = tid; t < nc * 2 * NP; t += kThreads3) {
      const int it = t / (2 * NP), rem = t - it * 2 * NP;
      const int w = rem / NP, i = rem - w * NP;
      const SubFaceModal3& f = A.sfm3[hang[c0 + it].x];
      const double* src = sy + (it * 2 + w) * N2 + i;
#pragma unroll
      for (int q = 0; q < NP; ++q) v[q] = src[q * NP];
      const double* R = A.tab + f.tab_rb;
      double* dst = reinterpret_cast<double*>(tr + f.own_off + i) + w;
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        double a = __ldg(R + k * kMaxN + k) * v[k];
#pragma unroll
        for (int m = k + 1; m < NP; ++m) a = fma(__ldg(R + k * kMaxN + m), v[m], a);
        dst[2 * k * NP] = a;
      }
    }
  }
}

template <int P, bool BR2>
__device__ __forceinline__ void apply3_tile(const ApplyArgs& A, const ApplyTile& T, int tile, double* sm,
                                            double* red) {
  using B = Modal3<P>;
  constexpr int NP = P + 1, N2 = NP * NP, N3 = N2 * NP;
  const int cnt = T.count, nl = cnt * N2, NQ = T.nq;
  double* tb = sm;
  double* sx = tb + B::SIZE;
  double* sg = sx + cnt * N3;
  double* sr = sg + cnt * N3;              // [cnt][6][N2] side residuals over a h
  double* sc = sr + cnt * 6 * N2;          // [cnt][6][N2] normal-derivative coefficients over a h
  double* sw = sc + cnt * 6 * N2;          // larger sides' sub-faces: [cap_c][4][N2]
  double* sb = sw + T.cap_c * 4 * N2;      // BR2, larger neighbours: [cap_b][NQ * NQ + NP * NQ]
  const double *E = tb, *O = tb + B::oO, *K = tb + B::oK, *S = tb + B::oS, *Q = tb + B::oQ;
  const int tid = threadIdx.x;
  const double2* tr = reinterpret_cast<const double2*>(A.tr);
  const ElemRec3* er = A.erec3 + T.first;
  for (int i = tid; i < B::SIZE; i += kThreads3) tb[i] = __ldg(A.tab + A.moff3[P] + i);
  for (int t = tid; t < cnt * N3; t += kThreads3) {
    const int e = t / N3;
    sx[t] = __ldg(A.xm + er[e].off + (t - e * N3));
  }
  // ---- whole sides (same-size neighbour, boundary, or a sub-face of a larger
  // neighbour, whose restricted trace is in place): diagonal in modes
  for (int t = tid; t < cnt * 6 * N2; t += kThreads3) {
    const int es = t / N2, q = t - es * N2;
    const int4 sd = __ldg(A.side3 + (int64_t)T.first * 6 + es);   // {record, first sub-face, sub-faces}
    double r = 0.0, c = 0.0;
    if (sd.z == 0) {
      const SubFaceModal3& f = A.sfm3[sd.x];
      const int i = q % NP, j = q / NP, npn = f.pn + 1;
      const double2 o = __ldg(tr + f.own_off + q);
      double J = o.x, F = o.y;
      const bool in = f.nb >= 0 && i < npn && j < npn;
      if (in) {
        const double2 n = __ldg(tr + f.nbr_off + j * npn + i);
        J -= n.x;
        F -= n.y;   // the neighbour's outward dn
      }
      r = fma(BR2 && in ? f.czx : f.cz, J, f.cf * F);
      c = f.cc * J;
    }
    sr[t] = r;
    sc[t] = c;
  }
  // ---- sub-faces smaller than the own side (C) and, for BR2, sub-faces of a
  // larger neighbour (its lifting), in rounds that fit the scratch
  const int2* hang = A.hang3 + T.hang;
  const int n_b = BR2 ? T.n_b : 0;
  for (int c0 = 0, b0 = 0; c0 < T.n_c || b0 < n_b; c0 += T.cap_c, b0 += T.cap_b) {
    const int nc = max(0, min(T.cap_c, T.n_c - c0)), nb = max(0, min(T.cap_b, n_b - b0));
    for (int t = tid; t < nc * N2; t += kThreads3) {   // J and the point-by-point residual
      const int it = t / N2, q = t - it * N2;
      const SubFaceModal3& f = A.sfm3[hang[c0 + it].x];
      const int i = q % NP, j = q / NP, npn = f.pn + 1;
      const double2 o = __ldg(tr + f.own_off + q);
      double J = o.x, F = o.y;
      const bool in = i < npn && j < npn;
      if (in) {
        const double2 n = __ldg(tr + f.nbr_off + j * npn + i);
        J -= n.x;
        F -= n.y;
      }
      double* X = sw + it * 4 * N2;
      X[q] = J;
      X[N2 + q] = BR2 ? (in ? fma(f.cx, J, f.cf * F) : f.cf * F) : fma(f.cz, J, f.cf * F);
    }
    for (int t = tid; t < nb * NQ * NQ; t += kThreads3) {   // J in the larger neighbour's modes
      const int it = t / (NQ * NQ), q = t - it * NQ * NQ;
      const SubFaceModal3& f = A.sfm3[hang[T.n_c + b0 + it].x];
      const int i = q % NQ, j = q / NQ, npn = f.pn + 1;
      if (i < npn && j < npn) {
        double J = -__ldg(tr + f.nbr_off + j * npn + i).x;
        if (i < NP && j < NP) J += __ldg(tr + f.own_off + j * NP + i).x;
        sb[it * (NQ * NQ + NP * NQ) + j * NQ + i] = J;
      }
    }
    __syncthreads();
    // first tangential axis: R^T J, and S J (BR2) or R^T of the residual
    for (int t = tid; t < nc * 2 * NP; t += kThreads3) {
      const int it = t / (2 * NP), rem = t - it * 2 * NP;
      const int w = rem / NP, n = rem - w * NP;
      const SubFaceModal3& f = A.sfm3[hang[c0 + it].x];
      const double* X = sw + it * 4 * N2 + (BR2 ? 0 : w) * N2 + n * NP;
      double* Y = sw + it * 4 * N2 + (2 + w) * N2 + n * NP;
      double v[NP];
#pragma unroll
      for (int q = 0; q < NP; ++q) v[q] = X[q];
      if (BR2 && w == 1) {
        const double* Sa = A.tab + f.tab_sa;
#pragma unroll
        for (int m = 0; m < NP; ++m) {
          double a = __ldg(Sa + m * NP) * v[0];
#pragma unroll
          for (int k = 1; k < NP; ++k) a = fma(__ldg(Sa + m * NP + k), v[k], a);
          Y[m] = a;
        }
      } else {
        const double* R = A.tab + f.tab_ra;
#pragma unroll
        for (int m = 0; m < NP; ++m) {
          double a = __ldg(R + m) * v[0];
#pragma unroll
          for (int k = 1; k <= m; ++k) a = fma(__ldg(R + k * kMaxN + m), v[k], a);
          Y[m] = a;
        }
      }
    }
    for (int t = tid; t < nb * NP * NQ; t += kThreads3) {
      const int it = t / (NP * NQ), rem = t - it * NP * NQ;
      const int i = rem % NP, n = rem / NP;
      const SubFaceModal3& f = A.sfm3[hang[T.n_c + b0 + it].x];
      const int npn = f.pn + 1;
      double* X = sb + it * (NQ * NQ + NP * NQ);
      if (i < npn && n < npn) {
        const double* Sa = A.tab + f.tab_sa + i * npn;
        double a = 0.0;
        for (int m = 0; m < npn; ++m) a = fma(__ldg(Sa + m), X[n * NQ + m], a);
        X[NQ * NQ + n * NP + i] = a;
      }
    }
    __syncthreads();
    // second tangential axis
    for (int t = tid; t < nc * 2 * NP; t += kThreads3) {
      const int it = t / (2 * NP), rem = t - it * 2 * NP;
      const int w = rem / NP, i = rem - w * NP;
      const SubFaceModal3& f = A.sfm3[hang[c0 + it].x];
      const double* Y = sw + it * 4 * N2 + (2 + w) * N2 + i;
      double* X = sw + it * 4 * N2 + w * N2 + i;
      double v[NP];
#pragma unroll
      for (int q = 0; q < NP; ++q) v[q] = Y[q * NP];
      if (BR2 && w == 1) {
        const double* Sb = A.tab + f.tab_sb;
#pragma unroll
        for (int m = 0; m < NP; ++m) {
          double a = __ldg(Sb + m * NP) * v[0];
#pragma unroll
          for (int k = 1; k < NP; ++k) a = fma(__ldg(Sb + m * NP + k), v[k], a);
          X[m * NP] = fma(f.cz, a, X[m * NP]);
        }
      } else {
        const double* R = A.tab + f.tab_rb;
#pragma unroll
        for (int m = 0; m < NP; ++m) {
          double a = __ldg(R + m) * v[0];
#pragma unroll
          for (int k = 1; k <= m; ++k) a = fma(__ldg(R + k * kMaxN + m), v[k], a);
          X[m * NP] = w == 0 ? f.cc * a : a;
        }
      }
    }
    for (int t = tid; t < nb * N2; t += kThreads3) {
      const int it = t / N2, q = t - it * N2;
      const int i = q % NP, j = q / NP;
      const int2 hg = hang[T.n_c + b0 + it];
      const SubFaceModal3& f = A.sfm3[hg.x];
      const int npn = f.pn + 1;
      if (i < npn && j < npn) {
        const double* Sb = A.tab + f.tab_sb + j * npn;
        const double* Y = sb + it * (NQ * NQ + NP * NQ) + NQ * NQ + i;
        double a = 0.0;
        for (int n = 0; n < npn; ++n) a = fma(__ldg(Sb + n), Y[n * NP], a);
        sr[hg.y * N2 + q] = fma(f.cx, a, sr[hg.y * N2 + q]);
      }
    }
    if (BR2) {   // back through R^T, after the own lifting joined the residual
#pragma unroll
      for (int ax = 0; ax < 2; ++ax) {
        __syncthreads();
        for (int t = tid; t < nc * NP; t += kThreads3) {
          const int it = t / NP, n = t - it * NP;
          const SubFaceModal3& f = A.sfm3[hang[c0 + it].x];
          double* X = sw + it * 4 * N2 + N2;
          const double* src = ax == 0 ? X + n * NP : X + N2 + n;
          double* dst = ax == 0 ? X + N2 + n * NP : X + n;
          const int st = ax == 0 ? 1 : NP;
          double v[NP];
#pragma unroll
          for (int q = 0; q < NP; ++q) v[q] = src[q * st];
          const double* R = A.tab + (ax == 0 ? f.tab_ra : f.tab_rb);
#pragma unroll
          for (int m = 0; m < NP; ++m) {
            double a = __ldg(R + m) * v[0];
#pragma unroll
            for (int k = 1; k <= m; ++k) a = fma(__ldg(R + k * kMaxN + m), v[k], a);
            dst[m * st] = a;
          }
        }
      }
    }
    __syncthreads();
    // every mode of a side adds its sub-faces of this round, in order
    if (nc > 0)
      for (int t = tid; t < cnt * 6 * N2; t += kThreads3) {
        const int es = t / N2, q = t - es * N2;
        const int4 sd = __ldg(A.side3 + (int64_t)T.first * 6 + es);
        const int lo = max(sd.y, c0), hi = min(sd.y + sd.z, c0 + nc);
        if (lo < hi) {
          double r = sr[t], c = sc[t];
          for (int g = lo; g < hi; ++g) {
            const double* X = sw + (g - c0) * 4 * N2 + q;
            c += X[0];
            r += X[N2];
          }
          sr[t] = r;
          sc[t] = c;
        }
      }
    __syncthreads();
  }
  __syncthreads();
  // ---- volume and lift, one thread per line of modes
  double v[NP], g[NP];
  auto line = [&](int ax, int e, int base, int st, int r) {
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = sx[base + q * st];
    if (ax == 2) {
      line_stiffness<NP, false>(v, g, K);
    } else {
#pragma unroll
      for (int q = 0; q < NP; ++q) g[q] = sg[base + q * st];
      line_stiffness<NP, true>(v, g, K);
    }
    const int f = (e * 6 + 2 * ax) * N2 + r;
    line_lift<NP>(g, S, Q, sr[f], sr[f + N2], sc[f], sc[f + N2]);
  };
  for (int l = tid; l < nl; l += kThreads3) {   // along z
    const int e = l / N2, r = l - e * N2, base = e * N3 + r;
    line(2, e, base, N2, r);
#pragma unroll
    for (int q = 0; q < NP; ++q) sg[base + q * N2] = g[q];
  }
  __syncthreads();
  for (int l = tid; l < nl; l += kThreads3) {   // along y
    const int e = l / N2, r = l - e * N2, base = e * N3 + (r / NP) * N2 + r % NP;
    line(1, e, base, NP, r);
#pragma unroll
    for (int q = 0; q < NP; ++q) sg[base + q * NP] = g[q];
  }
  __syncthreads();
  double part = 0.0;
  for (int l = tid; l < nl; l += kThreads3) {   // along x: x . y, then back to nodes
    const int e = l / N2, r = l - e * N2, base = e * N3 + r * NP;
    line(0, e, base, 1, r);
    if (A.dot_partial) {
      double d = v[0] * g[0];
#pragma unroll
      for (int q = 1; q < NP; ++q) d = fma(v[q], g[q], d);
      part = fma(er[e].ah, d, part);
    }
    line_to_nodes<NP>(g, E, O);
#pragma unroll
    for (int q = 0; q < NP; ++q) sg[base + q] = g[q];
  }
  __syncthreads();
  for (int l = tid; l < nl; l += kThreads3) {
    const int e = l / N2, r = l - e * N2, base = e * N3 + (r / NP) * N2 + r % NP;
#pragma unroll
    for (int q = 0; q < NP; ++q) g[q] = sg[base + q * NP];
    line_to_nodes<NP>(g, E, O);
#pragma unroll
    for (int q = 0; q < NP; ++q) sg[base + q * NP] = g[q];
  }
  __syncthreads();
  for (int l = tid; l < nl; l += kThreads3) {
    const int e = l / N2, r = l - e * N2, base = e * N3 + r;
#pragma unroll
    for (int q = 0; q < NP; ++q) g[q] = sg[base + q * N2];
    line_to_nodes<NP>(g, E, O);
    double* y = A.y + er[e].off + r;
    const double ah = er[e].ah;
#pragma unroll
    for (int q = 0; q < NP; ++q) y[q * N2] = ah * g[q];
  }
  if (A.dot_partial) {
    // tile partial of x . y (summed in tile order when the launch ends)
    const double tot = block_sum<kThreads3>(part, red);
    if (tid == 0) A.dot_partial[tile] = tot;
  }
}

}  // namespace dg
