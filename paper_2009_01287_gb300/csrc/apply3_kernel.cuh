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
// Three kernels per apply:
//  modal3  x^ of every element and the traces u and a grad u . n of its six
//          sides in modes;
//  hang3   per sub-face between a larger and a smaller side (a pair): the
//          larger side's traces restricted by R, J = jump and F = flux, and
//          the residuals of both sides, the larger side's back through R^T.
//          BR2's lifting on the larger side, R R^T J, serves both sides.  Its
//          own kernel, because an element can have anything from none to
//          dozens of them: taken inside the element's tile they made the
//          heaviest tile four times the mean and the SMs 54% busy on average;
//  apply3  one CTA per tile of elements of one degree P: side residuals point
//          by point in modes (same-size neighbours and the boundary) or summed
//          from the pairs' in order; then per line of modes K x^ plus the lift
//          of the two side residuals, along z, y, x, and the transposed
//          transform along x, y, z.
// Measured (GB300), apply of the 16^3 hp-random workload (1.7M unknowns, BR2):
// 689 us in nodal form with face-mass products, 350 in modes with the hanging
// sub-faces inside the tiles, 272 with their own kernel; 79k unknowns, SIPG,
// 62.8 / 48.6 / 33.0 us.  The FP64 operations alone (216.1 Mflop) are 0.204 ms
// on the large one at the measured 1.06 TFLOP/s.
// Every sum has a fixed order and there are no atomics on data: applies are
// bit-reproducible.
#pragma once

#include "modal.cuh"

namespace dg {

// Modes and traces of one tile.  UPDATE (inside PCG): x is p, formed here as
// z + beta p (first: z) and stored.
template <int P, bool UPDATE>
__device__ __forceinline__ void modal3_tile(const ApplyArgs& A, const ApplyTile& T, double* sm, double* p,
                                            const double* z, double beta, bool first) {
  using B = ModalTab<P>;
  constexpr int NP = P + 1, N2 = NP * NP, N3 = N2 * NP;
  double* tb = sm;
  double* sx = tb + B::SIZE;
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
}

// one line times R, upper triangular, or R^T
template <int NP>
__device__ __forceinline__ void line_restrict(const double (&v)[NP], double (&o)[NP], const double* R) {
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    double a = __ldg(R + k * kMaxN + k) * v[k];
#pragma unroll
    for (int m = k + 1; m < NP; ++m) a = fma(__ldg(R + k * kMaxN + m), v[m], a);
    o[k] = a;
  }
}
template <int NP>
__device__ __forceinline__ void line_restrict_t(const double (&v)[NP], double (&o)[NP], const double* R) {
#pragma unroll
  for (int m = 0; m < NP; ++m) {
    double a = __ldg(R + m) * v[0];
#pragma unroll
    for (int k = 1; k <= m; ++k) a = fma(__ldg(R + k * kMaxN + m), v[k], a);
    o[m] = a;
  }
}

// The hanging pairs of one tile (one degree P of the larger side).  Residuals
// over a h and normal-derivative coefficients over a h of either side go to
// the results part of the trace buffer.
template <int P, bool BR2>
__device__ __forceinline__ void hang3_tile(const ApplyArgs& A, const HangTile& T, double* sm) {
  constexpr int NP = P + 1, N2 = NP * NP;
  const int cnt = T.count, NS = T.ns, NM = NP > NS ? NP : NS;
  double* sX = sm;                    // [cnt][2][N2]: restricted u, dn; then J, residual
  double* sY = sX + cnt * 2 * N2;     // [cnt][2][N2]: half-way products
  const int tid = threadIdx.x;
  const HangPair* hp = A.hang3 + T.first;
  double2* tr = reinterpret_cast<double2*>(A.tr);
  const double* trd = A.tr;
  double v[NP], o[NP];
  auto load = [&](const double* p, int st) {
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = p[q * st];
  };
  auto store = [&](double* p, int st) {
#pragma unroll
    for (int q = 0; q < NP; ++q) p[q * st] = o[q];
  };
  for (int t = tid; t < cnt * 2 * NP; t += kThreads3) {   // R along the first axis
    const int it = t / (2 * NP), rem = t - it * 2 * NP, w = rem / NP, n = rem - w * NP;
    load(trd + 2 * (hp[it].src_b + n * NP) + w, 2);
    line_restrict<NP>(v, o, A.tab + hp[it].tab_ra);
    store(sY + (it * 2 + w) * N2 + n * NP, 1);
  }
  __syncthreads();
  for (int t = tid; t < cnt * 2 * NP; t += kThreads3) {   // and the second
    const int it = t / (2 * NP), rem = t - it * 2 * NP, w = rem / NP, i = rem - w * NP;
    load(sY + (it * 2 + w) * N2 + i, NP);
    line_restrict<NP>(v, o, A.tab + hp[it].tab_rb);
    store(sX + (it * 2 + w) * N2 + i, NP);
  }
  __syncthreads();
  // J and F of the larger side; the smaller side's are their negatives
  for (int t = tid; t < cnt * NM * NM; t += kThreads3) {
    const int it = t / (NM * NM), q = t - it * NM * NM, i = q % NM, j = q / NM;
    const HangPair& h = hp[it];
    const int ns = h.ns;
    const bool big = i < NP && j < NP, small = i < ns && j < ns;
    if (!big && !small) continue;
    double* X = sX + it * 2 * N2 + j * NP + i;
    double J = big ? X[0] : 0.0, F = big ? X[N2] : 0.0;
    if (small) {
      const double2 s = tr[h.src_s + j * ns + i];
      J -= s.x;
      F -= s.y;
      // (BR2: the larger side's lifting is added to the residual below)
      tr[h.dst_s + j * ns + i] = make_double2(-fma(h.cz_s, J, h.cf_s * F), -h.cc_s * J);
    }
    if (big) {
      X[0] = J;
      X[N2] = BR2 ? (small ? fma(h.cx_b, J, h.cf_b * F) : h.cf_b * F) : fma(h.cz_b, J, h.cf_b * F);
    }
  }
  __syncthreads();
  constexpr int W = BR2 ? 1 : 2;   // SIPG: J and the residual go back together
  for (int t = tid; t < cnt * W * NP; t += kThreads3) {
    const int it = t / (W * NP), rem = t - it * W * NP, w = rem / NP, n = rem - w * NP;
    load(sX + (it * 2 + w) * N2 + n * NP, 1);
    line_restrict_t<NP>(v, o, A.tab + hp[it].tab_ra);
    store(sY + (it * 2 + w) * N2 + n * NP, 1);
  }
  __syncthreads();
  for (int t = tid; t < cnt * W * NP; t += kThreads3) {
    const int it = t / (W * NP), rem = t - it * W * NP, w = rem / NP, i = rem - w * NP;
    const HangPair& h = hp[it];
    load(sY + (it * 2 + w) * N2 + i, NP);
    line_restrict_t<NP>(v, o, A.tab + h.tab_rb);
    if (BR2) store(sX + it * 2 * N2 + i, NP);   // R^T J: the lifting, and c2
    double* dst = A.tr + 2 * (h.dst_b + i) + (w == 0 ? 1 : 0);
    const double c = w == 0 ? h.cc_b : 1.0;
#pragma unroll
    for (int q = 0; q < NP; ++q) dst[2 * q * NP] = w == 0 ? c * o[q] : o[q];
  }
  if (!BR2) return;
  __syncthreads();
  for (int t = tid; t < cnt * NP; t += kThreads3) {   // R R^T J
    const int it = t / NP, n = t - it * NP;
    load(sX + it * 2 * N2 + n * NP, 1);
    line_restrict<NP>(v, o, A.tab + hp[it].tab_ra);
    store(sY + it * 2 * N2 + n * NP, 1);
  }
  __syncthreads();
  for (int t = tid; t < cnt * NP; t += kThreads3) {
    const int it = t / NP, i = t - it * NP;
    const HangPair& h = hp[it];
    load(sY + it * 2 * N2 + i, NP);
    line_restrict<NP>(v, o, A.tab + h.tab_rb);
    const int ns = h.ns;
    double* X = sX + it * 2 * N2 + N2 + i;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      X[q * NP] = fma(h.cz_b, o[q], X[q * NP]);
      if (i < ns && q < ns) {
        double2* d = tr + h.dst_s + q * ns + i;
        d->x = fma(-h.cx_s, o[q], d->x);
      }
    }
  }
  __syncthreads();
  for (int t = tid; t < cnt * NP; t += kThreads3) {   // the larger side's residual back
    const int it = t / NP, n = t - it * NP;
    load(sX + it * 2 * N2 + N2 + n * NP, 1);
    line_restrict_t<NP>(v, o, A.tab + hp[it].tab_ra);
    store(sY + it * 2 * N2 + n * NP, 1);
  }
  __syncthreads();
  for (int t = tid; t < cnt * NP; t += kThreads3) {
    const int it = t / NP, i = t - it * NP;
    load(sY + it * 2 * N2 + i, NP);
    line_restrict_t<NP>(v, o, A.tab + hp[it].tab_rb);
    store(A.tr + 2 * (hp[it].dst_b + i), 2 * NP);
  }
}

template <int P, bool BR2>
__device__ __forceinline__ void apply3_tile(const ApplyArgs& A, const ApplyTile& T, int tile, double* sm,
                                            double* red) {
  using B = ModalTab<P>;
  constexpr int NP = P + 1, N2 = NP * NP, N3 = N2 * NP;
  const int cnt = T.count, nl = cnt * N2;
  double* tb = sm;
  double* sx = tb + B::SIZE;
  double* sg = sx + cnt * N3;
  double* sr = sg + cnt * N3;              // [cnt][6][N2] side residuals over a h
  double* sc = sr + cnt * 6 * N2;          // [cnt][6][N2] normal-derivative coefficients over a h
  const double *E = tb, *O = tb + B::oO, *K = tb + B::oK, *S = tb + B::oS, *Q = tb + B::oQ;
  const int tid = threadIdx.x;
  const double2* tr = reinterpret_cast<const double2*>(A.tr);
  const ElemRec3* er = A.erec3 + T.first;
  for (int i = tid; i < B::SIZE; i += kThreads3) tb[i] = __ldg(A.tab + A.moff3[P] + i);
  for (int t = tid; t < cnt * N3; t += kThreads3) {
    const int e = t / N3;
    sx[t] = __ldg(A.xm + er[e].off + (t - e * N3));
  }
  // ---- side residuals: same-size neighbours and the boundary point by point
  // (diagonal in modes), hanging sides from their pairs' results, in order
  for (int t = tid; t < cnt * 6 * N2; t += kThreads3) {
    const int es = t / N2, q = t - es * N2;
    const SubFaceModal3& f = A.sfm3[(int64_t)T.first * 6 + es];
    double r, c;
    if (f.pairs == 0) {
      const int i = q % NP, j = q / NP, nn = f.nn;
      const double2 o = __ldg(tr + f.own_off + q);
      double J = o.x, F = o.y;
      const bool in = i < nn && j < nn;   // boundary: nn = 0
      if (in) {
        const double2 n = __ldg(tr + f.nbr_off + j * nn + i);
        J -= n.x;
        F -= n.y;   // the neighbour's outward dn
      }
      r = fma(BR2 && in ? f.czx : f.cz, J, f.cf * F);
      c = f.cc * J;
    } else {
      const double2* src = tr + f.own_off + q;
      const int pairs = f.pairs;
      const double2 first = __ldg(src);
      r = first.x;
      c = first.y;
      for (int g = 1; g < pairs; ++g) {
        const double2 n = __ldg(src + (int64_t)g * N2);
        r += n.x;
        c += n.y;
      }
    }
    sr[t] = r;
    sc[t] = c;
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
