// Matrix-free SIPG / BR2 operator y = A x on mapped squares (Section 2:
// element maps T_kappa onto general quadrilaterals; Eq. fe-problem; BR2 of
// Section 4.4), FP64.
//
// The elements are the images of the leaf boxes under the bilinear map of the
// lattice domain (DomainMap), so the geometric factors vary inside every
// element and the separable M / K contractions of boxes no longer apply.  The
// kernel works at Gauss points instead, with the same tiles, side traces and
// flat sub-face item lists as the box kernel:
//   volume  u at the (p+2)^2 Gauss points by sum factorisation (B = l_j(x_g),
//           D = l_j'(x_g)): grad_xi u = ((B (x) D) u, (D (x) B) u); at every
//           point the flux a w_g w_h G grad_xi u with G = det(J) J^-1 J^-T of
//           the map there (three factors per point, stored at setup); back to
//           the nodes with the transposed products: four passes of
//           O((p+1)(p+2)^2) work per element instead of two;
//   faces   (map_face kernel, before the tiles) one thread per (sub-face, Gauss
//           point) evaluates both sides' traces there (values and a-weighted
//           normal derivatives from the trace array, tangential derivatives
//           from the trace values) and, with the point's stored factors (the
//           arc-length weight w and w m for m = J^-1 n, n = J^-T nu / |J^-T nu|
//           the physical normal), writes three adjoint weights: of the test
//           function's value, of its tangential derivative and of its normal
//           derivative.  Seen from the other side the jump and the normal change
//           sign: the first and the third weight do, the second does not, so
//           one evaluation serves both sides.  In the tiles one thread per side
//           node sums its sub-faces' weights in sub-face order (deterministic)
//           with the side's basis tables, and the gather adds the
//           normal-derivative weights through l_k'(0 or 1) / h.
//   BR2     the mass matrix of a mapped element is not a Kronecker product, so
//           the lifting takes the block of each element's mass inverse on a
//           side's nodes (stored at setup): per sub-face the jump projected onto
//           both sides' nodes, the two blocks applied, and the lifted values
//           at its points added to the value weights.
// Applies are bit-reproducible (fixed sums, no atomics on data).
// Measured (GB300): apply of the 98k-unknown hp mesh on a quadrilateral 58.9 us
// with every tile evaluating its sub-faces itself (24 of 32 lanes active), 43.9
// with the weights formed once (22.6 of 27.3 MFLOP; the tiles' kernel 58 -> 36
// us, the weights' 6) and 42.4 without spills; PCG on 24k curved unknowns 70.3 ->
// 52.8 us per iteration (with the other changes measured beside it).
#pragma once

#include "apply_kernel.cuh"

namespace dg {

template <int P>
struct MapShape {
  static constexpr int NP = P + 1;
  static constexpr int NN = NP * NP;
  static constexpr int Q = P + 1 + kMapQExtra;
  static constexpr int QQ = Q * Q;
  static constexpr int EPB = apply_epb(P);
  // shared doubles: B, D (2 Q NP), x (EPB NN), stage 1 / 3 (2 EPB NP Q),
  // point fluxes (2 EPB QQ), side sums r, c2 (8 EPB NP)
  static constexpr int SMEM = 2 * Q * NP + EPB * NN + 2 * EPB * NP * Q + 2 * EPB * QQ + 8 * EPB * NP;
};

// Weights of a tile of sub-faces (MapFaceTile: rules of at most nq points, sides
// of at most nn nodes).
template <bool BR2>
__device__ __forceinline__ void map_face_tile(const ApplyArgs& A, const MapFaceTile& T, double* sm) {
  const int Q = T.nq, N = T.nn, cnt = T.count;
  const MapFace* faces = A.mface + T.first;
  const double2* tr = reinterpret_cast<const double2*>(A.tr);
  double* sj = sm;                    // BR2: [cnt][Q] w [[u]]
  double* sp = sj + cnt * Q;          // [cnt][2][N] projections, then
  double* sz = sp + cnt * 2 * N;      // [cnt][2][N] liftings
  for (int t = threadIdx.x; t < cnt * Q; t += kThreads3) {
    const int it = t / Q, g = t - it * Q;
    const MapFace& f = faces[it];
    const int qf = f.qf;
    if (g >= qf) continue;
    double u0 = 0.0, du0 = 0.0, f0 = 0.0;
    {
      const int np = f.np;
      const double2* src = tr + f.src_o;
      const double* Bo = A.tab + f.tab_bo + g * np;
      const double* Do = Bo + qf * np;
      for (int m = 0; m < np; ++m) {
        const double2 v = __ldg(src + m);
        const double b = __ldg(Bo + m);
        u0 = fma(b, v.x, u0);
        du0 = fma(__ldg(Do + m), v.x, du0);
        f0 = fma(b, v.y, f0);
      }
    }
    // the point's factors: w = w_g |J t| dt, w m_t, w m_n s (m = J^-1 n)
    const double* gf = A.gface + f.geo;
    const double w = __ldg(gf + g), wmt = __ldg(gf + qf + g), wmn = __ldg(gf + 2 * qf + g);
    double jmp = u0, flux = fma(f0, wmn, f.aih_o * du0 * wmt), cc = 1.0;   // w (a grad u-) . n
    if (f.npn > 0) {
      const int np = f.npn;
      const double2* src = tr + f.src_n;
      const double* Bn = A.tab + f.tab_bn + g * np;
      const double* Dn = Bn + qf * np;
      double u1 = 0.0, du1 = 0.0, f1 = 0.0;
      for (int m = 0; m < np; ++m) {
        const double2 v = __ldg(src + m);
        const double b = __ldg(Bn + m);
        u1 = fma(b, v.x, u1);
        du1 = fma(__ldg(Dn + m), v.x, du1);
        f1 = fma(b, v.y, f1);
      }
      jmp = u0 - u1;
      flux = 0.5 * (flux + fma(-f1, wmn, f.aih_n * du1 * wmt));
      cc = 0.5;
    }
    double* W = A.mw + f.w + 3 * g;
    W[0] = BR2 ? -flux : fma(f.sigma * jmp, w, -flux);   // of v-
    W[1] = -cc * jmp * wmt;                              // of d v- / d t (times a / h and l' at the side sums)
    W[2] = -cc * jmp * wmn;                              // of a times the outward normal derivative of v-
    if (BR2) sj[it * Q + g] = w * jmp;
  }
  if (!BR2) return;
  __syncthreads();
  // BR2 liftings (Section 4.4) on both sides: j = int phi_j [[u]] ds on each
  // side's nodes, z = (block of that element's mass inverse on the side) j, and
  // at every point the weight eta coef a w (z-(x_g) + z+(x_g)) of v-
  for (int t = threadIdx.x; t < cnt * 2 * N; t += kThreads3) {
    const int it = t / (2 * N), rem = t - it * 2 * N, sd = rem / N, j = rem - sd * N;
    const MapFace& f = faces[it];
    const int np = sd == 0 ? f.np : f.npn;
    if (j >= np) continue;
    const double* B = A.tab + (sd == 0 ? f.tab_bo : f.tab_bn) + j;
    double a = 0.0;
    for (int g = 0; g < f.qf; ++g) a = fma(__ldg(B + g * np), sj[it * Q + g], a);
    sp[t] = a;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < cnt * 2 * N; t += kThreads3) {
    const int it = t / (2 * N), rem = t - it * 2 * N, sd = rem / N, j = rem - sd * N;
    const MapFace& f = faces[it];
    const int np = sd == 0 ? f.np : f.npn;
    if (j >= np) continue;
    const double* G = A.gbr2 + (sd == 0 ? f.g_o : f.g_n) + j * np;
    double a = 0.0;
    for (int i = 0; i < np; ++i) a = fma(__ldg(G + i), sp[t - j + i], a);
    sz[t] = a;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < cnt * Q; t += kThreads3) {   // the thread that wrote the point's weights
    const int it = t / Q, g = t - it * Q;
    const MapFace& f = faces[it];
    if (g >= f.qf) continue;
    const double* z = sz + it * 2 * N;
    double v = 0.0;
    for (int i = 0; i < f.np; ++i) v = fma(__ldg(A.tab + f.tab_bo + g * f.np + i), z[i], v);
    for (int i = 0; i < f.npn; ++i) v = fma(__ldg(A.tab + f.tab_bn + g * f.npn + i), z[N + i], v);
    double* W = A.mw + f.w + 3 * g;
    W[0] = fma(f.cbr2 * __ldg(A.gface + f.geo + g), v, W[0]);
  }
}

// x with its sign bit flipped where s is negative zero's bit pattern
__device__ __forceinline__ double flip(double x, int s) {
  return __hiloint2double(__double2hiint(x) ^ s, __double2loint(x));
}

template <int P>
__device__ __forceinline__ void apply_map_tile(const ApplyArgs& A, const ApplyTile& T, int tile, double* sm,
                                               double* red) {
  using S = MapShape<P>;
  constexpr int NP = S::NP, NN = S::NN, Q = S::Q, QQ = S::QQ, EPB = S::EPB;
  double* sB = sm;                    // [Q][NP]
  double* sD = sB + Q * NP;
  double* sx = sD + Q * NP;           // [EPB][NN]
  double* sA1 = sx + EPB * NN;        // [EPB][NP][Q]; stage 3 reuses it
  double* sA2 = sA1 + EPB * NP * Q;
  double* sF1 = sA2 + EPB * NP * Q;   // [EPB][Q][Q]
  double* sF2 = sF1 + EPB * QQ;
  double* sr = sF2 + EPB * QQ;        // [EPB][4][NP]
  double* sc2 = sr + EPB * 4 * NP;

  const int tid = threadIdx.x;
  const int count = T.count;
  const MapOff mo = A.moff[P];
  for (int i = tid; i < Q * NP; i += blockDim.x) {
    sB[i] = __ldg(A.tab + mo.B + i);
    sD[i] = __ldg(A.tab + mo.D + i);
  }
  for (int t = tid; t < count * NN; t += blockDim.x) {
    const int e = t / NN;
    sx[t] = A.x[A.off[A.order[T.first + e]] + (t - e * NN)];
  }
  __syncthreads();
  // ---- volume stage 1: contract along x at the Gauss points (derivative and value)
  for (int t = tid; t < count * NP * Q; t += blockDim.x) {
    const int e = t / (NP * Q), rem = t - e * NP * Q;
    const int jy = rem / Q, g = rem - jy * Q;
    const double* xr = sx + e * NN + jy * NP;
    double a = 0.0, b = 0.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      a = fma(sD[g * NP + j], xr[j], a);
      b = fma(sB[g * NP + j], xr[j], b);
    }
    sA1[t] = a;
    sA2[t] = b;
  }
  __syncthreads();
  // ---- volume stage 2 and the flux at every Gauss point
  for (int t = tid; t < count * QQ; t += blockDim.x) {
    const int e = t / QQ, rem = t - e * QQ;
    const int gy = rem / Q, gxi = rem - gy * Q;
    const double* a1 = sA1 + e * NP * Q + gxi;
    const double* a2 = sA2 + e * NP * Q + gxi;
    double ux = 0.0, uy = 0.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      ux = fma(sB[gy * NP + j], a1[j * Q], ux);
      uy = fma(sD[gy * NP + j], a2[j * Q], uy);
    }
    // the point's factors a w_g w_h G (three planes per element)
    const double* G = A.gvol + A.goff[A.order[T.first + e]] + rem;
    const double g11 = __ldg(G), g12 = __ldg(G + QQ), g22 = __ldg(G + 2 * QQ);
    sF1[t] = fma(g11, ux, g12 * uy);
    sF2[t] = fma(g12, ux, g22 * uy);
  }
  // ---- faces: one thread per side node sums its sub-faces' weights in
  // sub-face order with the side's basis tables
  for (int t = tid; t < count * 4 * NP; t += blockDim.x) {
    const int e = t / (4 * NP);
    const int s = (t / NP) & 3;
    const int i = t % NP;
    const int k = A.order[T.first + e];
    const int rec0 = A.sf_ptr[4 * k + s], rec1 = A.sf_ptr[4 * k + s + 1];
    double r = 0.0, rt = 0.0, c2 = 0.0;
    for (int j = rec0; j < rec1; ++j) {
      const MapSide fm = A.mside[j];
      const double* W = A.mw + fm.w;
      const double* Bo = A.tab + fm.tab_bo + i;
      const double* Do = Bo + fm.qf * NP;
      for (int g = 0; g < fm.qf; ++g) {
        const double b = __ldg(Bo + g * NP);
        r = fma(b, flip(__ldg(W + 3 * g), fm.sign), r);
        rt = fma(__ldg(Do + g * NP), __ldg(W + 3 * g + 1), rt);
        c2 = fma(b, flip(__ldg(W + 3 * g + 2), fm.sign), c2);
      }
    }
    sr[t] = fma(A.aih[k], rt, r);
    sc2[t] = c2;
  }
  __syncthreads();
  // ---- volume stage 3: back along y (into the stage-1 arrays)
  for (int t = tid; t < count * NP * Q; t += blockDim.x) {
    const int e = t / (NP * Q), rem = t - e * NP * Q;
    const int iy = rem / Q, g = rem - iy * Q;
    const double* f1 = sF1 + e * QQ + g;
    const double* f2 = sF2 + e * QQ + g;
    double a = 0.0, b = 0.0;
#pragma unroll
    for (int gy = 0; gy < Q; ++gy) {
      a = fma(sB[gy * NP + iy], f1[gy * Q], a);
      b = fma(sD[gy * NP + iy], f2[gy * Q], b);
    }
    sA1[t] = a;
    sA2[t] = b;
  }
  __syncthreads();
  // ---- gather: volume stage 4 + side residuals + normal-derivative terms
  const BasisOff bo = A.boff[P];
  double part_dot = 0.0;
  for (int t = tid; t < count * NN; t += blockDim.x) {
    const int e = t / NN, node = t - e * NN;
    const int ix = node % NP, iy = node / NP;
    const int k = A.order[T.first + e];
    const double* c1 = sA1 + e * NP * Q + iy * Q;
    const double* c2v = sA2 + e * NP * Q + iy * Q;
    double y = 0.0;
#pragma unroll
    for (int g = 0; g < Q; ++g) {
      y = fma(sD[g * NP + ix], c1[g], y);
      y = fma(sB[g * NP + ix], c2v[g], y);
    }
    const double* d0 = A.tab + bo.d0;
    const double* d1 = A.tab + bo.d1;
    const double* c2 = sc2 + e * 4 * NP;
    const double* r = sr + e * 4 * NP;
    double gg = -__ldg(d0 + ix) * c2[0 * NP + iy];
    gg = fma(__ldg(d1 + ix), c2[1 * NP + iy], gg);
    gg = fma(-__ldg(d0 + iy), c2[2 * NP + ix], gg);
    gg = fma(__ldg(d1 + iy), c2[3 * NP + ix], gg);
    y = fma(gg, A.aih[k], y);
    if (ix == 0) y += r[0 * NP + iy];
    if (ix == P) y += r[1 * NP + iy];
    if (iy == 0) y += r[2 * NP + ix];
    if (iy == P) y += r[3 * NP + ix];
    A.y[A.off[k] + node] = y;
    part_dot = fma(y, sx[t], part_dot);
  }
  if (A.dot_partial) {
    // tile partial of x . y (summed in tile order when the launch ends)
    const double tot = block_sum<kThreads>(part_dot, red);
    if (tid == 0) A.dot_partial[tile] = tot;
  }
}

}  // namespace dg
