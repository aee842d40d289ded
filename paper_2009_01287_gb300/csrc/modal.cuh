// One-dimensional pieces of the operators in Legendre modes (squares and
// cubes): a line of NP values held by one thread, the tables of its degree in
// shared memory (read by all lanes at once).
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
struct ModalTab {
  static constexpr int NP = P + 1, H = NP / 2, HC = (NP + 1) / 2;
  static constexpr int oO = HC * HC, oK = oO + H * H, oS = oK + NP * NP, oQ = oS + NP;
  static constexpr int SIZE = oQ + NP;
};

}  // namespace dg
