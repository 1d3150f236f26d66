// lclb_pair.cuh -- the liquid-crystal algebra of two nodes at once (FP32 boxes
// of even width): molecular field, stress and the increment of Q of the
// one-node functions lc_node_f32 and q_increment_f32 in packed FP32x2.
//
// The order of the sums is theirs, operation by operation, and stays: a box
// near rest is driven by small differences of the stress, so a sum rounded in
// another order shows in the velocity at 3e-5 (measured over 345 boxes of mixed
// sizes), although neither order is the better one.  What is saved are
// operations that change no rounding: entries that symmetry repeats, factors of
// two and four (taken into constants and undone once), products with the zeros
// of the antisymmetric part, chiral terms of a nematic.
#pragma once
#include "lclb_f2.cuh"
#include "lclb_dev.cuh"

namespace lclb {

using LcPair = LcPairT<f2>;  // each value twice: one 8-byte load per packed operand

// lc_node_f32 of two nodes.  dq: the doubled first derivatives; CHIRAL: q0 != 0.
template <bool CHIRAL, bool NEED_P>
__device__ __forceinline__ void lc_pair(const LcPair& P, const f2 qi[5], const f2 dq[3][5],
                                        const f2 lap[5], f2 h[5], f2 p[9], f2* fprime) {
  const f2 a = qi[0], b = qi[1], c = qi[2], d = qi[3], e = qi[4];
  const f2 f = -a - d;
  const f2* X = dq[0];
  const f2* Y = dq[1];
  const f2* Z = dq[2];
  // Q.Q
  const f2 s0 = (a * a + b * b) + c * c, s1 = (a * b + b * d) + c * e, s2 = (a * c + b * e) + c * f;
  const f2 s3 = (b * b + d * d) + e * e, s4 = (b * c + d * e) + e * f, s5 = (c * c + e * e) + f * f;
  const f2 trq2 = s0 + s3 + s5;
  const f2 cb = P.c_lin + P.nA0g * trq2, tq3 = P.A0g3 * trq2;
  auto bulk = [&](f2 q, f2 s, f2 lp) { return f2((cb * q + P.A0g * s) + P.K * lp); };
  f2 h0 = bulk(a, s0, lap[0]), h1 = bulk(b, s1, lap[1]), h2 = bulk(c, s2, lap[2]), h3 = bulk(d, s3, lap[3]);
  f2 h4 = bulk(e, s4, lap[4]), h5 = f2((cb * f + P.A0g * s5) + P.nK * (lap[0] + lap[3]));
  f2 C[9];  // twice C_ab = eps_agd d_g Q_db
  const f2 tx = X[0] + X[3], ty = Y[0] + Y[3], tz = Z[0] + Z[3];  // minus the zz components
  if constexpr (CHIRAL) {
    C[0] = Y[2] - Z[1]; C[1] = Y[4] - Z[3]; C[2] = -ty - Z[4];
    C[3] = Z[0] - X[2]; C[4] = Z[1] - X[4]; C[5] = Z[2] + tx;
    C[6] = X[1] - Y[0]; C[7] = X[3] - Y[1]; C[8] = X[4] - Y[2];
    h0 = h0 + P.n2Kq * C[0];
    h1 = h1 + P.nKq * (C[1] + C[3]);
    h2 = h2 + P.nKq * (C[2] + C[6]);
    h3 = h3 + P.n2Kq * C[4];
    h4 = h4 + P.nKq * (C[5] + C[7]);
    h5 = h5 + P.n2Kq * C[8];
  }
  h0 = h0 - tq3;
  h3 = h3 - tq3;
  h5 = h5 - tq3;
  h[0] = h0; h[1] = h1; h[2] = h2; h[3] = h3; h[4] = h4;
  if constexpr (!NEED_P) return;
  // K <d_a Q, d_b Q>
  auto dd = [&](const f2* u, const f2* v, f2 tu, f2 tv) {
    const f2 on = (u[0] * v[0] + u[3] * v[3]) + tu * tv, off = (u[1] * v[1] + u[2] * v[2]) + u[4] * v[4];
    return f2(P.K4 * on + P.tK4 * off);
  };
  const f2 e0 = dd(X, X, tx, tx), e1 = dd(X, Y, tx, ty), e2 = dd(X, Z, tx, tz);
  const f2 e3 = dd(Y, Y, ty, ty), e4 = dd(Y, Z, ty, tz), e5 = dd(Z, Z, tz, tz);
  f2 t3 = a * s0;  // Tr Q^3
  t3 = t3 + b * s1; t3 = t3 + c * s2; t3 = t3 + b * s1; t3 = t3 + d * s3; t3 = t3 + e * s4;
  t3 = t3 + c * s2; t3 = t3 + e * s4; t3 = t3 + f * s5;
  f2 fp = P.fb2 * trq2 + P.nA0g3 * t3;
  fp = fp + P.fb4 * f2(trq2 * trq2);
  fp = fp + P.half * (e0 + e3 + e5);
  if constexpr (CHIRAL) {
    f2 qc = a * C[0];  // twice Q:C
    qc = qc + b * C[1]; qc = qc + c * C[2]; qc = qc + b * C[3]; qc = qc + d * C[4]; qc = qc + e * C[5];
    qc = qc + c * C[6]; qc = qc + e * C[7]; qc = qc + f * C[8];
    fp = fp + P.Kq * qc;
    fp = fp + P.Kqq * trq2;
  }
  // A = Q H
  const f2 a00 = (a * h0 + b * h1) + c * h2, a01 = (a * h1 + b * h3) + c * h4, a02 = (a * h2 + b * h4) + c * h5;
  const f2 a10 = (b * h0 + d * h1) + e * h2, a11 = (b * h1 + d * h3) + e * h4, a12 = (b * h2 + d * h4) + e * h5;
  const f2 a20 = (c * h0 + e * h1) + f * h2, a21 = (c * h1 + e * h3) + f * h4, a22 = (c * h2 + e * h4) + f * h5;
  const f2 qh2 = P.twoxi * (a00 + a11 + a22);
  const f2 dg = fp + P.third * qh2;
  f2 E[9] = {e0, e1, e2, e1, e3, e4, e2, e4, e5};
  if constexpr (CHIRAL) {
    // E_ab += 2 K q0 sum over g != b of eps(m, b, g) d_a Q_g. . Q_m.
    auto chi = [&](const f2* D, f2 t, f2* Ea) {
      const f2 zz = -t;
      const f2 u0 = ((D[1] * c + D[3] * e) + D[4] * f) - ((D[2] * b + D[4] * d) + zz * e);
      const f2 u1 = ((D[2] * a + D[4] * b) + zz * c) - ((D[0] * c + D[1] * e) + D[2] * f);
      const f2 u2 = ((D[0] * b + D[1] * d) + D[2] * e) - ((D[1] * a + D[3] * b) + D[4] * c);
      Ea[0] = Ea[0] + P.Kq * u0;
      Ea[1] = Ea[1] + P.Kq * u1;
      Ea[2] = Ea[2] + P.Kq * u2;
    };
    chi(X, tx, E);
    chi(Y, ty, E + 3);
    chi(Z, tz, E + 6);
  }
  auto diag = [&](f2 q, f2 A, f2 H, f2 Ed) {
    const f2 m = (qh2 * q + P.ntwoxi * A) + P.ntwoxi3 * H;
    return f2((m - Ed) + dg);
  };
  p[0] = diag(a, a00, h0, E[0]);
  p[4] = diag(d, a11, h3, E[4]);
  p[8] = diag(f, a22, h5, E[8]);
  auto off = [&](f2 q, f2 A, f2 At, f2 H, f2 Eab, f2 Eba, f2& pab, f2& pba) {
    const f2 m = (qh2 * q + P.nxi * (A + At)) + P.ntwoxi3 * H, df = A - At;
    pab = (m - Eab) + df;
    pba = (m - Eba) - df;
  };
  off(b, a01, a10, h1, E[1], E[3], p[1], p[3]);
  off(c, a02, a20, h2, E[2], E[6], p[2], p[6]);
  off(e, a12, a21, h4, E[5], E[7], p[5], p[7]);
  *fprime = fp;
}

// Local part of H(hi + lo) - H(hi), added to h (comp_h_f32 of two nodes).
__device__ __forceinline__ void comp_h_pair(const LcPair& P, const f2 qi[5], const f2 lo[5], f2 h[5]) {
  const f2 a = qi[0], b = qi[1], c = qi[2], d = qi[3], e = qi[4];
  const f2 la = lo[0], lb = lo[1], lc = lo[2], ld = lo[3], le = lo[4];
  const f2 f = -a - d, lf = -la - ld;
  f2 t2 = a * a, tl = a * la;  // Tr Q^2, Q:lo
  t2 = t2 + b * b; t2 = t2 + c * c; t2 = t2 + b * b; t2 = t2 + d * d; t2 = t2 + e * e;
  t2 = t2 + c * c; t2 = t2 + e * e; t2 = t2 + f * f;
  tl = tl + b * lb; tl = tl + c * lc; tl = tl + b * lb; tl = tl + d * ld; tl = tl + e * le;
  tl = tl + c * lc; tl = tl + e * le; tl = tl + f * lf;
  const f2 cb = P.c_lo + P.nA0g * t2, nt = -f2(P.A2 * tl);
  auto six = [](f2 x0, f2 l0, f2 y0, f2 m0, f2 x1, f2 l1, f2 y1, f2 m1, f2 x2, f2 l2, f2 y2, f2 m2) {
    f2 v = x0 * l0;
    v = v + y0 * m0; v = v + x1 * l1; v = v + y1 * m1; v = v + x2 * l2; v = v + y2 * m2;
    return v;
  };
  auto add = [&](int k, f2 ql) { h[k] = ((h[k] + cb * lo[k]) + P.A0g * ql) + nt * qi[k]; };
  add(0, six(a, la, la, a, b, lb, lb, b, c, lc, lc, c) + P.nq23 * tl);
  add(1, six(a, lb, la, b, b, ld, lb, d, c, le, lc, e));
  add(2, six(a, lc, la, c, b, le, lb, e, c, lf, lc, f));
  add(3, six(b, lb, lb, b, d, ld, ld, d, e, le, le, e) + P.nq23 * tl);
  add(4, six(b, lc, lb, c, d, le, ld, e, e, lf, le, f));
}

// Upwind parts of twice the velocities of the + and - face of one axis (ui, p,
// m: the velocity component of that axis at the node and its two neighbours):
// + face outflow of the node's own value with up, inflow of the neighbour's with
// dn; - face the other way round.
__device__ __forceinline__ void upwind_pair(f2 ui, f2 p, f2 m, f2 up[2], f2 dn[2]) {
  const f2 fp = ui + p, fm = ui + m;
  up[0] = pos_part(fp);
  dn[0] = neg_part(fp);
  up[1] = -neg_part(fm);
  dn[1] = -pos_part(fm);
}

// Twice the advective flux divergence of one component: per face one of the
// two products is an exact zero, the other the flux, added in face order.
__device__ __forceinline__ f2 advect_pair(const f2 up[6], const f2 dn[6], f2 q, const f2 n[6]) {
  f2 v = up[0] * q;
  v = v + dn[0] * n[0];
#pragma unroll
  for (int d = 1; d < 6; ++d) {
    v = v + up[d] * q;
    v = v + dn[d] * n[d];
  }
  return v;
}

// Increment of Q (q_increment_f32 of two nodes): adv twice the flux divergence,
// w twice the velocity gradient; h receives the compensation.  Sums are four
// times their values until the end.
__device__ __forceinline__ void q_pair(const LcPair& P, const f2 qi[5], const f2 adv[5], const f2 w[3][3], f2 h[5],
                                       const f2 lo[5], f2 d5[5]) {
  const f2 a = qi[0], b = qi[1], c = qi[2], d = qi[3], e = qi[4];
  const f2 f = -a - d;
  // 4 D (symmetric) and 4 Omega (antisymmetric)
  const f2 D00 = w[0][0] + w[0][0], D11 = w[1][1] + w[1][1], D22 = w[2][2] + w[2][2];
  const f2 D01 = w[0][1] + w[1][0], D02 = w[0][2] + w[2][0], D12 = w[1][2] + w[2][1];
  const f2 O01 = w[0][1] - w[1][0], O02 = w[0][2] - w[2][0], O12 = w[1][2] - w[2][1];
  const f2 O10 = w[1][0] - w[0][1], O20 = w[2][0] - w[0][2], O21 = w[2][1] - w[1][2];
  f2 tr = a * D00;  // Tr(Q W)
  tr = tr + b * D01; tr = tr + c * D02; tr = tr + b * D01; tr = tr + d * D11; tr = tr + e * D12;
  tr = tr + c * D02; tr = tr + e * D12; tr = tr + f * D22;
  // one term of D Q + Q D
  auto dq = [](f2 D1, f2 q1, f2 q2, f2 D2) { return f2(D1 * q1 + q2 * D2); };
  auto end = [&](f2 s, f2 D, f2 qt) { return f2((s + P.xi23 * D) + P.ntwoxi * f2(qt * tr)); };
  const f2 xi = P.xi;
  f2 s00 = xi * dq(D00, a, a, D00);
  s00 = s00 + xi * dq(D01, b, b, D01); s00 = s00 + O01 * b; s00 = s00 + b * O01;
  s00 = s00 + xi * dq(D02, c, c, D02); s00 = s00 + O02 * c; s00 = s00 + c * O02;
  s00 = end(s00, D00, a + P.third);
  f2 s11 = xi * dq(D01, b, b, D01);
  s11 = s11 + O10 * b; s11 = s11 + b * O10;
  s11 = s11 + xi * dq(D11, d, d, D11);
  s11 = s11 + xi * dq(D12, e, e, D12); s11 = s11 + O12 * e; s11 = s11 + e * O12;
  s11 = end(s11, D11, d + P.third);
  f2 s22 = xi * dq(D02, c, c, D02);
  s22 = s22 + O20 * c; s22 = s22 + c * O20;
  s22 = s22 + xi * dq(D12, e, e, D12); s22 = s22 + O21 * e; s22 = s22 + e * O21;
  s22 = s22 + xi * dq(D22, f, f, D22);
  s22 = end(s22, D22, f + P.third);
  f2 s01 = xi * dq(D00, b, a, D01);
  s01 = s01 + a * O10;
  s01 = s01 + xi * dq(D01, d, b, D11); s01 = s01 + O01 * d;
  s01 = s01 + xi * dq(D02, e, c, D12); s01 = s01 + O02 * e; s01 = s01 + c * O12;
  s01 = end(s01, D01, b);
  f2 s02 = xi * dq(D00, c, a, D02);
  s02 = s02 + a * O20;
  s02 = s02 + xi * dq(D01, e, b, D12); s02 = s02 + O01 * e; s02 = s02 + b * O21;
  s02 = s02 + xi * dq(D02, f, c, D22); s02 = s02 + O02 * f;
  s02 = end(s02, D02, c);
  f2 s12 = xi * dq(D01, c, b, D02);
  s12 = s12 + O10 * c; s12 = s12 + b * O20;
  s12 = s12 + xi * dq(D11, e, d, D12); s12 = s12 + d * O21;
  s12 = s12 + xi * dq(D12, f, e, D22); s12 = s12 + O12 * f;
  s12 = end(s12, D12, e);
  const f2 tr3 = P.third * (s00 + s11 + s22);
  comp_h_pair(P, qi, lo, h);
  const f2 s[5] = {s00, s01, s02, s11, s12};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    f2 v = (P.Gam4 * h[k] + s[k]) + P.ntwo * adv[k];
    if (k == 0 || k == 3) v = v - tr3;
    d5[k] = 0.25f * v;
  }
}

// The same with the flow frozen (u = 0).
__device__ __forceinline__ void q_pair_frozen(const LcPair& P, const f2 qi[5], f2 h[5], const f2 lo[5], f2 d5[5]) {
  comp_h_pair(P, qi, lo, h);
#pragma unroll
  for (int k = 0; k < 5; ++k) d5[k] = P.Gam * h[k];
}

}  // namespace lclb
