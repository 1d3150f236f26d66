// lclb_dev.cuh -- device-side data structures and per-node physics of the
// hybrid LB / Beris-Edwards solver (Lintuvuori et al., Sec. 2).
//
// Storage: structure of arrays [component][z][y][x], node index
// x + nx*(y + ny*z).  Populations are stored as deviations df_i = f_i - w_i rho0
// after collision (pull scheme: the next step gathers df_i(r - c_i)).
// Q stores (xx, xy, xz, yy, yz); zz = -xx - yy.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "f64_bits.cuh"

namespace lclb {

constexpr int NQ = 19;
constexpr int MAXCOL = 126;      // colloids per box (mask byte holds id + 1 in 7 bits)
constexpr uint8_t NEAR = 0x80;   // fluid node with a solid or wall node among its 18 neighbours
constexpr uint8_t IDMASK = 0x7F;
constexpr uint8_t WALLFLAG = 0xFF;  // "beyond a wall" marker in shared-memory flag planes

// D3Q19: rest; +x,-x,+y,-y,+z,-z; (1,1,0),(-1,-1,0),(1,-1,0),(-1,1,0),(1,0,1),(-1,0,-1),
// (1,0,-1),(-1,0,1),(0,1,1),(0,-1,-1),(0,1,-1),(0,-1,1); weights 1/3, 1/18, 1/36.
__host__ __device__ constexpr int cx(int q) {
  return q == 1 || q == 7 || q == 9 || q == 11 || q == 13 ? 1 : (q == 2 || q == 8 || q == 10 || q == 12 || q == 14 ? -1 : 0);
}
__host__ __device__ constexpr int cy(int q) {
  return q == 3 || q == 7 || q == 10 || q == 15 || q == 17 ? 1 : (q == 4 || q == 8 || q == 9 || q == 16 || q == 18 ? -1 : 0);
}
__host__ __device__ constexpr int cz(int q) {
  return q == 5 || q == 11 || q == 14 || q == 15 || q == 18 ? 1 : (q == 6 || q == 12 || q == 13 || q == 16 || q == 17 ? -1 : 0);
}
__host__ __device__ constexpr int opp(int q) { return q == 0 ? 0 : ((q & 1) ? q + 1 : q - 1); }
__host__ __device__ constexpr double wq(int q) { return q == 0 ? 1.0 / 3.0 : (q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0); }

struct DevParams {
  double rho0, tau, A0, gamma, K, q0, xi, Gamma, S0;
  double g[3];
  int lc_on, flow_on;
};

// The constants in the arithmetic type of the kernels (so that FP32 kernels
// never convert from FP64 per node).
template <typename T>
struct PhysT {
  T rho0, omega, pref, ptau;  // rho0, 1/tau, 1 - 1/(2 tau), (1 - 1/(2 tau)) tau = tau - 1/2
  T A0, gamma, K, q0, xi, Gamma;
  T S0, S0l;  // S0l: the part of S0 that FP32 drops
  T g[3];
};

// Constants of the packed FP32 functions (lclb_pair.cuh): one per field in the
// box's record, twice in the kernels' shared copy (T = f2).
template <typename T>
struct LcPairT {
  T A0g, nA0g, c_lin, A0g3, nA0g3;   // A0 g, H: Q beyond -A0 g Tr(Q^2), A0 g / 3
  T K, nK, K4, tK4;                  // K, K / 4, 2 K / 4
  T Kq, nKq, n2Kq, Kqq;              // K q0 (half of 2 K q0), 2 K q0^2
  T fb2, fb4, half, third;
  T twoxi, ntwoxi, nxi, ntwoxi3;     // 2 xi, -xi, -2 xi / 3
  T nsix;
  T xi, xi23, Gam4, ntwo;            // increment of Q (scaled by four)
  T c_lo, A2, nq23, Gam;
};
constexpr int LCPAIR_N = sizeof(LcPairT<float>) / sizeof(float);

// Formed on the device, once per upload of the record, by the expressions of the
// one-node functions (so that both round alike).
__device__ __forceinline__ void lc_pair_constants(LcPairT<float>& C, const PhysT<float>& P) {
  const float A0 = P.A0, g = P.gamma, K = P.K, q0 = P.q0, xi = P.xi;
  const float third = 1.f / 3.f;
  const float A0g = A0 * g, twoKq0 = 2.f * K * q0;
  const float c_lin = -A0 * (1.f - g * third) - 4.f * K * q0 * q0;
  const float A0g3 = A0g * third;
  C.A0g = A0g; C.nA0g = -A0g; C.c_lin = c_lin; C.A0g3 = A0g3; C.nA0g3 = -A0g3;
  C.K = K; C.nK = -K; C.K4 = 0.25f * K; C.tK4 = 0.5f * K;
  C.Kq = 0.5f * twoKq0; C.nKq = -0.5f * twoKq0; C.n2Kq = -twoKq0; C.Kqq = 2.f * K * q0 * q0;
  C.fb2 = 0.5f * A0 * (1.f - g * third); C.fb4 = 0.25f * A0g; C.half = 0.5f; C.third = third;
  const float twoxi = 2.f * xi, twoxi3 = twoxi * third;
  C.twoxi = twoxi; C.ntwoxi = -twoxi; C.nxi = -xi; C.ntwoxi3 = -twoxi3;
  C.nsix = -6.f;
  C.xi = xi; C.xi23 = 2.f * xi / 3.f; C.Gam4 = 4.f * P.Gamma; C.ntwo = -2.f;
  C.c_lo = -A0 * (1.f - g / 3.f) - 4.f * K * q0 * q0 - 6.f * K;
  C.A2 = 2.f * A0g; C.nq23 = -(2.f / 3.f); C.Gam = P.Gamma;
}

// Constants of the FP64 liquid-crystal algebra, every combination that the node
// functions multiply by formed once per box.
template <typename T>
struct LcK {
  T A0g, nA0g, nA3, c_lin;         // A0 g, its negative, -A0 g / 3, H: Q beyond -A0 g Tr(Q^2)
  T K, nKq0, n2Kq0, Kq0;           // K, -K q0, -2 K q0, K q0
  T f2c, f4c, K8;                  // f': Tr Q^2, (Tr Q^2)^2, K / 8
  T xi2, nt, nK4, up, dn, di;      // 2 xi, -2 xi / 3, -K / 4, 1 - xi, -(1 + xi), -2 xi
  T Gamma, g0, g1, g2;             // xi / 2, (xi + 1) / 4, (xi - 1) / 4
  T two, ntwo, third, nthird, nhalf;
};

// One colloid.  X, V, W: current state.  Xb, Vb, Wb: the state used when the
// post-collision populations now in memory were produced; the bounce-back of
// their streaming uses it.  acc: FP64 sums of the running step (F_hyd, T_hyd,
// F_lc, T_lc); Fh..Tlc: last completed step; imp/aimp: momentum received.
struct DevColloid {
  double X[3], V[3], W[3];
  double Xb[3], Vb[3], Wb[3];
  double a0, w, M, I;
  double Fext[3], Text[3];  // external force and torque
  int anchoring, mobile, strong, pad;
  double wfac;     // weight of Q0 in the surface value: w / (K + w), 1 for strong anchoring
  float ws[2];     // wfac and X as sums of two floats (48 bits), for the FP32 surface values
  float Xs[3][2];
  double acc[24];  // step sums: F_hyd, T_hyd, F_lc, T_lc, then the link drag tensors zv, zw (6 each, xx xy xz yy yz zz)
  double Fh[3], Th[3], Flc[3], Tlc[3];
  double imp[3], aimp[3];
  double rdp[3];  // momentum exchanged by the running re-discretisation
  // mobile colloids: the position of the last search for changed nodes and the
  // least distance of a node from the surface then; until the colloid has moved
  // that far no node can change (0: not searched yet)
  double Xref[3], margin;
};

__host__ __device__ inline void split_position(DevColloid& C) {
  for (int a = 0; a < 3; ++a) {
    C.Xs[a][0] = (float)C.X[a];
    C.Xs[a][1] = (float)(C.X[a] - (double)C.Xs[a][0]);
  }
}

// Per-box state flags kept on the device (the step kernels flip the buffer
// parities without a host round trip).
struct DevState {
  int fpar;       // f[fpar] holds the current populations
  int qpar;       // Q[qpar] holds the current order parameter
  int pre_valid;  // f[fpar] holds pre-collision values: next collide reads them in place
  int err;        // sticky error bits (1: link list overflow, 2: change list overflow, 4: overlap, 8: contact)
  int nchg;       // nodes whose solid/fluid status changes after the colloid update of this step
  int scan;       // 1: a mobile colloid has moved past its margin; search for changed nodes
  long long step;
  // first contact since the host last read it (see resolve_contacts): the
  // step, the colloid and its partner (-1: a z wall); cstep < 0: none
  long long cstep;
  int ccol, cpartner;
};

struct DevBox {
  int nx, ny, nz, wall_z;
  int pair;             // 1: FP32 box of even width (two-node paths of the stress kernel and the Q update)
  int nmobile;          // mobile colloids in the box (the colloid update tests contacts when > 0)
  int N, ncol;
  int nlinks_cap, chg_cap;
  int* chg;             // change list: (node, colloid << 1 | uncovered) pairs
  void* f[2];
  void* Q[2];
  // FP32 storage only (null for FP64): the BF16 remainder of each stored Q
  // component, so that hi + lo carries the increments that rounding hi alone
  // would drop (compensated storage; 5 comps, same layout as Q)
  __nv_bfloat16* Qlo[2];
  void* u;
  void* F;
  void* H;              // molecular field of the current Q at fluid nodes (5 comps), written by the stress kernels
  void* P;              // chemical stress at fluid nodes (9 comps, row-major P_ab), stored-stress variant only
  uint8_t* mask;
  DevColloid* col;
  DevState* st;
  int* gerr;            // error words of the box's group: [0] wait gave up, [1] contact in some box
  int* nlinks;          // device count of boundary links
  // fluid nodes next to a solid or wall (mask bit NEAR) and the other nodes of
  // their pairs (near_member), in node order: device count, capacity (a bound on
  // the count over the box's motion), counts per block of k_rediscretise
  int* nnear;
  int* near_node;
  int* near_cnt;
  int near_cap;
  int pad1;
  int* link_node;       // boundary links of this box, sorted by (colloid, node, dir)
  int8_t* link_dir;
  int8_t* link_col;
  DevParams p;
  PhysT<float> pf;
  PhysT<double> pd;
  LcK<double> kd;
  LcPairT<float> kp;    // written on the device (k_pair_constants)
};

// FP32 boxes of even width run the two-node paths of the stress kernel and
// the Q update over tiles 64 nodes wide (those phases' tile lists step x by
// 64): a lane holds two nodes, which the packed FP32x2 instructions evaluate
// at once.
__host__ __device__ __forceinline__ bool pair_width(int nx, bool fp32) { return fp32 && nx % 2 == 0; }
__device__ __forceinline__ bool pair_box(const DevBox& B) { return B.pair != 0; }

template <typename T>
__device__ __forceinline__ const PhysT<T>& phys(const DevBox& B);
template <>
__device__ __forceinline__ const PhysT<float>& phys<float>(const DevBox& B) { return B.pf; }
template <>
__device__ __forceinline__ const PhysT<double>& phys<double>(const DevBox& B) { return B.pd; }

// ---------------------------------------------------------------------------
// Small helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }
__device__ __forceinline__ int wrapn(int v, int n) {
  int r = v % n;
  return r < 0 ? r + n : r;
}

// Orders doubles (no NaN) as integers: an FP64 comparison takes a slot of the
// FP64 pipe (one instruction per 64 cycles for a warp), these do not.
__device__ __forceinline__ bool f64_ge(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return (x ^ ((x >> 63) & 0x7fffffffffffffffll)) >= (y ^ ((y >> 63) & 0x7fffffffffffffffll));
}

// Minimum-image displacement r - X along one axis (FP64, round-to-nearest
// operations only, matching a plain C evaluation).
__device__ __forceinline__ double minimg(double d, int L, bool periodic) {
  if (!periodic) return d;
  const double h = 0.5 * (double)L;
  if (f64_ge(d, h)) d = __dsub_rn(d, (double)L);
  else if (!f64_ge(d, -h)) d = __dadd_rn(d, (double)L);
  return d;
}

__device__ __forceinline__ void disp(const DevBox& B, double x, double y, double z, const double* X, double d[3]) {
  d[0] = minimg(__dsub_rn(x, X[0]), B.nx, true);
  d[1] = minimg(__dsub_rn(y, X[1]), B.ny, true);
  d[2] = minimg(__dsub_rn(z, X[2]), B.nz, !B.wall_z);
}

// Solid test of Sec. 2.2: |r - X|^2 < a0^2, evaluated as dx*dx + dy*dy + dz*dz
// left to right with no fused multiply-add, so that it agrees bit for bit with
// a plain FP64 C evaluation.
__device__ __forceinline__ bool inside_colloid(const DevBox& B, int x, int y, int z, const DevColloid& C) {
  double d[3];
  disp(B, (double)x, (double)y, (double)z, C.X, d);
  double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
  return r2 < __dmul_rn(C.a0, C.a0);
}

// Compensated storage of Q in FP32: a value v (FP64) is kept as hi = RN32(v)
// and lo = RNbf16(v - hi); the stored value is hi + lo.
__device__ __forceinline__ void split_q(double v, float& hi, __nv_bfloat16& lo) {
  hi = (float)v;
  lo = __double2bfloat16(v - (double)hi);
}

// hi + lo + d carried into a new (hi, lo): the exact sum hi + s of
// s = lo + d by Knuth's branch-free two-sum (hi' = RN(hi + s) and the exact
// error of that addition), the error then rounded to BF16.
__device__ __forceinline__ void add_compensated(float hi, float lo, float d, float& hi_out, __nv_bfloat16& lo_out) {
  const float s = lo + d;
  const float h = __fadd_rn(hi, s);
  const float bb = __fsub_rn(h, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(h, bb)), __fsub_rn(s, bb));
  hi_out = h;
  lo_out = __float2bfloat16_rn(err);
}

// Stored value of component k of node i of the current Q (hi + lo for FP32).
template <typename T>
__device__ __forceinline__ double load_q(const DevBox& B, int i, int k) {
  const int qpar = B.st->qpar;
  const size_t o = (size_t)k * B.N + i;
  if constexpr (sizeof(T) == 4)
    return (double)static_cast<const float*>(B.Q[qpar])[o] + (double)__bfloat162float(B.Qlo[qpar][o]);
  else
    return static_cast<const double*>(B.Q[qpar])[o];
}

// Q entry (a,b) of the 5-component storage.
template <typename T>
__device__ __forceinline__ T qab(const T* q, int a, int b) {
  if (a > b) { int t = a; a = b; b = t; }
  if (a == 0) return b == 0 ? q[0] : (b == 1 ? q[1] : q[2]);
  if (a == 1) return b == 1 ? q[3] : q[4];
  return -q[0] - q[3];
}

// Whether every eigenvalue of the symmetric traceless Q lies below t, decided
// in FP32 where that is safe: 1 yes, 0 no, -1 too close to call.  t I - Q is
// positive definite exactly when its three leading principal minors are
// positive (Sylvester's criterion); with M the sum of |t| and the |entries|,
// the FP32 evaluation (inputs rounded) of the minors is within 10 u M,
// 40 u M^2 and 150 u M^3 of the exact ones (u = 6e-8), so a minor further than
// the margins below from zero has its true sign.  FP64 runs at 1/64 of the
// FP32 rate on this GPU, and almost every node is far from the threshold.
__device__ __forceinline__ int below_f32(const float q[5], float t) {
  const float m00 = t - q[0], m11 = t - q[3], m22 = t + q[0] + q[3];
  const float M = fabsf(t) + fabsf(q[0]) + fabsf(q[1]) + fabsf(q[2]) + fabsf(q[3]) + fabsf(q[4]);
  if (!(M < 1e9f)) return -1;
  const float e1 = 1e-6f * M, e2 = 4e-6f * M * M, e3 = 1.6e-5f * M * M * M;
  if (m00 < -e1) return 0;
  if (!(m00 > e1)) return -1;
  const float p2 = m00 * m11 - q[1] * q[1];
  if (p2 < -e2) return 0;
  if (!(p2 > e2)) return -1;
  const float det = m00 * (m11 * m22 - q[4] * q[4]) - q[1] * (q[1] * m22 + q[4] * q[2]) - q[2] * (q[1] * q[4] + m11 * q[2]);
  if (det < -e3) return 0;
  return det > e3 ? 1 : -1;
}

// Sum and first moments of the 19 deviations in FP64, through the sums and
// differences of opposite directions (39 additions instead of the 76 of the
// 19 x 4 products; FP64 issue bounds the kernels that call it).
template <typename S, typename V>
__device__ __forceinline__ void pair_moments(const V v[NQ], S& sum, S m[3]) {
  sum = v[0];
  m[0] = m[1] = m[2] = S(0);
#pragma unroll
  for (int q = 1; q < NQ; q += 2) {
    const S a = v[q], b = v[q + 1], d = a - b;
    sum += a + b;
    if (cx(q)) m[0] += cx(q) > 0 ? d : -d;
    if (cy(q)) m[1] += cy(q) > 0 ? d : -d;
    if (cz(q)) m[2] += cz(q) > 0 ? d : -d;
  }
}
__device__ __forceinline__ void moments_f64(const double df[NQ], double& drho, double m[3]) {
  pair_moments<double>(df, drho, m);
}
// FP32 deviations: added as 64-bit integers at 2^-56 of the largest, which
// loses less than FP64 additions (2^-53 of the partial sums), and rounded to
// FP64 by integer instructions: no FP64 operation where there were 58, then 4
// and 4 conversions; infinities and NaN take the FP64 sums.
// F: a force whose half is added to the momentum.
__device__ __forceinline__ void moments_f64(const double df[NQ], const double F[3], double& drho, double m[3]) {
  pair_moments<double>(df, drho, m);
  for (int a = 0; a < 3; ++a) m[a] += 0.5 * F[a];
}
__device__ __forceinline__ void moments_f64(const float df[NQ], const float F[3], double& drho, double m[3]) {
  unsigned top = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) top = max(top, __float_as_uint(df[q]) & 0x7fffffffu);
#pragma unroll
  for (int a = 0; a < 3; ++a) top = max(top, __float_as_uint(F[a]) & 0x7fffffffu);
  if (top >= 0x7f800000u) {
    pair_moments<double>(df, drho, m);
    for (int a = 0; a < 3; ++a) m[a] += 0.5 * (double)F[a];
    return;
  }
  const int k = 182 - (int)(top >> 23);  // |df| 2^k < 2^56: 20 of them and the force fit 63 bits
  long long v[NQ], s, ms[3];
#pragma unroll
  for (int q = 0; q < NQ; ++q) v[q] = f32_to_fixed(df[q], k);
  pair_moments<long long>(v, s, ms);
  drho = fixed_to_f64(s, k);
#pragma unroll
  for (int a = 0; a < 3; ++a) m[a] = fixed_to_f64(ms[a] + f32_to_fixed(F[a], k - 1), k);
}
__device__ __forceinline__ void moments_f64(const float df[NQ], double& drho, double m[3]) {
  const float none[3] = {0.f, 0.f, 0.f};
  moments_f64(df, none, drho, m);
}

// The stored Q of node i rounded to FP32 (for decisions taken in FP32).
template <typename T>
__device__ __forceinline__ void load_q_f32(const DevBox& B, int qpar, int i, float q[5]) {
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const size_t o = (size_t)k * B.N + i;
    if constexpr (sizeof(T) == 4)
      q[k] = static_cast<const float*>(B.Q[qpar])[o] + __bfloat162float(B.Qlo[qpar][o]);
    else
      q[k] = (float)static_cast<const double*>(B.Q[qpar])[o];
  }
}

__device__ __forceinline__ double to_f64(float v) { return f32_to_f64(v); }
__device__ __forceinline__ double to_f64(double v) { return v; }

template <typename T>
__device__ __forceinline__ T ldg(const T* p) { return __ldg(p); }

// Minimum-image displacement and rigid velocity in the kernels' arithmetic
// type (used by the bounce-back of the LB kernel; the solid test itself is
// always FP64).
template <typename T>
__device__ __forceinline__ T minimg_t(T d, int L, bool periodic) {
  if (!periodic) return d;
  const T h = T(0.5) * T(L);
  if (d >= h) d -= T(L);
  else if (d < -h) d += T(L);
  return d;
}

template <typename T>
__device__ __forceinline__ void rigid_velocity_t(const DevBox& B, T x, T y, T z, const double* X, const double* V,
                                                 const double* W, T u[3]) {
  const T d0 = minimg_t(x - T(X[0]), B.nx, true);
  const T d1 = minimg_t(y - T(X[1]), B.ny, true);
  const T d2 = minimg_t(z - T(X[2]), B.nz, !B.wall_z);
  const T w0 = T(W[0]), w1 = T(W[1]), w2 = T(W[2]);
  u[0] = T(V[0]) + w1 * d2 - w2 * d1;
  u[1] = T(V[1]) + w2 * d0 - w0 * d2;
  u[2] = T(V[2]) + w0 * d1 - w1 * d0;
}

// Rigid-body velocity V + W x d.
__device__ __forceinline__ void rigid_velocity(const double* V, const double* W, const double d[3], double u[3]) {
  u[0] = V[0] + W[1] * d[2] - W[2] * d[1];
  u[1] = V[1] + W[2] * d[0] - W[0] * d[2];
  u[2] = V[2] + W[0] * d[1] - W[1] * d[0];
}

// Principal eigenvector of a symmetric traceless 3x3 matrix (5-component
// storage), from the closed-form trigonometric eigenvalue of a symmetric 3x3
// matrix (Smith, CACM 1961) and a cross product of two rows of (A - l I).
// FP64: the eigenvalue of the FP32 evaluation refined by two Newton steps on
// the characteristic polynomial det(A - l I) = -l^3 + (Tr A^2 / 2) l + det A
// (no FP64 transcendental functions, the slope in FP32), then the FP64 cross
// products.  One warp runs this chain per 32 nodes next to a planar colloid, and
// in a small box the step waits for it, so FP64 divisions and square roots are
// kept out.  The seed is 6e-8 / g off for a relative gap g to the second
// eigenvalue, and a step leaves the square of the error over g: to rounding
// for g > 0.05 (measured 1e-15), but two steps overshoot at g ~ 1e-3 and below.
// Where the slope, 3 l^2 - Tr A^2 / 2 ~ g, is small (a texture that is nearly
// uniaxial with negative order, as in defect cores), or A is so small or large
// that FP32 loses it, Jacobi rotations give the direction (1e-16 / g off).
template <typename T>
__device__ void principal_dir(const T* q, T n[3]);

// One rotation of the cyclic Jacobi method (Golub and Van Loan) that zeroes
// a_pq of a symmetric 3x3 matrix: r the third index, u and v columns p and q of
// the eigenvectors.
__device__ __forceinline__ void jacobi_rotate(double& app, double& aqq, double& apq, double& arp, double& arq,
                                              double u[3], double v[3]) {
  if (apq == 0.0) return;
  const double th = (aqq - app) / (2.0 * apq);
  const double t = copysign(1.0, th) / (fabs(th) + sqrt(th * th + 1.0));
  const double c = rsqrt(t * t + 1.0), s = t * c;
  app -= t * apq;
  aqq += t * apq;
  apq = 0.0;
  const double x = arp, y = arq;
  arp = c * x - s * y;
  arq = s * x + c * y;
  for (int k = 0; k < 3; ++k) {
    const double p = u[k], q = v[k];
    u[k] = c * p - s * q;
    v[k] = s * p + c * q;
  }
}

// Principal direction by Jacobi rotations (the matrix scaled to size 1).
inline __device__ __noinline__ void principal_dir_jacobi(const double* q, double n[3]) {
  double m = 0.0;
  for (int k = 0; k < 5; ++k) m = fmax(m, fabs(q[k]));
  const double sc = 1.0 / m;
  double a00 = q[0] * sc, a01 = q[1] * sc, a02 = q[2] * sc, a11 = q[3] * sc, a12 = q[4] * sc, a22 = -a00 - a11;
  double u[3] = {1.0, 0.0, 0.0}, v[3] = {0.0, 1.0, 0.0}, w[3] = {0.0, 0.0, 1.0};
  for (int sweep = 0; sweep < 8 && fabs(a01) + fabs(a02) + fabs(a12) > 1e-18; ++sweep) {
    jacobi_rotate(a00, a11, a01, a02, a12, u, v);
    jacobi_rotate(a00, a22, a02, a01, a12, u, w);
    jacobi_rotate(a11, a22, a12, a01, a02, v, w);
  }
  const double* e = a00 >= a11 ? (a00 >= a22 ? u : w) : (a11 >= a22 ? v : w);
  for (int k = 0; k < 3; ++k) n[k] = e[k];
}

// False: the two largest eigenvalues are too close for the Newton steps.
__device__ __forceinline__ bool principal_lambda_f64(const double* q, double& lam) {
  const double a00 = q[0], a01 = q[1], a02 = q[2], a11 = q[3], a12 = q[4], a22 = -q[0] - q[3];
  // FP32 seed: the largest eigenvalue by the trigonometric formula
  const float f00 = (float)q[0], f01 = (float)q[1], f02 = (float)q[2], f11 = (float)q[3], f12 = (float)q[4];
  const float f22 = -f00 - f11;
  const float p1 = f01 * f01 + f02 * f02 + f12 * f12;
  const float p2 = f00 * f00 + f11 * f11 + f22 * f22 + 2.f * p1;
  float lam32 = 0.f;
  if (p2 > 0.f) {
    const float pp = sqrtf(p2 / 6.f), ip = 1.f / pp;
    const float b00 = f00 * ip, b01 = f01 * ip, b02 = f02 * ip, b11 = f11 * ip, b12 = f12 * ip, b22 = f22 * ip;
    float r = (b00 * (b11 * b22 - b12 * b12) - b01 * (b01 * b22 - b12 * b02) + b02 * (b01 * b12 - b11 * b02)) / 2.f;
    r = fminf(1.f, fmaxf(-1.f, r));
    lam32 = 2.f * pp * cosf(acosf(r) / 3.f);
  }
  const double t2 = 0.5 * (a00 * a00 + a11 * a11 + a22 * a22 + 2.0 * (a01 * a01 + a02 * a02 + a12 * a12));
  const double det = a00 * (a11 * a22 - a12 * a12) - a01 * (a01 * a22 - a12 * a02) + a02 * (a01 * a12 - a11 * a02);
  lam = f32_to_f64(lam32);
  const float t2f = (float)t2;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const double f = (t2 - lam * lam) * lam + det;
    const float df = (float)(t2 - 3.0 * lam * lam);
    if (it == 0 && !(df < -0.06f * t2f && t2f > 1e-30f && t2f < 1e30f)) return false;
    lam -= f * f32_to_f64(1.f / df);
  }
  return true;
}

// 1/sqrt(v) in FP64 from the FP32 estimate and Newton steps (FP32 storage:
// one, relative error ~1e-14; FP64 storage: two, to rounding).
template <int STEPS>
__device__ __forceinline__ double rsqrt_f64(double v) {
  double r = f32_to_f64(rsqrtf((float)v));
#pragma unroll
  for (int k = 0; k < STEPS; ++k) r = r * (1.5 - 0.5 * v * r * r);
  return r;
}

template <typename T>
__device__ void principal_dir(const T* q, T n[3]) {
  T a00 = q[0], a01 = q[1], a02 = q[2], a11 = q[3], a12 = q[4], a22 = -q[0] - q[3];
  T p1 = a01 * a01 + a02 * a02 + a12 * a12;
  T p2 = a00 * a00 + a11 * a11 + a22 * a22 + T(2) * p1;
  if (!(p2 > T(0))) {
    n[0] = T(1); n[1] = T(0); n[2] = T(0);
    return;
  }
  T lam;
  if constexpr (sizeof(T) == 8) {
    if (!principal_lambda_f64(q, lam)) {
      principal_dir_jacobi(q, n);
      return;
    }
  } else {
    T p = sqrt(p2 / T(6));
    T b00 = a00 / p, b01 = a01 / p, b02 = a02 / p, b11 = a11 / p, b12 = a12 / p, b22 = a22 / p;
    T det = b00 * (b11 * b22 - b12 * b12) - b01 * (b01 * b22 - b12 * b02) + b02 * (b01 * b12 - b11 * b02);
    T r = det / T(2);
    r = r < T(-1) ? T(-1) : (r > T(1) ? T(1) : r);
    T phi = acos(r) / T(3);
    lam = T(2) * p * cos(phi);
  }
  T r0[3] = {a00 - lam, a01, a02}, r1[3] = {a01, a11 - lam, a12}, r2[3] = {a02, a12, a22 - lam};
  if constexpr (sizeof(T) == 8) {
    // the longest of the three row products, found in FP32, then that one in
    // FP64 (the others would be 24 of the chain's 110 FP64 instructions)
    const float f0[3] = {(float)r0[0], (float)r0[1], (float)r0[2]}, f1[3] = {f0[1], (float)r1[1], (float)r1[2]};
    const float f2[3] = {f0[2], f1[2], (float)r2[2]};
    auto len = [](const float* u, const float* v) {
      const float x = u[1] * v[2] - u[2] * v[1], y = u[2] * v[0] - u[0] * v[2], z = u[0] * v[1] - u[1] * v[0];
      return x * x + y * y + z * z;
    };
    const float l0 = len(f0, f1), l1 = len(f0, f2), l2 = len(f1, f2);
    if (fmaxf(l0, fmaxf(l1, l2)) > 1e-24f) {
      const bool u1 = l2 > l0 && l2 > l1, v2 = u1 || l1 > l0;  // rows (0,1), (0,2) or (1,2)
      const T u[3] = {u1 ? r1[0] : r0[0], u1 ? r1[1] : r0[1], u1 ? r1[2] : r0[2]};
      const T v[3] = {v2 ? r2[0] : r1[0], v2 ? r2[1] : r1[1], v2 ? r2[2] : r1[2]};
      n[0] = u[1] * v[2] - u[2] * v[1];
      n[1] = u[2] * v[0] - u[0] * v[2];
      n[2] = u[0] * v[1] - u[1] * v[0];
      const T sc = rsqrt_f64<2>(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
      n[0] *= sc; n[1] *= sc; n[2] *= sc;
      return;
    }
  }
  T c0[3] = {r0[1] * r1[2] - r0[2] * r1[1], r0[2] * r1[0] - r0[0] * r1[2], r0[0] * r1[1] - r0[1] * r1[0]};
  T c1[3] = {r0[1] * r2[2] - r0[2] * r2[1], r0[2] * r2[0] - r0[0] * r2[2], r0[0] * r2[1] - r0[1] * r2[0]};
  T c2[3] = {r1[1] * r2[2] - r1[2] * r2[1], r1[2] * r2[0] - r1[0] * r2[2], r1[0] * r2[1] - r1[1] * r2[0]};
  T n0 = c0[0] * c0[0] + c0[1] * c0[1] + c0[2] * c0[2];
  T n1 = c1[0] * c1[0] + c1[1] * c1[1] + c1[2] * c1[2];
  T n2 = c2[0] * c2[0] + c2[1] * c2[1] + c2[2] * c2[2];
  T nn = n0;
#pragma unroll
  for (int a = 0; a < 3; ++a) n[a] = c0[a];
  if (n1 > nn) {
    nn = n1;
#pragma unroll
    for (int a = 0; a < 3; ++a) n[a] = c1[a];
  }
  if (n2 > nn) {
    nn = n2;
#pragma unroll
    for (int a = 0; a < 3; ++a) n[a] = c2[a];
  }
  if (!(nn > T(0))) {
    n[0] = T(1); n[1] = T(0); n[2] = T(0);
    return;
  }
  const T s = T(1) / sqrt(nn);
  n[0] *= s; n[1] *= s; n[2] *= s;
}

// Surface order Q0 = S0 (n0 n0 - delta/3) (Eq. 7) at solid node (sx,sy,sz) of
// colloid c (c < 0: a z wall, homeotropic along z).  Homeotropic: n0 = unit
// normal s at the solid node; planar: n0 = projection of the fluid node's
// director (principal eigenvector of qf) on the plane normal to s.
template <typename T>
__device__ void surface_q0(const DevBox& B, int c, int sx, int sy, int sz, const T* qf, T q0[5]) {
  T n[3];
  if (c < 0) {
    n[0] = T(0); n[1] = T(0); n[2] = T(1);
  } else {
    const DevColloid& C = B.col[c];
    // the normal only orients Q0: the minimum-image offset is taken in FP64
    // (positions up to the box size), its normalisation in T
    double dd[3];
    disp(B, (double)sx, (double)sy, (double)sz, C.X, dd);
    const T d0 = T(dd[0]), d1 = T(dd[1]), d2 = T(dd[2]);
    const T r = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
    T s[3] = {d0 / r, d1 / r, d2 / r};
    if (C.anchoring == 0) {
      n[0] = s[0]; n[1] = s[1]; n[2] = s[2];
    } else {
      T nf[3];
      principal_dir(qf, nf);
      T ns = nf[0] * s[0] + nf[1] * s[1] + nf[2] * s[2];
      T p[3] = {nf[0] - ns * s[0], nf[1] - ns * s[1], nf[2] - ns * s[2]};
      T pn = sqrt(p[0] * p[0] + p[1] * p[1] + p[2] * p[2]);
      const T tiny = sizeof(T) == 8 ? T(1e-12) : T(1e-6);
      if (pn < tiny) {  // director along the normal: tangent s x e_k, k least aligned with s
        int k = 0;
        if (fabs(s[1]) < fabs(s[k])) k = 1;
        if (fabs(s[2]) < fabs(s[k])) k = 2;
        T e[3] = {T(0), T(0), T(0)};
        e[k] = T(1);
        p[0] = s[1] * e[2] - s[2] * e[1];
        p[1] = s[2] * e[0] - s[0] * e[2];
        p[2] = s[0] * e[1] - s[1] * e[0];
        pn = sqrt(p[0] * p[0] + p[1] * p[1] + p[2] * p[2]);
      }
      n[0] = p[0] / pn; n[1] = p[1] / pn; n[2] = p[2] / pn;
    }
  }
  T S0 = phys<T>(B).S0;
  T third = T(1) / T(3);
  q0[0] = S0 * (n[0] * n[0] - third);
  q0[1] = S0 * n[0] * n[1];
  q0[2] = S0 * n[0] * n[2];
  q0[3] = S0 * (n[1] * n[1] - third);
  q0[4] = S0 * n[1] * n[2];
}

// Value standing in for a solid (or wall) neighbour of a fluid node in the
// finite-difference stencil.  Strong anchoring: Q0.  Finite strength w: the
// minimiser of (w/2)|Qs - Q0|^2 + (K/2)|Qs - qf|^2, (K qf + w Q0)/(K + w).
// surf (if non-null) accumulates (w/2)|Qs - Q0|^2 (9 entries).
template <typename T>
__device__ void ghost_q(const DevBox& B, int c, int sx, int sy, int sz, const T* qf, T qs[5], double* surf) {
  T q0[5];
  surface_q0(B, c, sx, sy, sz, qf, q0);
  bool strong = (c < 0) || B.col[c].strong;
  if (strong) {
#pragma unroll
    for (int k = 0; k < 5; ++k) qs[k] = q0[k];
    return;
  }
  T w = T(B.col[c].w), K = phys<T>(B).K;
  T inv = T(1) / (K + w);
#pragma unroll
  for (int k = 0; k < 5; ++k) qs[k] = (K * qf[k] + w * q0[k]) * inv;
  if (surf) {
    double t = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        double dd = (double)qab(qs, a, b) - (double)qab(q0, a, b);
        t += dd * dd;
      }
    *surf += 0.5 * (double)B.col[c].w * t;
  }
}

// Neighbour indices of node (x,y,z) along +x,-x,+y,-y,+z,-z; -1 beyond a wall.
__device__ __forceinline__ void face_neighbours(const DevBox& B, int x, int y, int z, int nb[6], int cz6[2]) {
  int nx = B.nx, ny = B.ny, nz = B.nz;
  int xp = x + 1 == nx ? 0 : x + 1, xm = x == 0 ? nx - 1 : x - 1;
  int yp = y + 1 == ny ? 0 : y + 1, ym = y == 0 ? ny - 1 : y - 1;
  int zp, zm;
  if (B.wall_z) {
    zp = z + 1 < nz ? z + 1 : -1;
    zm = z > 0 ? z - 1 : -1;
  } else {
    zp = z + 1 == nz ? 0 : z + 1;
    zm = z == 0 ? nz - 1 : z - 1;
  }
  int row = nx * (y + ny * z);
  nb[0] = xp + row;
  nb[1] = xm + row;
  nb[2] = x + nx * (yp + ny * z);
  nb[3] = x + nx * (ym + ny * z);
  nb[4] = zp < 0 ? -1 : x + nx * (y + ny * zp);
  nb[5] = zm < 0 ? -1 : x + nx * (y + ny * zm);
  cz6[0] = zp;
  cz6[1] = zm;
}

// Q at a fluid node and its six face neighbours (surface values for solid or
// wall neighbours).  Returns the centre in qi, neighbours in qn[6][5].
template <typename T>
__device__ __forceinline__ void gather_q(const DevBox& B, const T* __restrict__ Q, int x, int y, int z, int i,
                                         uint8_t m, T qi[5], T qn[6][5], double* surf) {
  const int N = B.N;
#pragma unroll
  for (int k = 0; k < 5; ++k) qi[k] = ldg(Q + (size_t)k * N + i);
  int nb[6], zz[2];
  face_neighbours(B, x, y, z, nb, zz);
  if (!(m & NEAR)) {
#pragma unroll
    for (int d = 0; d < 6; ++d)
#pragma unroll
      for (int k = 0; k < 5; ++k) qn[d][k] = ldg(Q + (size_t)k * N + nb[d]);
    return;
  }
  const int nx = B.nx, ny = B.ny;
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    int j = nb[d];
    int c = -1;
    bool solid;
    if (j < 0) {
      solid = true;
    } else {
      uint8_t mj = B.mask[j] & IDMASK;
      solid = mj != 0;
      c = (int)mj - 1;
    }
    if (!solid) {
#pragma unroll
      for (int k = 0; k < 5; ++k) qn[d][k] = ldg(Q + (size_t)k * N + j);
    } else {
      int sx = x, sy = y, sz = z;
      if (d == 0) sx = x + 1 == nx ? 0 : x + 1;
      if (d == 1) sx = x == 0 ? nx - 1 : x - 1;
      if (d == 2) sy = y + 1 == ny ? 0 : y + 1;
      if (d == 3) sy = y == 0 ? ny - 1 : y - 1;
      if (d == 4) sz = zz[0];
      if (d == 5) sz = zz[1];
      ghost_q(B, c, sx, sy, sz, qi, qn[d], surf);
    }
  }
}

// Surface order Q0 (Eq. 7) in FP64: the unit normal s at solid node
// (sx, sy, sz) of colloid c (c < 0: a z wall, n0 = z); homeotropic n0 = s,
// planar n0 = nf projected on the plane normal to s (nf: the fluid node's
// director), the tie-break s x e_k as surface_q0.
template <typename T>
__device__ __forceinline__ void surface_q0_near(const DevBox& B, int c, int sx, int sy, int sz, const double nf[3],
                                                double q0[5]) {
  constexpr int ST = sizeof(T) == 8 ? 2 : 1;
  double n[3];
  if (c < 0) {
    n[0] = 0.0; n[1] = 0.0; n[2] = 1.0;
  } else {
    const DevColloid& C = B.col[c];
    double d[3];
    disp(B, (double)sx, (double)sy, (double)sz, C.X, d);
    const double ri = rsqrt_f64<ST>(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    const double sv[3] = {d[0] * ri, d[1] * ri, d[2] * ri};
    if (C.anchoring == 0) {
      n[0] = sv[0]; n[1] = sv[1]; n[2] = sv[2];
    } else {
      const double ns = nf[0] * sv[0] + nf[1] * sv[1] + nf[2] * sv[2];
      double pv[3] = {nf[0] - ns * sv[0], nf[1] - ns * sv[1], nf[2] - ns * sv[2]};
      double p2 = pv[0] * pv[0] + pv[1] * pv[1] + pv[2] * pv[2];
      if (p2 < 1e-24) {  // director along the normal: tangent s x e_k, k least aligned with s
        int k = 0;
        if (fabs(sv[1]) < fabs(sv[k])) k = 1;
        if (fabs(sv[2]) < fabs(sv[k])) k = 2;
        double e[3] = {0.0, 0.0, 0.0};
        e[k] = 1.0;
        pv[0] = sv[1] * e[2] - sv[2] * e[1];
        pv[1] = sv[2] * e[0] - sv[0] * e[2];
        pv[2] = sv[0] * e[1] - sv[1] * e[0];
        p2 = pv[0] * pv[0] + pv[1] * pv[1] + pv[2] * pv[2];
      }
      const double pi = rsqrt_f64<ST>(p2);
      n[0] = pv[0] * pi; n[1] = pv[1] * pi; n[2] = pv[2] * pi;
    }
  }
  const double S0 = B.pd.S0, third = 1.0 / 3.0;
  q0[0] = S0 * (n[0] * n[0] - third);
  q0[1] = S0 * n[0] * n[1];
  q0[2] = S0 * n[0] * n[2];
  q0[3] = S0 * (n[1] * n[1] - third);
  q0[4] = S0 * n[1] * n[2];
}

// a - b rounded, and its rounding error (Knuth's two-sum).
__device__ __forceinline__ float two_diff(float a, float b, float& e) {
  const float t = __fsub_rn(a, b), bb = __fsub_rn(a, t);
  e = __fadd_rn(__fsub_rn(a, __fadd_rn(t, bb)), __fsub_rn(bb, b));
  return t;
}

// w (Q0 - Q) for a homeotropic solid face in FP32 storage, in sums of two
// floats (48 bits; every step below keeps the error of the FP32 operation
// before it): n0 = d / |d| from the split position of the colloid, 1/|d| by one
// corrected estimate, and the difference to Q = qh + ql rounded once at the
// end, as the FP64 evaluation of surface_q0_near rounds it.  The FP64 one is
// some 100 instructions of 64 cycles each for a lone warp, this one as many
// FP32 instructions.
__device__ __forceinline__ void surface_dn_normal(const DevBox& B, const DevColloid& C, const int s[3],
                                                  const float qh[5], const float ql[5], float dn[5]) {
  float dh[3], dl[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int L = a == 0 ? B.nx : (a == 1 ? B.ny : B.nz);
    // node minus X: the minimum image is taken on the integer (exact in FP32),
    // decided on both parts of the difference, then the difference to the high
    // part with its rounding error, which is no zero where X is small beside it
    // (a colloid at a low face of the box)
    const float xh = C.Xs[a][0], xl = C.Xs[a][1];
    int si = s[a];
    float e, t = two_diff((float)si, xh, e);
    if (a < 2 || !B.wall_z) {
      const float h = 0.5f * (float)L;
      if (t - h >= xl - e) si -= L;
      else if (t + h < xl - e) si += L;
    }
    t = two_diff((float)si, xh, e);
    const float low = e - xl;
    dh[a] = t + low;
    dl[a] = (t - dh[a]) + low;
  }
  // |d|^2 = rh + rl
  float ph[3], rl = 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    ph[a] = dh[a] * dh[a];
    rl += fmaf(dh[a], dh[a], -ph[a]) + 2.f * dh[a] * dl[a];
  }
  const float s01 = ph[0] + ph[1], b01 = s01 - ph[0];
  rl += (ph[0] - (s01 - b01)) + (ph[1] - b01);
  const float rh = s01 + ph[2], b2 = rh - s01;
  rl += (s01 - (rh - b2)) + (ph[2] - b2);
  // 1/|d| = r + rc
  const float r = rsqrtf(rh), rr = r * r, re = fmaf(r, r, -rr);
  const float eps = -(fmaf(rr, rh, -1.f) + fmaf(rr, rl, re * rh));
  const float rc = 0.5f * r * eps;
  float nh[3], nl[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float p = dh[a] * r, e = fmaf(dh[a], r, -p) + fmaf(dh[a], rc, dl[a] * r);
    nh[a] = p + e;
    nl[a] = e - (nh[a] - p);
  }
  const float th = 1.f / 3.f, tl = -9.934107e-9f;  // 1/3 - th
  const float S0h = B.pf.S0, S0l = B.pf.S0l, wh = C.ws[0], wl = C.ws[1];
  const int ia[5] = {0, 0, 0, 1, 1}, ib[5] = {0, 1, 2, 1, 2};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int a = ia[k], b = ib[k];
    float ph2 = nh[a] * nh[b], pl = fmaf(nh[a], nh[b], -ph2) + fmaf(nh[a], nl[b], nl[a] * nh[b]);
    if (a == b) {
      const float t = ph2 - th, bb = t - ph2;
      pl += ((ph2 - (t - bb)) + (-th - bb)) - tl;
      ph2 = t;
    }
    // S0 (n n - delta/3) - qh - ql
    const float q = S0h * ph2, qe = fmaf(S0h, ph2, -q) + fmaf(S0h, pl, S0l * ph2);
    const float t = q - qh[k], bb = t - q;
    const float D = t, E = ((q - (t - bb)) + (-qh[k] - bb)) + (qe - ql[k]);
    dn[k] = fmaf(D, wh, fmaf(E, wh, D * wl));
  }
}

// Derivatives from the face-neighbour values: twice the central first
// differences, dq[g][k] = 2 d_g Q_k (the halves are taken into the constants
// of lc_node_d), and the 7-point Laplacian (Sec. 2.2: one stencil at all fluid
// nodes, surface values standing in for solid neighbours).
template <typename T>
__device__ __forceinline__ void derivatives(const T qi[5], const T qn[6][5], T dq[3][5], T lap[5]) {
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    dq[0][k] = qn[0][k] - qn[1][k];
    dq[1][k] = qn[2][k] - qn[3][k];
    dq[2][k] = qn[4][k] - qn[5][k];
    const T n6 = (qn[0][k] + qn[1][k]) + (qn[2][k] + qn[3][k]) + (qn[4][k] + qn[5][k]);
    lap[k] = n6 + T(-6) * qi[k];
  }
}

// All liquid-crystal quantities of one fluid node from its Q, the doubled
// first derivatives dq[g][k] = 2 d_g Q_k and the Laplacian lap[k]:
//   H   = cb Q + A0 g (Q.Q - Tr(Q^2) I/3) + K lap Q - 2 K q0 (C + C^T),
//         cb = -A0(1 - g/3) - A0 g Tr(Q^2) - 4 K q0^2, C_ab = eps_agd d_g Q_db  (Eqs. 1, 2)
//   f'  = A0/2 (1-g/3) Tr Q^2 - A0 g/3 Tr Q^3 + A0 g/4 (Tr Q^2)^2
//         + K/2 |grad Q|^2 + 2 K q0 Q:C + 2 K q0^2 Tr Q^2                        (Eq. 1)
//   P   = f' I + 2 xi (Q + I/3) Q:H - xi (A + A^T) - (2 xi/3) H - E + A - A^T,
//         A = Q H,  E_ab = K <d_a Q, d_b Q> + 2 K q0 sum_gn d_a Q_gn eps_mbg Q_mn  (Eq. 4)
// The algebra is written out in the five stored components with what
// tracelessness gives (off-diagonal Q.Q from two products each, H_zz from H_xx
// and H_yy, the commutator and anticommutator of Q and H from the nine entries
// of Q H): about 290 operations a node against 470 for the 3x3 loops of
// lc_node_f32, which matters where FP64 issue bounds the step (k_stress FP64,
// 64^3: 84-87 % of the FP64 pipe).  The chiral stress term is skipped when
// q0 = 0 (uniform over a box).  FP64 storage only (T = double): FP32 keeps the
// order of lc_node_f32.  chiral: q0 != 0; NEED_P false: the molecular field
// alone.
template <typename T, bool NEED_P = true>
__device__ __forceinline__ void lc_node_d(const LcK<T>& P, bool chiral, const T qi[5], const T dq[3][5],
                                          const T lap[5], T h[5], T p[9], T* fprime) {
  const T a = qi[0], b = qi[1], c = qi[2], d = qi[3], e = qi[4];
  const T f = -a - d;
  const T nb = -b, nc = -c, ne = -e;
  // Q.Q: (xx, xy, xz, yy, yz, zz)
  const T bb = b * b, cc = c * c, ee = e * e;
  const T s0 = a * a + (bb + cc), s3 = d * d + (bb + ee), s5 = f * f + (cc + ee);
  const T s1 = c * e + nb * f, s2 = b * e + nc * d, s4 = b * c + ne * a;
  const T trq2 = s0 + s3 + s5;
  // 2 (C_ab + C_ba) off the diagonal, 2 C_aa on it
  const T* X = dq[0];
  const T* Y = dq[1];
  const T* Z = dq[2];
  const T tx = X[0] + X[3], ty = Y[0] + Y[3], tz = Z[0] + Z[3];  // minus the zz components
  const T c0 = Y[2] - Z[1], c3 = Z[1] - X[4], c5 = X[4] - Y[2];
  const T c1 = (Y[4] - Z[3]) + (Z[0] - X[2]);
  const T c2 = (X[1] - Z[4]) - (Y[0] + ty);
  const T c4 = (Z[2] - Y[1]) + (X[3] + tx);
  const T cb = P.c_lin + P.nA0g * trq2;
  // the bulk terms are O(A0 q^2) and cancel near equilibrium: they are summed
  // among themselves first, each product but one unrounded, so that the small
  // gradient terms are not rounded at their size
  h[0] = T(P.nA3 * trq2 + T(cb * a + P.A0g * s0)) + T(P.K * lap[0] + P.n2Kq0 * c0);
  h[1] = T(cb * b + P.A0g * s1) + T(P.K * lap[1] + P.nKq0 * c1);
  h[2] = T(cb * c + P.A0g * s2) + T(P.K * lap[2] + P.nKq0 * c2);
  h[3] = T(P.nA3 * trq2 + T(cb * d + P.A0g * s3)) + T(P.K * lap[3] + P.n2Kq0 * c3);
  h[4] = T(cb * e + P.A0g * s4) + T(P.K * lap[4] + P.nKq0 * c4);
  if constexpr (!NEED_P) return;
  const T hz = -h[0] - h[3];
  // <2 d_a Q, 2 d_b Q> for the six pairs (double contraction over the five
  // stored components of two traceless symmetric tensors)
  auto dd = [&](const T* u, const T* v, T tu, T tv) {
    const T on = u[0] * v[0] + (u[3] * v[3] + tu * tv);
    return T(on + P.two * T(u[1] * v[1] + (u[2] * v[2] + u[4] * v[4])));
  };
  const T e0 = dd(X, X, tx, tx), e1 = dd(X, Y, tx, ty), e2 = dd(X, Z, tx, tz);
  const T e3 = dd(Y, Y, ty, ty), e4 = dd(Y, Z, ty, tz), e5 = dd(Z, Z, tz, tz);
  const T qc = a * c0 + (d * c3 + (f * c5 + (b * c1 + (c * c2 + e * c4))));  // 2 Q:C
  const T trq3 = a * s0 + (d * s3 + (f * s5 + P.two * T(b * s1 + (c * s2 + e * s4))));
  const T fp = P.f2c * trq2 + (P.nA3 * trq3 + (P.f4c * T(trq2 * trq2) + (P.K8 * (e0 + e3 + e5) + P.Kq0 * qc)));
  // A = Q H
  const T h0 = h[0], h1 = h[1], h2 = h[2], h3 = h[3], h4 = h[4];
  const T a00 = a * h0 + (b * h1 + c * h2), a01 = a * h1 + (b * h3 + c * h4), a02 = a * h2 + (b * h4 + c * hz);
  const T a10 = b * h0 + (d * h1 + e * h2), a11 = b * h1 + (d * h3 + e * h4), a12 = b * h2 + (d * h4 + e * hz);
  const T a20 = c * h0 + (e * h1 + f * h2), a21 = c * h1 + (e * h3 + f * h4), a22 = c * h2 + (e * h4 + f * hz);
  const T qh2 = P.xi2 * (a00 + a11 + a22);
  const T nt = P.nt, nK4 = P.nK4, up = P.up, dn = P.dn, di = P.di;
  const T dg = fp + P.third * qh2;
  const T z1 = qh2 * b + (nt * h1 + nK4 * e1), z2 = qh2 * c + (nt * h2 + nK4 * e2), z4 = qh2 * e + (nt * h4 + nK4 * e4);
  p[0] = qh2 * a + (nt * h0 + (nK4 * e0 + (di * a00 + dg)));
  p[4] = qh2 * d + (nt * h3 + (nK4 * e3 + (di * a11 + dg)));
  p[8] = qh2 * f + (nt * hz + (nK4 * e5 + (di * a22 + dg)));
  p[1] = up * a01 + (dn * a10 + z1);
  p[3] = up * a10 + (dn * a01 + z1);
  p[2] = up * a02 + (dn * a20 + z2);
  p[6] = up * a20 + (dn * a02 + z2);
  p[5] = up * a12 + (dn * a21 + z4);
  p[7] = up * a21 + (dn * a12 + z4);
  if (chiral) {
    // chiral part of E: twice the axial vector of (d_a Q) Q
    const T fd = f - d, af = a - f, da = d - a;
    auto chi = [&](const T* D, T tD, T& p0, T& p1, T& p2) {
      const T m0 = D[3] + tD, m1 = D[0] + tD, m2 = D[0] - D[3];
      p0 = p0 + P.nKq0 * T(D[1] * c + (D[2] * nb + (D[4] * fd + e * m0)));
      p1 = p1 + P.nKq0 * T(D[2] * af + (D[4] * b + (D[1] * ne + nc * m1)));
      p2 = p2 + P.nKq0 * T(b * m2 + (D[1] * da + (D[2] * e + D[4] * nc)));
    };
    chi(X, tx, p[0], p[1], p[2]);
    chi(Y, ty, p[3], p[4], p[5]);
    chi(Z, tz, p[6], p[7], p[8]);
  }
  *fprime = fp;
}

// The same in FP32 (dq2: the doubled first derivatives): H, f' and P by sums
// over the 3x3 matrices, in an order that stays as it is (see lclb_pair.cuh,
// which evaluates two nodes at once in the same order).
template <bool NEED_P>
__device__ __forceinline__ void lc_node_f32(const PhysT<float>& P, const float qi[5], const float dq2[3][5],
                                            const float lap[5], float h[5], float p[9], float* fprime) {
  const float A0 = P.A0, g = P.gamma, K = P.K, q0 = P.q0, xi = P.xi;
  const float third = float(1) / float(3);
  const float A0g = A0 * g, twoKq0 = float(2) * K * q0;
  const float c_lin = -A0 * (float(1) - g * third) - float(4) * K * q0 * q0;  // H: coefficient of Q beyond -A0 g Tr(Q^2)
  const float A0g3 = A0g * third;
  float dq[3][5];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int k = 0; k < 5; ++k) dq[a][k] = 0.5f * dq2[a][k];
  // Q (3x3), D[g] = d_g Q (3x3 each) from the 5 stored components
  float Q[3][3], D[3][3][3], S2[3][3], Cm[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      Q[a][b] = qab(qi, a, b);
#pragma unroll
      for (int gg = 0; gg < 3; ++gg) D[gg][a][b] = qab(dq[gg], a, b);
    }
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a; b < 3; ++b) {
      S2[a][b] = Q[a][0] * Q[0][b] + Q[a][1] * Q[1][b] + Q[a][2] * Q[2][b];
      S2[b][a] = S2[a][b];
    }
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) Cm[a][b] = D[(a + 1) % 3][(a + 2) % 3][b] - D[(a + 2) % 3][(a + 1) % 3][b];
  const float trq2 = S2[0][0] + S2[1][1] + S2[2][2];
  const float cb = c_lin - A0g * trq2;
  const float tq3 = A0g3 * trq2;
  float H[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a; b < 3; ++b) {
      const int k = a == 0 ? b : (a == 1 ? 2 + b : 5);
      const float lp = k < 5 ? lap[k] : -(lap[0] + lap[3]);
      float v = cb * Q[a][b] + A0g * S2[a][b] + K * lp - twoKq0 * (Cm[a][b] + Cm[b][a]);
      if (a == b) v = v - tq3;
      H[a][b] = v;
      H[b][a] = v;
    }
  h[0] = H[0][0]; h[1] = H[0][1]; h[2] = H[0][2]; h[3] = H[1][1]; h[4] = H[1][2];
  if (!NEED_P) return;
  // E_ab = K d_aQ : d_bQ; both factors are symmetric and traceless, so the
  // double contraction over the 5 stored components is
  // A_xx B_xx + A_yy B_yy + A_zz B_zz + 2 (A_xy B_xy + A_xz B_xz + A_yz B_yz)
  // with A_zz = -(A_xx + A_yy)
  float E[3][3], tz[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) tz[a] = dq[a][0] + dq[a][3];
  const float twoK = float(2) * K;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a; b < 3; ++b) {
      const float e = K * (dq[a][0] * dq[b][0] + dq[a][3] * dq[b][3] + tz[a] * tz[b]) +
                  twoK * (dq[a][1] * dq[b][1] + dq[a][2] * dq[b][2] + dq[a][4] * dq[b][4]);
      E[a][b] = e;
      E[b][a] = e;
    }
  const float Kgrad2 = E[0][0] + E[1][1] + E[2][2];  // K |grad Q|^2
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      // the chiral part: sum over g != b of eps(m, b, g) d_a Q_g. . Q_m. (m = 3 - b - g);
      // eps(m, b, g) = +1 for g = b + 1, m = b + 2 and -1 for g = b + 2, m = b + 1 (mod 3)
      const int g1 = (b + 1) % 3, g2 = (b + 2) % 3;
      const float e2 = (D[a][g1][0] * Q[g2][0] + D[a][g1][1] * Q[g2][1] + D[a][g1][2] * Q[g2][2]) -
                   (D[a][g2][0] * Q[g1][0] + D[a][g2][1] * Q[g1][1] + D[a][g2][2] * Q[g1][2]);
      E[a][b] = E[a][b] + twoKq0 * e2;
    }
  float trq3 = float(0), qc = float(0);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      trq3 = trq3 + Q[a][b] * S2[a][b];
      qc = qc + Q[a][b] * Cm[a][b];
    }
  const float fb2 = float(0.5) * A0 * (float(1) - g * third), fb4 = float(0.25) * A0g;
  const float fp = (fb2 * trq2 - A0g3 * trq3) + fb4 * (trq2 * trq2) + float(0.5) * Kgrad2 + twoKq0 * qc +
               (float(2) * K * q0 * q0) * trq2;
  float Am[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) Am[a][b] = Q[a][0] * H[0][b] + Q[a][1] * H[1][b] + Q[a][2] * H[2][b];
  const float qh = Am[0][0] + Am[1][1] + Am[2][2];
  const float twoxi = float(2) * xi, twoxi3 = twoxi * third;
  const float qh2 = twoxi * qh;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      // 2 xi (Q + I/3) Q:H - xi (A + A^T) - (2 xi/3) H - E + A - A^T, plus f' on the diagonal
      float v = qh2 * Q[a][b] - xi * (Am[a][b] + Am[b][a]) - twoxi3 * H[a][b] - E[a][b] + (Am[a][b] - Am[b][a]);
      if (a == b) v = v + (fp + third * qh2);
      p[3 * a + b] = v;
    }
  *fprime = fp;
}

// One node in the storage's arithmetic, from its derivatives or its face
// neighbours.
template <typename T, bool NEED_P = true>
__device__ __forceinline__ void lc_node_dq(const DevBox& B, const T qi[5], const T dq[3][5], const T lap[5], T h[5],
                                           T p[9], T* fprime) {
  if constexpr (sizeof(T) == 4) lc_node_f32<NEED_P>(B.pf, qi, dq, lap, h, p, fprime);
  else lc_node_d<T, NEED_P>(B.kd, B.p.q0 != 0.0, qi, dq, lap, h, p, fprime);
}
template <typename T, bool NEED_P = true>
__device__ __forceinline__ void lc_node(const DevBox& B, const T qi[5], const T qn[6][5], T h[5], T p[9],
                                        T* fprime) {
  T dq[3][5], lap[5];
  derivatives(qi, qn, dq, lap);
  lc_node_dq<T, NEED_P>(B, qi, dq, lap, h, p, fprime);
}

template <typename T>
__device__ __forceinline__ T pos_part(T v) {
  return v > T(0) ? v : T(0);
}

// Increment of Q in one step (Eq. 2) at one node, FP64 storage:
//   co-rotation S = X + X^T - 2 xi (Q + I/3) Tr(QW), X = G (Q + I/3),
//     G = xi D + Omega: 27 products for X instead of 72 for its four factors;
//   upwind fluxes: with the positive and negative parts of the face velocity
//     the six fluxes are one product per neighbour and component plus one
//     with the node's own Q, adv = (self Q_i + sum_d cd[d] Q_d) / 2 (35
//     multiply-adds and 6 selects instead of 30 and 30).
// flow_terms: G (row-major), cd and self from the velocities ui and un of the
// node and its six face neighbours; open[d] = false closes face d (solid or
// wall) to the flux.
template <typename T>
__device__ __forceinline__ void flow_terms(const LcK<T>& P, const T ui[3], const T un[6][3], const bool open[6],
                                           T G[9], T cd[6], T& self) {
  // w[a][b] = 2 d_b u_a
  T w[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) w[i][j] = un[2 * j][i] - un[2 * j + 1][i];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const T uf = ui[k >> 1] + un[k][k >> 1];
    T up = pos_part(uf);
    T dn = uf - up;
    if (!open[k]) up = dn = T(0);
    // + face: outflow up Q_i + dn Q_d; - face: minus (up Q_d + dn Q_i)
    cd[k] = (k & 1) ? T(-up) : dn;
    const T own = (k & 1) ? T(-dn) : up;
    self = k ? T(self + own) : own;
  }
  const T g0 = P.g0, g1 = P.g1, g2 = P.g2;
  G[0] = g0 * w[0][0];
  G[4] = g0 * w[1][1];
  G[8] = g0 * w[2][2];
  G[1] = g1 * w[0][1] + g2 * w[1][0];
  G[3] = g1 * w[1][0] + g2 * w[0][1];
  G[2] = g1 * w[0][2] + g2 * w[2][0];
  G[6] = g1 * w[2][0] + g2 * w[0][2];
  G[5] = g1 * w[1][2] + g2 * w[2][1];
  G[7] = g1 * w[2][1] + g2 * w[1][2];
}

// Twice the advective flux divergence of one component.
template <typename T>
__device__ __forceinline__ T advect(const T cd[6], T self, T q, const T n[6]) {
  T v = self * q;
#pragma unroll
  for (int d = 0; d < 6; ++d) v = v + cd[d] * n[d];
  return v;
}

// FLOW = false: the flow is frozen (u = 0), G and adv are not read.
template <bool FLOW, typename T>
__device__ __forceinline__ void q_increment(const LcK<T>& P, const T qi[5], const T adv[5], const T G[9],
                                            const T h[5], T d5[5]) {
  if constexpr (!FLOW) {
#pragma unroll
    for (int k = 0; k < 5; ++k) d5[k] = P.Gamma * h[k];
    return;
  }
  const T a = qi[0], b = qi[1], c = qi[2], d = qi[3], e = qi[4];
  const T f = -a - d;
  const T at = a + P.third, dt = d + P.third, ft = f + P.third;
  const T tm = P.ntwo * T(a * G[0] + (d * G[4] + (f * G[8] + (b * (G[1] + G[3]) + (c * (G[2] + G[6]) + e * (G[5] + G[7]))))));
  const T x00 = G[0] * at + (G[1] * b + G[2] * c), x11 = G[3] * b + (G[4] * dt + G[5] * e);
  const T x22 = G[6] * c + (G[7] * e + G[8] * ft);
  T S[5];
  S[0] = P.two * x00 + tm * at;
  S[3] = P.two * x11 + tm * dt;
  const T s5 = P.two * x22 + tm * ft;
  S[1] = (G[0] * b + (G[1] * dt + G[2] * e)) + (G[3] * at + (G[4] * b + (G[5] * c + tm * b)));
  S[2] = (G[0] * c + (G[1] * e + G[2] * ft)) + (G[6] * at + (G[7] * b + (G[8] * c + tm * c)));
  S[4] = (G[3] * c + (G[4] * e + G[5] * ft)) + (G[6] * b + (G[7] * dt + (G[8] * e + tm * e)));
  const T tr3 = P.nthird * (S[0] + S[3] + s5);
  S[0] = S[0] + tr3;
  S[3] = S[3] + tr3;
#pragma unroll
  for (int k = 0; k < 5; ++k) d5[k] = S[k] + (P.Gamma * h[k] + P.nhalf * adv[k]);
}

// FP32 storage: H was evaluated at hi, the stored Q is hi + lo.  Adds the local
// part of H(hi + lo) - H(hi) to first order: the bulk terms' derivative at hi
// applied to lo, and lo's own term -6 K lo of the Laplacian (the neighbours' lo
// enter K lap and the gradient terms at the ~1e-9 level).  Without it the
// relaxation stalls where A0 lo ~ the residual.
__device__ __forceinline__ void comp_h_f32(const PhysT<float>& P, const float qi[5], const float lo[5], float h[5]) {
  const int ia[5] = {0, 0, 0, 1, 1}, ib[5] = {0, 1, 2, 1, 2};
  const float A0 = P.A0, g = P.gamma, K = P.K, q0 = P.q0;
  float Qm[3][3], Lm[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      Qm[a][b] = qab(qi, a, b);
      Lm[a][b] = qab(lo, a, b);
    }
  float trq2 = float(0), trql = float(0);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      trq2 += Qm[a][b] * Qm[a][b];
      trql += Qm[a][b] * Lm[a][b];
    }
  const float cb = -A0 * (float(1) - g / float(3)) - A0 * g * trq2 - float(4) * K * q0 * q0 - float(6) * K;
  const float A0g = A0 * g;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int a = ia[k], b = ib[k];
    float ql = float(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) ql += Qm[a][c] * Lm[c][b] + Lm[a][c] * Qm[c][b];
    if (a == b) ql -= float(2) / float(3) * trql;
    h[k] += cb * lo[k] + A0g * ql - float(2) * A0g * trql * qi[k];
  }
}

// Increment of Q of one node, FP32 storage (h receives the compensation; fl[d]
// false closes face d).  The order of the sums stays as it is (see
// lclb_pair.cuh).  FLOW false: the flow is frozen (u = 0).
template <bool FLOW>
__device__ __forceinline__ void q_increment_f32(const PhysT<float>& P, const float qi[5], const float qn[6][5],
                                                const float ui[3], const float un[6][3], const bool fl[6], float h[5],
                                                const float lo[5], float d5[5]) {
  const float Gam = P.Gamma, xi = P.xi;
  if constexpr (!FLOW) {
    comp_h_f32(P, qi, lo, h);
#pragma unroll
    for (int k = 0; k < 5; ++k) d5[k] = Gam * h[k];
    return;
  }
  // velocity gradient W_ab = d_b u_a
  float W[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) W[a][b] = float(0.5) * (un[2 * b][a] - un[2 * b + 1][a]);
  // advective fluxes through the six faces (zero across solid faces)
  float adv[5] = {float(0), float(0), float(0), float(0), float(0)};
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    if (!fl[d]) continue;
    const int ax = d >> 1;
    const float uf = float(0.5) * (ui[ax] + un[d][ax]);
    const bool plus = (d & 1) == 0;
    // + face: upwind is i when uf > 0; - face: upwind is the neighbour when uf > 0
    const bool take_i = plus ? (uf > float(0)) : !(uf > float(0));
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const float fl_ = uf * (take_i ? qi[k] : qn[d][k]);
      adv[k] += plus ? fl_ : -fl_;
    }
  }
  // co-rotation S = xi (D Qt + Qt D) + (Om Q - Q Om) - 2 xi Qt Tr(Q W), Qt = Q + I/3
  float D[3][3], Om[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      D[a][b] = float(0.5) * (W[a][b] + W[b][a]);
      Om[a][b] = float(0.5) * (W[a][b] - W[b][a]);
    }
  float trQW = float(0);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) trQW += qab(qi, a, b) * D[a][b];
  float dQ[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      float s = float(0);
#pragma unroll
      for (int c = 0; c < 3; ++c)
        s += xi * (D[a][c] * qab(qi, c, b) + qab(qi, a, c) * D[c][b]) + Om[a][c] * qab(qi, c, b) -
             qab(qi, a, c) * Om[c][b];
      s += xi * float(2) / float(3) * D[a][b];
      s -= float(2) * xi * (qab(qi, a, b) + (a == b ? float(1) / float(3) : float(0))) * trQW;
      dQ[a][b] = s;
    }
  const float tr = dQ[0][0] + dQ[1][1] + dQ[2][2];
  comp_h_f32(P, qi, lo, h);
  const int ia[5] = {0, 0, 0, 1, 1}, ib[5] = {0, 1, 2, 1, 2};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    float v = Gam * h[k] + dQ[ia[k]][ib[k]] - adv[k];
    if (ia[k] == ib[k]) v -= tr / float(3);
    d5[k] = v;
  }
}

}  // namespace lclb
