// lclb_kernels.cu -- sm_103a kernels of one coupled step (Lintuvuori et al., Sec. 2.2):
//   k_stress  molecular field H and stress P of every fluid node, stored, and
//             the colloid LC force/torque (Eqs. 4, 8).
//   k_lbp     pull-scheme stream + BGK collide with Guo forcing, bounce-back on
//             links inline (moving-surface term), body force from the stored P;
//             writes df* and u.
//   k_lc      Beris-Edwards update of Q (Eq. 2 with co-rotation and upwind
//             advective face fluxes), residual partials, momentum exchange over
//             the boundary links -> F_hyd, T_hyd, colloid update and
//             buffer-parity flip.
//   k_relax   the whole step when the flow is frozen.
// Other variants of the step: k_flb (stress and LB fused), k_force + k_lb (body
// force stored), k_step (all phases in one launch), and k_links and k_colloid,
// the last two parts of k_lc as launches of their own.
// All step kernels walk a work list of (box, x0, y0, z0) tiles, so that one
// launch serves one box or a batch of boxes of different sizes.
#include <cstdio>

#include "lclb_pair.cuh"
#include "lclb_internal.h"
#include "lclb_barrier.h"

namespace lclb {

constexpr int TX = 32;

// Loads of data that the same launch may have written (the persistent step
// kernel: stress, velocity, post-collision populations, colloid sums) go
// through L2 only (CG); data produced by earlier launches may take the
// read-only path.
template <bool CG, typename T>
__device__ __forceinline__ T ldx(const T* p) {
  if constexpr (CG) return __ldcg(p);
  else return __ldg(p);
}

// L2 eviction priorities (PTX createpolicy, cache hints on the loads and
// stores; no setting of the device changes): the stress, molecular field and
// velocity that the next kernels of the step read are stored to stay
// (evict_last), the populations, read and written once per step, to go first
// (evict_first), so the 129 MB L2 keeps the intermediates between kernels.
__device__ __forceinline__ uint64_t l2_keep() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_stream() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void st_hint(float* a, float v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(a), "f"(v), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_hint(double* a, double v, uint64_t) { *a = v; }
__device__ __forceinline__ float ld_hint(const float* a, uint64_t pol) {
  float v;
  asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(a), "l"(pol));
  return v;
}
__device__ __forceinline__ double ld_hint(const double* a, uint64_t) { return __ldg(a); }

// ---------------------------------------------------------------------------
// reductions
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}

// Block sum of NV doubles per thread; result valid in thread 0.  sred needs
// 32*NV doubles.  Must be called by all threads of the block.
template <int NV>
__device__ void block_sum(double v[NV], double* sred, bool is_max_last = false) {
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  const int lane = tid & 31, wid = tid >> 5, nw = (blockDim.x * blockDim.y + 31) >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = (is_max_last && k == NV - 1) ? warp_max(v[k]) : warp_sum(v[k]);
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) sred[k * 32 + wid] = v[k];
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double t = lane < nw ? sred[k * 32 + lane] : 0.0;
      v[k] = (is_max_last && k == NV - 1) ? warp_max(t) : warp_sum(t);
    }
  }
  __syncthreads();
}

// Residual partials of a warp's row of a Q-update tile: the sum of squares
// and the max over its lanes, written by lane 0 to part[2 wy], part[2 wy + 1]
// (one record per warp, so a tile needs no block barrier and no FP64 sum).
template <typename T>
__device__ __forceinline__ void warp_residual(double* part, int wy, int lane, T rsum, T rmax) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rsum += __shfl_down_sync(0xffffffffu, rsum, o);
    const T m = __shfl_down_sync(0xffffffffu, rmax, o);
    rmax = m > rmax ? m : rmax;
  }
  if (lane == 0) {
    part[2 * wy] = (double)rsum;
    part[2 * wy + 1] = (double)rmax;
  }
}

// Sums of NV values over the 32 lanes, eight at a time: each exchange halves
// the values a lane carries, so a sum takes 9 FP64 additions per eight values
// instead of 40 (an FP64 instruction occupies a warp for 64 cycles).  fn(k, sum)
// is called once per value by one lane.  All lanes call it.
template <int NV, typename Fn>
__device__ __forceinline__ void warp_sums(const double* v, Fn fn) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k0 = 0; k0 < NV; k0 += 8) {
    double t[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) t[k] = k0 + k < NV ? v[k0 + k] : 0.0;
#pragma unroll
    for (int w = 4, o = 16; w >= 1; w >>= 1, o >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < w; ++k) {
        const double give = up ? t[k] : t[k + w], keep = up ? t[k + w] : t[k];
        t[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    t[0] += __shfl_xor_sync(0xffffffffu, t[0], 2);
    t[0] += __shfl_xor_sync(0xffffffffu, t[0], 1);
    const int k = k0 + (lane >> 2);
    if ((lane & 3) == 0 && k < NV) fn(k, t[0]);
  }
}

// Add per-lane contributions v[0..NV-1] (for colloid id c, -1: none) into
// acc[off..off+NV-1] of each colloid with one FP64 atomic per (warp, colloid,
// component).  Must be called by all 32 lanes of a converged warp.
template <int NV = 6>
__device__ __forceinline__ void warp_flush_colloid(DevColloid* col, int c, const double* v, int off) {
  unsigned pend = __ballot_sync(0xffffffffu, c >= 0);
  while (pend) {
    const int leader = __ffs(pend) - 1;
    const int cc = __shfl_sync(0xffffffffu, c, leader);
    const bool mine = (c == cc);
    double w[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) w[k] = mine ? v[k] : 0.0;
    warp_sums<NV>(w, [&](int k, double t) {
      if (t != 0.0) atomicAdd(&col[cc].acc[off + k], t);
    });
    if (mine) c = -1;
    pend = __ballot_sync(0xffffffffu, c >= 0);
  }
}

// The block's shared copy of box b's record, copied by all threads in 4-byte
// words (DevBox is a multiple of 8 bytes and 8-byte aligned).
static_assert(sizeof(DevBox) % 4 == 0, "DevBox is copied in 4-byte words");
__device__ __forceinline__ void load_box(DevBox& sb, const DevBox* boxes, int b) {
  __syncthreads();
  const unsigned* src = reinterpret_cast<const unsigned*>(boxes + b);
  unsigned* dst = reinterpret_cast<unsigned*>(&sb);
  const int nthr = blockDim.x * blockDim.y;
  for (int k = threadIdx.x + blockDim.x * threadIdx.y; k < (int)(sizeof(DevBox) / 4); k += nthr) dst[k] = src[k];
  __syncthreads();
}

// The constants of the two-node paths from the shared record.
__device__ __forceinline__ void load_k2(LcPair& k2, const DevBox& B) {
  const float* src = reinterpret_cast<const float*>(&B.kp);
  f2* dst = reinterpret_cast<f2*>(&k2);
  const int nthr = blockDim.x * blockDim.y;
  for (int k = threadIdx.x + blockDim.x * threadIdx.y; k < LCPAIR_N; k += nthr) dst[k] = f2(src[k]);
  __syncthreads();
}

// Tile loops: reload the shared box record only when the tile's box changes
// (b is uniform over the block, so the barriers are too).
__device__ __forceinline__ void load_box(DevBox& sb, const DevBox* boxes, int b, int& cur) {
  if (b == cur) return;
  load_box(sb, boxes, b);
  cur = b;
}
template <typename T>
__device__ __forceinline__ void load_box(DevBox& sb, LcPair& k2, const DevBox* boxes, int b, int& cur) {
  if (b == cur) return;
  load_box(sb, boxes, b);
  if constexpr (sizeof(T) == 4) load_k2(k2, sb);
  cur = b;
}

// ---------------------------------------------------------------------------
// shared pieces of the force / LB kernels
// ---------------------------------------------------------------------------
// Stress P (9 comps) of fluid node (gx,gy,kk) into sP[c*HP] (c = 0..8); the
// node's mask byte decides fluid/solid.  Returns the flag stored with it:
// 0 fluid, colloid id + 1, or WALLFLAG.  When hout is non-null (an interior
// position of the tile) the molecular field H is also stored there, for the
// Q update of the same step.
template <typename T>
__device__ __forceinline__ uint8_t stress_at(const DevBox& B, const PhysT<T>& PP, const T* __restrict__ Q, int gx,
                                             int gy, int kk, T* sP, int HP, T* hout) {
  const int i = gx + B.nx * (gy + B.ny * kk);
  const uint8_t m = B.mask[i];
  const uint8_t flag = m & IDMASK;
  if (flag != 0) return flag;
  T qi[5], qn[6][5], h[5], p[9], fp;
  gather_q(B, Q, gx, gy, kk, i, m, qi, qn, nullptr);
  lc_node<T>(B, qi, qn, h, p, &fp);
#pragma unroll
  for (int c = 0; c < 9; ++c) sP[c * HP] = p[c];
  if (hout) {
#pragma unroll
    for (int c = 0; c < 5; ++c) hout[(size_t)c * B.N + i] = h[c];
  }
  return 0;
}

// Colloid c takes -sgn P_{.,ax}(i) through the face of fluid node (x, y, kc)
// on its side (Eq. 8), with the moment about its centre; summed per thread
// into my_acc (F, T) for colloid my_c.
template <typename T>
__device__ __forceinline__ void colloid_face(const DevBox& B, int c, int ax, T sgn, const T pcv[3], int x, int y,
                                             int kc, int& my_c, double my_acc[6]) {
  const DevColloid& C = B.col[c];
  const T ff[3] = {-sgn * pcv[0], -sgn * pcv[1], -sgn * pcv[2]};
  double rd[3];
  const double hx2 = 0.5 * (double)(ax == 0 ? sgn : 0), hy2 = 0.5 * (double)(ax == 1 ? sgn : 0),
               hz2 = 0.5 * (double)(ax == 2 ? sgn : 0);
  disp(B, (double)x + hx2, (double)y + hy2, (double)kc + hz2, C.X, rd);
  // the face force is in T; its moment arm from the FP64 offset, taken in T
  const T r[3] = {T(rd[0]), T(rd[1]), T(rd[2])};
  const T tq[3] = {r[1] * ff[2] - r[2] * ff[1], r[2] * ff[0] - r[0] * ff[2], r[0] * ff[1] - r[1] * ff[0]};
  if (my_c >= 0 && my_c != c) {  // a second colloid at this node: flush the first directly
    for (int a = 0; a < 6; ++a) {
      atomicAdd(&B.col[my_c].acc[6 + a], my_acc[a]);
      my_acc[a] = 0.0;
    }
  }
  my_c = c;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    my_acc[a] += (double)ff[a];
    my_acc[3 + a] += (double)tq[a];
  }
}

// Body force at interior fluid position pc (plane slot s0; the planes below
// and above in slots sm, sp): F_a = sum_d [P_ad(face +d) - P_ad(face -d)],
// a fluid-fluid face carrying (P_i + P_j)/2 and a solid or wall face P_i.
// Each colloid face adds -(+-P_.d(i)) to the colloid's LC force (and its
// moment about X to the torque) in the thread's accumulator.
template <typename T>
__device__ __forceinline__ void face_force(const DevBox& B, const T* sP, const uint8_t* sFl, int HP, int HX, int s0,
                                           int sm, int sp, int pc, int x, int y, int kc, bool acc, T Fv[3],
                                           int& my_c, double my_acc[6]) {
  Fv[0] = Fv[1] = Fv[2] = T(0);
  const int nslot[6] = {s0, s0, s0, s0, sp, sm};
  const int npos[6] = {pc + 1, pc - 1, pc + HX, pc - HX, pc, pc};
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const int ax = d >> 1;
    const T sgn = (d & 1) ? T(-1) : T(1);
    const uint8_t fj = sFl[nslot[d] * HP + npos[d]];
    T pcv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      pcv[a] = sP[(s0 * 9 + 3 * a + ax) * HP + pc];
      const T face = (fj == 0) ? T(0.5) * (pcv[a] + sP[(nslot[d] * 9 + 3 * a + ax) * HP + npos[d]]) : pcv[a];
      Fv[a] += sgn * face;
    }
    if (acc && fj != 0 && fj != WALLFLAG) colloid_face(B, fj - 1, ax, sgn, pcv, x, y, kc, my_c, my_acc);
  }
}

// ---------------------------------------------------------------------------
// k_force: body force alone
// ---------------------------------------------------------------------------
// Shared memory: P of three z planes over the tile plus a one-node halo,
// [3][9][(TX+2)(TY+2)] in T, then one flag byte per position.
template <typename T, int TY>
__global__ void __launch_bounds__(TX * TY) k_force(const DevBox* __restrict__ boxes, const int4* __restrict__ tiles,
                                                   int ntiles, int zc, int mode, double* __restrict__ part) {
  constexpr int HX = TX + 2, HY = TY + 2, HP = HX * HY, NT = TX * TY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sP = reinterpret_cast<T*>(smem_raw);
  uint8_t* sFl = smem_raw + sizeof(T) * 27 * HP;
  __shared__ DevBox B;
  const int tid = threadIdx.x + TX * threadIdx.y;

  int cur_box = -1;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int4 td = tiles[t];
    load_box(B, boxes, td.x, cur_box);
    if (!B.p.lc_on) continue;
    const PhysT<T>& PP = phys<T>(B);
    int my_c = -1;
    double my_acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const T* __restrict__ Q = static_cast<const T*>(B.Q[B.st->qpar]);
    T* __restrict__ Fout = static_cast<T*>(B.F);
    const int x0 = td.y, y0 = td.z, z0 = td.w;
    const int nx = B.nx, ny = B.ny, nz = B.nz, N = B.N;
    const int vx = min(TX, nx - x0), vy = min(TY, ny - y0);
    const int zend = min(z0 + zc, nz);
    __syncthreads();
    for (int k = z0 - 1; k <= zend; ++k) {
      const int slot = (k - z0 + 1) % 3;
      const bool wallplane = B.wall_z && (k < 0 || k >= nz);
      const int kk = B.wall_z ? k : wrapn(k, nz);
      for (int pidx = tid; pidx < HP; pidx += NT) {
        const int hx = pidx % HX, hy = pidx / HX;
        if (hx > vx + 1 || hy > vy + 1) continue;
        uint8_t flag = WALLFLAG;
        if (!wallplane) {
          const bool inner = hx >= 1 && hx <= vx && hy >= 1 && hy <= vy && k >= z0 && k < zend;
          flag = stress_at(B, PP, Q, wrapn(x0 - 1 + hx, nx), wrapn(y0 - 1 + hy, ny), kk, sP + slot * 9 * HP + pidx,
                           HP, inner ? static_cast<T*>(B.H) : (T*)nullptr);
        }
        sFl[slot * HP + pidx] = flag;
      }
      __syncthreads();
      if (k >= z0 + 1) {
        const int kc = k - 1;
        const int tx = threadIdx.x, ty = threadIdx.y;
        const int pc = (tx + 1) + HX * (ty + 1);
        if (tx < vx && ty < vy && sFl[((k - z0) % 3) * HP + pc] == 0) {
          T Fv[3];
          face_force(B, sP, sFl, HP, HX, (k - z0) % 3, (k - z0 - 1) % 3, slot, pc, x0 + tx, y0 + ty, kc,
                     (mode & FORCE_ACC) != 0, Fv, my_c, my_acc);
          const int ic = (x0 + tx) + nx * ((y0 + ty) + ny * kc);
#pragma unroll
          for (int a = 0; a < 3; ++a) Fout[(size_t)a * N + ic] = Fv[a];
        }
      }
      __syncthreads();
    }
    if (mode & FORCE_ACC) warp_flush_colloid(B.col, my_c, my_acc, 6);
  }
}

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// Moving-surface term of the bounced populations: ms[q] is the mask byte of
// node r - c_q (colloid id + 1, 0 fluid, WALLFLAG).  The colloid's state is
// read and converted once per node (a node rarely touches two), and a colloid
// at rest adds nothing.
template <typename T>
__device__ __forceinline__ void bounce_correction(const DevBox& B, int x, int y, int z, const uint8_t ms[NQ],
                                                  T df[NQ]) {
  const T rho0 = phys<T>(B).rho0;
  unsigned todo = 0;
#pragma unroll
  for (int q = 1; q < NQ; ++q)
    if (ms[q] != 0 && ms[q] != WALLFLAG) todo |= 1u << q;
  while (todo) {
    int id = 0;
    const int first = __ffs(todo) - 1;
#pragma unroll
    for (int q = 1; q < NQ; ++q)
      if (q == first) id = ms[q];
    const DevColloid& C = B.col[id - 1];
    T X[3], V[3], W[3];
    bool moving = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      X[a] = T(C.Xb[a]);
      V[a] = T(C.Vb[a]);
      W[a] = T(C.Wb[a]);
      moving = moving || V[a] != T(0) || W[a] != T(0);
    }
#pragma unroll
    for (int q = 1; q < NQ; ++q) {
      if (ms[q] != id) continue;
      todo &= ~(1u << q);
      if (!moving) continue;
      // u_b = V + W x d at the link midpoint r - c_q / 2
      const T d0 = minimg_t(T(x) - T(0.5 * cx(q)) - X[0], B.nx, true);
      const T d1 = minimg_t(T(y) - T(0.5 * cy(q)) - X[1], B.ny, true);
      const T d2 = minimg_t(T(z) - T(0.5 * cz(q)) - X[2], B.nz, !B.wall_z);
      T cub = T(0);
      if (cx(q)) cub += T(cx(q)) * (V[0] + W[1] * d2 - W[2] * d1);
      if (cy(q)) cub += T(cy(q)) * (V[1] + W[2] * d0 - W[0] * d2);
      if (cz(q)) cub += T(cz(q)) * (V[2] + W[0] * d1 - W[1] * d0);
      df[q] += mul_rn(T(6.0 * wq(q)) * rho0, cub);  // (rounded before it is added)
    }
  }
}

// ---------------------------------------------------------------------------
// pull with bounce-back (shared by the LB kernels and the export/diagnostic kernels)
// ---------------------------------------------------------------------------
// Gathers the pre-collision deviations df_q(r) = df*_q(r - c_q) for fluid
// node r, or, when r - c_q is solid (colloid) or beyond a wall, the bounced
// population df*_{-q}(r) + 6 w_q rho0 (c_q . u_b) with u_b the rigid velocity
// at the link midpoint r - c_q/2 of the state that produced df* (Vb, Wb, Xb).
template <typename T>
__device__ __forceinline__ void pull(const DevBox& B, const T* __restrict__ fin, int x, int y, int z, int i, uint8_t m,
                                     bool pre, T df[NQ]) {
  const int N = B.N;
  if (pre) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) df[q] = ldg(fin + (size_t)q * N + i);
    return;
  }
  const int nx = B.nx, ny = B.ny, nz = B.nz;
  const int xs[3] = {x == 0 ? nx - 1 : x - 1, x, x + 1 == nx ? 0 : x + 1};
  const int ys[3] = {y == 0 ? ny - 1 : y - 1, y, y + 1 == ny ? 0 : y + 1};
  int zs[3];
  if (B.wall_z) {
    zs[0] = z - 1; zs[1] = z; zs[2] = z + 1;
  } else {
    zs[0] = z == 0 ? nz - 1 : z - 1; zs[1] = z; zs[2] = z + 1 == nz ? 0 : z + 1;
  }
  if (!(m & NEAR)) {
    const uint64_t pol = l2_stream();
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int s = xs[1 - cx(q)] + nx * (ys[1 - cy(q)] + ny * zs[1 - cz(q)]);
      df[q] = ld_hint(fin + (size_t)q * N + s, pol);
    }
    return;
  }
  // near node: the 18 mask bytes, then the 19 populations, each in one round of
  // independent loads (taken direction by direction, the dependent pairs of
  // loads were most of the time of a small box's LB kernel)
  int s[NQ];
  uint8_t ms[NQ];
  s[0] = i;
  ms[0] = 0;
#pragma unroll
  for (int q = 1; q < NQ; ++q) {
    const int zsrc = zs[1 - cz(q)];
    const bool in = zsrc >= 0 && zsrc < nz;
    s[q] = in ? xs[1 - cx(q)] + nx * (ys[1 - cy(q)] + ny * zsrc) : i;
    ms[q] = B.mask[s[q]] & IDMASK;
    if (!in) ms[q] = WALLFLAG;
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q) df[q] = ldg(fin + (ms[q] == 0 ? (size_t)q * N + s[q] : (size_t)opp(q) * N + i));
  bounce_correction<T>(B, x, y, z, ms, df);
}

// Collide at fluid node i with force (Fx,Fy,Fz) (BGK + Guo, deviation form):
// rho = rho0 + sum df, u = (sum df c + F/2)/rho,
// df*_q = df_q - omega (df_q - df_eq_q) + (1 - 1/2tau) w_q [3(c - u) + 9 (c.u) c].F,
// df_eq_q = w_q [drho + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u^2)].  Writes df* and u.
// FP32 storage: direction by direction, in an order that stays as it is (see
// lclb_pair.cuh); opposite directions share c.u and c.F.
__device__ __forceinline__ void collide_store(const PhysT<float>& PP, float* __restrict__ fout,
                                              float* __restrict__ ub, int N, int i, const float df[NQ], float Fx,
                                              float Fy, float Fz) {
  float drho = 0.f, mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    drho += df[q];
    if (cx(q)) mx += cx(q) > 0 ? df[q] : -df[q];
    if (cy(q)) my += cy(q) > 0 ? df[q] : -df[q];
    if (cz(q)) mz += cz(q) > 0 ? df[q] : -df[q];
  }
  const float rho = PP.rho0 + drho;
  const float inv = 1.f / rho;
  const float ux = (mx + 0.5f * Fx) * inv, uy = (my + 0.5f * Fy) * inv, uz = (mz + 0.5f * Fz) * inv;
  const float usq = ux * ux + uy * uy + uz * uz;
  const float uF = ux * Fx + uy * Fy + uz * Fz;
  const float omega = PP.omega, pref = PP.pref;
  const uint64_t pol_stream = l2_stream(), pol_keep = l2_keep();
  auto put = [&](int q, float w, float cu, float cF) {
    const float eq = w * (drho + rho * (3.f * cu + 4.5f * cu * cu - 1.5f * usq));
    const float src = pref * w * (3.f * (cF - uF) + 9.f * cu * cF);
    st_hint(fout + (size_t)q * N + i, df[q] - omega * (df[q] - eq) + src, pol_stream);
  };
  put(0, float(wq(0)), 0.f, 0.f);
#pragma unroll
  for (int q = 1; q < NQ; q += 2) {
    float cu = 0.f, cF = 0.f;
    if (cx(q)) { cu += cx(q) > 0 ? ux : -ux; cF += cx(q) > 0 ? Fx : -Fx; }
    if (cy(q)) { cu += cy(q) > 0 ? uy : -uy; cF += cy(q) > 0 ? Fy : -Fy; }
    if (cz(q)) { cu += cz(q) > 0 ? uz : -uz; cF += cz(q) > 0 ? Fz : -Fz; }
    put(q, float(wq(q)), cu, cF);
    put(q + 1, float(wq(q)), -cu, -cF);
  }
  st_hint(ub + i, ux, pol_keep);
  st_hint(ub + (size_t)N + i, uy, pol_keep);
  st_hint(ub + (size_t)2 * N + i, uz, pol_keep);
}

__device__ __forceinline__ void collide_store(const PhysT<double>& PP, double* __restrict__ fout,
                                              double* __restrict__ ub, int N, int i, const double df[NQ], double Fx,
                                              double Fy, double Fz) {
  using T = double;
  // Opposite directions share all but a sign: with c.j the odd part (j = 3 rho u +
  // 3 (tau - 1/2) F) and an even part base + (c.u)(c.g) (g = 1.5 j + 4.5 (tau - 1/2) F),
  // df*_q = df_q + omega (w_q (even + c.j) - df_q), the bracket small near
  // equilibrium so that df_q is rounded once.  About 150 operations a node instead
  // of 420 direction by direction: FP64 issue bounds the kernel (k_lbp, 64^3:
  // 229 -> 109 us).
  T drho = df[0], mx = T(0), my = T(0), mz = T(0);
#pragma unroll
  for (int q = 1; q < NQ; q += 2) {
    const T s = df[q] + df[q + 1], d = df[q] - df[q + 1];
    drho += s;
    if (cx(q)) mx += cx(q) > 0 ? d : -d;
    if (cy(q)) my += cy(q) > 0 ? d : -d;
    if (cz(q)) mz += cz(q) > 0 ? d : -d;
  }
  const T omega = PP.omega, pt = PP.ptau;
  const T rho = PP.rho0 + drho;
  const T inv = T(1) / rho;
  const T ux = (mx + T(0.5) * Fx) * inv, uy = (my + T(0.5) * Fy) * inv, uz = (mz + T(0.5) * Fz) * inv;
  const T usq = ux * ux + uy * uy + uz * uz;
  const T uF = ux * Fx + uy * Fy + uz * Fz;
  const T r3 = T(3) * rho, p3 = T(3) * pt, p45 = T(4.5) * pt;
  const T jx = r3 * ux + p3 * Fx, jy = r3 * uy + p3 * Fy, jz = r3 * uz + p3 * Fz;
  const T gx = T(1.5) * jx + p45 * Fx, gy = T(1.5) * jy + p45 * Fy, gz = T(1.5) * jz + p45 * Fz;
  const T base = drho - (T(0.5) * r3 * usq + p3 * uF);
  const uint64_t pol_stream = l2_stream(), pol_keep = l2_keep();
  st_hint(fout + i, df[0] + omega * (T(wq(0)) * base - df[0]), pol_stream);
#pragma unroll
  for (int q = 1; q < NQ; q += 2) {
    const T w = T(wq(q));
    T cu = T(0), cg = T(0), cj = T(0);
    if (cx(q)) { cu += cx(q) > 0 ? ux : -ux; cg += cx(q) > 0 ? gx : -gx; cj += cx(q) > 0 ? jx : -jx; }
    if (cy(q)) { cu += cy(q) > 0 ? uy : -uy; cg += cy(q) > 0 ? gy : -gy; cj += cy(q) > 0 ? jy : -jy; }
    if (cz(q)) { cu += cz(q) > 0 ? uz : -uz; cg += cz(q) > 0 ? gz : -gz; cj += cz(q) > 0 ? jz : -jz; }
    const T even = base + cu * cg;
    st_hint(fout + (size_t)q * N + i, df[q] + omega * (w * (even + cj) - df[q]), pol_stream);
    st_hint(fout + (size_t)(q + 1) * N + i, df[q + 1] + omega * (w * (even - cj) - df[q + 1]), pol_stream);
  }
  st_hint(ub + i, ux, pol_keep);
  st_hint(ub + (size_t)N + i, uy, pol_keep);
  st_hint(ub + (size_t)2 * N + i, uz, pol_keep);
}

template <typename T>
__device__ __forceinline__ void solid_velocity(const DevBox& B, T* __restrict__ ub, int x, int y, int z, int i,
                                               uint8_t m) {
  const DevColloid& C = B.col[(m & IDMASK) - 1];
  T ur[3];
  rigid_velocity_t<T>(B, T(x), T(y), T(z), C.X, C.V, C.W, ur);
#pragma unroll
  for (int a = 0; a < 3; ++a) ub[(size_t)a * B.N + i] = ur[a];
}

// ---------------------------------------------------------------------------
// k_lb: collide/stream with the body force read from memory
// ---------------------------------------------------------------------------
template <typename T, int TY>
__global__ void __launch_bounds__(TX * TY, (sizeof(T) == 4 ? 768 : 384) / (TX * TY)) k_lb(
    const DevBox* __restrict__ boxes, const int4* __restrict__ tiles, int ntiles, int zc, int mode,
    double* __restrict__ part) {
  __shared__ DevBox B;
  int cur_box = -1;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int4 td = tiles[t];
    load_box(B, boxes, td.x, cur_box);
    if (!B.p.flow_on) continue;
    const PhysT<T>& PP = phys<T>(B);
    const int fpar = B.st->fpar;
    const bool pre = B.st->pre_valid != 0;
    const T* __restrict__ fin = static_cast<const T*>(B.f[fpar]);
    T* __restrict__ fout = static_cast<T*>(B.f[fpar ^ 1]);
    const T* __restrict__ Fb = static_cast<const T*>(B.F);
    T* __restrict__ ub = static_cast<T*>(B.u);
    const int nx = B.nx, ny = B.ny, N = B.N;
    const int x = td.y + threadIdx.x, y = td.z + threadIdx.y;
    const int zend = min(td.w + zc, B.nz);
    if (x >= nx || y >= ny) continue;
    const bool lc = B.p.lc_on != 0;
    for (int z = td.w; z < zend; ++z) {
      const int i = x + nx * (y + ny * z);
      const uint8_t m = B.mask[i];
      if (m & IDMASK) {
        solid_velocity(B, ub, x, y, z, i, m);
        continue;
      }
      T df[NQ];
      pull(B, fin, x, y, z, i, m, pre, df);
      T Fx = PP.g[0], Fy = PP.g[1], Fz = PP.g[2];
      if (lc) {
        Fx += Fb[i];
        Fy += Fb[(size_t)N + i];
        Fz += Fb[(size_t)2 * N + i];
      }
      collide_store(PP, fout, ub, N, i, df, Fx, Fy, Fz);
    }
  }
}

// ---------------------------------------------------------------------------
// x-neighbour values from the adjacent lanes
// ---------------------------------------------------------------------------
// The lanes of a warp hold consecutive x of one row, so the K values of the
// x +- 1 neighbours of a node come from lanes +- 1 by shuffles; a lane whose
// neighbour is not held by the adjacent lane (the tile's edge lanes, the
// periodic wrap, the end of a ragged row) loads it.  All 32 lanes call this.
// xn[0] = x + 1, xn[1] = x - 1 (the order of face_neighbours).
template <typename T, int K, bool CG = false>
__device__ __forceinline__ void x_neighbours(const T* __restrict__ F, size_t N, const T self[K], int lane, int x,
                                             int nx, int row, bool valid, T xn[2][K]) {
#pragma unroll
  for (int k = 0; k < K; ++k) {
    xn[0][k] = __shfl_down_sync(0xffffffffu, self[k], 1);
    xn[1][k] = __shfl_up_sync(0xffffffffu, self[k], 1);
  }
  if (!valid) return;
  if (lane == TX - 1 || x + 1 >= nx) {
    const int j = (x + 1 == nx ? 0 : x + 1) + row;
#pragma unroll
    for (int k = 0; k < K; ++k) xn[0][k] = ldx<CG>(F + (size_t)k * N + j);
  }
  if (lane == 0) {
    const int j = (x == 0 ? nx - 1 : x - 1) + row;
#pragma unroll
    for (int k = 0; k < K; ++k) xn[1][k] = ldx<CG>(F + (size_t)k * N + j);
  }
}

// Values of the thread's own column (x, y) down the z march: at the start of
// a tile, z0 - 1 and z0 (the plane below z0 wraps in a periodic box; beyond a
// wall the value is 0 and unused, such nodes being near nodes).  Each step
// loads z + 1 into pc[3], takes z into pc[0] and z - 1 into pc[4]
// (pc[1], pc[2] are the x-neighbours), and column_roll moves the window up.
template <typename T, int K>
__device__ __forceinline__ void column_start(const DevBox& B, const T* __restrict__ F, int x, int y, int z0,
                                             bool valid, T cz[2][K]) {
  const int zm = z0 > 0 ? z0 - 1 : (B.wall_z ? -1 : B.nz - 1);
  const size_t N = (size_t)B.N;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    cz[0][k] = (valid && zm >= 0) ? ldg(F + (size_t)k * N + x + B.nx * (y + B.ny * zm)) : T(0);
    cz[1][k] = valid ? ldg(F + (size_t)k * N + x + B.nx * (y + B.ny * z0)) : T(0);
  }
}

template <typename T, int K>
__device__ __forceinline__ void column_next(const DevBox& B, const T* __restrict__ F, int x, int y, int z, bool valid,
                                            const T cz[2][K], T pc[5][K]) {
  const int zp = z + 1 < B.nz ? z + 1 : (B.wall_z ? -1 : 0);
  const size_t N = (size_t)B.N;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    pc[0][k] = cz[1][k];
    pc[4][k] = cz[0][k];
    pc[3][k] = (valid && zp >= 0) ? ldg(F + (size_t)k * N + x + B.nx * (y + B.ny * zp)) : T(0);
  }
}

template <typename T, int K>
__device__ __forceinline__ void column_roll(T cz[2][K], const T pc[5][K]) {
#pragma unroll
  for (int k = 0; k < K; ++k) {
    cz[0][k] = pc[0][k];
    cz[1][k] = pc[3][k];
  }
}

// ---------------------------------------------------------------------------
// stored-stress variant: k_stress stores H and P once per fluid node, k_lbp
// takes the body force from the stored P
// ---------------------------------------------------------------------------
// Node i of the stored-stress kernel: gather (surface values at solid or wall
// faces when near), H, P, stores, and for near nodes the colloid LC force.
// A plain node (NEAR_NODE false) takes its own Q and that of its x- and
// z-neighbours from pq (self, x + 1, x - 1, z + 1, z - 1: gathered by the warp
// and rolled down the thread's column) and loads the y-neighbours.
//
// Near node: derivatives from the differences to the six neighbours, the
// difference to a solid or wall neighbour being w/(K + w) (Q0 - Q) (1 for
// strong anchoring) with Q0 in FP64.  FP32 storage takes the compensated
// values, (hi_j - hi_i) + (lo_j - lo_i), and the surface difference in FP64:
// with hi alone the rounding of Q (~3e-8) enters the Laplacian of every node at
// the colloid surface, and the colloid's LC force, a small sum of large face
// terms, would carry it at ~1e-4 relative.
//
// A warp evaluates 32 near nodes.  Their solid faces (one or two per node of
// the six) are packed into a queue and shared out over the lanes, once for the
// surface values and once for the colloid force, because the FP64 arithmetic
// of a face is a chain of some 60 dependent operations that every lane of the
// warp would otherwise run through six times.  scratch: shared memory of the
// warp (NearScratch<T>).
template <typename T>
struct NearScratch {
  uint16_t face[192];  // lane | d << 8 of each solid face
  T dn[192][5];        // Qs - Q of each solid face
};

// a b - c d, one product rounded (FP32: the second for a - face, the first for a
// + face, as the torque of a face has always been summed).
__device__ __forceinline__ float cross_term(bool minus, float a, float b, float c, float d) {
  return minus ? __fmaf_rn(a, b, -__fmul_rn(c, d)) : __fmaf_rn(-c, d, __fmul_rn(a, b));
}
__device__ __forceinline__ double cross_term(bool, double a, double b, double c, double d) { return a * b - c * d; }

// FROZEN (flow frozen): the node's Q is updated at once, dQ = Gamma H, and its
// residual added to rs (sum of squares, max), instead of storing H and P.
template <typename T>
__device__ __forceinline__ void store_q_next(const DevBox& B, int qpar, size_t i, int k, T q, float lo, T d) {
  const size_t o = (size_t)k * B.N + i;
  if constexpr (sizeof(T) == 4) {
    // compensated FP32 storage: hi + lo + increment carried exactly into hi, to BF16 in lo
    float hi;
    __nv_bfloat16 lo_out;
    add_compensated(q, lo, d, hi, lo_out);
    static_cast<float*>(B.Q[qpar ^ 1])[o] = hi;
    B.Qlo[qpar ^ 1][o] = lo_out;
  } else {
    static_cast<T*>(B.Q[qpar ^ 1])[o] = q + d;
  }
}
template <typename T>
__device__ __forceinline__ void add_residual(const T d5[5], T& rsum, T& rmax) {
  const T dzz = -d5[0] - d5[3];
  rsum += d5[0] * d5[0] + d5[3] * d5[3] + dzz * dzz + T(2) * (d5[1] * d5[1] + d5[2] * d5[2] + d5[4] * d5[4]);
  T mx = fabs(dzz);
#pragma unroll
  for (int k = 0; k < 5; ++k) mx = fmax(mx, fabs(d5[k]));
  rmax = fmax(rmax, mx);
}

template <typename T, bool FROZEN = false>
__device__ __noinline__ void near_stress(const DevBox& B, int i, int mode, NearScratch<T>& sc, T* rs = nullptr,
                                         double* fe = nullptr) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const bool valid = i >= 0;
  if (!__ballot_sync(full, valid)) return;
  const int N = B.N, nx = B.nx, ny = B.ny, qpar = B.st->qpar;
  const int j0 = valid ? i : 0;
  const int x = j0 % nx, y = (j0 / nx) % ny, z = j0 / (nx * ny);
  const T* __restrict__ Q = static_cast<const T*>(B.Q[qpar]);
  const __nv_bfloat16* __restrict__ Lo = B.Qlo[qpar];
  constexpr bool comp = sizeof(T) == 4;
  T qh[5];
  float ql[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    qh[k] = ldg(Q + (size_t)k * N + j0);
    ql[k] = 0.f;
    if constexpr (comp) ql[k] = __bfloat162float(Lo[(size_t)k * N + j0]);
  }
  int nb[6], zz[2], cf[6];
  face_neighbours(B, x, y, z, nb, zz);
#pragma unroll
  for (int d = 0; d < 6; ++d) cf[d] = (int)(B.mask[nb[d] < 0 ? j0 : nb[d]] & IDMASK);
  unsigned solid = 0;  // solid faces of the node
#pragma unroll
  for (int d = 0; d < 6; ++d)
    if (valid && (nb[d] < 0 || cf[d] != 0)) solid |= 1u << d;
  // differences to the fluid neighbours (their loads are in flight under the
  // arithmetic of the surface values)
  T dn[6][5];
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const size_t j = ((solid >> d) & 1u) || nb[d] < 0 ? j0 : nb[d];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      dn[d][k] = ldg(Q + (size_t)k * N + j) - qh[k];
      if constexpr (comp) dn[d][k] += __bfloat162float(Lo[(size_t)k * N + j]) - ql[k];
    }
  }
  bool planar = false;
#pragma unroll
  for (int d = 0; d < 6; ++d)
    if (((solid >> d) & 1u) && nb[d] >= 0 && B.col[cf[d] - 1].anchoring != 0) planar = true;
  // Q in FP64 where a face evaluates its surface value in FP64: planar
  // anchoring, walls, FP64 storage
  const bool wall_face = B.wall_z && (((solid >> 4) & 1u && nb[4] < 0) || ((solid >> 5) & 1u && nb[5] < 0));
  double nf[3] = {1.0, 0.0, 0.0}, qid[5];
  if (!comp || planar || wall_face || max(nx, max(ny, B.nz)) >= (1 << 22)) {
#pragma unroll
    for (int k = 0; k < 5; ++k) qid[k] = comp ? to_f64(qh[k]) + f32_to_f64(ql[k]) : to_f64(qh[k]);
  } else {
#pragma unroll
    for (int k = 0; k < 5; ++k) qid[k] = 0.0;
  }
  if (planar) principal_dir<double>(qid, nf);
  // queue of solid faces; slot[d]: position of this node's face d
  int slot[6], nface = 0;
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const unsigned m = __ballot_sync(full, (solid >> d) & 1u);
    slot[d] = nface + __popc(m & ((1u << lane) - 1u));
    if ((solid >> d) & 1u) sc.face[slot[d]] = (uint16_t)(lane | (d << 8));
    nface += __popc(m);
  }
  __syncwarp();
  // node, direction and colloid (-1: wall) of face t on this lane
  auto face_of = [&](int t, int& own, int& d, int& c, int s[3]) {
    const int e = t < nface ? sc.face[t] : lane;
    own = e & 31;
    d = e >> 8;
    s[0] = __shfl_sync(full, x, own);
    s[1] = __shfl_sync(full, y, own);
    s[2] = __shfl_sync(full, z, own);
    const int ax = d >> 1, up = (d & 1) ? -1 : 1;
    s[0] = ax == 0 ? wrap1(s[0] + up, nx) : s[0];
    s[1] = ax == 1 ? wrap1(s[1] + up, ny) : s[1];
    const int zs = ax == 2 ? s[2] + up : s[2];
    const bool out = B.wall_z && (zs < 0 || zs >= B.nz);
    s[2] = out ? zs : wrap1(zs, B.nz);
    c = t < nface && !out ? (int)(B.mask[s[0] + nx * (s[1] + ny * s[2])] & IDMASK) - 1 : -1;
  };
  for (int t0 = 0; t0 < nface; t0 += 32) {
    const int t = t0 + lane;
    int own, d, c, s[3];
    face_of(t, own, d, c, s);
    // (node coordinates, one box further for an image, are exact in FP32)
    const bool normal = comp && c >= 0 && B.col[c].anchoring == 0 && max(nx, max(ny, B.nz)) < (1 << 22);
    if constexpr (comp) {
      if (__ballot_sync(full, t < nface && normal)) {
        float ho[5], lo[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          ho[k] = __shfl_sync(full, qh[k], own);
          lo[k] = __shfl_sync(full, ql[k], own);
        }
        if (t < nface && normal) surface_dn_normal(B, B.col[c], s, ho, lo, sc.dn[t]);
      }
    }
    if (__ballot_sync(full, t < nface && !normal)) {
      double nfo[3], qo[5];
#pragma unroll
      for (int a = 0; a < 3; ++a) nfo[a] = __shfl_sync(full, nf[a], own);
#pragma unroll
      for (int k = 0; k < 5; ++k) qo[k] = __shfl_sync(full, qid[k], own);
      if (t < nface && !normal) {
        double q0[5];
        surface_q0_near<T>(B, c, s[0], s[1], s[2], nfo, q0);
        const double w = c < 0 ? 1.0 : B.col[c].wfac;
#pragma unroll
        for (int k = 0; k < 5; ++k) sc.dn[t][k] = (T)(w * (q0[k] - qo[k]));
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int d = 0; d < 6; ++d)
    if ((solid >> d) & 1u)
#pragma unroll
      for (int k = 0; k < 5; ++k) dn[d][k] = sc.dn[slot[d]][k];
  T qi[5], dq[3][5], lap[5], h[5], p[9], fp;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    qi[k] = qh[k] + (T)ql[k];
    dq[0][k] = dn[0][k] - dn[1][k];  // doubled, as derivatives()
    dq[1][k] = dn[2][k] - dn[3][k];
    dq[2][k] = dn[4][k] - dn[5][k];
    lap[k] = (dn[0][k] + dn[1][k]) + (dn[2][k] + dn[3][k]) + (dn[4][k] + dn[5][k]);
  }
  lc_node_dq<T>(B, qi, dq, lap, h, p, &fp);
  if constexpr (FROZEN) {
    if (valid) {
      T d5[5];
      if constexpr (comp) q_increment_f32<false>(B.pf, qh, nullptr, nullptr, nullptr, nullptr, h, ql, d5);
      else q_increment<false, T>(B.kd, qh, nullptr, nullptr, h, d5);
#pragma unroll
      for (int k = 0; k < 5; ++k) store_q_next<T>(B, qpar, i, k, qh[k], ql[k], d5[k]);
      add_residual(d5, rs[0], rs[1]);
    }
  } else if (valid) {
    T* Hb = static_cast<T*>(B.H);
    T* Pb = static_cast<T*>(B.P);
#pragma unroll
    for (int c = 0; c < 5; ++c) Hb[(size_t)c * N + i] = h[c];
    if (B.p.flow_on || (mode & FORCE_P)) {  // with the flow frozen only exports read the stress
#pragma unroll
      for (int c = 0; c < 9; ++c) Pb[(size_t)c * N + i] = p[c];
    }
  }
  if (fe && valid) {
    // free energy of the node, and of its weakly anchored faces (w/2)|Qs - Q0|^2
    // with Qs - Q0 = -(K/w)(Qs - Q), squared in FP64
    *fe += to_f64(fp);
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      if (!((solid >> d) & 1u) || nb[d] < 0) continue;
      const DevColloid& C = B.col[cf[d] - 1];
      if (C.strong) continue;
      const double r = B.p.K / C.w;
      double e[5], s2 = 0.0;
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        e[k] = r * to_f64(dn[d][k]);
        s2 += (k == 0 || k == 3 ? 1.0 : 2.0) * e[k] * e[k];
      }
      s2 += (e[0] + e[3]) * (e[0] + e[3]);
      *fe += 0.5 * C.w * s2;
    }
  }
  if (!(mode & FORCE_ACC)) return;
  for (int t0 = 0; t0 < nface; t0 += 32) {
    const int t = t0 + lane;
    int own, d, c, s[3];
    face_of(t, own, d, c, s);
    T po[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) po[k] = __shfl_sync(full, p[k], own);
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (t < nface && c >= 0) {
      // the colloid takes -sgn P_{.,ax} of the fluid node (Eq. 8) at the face
      // centre, half a step back from the solid node, with the moment about
      // its centre (arm from the FP64 offset, taken in T)
      const int ax = d >> 1;
      const T sgn = (d & 1) ? T(-1) : T(1);
      const T ff[3] = {-sgn * (ax == 0 ? po[0] : (ax == 1 ? po[1] : po[2])),
                       -sgn * (ax == 0 ? po[3] : (ax == 1 ? po[4] : po[5])),
                       -sgn * (ax == 0 ? po[6] : (ax == 1 ? po[7] : po[8]))};
      const int back = (d & 1) ? 1 : -1;
      double fc[3], rd[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int L = a == 0 ? nx : (a == 1 ? ny : B.nz);
        fc[a] = (double)(ax == a ? wrap1(s[a] + back, L) : s[a]);
        if (ax == a) fc[a] -= 0.5 * back;
      }
      disp(B, fc[0], fc[1], fc[2], B.col[c].X, rd);
      const T r[3] = {T(rd[0]), T(rd[1]), T(rd[2])};
#pragma unroll
      for (int a = 0; a < 3; ++a) v[a] = to_f64(ff[a]);
      v[3] = to_f64(cross_term((d & 1) != 0, r[1], ff[2], r[2], ff[1]));
      v[4] = to_f64(cross_term((d & 1) != 0, r[2], ff[0], r[0], ff[2]));
      v[5] = to_f64(cross_term((d & 1) != 0, r[0], ff[1], r[1], ff[0]));
    }
    __syncwarp();
    warp_flush_colloid(B.col, t < nface ? c : -1, v, 6);
  }
}

// Plain node, one per lane: own Q and that of the x- and z-neighbours from pq.
template <typename T>
__device__ __forceinline__ void stress_node(const DevBox& B, const PhysT<T>& PP, const T* __restrict__ Q,
                                            T* __restrict__ Hb, T* __restrict__ Pb, int x, int y, int z, int i,
                                            const T (*pq)[5], int mode, T& fp) {
  const int N = B.N;
  T qi[5], qn[6][5], h[5], p[9];
  int nb[6], zz[2];
  face_neighbours(B, x, y, z, nb, zz);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    qi[k] = pq[0][k];
    qn[0][k] = pq[1][k];
    qn[1][k] = pq[2][k];
    qn[4][k] = pq[3][k];
    qn[5][k] = pq[4][k];
  }
#pragma unroll
  for (int d = 2; d < 4; ++d)
#pragma unroll
    for (int k = 0; k < 5; ++k) qn[d][k] = ldg(Q + (size_t)k * N + nb[d]);
  lc_node<T>(B, qi, qn, h, p, &fp);
#pragma unroll
  for (int c = 0; c < 5; ++c) Hb[(size_t)c * N + i] = h[c];
  if (B.p.flow_on || (mode & FORCE_P)) {  // with the flow frozen only exports read the stress
#pragma unroll
    for (int c = 0; c < 9; ++c) Pb[(size_t)c * N + i] = p[c];
  }
}

// Stress tile of k_step: H and P stored once per fluid node.  A warp evaluates its row's
// nodes away from solids and walls together; nodes next to a solid or wall
// (surface values, colloid faces) are queued per warp and evaluated 32 at a
// time, so a row that crosses a colloid does not run the surface path with
// most of its lanes idle.
template <typename T, int TY>
__device__ __forceinline__ void stress_tile(const DevBox& B, const int4 td, int zc, int mode, int (*sq)[2 * TX],
                                            NearScratch<T>& sc) {
  if (!B.p.lc_on) return;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const PhysT<T>& PP = phys<T>(B);
  const T* __restrict__ Q = static_cast<const T*>(B.Q[B.st->qpar]);
  T* __restrict__ Hb = static_cast<T*>(B.H);
  T* __restrict__ Pb = static_cast<T*>(B.P);
  const int nx = B.nx, ny = B.ny;
  const int x = td.y + lane, y = td.z + wy;
  const int zend = min(td.w + zc, B.nz);
  const bool valid = x < nx && y < ny;
  int nq = 0;  // queued near nodes of this warp (warp-uniform)
  T qz[2][5];  // Q of the thread's own column at z - 1 and z, rolled down the z march
  column_start<T, 5>(B, Q, x, y, td.w, valid, qz);
  for (int z = td.w; z < zend; ++z) {
    const int i = x + nx * (y + ny * z);
    const uint8_t m = valid ? B.mask[i] : (uint8_t)1;
    const bool fluid = (m & IDMASK) == 0;
    const bool near = fluid && (m & NEAR);
    T pq[5][5];
    column_next<T, 5>(B, Q, x, y, z, valid, qz, pq);
    x_neighbours<T, 5>(Q, (size_t)B.N, pq[0], lane, x, nx, nx * (y + ny * z), valid, &pq[1]);
    T fp;
    if (fluid && !near) stress_node<T>(B, PP, Q, Hb, Pb, x, y, z, i, pq, mode, fp);
    const unsigned nb = __ballot_sync(0xffffffffu, near);
    if (nb) {
      if (near) sq[wy][nq + __popc(nb & ((1u << lane) - 1u))] = i;
      nq += __popc(nb);
      __syncwarp();
      if (nq >= TX) {
        near_stress<T>(B, sq[wy][lane], mode, sc);
        __syncwarp();
        nq -= TX;
        if (lane < nq) sq[wy][lane] = sq[wy][TX + lane];
        __syncwarp();
      }
    }
    column_roll<T, 5>(qz, pq);
  }
  near_stress<T>(B, lane < nq ? sq[wy][lane] : -1, mode, sc);
  __syncwarp();
}

// ---------------------------------------------------------------------------
// two-node paths of the FP32 kernels (boxes of even width)
// ---------------------------------------------------------------------------
// A lane holds the nodes x and x + 1 (x even) of its row, so a warp covers 64
// columns: the fields move as float2, the x-neighbours of the pair come from
// the adjacent lanes by one shuffle per component, and the per-node
// arithmetic of the two nodes runs together in packed FP32x2 (f2).  A pair
// with a node next to a solid or wall sends its fluid nodes through the
// per-warp queue of the one-node path.
__device__ __forceinline__ f2 ld2(const float* p) { return f2(__ldg(reinterpret_cast<const float2*>(p))); }
__device__ __forceinline__ void st2(float* p, f2 v) { *reinterpret_cast<float2*>(p) = v.v; }
__device__ __forceinline__ void st2_keep(float* p, f2 v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(p), "f"(v.v.x), "f"(v.v.y), "l"(pol)
               : "memory");
}

template <bool CG>
__device__ __forceinline__ f2 ldx2(const float* p) {
  const float2* q = reinterpret_cast<const float2*>(p);
  if constexpr (CG) return f2(__ldcg(q));
  else return f2(__ldg(q));
}

// The pair's values of a field row shifted by -s (s = +1: the nodes x - 1, x;
// s = -1: x + 1, x + 2), from the float2 v of the nodes x, x + 1 of the same
// row.  All lanes call it; edge lanes load the outside node from src_row.
template <bool CG>
__device__ __forceinline__ f2 shift_pair(f2 v, int s, int lane, bool valid, int x, int nx, const float* src_row) {
  const float left = __shfl_up_sync(0xffffffffu, v.v.y, 1);
  const float right = __shfl_down_sync(0xffffffffu, v.v.x, 1);
  if (s > 0) {
    float l = left;
    if (valid && lane == 0) l = ldx<CG>(src_row + (x == 0 ? nx - 1 : x - 1));
    return f2(l, v.v.x);
  }
  float r = right;
  if (valid && (lane == TX - 1 || x + 2 >= nx)) r = ldx<CG>(src_row + (x + 2 >= nx ? x + 2 - nx : x + 2));
  return f2(v.v.y, r);
}

// Push node j (when cond) onto the warp's queue sq[wy], evaluating 32 queued
// nodes with fn(j) whenever the queue holds 32 or more.  All lanes call it.
template <typename Fn>
__device__ __forceinline__ void queue_push(int (*sq)[2 * TX], int wy, int lane, int& nq, bool cond, int j, Fn fn) {
  const unsigned nb = __ballot_sync(0xffffffffu, cond);
  if (!nb) return;
  if (cond) sq[wy][nq + __popc(nb & ((1u << lane) - 1u))] = j;
  nq += __popc(nb);
  __syncwarp();
  if (nq >= TX) {
    fn(sq[wy][lane]);
    __syncwarp();
    nq -= TX;
    if (lane < nq) sq[wy][lane] = sq[wy][TX + lane];
    __syncwarp();
  }
}

// Stress tile of k_step, two nodes per lane: H and P of the pair from packed
// derivatives (the z-neighbours rolled down the column as in stress_tile).
// The loads of the next plane (mask, the column's z + 1 and the rows y +- 1)
// are issued before the current plane is evaluated, so their latency is
// covered by that plane's arithmetic rather than by other warps.
template <int TY>
__device__ __forceinline__ void stress_tile_pair(const DevBox& B, const LcPair& K2, const int4 td, int zc, int mode,
                                                 int (*sq)[2 * TX], NearScratch<float>& sc) {
  if (!B.p.lc_on) return;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const float* __restrict__ Q = static_cast<const float*>(B.Q[B.st->qpar]);
  float* __restrict__ Hb = static_cast<float*>(B.H);
  float* __restrict__ Pb = static_cast<float*>(B.P);
  const int nx = B.nx, ny = B.ny, nz = B.nz;
  const size_t N = (size_t)B.N;
  const int x = td.y + 2 * lane, y = td.z + wy;
  const int zend = min(td.w + zc, nz);
  const bool valid = x < nx && y < ny;
  const int yp = y + 1 == ny ? 0 : y + 1, ym = y == 0 ? ny - 1 : y - 1;
  int nq = 0;
  auto near_fn = [&](int j) { near_stress<float>(B, j, mode, sc); };
  f2 qz[2][5];  // the pair's Q at z - 1 and z, rolled down the z march
  f2 pz[5], pyp[5], pym[5];  // next plane's loads: the pair's Q at z + 1, the rows y + 1 and y - 1 at z
  unsigned pm2;              // and the pair's mask bytes at z
  auto fetch = [&](int z) {
    const int zp = z + 1 < nz ? z + 1 : (B.wall_z ? -1 : 0);
    pm2 = valid ? (unsigned)*reinterpret_cast<const uint16_t*>(B.mask + x + nx * (y + ny * z)) : 0x0101u;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      pz[k] = (valid && zp >= 0) ? ld2(Q + k * N + x + nx * (y + ny * zp)) : f2(0.f);
      pyp[k] = valid ? ld2(Q + k * N + x + nx * (yp + ny * z)) : f2(0.f);
      pym[k] = valid ? ld2(Q + k * N + x + nx * (ym + ny * z)) : f2(0.f);
    }
  };
  {
    const int zm = td.w > 0 ? td.w - 1 : (B.wall_z ? -1 : nz - 1);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      qz[0][k] = (valid && zm >= 0) ? ld2(Q + k * N + x + nx * (y + ny * zm)) : f2(0.f);
      qz[1][k] = valid ? ld2(Q + k * N + x + nx * (y + ny * td.w)) : f2(0.f);
    }
  }
  if (td.w < zend) fetch(td.w);
  for (int z = td.w; z < zend; ++z) {
    const int row = nx * (y + ny * z);
    const int i = x + row;
    const unsigned m2 = pm2;
    const uint8_t mA = (uint8_t)(m2 & 0xffu), mB = (uint8_t)(m2 >> 8);
    const bool fA = (mA & IDMASK) == 0, fB = (mB & IDMASK) == 0;
    const bool plain = fA && fB && !(mA & NEAR) && !(mB & NEAR);
    f2 qn[6][5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      qn[4][k] = pz[k];
      qn[2][k] = pyp[k];
      qn[3][k] = pym[k];
      qn[5][k] = qz[0][k];
    }
    if (z + 1 < zend) fetch(z + 1);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      qn[0][k] = shift_pair<false>(qz[1][k], -1, lane, valid, x, nx, Q + k * N + row);
      qn[1][k] = shift_pair<false>(qz[1][k], 1, lane, valid, x, nx, Q + k * N + row);
    }
    if (plain) {
      f2 dq[3][5], lap[5], h[5], p[9], fp;
      derivatives(qz[1], qn, dq, lap);
      lc_pair<true, true>(K2, qz[1], dq, lap, h, p, &fp);
      const uint64_t keep = l2_keep();
#pragma unroll
      for (int c = 0; c < 5; ++c) st2_keep(Hb + c * N + i, h[c], keep);
#pragma unroll
      for (int c = 0; c < 9; ++c) st2_keep(Pb + c * N + i, p[c], keep);
    }
    queue_push(sq, wy, lane, nq, fA && !plain, i, near_fn);
    queue_push(sq, wy, lane, nq, fB && !plain, i + 1, near_fn);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      qz[0][k] = qz[1][k];
      qz[1][k] = qn[4][k];
    }
  }
  near_fn(lane < nq ? sq[wy][lane] : -1);
  __syncwarp();
}

// ---------------------------------------------------------------------------
// nodes next to a solid or wall, and the plain tiles of the step kernels
// ---------------------------------------------------------------------------
// k_stress, k_lbp and k_lc take two kinds of work units: groups of 32 near
// nodes from the box's list, one per warp, and tiles, which leave the near
// nodes out.  The groups come first in the launch and spread over all SMs.  (With
// the near nodes queued by the warp that meets them, the warps whose column
// crosses a colloid ran batch after batch of the long surface path while the
// rest of the GPU had finished: 38 us for the stress of a 37 x 29 x 23 box with
// two colloids.)  Calls fn(B, node) for the group's node of this lane, or
// fn(B, -1).
template <int TY, typename Fn>
__device__ __forceinline__ void near_group(const DevBox& B, const int2* __restrict__ groups, int block, Fn fn) {
  const int e = groups[block * TY + threadIdx.y].y + (int)threadIdx.x;
  const int n = min(*B.nnear, B.near_cap);
  fn(e < n ? B.near_node[e] : -1);
}

// Planes of NC float components over a tile of 64 x TY columns and the rows
// y0 - 1 .. y0 + TY, four z planes in a ring in shared memory.  Per row: the 64
// columns, then the columns x0 - 1 and x0 + 64 (wrapped; the tile's own rows
// only).  A plane is copied by cp.async one plane of arithmetic ahead, so the
// march waits neither for memory nor holds prefetched values in registers;
// one barrier per plane separates the copies into a slot from its last reads.
template <int NC, int TY>
struct Ring {
  static constexpr int PW = 68, RY = TY + 2, PLANE = NC * RY * PW, SLOTS = 4;
  static constexpr size_t BYTES = sizeof(float) * PLANE * SLOTS;
};

__device__ __forceinline__ void cp_async8(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Columns of the tile at (td.y, td.z): where a lane finds its neighbours, and
// what the thread copies of each plane.  The 64 columns of the RY rows of a
// component are 16 RY pieces of 16 bytes, one per thread (rows whose length or
// base is not a multiple of 16 bytes: pieces of 8 bytes in turns); the two edge
// columns of all components are one 4-byte copy per thread, at offsets that are
// kept from plane to plane.  (Each lane copying its own pair, its row's edges
// and, by turns, the rows above and below took 24 copies a plane and warp for
// 5 components and 43 for 8, with their addresses a quarter of the kernels'
// instructions.  When that was changed, 128^3: k_stress 59 -> 44 us, k_lc 71 -> 53;
// 256 x 192 x 160: 167 -> 126 and 207 -> 162; a step of k_relax at 96^3 26.5 ->
// 22.2.)
struct RingLane {
  int x, y, row;   // node column, row start of y (node index)
  int li, ri;      // ring columns of x - 1 and x + 2
  int src, dst;    // first piece: offset in a plane of a component (-1: none), ring index
  int esrc, edst;  // edge value: offset in a plane (-1: none), ring index
  bool wide;       // pieces of 16 bytes
  bool valid;      // the lane's pair is a node pair
};

// Start of ring row r (0 .. RY - 1) of the tile in a plane, or -1: not read.
__device__ __forceinline__ int ring_row(const DevBox& B, const int4 td, int vy, int r) {
  if (r > vy + 1) return -1;
  int y = td.z + r - 1;
  y = y < 0 ? B.ny - 1 : (y >= B.ny ? 0 : y);
  return B.nx * y;
}

// Components 0 .. NF - 1 of the ring are F's, the next NC - NF are G's.
template <int NC, int TY, int NF>
__device__ __forceinline__ RingLane ring_lane(const DevBox& B, const int4 td, const float* F, const float* G) {
  using Rg = Ring<NC, TY>;
  static_assert(16 * Rg::RY <= 32 * TY && 2 * NC <= 32, "one piece and one edge value per thread");
  RingLane R;
  const int lane = threadIdx.x, nx = B.nx, ny = B.ny, t = lane + 32 * (int)threadIdx.y;
  const int vx = min(64, nx - td.y), vy = min(TY, ny - td.z);
  R.x = td.y + 2 * lane;
  R.y = td.z + (int)threadIdx.y;
  R.valid = R.x < nx && R.y < ny;
  R.row = nx * R.y;
  R.li = lane == 0 ? 64 : 2 * lane - 1;
  R.ri = 2 * lane + 2 >= vx ? 65 : 2 * lane + 2;
  R.wide = (nx & 3) == 0 && ((reinterpret_cast<uintptr_t>(F) | reinterpret_cast<uintptr_t>(G)) & 15) == 0;
  const int r = R.wide ? t >> 4 : t >> 5, c = R.wide ? 4 * (t & 15) : 2 * lane;
  const int row = r < Rg::RY && c < vx ? ring_row(B, td, vy, r) : -1;
  R.src = row < 0 ? -1 : row + td.y + c;
  R.dst = r * Rg::PW + c;
  const int k = t / (2 * TY), ry = (t >> 1) % TY, side = t & 1;
  const int xe = side ? (td.y + vx >= nx ? 0 : td.y + vx) : (td.y == 0 ? nx - 1 : td.y - 1);
  R.esrc = k < NC && ry < vy ? xe + nx * (td.z + ry) : -1;
  R.edst = (k * Rg::RY + ry + 1) * Rg::PW + 64 + side;
  return R;
}

// Copies plane z (-1 .. nz; wrapped, or nothing beyond a wall) of all
// components (strides N) into the ring.
template <int NC, int TY, int NF>
__device__ __forceinline__ void ring_load(float* ring, const DevBox& B, const RingLane& R, const int4 td,
                                          const float* __restrict__ F, const float* __restrict__ G, int z, int slot) {
  using Rg = Ring<NC, TY>;
  const int nz = B.nz;
  if (B.wall_z && (z < 0 || z >= nz)) return;
  const size_t base = (size_t)B.nx * B.ny * (z < 0 ? z + nz : (z >= nz ? z - nz : z));
  const size_t N = (size_t)B.N;
  float* dst = ring + slot * Rg::PLANE;
  if (R.esrc >= 0) {
    const int k = ((int)threadIdx.x + 32 * (int)threadIdx.y) / (2 * TY);
    cp_async4(dst + R.edst, (k < NF ? F + k * N : G + (k - NF) * N) + base + R.esrc);
  }
  if (R.wide) {
    if (R.src >= 0) {
      const float* p = F + base + R.src;
      const float* q = G + base + R.src;
#pragma unroll
      for (int k = 0; k < NC; ++k)
        cp_async16(dst + k * (Rg::RY * Rg::PW) + R.dst, k < NF ? p + k * N : q + (k - NF) * N);
    }
  } else {
    const int vx = min(64, B.nx - td.y), vy = min(TY, B.ny - td.z), c = 2 * (int)threadIdx.x;
    if (c < vx)
#pragma unroll 1
      for (int e = threadIdx.y; e < NC * (vy + 2); e += TY) {
        const int k = e / (vy + 2), r = e % (vy + 2);
        cp_async8(dst + (k * Rg::RY + r) * Rg::PW + c,
                  (k < NF ? F + k * N : G + (k - NF) * N) + base + ring_row(B, td, vy, r) + td.y + c);
      }
  }
}

__device__ __forceinline__ f2 sh2(const float* p) { return f2(*reinterpret_cast<const float2*>(p)); }

// Values of component k at the pair's own column and its six neighbours
// (the order of face_neighbours) in ring plane slot, from slots sm (z - 1)
// and sp (z + 1).
template <int NC, int TY>
__device__ __forceinline__ void ring_gather(const float* ring, const RingLane& R, int k, int s0, int sm, int sp,
                                            f2& own, f2 n[6]) {
  using Rg = Ring<NC, TY>;
  const int off = (k * Rg::RY + (int)threadIdx.y + 1) * Rg::PW, c = 2 * (int)threadIdx.x;
  const float* p = ring + s0 * Rg::PLANE + off;
  own = sh2(p + c);
  n[0] = f2(own.v.y, p[R.ri]);
  n[1] = f2(p[R.li], own.v.x);
  n[2] = sh2(p + Rg::PW + c);
  n[3] = sh2(p - Rg::PW + c);
  n[4] = sh2(ring + sp * Rg::PLANE + off + c);
  n[5] = sh2(ring + sm * Rg::PLANE + off + c);
}

__device__ __forceinline__ bool plain_node(unsigned m) { return (m & (IDMASK | NEAR)) == 0; }
// Both nodes of a pair are plain (two mask bytes).
__device__ __forceinline__ bool plain_pair(unsigned m2) { return (m2 & ((IDMASK | NEAR) * 0x0101u)) == 0; }

// Stress of a tile of plain nodes, two nodes per lane, Q from the ring.
template <int TY, bool FE, bool CHIRAL>
__device__ __forceinline__ void stress_ring(const DevBox& B, const LcPair& K2, const int4 td, int zc, int mode,
                                            float* ring, double& fe) {
  if (!B.p.lc_on) return;
  const float* __restrict__ Q = static_cast<const float*>(B.Q[B.st->qpar]);
  float* __restrict__ Hb = static_cast<float*>(B.H);
  float* __restrict__ Pb = static_cast<float*>(B.P);
  const RingLane R = ring_lane<5, TY, 5>(B, td, Q, Q);
  const int nz = B.nz, zend = min(td.w + zc, nz);
  const size_t N = (size_t)B.N;
  const uint64_t keep = l2_keep();
  const bool store_p = B.p.flow_on || (mode & FORCE_P);
  const uint8_t* mp = B.mask + R.x + R.row;
  const int plane = B.nx * B.ny;
  __syncthreads();  // the ring's last reads (previous tile) are done
#pragma unroll 1
  for (int k = -1; k <= 1; ++k) ring_load<5, TY, 5>(ring, B, R, td, Q, Q, td.w + k, (k + 1) & 3);
  cp_async_commit();
  unsigned m2 = R.valid ? (unsigned)*reinterpret_cast<const uint16_t*>(mp + (size_t)plane * td.w) : 0x0101u;
  for (int z = td.w; z < zend; ++z) {
    const int s0 = (z - td.w + 1) & 3;
    cp_async_wait0();
    __syncthreads();
    const bool plain = plain_pair(m2);
    if (z + 1 < zend) {
      ring_load<5, TY, 5>(ring, B, R, td, Q, Q, z + 2, (s0 + 2) & 3);
      if (R.valid) m2 = (unsigned)*reinterpret_cast<const uint16_t*>(mp + (size_t)plane * (z + 1));
    }
    cp_async_commit();
    if (!plain) continue;
    f2 qi[5], dq[3][5], lap[5], h[5], p[9], fp;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      f2 n[6];
      ring_gather<5, TY>(ring, R, k, s0, (s0 + 3) & 3, (s0 + 1) & 3, qi[k], n);
      dq[0][k] = n[0] - n[1];
      dq[1][k] = n[2] - n[3];
      dq[2][k] = n[4] - n[5];
      lap[k] = ((n[0] + n[1]) + (n[2] + n[3]) + (n[4] + n[5])) + K2.nsix * qi[k];
    }
    lc_pair<CHIRAL, true>(K2, qi, dq, lap, h, p, &fp);
    if constexpr (FE) fe += f32_to_f64(fp.v.x) + f32_to_f64(fp.v.y);
    const size_t i = (size_t)R.x + R.row + (size_t)plane * z;
#pragma unroll
    for (int c = 0; c < 5; ++c) st2_keep(Hb + c * N + i, h[c], keep);
    if (store_p) {  // with the flow frozen only exports read the stress
#pragma unroll
      for (int c = 0; c < 9; ++c) st2_keep(Pb + c * N + i, p[c], keep);
    }
  }
}

// Stress of a tile of plain nodes, one node per lane (odd widths, FP64).
template <typename T, bool FE>
__device__ __forceinline__ void stress_plain(const DevBox& B, const int4 td, int zc, int mode, double& fe) {
  if (!B.p.lc_on) return;
  const int lane = threadIdx.x;
  const T* __restrict__ Q = static_cast<const T*>(B.Q[B.st->qpar]);
  const int nx = B.nx, ny = B.ny, x = td.y + lane, y = td.z + (int)threadIdx.y;
  const int zend = min(td.w + zc, B.nz);
  const bool valid = x < nx && y < ny;
  T qz[2][5];
  column_start<T, 5>(B, Q, x, y, td.w, valid, qz);
  for (int z = td.w; z < zend; ++z) {
    const int i = x + nx * (y + ny * z);
    const uint8_t m = valid ? B.mask[i] : (uint8_t)1;
    T pq[5][5];
    column_next<T, 5>(B, Q, x, y, z, valid, qz, pq);
    x_neighbours<T, 5>(Q, (size_t)B.N, pq[0], lane, x, nx, nx * (y + ny * z), valid, &pq[1]);
    if (plain_node(m)) {
      T fp;
      stress_node<T>(B, phys<T>(B), Q, static_cast<T*>(B.H), static_cast<T*>(B.P), x, y, z, i, pq, mode, fp);
      if constexpr (FE) fe += to_f64(fp);
    }
    column_roll<T, 5>(qz, pq);
  }
}

// Sum of fe over the block's TY warps in warp order, by thread (0, 0) into *out.
template <int TY>
__device__ __forceinline__ void block_fe(double fe, double* out) {
  __shared__ double s_fe[TY];
  warp_sums<1>(&fe, [&](int, double t) { s_fe[threadIdx.y] = t; });
  __syncthreads();
  if (threadIdx.x + threadIdx.y == 0) {
    double t = 0.0;
    for (int k = 0; k < TY; ++k) t += s_fe[k];
    *out = t;
  }
  __syncthreads();
}

// H and P stored once per fluid node, and the colloid LC force from the near
// nodes.  FE (diagnostics): the free energy of each tile into part and of each
// block of near groups into L.fepart.
// FP32 tiles of even width: two nodes per lane from the ring, packed arithmetic,
// about 600 instructions a pair and warp, 16 warps per SM at 128 registers; bound
// by issue and by the FP32 pipe, which a packed instruction holds for two cycles
// (76 bytes a node: 23 us at 128^3).  One or two rows of a tile per thread, and 168
// registers with fewer warps, measured the same or slower.  FP64: bound by the
// FP64 pipe (84 % busy).  Near groups: a chain of FP64 surface values, 64 cycles
// an instruction and warp, spread over all SMs.  128^3 with one
// colloid: near nodes queued by tiles and Q by shuffles and loads 75 us, near
// groups and the ring 58, its copies in 16-byte pieces 44, the tiles of chiral and
// other boxes compiled apart 41 (one code with branches on q0: 52); 256 x 192 x
// 160, nematic: 117.
template <typename T, int TY, bool FE>
__global__ void __launch_bounds__(TX * TY, (sizeof(T) == 4 ? 512 : 256) / (TX * TY)) k_stress(Launch L, int mode,
                                                                                             double* __restrict__ part) {
  __shared__ DevBox B;
  __shared__ LcPair K2;
  extern __shared__ __align__(16) float ring[];
  int cur_box = -1;
  const int nn = L.ngroups / TY, units = nn + L.ntiles;
  for (int t = blockIdx.x; t < units; t += gridDim.x) {
    const int4 td = t < nn ? make_int4(L.groups[t * TY].x, 0, 0, 0) : L.tiles[t - nn];
    load_box<T>(B, K2, L.boxes, td.x, cur_box);
    double fe = 0.0;
    if (t < nn) {
      if (B.p.lc_on)
        near_group<TY>(B, L.groups, t, [&](int j) {
          near_stress<T>(B, j, mode, reinterpret_cast<NearScratch<T>*>(ring)[threadIdx.y], nullptr, FE ? &fe : nullptr);
        });
      __syncthreads();
    } else {
      bool done = false;
      if constexpr (sizeof(T) == 4) {
        if (pair_box(B)) {
          if (B.p.q0 != 0.0) stress_ring<TY, FE, true>(B, K2, td, L.zc, mode, ring, fe);
          else stress_ring<TY, FE, false>(B, K2, td, L.zc, mode, ring, fe);
          done = true;
        }
      }
      if (!done) stress_plain<T, FE>(B, td, L.zc, mode, fe);
    }
    if constexpr (FE) block_fe<TY>(fe, t < nn ? L.fepart + t : part + (t - nn));
  }
}

// Body force at fluid node i from the stored stress: the face divergence of
// k_flb, sum over the six faces of +-(face value), the face value the mean of
// the two nodes' P or, across a solid or wall face, P(i).  With six fluid
// neighbours the P(i) halves cancel.
template <typename T, bool CG = false>
__device__ __forceinline__ void stored_force(const DevBox& B, const T* __restrict__ Pb, int x, int y, int z, int i,
                                             uint8_t m, T F[3]) {
  const size_t N = (size_t)B.N;
  int nb[6], zz[2];
  face_neighbours(B, x, y, z, nb, zz);
  if (!(m & NEAR)) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const T* Pa = Pb + (size_t)(3 * a) * N;
      F[a] = T(0.5) * ((ldx<CG>(Pa + nb[0]) - ldx<CG>(Pa + nb[1])) + (ldx<CG>(Pa + N + nb[2]) - ldx<CG>(Pa + N + nb[3])) +
                       (ldx<CG>(Pa + 2 * N + nb[4]) - ldx<CG>(Pa + 2 * N + nb[5])));
    }
    return;
  }
  // near node: the six mask bytes, then all stress values, in one round of
  // loads each (a closed face reads P(i), which is its face value)
  size_t j[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) j[d] = nb[d] >= 0 && (B.mask[nb[d] < 0 ? i : nb[d]] & IDMASK) == 0 ? nb[d] : i;
  T v[6][3], pc[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) pc[c] = ldx<CG>(Pb + (size_t)c * N + i);
#pragma unroll
  for (int d = 0; d < 6; ++d)
#pragma unroll
    for (int a = 0; a < 3; ++a) v[d][a] = ldx<CG>(Pb + (size_t)(3 * a + (d >> 1)) * N + j[d]);
  F[0] = F[1] = F[2] = T(0);
#pragma unroll
  for (int d = 0; d < 6; ++d)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const T face = T(0.5) * (pc[3 * a + (d >> 1)] + v[d][a]);
      F[a] += (d & 1) ? -face : face;
    }
}

// One fluid node of k_lbp: pull (bounce-back only for near nodes), body force
// from the stored P, collide, store.  For a plain node the mask handed down
// has the near bit cleared, which removes the neighbour checks at compile time.
template <typename T, bool NEAR_NODE, bool CG = false>
__device__ __forceinline__ void lbp_node(const DevBox& B, const PhysT<T>& PP, const T* __restrict__ fin,
                                         T* __restrict__ fout, const T* __restrict__ Pb, T* __restrict__ ub, int x,
                                         int y, int z, int i, uint8_t m, bool pre, bool lc) {
  const uint8_t mm = NEAR_NODE ? m : (uint8_t)(m & (uint8_t)~NEAR);
  T df[NQ];
  pull(B, fin, x, y, z, i, mm, pre, df);
  T Fx = PP.g[0], Fy = PP.g[1], Fz = PP.g[2];
  if (lc) {
    T Fv[3];
    stored_force<T, CG>(B, Pb, x, y, z, i, mm, Fv);
    Fx += Fv[0];
    Fy += Fv[1];
    Fz += Fv[2];
  }
  collide_store(PP, fout, ub, B.N, i, df, Fx, Fy, Fz);
}

// LB tile of k_step: as there, a warp collides the plain fluid nodes of its row
// together and queues the nodes next to a solid or wall (bounce-back links,
// solid faces of the force) in shared memory, 32 at a time.
template <typename T, int TY, bool CG>
__device__ __forceinline__ void lbp_tile(const DevBox& B, const int4 td, int zc, int (*sq)[2 * TX]) {
  if (!B.p.flow_on) return;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const PhysT<T>& PP = phys<T>(B);
  const int fpar = B.st->fpar;
  const bool pre = B.st->pre_valid != 0;
  const T* __restrict__ fin = static_cast<const T*>(B.f[fpar]);
  T* __restrict__ fout = static_cast<T*>(B.f[fpar ^ 1]);
  const T* __restrict__ Pb = static_cast<const T*>(B.P);
  T* __restrict__ ub = static_cast<T*>(B.u);
  const int nx = B.nx, ny = B.ny;
  const int x = td.y + lane, y = td.z + wy;
  const int zend = min(td.w + zc, B.nz);
  const bool valid = x < nx && y < ny;
  const bool lc = B.p.lc_on != 0;
  int nq = 0;
  for (int z = td.w; z < zend; ++z) {
    const int i = x + nx * (y + ny * z);
    const uint8_t m = valid ? B.mask[i] : (uint8_t)0;
    const bool fluid = valid && (m & IDMASK) == 0;
    const bool near = fluid && (m & NEAR);
    if (valid && !fluid) solid_velocity(B, ub, x, y, z, i, m);
    if (fluid && !near) lbp_node<T, false, CG>(B, PP, fin, fout, Pb, ub, x, y, z, i, m, pre, lc);
    const unsigned nb = __ballot_sync(0xffffffffu, near);
    if (nb) {
      if (near) sq[wy][nq + __popc(nb & ((1u << lane) - 1u))] = i;
      nq += __popc(nb);
      __syncwarp();
      if (nq >= TX) {
        const int j = sq[wy][lane];
        lbp_node<T, true, CG>(B, PP, fin, fout, Pb, ub, j % nx, (j / nx) % ny, j / (nx * ny), j, B.mask[j], pre, lc);
        __syncwarp();
        nq -= TX;
        if (lane < nq) sq[wy][lane] = sq[wy][TX + lane];
        __syncwarp();
      }
    }
  }
  if (lane < nq) {
    const int j = sq[wy][lane];
    lbp_node<T, true, CG>(B, PP, fin, fout, Pb, ub, j % nx, (j / nx) % ny, j / (nx * ny), j, B.mask[j], pre, lc);
  }
  __syncwarp();
}

// Tile of k_lbp: the plain nodes collided, solid nodes given the colloid's
// velocity.
template <typename T>
__device__ __forceinline__ void lbp_plain(const DevBox& B, const int4 td, int zc) {
  const int nx = B.nx, ny = B.ny, x = td.y + (int)threadIdx.x, y = td.z + (int)threadIdx.y;
  if (x >= nx || y >= ny) return;
  const int fpar = B.st->fpar, zend = min(td.w + zc, B.nz);
  const bool pre = B.st->pre_valid != 0, lc = B.p.lc_on != 0;
  const T* __restrict__ fin = static_cast<const T*>(B.f[fpar]);
  T* __restrict__ fout = static_cast<T*>(B.f[fpar ^ 1]);
  for (int z = td.w; z < zend; ++z) {
    const int i = x + nx * (y + ny * z);
    const uint8_t m = B.mask[i];
    if (plain_node(m))
      lbp_node<T, false>(B, phys<T>(B), fin, fout, static_cast<const T*>(B.P), static_cast<T*>(B.u), x, y, z, i, m,
                         pre, lc);
    else if (m & IDMASK)
      solid_velocity(B, static_cast<T*>(B.u), x, y, z, i, m);
  }
}

// Near node of k_lbp (a listed node that is not next to a solid is a plain
// node here: the tiles collide it).
template <typename T>
__device__ __forceinline__ void near_lbp(const DevBox& B, int j) {
  if (j < 0 || !(B.mask[j] & NEAR)) return;
  const int fpar = B.st->fpar;
  lbp_node<T, true>(B, phys<T>(B), static_cast<const T*>(B.f[fpar]), static_cast<T*>(B.f[fpar ^ 1]),
                    static_cast<const T*>(B.P), static_cast<T*>(B.u), j % B.nx, (j / B.nx) % B.ny,
                    j / (B.nx * B.ny), j, B.mask[j], B.st->pre_valid != 0, B.p.lc_on != 0);
}

// Bound by the memory system: 38 population streams of 4 bytes a node, 18
// stress values and 3 velocities: 159 MB of populations read and written and 75
// MB of stress at 128^3 (70 us under the profiler, 5.0 TB/s; 76 in the step, 280
// at 256 x 192 x 160).  What hides the
// latency is warps: 64 registers for 32 warps per SM 77 us, 80 registers 87, 48
// registers 88.  The rows of the next plane staged in shared memory by 16-byte
// asynchronous copies, which leaves 20 warps per SM: 94.  (Opposite directions
// collided together, in a sum of another order, saved 2 us.)
template <typename T, int TY>
__global__ void __launch_bounds__(TX * TY, (sizeof(T) == 4 ? 1024 : 384) / (TX * TY)) k_lbp(Launch L) {
  __shared__ DevBox B;
  int cur_box = -1;
  const int nn = L.ngroups / TY, units = nn + L.ntiles;
  for (int t = blockIdx.x; t < units; t += gridDim.x) {
    const int4 td = t < nn ? make_int4(L.groups[t * TY].x, 0, 0, 0) : L.tiles[t - nn];
    load_box(B, L.boxes, td.x, cur_box);
    if (!B.p.flow_on) continue;
    if (t < nn) {
      near_group<TY>(B, L.groups, t, [&](int j) { near_lbp<T>(B, j); });
      continue;
    }
    lbp_plain<T>(B, td, L.zc);
  }
}

// ---------------------------------------------------------------------------
// k_flb: stress + body force + collide/stream fused (the step kernel)
// ---------------------------------------------------------------------------
// Tile: 32 x BY interior columns marching z.  Threads: 32*(BY+2) cover the
// stress positions of the tile rows and the two y-halo rows (whole warps),
// one more warp the two x-halo columns, so every halo position of a plane is
// computed in a single pass.  Warps 1..BY then run the body force and the LB
// collide of their interior node; the stress never leaves shared memory and
// the body force never reaches HBM.
template <typename T, int BY>
__global__ void __launch_bounds__(32 * (BY + 3), (sizeof(T) == 4 && BY <= 4) ? 2 : 1) k_flb(
    const DevBox* __restrict__ boxes, const int4* __restrict__ tiles, int ntiles, int zc, int mode,
    double* __restrict__ part) {
  constexpr int HX = TX + 2, HY = BY + 2, HP = HX * HY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sP = reinterpret_cast<T*>(smem_raw);
  uint8_t* sFl = smem_raw + sizeof(T) * 27 * HP;
  __shared__ DevBox B;
  const int tid = threadIdx.x;
  // this thread's stress position (hx, hy) in the halo'd plane, or none
  int hx, hy;
  if (tid < 32 * HY) {
    hx = 1 + (tid & 31);
    hy = tid >> 5;
  } else {
    const int k = tid - 32 * HY;
    hx = k < HY ? 0 : (k < 2 * HY ? HX - 1 : -1);
    hy = k < HY ? k : k - HY;
  }
  const int pidx = hx >= 0 ? hx + HX * hy : -1;
  const bool lbthread = tid >= 32 && tid < 32 * (BY + 1);
  const int tx = tid & 31, ty = (tid >> 5) - 1;

  int cur_box = -1;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int4 td = tiles[t];
    load_box(B, boxes, td.x, cur_box);
    const PhysT<T>& PP = phys<T>(B);
    const bool lc = B.p.lc_on != 0, flow = B.p.flow_on != 0;
    if (!flow && !lc) continue;
    int my_c = -1;
    double my_acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const T* __restrict__ Q = static_cast<const T*>(B.Q[B.st->qpar]);
    const int fpar = B.st->fpar;
    const bool pre = B.st->pre_valid != 0;
    const T* __restrict__ fin = static_cast<const T*>(B.f[fpar]);
    T* __restrict__ fout = static_cast<T*>(B.f[fpar ^ 1]);
    T* __restrict__ ub = static_cast<T*>(B.u);
    const int x0 = td.y, y0 = td.z, z0 = td.w;
    const int nx = B.nx, ny = B.ny, nz = B.nz, N = B.N;
    const int vx = min(TX, nx - x0), vy = min(BY, ny - y0);
    const int zend = min(z0 + zc, nz);
    const bool mypos = pidx >= 0 && hx <= vx + 1 && hy <= vy + 1;
    const int gx = wrapn(x0 - 1 + hx, nx), gy = wrapn(y0 - 1 + hy, ny);
    const bool myint = lbthread && tx < vx && ty < vy;
    for (int k = z0 - 1; k <= zend; ++k) {
      const int slot = (k - z0 + 1) % 3;
      if (lc && mypos) {
        const bool wallplane = B.wall_z && (k < 0 || k >= nz);
        const int kk = B.wall_z ? k : wrapn(k, nz);
        const bool inner = hx >= 1 && hx <= vx && hy >= 1 && hy <= vy && k >= z0 && k < zend;
        sFl[slot * HP + pidx] =
            wallplane ? WALLFLAG
                      : stress_at(B, PP, Q, gx, gy, kk, sP + slot * 9 * HP + pidx, HP,
                                  inner ? static_cast<T*>(B.H) : (T*)nullptr);
      }
      __syncthreads();
      if (k >= z0 + 1 && myint) {
        const int kc = k - 1;
        const int x = x0 + tx, y = y0 + ty;
        const int i = x + nx * (y + ny * kc);
        const uint8_t m = B.mask[i];
        if (m & IDMASK) {
          if (flow) solid_velocity(B, ub, x, y, kc, i, m);
        } else {
          T Fv[3] = {T(0), T(0), T(0)};
          if (lc)
            face_force(B, sP, sFl, HP, HX, (k - z0) % 3, (k - z0 - 1) % 3, slot, (tx + 1) + HX * (ty + 1), x, y, kc,
                       (mode & FORCE_ACC) != 0, Fv, my_c, my_acc);
          if (flow) {
            T df[NQ];
            pull(B, fin, x, y, kc, i, m, pre, df);
            collide_store(PP, fout, ub, N, i, df, Fv[0] + PP.g[0], Fv[1] + PP.g[1], Fv[2] + PP.g[2]);
          }
        }
      }
      __syncthreads();
    }
    if (mode & FORCE_ACC) warp_flush_colloid(B.col, my_c, my_acc, 6);
  }
}

// ---------------------------------------------------------------------------
// k_lc: Beris-Edwards update
// ---------------------------------------------------------------------------
// Beris-Edwards update of fluid node i (Eq. 2): co-rotation from the central
// velocity gradient, upwind advective fluxes through the faces (zero across
// solid or wall faces, which only near nodes have), H stored by the stress
// kernel of this step; Q^{n+1} stored, residual folded into (rsum, rmax).
// A plain node (NEAR_NODE false) takes its own Q and u and those of its
// x-neighbours from pq and pu (self, x + 1, x - 1; gathered by the warp).
// Holding the z-neighbours in registers down the z march, as the stress
// kernel does, pushed this kernel past its 96-register cap (spills, 76 us
// against 71 us).
template <typename T, bool NEAR_NODE, bool CG = false>
__device__ __forceinline__ void lc_update_node(const DevBox& B, const PhysT<T>& PP, const T* __restrict__ Q,
                                               const __nv_bfloat16* __restrict__ Lin, const T* __restrict__ U, int qpar,
                                               int x, int y, int z, int i, T& rsum, T& rmax,
                                               const T (*pq)[5] = nullptr, const T (*pu)[3] = nullptr,
                                               const float* plo = nullptr) {
  const int N = B.N;
  // H of this node was stored by the stress kernel of this step; Q of the
  // fluid face neighbours is needed only for the advective fluxes (zero
  // across solid faces), so no surface values are formed here.  Near nodes
  // read the six mask bytes first and then everything else in one round of
  // independent loads (a closed face loads the node's own Q, unused).
  float lo[5];
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int c = 0; c < 5; ++c) lo[c] = NEAR_NODE ? __bfloat162float(Lin[(size_t)c * N + i]) : plo[c];
  }
  const T* __restrict__ Hb = static_cast<const T*>(B.H);
  T qi[5], qn[6][5], h[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    qi[c] = NEAR_NODE ? ldg(Q + (size_t)c * N + i) : pq[0][c];
    h[c] = ldx<CG>(Hb + (size_t)c * N + i);
  }
  int nb[6], zz[2];
  face_neighbours(B, x, y, z, nb, zz);
  T ui[3], un[6][3];
  bool fl[6];
#pragma unroll
  for (int a = 0; a < 3; ++a) ui[a] = NEAR_NODE ? ldx<CG>(U + (size_t)a * N + i) : pu[0][a];
#pragma unroll
  for (int d = 0; d < 6; ++d) fl[d] = !NEAR_NODE || (nb[d] >= 0 && (B.mask[nb[d] < 0 ? i : nb[d]] & IDMASK) == 0);
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const int j = nb[d];
    if (!NEAR_NODE && d < 2) {
#pragma unroll
      for (int a = 0; a < 3; ++a) un[d][a] = pu[1 + d][a];
#pragma unroll
      for (int c = 0; c < 5; ++c) qn[d][c] = pq[1 + d][c];
      continue;
    }
    const size_t ju = NEAR_NODE && j < 0 ? i : j, jq = fl[d] ? j : i;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      un[d][a] = ldx<CG>(U + (size_t)a * N + ju);
      if (NEAR_NODE && j < 0) un[d][a] = T(0);
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) qn[d][c] = ldg(Q + (size_t)c * N + jq);
  }
  T d5[5];
  if constexpr (sizeof(T) == 4) {
    q_increment_f32<true>(PP, qi, qn, ui, un, fl, h, lo, d5);
  } else {
    T G[9], cd[6], self, adv[5];
    flow_terms<T>(B.kd, ui, un, fl, G, cd, self);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const T n[6] = {qn[0][k], qn[1][k], qn[2][k], qn[3][k], qn[4][k], qn[5][k]};
      adv[k] = advect(cd, self, qi[k], n);
    }
    q_increment<true, T>(B.kd, qi, adv, G, h, d5);
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) store_q_next<T>(B, qpar, i, k, qi[k], sizeof(T) == 4 ? lo[k] : 0.f, d5[k]);
  add_residual(d5, rsum, rmax);
}

// Q-update tile of k_step: plain nodes of a warp's row together, nodes
// next to a solid or wall queued and updated 32 at a time.  part (if non-null)
// receives the tile's residual partials (sum of squares, max), one record per
// warp (TY records per tile).
template <typename T, int TY, bool CG>
__device__ __forceinline__ void lc_tile(const DevBox& B, const int4 td, int zc, double* part, int (*sq)[2 * TX]) {
  if (!B.p.lc_on) return;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int qpar = B.st->qpar;
  const T* __restrict__ Q = static_cast<const T*>(B.Q[qpar]);
  const __nv_bfloat16* __restrict__ Lin = B.Qlo[qpar];
  const T* __restrict__ U = static_cast<const T*>(B.u);
  const int nx = B.nx, ny = B.ny;
  const int x = td.y + lane, y = td.z + wy;
  const int zend = min(td.w + zc, B.nz);
  const bool valid = x < nx && y < ny;
  const PhysT<T>& PP = phys<T>(B);
  T rsum = T(0), rmax = T(0);  // per-thread residual (sum of squares, max), in T
  int nq = 0;
  for (int z = td.w; z < zend; ++z) {
    const int i = x + nx * (y + ny * z);
    const uint8_t m = valid ? B.mask[i] : (uint8_t)1;
    const bool fluid = (m & IDMASK) == 0;
    const bool near = fluid && (m & NEAR);
    T pq[3][5], pu[3][3];
    float plo[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) pq[0][k] = valid ? ldg(Q + (size_t)k * B.N + i) : T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) pu[0][a] = valid ? ldx<CG>(U + (size_t)a * B.N + i) : T(0);
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int k = 0; k < 5; ++k) plo[k] = (valid && fluid && !near) ? __bfloat162float(Lin[(size_t)k * B.N + i]) : 0.f;
    }
    const int row = nx * (y + ny * z);
    x_neighbours<T, 5>(Q, (size_t)B.N, pq[0], lane, x, nx, row, valid, &pq[1]);
    x_neighbours<T, 3, CG>(U, (size_t)B.N, pu[0], lane, x, nx, row, valid, &pu[1]);
    if (fluid && !near)
      lc_update_node<T, false, CG>(B, PP, Q, Lin, U, qpar, x, y, z, i, rsum, rmax, pq, pu, plo);
    const unsigned nb = __ballot_sync(0xffffffffu, near);
    if (nb) {
      if (near) sq[wy][nq + __popc(nb & ((1u << lane) - 1u))] = i;
      nq += __popc(nb);
      __syncwarp();
      if (nq >= TX) {
        const int j = sq[wy][lane];
        lc_update_node<T, true, CG>(B, PP, Q, Lin, U, qpar, j % nx, (j / nx) % ny, j / (nx * ny), j, rsum, rmax);
        __syncwarp();
        nq -= TX;
        if (lane < nq) sq[wy][lane] = sq[wy][TX + lane];
        __syncwarp();
      }
    }
  }
  if (lane < nq) {
    const int j = sq[wy][lane];
    lc_update_node<T, true, CG>(B, PP, Q, Lin, U, qpar, j % nx, (j / nx) % ny, j / (nx * ny), j, rsum, rmax);
  }
  __syncwarp();
  if (part) warp_residual<T>(part, wy, lane, rsum, rmax);
}

// Q-update tile of k_step, two nodes per lane (FP32 boxes of even width; tiles 64 wide): the
// Beris-Edwards update of lc_update_node for the nodes x, x + 1 at once, in
// packed FP32x2 arithmetic, with Q, u, H and the BF16 remainder of Q moved as
// pairs.
__device__ __forceinline__ void lc_update_pair(const DevBox& B, const LcPair& K2, float* __restrict__ Qo,
                                               __nv_bfloat16* __restrict__ Lout, int i, const f2 qi[5],
                                               const f2 qn[6][5], const f2 ui[3], const f2 un[6][3], const f2 hin[5],
                                               const f2 lo[5], float& rsum, float& rmax) {
  const size_t N = (size_t)B.N;
  f2 w[3][3], up[6], dn[6], adv[5], h[5], d5[5];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    upwind_pair(ui[a], un[2 * a][a], un[2 * a + 1][a], up + 2 * a, dn + 2 * a);
#pragma unroll
    for (int j = 0; j < 3; ++j) w[a][j] = un[2 * j][a] - un[2 * j + 1][a];
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const f2 n[6] = {qn[0][k], qn[1][k], qn[2][k], qn[3][k], qn[4][k], qn[5][k]};
    adv[k] = advect_pair(up, dn, qi[k], n);
    h[k] = hin[k];
  }
  q_pair(K2, qi, adv, w, h, lo, d5);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const f2 v = d5[k];
    // compensated storage: hi + lo + v carried exactly into (hi, lo) (two-sum)
    const f2 sv = lo[k] + v;
    const f2 hn = qi[k] + sv;
    const f2 bb = hn - qi[k];
    const f2 err = (qi[k] - (hn - bb)) + (sv - bb);
    st2(Qo + (size_t)k * N + i, hn);
    *reinterpret_cast<__nv_bfloat162*>(Lout + (size_t)k * N + i) = __float22bfloat162_rn(err.v);
  }
  const f2 dzz = -(d5[0] + d5[3]);
  const f2 r2 = d5[0] * d5[0] + d5[3] * d5[3] + dzz * dzz + 2.f * (d5[1] * d5[1] + d5[2] * d5[2] + d5[4] * d5[4]);
  rsum += r2.v.x + r2.v.y;
  float mx = fmaxf(fabsf(dzz.v.x), fabsf(dzz.v.y));
#pragma unroll
  for (int k = 0; k < 5; ++k) mx = fmaxf(mx, fmaxf(fabsf(d5[k].v.x), fabsf(d5[k].v.y)));
  rmax = fmaxf(rmax, mx);
}

template <int TY, bool CG>
__device__ __forceinline__ void lc_tile_pair(const DevBox& B, const LcPair& K2, const int4 td, int zc, double* part,
                                             int (*sq)[2 * TX]) {
  if (!B.p.lc_on) return;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int qpar = B.st->qpar;
  const float* __restrict__ Q = static_cast<const float*>(B.Q[qpar]);
  float* __restrict__ Qo = static_cast<float*>(B.Q[qpar ^ 1]);
  const __nv_bfloat16* __restrict__ Lin = B.Qlo[qpar];
  __nv_bfloat16* __restrict__ Lout = B.Qlo[qpar ^ 1];
  const float* __restrict__ U = static_cast<const float*>(B.u);
  const float* __restrict__ Hb = static_cast<const float*>(B.H);
  const int nx = B.nx, ny = B.ny, nz = B.nz;
  const size_t N = (size_t)B.N;
  const int x = td.y + 2 * lane, y = td.z + wy;
  const int zend = min(td.w + zc, nz);
  const bool valid = x < nx && y < ny;
  const int yp = y + 1 == ny ? 0 : y + 1, ym = y == 0 ? ny - 1 : y - 1;
  float rsum = 0.f, rmax = 0.f;
  int nq = 0;
  auto near_fn = [&](int j) {
    lc_update_node<float, true, CG>(B, B.pf, Q, Lin, U, qpar, j % nx, (j / nx) % ny, j / (nx * ny), j, rsum, rmax);
  };
  for (int z = td.w; z < zend; ++z) {
    const int row = nx * (y + ny * z);
    const int i = x + row;
    const unsigned m2 = valid ? (unsigned)*reinterpret_cast<const uint16_t*>(B.mask + i) : 0x0101u;
    const uint8_t mA = (uint8_t)(m2 & 0xffu), mB = (uint8_t)(m2 >> 8);
    const bool fA = (mA & IDMASK) == 0, fB = (mB & IDMASK) == 0;
    const bool plain = fA && fB && !(mA & NEAR) && !(mB & NEAR);
    f2 qi[5], ui[3], qn[6][5], un[6][3];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      qi[k] = valid ? ldx2<false>(Q + k * N + i) : f2(0.f);
      qn[0][k] = shift_pair<false>(qi[k], -1, lane, valid, x, nx, Q + k * N + row);
      qn[1][k] = shift_pair<false>(qi[k], 1, lane, valid, x, nx, Q + k * N + row);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ui[a] = valid ? ldx2<CG>(U + a * N + i) : f2(0.f);
      un[0][a] = shift_pair<CG>(ui[a], -1, lane, valid, x, nx, U + a * N + row);
      un[1][a] = shift_pair<CG>(ui[a], 1, lane, valid, x, nx, U + a * N + row);
    }
    if (plain) {
      const int zp = z + 1 == nz ? 0 : z + 1, zm = z == 0 ? nz - 1 : z - 1;  // no wall next to a plain node
      const int jr[4] = {x + nx * (yp + ny * z), x + nx * (ym + ny * z), x + nx * (y + ny * zp),
                         x + nx * (y + ny * zm)};
      f2 h[5], lo[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
#pragma unroll
        for (int d = 0; d < 4; ++d) qn[2 + d][k] = ldx2<false>(Q + k * N + jr[d]);
        h[k] = ldx2<CG>(Hb + k * N + i);
        lo[k] = f2(__bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(Lin + k * N + i)));
      }
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int d = 0; d < 4; ++d) un[2 + d][a] = ldx2<CG>(U + a * N + jr[d]);
      lc_update_pair(B, K2, Qo, Lout, i, qi, qn, ui, un, h, lo, rsum, rmax);
    }
    queue_push(sq, wy, lane, nq, valid && fA && !plain, i, near_fn);
    queue_push(sq, wy, lane, nq, valid && fB && !plain, i + 1, near_fn);
  }
  if (lane < nq) near_fn(sq[wy][lane]);
  __syncwarp();
  if (part) warp_residual<float>(part, wy, lane, rsum, rmax);
}

// ---------------------------------------------------------------------------
// k_links: momentum exchange on the boundary links
// ---------------------------------------------------------------------------
// Per link (fluid r, direction b into colloid c): dp = c_b (2 df*_b(r) -
// 6 w_b rho0 c_b.u_b), u_b the rigid velocity at r + c_b/2; torque
// (r + c_b/2 - X) x dp.  The constant w_b rho0 part of 2 f*_b sums to zero
// over a closed surface and is left out.
// One chunk of links (box record B, first link l0, count n) by all threads of
// the block; sblk holds 18 doubles, sc0 one int of shared memory.
template <typename T, bool CG>
__device__ __forceinline__ void links_chunk(const DevBox& B, int l0, int n, double* sblk, int* sc0) {
  if (!B.p.flow_on) return;
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  const int nthr = blockDim.x * blockDim.y;
  const int nl = *B.nlinks;
  for (int base = l0; base < l0 + n; base += nthr) {
    const int l = base + tid;
    int my_c = -1;
    bool mob = false;
    // dp (3), torque (3), then for mobile colloids the drag tensors zv, zw (6 + 6)
    double v[18];
#pragma unroll
    for (int k = 0; k < 18; ++k) v[k] = 0.0;
    // the sub-chunk's first colloid is summed in shared memory (links are sorted by colloid)
    __syncthreads();
    if (tid < 18) sblk[tid] = 0.0;
    if (tid == 0) *sc0 = (base < nl && base < B.nlinks_cap) ? (int)B.link_col[base] : -1;
    __syncthreads();
    if (l < l0 + n && l < nl && l < B.nlinks_cap) {
      const int i = B.link_node[l];
      const int q = B.link_dir[l];
      const int c = B.link_col[l];
      const T* fout = static_cast<const T*>(B.f[B.st->fpar ^ 1]);
      const double dfq = to_f64(ldx<CG>(fout + (size_t)q * B.N + i));
      const int x = i % B.nx, y = (i / B.nx) % B.ny, z = i / (B.nx * B.ny);
      int qx = 0, qy = 0, qz = 0;
      switch (q) {
#define LCLB_CASE(k) case k: qx = cx(k); qy = cy(k); qz = cz(k); break;
        LCLB_CASE(1) LCLB_CASE(2) LCLB_CASE(3) LCLB_CASE(4) LCLB_CASE(5) LCLB_CASE(6) LCLB_CASE(7) LCLB_CASE(8)
        LCLB_CASE(9) LCLB_CASE(10) LCLB_CASE(11) LCLB_CASE(12) LCLB_CASE(13) LCLB_CASE(14) LCLB_CASE(15)
        LCLB_CASE(16) LCLB_CASE(17) LCLB_CASE(18)
#undef LCLB_CASE
        default: break;
      }
      const DevColloid& C = B.col[c];
      double d[3];
      disp(B, x + 0.5 * qx, y + 0.5 * qy, z + 0.5 * qz, C.X, d);
      // with rc = d x c_b, c_b.(V + W x d) = c_b.V + W.rc and the torque of
      // dp = mag c_b is mag rc
      const double cc[3] = {(double)qx, (double)qy, (double)qz};
      const double rc[3] = {d[1] * cc[2] - d[2] * cc[1], d[2] * cc[0] - d[0] * cc[2], d[0] * cc[1] - d[1] * cc[0]};
      const double zk = (q <= 6 ? 6.0 / 18.0 : 6.0 / 36.0) * B.p.rho0;
      const double cub = cc[0] * C.V[0] + cc[1] * C.V[1] + cc[2] * C.V[2] + rc[0] * C.W[0] + rc[1] * C.W[1] + rc[2] * C.W[2];
      const double mag = 2.0 * dfq - zk * cub;
      my_c = c;
      for (int a = 0; a < 3; ++a) {
        v[a] = cc[a] * mag;
        v[3 + a] = rc[a] * mag;
      }
      mob = C.mobile != 0;
      if (mob) {
        // the part of dp linear in the rigid velocity, -6 w rho0 c (c.(V + W x d)):
        // coefficients 6 w rho0 c c (V-V) and 6 w rho0 (d x c)(d x c) (W-W)
        const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          v[6 + k] = zk * (cc[ia[k]] * cc[ib[k]]);
          v[12 + k] = zk * rc[ia[k]] * rc[ib[k]];
        }
      }
    }
    const int c0 = *sc0;
    const bool main = (my_c == c0) && c0 >= 0;
    const bool warp_main = __all_sync(0xffffffffu, main || my_c < 0);
    const bool warp_mob = __any_sync(0xffffffffu, mob);
    if (warp_main) {
      auto add = [&](int k, double t) {
        if (t != 0.0) atomicAdd(&sblk[k], t);
      };
      if (warp_mob) warp_sums<18>(v, add);
      else warp_sums<6>(v, add);
    } else {
      warp_flush_colloid<6>(B.col, my_c, v, 0);
      if (warp_mob) warp_flush_colloid<12>(B.col, mob ? my_c : -1, v + 6, 12);
    }
    __syncthreads();
    if (tid < 18 && c0 >= 0 && sblk[tid] != 0.0) atomicAdd(&B.col[c0].acc[tid < 6 ? tid : tid + 6], sblk[tid]);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_links(const DevBox* __restrict__ boxes, const int2* __restrict__ chunks,
                                               int nchunks) {
  __shared__ DevBox B;
  __shared__ double sblk[18];
  __shared__ int sc0;
  for (int ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
    const int2 cd = chunks[ch];
    load_box(B, boxes, cd.x);
    links_chunk<T, false>(B, cd.y, LINK_CHUNK, sblk, &sc0);
  }
}

// x = A^{-1} b for a symmetric 3x3 A given as (xx, xy, xz, yy, yz, zz) plus
// s on the diagonal (adjugate over determinant; A is positive definite).
__device__ void solve_sym3(const double* a, double s, const double* b, double* x) {
  const double m00 = a[0] + s, m01 = a[1], m02 = a[2], m11 = a[3] + s, m12 = a[4], m22 = a[5] + s;
  const double c00 = m11 * m22 - m12 * m12, c01 = m02 * m12 - m01 * m22, c02 = m01 * m12 - m02 * m11;
  const double c11 = m00 * m22 - m02 * m02, c12 = m01 * m02 - m00 * m12, c22 = m00 * m11 - m01 * m01;
  const double det = m00 * c00 + m01 * c01 + m02 * c02;
  x[0] = (c00 * b[0] + c01 * b[1] + c02 * b[2]) / det;
  x[1] = (c01 * b[0] + c11 * b[1] + c12 * b[2]) / det;
  x[2] = (c02 * b[0] + c12 * b[1] + c22 * b[2]) / det;
}

// ---------------------------------------------------------------------------
// k_colloid: colloid update ("molecular dynamics-like step", Sec. 2.2) and the
// end-of-step parity flip.  One block per box, one thread per colloid.  The
// velocity-dependent part of the link force is taken at the new velocity:
// V' = V + (M + zv)^{-1} (F_hyd + F_lc + F_ext), W' = W + (I + zw)^{-1} (T_hyd + T_lc + T_ext).
// ---------------------------------------------------------------------------
// Contact partner of colloid c at the current positions: -1 for a z wall,
// the lowest index of a colloid it touches, -2 for none.  The paper treats no
// contact (interactions between colloids are left to later work, Sec. 3.2);
// the reading taken: two colloids touch when their centres (minimum image)
// are closer than the sum of their radii, a colloid touches a wall when its
// surface passes the plane of the half-way bounce-back, z = -1/2 or nz - 1/2.
__device__ int contact_partner(const DevBox& B, int c) {
  const DevColloid& C = B.col[c];
  if (B.wall_z && (C.X[2] - C.a0 < -0.5 || C.X[2] + C.a0 > B.nz - 0.5)) return -1;
  for (int d = 0; d < B.ncol; ++d) {
    if (d == c) continue;
    double r[3];
    disp(B, C.X[0], C.X[1], C.X[2], B.col[d].X, r);
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(r[0], r[0]), __dmul_rn(r[1], r[1])), __dmul_rn(r[2], r[2]));
    const double s = __dadd_rn(C.a0, B.col[d].a0);
    if (r2 < __dmul_rn(s, s)) return d;
  }
  return -2;
}

// A mobile colloid whose new position touches a wall or another colloid is
// put back where it was before this step's move (its new velocities stand),
// so that no node is ever inside two colloids.  Every mobile colloid is tested
// at the same positions, then those in contact are put back; a colloid put
// back can be touched by another's move, so the test repeats until a pass
// puts none back.  The first contact since the host last read it (lowest
// colloid index of that pass) is kept in the box state and flagged in the
// group's error words; the host reports it as LC_ERR_OVERLAP.  All threads of
// the block call this (it holds block barriers).
__device__ void resolve_contacts(const DevBox& B, int tid, int nthr) {
  __shared__ signed char s_hit[MAXCOL];  // -2 no contact, else the partner
  __shared__ unsigned char s_back[MAXCOL];
  __shared__ int s_any;
  for (int c = tid; c < B.ncol; c += nthr) s_back[c] = 0;
  for (int pass = 0; pass <= B.ncol; ++pass) {
    __syncthreads();
    for (int c = tid; c < B.ncol; c += nthr)
      s_hit[c] = (signed char)((B.col[c].mobile && !s_back[c]) ? contact_partner(B, c) : -2);
    if (tid == 0) s_any = 0;
    __syncthreads();
    for (int c = tid; c < B.ncol; c += nthr) {
      if (s_hit[c] == -2) continue;
      DevColloid& C = B.col[c];
      for (int a = 0; a < 3; ++a) C.X[a] = C.Xb[a];
      s_back[c] = 1;
      s_any = 1;
    }
    if (tid == 0) {
      DevState* st = B.st;
      for (int c = 0; c < B.ncol; ++c) {
        if (s_hit[c] == -2) continue;
        if (st->cstep < 0) {
          st->cstep = st->step;
          st->ccol = c;
          st->cpartner = s_hit[c];
        }
        st->err |= 8;
        atomicOr(B.gerr + 1, 1);
        break;
      }
    }
    __syncthreads();
    if (!s_any) break;
  }
}

template <bool CG>
__device__ __forceinline__ void colloid_box(const DevBox& B, bool commit = true) {
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  const int nthr = blockDim.x * blockDim.y;
  if (!commit) {
    for (int c = tid; c < B.ncol; c += nthr)
      for (int k = 0; k < 24; ++k) B.col[c].acc[k] = 0.0;
    return;
  }
  for (int c = tid; c < B.ncol; c += nthr) {
    DevColloid& C = B.col[c];
    double acc[24];
    for (int k = 0; k < 24; ++k) acc[k] = CG ? __ldcg(&C.acc[k]) : C.acc[k];
    for (int a = 0; a < 3; ++a) {
      C.Fh[a] = acc[a];
      C.Th[a] = acc[3 + a];
      C.Flc[a] = acc[6 + a];
      C.Tlc[a] = acc[9 + a];
    }
    for (int a = 0; a < 3; ++a) {
      C.imp[a] += C.Fh[a] + C.Flc[a];
      C.aimp[a] += C.Th[a] + C.Tlc[a];
      C.Xb[a] = C.X[a];
      C.Vb[a] = C.V[a];
      C.Wb[a] = C.W[a];
    }
    if (C.mobile) {
      const double fv[3] = {C.Fh[0] + C.Flc[0] + C.Fext[0], C.Fh[1] + C.Flc[1] + C.Fext[1],
                            C.Fh[2] + C.Flc[2] + C.Fext[2]};
      const double tv[3] = {C.Th[0] + C.Tlc[0] + C.Text[0], C.Th[1] + C.Tlc[1] + C.Text[1],
                            C.Th[2] + C.Tlc[2] + C.Text[2]};
      double dv[3], dw[3];
      solve_sym3(acc + 12, C.M, fv, dv);
      solve_sym3(acc + 18, C.I, tv, dw);
      for (int a = 0; a < 3; ++a) {
        C.V[a] += dv[a];
        C.W[a] += dw[a];
      }
      const int L[3] = {B.nx, B.ny, B.nz};
      for (int a = 0; a < 3; ++a) {
        C.X[a] += C.V[a];
        if (a < 2 || !B.wall_z) {
          if (C.X[a] >= L[a]) C.X[a] -= L[a];
          if (C.X[a] < 0) C.X[a] += L[a];
        }
      }
    }
    for (int k = 0; k < 24; ++k) C.acc[k] = 0.0;
  }
  if (B.nmobile) {
    resolve_contacts(B, tid, nthr);
    // has a colloid moved as far as the node nearest to its surface?  (1e-9:
    // far above the rounding of the solid test, far below any margin that
    // saves a search)
    __shared__ int s_scan;
    if (tid == 0) s_scan = 0;
    __syncthreads();
    for (int c = tid; c < B.ncol; c += nthr) {
      const DevColloid& C = B.col[c];
      if (!C.mobile) continue;
      double r[3];
      disp(B, C.X[0], C.X[1], C.X[2], C.Xref, r);
      if (!(sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]) + 1e-9 < C.margin)) s_scan = 1;
    }
    __syncthreads();
    for (int c = tid; c < B.ncol; c += nthr)
      if (B.col[c].mobile) split_position(B.col[c]);
    if (s_scan)
      for (int c = tid; c < B.ncol; c += nthr) {
        DevColloid& C = B.col[c];
        for (int a = 0; a < 3; ++a) C.Xref[a] = C.X[a];
        C.margin = 1.0;
      }
    if (tid == 0) B.st->scan = s_scan;
  }
  if (tid == 0) {
    DevState* st = B.st;
    if (B.p.flow_on) {
      st->fpar ^= 1;
      st->pre_valid = 0;
    }
    if (B.p.lc_on) st->qpar ^= 1;
    st->step += 1;
    st->nchg = 0;
  }
}

// Stores Q + d5 of a pair (compensated: hi + lo + increment carried exactly into
// (hi, lo) by two-sum) and adds its residual.
__device__ __forceinline__ void store_pair(float* q, __nv_bfloat16* l, size_t N, const f2 qi[5], const f2 lo[5],
                                           const f2 d5[5], float& rsum, float& rmax) {
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const f2 sv = lo[k] + d5[k];
    const f2 hn = qi[k] + sv;
    const f2 bb = hn - qi[k];
    const f2 err = (qi[k] - (hn - bb)) + (sv - bb);
    st2(q + k * N, hn);
    *reinterpret_cast<__nv_bfloat162*>(l + k * N) = __float22bfloat162_rn(err.v);
  }
  const f2 dzz = -(d5[0] + d5[3]);
  const f2 r2 = d5[0] * d5[0] + d5[3] * d5[3] + dzz * dzz + 2.f * (d5[1] * d5[1] + d5[2] * d5[2] + d5[4] * d5[4]);
  float mx = fmaxf(fabsf(dzz.v.x), fabsf(dzz.v.y));
#pragma unroll
  for (int k = 0; k < 5; ++k) mx = fmaxf(mx, fmaxf(fabsf(d5[k].v.x), fabsf(d5[k].v.y)));
  rsum += r2.v.x + r2.v.y;
  rmax = fmaxf(rmax, mx);
}

// ---------------------------------------------------------------------------
// k_lc: Q update, link exchange and colloid update in one launch
// ---------------------------------------------------------------------------
// Q update of a tile of plain nodes, two nodes per lane: Q and u from the
// ring, H and the remainder of Q from global memory, issued before the ring
// reads of the plane.
template <int TY>
__device__ __forceinline__ void lc_ring(const DevBox& B, const LcPair& K2, const int4 td, int zc, float* ring,
                                        float& rsum, float& rmax) {
  if (!B.p.lc_on) return;
  const int qpar = B.st->qpar;
  const float* __restrict__ Q = static_cast<const float*>(B.Q[qpar]);
  float* __restrict__ Qo = static_cast<float*>(B.Q[qpar ^ 1]);
  const __nv_bfloat16* __restrict__ Lin = B.Qlo[qpar];
  __nv_bfloat16* __restrict__ Lout = B.Qlo[qpar ^ 1];
  const float* __restrict__ U = static_cast<const float*>(B.u);
  const float* __restrict__ Hb = static_cast<const float*>(B.H);
  const RingLane R = ring_lane<8, TY, 5>(B, td, Q, U);
  const int nz = B.nz, zend = min(td.w + zc, nz), plane = B.nx * B.ny;
  const size_t N = (size_t)B.N;
  const uint8_t* mp = B.mask + R.x + R.row;
  __syncthreads();
#pragma unroll 1
  for (int k = -1; k <= 1; ++k) ring_load<8, TY, 5>(ring, B, R, td, Q, U, td.w + k, (k + 1) & 3);
  cp_async_commit();
  unsigned m2 = R.valid ? (unsigned)*reinterpret_cast<const uint16_t*>(mp + (size_t)plane * td.w) : 0x0101u;
  for (int z = td.w; z < zend; ++z) {
    const int s0 = (z - td.w + 1) & 3, sm = (s0 + 3) & 3, sp = (s0 + 1) & 3;
    const size_t i = (size_t)R.x + R.row + (size_t)plane * z;
    const bool plain = plain_pair(m2);
    float2 hr[5];
    __nv_bfloat162 lr[5];
    if (plain) {
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        hr[k] = __ldg(reinterpret_cast<const float2*>(Hb + k * N + i));
        lr[k] = *reinterpret_cast<const __nv_bfloat162*>(Lin + k * N + i);
      }
    }
    cp_async_wait0();
    __syncthreads();
    if (z + 1 < zend) {
      ring_load<8, TY, 5>(ring, B, R, td, Q, U, z + 2, (s0 + 2) & 3);
      if (R.valid) m2 = (unsigned)*reinterpret_cast<const uint16_t*>(mp + (size_t)plane * (z + 1));
    }
    cp_async_commit();
    if (!plain) continue;
    // the fluxes first, one component's neighbours at a time, then the velocity
    // gradient, for which the velocities are read again: all of them at once
    // would push the kernel past its registers
    f2 qi[5], adv[5], w[3][3], d5[5];
    {
      f2 up[6], dn[6];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        f2 ui, n[6];
        ring_gather<8, TY>(ring, R, 5 + a, s0, sm, sp, ui, n);
        upwind_pair(ui, n[2 * a], n[2 * a + 1], up + 2 * a, dn + 2 * a);
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        f2 n[6];
        asm volatile("" ::: "memory");
        ring_gather<8, TY>(ring, R, k, s0, sm, sp, qi[k], n);
        adv[k] = advect_pair(up, dn, qi[k], n);
      }
    }
    asm volatile("" ::: "memory");
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      f2 ui, n[6];
      ring_gather<8, TY>(ring, R, 5 + a, s0, sm, sp, ui, n);
#pragma unroll
      for (int j = 0; j < 3; ++j) w[a][j] = n[2 * j] - n[2 * j + 1];
    }
    f2 h[5], lo[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      h[k] = f2(hr[k]);
      lo[k] = f2(__bfloat1622float2(lr[k]));
    }
    q_pair(K2, qi, adv, w, h, lo, d5);
    store_pair(Qo + i, Lout + i, N, qi, lo, d5, rsum, rmax);
  }
}

// Q update of a tile of plain nodes, one node per lane.
template <typename T>
__device__ __forceinline__ void lc_plain(const DevBox& B, const int4 td, int zc, T& rsum, T& rmax) {
  if (!B.p.lc_on) return;
  const int lane = threadIdx.x, qpar = B.st->qpar;
  const T* __restrict__ Q = static_cast<const T*>(B.Q[qpar]);
  const __nv_bfloat16* __restrict__ Lin = B.Qlo[qpar];
  const T* __restrict__ U = static_cast<const T*>(B.u);
  const int nx = B.nx, ny = B.ny, x = td.y + lane, y = td.z + (int)threadIdx.y;
  const int zend = min(td.w + zc, B.nz);
  const bool valid = x < nx && y < ny;
  for (int z = td.w; z < zend; ++z) {
    const int row = nx * (y + ny * z), i = x + row;
    const uint8_t m = valid ? B.mask[i] : (uint8_t)1;
    const bool plain = plain_node(m);
    T pq[3][5], pu[3][3];
    float plo[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) pq[0][k] = valid ? ldg(Q + (size_t)k * B.N + i) : T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) pu[0][a] = valid ? ldg(U + (size_t)a * B.N + i) : T(0);
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int k = 0; k < 5; ++k) plo[k] = plain ? __bfloat162float(Lin[(size_t)k * B.N + i]) : 0.f;
    }
    x_neighbours<T, 5>(Q, (size_t)B.N, pq[0], lane, x, nx, row, valid, &pq[1]);
    x_neighbours<T, 3>(U, (size_t)B.N, pu[0], lane, x, nx, row, valid, &pu[1]);
    if (plain)
      lc_update_node<T, false>(B, phys<T>(B), Q, Lin, U, qpar, x, y, z, i, rsum, rmax, pq, pu, plo);
  }
}

// Near node of k_lc.
template <typename T>
__device__ __forceinline__ void near_lc(const DevBox& B, int j, T& rsum, T& rmax) {
  if (j < 0) return;
  const int qpar = B.st->qpar;
  T rs = T(0), rm = T(0);
  lc_update_node<T, true>(B, phys<T>(B), static_cast<const T*>(B.Q[qpar]), B.Qlo[qpar], static_cast<const T*>(B.u),
                          qpar, j % B.nx, (j / B.nx) % B.ny, j / (B.nx * B.ny), j, rs, rm);
  rsum += rs;
  rmax = fmax(rmax, rm);
}

// The work units of a box are counted as they finish; the block that finishes
// the last one of a box (near groups, link chunks and tiles) runs its colloid
// update and parity flip, so a step takes no separate launches for the link
// exchange and the colloid update (16 and 6 us beside or after a 62 us update
// at 128^3, and most of the step of a small box).  The counter is zero again
// when the launch ends.  All threads of the block call this.
__device__ __forceinline__ void lc_commit(const Launch& L, int b, unsigned n) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x + threadIdx.y == 0) s_last = atomicAdd(L.done + b, n) + n == L.total[b];
  __syncthreads();
  if (s_last) {
    __threadfence();
    colloid_box<true>(L.boxes[b]);
    if (threadIdx.x + threadIdx.y == 0) L.done[b] = 0;
  }
  __syncthreads();
}

// Q update of all nodes, link exchange and colloid update.  FP32 tiles of even
// width: as k_stress, Q and u from the ring (8 components), H and the remainder
// of Q loaded per pair ahead of the plane's barrier; 128 registers, one
// component's neighbours read at a time (all at once spill).  Bound by issue:
// 128^3 67 + 16 us (links) + 6 (colloid) as three launches, 60 us for all of it now
// (55 with shorter sums in another order, see lclb_pair.cuh); 256 x 192 x 160 186 us.
template <typename T, int TY>
__global__ void __launch_bounds__(TX * TY, (sizeof(T) == 4 ? 512 : 256) / (TX * TY)) k_lc(Launch L, int mode,
                                                                                         double* __restrict__ part) {
  __shared__ DevBox B;
  __shared__ LcPair K2;
  __shared__ double sblk[18];
  __shared__ int sc0;
  extern __shared__ __align__(16) float ring[];
  const bool commit = (mode & LC_COMMIT) != 0;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int nn = L.ngroups / TY, nl = commit ? L.nchunks : 0, units = nn + nl + L.ntiles;
  int cur_box = -1, run_box = -1;
  unsigned run_n = 0;
  for (int t = blockIdx.x; t < units; t += gridDim.x) {
    const int4 td = t < nn ? make_int4(L.groups[t * TY].x, 0, 0, 0)
                           : (t < nn + nl ? make_int4(L.chunks[t - nn].x, L.chunks[t - nn].y, 0, 0) : L.tiles[t - nn - nl]);
    if (commit && td.x != run_box) {
      if (run_n) lc_commit(L, run_box, run_n);
      run_box = td.x;
      run_n = 0;
    }
    ++run_n;
    load_box<T>(B, K2, L.boxes, td.x, cur_box);
    T rsum = T(0), rmax = T(0);  // per-thread residual (sum of squares, max), in T
    if (t < nn) {
      if (B.p.lc_on)
        near_group<TY>(B, L.groups, t, [&](int j) { near_lc<T>(B, j, rsum, rmax); });
      __syncwarp();
      if (mode & LC_RESID) warp_residual<T>(L.npart + 2 * (size_t)t * TY, wy, lane, rsum, rmax);
      continue;
    }
    if (t < nn + nl) {
      links_chunk<T, false>(B, td.y, TX * TY, sblk, &sc0);
      continue;
    }
    bool done = false;
    if constexpr (sizeof(T) == 4) {
      if (pair_box(B)) {
        lc_ring<TY>(B, K2, td, L.zc, ring, rsum, rmax);
        done = true;
      }
    }
    if (!done) lc_plain<T>(B, td, L.zc, rsum, rmax);
    __syncwarp();
    if (mode & LC_RESID) warp_residual<T>(part + 2 * (size_t)(t - nn - nl) * TY, wy, lane, rsum, rmax);
  }
  if (commit && run_n) lc_commit(L, run_box, run_n);
}

// ---------------------------------------------------------------------------
// k_relax: the whole step of boxes whose flow is frozen
// ---------------------------------------------------------------------------
// With u = 0 the step is dQ = Gamma H (Eq. 2): no stress, no populations, no
// flux, so H is used where it is formed and each node moves its Q twice (60
// bytes with the remainder) instead of the 190 of the separate stress and Q
// update.  Near nodes still take their stress for the colloid's LC force.
// Bound by issue of the molecular field (about 140 packed operations a pair);
// 96^3: 105 us for the launches of the general step, 69 without its stores and
// loads, 30 as one launch, 22 with the ring copied in 16-byte pieces.
template <int TY, bool CHIRAL>
__device__ __forceinline__ void relax_ring(const DevBox& B, const LcPair& K2, const int4 td, int zc, float* ring,
                                           float& rsum, float& rmax) {
  const int qpar = B.st->qpar;
  const float* __restrict__ Q = static_cast<const float*>(B.Q[qpar]);
  float* __restrict__ Qo = static_cast<float*>(B.Q[qpar ^ 1]);
  const __nv_bfloat16* __restrict__ Lin = B.Qlo[qpar];
  __nv_bfloat16* __restrict__ Lout = B.Qlo[qpar ^ 1];
  const RingLane R = ring_lane<5, TY, 5>(B, td, Q, Q);
  const int zend = min(td.w + zc, B.nz), plane = B.nx * B.ny;
  const size_t N = (size_t)B.N;
  const uint8_t* mp = B.mask + R.x + R.row;
  __syncthreads();
#pragma unroll 1
  for (int k = -1; k <= 1; ++k) ring_load<5, TY, 5>(ring, B, R, td, Q, Q, td.w + k, (k + 1) & 3);
  cp_async_commit();
  unsigned m2 = R.valid ? (unsigned)*reinterpret_cast<const uint16_t*>(mp + (size_t)plane * td.w) : 0x0101u;
  for (int z = td.w; z < zend; ++z) {
    const int s0 = (z - td.w + 1) & 3;
    const size_t i = (size_t)R.x + R.row + (size_t)plane * z;
    const bool plain = plain_pair(m2);
    __nv_bfloat162 lr[5];
    if (plain) {
#pragma unroll
      for (int k = 0; k < 5; ++k) lr[k] = *reinterpret_cast<const __nv_bfloat162*>(Lin + k * N + i);
    }
    cp_async_wait0();
    __syncthreads();
    if (z + 1 < zend) {
      ring_load<5, TY, 5>(ring, B, R, td, Q, Q, z + 2, (s0 + 2) & 3);
      if (R.valid) m2 = (unsigned)*reinterpret_cast<const uint16_t*>(mp + (size_t)plane * (z + 1));
    }
    cp_async_commit();
    if (!plain) continue;
    f2 qi[5], dq[3][5], lap[5], h[5], p[9], fp, lo[5], d5[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      f2 n[6];
      ring_gather<5, TY>(ring, R, k, s0, (s0 + 3) & 3, (s0 + 1) & 3, qi[k], n);
      dq[0][k] = n[0] - n[1];
      dq[1][k] = n[2] - n[3];
      dq[2][k] = n[4] - n[5];
      lap[k] = ((n[0] + n[1]) + (n[2] + n[3]) + (n[4] + n[5])) + K2.nsix * qi[k];
      lo[k] = f2(__bfloat1622float2(lr[k]));
    }
    lc_pair<CHIRAL, false>(K2, qi, dq, lap, h, p, &fp);
    q_pair_frozen(K2, qi, h, lo, d5);
    store_pair(Qo + i, Lout + i, N, qi, lo, d5, rsum, rmax);
  }
}

template <typename T>
__device__ __forceinline__ void relax_plain(const DevBox& B, const int4 td, int zc, T& rsum, T& rmax) {
  const int lane = threadIdx.x, qpar = B.st->qpar;
  const T* __restrict__ Q = static_cast<const T*>(B.Q[qpar]);
  const size_t N = (size_t)B.N;
  const int nx = B.nx, ny = B.ny, x = td.y + lane, y = td.z + (int)threadIdx.y;
  const int zend = min(td.w + zc, B.nz);
  const bool valid = x < nx && y < ny;
  T qz[2][5];
  column_start<T, 5>(B, Q, x, y, td.w, valid, qz);
  for (int z = td.w; z < zend; ++z) {
    const int row = nx * (y + ny * z), i = x + row;
    const bool plain = valid && plain_node(B.mask[i]);
    T pq[5][5];
    column_next<T, 5>(B, Q, x, y, z, valid, qz, pq);
    x_neighbours<T, 5>(Q, N, pq[0], lane, x, nx, row, valid, &pq[1]);
    if (plain) {
      float lo[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
      T qn[6][5], h[5], p[9], fp, d5[5];
      const int yp = nx * ((y + 1 == ny ? 0 : y + 1) + ny * z) + x, ym = nx * ((y == 0 ? ny - 1 : y - 1) + ny * z) + x;
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        if constexpr (sizeof(T) == 4) lo[k] = __bfloat162float(B.Qlo[qpar][k * N + i]);
        qn[0][k] = pq[1][k];
        qn[1][k] = pq[2][k];
        qn[2][k] = ldg(Q + k * N + yp);
        qn[3][k] = ldg(Q + k * N + ym);
        qn[4][k] = pq[3][k];
        qn[5][k] = pq[4][k];
      }
      lc_node<T, false>(B, pq[0], qn, h, p, &fp);
      if constexpr (sizeof(T) == 4) q_increment_f32<false>(B.pf, pq[0], nullptr, nullptr, nullptr, nullptr, h, lo, d5);
      else q_increment<false, T>(B.kd, pq[0], nullptr, nullptr, h, d5);
#pragma unroll
      for (int k = 0; k < 5; ++k) store_q_next<T>(B, qpar, i, k, pq[0][k], lo[k], d5[k]);
      add_residual(d5, rsum, rmax);
    }
    column_roll<T, 5>(qz, pq);
  }
}

template <typename T, int TY>
__global__ void __launch_bounds__(TX * TY, (sizeof(T) == 4 ? 640 : 256) / (TX * TY)) k_relax(Launch L, int mode,
                                                                                            double* __restrict__ part) {
  __shared__ DevBox B;
  __shared__ LcPair K2;
  extern __shared__ __align__(16) float ring[];
  const bool commit = (mode & LC_COMMIT) != 0;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int nn = L.ngroups / TY, units = nn + L.ntiles;
  int cur_box = -1, run_box = -1;
  unsigned run_n = 0;
  for (int t = blockIdx.x; t < units; t += gridDim.x) {
    const int4 td = t < nn ? make_int4(L.groups[t * TY].x, 0, 0, 0) : L.tiles[t - nn];
    if (commit && td.x != run_box) {
      if (run_n) lc_commit(L, run_box, run_n);
      run_box = td.x;
      run_n = 0;
    }
    ++run_n;
    load_box<T>(B, K2, L.boxes, td.x, cur_box);
    T rs[2] = {T(0), T(0)};
    if (B.p.lc_on) {
      if (t < nn) {
        near_group<TY>(B, L.groups, t, [&](int j) {
          near_stress<T, true>(B, j, (mode & LC_FLC) ? FORCE_ACC : 0, reinterpret_cast<NearScratch<T>*>(ring)[wy], rs);
        });
        __syncthreads();
      } else {
        bool done = false;
        if constexpr (sizeof(T) == 4) {
          if (pair_box(B)) {
            if (B.p.q0 != 0.0) relax_ring<TY, true>(B, K2, td, L.zc, ring, rs[0], rs[1]);
            else relax_ring<TY, false>(B, K2, td, L.zc, ring, rs[0], rs[1]);
            done = true;
          }
        }
        if (!done) relax_plain<T>(B, td, L.zc, rs[0], rs[1]);
      }
    }
    __syncwarp();
    if (mode & LC_RESID)
      warp_residual<T>(t < nn ? L.npart + 2 * (size_t)t * TY : part + 2 * (size_t)(t - nn) * TY, wy, lane, rs[0], rs[1]);
  }
  if (commit && run_n) lc_commit(L, run_box, run_n);
}

__global__ void k_colloid(const DevBox* __restrict__ boxes, int nboxes) {
  const int b = blockIdx.x;
  if (b >= nboxes) return;
  colloid_box<false>(boxes[b]);
}

// ---------------------------------------------------------------------------
// k_step: one coupled step of every box as one persistent launch
// ---------------------------------------------------------------------------
// The blocks take work items in list order from an atomic counter.  The list
// is ordered so that every item comes after the items it waits for (stress of
// z chunks c - 1, c, c + 1 before the LB of chunk c; LB of c - 1, c, c + 1
// before the Q update of c; all LB tiles before the link exchange; all tiles
// and links before the colloid update), so the earliest unfinished item
// never waits on an item no block has taken, and the launch cannot deadlock
// whether or not all blocks are resident.  The phases of different chunks run
// side by side, so the HBM-bound LB overlaps the arithmetic-bound stress and
// Q update, and the stress, velocity and molecular field of a chunk are read
// back while they are still in L2.  Waits are bounded: after spin_limit
// polls the item is skipped (its outputs are then stale), *err is set and the
// host reports a timeout.

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

template <typename T, int TY>
__global__ void __launch_bounds__(TX * TY, (sizeof(T) == 4 ? 512 : 256) / (TX * TY)) k_step(
    DevBox* __restrict__ boxes, const StepItem* __restrict__ items, int nitems, int zc, unsigned* __restrict__ sync,
    double* __restrict__ part, int spin_limit, int commit, int* __restrict__ err) {
  __shared__ DevBox B;
  __shared__ LcPair K2;
  __shared__ double sblk[18];
  __shared__ int sq[TY][2 * TX];
  __shared__ int s_item, s_ok, s_sc0;
  extern __shared__ __align__(16) float step_smem[];
  NearScratch<T>& sc = reinterpret_cast<NearScratch<T>*>(step_smem)[threadIdx.y];
  const int tid = threadIdx.x + TX * threadIdx.y;
  int cur_box = -1;
  for (;;) {
    if (tid == 0) s_item = (int)atomicAdd(&sync[0], 1u);
    __syncthreads();
    const int it = s_item;
    if (it >= nitems) break;
    const StepItem I = items[it];
    if (tid == 0) {
      int ok = 1;
      for (int k = 0; k < 4 && ok; ++k) {
        if (I.wc[k] < 0) continue;
        const unsigned target = (unsigned)I.wt[k];
        for (int spin = 0; ld_acquire_u32(&sync[I.wc[k]]) < target; ++spin) {
          // give up after spin_limit polls, or at once when another wait of
          // this launch already gave up
          if (spin >= spin_limit || ((spin & 255) == 255 && ld_acquire_u32(reinterpret_cast<unsigned*>(err)) != 0)) {
            ok = 0;
            break;
          }
          __nanosleep(100);
        }
      }
      if (!ok) atomicOr(err, 1);
      s_ok = ok;
    }
    __syncthreads();
    if (s_ok) {
      load_box<T>(B, K2, boxes, I.box, cur_box);
      const int4 td = make_int4(I.box, I.x0, I.y0, I.z0);
      switch (I.kind) {
        case ITEM_STRESS:
          if constexpr (sizeof(T) == 4) {
            if (pair_box(B)) {
              stress_tile_pair<TY>(B, K2, td, zc, FORCE_ACC, sq, sc);
              break;
            }
          }
          stress_tile<T, TY>(B, td, zc, FORCE_ACC, sq, sc);
          break;
        case ITEM_LB: lbp_tile<T, TY, true>(B, td, zc, sq); break;
        case ITEM_LC:
          if constexpr (sizeof(T) == 4) {
            if (pair_box(B)) {
              lc_tile_pair<TY, true>(B, K2, td, zc, part + 2 * (size_t)I.part * TY, sq);
              break;
            }
          }
          lc_tile<T, TY, true>(B, td, zc, part + 2 * (size_t)I.part * TY, sq);
          break;
        case ITEM_LINKS: links_chunk<T, true>(B, I.x0, LINK_CHUNK, sblk, &s_sc0); break;
        default: colloid_box<true>(B, commit != 0); break;
      }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      if (I.dc[0] >= 0) atomicAdd(&sync[I.dc[0]], 1u);
      if (I.dc[1] >= 0) atomicAdd(&sync[I.dc[1]], 1u);
    }
  }
}

// ---------------------------------------------------------------------------
// geometry: solid mask, near flags, boundary links (cold path)
// ---------------------------------------------------------------------------
__global__ void k_pair_constants(DevBox* __restrict__ boxes, int b) { lc_pair_constants(boxes[b].kp, boxes[b].pf); }

__global__ void k_mask(DevBox* __restrict__ boxes, int b) {
  const DevBox& B = boxes[b];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B.N) return;
  const int x = i % B.nx, y = (i / B.nx) % B.ny, z = i / (B.nx * B.ny);
  uint8_t id = 0;
  for (int c = 0; c < B.ncol; ++c)
    if (inside_colloid(B, x, y, z, B.col[c])) {
      if (id == 0) id = (uint8_t)(c + 1);
      else atomicOr(&B.st->err, 4);  // overlap
    }
  B.mask[i] = id;
}

__global__ void k_near(DevBox* __restrict__ boxes, int b) {
  const DevBox& B = boxes[b];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B.N) return;
  uint8_t m = B.mask[i];
  if (m & IDMASK) return;
  const int x = i % B.nx, y = (i / B.nx) % B.ny, z = i / (B.nx * B.ny);
  bool near = false;
#pragma unroll
  for (int q = 1; q < NQ; ++q) {
    const int zz = z + cz(q);
    if (B.wall_z && (zz < 0 || zz >= B.nz)) {
      near = true;
      continue;
    }
    const int j = wrap1(x + cx(q), B.nx) + B.nx * (wrap1(y + cy(q), B.ny) + B.ny * wrap1(zz, B.nz));
    if (B.mask[j] & IDMASK) near = true;
  }
  B.mask[i] = near ? (uint8_t)(m | NEAR) : (uint8_t)(m & ~NEAR);
}

// Whether fluid node i is on the box's near list: next to a solid or wall, or,
// in boxes whose tiles evaluate two nodes at once, the other node of such a
// node's pair (the tiles leave the pair out whole).  The list is evaluated from
// the compensated Q; with that other node's stress from the FP32 part of Q alone,
// a mobile colloid's force, a small sum over these nodes, was 1e-5 to 4e-5 off
// what it is with it.
__device__ __forceinline__ bool near_member(const DevBox& B, int i) {
  if (i >= B.N) return false;
  const uint8_t m = B.mask[i];
  if (m & IDMASK) return false;
  return (m & NEAR) || (pair_box(B) && (B.mask[i ^ 1] & NEAR));
}

// The list is in node order, so that a box's residual, which is summed over it in
// FP32, is the same for every handle with the same state: nodes counted per
// block, the counts scanned, and each block's nodes written behind those of the
// blocks before it.
// Rank of a listed node among those of the block's 256 nodes (all threads call
// it; s: 8 ints of shared memory).
__device__ __forceinline__ int near_rank(bool near, int* s) {
  const unsigned m = __ballot_sync(0xffffffffu, near);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) s[wid] = __popc(m);
  __syncthreads();
  int r = __popc(m & ((1u << lane) - 1u));
  for (int k = 0; k < wid; ++k) r += s[k];
  return r;
}

__global__ void __launch_bounds__(256) k_near_count(const DevBox* __restrict__ boxes, int b, int* blocksum) {
  const int n = __syncthreads_count(near_member(boxes[b], blockIdx.x * blockDim.x + threadIdx.x));
  if (threadIdx.x == 0) blocksum[blockIdx.x] = n;
}

__global__ void __launch_bounds__(256) k_near_write(const DevBox* __restrict__ boxes, int b, const int* blockoff) {
  __shared__ int s[8];
  const DevBox& B = boxes[b];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool near = near_member(B, i);
  const int at = blockoff[blockIdx.x] + near_rank(near, s);
  if (near && at < B.near_cap) B.near_node[at] = i;
}

// Number of links from fluid node i into colloid c (bit q set in *bits).
__device__ __forceinline__ int links_at(const DevBox& B, int i, int c, unsigned* bits) {
  unsigned bm = 0;
  if ((B.mask[i] & IDMASK) == 0 && (B.mask[i] & NEAR)) {
    const int x = i % B.nx, y = (i / B.nx) % B.ny, z = i / (B.nx * B.ny);
#pragma unroll
    for (int q = 1; q < NQ; ++q) {
      const int zz = z + cz(q);
      if (B.wall_z && (zz < 0 || zz >= B.nz)) continue;
      const int j = wrap1(x + cx(q), B.nx) + B.nx * (wrap1(y + cy(q), B.ny) + B.ny * wrap1(zz, B.nz));
      if ((B.mask[j] & IDMASK) == (uint8_t)(c + 1)) bm |= 1u << q;
    }
  }
  *bits = bm;
  return __popc(bm);
}

__global__ void __launch_bounds__(256) k_link_count(const DevBox* __restrict__ boxes, int b, int c, int* blocksum) {
  const DevBox& B = boxes[b];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned bits;
  int n = i < B.N ? links_at(B, i, c, &bits) : 0;
  __shared__ int s[8];
  int v = n;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int k = 0; k < 8; ++k) t += s[k];
    blocksum[blockIdx.x] = t;
  }
}

// Exclusive scan of n ints in one block (deterministic); total -> *total.
__global__ void __launch_bounds__(1024) k_scan(int* a, int n, int base, int* total) {
  __shared__ int s[1024];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = base;
  __syncthreads();
  for (int off = 0; off < n; off += 1024) {
    const int i = off + threadIdx.x;
    const int v = i < n ? a[i] : 0;
    s[threadIdx.x] = v;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {
      int t = threadIdx.x >= d ? s[threadIdx.x - d] : 0;
      __syncthreads();
      s[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < n) a[i] = carry + s[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry += s[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(256) k_link_write(const DevBox* __restrict__ boxes, int b, int c,
                                                    const int* blockoff) {
  const DevBox& B = boxes[b];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned bits = 0;
  const int n = i < B.N ? links_at(B, i, c, &bits) : 0;
  __shared__ int s[256];
  s[threadIdx.x] = n;
  __syncthreads();
  for (int d = 1; d < 256; d <<= 1) {
    int t = threadIdx.x >= d ? s[threadIdx.x - d] : 0;
    __syncthreads();
    s[threadIdx.x] += t;
    __syncthreads();
  }
  int pos = blockoff[blockIdx.x] + s[threadIdx.x] - n;
  for (int q = 1; q < NQ; ++q)
    if (bits & (1u << q)) {
      if (pos < B.nlinks_cap) {
        B.link_node[pos] = i;
        B.link_dir[pos] = (int8_t)q;
        B.link_col[pos] = (int8_t)c;
      } else {
        atomicOr(&B.st->err, 1);
      }
      ++pos;
    }
}

// ---------------------------------------------------------------------------
// init, export, diagnostics (cold path)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t splitmix64(uint64_t s) {
  uint64_t z = s + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

// Stores FP64 value v as component k of node i in both Q buffers (FP32:
// compensated, hi and its BF16 remainder).
template <typename T>
__device__ __forceinline__ void store_q(const DevBox& B, int i, int k, double v) {
  const size_t o = (size_t)k * B.N + i;
  if constexpr (sizeof(T) == 4) {
    float hi;
    __nv_bfloat16 lo;
    split_q(v, hi, lo);
    static_cast<float*>(B.Q[0])[o] = hi;
    static_cast<float*>(B.Q[1])[o] = hi;
    B.Qlo[0][o] = lo;
    B.Qlo[1][o] = lo;
  } else {
    static_cast<double*>(B.Q[0])[o] = v;
    static_cast<double*>(B.Q[1])[o] = v;
  }
}

// Stores FP64 value v as component k of node i of the current Q buffer only.
template <typename T>
__device__ __forceinline__ void store_q_cur(const DevBox& B, int i, int k, double v) {
  const int qpar = B.st->qpar;
  const size_t o = (size_t)k * B.N + i;
  if constexpr (sizeof(T) == 4) {
    float hi;
    __nv_bfloat16 lo;
    split_q(v, hi, lo);
    static_cast<float*>(B.Q[qpar])[o] = hi;
    B.Qlo[qpar][o] = lo;
  } else {
    static_cast<double*>(B.Q[qpar])[o] = v;
  }
}

// kind 0: uniaxial along (n0,n1,n2); kind 1: helix along axis (int)n0.
template <typename T>
__global__ void k_init_q(DevBox* __restrict__ boxes, int b, int kind, double n0, double n1, double n2, double amp,
                         unsigned long long seed) {
  const DevBox& B = boxes[b];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B.N) return;
  const int x = i % B.nx, y = (i / B.nx) % B.ny, z = i / (B.nx * B.ny);
  double d[3];
  if (kind == 0) {
    const double nn = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(n0, n0), __dmul_rn(n1, n1)), __dmul_rn(n2, n2)));
    d[0] = n0 / nn; d[1] = n1 / nn; d[2] = n2 / nn;
  } else {
    const int ax = (int)n0, bb = (ax + 1) % 3, cc = (ax + 2) % 3;
    const int r[3] = {x, y, z};
    const double ph = B.p.q0 * r[ax];
    d[0] = d[1] = d[2] = 0.0;
    d[bb] = cos(ph);
    d[cc] = sin(ph);
  }
  // S0 (d_a d_b - delta_ab/3) with round-to-nearest operations only (no
  // contraction), so FP64 storage agrees bit for bit with a plain C evaluation.
  const double S0 = B.p.S0, third = 1.0 / 3.0;
  const double v[5] = {__dmul_rn(S0, __dsub_rn(__dmul_rn(d[0], d[0]), third)), __dmul_rn(S0, __dmul_rn(d[0], d[1])),
                       __dmul_rn(S0, __dmul_rn(d[0], d[2])), __dmul_rn(S0, __dsub_rn(__dmul_rn(d[1], d[1]), third)),
                       __dmul_rn(S0, __dmul_rn(d[1], d[2]))};
  for (int k = 0; k < 5; ++k) {
    const uint64_t r = splitmix64((uint64_t)seed ^ (uint64_t)(5LL * i + k));
    const double u = (double)(r >> 11) * (1.0 / 9007199254740992.0);
    const double val = __dadd_rn(v[k], __dmul_rn(amp, __dsub_rn(2.0 * u, 1.0)));
    store_q<T>(B, i, k, val);
  }
}

// Convert FP64 input to storage: which 0 = Q (both buffers), 1 = f (pre-collision,
// full f -> deviation into f[fpar], pre_valid set by the host).
template <typename T>
__global__ void k_set_field(DevBox* __restrict__ boxes, int b, int which, const double* __restrict__ src) {
  const DevBox& B = boxes[b];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B.N) return;
  if (which == 0) {
    for (int k = 0; k < 5; ++k) store_q<T>(B, i, k, src[(size_t)k * B.N + i]);
  } else {
    T* f = static_cast<T*>(B.f[B.st->fpar]);
    for (int q = 0; q < NQ; ++q) f[(size_t)q * B.N + i] = T(src[(size_t)q * B.N + i] - wq(q) * B.p.rho0);
  }
}

// Exports.  Q: the 5 N stored values in order, VEC per thread (hi + lo, or the
// FP64 values).
template <typename T, int VEC>
__global__ void __launch_bounds__(256) k_export_q(const DevBox* __restrict__ boxes, int b, double* __restrict__ out) {
  const DevBox& B = boxes[b];
  const int qpar = B.st->qpar;
  const size_t n = 5 * (size_t)B.N, e0 = (blockIdx.x * (size_t)256 + threadIdx.x) * VEC;
  const T* __restrict__ Q = static_cast<const T*>(B.Q[qpar]);
  const __nv_bfloat16* __restrict__ lo = B.Qlo[qpar];
  if constexpr (sizeof(T) == 4 && VEC == 4) {
    if (e0 + 4 <= n) {
      const float4 h = *reinterpret_cast<const float4*>(Q + e0);
      const __nv_bfloat162 l0 = *reinterpret_cast<const __nv_bfloat162*>(lo + e0);
      const __nv_bfloat162 l1 = *reinterpret_cast<const __nv_bfloat162*>(lo + e0 + 2);
      double2* o = reinterpret_cast<double2*>(out + e0);
      o[0] = make_double2(f32_to_f64(h.x) + f32_to_f64(__low2float(l0)), f32_to_f64(h.y) + f32_to_f64(__high2float(l0)));
      o[1] = make_double2(f32_to_f64(h.z) + f32_to_f64(__low2float(l1)), f32_to_f64(h.w) + f32_to_f64(__high2float(l1)));
      return;
    }
  }
  for (size_t e = e0; e < e0 + VEC && e < n; ++e) {
    if constexpr (sizeof(T) == 4) out[e] = (double)Q[e] + (double)__bfloat162float(lo[e]);
    else out[e] = Q[e];
  }
}

// Other fields.  which: LC_F_PRE, LC_RHO, LC_U, LC_FORCE, LC_SOLID.  The force
// is the face divergence of the stored stress, as the LB kernel takes it.
// Velocity from FP32 storage: 37 loads a node, so 64 registers for 32 warps per
// SM (98 registers: 16 warps), and 8 FP64 operations a node with the half force
// added among the integers (23 with conversions before): 256 x 192 x 160 694 ->
// 364 us (a quarter more than the LB kernel, which loads the same), 128^3 189 ->
// 98.
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_export(const DevBox* __restrict__ boxes, int b, int which,
                                                double* __restrict__ out) {
  const DevBox& B = boxes[b];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B.N) return;
  const int N = B.N;
  const uint8_t m = B.mask[i];
  const int x = i % B.nx, y = (i / B.nx) % B.ny, z = i / (B.nx * B.ny);
  if (which == EXP_SOLID) {
    out[i] = (m & IDMASK) ? (double)((m & IDMASK) - 1) : -1.0;
    return;
  }
  T F[3] = {T(0), T(0), T(0)};
  if ((which == EXP_FORCE || which == EXP_U) && !(m & IDMASK) && B.p.lc_on)
    stored_force<T>(B, static_cast<const T*>(B.P), x, y, z, i, m, F);
  if (which == EXP_FORCE) {
    for (int a = 0; a < 3; ++a) out[(size_t)a * N + i] = (double)F[a];
    return;
  }
  if (m & IDMASK) {
    if (which == EXP_F) {
      for (int q = 0; q < NQ; ++q) out[(size_t)q * N + i] = 0.0;
    } else if (which == EXP_RHO) {
      out[i] = B.p.rho0;
    } else {
      const DevColloid& C = B.col[(m & IDMASK) - 1];
      double d[3], ur[3];
      disp(B, (double)x, (double)y, (double)z, C.X, d);
      rigid_velocity(C.V, C.W, d, ur);
      for (int a = 0; a < 3; ++a) out[(size_t)a * N + i] = ur[a];
    }
    return;
  }
  T df[NQ];
  pull(B, static_cast<const T*>(B.f[B.st->fpar]), x, y, z, i, m, B.st->pre_valid != 0, df);
  if (which == EXP_F) {
    for (int q = 0; q < NQ; ++q) out[(size_t)q * N + i] = wq(q) * B.p.rho0 + (double)df[q];
    return;
  }
  double drho, mm[3];
  moments_f64(df, F, drho, mm);
  const double rho = B.p.rho0 + drho;
  if (which == EXP_RHO) {
    out[i] = rho;
    return;
  }
  // 1/rho by Newton from the FP32 reciprocal (to rounding in two steps)
  const float rf = (float)rho;
  double inv;
  if (rf > 1e-30f && rf < 1e30f) {
    inv = f32_to_f64(1.f / rf);
    inv = inv * (2.0 - rho * inv);
    inv = inv * (2.0 - rho * inv);
  } else {
    inv = 1.0 / rho;
  }
  const bool forced = B.p.g[0] != 0.0 || B.p.g[1] != 0.0 || B.p.g[2] != 0.0;
  for (int a = 0; a < 3; ++a) {
    double m = mm[a];
    if (forced) m += 0.5 * B.p.g[a];
    out[(size_t)a * N + i] = m * inv;
  }
}

// Diagnostics per block: [0] sum(df), [1..3] sum(df c), [4] fluid nodes,
// [5] defect nodes (3/2 lambda_max(Q) < 0.435).  Bound by FP64 issue: the
// moments of FP32 populations are summed as integers, a thread sums DIAG_PER
// nodes before the block reduction, and the defect test runs in FP32 except at
// nodes too close to the threshold (with the closed-form eigenvalue in FP64 at
// every node and 19 x 4 products: 1102 us at 128^3).  At 64 registers 32 warps
// fit an SM: 158 -> 115 us at 128^3.
constexpr int DIAG_PER = 4;
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_diag_state(const DevBox* __restrict__ boxes, int b,
                                                                              double* __restrict__ part) {
  const DevBox& B = boxes[b];
  double v[6] = {0, 0, 0, 0, 0, 0};
  __shared__ double sred[32 * 6];
  int nfl = 0, ndef = 0;
  const int nx = B.nx, ny = B.ny, N = B.N, qpar = B.st->qpar;
  for (int r = 0; r < DIAG_PER; ++r) {
    const long long il = ((long long)blockIdx.x * DIAG_PER + r) * 256 + threadIdx.x;
    if (il >= N) break;
    const int i = (int)il;
    const uint8_t m = B.mask[i];
    if (m & IDMASK) continue;
    const int x = i % nx, y = (i / nx) % ny, z = i / (nx * ny);
    T df[NQ];
    pull(B, static_cast<const T*>(B.f[B.st->fpar]), x, y, z, i, m, B.st->pre_valid != 0, df);
    double drho, mom[3];
    moments_f64(df, drho, mom);
    v[0] += drho;
    v[1] += mom[0];
    v[2] += mom[1];
    v[3] += mom[2];
    ++nfl;
    float qf[5];
    load_q_f32<T>(B, qpar, i, qf);
    int low = below_f32(qf, 0.29f);
    if (low < 0) {
      double q[5];
      for (int k = 0; k < 5; ++k) q[k] = load_q<T>(B, i, k);
      // largest eigenvalue of the traceless symmetric Q (closed form, as in principal_dir)
      double a00 = q[0], a01 = q[1], a02 = q[2], a11 = q[3], a12 = q[4], a22 = -q[0] - q[3];
      double p1 = a01 * a01 + a02 * a02 + a12 * a12;
      double p2 = a00 * a00 + a11 * a11 + a22 * a22 + 2.0 * p1;
      double lam = 0.0;
      if (p2 > 0.0) {
        double p = sqrt(p2 / 6.0);
        double b00 = a00 / p, b01 = a01 / p, b02 = a02 / p, b11 = a11 / p, b12 = a12 / p, b22 = a22 / p;
        double det = b00 * (b11 * b22 - b12 * b12) - b01 * (b01 * b22 - b12 * b02) + b02 * (b01 * b12 - b11 * b02);
        double r3 = fmin(1.0, fmax(-1.0, det / 2.0));
        lam = 2.0 * p * cos(acos(r3) / 3.0);
      }
      low = 1.5 * lam < 0.435;
    }
    ndef += low;
  }
  v[4] = (double)nfl;
  v[5] = (double)ndef;
  block_sum<6>(v, sred);
  if (threadIdx.x == 0)
    for (int k = 0; k < 6; ++k) part[6 * blockIdx.x + k] = v[k];
}

// Deterministic sum of n records of width w starting at rec0, one block per
// column k; out[k] = sum, or max for columns flagged in maxmask.
__global__ void __launch_bounds__(256) k_reduce(const double* __restrict__ part, int rec0, int n, int w,
                                                unsigned maxmask, double* __restrict__ out) {
  __shared__ double s[256];
  const int k = blockIdx.x;
  const bool ismax = (maxmask >> k) & 1u;
  double v = 0.0;
  for (int r = threadIdx.x; r < n; r += 256) {
    const double x = part[(size_t)(rec0 + r) * w + k];
    v = ismax ? fmax(v, x) : v + x;
  }
  s[threadIdx.x] = v;
  __syncthreads();
  for (int d = 128; d > 0; d >>= 1) {
    if (threadIdx.x < d) s[threadIdx.x] = ismax ? fmax(s[threadIdx.x], s[threadIdx.x + d]) : s[threadIdx.x] + s[threadIdx.x + d];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[k] = s[0];
}

// ---------------------------------------------------------------------------
// re-discretisation of moving colloids (Sec. 2.2, last paragraph)
// ---------------------------------------------------------------------------
// One launch (k_rediscretise) after the colloid update, which has flagged the
// boxes where a mobile colloid moved past its margin (DevState::scan); without
// one every block returns at once.  Phases, with a grid barrier between them
// (the launch is cooperative, so all its blocks are resident):
//   rd_find   nodes of the colloid's bounding region whose solid test at the
//             new X differs from the mask -> change list; the least distance
//             of a node from the surface -> margin
//   rd_pull   pre-collision populations of the step just streamed, pulled
//             with the old mask and the old colloid state, into the other
//             buffer (the next collide reads them in place)
//   rd_apply  covered nodes hand their momentum sum_q df_q c_q to the
//             colloid; uncovered nodes take f_eq(rho_bar, u_b) and the
//             mean Q of their fluid face neighbours (fluid before and after)
//   rd_mask   mask bits of the changed nodes; rd_near the near flags of the
//             region; rd_count the near nodes of each block's part of the box;
//             rd_links the boundary links and near list; rd_finish the box state.
// As eight launches that returned at once they took 52 us of the 113 us step
// of a 64^3 box with one mobile colloid.
__device__ __forceinline__ int region_lo(double c, double r) { return (int)floor(c - r - 2.0); }

// Node (x,y,z) of the bounding region of colloid C: index k of n = nx*ny*nz region
// nodes; returns false when the region node falls outside a z wall.
__device__ __forceinline__ bool region_node(const DevBox& B, const DevColloid& C, int k, int& x, int& y, int& z) {
  const int lx = region_lo(C.X[0], C.a0), ly = region_lo(C.X[1], C.a0), lz = region_lo(C.X[2], C.a0);
  const int ex = min(B.nx, (int)ceil(2.0 * C.a0) + 5), ey = min(B.ny, (int)ceil(2.0 * C.a0) + 5),
            ez = min(B.nz, (int)ceil(2.0 * C.a0) + 5);
  const int ix = k % ex, iy = (k / ex) % ey, iz = k / (ex * ey);
  x = wrapn(lx + ix, B.nx);
  y = wrapn(ly + iy, B.ny);
  z = lz + iz;
  if (B.wall_z) return z >= 0 && z < B.nz;
  z = wrapn(z, B.nz);
  return true;
}

__device__ __forceinline__ int region_size(const DevBox& B, const DevColloid& C) {
  const int e = (int)ceil(2.0 * C.a0) + 5;
  return min(B.nx, e) * min(B.ny, e) * min(B.nz, e);
}

// New solid owner of node (x,y,z): colloid index + 1, or 0.  No node is
// inside two colloids: add_colloid refuses a colloid that touches another and
// the colloid update puts back a move into contact (resolve_contacts), so the
// first colloid found is the only one.
__device__ __forceinline__ int new_owner(const DevBox& B, int x, int y, int z) {
  for (int c = 0; c < B.ncol; ++c)
    if (inside_colloid(B, x, y, z, B.col[c])) return c + 1;
  return 0;
}

// Words that other blocks of the same launch write: read through L2.
__device__ __forceinline__ int ld_state(const int* p) { return __ldcg(p); }

__device__ void rd_find(DevBox* __restrict__ boxes, const int2* __restrict__ mob, int nmob) {
  for (int p = 0; p < nmob; ++p) {
    const DevBox& B = boxes[mob[p].x];
    if (!B.st->scan) continue;
    DevColloid& C = B.col[mob[p].y];
    const int c = mob[p].y, n = region_size(B, C);
    double gap = 1.0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
      int x, y, z;
      if (!region_node(B, C, k, x, y, z)) continue;
      const int i = x + B.nx * (y + B.ny * z);
      const int old = B.mask[i] & IDMASK;
      const bool in_new = inside_colloid(B, x, y, z, C);
      double r[3];
      disp(B, (double)x, (double)y, (double)z, C.X, r);
      gap = fmin(gap, fabs(sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]) - C.a0));
      int code = -1;
      if (in_new && old == 0) code = c << 1;                 // covered
      else if (!in_new && old == c + 1) code = (c << 1) | 1;  // uncovered
      else if (in_new && old != 0 && old != c + 1) atomicOr(&B.st->err, 4);
      if (code >= 0) {
        const int slot = atomicAdd(&B.st->nchg, 1);
        if (slot < B.chg_cap) {
          B.chg[2 * slot] = i;
          B.chg[2 * slot + 1] = code;
        } else {
          atomicOr(&B.st->err, 2);
        }
      }
    }
    // positive doubles order as their bits
    if (gap < 1.0) atomicMin(reinterpret_cast<unsigned long long*>(&C.margin), (unsigned long long)__double_as_longlong(gap));
  }
}

template <typename T>
__device__ void rd_pull(DevBox* __restrict__ boxes, int nboxes) {
  for (int b = 0; b < nboxes; ++b) {
    const DevBox& B = boxes[b];
    if (ld_state(&B.st->nchg) == 0 || !B.p.flow_on) continue;
    const int fpar = B.st->fpar;
    const bool pre = B.st->pre_valid != 0;
    const T* fin = static_cast<const T*>(B.f[fpar]);
    T* fpre = static_cast<T*>(B.f[fpar ^ 1]);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B.N; i += gridDim.x * blockDim.x) {
      const uint8_t m = B.mask[i];
      if (m & IDMASK) continue;
      const int x = i % B.nx, y = (i / B.nx) % B.ny, z = i / (B.nx * B.ny);
      T df[NQ];
      pull(B, fin, x, y, z, i, m, pre, df);
#pragma unroll
      for (int q = 0; q < NQ; ++q) fpre[(size_t)q * B.N + i] = df[q];
    }
  }
}

template <typename T>
__device__ void rd_apply(DevBox* __restrict__ boxes, int nboxes) {
  for (int b = 0; b < nboxes; ++b) {
    DevBox& B = boxes[b];
    const int nchg = min(ld_state(&B.st->nchg), B.chg_cap);
    if (nchg == 0) continue;
    const int fpar = B.st->fpar;
    T* fpre = static_cast<T*>(B.f[fpar ^ 1]);
    const int N = B.N;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nchg; k += gridDim.x * blockDim.x) {
      const int i = B.chg[2 * k], code = B.chg[2 * k + 1];
      const int c = code >> 1;
      DevColloid& C = B.col[c];
      const int x = i % B.nx, y = (i / B.nx) % B.ny, z = i / (B.nx * B.ny);
      if ((code & 1) == 0) {  // covered: its fluid momentum goes to the colloid
        if (B.p.flow_on) {
          double mom[3] = {0.0, 0.0, 0.0};
          for (int q = 0; q < NQ; ++q) {
            const double d = (double)fpre[(size_t)q * N + i];
            mom[0] += cx(q) * d;
            mom[1] += cy(q) * d;
            mom[2] += cz(q) * d;
            fpre[(size_t)q * N + i] = T(0);
          }
          for (int a = 0; a < 3; ++a) {
            atomicAdd(&C.imp[a], mom[a]);
            atomicAdd(&C.rdp[a], mom[a]);
          }
        }
        continue;
      }
      // uncovered: neighbours fluid before and after
      double rsum = 0.0, qsum[5] = {0, 0, 0, 0, 0};
      int cnt = 0;
      for (int d = 0; d < 6; ++d) {
        int xx = x, yy = y, zz = z;
        if (d == 0) xx = wrap1(x + 1, B.nx);
        if (d == 1) xx = wrap1(x - 1, B.nx);
        if (d == 2) yy = wrap1(y + 1, B.ny);
        if (d == 3) yy = wrap1(y - 1, B.ny);
        if (d == 4) zz = z + 1;
        if (d == 5) zz = z - 1;
        if (B.wall_z) {
          if (zz < 0 || zz >= B.nz) continue;
        } else {
          zz = wrap1(zz, B.nz);
        }
        const int j = xx + B.nx * (yy + B.ny * zz);
        if ((B.mask[j] & IDMASK) != 0 || new_owner(B, xx, yy, zz) != 0) continue;
        double rj = B.p.rho0;
        if (B.p.flow_on)
          for (int q = 0; q < NQ; ++q) rj += (double)fpre[(size_t)q * N + j];
        rsum += rj;
        for (int kk = 0; kk < 5; ++kk) qsum[kk] += load_q<T>(B, j, kk);
        ++cnt;
      }
      const double rb = cnt ? rsum / cnt : B.p.rho0;
      double dd[3], ubv[3];
      disp(B, (double)x, (double)y, (double)z, C.X, dd);
      rigid_velocity(C.V, C.W, dd, ubv);
      if (B.p.flow_on) {
        const double uu = ubv[0] * ubv[0] + ubv[1] * ubv[1] + ubv[2] * ubv[2];
        for (int q = 0; q < NQ; ++q) {
          const double cu = cx(q) * ubv[0] + cy(q) * ubv[1] + cz(q) * ubv[2];
          const double feq = wq(q) * rb * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu);
          fpre[(size_t)q * N + i] = T(feq - wq(q) * B.p.rho0);
        }
        for (int a = 0; a < 3; ++a) {
          atomicAdd(&C.imp[a], -rb * ubv[a]);
          atomicAdd(&C.rdp[a], -rb * ubv[a]);
        }
      }
      if (cnt)
        for (int kk = 0; kk < 5; ++kk) store_q_cur<T>(B, i, kk, qsum[kk] / cnt);
    }
  }
}

__device__ void rd_mask(DevBox* __restrict__ boxes, int nboxes) {
  for (int b = 0; b < nboxes; ++b) {
    const DevBox& B = boxes[b];
    const int nchg = min(ld_state(&B.st->nchg), B.chg_cap);
    if (nchg == 0) continue;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nchg; k += gridDim.x * blockDim.x) {
      const int i = B.chg[2 * k], code = B.chg[2 * k + 1];
      B.mask[i] = (code & 1) ? (uint8_t)0 : (uint8_t)((code >> 1) + 1);
    }
  }
}

__device__ void rd_near(DevBox* __restrict__ boxes, const int2* __restrict__ mob, int nmob) {
  for (int p = 0; p < nmob; ++p) {
    const DevBox& B = boxes[mob[p].x];
    if (ld_state(&B.st->nchg) == 0) continue;
    const DevColloid& C = B.col[mob[p].y];
    const int n = region_size(B, C);
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
      int x, y, z;
      if (!region_node(B, C, k, x, y, z)) continue;
      const int i = x + B.nx * (y + B.ny * z);
      const uint8_t m = B.mask[i];
      if (m & IDMASK) {
        B.mask[i] = m & IDMASK;
        continue;
      }
      bool near = false;
      for (int q = 1; q < NQ; ++q) {
        const int zz = z + cz(q);
        if (B.wall_z && (zz < 0 || zz >= B.nz)) {
          near = true;
          continue;
        }
        const int j = wrap1(x + cx(q), B.nx) + B.nx * (wrap1(y + cy(q), B.ny) + B.ny * wrap1(zz, B.nz));
        if (B.mask[j] & IDMASK) near = true;
      }
      B.mask[i] = near ? NEAR : (uint8_t)0;
    }
  }
}

// The block's part of the nodes of box B: whole 256s, in block order.
__device__ __forceinline__ void near_part(const DevBox& B, int& lo, int& hi) {
  const long long per = ((B.N + 255LL) / 256 + gridDim.x - 1) / gridDim.x * 256;
  lo = (int)min((long long)B.N, per * blockIdx.x);
  hi = (int)min((long long)B.N, per * (blockIdx.x + 1LL));
}
__device__ __forceinline__ int warp_total(int v) {
  return __reduce_add_sync(0xffffffffu, v);
}

__device__ void rd_count(DevBox* __restrict__ boxes, int nboxes) {
  for (int b = 0; b < nboxes; ++b) {
    const DevBox& B = boxes[b];
    if (ld_state(&B.st->nchg) == 0) continue;
    int lo, hi, n = 0;
    near_part(B, lo, hi);
    for (int base = lo; base < hi; base += 256) {
      const int i = base + (int)threadIdx.x;
      n += __syncthreads_count(i < hi && near_member(B, i));
    }
    if (threadIdx.x == 0) B.near_cnt[blockIdx.x] = n;
  }
}

// Rebuild the boundary links (unordered; lc_lb_get_links sorts them; their count
// is zeroed with the near flags) and the near-node lists of boxes whose solid set
// changed.
__device__ void rd_links(DevBox* __restrict__ boxes, int nboxes) {
  __shared__ int s_off[8];
  for (int b = 0; b < nboxes; ++b) {
    const DevBox& B = boxes[b];
    if (ld_state(&B.st->nchg) == 0) continue;
    {  // near nodes of the block's part, behind those of the blocks before it
      int lo, hi, before = 0;
      near_part(B, lo, hi);
      for (int k = threadIdx.x; k < (int)blockIdx.x; k += blockDim.x) before += __ldcg(B.near_cnt + k);
      before = warp_total(before);
      __syncthreads();
      if ((threadIdx.x & 31) == 0) s_off[threadIdx.x >> 5] = before;
      __syncthreads();
      int at = 0;
      for (int k = 0; k < 8; ++k) at += s_off[k];
      for (int base = lo; base < hi; base += 256) {
        const int i = base + (int)threadIdx.x;
        const bool near = i < hi && near_member(B, i);
        const int pos = at + near_rank(near, s_off);
        if (near && pos < B.near_cap) B.near_node[pos] = i;
        at += __syncthreads_count(near);
      }
      if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *B.nnear = at;
    }
    for (int c = 0; c < B.ncol; ++c) {
      const DevColloid& C = B.col[c];
      const int n = region_size(B, C);
      for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        int x, y, z;
        if (!region_node(B, C, k, x, y, z)) continue;
        const int i = x + B.nx * (y + B.ny * z);
        unsigned bits;
        const int nl = links_at(B, i, c, &bits);
        if (!nl) continue;
        int pos = atomicAdd(B.nlinks, nl);
        for (int q = 1; q < NQ; ++q)
          if (bits & (1u << q)) {
            if (pos < B.nlinks_cap) {
              B.link_node[pos] = i;
              B.link_dir[pos] = (int8_t)q;
              B.link_col[pos] = (int8_t)c;
            } else {
              atomicOr(&B.st->err, 1);
            }
            ++pos;
          }
      }
    }
  }
}

// The next collide reads the pulled populations in place; the momentum
// exchanged by the re-discretisation changes each mobile colloid's velocity.
__device__ void rd_finish(DevBox* __restrict__ boxes, int b) {
  DevBox& B = boxes[b];
  DevState* st = B.st;
  if (ld_state(&st->nchg) == 0) return;
  if (B.p.flow_on) {
    st->fpar ^= 1;
    st->pre_valid = 1;
  }
  for (int c = 0; c < B.ncol; ++c) {
    DevColloid& C = B.col[c];
    if (C.mobile)
      for (int a = 0; a < 3; ++a) C.V[a] += C.rdp[a] / C.M;
    for (int a = 0; a < 3; ++a) C.rdp[a] = 0.0;
  }
  if (ld_state(B.nlinks) > B.nlinks_cap || ld_state(B.nnear) > B.near_cap) atomicOr(&st->err, 1);
}

// The word of the launch's barrier and the group's error word.
struct GridWords {
  unsigned* bar;
  int* err;
  __device__ unsigned word() const { return ld_acquire_u32(bar); }
  __device__ unsigned arrive(unsigned add) const {
    __threadfence();
    return atomicAdd(bar, add);
  }
  __device__ bool failed() const { return ld_acquire_u32(reinterpret_cast<const unsigned*>(err)) != 0u; }
  __device__ void fail() const { atomicOr(err, 1); }
  __device__ void pause() const { __nanosleep(40); }
};

__device__ bool grid_barrier(unsigned* bar, int* err, int spin_limit) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    GridWords w{bar, err};
    s_ok = barrier_wait(w, gridDim.x, blockIdx.x == 0, spin_limit);
    __threadfence();
  }
  __syncthreads();
  return s_ok != 0;
}

template <typename T>
__global__ void __launch_bounds__(256) k_rediscretise(DevBox* __restrict__ boxes, int nboxes,
                                                      const int2* __restrict__ mob, int nmob, unsigned* bar, int* err,
                                                      int spin_limit) {
  // (a wait that gave up in an earlier step: the state is invalid until the host
  // has reported it)
  bool any = false;
  if (*err == 0)
    for (int b = threadIdx.x; b < nboxes; b += blockDim.x) any = any || (boxes[b].nmobile && boxes[b].st->scan);
  if (!__syncthreads_or(any)) return;
  rd_find(boxes, mob, nmob);
  if (!grid_barrier(bar, err, spin_limit)) return;
  any = false;
  for (int b = threadIdx.x; b < nboxes; b += blockDim.x) any = any || ld_state(&boxes[b].st->nchg) != 0;
  if (!__syncthreads_or(any)) return;
  rd_pull<T>(boxes, nboxes);
  if (!grid_barrier(bar, err, spin_limit)) return;
  rd_apply<T>(boxes, nboxes);
  if (!grid_barrier(bar, err, spin_limit)) return;
  rd_mask(boxes, nboxes);
  if (!grid_barrier(bar, err, spin_limit)) return;
  rd_near(boxes, mob, nmob);
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b < nboxes; b += blockDim.x)
      if (ld_state(&boxes[b].st->nchg) > 0) *boxes[b].nlinks = 0;
  if (!grid_barrier(bar, err, spin_limit)) return;
  rd_count(boxes, nboxes);
  if (!grid_barrier(bar, err, spin_limit)) return;
  rd_links(boxes, nboxes);
  if (!grid_barrier(bar, err, spin_limit)) return;
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b < nboxes; b += blockDim.x) rd_finish(boxes, b);
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
// An error that is returned to the caller is taken from the runtime, so that the
// next launch does not report it again.
static cudaError_t taken(cudaError_t e) {
  cudaGetLastError();
  return e;
}

template <typename T, int TY>
static cudaError_t launch_force_t(const Launch& L, int mode, double* part) {
  constexpr int HP = (TX + 2) * (TY + 2);
  const size_t smem = sizeof(T) * 27 * HP + 3 * HP;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_force<T, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr = true;
  }
  k_force<T, TY><<<L.grid, dim3(TX, TY), smem, L.stream>>>(L.boxes, L.tiles, L.ntiles, L.zc, mode, part);
  return cudaGetLastError();
}

template <typename T, int TY>
static cudaError_t launch_lb_t(const Launch& L, int mode, double* part) {
  k_lb<T, TY><<<L.grid, dim3(TX, TY), 0, L.stream>>>(L.boxes, L.tiles, L.ntiles, L.zc, mode, part);
  return cudaGetLastError();
}

template <typename T, int BY>
static cudaError_t launch_flb_t(const Launch& L, int mode, double* part) {
  constexpr int HP = (TX + 2) * (BY + 2);
  const size_t smem = sizeof(T) * 27 * HP + 3 * HP;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_flb<T, BY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr = true;
  }
  k_flb<T, BY><<<L.grid, 32 * (BY + 3), smem, L.stream>>>(L.boxes, L.tiles, L.ntiles, L.zc, mode, part);
  return cudaGetLastError();
}

// Dynamic shared memory of the kernels that march with a Ring (0: FP64).
template <typename T, int NC, int TY>
constexpr size_t ring_bytes() { return sizeof(T) == 4 ? Ring<NC, TY>::BYTES : 0; }

template <typename T, int TY>
static cudaError_t launch_stress_t(const Launch& L, int mode, double* part) {
  constexpr size_t ring = ring_bytes<T, 5, TY>(), near = sizeof(NearScratch<T>) * TY, smem = ring > near ? ring : near;
  auto* fn = (mode & FORCE_FE) ? k_stress<T, TY, true> : k_stress<T, TY, false>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return taken(e);
  fn<<<L.grid, dim3(TX, TY), smem, L.stream>>>(L, mode, part);
  return cudaGetLastError();
}

template <typename T, int TY>
static cudaError_t launch_lbp_t(const Launch& L, int, double*) {
  k_lbp<T, TY><<<L.grid, dim3(TX, TY), 0, L.stream>>>(L);
  return cudaGetLastError();
}

template <typename T, int TY>
static cudaError_t launch_lc_t(const Launch& L, int mode, double* part) {
  constexpr size_t smem = ring_bytes<T, 8, TY>();
  if (smem > 0) {
    cudaError_t e = cudaFuncSetAttribute(k_lc<T, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return taken(e);
  }
  k_lc<T, TY><<<L.grid, dim3(TX, TY), smem, L.stream>>>(L, mode, part);
  return cudaGetLastError();
}

template <typename T, int TY>
static cudaError_t launch_relax_t(const Launch& L, int mode, double* part) {
  constexpr size_t ring = ring_bytes<T, 5, TY>(), near = sizeof(NearScratch<T>) * TY, smem = ring > near ? ring : near;
  cudaError_t e = cudaFuncSetAttribute(k_relax<T, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return taken(e);
  k_relax<T, TY><<<L.grid, dim3(TX, TY), smem, L.stream>>>(L, mode, part);
  return cudaGetLastError();
}

#define LCLB_DISPATCH_TY(FN, T)                      \
  switch (L.ty) {                                    \
    case 2: return FN<T, 2>(L, mode, part);          \
    case 4: return FN<T, 4>(L, mode, part);          \
    case 8: return FN<T, 8>(L, mode, part);          \
    default: return cudaErrorInvalidValue;           \
  }

cudaError_t launch_force(int prec, const Launch& L, int mode, double* part) {
  if (prec == 0) { LCLB_DISPATCH_TY(launch_force_t, float) }
  LCLB_DISPATCH_TY(launch_force_t, double)
}
cudaError_t launch_lb(int prec, const Launch& L, int mode, double* part) {
  if (prec == 0) { LCLB_DISPATCH_TY(launch_lb_t, float) }
  LCLB_DISPATCH_TY(launch_lb_t, double)
}
cudaError_t launch_flb(int prec, const Launch& L, int mode, double* part) {
  if (prec == 0) {
    switch (L.ty) {
      case 4: return launch_flb_t<float, 4>(L, mode, part);
      case 6: return launch_flb_t<float, 6>(L, mode, part);
      case 8: return launch_flb_t<float, 8>(L, mode, part);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (L.ty) {
    case 4: return launch_flb_t<double, 4>(L, mode, part);
    case 6: return launch_flb_t<double, 6>(L, mode, part);
    case 8: return launch_flb_t<double, 8>(L, mode, part);
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t launch_lc(int prec, const Launch& L, int mode, double* part) {
  if (prec == 0) { LCLB_DISPATCH_TY(launch_lc_t, float) }
  LCLB_DISPATCH_TY(launch_lc_t, double)
}
cudaError_t launch_relax(int prec, const Launch& L, int mode, double* part) {
  if (prec == 0) { LCLB_DISPATCH_TY(launch_relax_t, float) }
  LCLB_DISPATCH_TY(launch_relax_t, double)
}
cudaError_t launch_stress(int prec, const Launch& L, int mode, double* part) {
  if (prec == 0) { LCLB_DISPATCH_TY(launch_stress_t, float) }
  LCLB_DISPATCH_TY(launch_stress_t, double)
}
cudaError_t launch_lbp(int prec, const Launch& L, int mode, double* part) {
  if (prec == 0) { LCLB_DISPATCH_TY(launch_lbp_t, float) }
  LCLB_DISPATCH_TY(launch_lbp_t, double)
}

cudaError_t launch_links(int prec, const DevBox* boxes, const int2* chunks, int nchunks, int grid, cudaStream_t s) {
  if (nchunks <= 0) return cudaSuccess;
  if (prec == 0) k_links<float><<<grid, LINK_CHUNK, 0, s>>>(boxes, chunks, nchunks);
  else k_links<double><<<grid, LINK_CHUNK, 0, s>>>(boxes, chunks, nchunks);
  return cudaGetLastError();
}

cudaError_t launch_colloid(DevBox* boxes, int nboxes, cudaStream_t s) {
  k_colloid<<<nboxes, 128, 0, s>>>(boxes, nboxes);
  return cudaGetLastError();
}

template <typename T, int TY>
static cudaError_t launch_step_t(DevBox* boxes, const StepItem* items, int nitems, int zc, unsigned* sync,
                                 double* part, int spin_limit, int commit, int* err, int grid, cudaStream_t s) {
  constexpr size_t smem = sizeof(NearScratch<T>) * TY;
  cudaError_t e = cudaFuncSetAttribute(k_step<T, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return taken(e);
  k_step<T, TY><<<grid, dim3(TX, TY), smem, s>>>(boxes, items, nitems, zc, sync, part, spin_limit, commit, err);
  return cudaGetLastError();
}

cudaError_t launch_step(int prec, int ty, DevBox* boxes, const StepItem* items, int nitems, int zc, unsigned* sync,
                        double* part, int spin_limit, int commit, int* err, int grid, cudaStream_t s) {
#define LCLB_STEP_CASE(T, Y) \
  case Y: return launch_step_t<T, Y>(boxes, items, nitems, zc, sync, part, spin_limit, commit, err, grid, s);
  if (prec == 0) {
    switch (ty) { LCLB_STEP_CASE(float, 2) LCLB_STEP_CASE(float, 4) LCLB_STEP_CASE(float, 8) default: break; }
  } else {
    switch (ty) { LCLB_STEP_CASE(double, 2) LCLB_STEP_CASE(double, 4) LCLB_STEP_CASE(double, 8) default: break; }
  }
#undef LCLB_STEP_CASE
  return cudaErrorInvalidValue;
}

int step_blocks_per_sm(int prec, int ty) {
  int n = 0;
  cudaError_t e = cudaErrorInvalidValue;
#define LCLB_OCC(T, Y) \
  case Y: \
    e = cudaFuncSetAttribute(k_step<T, Y>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NearScratch<T>) * Y); \
    if (e == cudaSuccess) \
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step<T, Y>, TX * Y, sizeof(NearScratch<T>) * Y); \
    break;
  if (prec == 0) {
    switch (ty) { LCLB_OCC(float, 2) LCLB_OCC(float, 4) LCLB_OCC(float, 8) default: break; }
  } else {
    switch (ty) { LCLB_OCC(double, 2) LCLB_OCC(double, 4) LCLB_OCC(double, 8) default: break; }
  }
#undef LCLB_OCC
  return e == cudaSuccess && n > 0 ? n : 1;
}

static inline int nblk(int N, int bs) { return (N + bs - 1) / bs; }

cudaError_t launch_pair_constants(DevBox* boxes, int b, cudaStream_t s) {
  k_pair_constants<<<1, 1, 0, s>>>(boxes, b);
  return cudaGetLastError();
}

cudaError_t launch_geometry(DevBox* boxes, int b, int N, cudaStream_t s) {
  k_mask<<<nblk(N, 256), 256, 0, s>>>(boxes, b);
  k_near<<<nblk(N, 256), 256, 0, s>>>(boxes, b);
  return cudaGetLastError();
}

cudaError_t launch_near_list(DevBox* boxes, int b, int N, int* blocksum, int* total, cudaStream_t s) {
  const int nb = nblk(N, 256);
  k_near_count<<<nb, 256, 0, s>>>(boxes, b, blocksum);
  k_scan<<<1, 1024, 0, s>>>(blocksum, nb, 0, total);
  k_near_write<<<nb, 256, 0, s>>>(boxes, b, blocksum);
  return cudaGetLastError();
}

cudaError_t launch_link_build(DevBox* boxes, int b, int N, int c, int* blocksum, int base, int* total,
                              cudaStream_t s) {
  const int nb = nblk(N, 256);
  k_link_count<<<nb, 256, 0, s>>>(boxes, b, c, blocksum);
  k_scan<<<1, 1024, 0, s>>>(blocksum, nb, base, total);
  k_link_write<<<nb, 256, 0, s>>>(boxes, b, c, blocksum);
  return cudaGetLastError();
}

cudaError_t launch_init_q(int prec, DevBox* boxes, int b, int N, int kind, const double* n, double amp,
                          unsigned long long seed, cudaStream_t s) {
  if (prec == 0) k_init_q<float><<<nblk(N, 256), 256, 0, s>>>(boxes, b, kind, n[0], n[1], n[2], amp, seed);
  else k_init_q<double><<<nblk(N, 256), 256, 0, s>>>(boxes, b, kind, n[0], n[1], n[2], amp, seed);
  return cudaGetLastError();
}

cudaError_t launch_set_field(int prec, DevBox* boxes, int b, int N, int which, const double* src, cudaStream_t s) {
  if (prec == 0) k_set_field<float><<<nblk(N, 256), 256, 0, s>>>(boxes, b, which, src);
  else k_set_field<double><<<nblk(N, 256), 256, 0, s>>>(boxes, b, which, src);
  return cudaGetLastError();
}

cudaError_t launch_export_q(int prec, const DevBox* boxes, int b, int N, bool vec, double* out, cudaStream_t s) {
  const size_t n = 5 * (size_t)N;
  const unsigned g1 = (unsigned)((n + 255) / 256), g4 = (unsigned)((n + 1023) / 1024);
  if (prec != 0) k_export_q<double, 1><<<g1, 256, 0, s>>>(boxes, b, out);
  else if (vec) k_export_q<float, 4><<<g4, 256, 0, s>>>(boxes, b, out);
  else k_export_q<float, 1><<<g1, 256, 0, s>>>(boxes, b, out);
  return cudaGetLastError();
}

cudaError_t launch_export(int prec, const DevBox* boxes, int b, int N, int which, double* out, cudaStream_t s) {
  if (prec == 0) k_export<float><<<nblk(N, 256), 256, 0, s>>>(boxes, b, which, out);
  else k_export<double><<<nblk(N, 256), 256, 0, s>>>(boxes, b, which, out);
  return cudaGetLastError();
}


cudaError_t launch_rediscretise(int prec, DevBox* boxes, int nboxes, const int2* mob, int nmob, int nsm,
                                unsigned* bar, int* err, int spin_limit, cudaStream_t s) {
  if (nmob <= 0) return cudaSuccess;
  // one block per SM: all resident, which the cooperative launch guarantees
  void* args[] = {&boxes, &nboxes, &mob, &nmob, &bar, &err, &spin_limit};
  const void* fn = prec == 0 ? (const void*)k_rediscretise<float> : (const void*)k_rediscretise<double>;
  cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(nsm), dim3(256), args, 0, s);
  if (e != cudaSuccess) return taken(e);
  return cudaGetLastError();
}

int diag_state_blocks(int N) { return (N - 1) / (256 * DIAG_PER) + 1; }

cudaError_t launch_diag_state(int prec, const DevBox* boxes, int b, int N, double* part, cudaStream_t s) {
  if (prec == 0) k_diag_state<float><<<diag_state_blocks(N), 256, 0, s>>>(boxes, b, part);
  else k_diag_state<double><<<diag_state_blocks(N), 256, 0, s>>>(boxes, b, part);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const double* part, int rec0, int n, int w, unsigned maxmask, double* out, cudaStream_t s) {
  k_reduce<<<w, 256, 0, s>>>(part, rec0, n, w, maxmask, out);
  return cudaGetLastError();
}

}  // namespace lclb
