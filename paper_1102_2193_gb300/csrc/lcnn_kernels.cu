// lcnn_kernels.cu -- kernels of the learned warm start: a small 3D U-Net that
// proposes the relaxed Q around a colloid, trained on fields the solver
// itself relaxes.  Activations are channels-last BF16 ([position][channel],
// position = x + W*(y + H*z)), weights [C_out][taps][C_in] BF16 with FP32
// masters; every convolution accumulates in FP32 on the tensor cores
// (mma.sync m16n8k16 bf16, implicit GEMM).  Boundaries are periodic, like the
// boxes the fields come from.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "../../include/lc_nn.h"
#include "f64_bits.cuh"

namespace lcnn {

__device__ __forceinline__ int wrapi(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// Position of tap t (0..26, (dz+1)*9 + (dy+1)*3 + (dx+1)) around p; taps == 1: p itself.
__device__ __forceinline__ int tap_pos(int p, int t, int taps, int W, int H, int D) {
  if (taps == 1) return p;
  const int x = p % W, y = (p / W) % H, z = p / (W * H);
  const int dz = t / 9 - 1, dy = (t / 3) % 3 - 1, dx = t % 3 - 1;
  return wrapi(x + dx, W) + W * (wrapi(y + dy, H) + H * wrapi(z + dz, D));
}

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], const uint32_t b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t ld2(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// out[p][co] = act(bias[co] + sum_{t, ci} w[co][t][ci] in[tap(p, t)][ci]).
// One warp: 16 consecutive positions x all C_out (NT = C_out/8 tiles of 8).
// A fragment (16 positions x 16 channels of one tap), B fragment (16
// channels x 8 output channels), C: FP32.
template <int NT>
__global__ void __launch_bounds__(128) k_conv_fwd(const __nv_bfloat16* __restrict__ in, const __nv_bfloat16* __restrict__ w,
                                                  const float* __restrict__ bias, float* __restrict__ out32,
                                                  __nv_bfloat16* __restrict__ out16, int npos, int W, int H, int D,
                                                  int cin, int taps, int relu) {
  constexpr int COUT = NT * 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int p0 = (blockIdx.x * 4 + warp) * 16;
  if (p0 >= npos) return;
  const int g = lane >> 2, tg = lane & 3;
  float acc[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
  const int pa = min(p0 + g, npos - 1), pb = min(p0 + g + 8, npos - 1);
  for (int t = 0; t < taps; ++t) {
    const int qa = tap_pos(pa, t, taps, W, H, D), qb = tap_pos(pb, t, taps, W, H, D);
    const __nv_bfloat16* ra = in + (size_t)qa * cin;
    const __nv_bfloat16* rb = in + (size_t)qb * cin;
    for (int c0 = 0; c0 < cin; c0 += 16) {
      uint32_t a[4];
      a[0] = ld2(ra + c0 + tg * 2);
      a[1] = ld2(rb + c0 + tg * 2);
      a[2] = ld2(ra + c0 + 8 + tg * 2);
      a[3] = ld2(rb + c0 + 8 + tg * 2);
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const __nv_bfloat16* wr = w + ((size_t)(j * 8 + g) * taps + t) * cin + c0;
        uint32_t b[2] = {ld2(wr + tg * 2), ld2(wr + 8 + tg * 2)};
        mma_bf16(acc[j], a, b);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < NT; ++j) {
    const int co = j * 8 + tg * 2;
    const float b0 = bias ? bias[co] : 0.f, b1 = bias ? bias[co + 1] : 0.f;
    float v[4] = {acc[j][0] + b0, acc[j][1] + b1, acc[j][2] + b0, acc[j][3] + b1};
    if (relu)
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = fmaxf(v[k], 0.f);
    const int rows[2] = {p0 + g, p0 + g + 8};
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (rows[r] >= npos) continue;
      const size_t o = (size_t)rows[r] * COUT + co;
      if (out32) {
        out32[o] = v[2 * r];
        out32[o + 1] = v[2 * r + 1];
      }
      if (out16) {
        out16[o] = __float2bfloat16_rn(v[2 * r]);
        out16[o + 1] = __float2bfloat16_rn(v[2 * r + 1]);
      }
    }
  }
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void ldm4(uint32_t r[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldm2(uint32_t r[2], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldm4t(uint32_t r[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
// Byte offset of half h (8 channels, 16 bytes) of row p in a tile of 32-byte
// rows (16 channels): the halves swap every four rows, so the eight rows of
// an 8x8 ldmatrix, consecutive from any start, fall in eight different 16-byte
// bank groups.
__device__ __forceinline__ uint32_t row32(int p, int h) {
  return (uint32_t)(p << 5) + (uint32_t)(((h ^ (p >> 2)) & 1) << 4);
}
__device__ __forceinline__ int modn(int v, int n) {
  const int r = v % n;
  return r < 0 ? r + n : r;
}

// Periodic 3x3x3 convolution over a TX x TY x TZ box of positions per block:
// for each 16 input channels the box with its one-node halo (32 bytes a
// position) and the 27 x COUT x 16 weights go to shared memory once, and the
// 27 taps read their A fragments there by ldmatrix at shifted row addresses.
// k_conv_fwd, which this replaces for 3x3x3 kernels, read every position 27
// times through L1 with 4-byte loads (16 -> 16 channels at 128^3: 740 us).
// A warp holds MT 16-position tiles x NT 8-channel tiles, so one B fragment
// serves MT products; in boxes 16 wide its tiles are MT consecutive rows of y,
// so the MT + 2 rows of A that one (dx, dz) needs serve all three dy (shared
// memory reads bound the kernel: 61 % of its wavefronts with 12 loads of A per
// (dx, dz) instead of 6).  MT and NT are bounded by the accumulator registers,
// the tile by 2 or 3 blocks per SM.  FP32 accumulation in the order (16-channel group,
// tap).  blockIdx.y picks the group of NT * 8 output channels.
template <int NT, int MT, int NW, int TX, int TY, int TZ>
__global__ void __launch_bounds__(32 * NW, NW == 8 ? (NT <= 2 ? 3 : (NT <= 4 ? 2 : 1)) : 6) k_conv_tile(const __nv_bfloat16* __restrict__ in,
                                                       const __nv_bfloat16* __restrict__ w,
                                                       const float* __restrict__ bias, float* __restrict__ out32,
                                                       __nv_bfloat16* __restrict__ out16, int W, int H, int D, int cin,
                                                       int cout, int relu, int ntx, int nty) {
  static_assert(TX * TY * TZ == 16 * MT * NW, "one 16-position tile per (warp, MT)");
  static_assert(TX != 16 || TY % MT == 0, "a warp's rows share z");
  constexpr int HX = TX + 2, HY = TY + 2, HZ = TZ + 2, HP = HX * HY * HZ, NTHR = 32 * NW;
  constexpr int NPT = (HP + NTHR - 1) / NTHR, NWR = 27 * NT * 8;
  extern __shared__ __align__(128) unsigned char smem[];
  const uint32_t sA = smem_addr(smem), sW = sA + HP * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % nty, bz = blockIdx.x / (ntx * nty);
  const int x0 = bx * TX, y0 = by * TY, z0 = bz * TZ, co0 = blockIdx.y * NT * 8;
  int pos[NPT];
#pragma unroll
  for (int k = 0; k < NPT; ++k) {
    const int p = tid + k * NTHR;
    pos[k] = modn(x0 + p % HX - 1, W) + W * (modn(y0 + (p / HX) % HY - 1, H) + H * modn(z0 + p / (HX * HY) - 1, D));
  }
  int rowp[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    const int m = (warp * MT + i) * 16 + (lane & 15);
    rowp[i] = m % TX + HX * ((m / TX) % TY + HY * (m / (TX * TY)));
  }
  const int ahalf = lane >> 4;                                // A: rows lane & 15, channels 8 ahalf..
  const int brow = ((lane >> 4) & 1) * 8 + (lane & 7);        // B: output channel within a pair of 8-tiles
  const int bhalf = (lane >> 3) & 1;
  float acc[MT][NT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[i][j][0] = acc[i][j][1] = acc[i][j][2] = acc[i][j][3] = 0.f;
  for (int c0 = 0; c0 < cin; c0 += 16) {
    if (c0) __syncthreads();
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      const int p = tid + k * NTHR;
      if (p < HP) {
        const __nv_bfloat16* src = in + (size_t)pos[k] * cin + c0;
        cp16(sA + row32(p, 0), src);
        cp16(sA + row32(p, 1), src + 8);
      }
    }
    for (int r = tid; r < NWR; r += NTHR) {
      const int t = r / (NT * 8), co = r % (NT * 8);
      const __nv_bfloat16* src = w + ((size_t)(co0 + co) * 27 + t) * cin + c0;
      cp16(sW + row32(r, 0), src);
      cp16(sW + row32(r, 1), src + 8);
    }
    cp_wait_all();
    __syncthreads();
    // B fragments of tap t
    auto load_b = [&](int t, uint32_t b[NT][2]) {
#pragma unroll
      for (int j = 0; j + 1 < NT; j += 2) {
        uint32_t q[4];
        ldm4(q, sW + row32(t * NT * 8 + j * 8 + brow, bhalf));
        b[j][0] = q[0];
        b[j][1] = q[1];
        b[j + 1][0] = q[2];
        b[j + 1][1] = q[3];
      }
      if constexpr (NT & 1) ldm2(b[NT - 1], sW + row32(t * NT * 8 + (NT - 1) * 8 + (lane & 7), bhalf));
    };
#pragma unroll 1
    for (int dz = 0; dz < 3; ++dz)
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) {
        uint32_t a[MT + 2][4], b[NT][2];
        if constexpr (TX == 16) {
#pragma unroll
          for (int i = 0; i < MT + 2; ++i) ldm4(a[i], sA + row32(rowp[0] + dx + HX * (i + HY * dz), ahalf));
        }
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
          if constexpr (TX != 16) {
#pragma unroll
            for (int i = 0; i < MT; ++i) ldm4(a[i + dy], sA + row32(rowp[i] + dx + HX * (dy + HY * dz), ahalf));
          }
          load_b(dz * 9 + dy * 3 + dx, b);
#pragma unroll
          for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j) mma_bf16(acc[i][j], a[i + dy], b[j]);
        }
      }
  }
  const int g = lane >> 2, tg = lane & 3;
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int m = (warp * MT + i) * 16 + g + 8 * r;
      const int x = x0 + m % TX, y = y0 + (m / TX) % TY, z = z0 + m / (TX * TY);
      if (x >= W || y >= H || z >= D) continue;
      const size_t o = ((size_t)x + (size_t)W * (y + (size_t)H * z)) * cout + co0 + tg * 2;
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        float v0 = acc[i][j][2 * r], v1 = acc[i][j][2 * r + 1];
        if (bias) {
          v0 += bias[co0 + j * 8 + tg * 2];
          v1 += bias[co0 + j * 8 + tg * 2 + 1];
        }
        if (relu) {
          v0 = fmaxf(v0, 0.f);
          v1 = fmaxf(v1, 0.f);
        }
        if (out32) {
          out32[o + j * 8] = v0;
          out32[o + j * 8 + 1] = v1;
        }
        if (out16) {
          out16[o + j * 8] = __float2bfloat16_rn(v0);
          out16[o + j * 8 + 1] = __float2bfloat16_rn(v1);
        }
      }
    }
}

// Partial dW of the 3x3x3 kernel: block (chunk, 16 output channels x 16 input
// channels, tap group) sums its boxes of 16 x TY x TZ positions (boxes chunk,
// chunk + nchunk, ... in order) with the input box and its halo and the
// output-gradient box in shared memory; nine warps take TPW taps each.  Both
// operands are position-major, so A (dout^T) and B (shifted input) are read by
// transposing ldmatrix, a tap being a shifted row address; one A fragment
// serves TPW taps.  k_conv_wgrad read both through 2-byte global loads, once
// per tap (16 x 16 channels at 64^3: 185 us).  Positions past the end of a
// ragged box read a row of zeros on both sides.
template <int TPW, int TY, int TZ>
__global__ void __launch_bounds__(288) k_wgrad_tile(const __nv_bfloat16* __restrict__ dout,
                                                    const __nv_bfloat16* __restrict__ in, float* __restrict__ part,
                                                    int W, int H, int D, int cin, int cout, int ntx, int nty, int ntz,
                                                    int nchunk) {
  constexpr int TX = 16, HX = TX + 2, HY = TY + 2, HZ = TZ + 2, HP = HX * HY * HZ, NP = TX * TY * TZ, NTHR = 288;
  extern __shared__ __align__(128) unsigned char smem[];
  const uint32_t sI = smem_addr(smem), sD = sI + (HP + 1) * 32, zrow = sI + HP * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nci = cin / 16, co0 = (blockIdx.y / nci) * 16, ci0 = (blockIdx.y % nci) * 16;
  const int t0 = (blockIdx.z * 9 + warp) * TPW;
  float acc[TPW][2][4];
#pragma unroll
  for (int k = 0; k < TPW; ++k)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[k][j][0] = acc[k][j][1] = acc[k][j][2] = acc[k][j][3] = 0.f;
  int off[TPW];
#pragma unroll
  for (int k = 0; k < TPW; ++k) {
    const int t = t0 + k;
    off[k] = t % 3 + HX * ((t / 3) % 3 + HY * (t / 9));
  }
  if (tid < 8) reinterpret_cast<uint32_t*>(smem)[HP * 8 + tid] = 0u;
  const int ar = ((lane >> 4) & 1) * 8 + (lane & 7), ah = (lane >> 3) & 1;  // A: position, output-channel half
  const int br = ((lane >> 3) & 1) * 8 + (lane & 7), bh = lane >> 4;        // B: position, input-channel half
  for (int tile = blockIdx.x; tile < ntx * nty * ntz; tile += nchunk) {
    const int x0 = (tile % ntx) * TX, y0 = ((tile / ntx) % nty) * TY, z0 = (tile / (ntx * nty)) * TZ;
    __syncthreads();
    for (int p = tid; p < HP; p += NTHR) {
      const int q = modn(x0 + p % HX - 1, W) + W * (modn(y0 + (p / HX) % HY - 1, H) + H * modn(z0 + p / (HX * HY) - 1, D));
      const __nv_bfloat16* src = in + (size_t)q * cin + ci0;
      cp16(sI + row32(p, 0), src);
      cp16(sI + row32(p, 1), src + 8);
    }
    for (int m = tid; m < NP; m += NTHR) {
      const int x = x0 + m % TX, y = y0 + (m / TX) % TY, z = z0 + m / (TX * TY);
      if (x < W && y < H && z < D) {
        const __nv_bfloat16* src = dout + ((size_t)x + (size_t)W * (y + (size_t)H * z)) * cout + co0;
        cp16(sD + row32(m, 0), src);
        cp16(sD + row32(m, 1), src + 8);
      } else {
        uint4* d = reinterpret_cast<uint4*>(smem + (HP + 1) * 32 + m * 32);
        d[0] = d[1] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    cp_wait_all();
    __syncthreads();
    const bool xin = x0 + br < W;
    for (int s = 0; s < TY * TZ; ++s) {
      const int yy = s % TY, zz = s / TY;
      if (y0 + yy >= H || z0 + zz >= D) continue;
      const int base = br + HX * (yy + HY * zz);
      uint32_t a[4];
      ldm4t(a, sD + row32(s * 16 + ar, ah));
#pragma unroll
      for (int k = 0; k < TPW; ++k) {
        uint32_t b[4];
        ldm4t(b, xin ? sI + row32(base + off[k], bh) : zrow);
        mma_bf16(acc[k][0], a, b);
        mma_bf16(acc[k][1], a, b + 2);
      }
    }
  }
  const int g = lane >> 2, tg = lane & 3;
  float* dw = part + (size_t)blockIdx.x * cout * 27 * cin;
#pragma unroll
  for (int k = 0; k < TPW; ++k)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float* o = dw + ((size_t)(co0 + g + 8 * r) * 27 + t0 + k) * cin + ci0 + j * 8 + tg * 2;
        o[0] = acc[k][j][2 * r];
        o[1] = acc[k][j][2 * r + 1];
      }
}

// Partial dW of the 1x1x1 kernel: block (chunk, 16 output x 16 input channels)
// takes its chunk 512 positions at a time through shared memory, as
// k_wgrad_tile without taps: eight warps take every eighth group of 16
// positions, and their sums are added in warp order (k_conv_wgrad, with its
// 2-byte loads, 105 us for 16 x 16 channels at 64^3).
__global__ void __launch_bounds__(256) k_wgrad_1(const __nv_bfloat16* __restrict__ dout,
                                                 const __nv_bfloat16* __restrict__ in, float* __restrict__ part,
                                                 int npos, int cin, int cout, int chunk) {
  constexpr int NP = 512;
  __shared__ __align__(128) unsigned char buf[2 * NP * 32];
  const uint32_t sI = smem_addr(buf), sD = sI + NP * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nci = cin / 16, co0 = (blockIdx.y / nci) * 16, ci0 = (blockIdx.y % nci) * 16;
  const int pend = min(npos, (int)(blockIdx.x + 1) * chunk);
  const int ar = ((lane >> 4) & 1) * 8 + (lane & 7), ah = (lane >> 3) & 1;
  const int br = ((lane >> 3) & 1) * 8 + (lane & 7), bh = lane >> 4;
  float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
  for (int p0 = blockIdx.x * chunk; p0 < pend; p0 += NP) {
    __syncthreads();
    for (int m = tid; m < NP; m += 256) {
      const int p = p0 + m;
      if (p < pend) {
        cp16(sI + row32(m, 0), in + (size_t)p * cin + ci0);
        cp16(sI + row32(m, 1), in + (size_t)p * cin + ci0 + 8);
        cp16(sD + row32(m, 0), dout + (size_t)p * cout + co0);
        cp16(sD + row32(m, 1), dout + (size_t)p * cout + co0 + 8);
      } else {
        uint4* a = reinterpret_cast<uint4*>(buf + m * 32);
        uint4* b = reinterpret_cast<uint4*>(buf + NP * 32 + m * 32);
        a[0] = a[1] = b[0] = b[1] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    cp_wait_all();
    __syncthreads();
    for (int g = warp; g < NP / 16; g += 8) {
      uint32_t a[4], b[4];
      ldm4t(a, sD + row32(g * 16 + ar, ah));
      ldm4t(b, sI + row32(g * 16 + br, bh));
      mma_bf16(acc[0], a, b);
      mma_bf16(acc[1], a, b + 2);
    }
  }
  __syncthreads();
  float* red = reinterpret_cast<float*>(buf);  // [warp][16 co][16 ci]
  const int g = lane >> 2, tg = lane & 3;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int k = 0; k < 4; ++k) red[warp * 256 + (g + (k >> 1) * 8) * 16 + j * 8 + tg * 2 + (k & 1)] = acc[j][k];
  __syncthreads();
  float v = 0.f;
  for (int w = 0; w < 8; ++w) v += red[w * 256 + tid];
  part[(size_t)blockIdx.x * cout * cin + (size_t)(co0 + tid / 16) * cin + ci0 + tid % 16] = v;
}

// Partial dW[co][t][ci] = sum_p dout[p][co] in[tap(p, t)][ci] over one chunk
// of positions, stored for the chunk (part[chunk][co][t][ci]); one warp per
// (chunk, tap, 16 output channels).  A = dout^T (16 C_out x 16 positions),
// B = shifted input (16 positions x 8 C_in).
template <int NTI>
__global__ void __launch_bounds__(32) k_conv_wgrad(const __nv_bfloat16* __restrict__ dout,
                                                   const __nv_bfloat16* __restrict__ in, float* __restrict__ part,
                                                   int npos, int W, int H, int D, int cin, int cout, int taps,
                                                   int chunk) {
  const int lane = threadIdx.x, g = lane >> 2, tg = lane & 3;
  const int t = blockIdx.y, co0 = blockIdx.z * 16;
  const int pbeg = blockIdx.x * chunk, pend = min(npos, pbeg + chunk);
  float acc[NTI][4];
#pragma unroll
  for (int j = 0; j < NTI; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
  for (int p0 = pbeg; p0 < pend; p0 += 16) {
    // A[m = co][k = position]: a0 (g, 2tg..2tg+1), a1 (g+8, ...), a2 (g, 2tg+8..), a3 (g+8, 2tg+8..)
    int pk[4] = {p0 + tg * 2, p0 + tg * 2 + 1, p0 + tg * 2 + 8, p0 + tg * 2 + 9};
    __nv_bfloat16 da[4], db[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool ok = pk[k] < pend;
      da[k] = ok ? dout[(size_t)pk[k] * cout + co0 + g] : zero;
      db[k] = ok ? dout[(size_t)pk[k] * cout + co0 + g + 8] : zero;
    }
    uint32_t a[4] = {pack2(da[0], da[1]), pack2(db[0], db[1]), pack2(da[2], da[3]), pack2(db[2], db[3])};
    int qk[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) qk[k] = pk[k] < pend ? tap_pos(pk[k], t, taps, W, H, D) : -1;
#pragma unroll
    for (int j = 0; j < NTI; ++j) {
      // B[k = position][n = ci]: b0 rows 2tg, 2tg+1 col g; b1 rows 2tg+8, 2tg+9
      __nv_bfloat16 e[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) e[k] = qk[k] >= 0 ? in[(size_t)qk[k] * cin + j * 8 + g] : zero;
      uint32_t b[2] = {pack2(e[0], e[1]), pack2(e[2], e[3])};
      mma_bf16(acc[j], a, b);
    }
  }
  float* dw = part + (size_t)blockIdx.x * cout * taps * cin;
#pragma unroll
  for (int j = 0; j < NTI; ++j) {
    const int ci = j * 8 + tg * 2;
    dw[((size_t)(co0 + g) * taps + t) * cin + ci] = acc[j][0];
    dw[((size_t)(co0 + g) * taps + t) * cin + ci + 1] = acc[j][1];
    dw[((size_t)(co0 + g + 8) * taps + t) * cin + ci] = acc[j][2];
    dw[((size_t)(co0 + g + 8) * taps + t) * cin + ci + 1] = acc[j][3];
  }
}

// dw[e] += sum over the chunks of part[chunk][e]: eight threads per element
// take every eighth chunk each, in order, and their sums are added in order
// (one thread per element left the sum of 256 chunks to a chain of dependent
// adds in a few blocks: 15 us; now bound by the read of the partials).
__global__ void __launch_bounds__(256) k_wgrad_sum(const float* __restrict__ part, float* __restrict__ dw, int nchunk,
                                                   size_t nw) {
  __shared__ float sp[8][32];
  const size_t e = blockIdx.x * (size_t)32 + threadIdx.x;
  float v = 0.f;
  if (e < nw)
    for (int c = threadIdx.y; c < nchunk; c += 8) v += part[(size_t)c * nw + e];
  sp[threadIdx.y][threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.y == 0 && e < nw) {
    for (int k = 1; k < 8; ++k) v += sp[k][threadIdx.x];
    dw[e] += v;
  }
}

// Weights of the input-gradient convolution: w'[ci][t][co] = w[co][taps-1-t][ci].
__global__ void k_flip_weights(const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ wt, int cout, int cin,
                               int taps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= cout * cin * taps) return;
  const int co = i / (taps * cin), t = (i / cin) % taps, ci = i % cin;
  wt[((size_t)ci * taps + (taps - 1 - t)) * cout + co] = w[i];
}

// db[ch] += sum_p dout[p][ch]: a cluster of 16 blocks takes up to 16 channels;
// a thread adds the positions of its residue class for its V channels (rows of
// 16 bytes, eight in flight per thread: 64 KB per SM cover the latency of the
// memory), the block sums go through distributed shared memory and are added
// in block order, so the result is the same on every run.  16 channels at 64^3:
// one block per channel 223 us, clusters of 8 with 4-byte loads 80 us, with
// 512 threads 17 us.
constexpr int BIAS_CLUSTER = 16, BIAS_THREADS = 1024;
template <int V>
__global__ void __launch_bounds__(BIAS_THREADS) k_bias_grad(const float* __restrict__ dout, float* __restrict__ db,
                                                            int npos, int c) {
  constexpr int COLS = 16 / V, ROWS = BIAS_THREADS / COLS, UNROLL = 8;
  __shared__ float s[ROWS][17];
  __shared__ float tot[16];
  const int tid = threadIdx.x, rank = blockIdx.x % BIAS_CLUSTER, c0 = (blockIdx.x / BIAS_CLUSTER) * 16;
  const int col = (tid % COLS) * V, row = tid / COLS;
  float v[V];
#pragma unroll
  for (int j = 0; j < V; ++j) v[j] = 0.f;
  if (c0 + col < c) {
    const size_t step = (size_t)ROWS * BIAS_CLUSTER;
    size_t p = (size_t)rank * ROWS + row;
    const float* src = dout + c0 + col;
    for (; p + (UNROLL - 1) * step < (size_t)npos; p += UNROLL * step) {
      float t[UNROLL][V];
#pragma unroll
      for (int k = 0; k < UNROLL; ++k) {
        if constexpr (V == 4) *reinterpret_cast<float4*>(t[k]) = *reinterpret_cast<const float4*>(src + (p + k * step) * c);
        else t[k][0] = src[(p + k * step) * c];
      }
#pragma unroll
      for (int k = 0; k < UNROLL; ++k)
#pragma unroll
        for (int j = 0; j < V; ++j) v[j] += t[k][j];
    }
    for (; p < (size_t)npos; p += step)
#pragma unroll
      for (int j = 0; j < V; ++j) v[j] += src[p * c + j];
  }
#pragma unroll
  for (int j = 0; j < V; ++j) s[row][col + j] = v[j];
  __syncthreads();
  // a warp per channel adds the rows in a fixed tree
  const int ch = tid >> 5, lane = tid & 31;
  if (ch < 16) {
    float t = 0.f;
    for (int r = lane; r < ROWS; r += 32) t += s[r][ch];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) tot[ch] = t;
  }
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  cl.sync();
  if (rank == 0 && tid < 16 && c0 + tid < c) {
    float u = 0.f;
    for (int r = 0; r < BIAS_CLUSTER; ++r) u += cl.map_shared_rank(tot, r)[tid];
    db[c0 + tid] += u;
  }
  cl.sync();
}

// dz = dy * (y > 0) (ReLU backward from the stored activation); also to BF16.
__global__ void k_relu_bwd(const float* __restrict__ dy, const __nv_bfloat16* __restrict__ y, float* __restrict__ dz32,
                           __nv_bfloat16* __restrict__ dz16, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float v = __bfloat162float(y[i]) > 0.f ? dy[i] : 0.f;
    if (dz32) dz32[i] = v;
    if (dz16) dz16[i] = __float2bfloat16_rn(v);
  }
}

__global__ void k_cast_bf16(const float* __restrict__ a, __nv_bfloat16* __restrict__ b, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = __float2bfloat16_rn(a[i]);
}

// 2x2x2 mean pooling (channels last) and its adjoint.
template <int VEC>
__global__ void k_pool2(const __nv_bfloat16* __restrict__ in, __nv_bfloat16* __restrict__ out, int S, int c) {
  const int So = S / 2, cv = c / VEC;
  const size_t n = (size_t)So * So * So * cv;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const unsigned p = n >> 32 ? (unsigned)(i / (unsigned)cv) : (unsigned)i / (unsigned)cv;
    const int ch = (int)(i - (size_t)p * cv) * VEC;
    const int x = p % So, y = (p / So) % So, z = p / ((unsigned)So * So);
    float s[VEC];
#pragma unroll
    for (int j = 0; j < VEC; ++j) s[j] = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int xx = 2 * x + (k & 1), yy = 2 * y + ((k >> 1) & 1), zz = 2 * z + (k >> 2);
      const __nv_bfloat16* src = in + ((size_t)xx + (size_t)S * (yy + (size_t)S * zz)) * c + ch;
      if constexpr (VEC == 8) {
        const uint4 q = *reinterpret_cast<const uint4*>(src);
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 f = __bfloat1622float2(h[j]);
          s[2 * j] += f.x;
          s[2 * j + 1] += f.y;
        }
      } else {
        s[0] += __bfloat162float(src[0]);
      }
    }
    if constexpr (VEC == 8) {
      uint4 q;
      __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&q);
#pragma unroll
      for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(0.125f * s[2 * j], 0.125f * s[2 * j + 1]);
      reinterpret_cast<uint4*>(out)[i] = q;
    } else {
      out[i] = __float2bfloat16_rn(0.125f * s[0]);
    }
  }
}

__global__ void k_pool2_bwd(const float* __restrict__ dout, float* __restrict__ din, int S, int c) {
  const size_t n = (size_t)S * S * S * c;
  const int So = S / 2;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int ch = (int)(i % c);
    const size_t p = i / c;
    const int x = (int)(p % S), y = (int)((p / S) % S), z = (int)(p / ((size_t)S * S));
    din[i] += 0.125f * dout[((size_t)(x / 2) + (size_t)So * ((y / 2) + (size_t)So * (z / 2))) * c + ch];
  }
}

// Nearest x2 upsampling of a (So^3, c1) tensor into channels [0, c1) of a
// (2So)^3 tensor with c1 + c2 channels, and the copy of the skip tensor
// (c2 channels) into channels [c1, c1 + c2).
// VEC channels per thread (8 when c1, c2 and the pointers allow 16-byte moves,
// else 1; element-wise at 128^3 x 48 channels: 357 us against the 45 us that
// its bytes take).
template <int VEC>
__global__ void k_up2_concat(const __nv_bfloat16* __restrict__ lo, const __nv_bfloat16* __restrict__ skip,
                             __nv_bfloat16* __restrict__ out, int S, int c1, int c2) {
  const int cv = (c1 + c2) / VEC, So = S / 2;
  const size_t n = (size_t)S * S * S * cv;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const unsigned p = n >> 32 ? (unsigned)(i / (unsigned)cv) : (unsigned)i / (unsigned)cv;
    const int ch = (int)(i - (size_t)p * cv) * VEC;
    const __nv_bfloat16* src;
    if (ch < c1) {
      const unsigned x = p % S, y = (p / S) % S, z = p / ((unsigned)S * S);
      src = lo + ((size_t)(x / 2) + (size_t)So * ((y / 2) + (size_t)So * (z / 2))) * c1 + ch;
    } else {
      src = skip + (size_t)p * c2 + (ch - c1);
    }
    if constexpr (VEC == 8)
      reinterpret_cast<uint4*>(out)[i] = *reinterpret_cast<const uint4*>(src);
    else
      out[i] = *src;
  }
}

// Adjoint: d(lo) = sum of the 8 children of channels [0, c1); d(skip) += channels [c1, c).
__global__ void k_up2_concat_bwd(const float* __restrict__ dout, float* __restrict__ dlo, float* __restrict__ dskip,
                                 int S, int c1, int c2) {
  const int c = c1 + c2, So = S / 2;
  const size_t nlo = (size_t)So * So * So * c1;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nlo; i += (size_t)gridDim.x * blockDim.x) {
    const int ch = (int)(i % c1);
    const size_t p = i / c1;
    const int x = (int)(p % So), y = (int)((p / So) % So), z = (int)(p / ((size_t)So * So));
    float s = 0.f;
    for (int k = 0; k < 8; ++k) {
      const int xx = 2 * x + (k & 1), yy = 2 * y + ((k >> 1) & 1), zz = 2 * z + (k >> 2);
      s += dout[((size_t)xx + (size_t)S * (yy + (size_t)S * zz)) * c + ch];
    }
    dlo[i] = s;
  }
  const size_t nsk = (size_t)S * S * S * c2;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nsk; i += (size_t)gridDim.x * blockDim.x) {
    const size_t p = i / c2;
    dskip[i] += dout[p * c + c1 + (i % c2)];
  }
}

// Masked mean-square error over fluid positions and the 5 Q components of
// pred = base + out[:, 0:5] (out has cout channels); grad w.r.t. out.
__global__ void k_mse(const float* __restrict__ out, const float* __restrict__ base, const float* __restrict__ target,
                      const float* __restrict__ fluid, float* __restrict__ grad, double* __restrict__ loss, int npos,
                      int cout, double inv_count, bool vec) {
  __shared__ double s[256];
  double acc = 0.0;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npos; p += gridDim.x * blockDim.x) {
    const float m = fluid[p];
    if (cout == 16 && vec) {  // the position's gradient row in four 16-byte stores
      float g[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (m > 0.f)
        for (int c = 0; c < 5; ++c) {
          const float d = out[(size_t)p * 16 + c] + base[(size_t)p * 5 + c] - target[(size_t)p * 5 + c];
          const double dd = f32_to_f64(d);
          acc += dd * dd;
          g[c] = (float)(2.0 * inv_count) * d;
        }
      if (grad) {
        float4* o = reinterpret_cast<float4*>(grad + (size_t)p * 16);
        o[0] = make_float4(g[0], g[1], g[2], g[3]);
        o[1] = make_float4(g[4], 0.f, 0.f, 0.f);
        o[2] = o[3] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      continue;
    }
    for (int c = 0; c < cout; ++c) {
      float gv = 0.f;
      if (c < 5 && m > 0.f) {
        const float d = out[(size_t)p * cout + c] + base[(size_t)p * 5 + c] - target[(size_t)p * 5 + c];
        acc += (double)d * d;
        gv = (float)(2.0 * inv_count) * d;
      }
      if (grad) grad[(size_t)p * cout + c] = gv;
    }
  }
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int d = blockDim.x / 2; d > 0; d >>= 1) {
    if (threadIdx.x < d) s[threadIdx.x] += s[threadIdx.x + d];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(loss, s[0] * inv_count);
}

// Cube means of the masked error (one thread per cube and component) and
// their squared sum; then each fluid position's share of the gradient.
__global__ void k_mse_coarse_blocks(const float* __restrict__ out, const float* __restrict__ base,
                                    const float* __restrict__ target, const float* __restrict__ fluid,
                                    float* __restrict__ blk, double* __restrict__ loss, int S, int b, int cout,
                                    double inv_count) {
  __shared__ double s[256];
  const int nc = S / b;
  const int ncube = nc * nc * nc;
  double acc = 0.0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ncube * 5; t += gridDim.x * blockDim.x) {
    const int cube = t / 5, c = t % 5;
    const int cx = cube % nc, cy = (cube / nc) % nc, cz = cube / (nc * nc);
    double sum = 0.0;
    for (int dz = 0; dz < b; ++dz)
      for (int dy = 0; dy < b; ++dy)
        for (int dx = 0; dx < b; ++dx) {
          const size_t p = (size_t)(cx * b + dx) + (size_t)S * ((cy * b + dy) + (size_t)S * (cz * b + dz));
          if (fluid[p] > 0.f) sum += (double)(out[p * cout + c] + base[p * 5 + c] - target[p * 5 + c]);
        }
    const double e = sum / ((double)b * b * b);
    blk[t] = (float)e;
    acc += e * e;
  }
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int d = blockDim.x / 2; d > 0; d >>= 1) {
    if (threadIdx.x < d) s[threadIdx.x] += s[threadIdx.x + d];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(loss, s[0] * inv_count);
}

__global__ void k_mse_coarse_grad(const float* __restrict__ fluid, const float* __restrict__ blk,
                                  float* __restrict__ grad, int S, int b, int cout, double inv_count) {
  const int nc = S / b;
  const size_t npos = (size_t)S * S * S;
  const float g = (float)(2.0 * inv_count / ((double)b * b * b));
  for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < npos; p += (size_t)gridDim.x * blockDim.x) {
    if (!(fluid[p] > 0.f)) continue;
    const int x = (int)(p % S), y = (int)((p / S) % S), z = (int)(p / ((size_t)S * S));
    const int cube = x / b + nc * (y / b + nc * (z / b));
    for (int c = 0; c < 5; ++c) grad[p * cout + c] += g * blk[cube * 5 + c];
  }
}

// Adam on FP32 masters with a BF16 working copy.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       __nv_bfloat16* __restrict__ p16, size_t n, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (p16) p16[i] = __float2bfloat16_rn(pi);
  }
}

// Network input (channels last, cpad >= 9 channels, the rest zero):
// [solid indicator, Q xx,xy,xz,yy,yz, R/32, p/64, 20 w] from FP64 SoA fields.
// vec (cpad == 16, x16 and base 16-byte aligned): the position's 32 bytes in two
// stores, and the base of the block's 256 positions through shared memory in
// whole lines.
__global__ void __launch_bounds__(256) k_pack_input(const double* __restrict__ solid, const double* __restrict__ q,
                                                    float r, float pitch, float w, __nv_bfloat16* __restrict__ x16,
                                                    float* __restrict__ base, float* __restrict__ fluid,
                                                    double* __restrict__ nfluid, int npos, int cpad, bool vec) {
  __shared__ __align__(16) float sb[256 * 5];
  int cnt = 0;
  for (int p0 = blockIdx.x * 256; p0 < npos; p0 += gridDim.x * 256) {
    const int p = p0 + threadIdx.x;
    const bool in = p < npos;
    float v[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, r / 32.f, pitch / 64.f, 20.f * w};
    if (in) {
      // solid < 0, >= 0 by the bits (an FP64 comparison is a slot of the FP64 pipe;
      // NaN is neither)
      const long long sbits = __double_as_longlong(solid[p]);
      const bool nan = (sbits & 0x7fffffffffffffffll) > 0x7ff0000000000000ll, zero = (sbits << 1) == 0;
      cnt += !nan && !zero && sbits < 0;
      const bool sol = !nan && (zero || sbits > 0);
      v[0] = sol ? 1.f : 0.f;
      for (int c = 0; c < 5; ++c) v[1 + c] = (float)q[(size_t)c * npos + p];
      if (vec) {
        __nv_bfloat162 h[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          h[k] = __floats2bfloat162_rn(2 * k < 9 ? v[2 * k] : 0.f, 2 * k + 1 < 9 ? v[2 * k + 1] : 0.f);
        uint4* d = reinterpret_cast<uint4*>(x16 + (size_t)p * 16);
        d[0] = *reinterpret_cast<uint4*>(h);
        d[1] = *reinterpret_cast<uint4*>(h + 4);
      } else {
        for (int c = 0; c < cpad; ++c) x16[(size_t)p * cpad + c] = __float2bfloat16_rn(c < 9 ? v[c] : 0.f);
        if (base)
          for (int c = 0; c < 5; ++c) base[(size_t)p * 5 + c] = v[1 + c];
      }
      if (fluid) fluid[p] = sol ? 0.f : 1.f;
    }
    if (vec && base) {
      __syncthreads();
      for (int c = 0; c < 5; ++c) sb[threadIdx.x * 5 + c] = v[1 + c];
      __syncthreads();
      const int n = min(256, npos - p0) * 5;
      float* dst = base + (size_t)p0 * 5;
      for (int k = threadIdx.x * 4; k < n; k += 1024) {
        if (k + 4 <= n) *reinterpret_cast<float4*>(dst + k) = *reinterpret_cast<const float4*>(sb + k);
        else
          for (int j = k; j < n; ++j) dst[j] = sb[j];
      }
    }
  }
  if (nfluid) {
    // one FP64 atomic per block of a grid that fits the GPU (one per warp, all
    // to one address, was the kernel's time: 131 us at 128^3 for 32 us of bytes)
    __shared__ int sc[8];
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0) sc[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
      int t = 0;
      for (int k = 0; k < 8; ++k) t += sc[k];
      if (t) atomicAdd(nfluid, (double)t);
    }
  }
}

// SoA FP64 [5][npos] -> channels-last FP32 (npos x 5).
__global__ void k_from_soa(const double* __restrict__ q, float* __restrict__ a, int npos) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npos; p += gridDim.x * blockDim.x)
    for (int c = 0; c < 5; ++c) a[(size_t)p * 5 + c] = (float)q[(size_t)c * npos + p];
}

// Channels-last (npos, 5) FP32 -> SoA FP64 [5][npos].
__global__ void k_to_soa(const float* __restrict__ a, const float* __restrict__ base, double* __restrict__ q, int npos,
                         int cout) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npos; p += gridDim.x * blockDim.x)
    for (int c = 0; c < 5; ++c) {
      const double v = f32_to_f64(a[(size_t)p * cout + c]);
      q[(size_t)c * npos + p] = base ? v + f32_to_f64(base[(size_t)p * 5 + c]) : v + 0.0;
    }
}

// Trilinear x2 upsampling of a periodic SoA field [c][S^3] (cell-centred: the
// fine node 2i + 1/2 +- 1/4 of coarse node i) to [c][(2S)^3].
__global__ void k_trilinear2(const double* __restrict__ a, double* __restrict__ b, int S, int c) {
  const int F = 2 * S;
  const size_t n = (size_t)F * F * F;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n * c; i += (size_t)gridDim.x * blockDim.x) {
    const int ch = (int)(i / n);
    const size_t p = i % n;
    const int X = (int)(p % F), Y = (int)((p / F) % F), Z = (int)(p / ((size_t)F * F));
    int i0[3], i1[3];
    float t[3];
    const int P[3] = {X, Y, Z};
    for (int k = 0; k < 3; ++k) {
      // fine coordinate in coarse units: (P + 0.5)/2 - 0.5
      const float u = 0.5f * (P[k] + 0.5f) - 0.5f;
      const int f = (int)floorf(u);
      t[k] = u - f;
      i0[k] = wrapi(f, S);
      i1[k] = wrapi(f + 1, S);
    }
    double v = 0.0;
    for (int k = 0; k < 8; ++k) {
      const int xx = (k & 1) ? i1[0] : i0[0], yy = (k & 2) ? i1[1] : i0[1], zz = (k & 4) ? i1[2] : i0[2];
      const double wgt = ((k & 1) ? t[0] : 1 - t[0]) * ((k & 2) ? t[1] : 1 - t[1]) * ((k & 4) ? t[2] : 1 - t[2]);
      v += wgt * a[(size_t)ch * S * S * S + xx + (size_t)S * (yy + (size_t)S * zz)];
    }
    b[i] = v;
  }
}

static inline int grid_for(size_t n, int bs = 256) {
  size_t g = (n + bs - 1) / bs;
  return (int)(g > 65535 * 8 ? 65535 * 8 : (g < 1 ? 1 : g));
}

// The status of a runtime call that may have failed; its error is taken, so that
// the next call does not report it again.
static inline int taken(cudaError_t e) {
  if (e == cudaSuccess) return LC_NN_OK;
  cudaGetLastError();
  return LC_NN_ERR_CUDA;
}

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

template <int NT, int MT, int NW, int TX, int TY, int TZ>
static int launch_conv_tile(const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias, float* out32,
                            __nv_bfloat16* out16, int W, int H, int D, int cin, int cout, int relu, cudaStream_t s) {
  constexpr int smem = ((TX + 2) * (TY + 2) * (TZ + 2) + 27 * NT * 8) * 32;
  auto* fn = k_conv_tile<NT, MT, NW, TX, TY, TZ>;
  if (taken(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != LC_NN_OK) return LC_NN_ERR_CUDA;
  const int ntx = (W + TX - 1) / TX, nty = (H + TY - 1) / TY, ntz = (D + TZ - 1) / TZ;
  fn<<<dim3((unsigned)ntx * nty * ntz, cout / (NT * 8)), 32 * NW, smem, s>>>(in, w, bias, out32, out16, W, H, D, cin,
                                                                            cout, relu, ntx, nty);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

// Boxes of 16 x 8 x 4 positions and all output channels per block while they
// fill the GPU (152 SMs x 2 blocks), else boxes of 128 positions (16 x 4 x 2, or
// 8 x 4 x 4 where the tensor is no wider than 8) with the output channels split
// in groups of 16 over the blocks.
static int conv_tiled(const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias, float* out32,
                      __nv_bfloat16* out16, int W, int H, int D, int cin, int cout, int relu, cudaStream_t s) {
  if (cout != 8 && cout % 16) return LC_NN_ERR_ARG;
  const long long big = (long long)((W + 15) / 16) * ((H + 7) / 8) * ((D + 3) / 4);
#define LCNN_BIG(NT) return launch_conv_tile<NT, 4, 8, 16, 8, 4>(in, w, bias, out32, out16, W, H, D, cin, cout, relu, s)
  if (big >= 256) {
    switch (cout / 8) {
      case 1: LCNN_BIG(1);
      case 2: LCNN_BIG(2);
      case 4: case 8: LCNN_BIG(4);
      case 6: LCNN_BIG(6);
      case 10: LCNN_BIG(5);
      default: return LC_NN_ERR_ARG;
    }
  }
#undef LCNN_BIG
  if (W > 8) {
    if (cout == 8) return launch_conv_tile<1, 2, 4, 16, 4, 2>(in, w, bias, out32, out16, W, H, D, cin, cout, relu, s);
    return launch_conv_tile<2, 2, 4, 16, 4, 2>(in, w, bias, out32, out16, W, H, D, cin, cout, relu, s);
  }
  if (cout == 8) return launch_conv_tile<1, 2, 4, 8, 4, 4>(in, w, bias, out32, out16, W, H, D, cin, cout, relu, s);
  return launch_conv_tile<2, 2, 4, 8, 4, 4>(in, w, bias, out32, out16, W, H, D, cin, cout, relu, s);
}

static int launch_bias_grad(const float* dout, float* db, int npos, int c, cudaStream_t s) {
  auto* fn = c % 4 == 0 && aligned16(dout) ? k_bias_grad<4> : k_bias_grad<1>;
  if (taken(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != LC_NN_OK) return LC_NN_ERR_CUDA;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  cfg.gridDim = dim3((c + 15) / 16 * BIAS_CLUSTER);
  cfg.blockDim = dim3(BIAS_THREADS);
  cfg.stream = s;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = BIAS_CLUSTER;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return taken(cudaLaunchKernelEx(&cfg, fn, dout, db, npos, c));
}

template <int TPW, int TY, int TZ>
static int launch_wgrad_tile(const __nv_bfloat16* dout, const __nv_bfloat16* in, float* part, int W, int H, int D,
                             int cin, int cout, int nchunk, cudaStream_t s) {
  constexpr int smem = (18 * (TY + 2) * (TZ + 2) + 1 + 16 * TY * TZ) * 32;
  auto* fn = k_wgrad_tile<TPW, TY, TZ>;
  if (taken(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != LC_NN_OK) return LC_NN_ERR_CUDA;
  fn<<<dim3(nchunk, (cout / 16) * (cin / 16), 3 / TPW), 288, smem, s>>>(
      dout, in, part, W, H, D, cin, cout, (W + 15) / 16, (H + TY - 1) / TY, (D + TZ - 1) / TZ, nchunk);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

}  // namespace lcnn

using namespace lcnn;

extern "C" {

int lc_nn_conv3d_fwd(const void* in, const void* w, const float* bias, float* out32, void* out16, int W, int H, int D,
                     int cin, int cout, int taps, int relu, void* stream) {
  if (!in || !w || (!out32 && !out16) || cin % 16 || cout % 8 || cout > 80 || (taps != 27 && taps != 1) || W < 1 ||
      H < 1 || D < 1)
    return LC_NN_ERR_ARG;
  const int npos = W * H * D;
  const dim3 grid((npos + 63) / 64);
  cudaStream_t s = (cudaStream_t)stream;
  auto* a = (const __nv_bfloat16*)in;
  auto* b = (const __nv_bfloat16*)w;
  auto* o16 = (__nv_bfloat16*)out16;
  // 3x3x3: input tiles in shared memory (16-byte copies, so aligned tensors);
  // 1x1x1 has no taps to share, and unaligned tensors take 4-byte loads
  if (taps == 27 && aligned16(in) && aligned16(w)) return conv_tiled(a, b, bias, out32, o16, W, H, D, cin, cout, relu, s);
  switch (cout / 8) {
    case 1: k_conv_fwd<1><<<grid, 128, 0, s>>>(a, b, bias, out32, o16, npos, W, H, D, cin, taps, relu); break;
    case 2: k_conv_fwd<2><<<grid, 128, 0, s>>>(a, b, bias, out32, o16, npos, W, H, D, cin, taps, relu); break;
    case 4: k_conv_fwd<4><<<grid, 128, 0, s>>>(a, b, bias, out32, o16, npos, W, H, D, cin, taps, relu); break;
    case 6: k_conv_fwd<6><<<grid, 128, 0, s>>>(a, b, bias, out32, o16, npos, W, H, D, cin, taps, relu); break;
    case 8: k_conv_fwd<8><<<grid, 128, 0, s>>>(a, b, bias, out32, o16, npos, W, H, D, cin, taps, relu); break;
    case 10: k_conv_fwd<10><<<grid, 128, 0, s>>>(a, b, bias, out32, o16, npos, W, H, D, cin, taps, relu); break;
    default: return LC_NN_ERR_ARG;
  }
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_conv3d_dgrad(const void* dout, const void* w, void* wt_scratch, float* din32, void* din16, int W, int H,
                       int D, int cin, int cout, int taps, void* stream) {
  if (!dout || !w || !wt_scratch || cout % 16 || cin % 8) return LC_NN_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const int n = cout * cin * taps;
  k_flip_weights<<<(n + 255) / 256, 256, 0, s>>>((const __nv_bfloat16*)w, (__nv_bfloat16*)wt_scratch, cout, cin, taps);
  if (cudaGetLastError() != cudaSuccess) return LC_NN_ERR_CUDA;
  return lc_nn_conv3d_fwd(dout, wt_scratch, nullptr, din32, din16, W, H, D, cout, cin, taps, 0, stream);
}

// Positions per chunk of the weight gradient: 1024, more when that would give
// more than 256 chunks (a multiple of 16, the MMA's K).
static int wgrad_chunk(int npos) {
  int chunk = 1024;
  while ((npos + chunk - 1) / chunk > 256) chunk *= 2;
  return chunk;
}

size_t lc_nn_wgrad_partial_floats(int W, int H, int D, int cin, int cout, int taps) {
  const int npos = W * H * D;
  if (npos <= 0) return 0;
  const int nchunk = (npos + wgrad_chunk(npos) - 1) / wgrad_chunk(npos);
  return (size_t)nchunk * cout * taps * cin;
}

int lc_nn_conv3d_wgrad(const void* dout, const void* in, float* dw, float* partial, int W, int H, int D, int cin,
                       int cout, int taps, void* stream) {
  if (!dout || !in || !dw || !partial || cout % 16 || cin % 8 || cin > 80) return LC_NN_ERR_ARG;
  const int npos = W * H * D;
  if (npos <= 0) return LC_NN_ERR_ARG;
  if (cin != 8 && cin != 16 && cin != 32 && cin != 48 && cin != 80) return LC_NN_ERR_ARG;  // the same for every path
  const int chunk = wgrad_chunk(npos);
  const int nchunk = (npos + chunk - 1) / chunk;
  const dim3 grid(nchunk, taps, cout / 16);
  cudaStream_t s = (cudaStream_t)stream;
  auto* a = (const __nv_bfloat16*)dout;
  auto* b = (const __nv_bfloat16*)in;
  const size_t nw = (size_t)cout * taps * cin;
  const dim3 sblk(32, 8);
  const unsigned sgrid = (unsigned)((nw + 31) / 32);
  if (taps == 27 && cin % 16 == 0 && aligned16(dout) && aligned16(in)) {
    // the boxes of the chunks are summed in box order; the taps of one chunk
    // go to three blocks where the chunks alone leave SMs idle
    const int rc = nchunk * (cout / 16) * (cin / 16) >= 256
                       ? launch_wgrad_tile<3, 8, 4>(a, b, partial, W, H, D, cin, cout, nchunk, s)
                       : launch_wgrad_tile<1, 4, 4>(a, b, partial, W, H, D, cin, cout, nchunk, s);
    if (rc != LC_NN_OK) return rc;
    k_wgrad_sum<<<sgrid, sblk, 0, s>>>(partial, dw, nchunk, nw);
    return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
  }
  if (taps == 1 && cin % 16 == 0 && aligned16(dout) && aligned16(in)) {
    k_wgrad_1<<<dim3(nchunk, (cout / 16) * (cin / 16)), 256, 0, s>>>(a, b, partial, npos, cin, cout, chunk);
    k_wgrad_sum<<<sgrid, sblk, 0, s>>>(partial, dw, nchunk, nw);
    return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
  }
  switch (cin / 8) {
    case 1: k_conv_wgrad<1><<<grid, 32, 0, s>>>(a, b, partial, npos, W, H, D, cin, cout, taps, chunk); break;
    case 2: k_conv_wgrad<2><<<grid, 32, 0, s>>>(a, b, partial, npos, W, H, D, cin, cout, taps, chunk); break;
    case 4: k_conv_wgrad<4><<<grid, 32, 0, s>>>(a, b, partial, npos, W, H, D, cin, cout, taps, chunk); break;
    case 6: k_conv_wgrad<6><<<grid, 32, 0, s>>>(a, b, partial, npos, W, H, D, cin, cout, taps, chunk); break;
    case 10: k_conv_wgrad<10><<<grid, 32, 0, s>>>(a, b, partial, npos, W, H, D, cin, cout, taps, chunk); break;
    default: return LC_NN_ERR_ARG;
  }
  k_wgrad_sum<<<sgrid, sblk, 0, s>>>(partial, dw, nchunk, nw);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_bias_grad(const float* dout, float* db, int npos, int c, void* stream) {
  return launch_bias_grad(dout, db, npos, c, (cudaStream_t)stream);
}

int lc_nn_relu_bwd(const float* dy, const void* y, float* dz32, void* dz16, size_t n, void* stream) {
  k_relu_bwd<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(dy, (const __nv_bfloat16*)y, dz32, (__nv_bfloat16*)dz16, n);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_cast_bf16(const float* a, void* b, size_t n, void* stream) {
  k_cast_bf16<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(a, (__nv_bfloat16*)b, n);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_pool2(const void* in, void* out, int S, int c, void* stream) {
  if (S % 2) return LC_NN_ERR_ARG;
  const size_t n = (size_t)(S / 2) * (S / 2) * (S / 2) * c;
  if (c % 8 == 0 && aligned16(in) && aligned16(out))
    k_pool2<8><<<grid_for(n / 8), 256, 0, (cudaStream_t)stream>>>((const __nv_bfloat16*)in, (__nv_bfloat16*)out, S, c);
  else
    k_pool2<1><<<grid_for(n), 256, 0, (cudaStream_t)stream>>>((const __nv_bfloat16*)in, (__nv_bfloat16*)out, S, c);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_pool2_bwd(const float* dout, float* din, int S, int c, void* stream) {
  k_pool2_bwd<<<grid_for((size_t)S * S * S * c), 256, 0, (cudaStream_t)stream>>>(dout, din, S, c);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_up2_concat(const void* lo, const void* skip, void* out, int S, int c1, int c2, void* stream) {
  if (S % 2) return LC_NN_ERR_ARG;
  const size_t n = (size_t)S * S * S * (c1 + c2);
  if (c1 % 8 == 0 && c2 % 8 == 0 && aligned16(lo) && aligned16(skip) && aligned16(out))
    k_up2_concat<8><<<grid_for(n / 8), 256, 0, (cudaStream_t)stream>>>(
        (const __nv_bfloat16*)lo, (const __nv_bfloat16*)skip, (__nv_bfloat16*)out, S, c1, c2);
  else
    k_up2_concat<1><<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(
        (const __nv_bfloat16*)lo, (const __nv_bfloat16*)skip, (__nv_bfloat16*)out, S, c1, c2);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_up2_concat_bwd(const float* dout, float* dlo, float* dskip, int S, int c1, int c2, void* stream) {
  k_up2_concat_bwd<<<grid_for((size_t)S * S * S * c2), 256, 0, (cudaStream_t)stream>>>(dout, dlo, dskip, S, c1, c2);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_mse(const float* out, const float* base, const float* target, const float* fluid, float* grad,
              double* loss, int npos, int cout, double inv_count, void* stream) {
  k_mse<<<grid_for(npos), 256, 0, (cudaStream_t)stream>>>(out, base, target, fluid, grad, loss, npos, cout, inv_count,
                                                            aligned16(grad));
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_mse_coarse(const float* out, const float* base, const float* target, const float* fluid, float* grad,
                     double* loss, float* blk, int S, int b, int cout, double inv_count, void* stream) {
  if (b < 1 || S < 1 || S % b != 0 || cout < 5 || !blk || !loss) return LC_NN_ERR_ARG;
  const int nc = S / b;
  cudaStream_t st = (cudaStream_t)stream;
  k_mse_coarse_blocks<<<grid_for((size_t)nc * nc * nc * 5), 256, 0, st>>>(out, base, target, fluid, blk, loss, S, b,
                                                                           cout, inv_count);
  if (grad) k_mse_coarse_grad<<<grid_for((size_t)S * S * S), 256, 0, st>>>(fluid, blk, grad, S, b, cout, inv_count);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_adam(float* p, const float* g, float* m, float* v, void* p16, size_t n, float lr, float b1, float b2,
               float eps, int step, void* stream) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_adam<<<grid_for(n), 256, 0, (cudaStream_t)stream>>>(p, g, m, v, (__nv_bfloat16*)p16, n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_pack_input(const double* solid, const double* q, double R, double pitch, double w, void* x16, float* base,
                     float* fluid, double* nfluid, int npos, int cpad, void* stream) {
  if (cpad < 9) return LC_NN_ERR_ARG;
  k_pack_input<<<std::min(grid_for(npos), 8 * 152), 256, 0, (cudaStream_t)stream>>>(solid, q, (float)R, (float)pitch, (float)w,
                                                                   (__nv_bfloat16*)x16, base, fluid, nfluid, npos, cpad,
                                                                   cpad == 16 && aligned16(x16) && aligned16(base));
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_from_soa(const double* q, float* a, int npos, void* stream) {
  k_from_soa<<<grid_for(npos), 256, 0, (cudaStream_t)stream>>>(q, a, npos);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_to_soa(const float* a, const float* base, double* q, int npos, int cout, void* stream) {
  k_to_soa<<<grid_for(npos), 256, 0, (cudaStream_t)stream>>>(a, base, q, npos, cout);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

int lc_nn_trilinear2(const double* a, double* b, int S, int c, void* stream) {
  k_trilinear2<<<grid_for((size_t)8 * S * S * S * c), 256, 0, (cudaStream_t)stream>>>(a, b, S, c);
  return cudaGetLastError() == cudaSuccess ? LC_NN_OK : LC_NN_ERR_CUDA;
}

}  // extern "C"
