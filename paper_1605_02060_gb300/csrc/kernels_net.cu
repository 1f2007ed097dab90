// Kernels of the learned warm start: a small 3D convolutional encoder-decoder that maps a
// template/target mask pair to an initial velocity field, trained and evaluated entirely here.
//
// Layout: activations [B][C][n][n][n] float32 (x fastest); weights [Co][Ci][k^3] (k = 3 or 1)
// stored bf16 for the forward and data-gradient products (FP32 master copy for the optimiser),
// all products accumulated in FP32.  3x3x3 convolutions use zero padding 1.
//
//   conv_fwd   y[b,co,v] = bias[co] + sum_ci sum_t w[co,ci,t] x[b,ci,v+o(t)]   (+ ReLU)
//   conv_dgrad dx[b,ci,v] = sum_co sum_t w[co,ci,t] dy[b,co,v-o(t)]  (= conv_fwd with the
//              transposed, flipped kernel, since o(26-t) = -o(t))
//   conv_wgrad dw[co,ci,t] += sum_b sum_v dy[b,co,v] x[b,ci,v+o(t)],  db[co] += sum dy[b,co,v]
//              (fixed-order partial sums in caller scratch: the same bits on every run)
// plus 2x average pooling, 2x nearest upsampling, channel concatenation, ReLU backward, the MSE
// loss and Adam.  Convolutions whose input channels come in groups of 16 run on the tensor cores
// (kernels_conv_tc.cu); the others (the 2-channel network input, the 3-channel head gradient)
// here: 8x8x4 output voxels x 16 output channels per block, input channels staged 8 at a time
// with a one-voxel halo in shared memory.
#include <cuda_bf16.h>

#include "kernels.h"

namespace lddmm {

namespace {

constexpr int BX = 8, BY = 8, BZ = 4, NTV = BX * BY * BZ;   // 256 voxels per block
constexpr int CT = 16;                                      // output channels per block
constexpr int CC = 8;                                       // input channels per stage
constexpr int HXn = BX + 2, HYn = BY + 2, HZn = BZ + 2, HV = HXn * HYn * HZn;

__device__ __forceinline__ float xval(const float* __restrict__ x, int n, int gx, int gy, int gz) {
  return (gx >= 0 && gx < n && gy >= 0 && gy < n && gz >= 0 && gz < n)
             ? __ldg(x + ((size_t)gz * n + gy) * n + gx)
             : 0.f;
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// Forward convolution (also the data gradient with transposed weights).
// grid: (tiles of 8x8x4, ceil(Co/16), B); block: 256 threads, one output voxel each.
__global__ void __launch_bounds__(NTV) k_conv_fwd(const float* __restrict__ x,
                                                  const __nv_bfloat16* __restrict__ w,
                                                  const float* __restrict__ bias,
                                                  float* __restrict__ y, int Ci, int Co, int n,
                                                  int ks, int relu, int accumulate) {
  __shared__ float xs[CC][HV];
  __shared__ __align__(16) float ws[CC][27][CT];
  const int tid = threadIdx.x;
  const int ntx = (n + BX - 1) / BX, nty = (n + BY - 1) / BY;
  const int tile = blockIdx.x;
  const int tx0 = (tile % ntx) * BX, ty0 = ((tile / ntx) % nty) * BY, tz0 = (tile / (ntx * nty)) * BZ;
  const int co0 = blockIdx.y * CT, b = blockIdx.z;
  const int lx = tid % BX, ly = (tid / BX) % BY, lz = tid / (BX * BY);
  const int gx = tx0 + lx, gy = ty0 + ly, gz = tz0 + lz;
  const size_t nv = (size_t)n * n * n;
  const int taps = ks * ks * ks, pad = ks / 2;
  float acc[CT];
#pragma unroll
  for (int c = 0; c < CT; ++c) acc[c] = 0.f;
  for (int ci0 = 0; ci0 < Ci; ci0 += CC) {
    const int cc = min(CC, Ci - ci0);
    // input tile (with halo) for cc channels
    for (int i = tid; i < cc * HV; i += NTV) {
      const int c = i / HV, h = i % HV;
      const int hx = h % HXn, hy = (h / HXn) % HYn, hz = h / (HXn * HYn);
      xs[c][h] = xval(x + ((size_t)b * Ci + ci0 + c) * nv, n, tx0 + hx - 1, ty0 + hy - 1, tz0 + hz - 1);
    }
    // weights [c][t][co] as float
    for (int i = tid; i < cc * taps * CT; i += NTV) {
      const int co = i % CT, t = (i / CT) % taps, c = i / (CT * taps);
      const int gco = co0 + co;
      ws[c][t][co] = gco < Co ? __bfloat162float(w[((size_t)gco * Ci + ci0 + c) * taps + t]) : 0.f;
    }
    __syncthreads();
    for (int c = 0; c < cc; ++c) {
      for (int t = 0; t < taps; ++t) {
        int ox, oy, oz;
        if (ks == 3) { ox = t % 3 - 1; oy = (t / 3) % 3 - 1; oz = t / 9 - 1; }
        else { ox = oy = oz = 0; }
        const float xv = xs[c][((lz + 1 + oz) * HYn + (ly + 1 + oy)) * HXn + (lx + 1 + ox)];
        const float4* w4 = reinterpret_cast<const float4*>(&ws[c][t][0]);
#pragma unroll
        for (int q = 0; q < CT / 4; ++q) {
          const float4 wv = w4[q];
          acc[4 * q] = fmaf(wv.x, xv, acc[4 * q]);
          acc[4 * q + 1] = fmaf(wv.y, xv, acc[4 * q + 1]);
          acc[4 * q + 2] = fmaf(wv.z, xv, acc[4 * q + 2]);
          acc[4 * q + 3] = fmaf(wv.w, xv, acc[4 * q + 3]);
        }
      }
    }
    __syncthreads();
  }
  (void)pad;
  if (gx < n && gy < n && gz < n) {
    const size_t v = ((size_t)gz * n + gy) * n + gx;
#pragma unroll
    for (int c = 0; c < CT; ++c) {
      const int co = co0 + c;
      if (co >= Co) break;
      float r = acc[c] + (bias ? bias[co] : 0.f);
      float* o = y + ((size_t)b * Co + co) * nv + v;
      if (accumulate) r += *o;
      if (relu) r = fmaxf(r, 0.f);
      *o = r;
    }
  }
}

// wT[ci][co][t'] = w[co][ci][taps-1-t'] (bf16): the data-gradient kernel in forward form.
__global__ void k_transpose_flip(const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ wT,
                                 int Ci, int Co, int taps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Ci * Co * taps) return;
  const int t = i % taps, co = (i / taps) % Co, ci = i / (taps * Co);
  wT[i] = w[((size_t)co * Ci + ci) * taps + (taps - 1 - t)];
}

// Weight gradient, deterministic.  dw[co][ci][t] is a product of Co x B n^3 by B n^3 x 27 Ci in
// FP32 (274 GFLOP in a training step at 64^3, batch 8), so the FP32 pipes bound it and everything
// else has to stay off their issue slots.  A block owns 16 output channels x CIT input channels
// and the voxel tiles (units) g, g + G, ...; it stages a unit's x (with halo, [voxel][ci], rows
// of CIT + 1 words: conflict free both ways) and dy ([voxel][16 co], 16-byte quads swizzled by
// voxel) in shared memory by 4-byte asynchronous copies into two buffers, the next unit's under
// the products of this one.  A thread owns one input channel, one dz, 8 output channels and one
// of the KS slices of the tile's rows: it walks its rows in x with a 3 x 3 window of x in
// registers, so a voxel costs 3 + 2 shared loads for 72 FMAs.  One block of 12 warps per SM: the
// 72 sums want 167 registers.  The step's 15 weight gradients take 7.6 ms (36 TFLOP/s); one
// (co, tap) per thread with two shared loads per FMA took 57.3 ms, this kernel with three blocks
// of 6 warps at 96 registers (spilled sums) 14.3 ms, with two and loads through registers
// 10.3 ms.  Packed fma.rn.f32x2 gains nothing (7.7 ms).
// Partial sums part[g][co][ci][t] (and partb[g][co], from the blocks of the first input
// channels) are added over g in a fixed order by k_wgrad_reduce: no floating-point atomics, the
// same bits on every run.
constexpr int WG_NT = 384, WG_TV = 256;

struct WgTile {
  int tx, ty, tz;      // voxels of a unit (tx * ty * tz <= WG_TV)
  int ntx, nty, ntz;   // units of a sample along each axis
};

// 4 bytes to shared memory, asynchronously; zeros when !in (the address is then not read)
__device__ __forceinline__ void cp4(float* dst, const float* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(in ? 4 : 0)
               : "memory");
}

template <int CIT>
__global__ void __launch_bounds__(WG_NT, 1) k_wgrad3(const float* __restrict__ x,
                                                     const float* __restrict__ dy,
                                                     float* __restrict__ part,
                                                     float* __restrict__ partb, int B, int Ci,
                                                     int Co, int n, WgTile tl, int G) {
  constexpr int KS = WG_NT / (6 * CIT), XS = CIT + 1, NW = WG_NT / 32;
  extern __shared__ __align__(16) float wg_smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ci = tid % CIT, cog = (tid / CIT) & 1, dz = (tid / (2 * CIT)) % 3, ks = tid / (6 * CIT);
  const int nci = (Ci + CIT - 1) / CIT;
  const int ci0 = (blockIdx.y % nci) * CIT, co0 = (blockIdx.y / nci) * 16;
  const int HX = tl.tx + 2, HY = tl.ty + 2, HZ = tl.tz + 2, HXY = HX * HY;
  const int rows = tl.ty * tl.tz, TV = rows * tl.tx;
  const int tiles = tl.ntx * tl.nty * tl.ntz;
  const size_t nv = (size_t)n * n * n;
  // two buffers of dy [WG_TV][16] (quads swizzled) and x [(tz+2)(ty+2)(tx+2)][XS]
  const int bufw = (WG_TV * 16 + HXY * HZ * XS + 3) & ~3;
  const bool bias = partb && ci0 == 0;
  float bsum = 0.f;                           // channel tid % 16, voxels tid / 16, + NT / 16, ...
  float s[8][9];
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int t = 0; t < 9; ++t) s[c][t] = 0.f;
  auto stage = [&](int u, float* dys) {
    float* xs = dys + WG_TV * 16;
    const int b = u / tiles, tile = u - b * tiles;
    const int tx0 = (tile % tl.ntx) * tl.tx, ty0 = ((tile / tl.ntx) % tl.nty) * tl.ty,
              tz0 = (tile / (tl.ntx * tl.nty)) * tl.tz;
    // Warp w of the 12 takes the channels w % CG, + CG, ... and the positions of its third (or
    // sixth) of the tile; a lane's position is decoded once for all channels and planes.  The
    // addresses are clamped into the tensor, what lies outside the grid arrives as zero.
    constexpr int CG = CIT < 4 ? CIT : 4, PG = NW / CG;
    const float* xb = x + ((size_t)b * Ci + ci0) * nv;
    const int cw = warp % CG, pw = (warp / CG) * 32 + lane;
    const int cmax = Ci - 1 - ci0;
    for (int e = pw; e < HXY; e += PG * 32) {
      const int hy = e / HX, hx = e - hy * HX;
      const int gx = tx0 + hx - 1, gy = ty0 + hy - 1;
      const bool inxy = gx >= 0 && gx < n && gy >= 0 && gy < n;
      const int oxy = inxy ? gy * n + gx : 0;
      float* d = xs + e * XS + cw;
      for (int hz = 0; hz < HZ; ++hz, d += HXY * XS) {
        const int gz = tz0 + hz - 1;
        const bool in = inxy && gz >= 0 && gz < n;
        const float* p = xb + (size_t)(in ? gz : 0) * n * n + oxy;
#pragma unroll
        for (int k = 0; k < CIT / CG; ++k) {
          const int c = cw + k * CG;
          cp4(d + k * CG, p + (size_t)min(c, cmax) * nv, in && c <= cmax);
        }
      }
    }
    const float* dyb = dy + ((size_t)b * Co + co0) * nv;
    const int gw = warp & 3, omax = Co - 1 - co0;
    for (int v = (warp >> 2) * 32 + lane; v < TV; v += NW / 4 * 32) {
      const int lx = v % tl.tx, r = v / tl.tx, ly = r % tl.ty, lz = r / tl.ty;
      const int gx = tx0 + lx, gy = ty0 + ly, gz = tz0 + lz;
      const bool in = gx < n && gy < n && gz < n;
      const float* p = dyb + (in ? ((size_t)gz * n + gy) * n + gx : 0);
      float* d = dys + v * 16 + gw;
      const int sw = (v >> 1) & 3;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = gw + 4 * k;
        cp4(d + ((k ^ sw) << 2), p + (size_t)min(c, omax) * nv, in && c <= omax);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int units = tiles * B;
  int buf = 0;
  if ((int)blockIdx.x < units) stage(blockIdx.x, wg_smem);
  for (int u = blockIdx.x; u < units; u += G, buf ^= 1) {
    const float* dys = wg_smem + buf * bufw;
    const float* xs = dys + WG_TV * 16;
    if (u + G < units) {
      stage(u + G, wg_smem + (buf ^ 1) * bufw);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    for (int r = ks; r < rows; r += KS) {
      const int ly = r % tl.ty, lz = r / tl.ty;
      const float* xr = xs + (((lz + dz) * HY + ly) * HX) * XS + ci;
      float w[3][3];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int e = 0; e < 2; ++e) w[d][e] = xr[(d * HX + e) * XS];
      int v = r * tl.tx;
#pragma unroll 3
      for (int lx = 0; lx < tl.tx; ++lx, ++v) {
#pragma unroll
        for (int d = 0; d < 3; ++d) w[d][2] = xr[(d * HX + lx + 2) * XS];
        const int sw = (v >> 1) & 3;
        const float4 p0 = reinterpret_cast<const float4*>(dys)[v * 4 + ((2 * cog) ^ sw)];
        const float4 p1 = reinterpret_cast<const float4*>(dys)[v * 4 + ((2 * cog + 1) ^ sw)];
        const float g8[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
          for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int e = 0; e < 3; ++e) s[c][d * 3 + e] = fmaf(g8[c], w[d][e], s[c][d * 3 + e]);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          w[d][0] = w[d][1];
          w[d][1] = w[d][2];
        }
      }
    }
    if (bias) {
      const int c = tid & 15, q = c >> 2;
      for (int v = tid >> 4; v < TV; v += WG_NT / 16)
        bsum += dys[(v * 4 + (q ^ ((v >> 1) & 3))) * 4 + (c & 3)];
    }
    __syncthreads();
  }
  // the KS row slices are added in order, through shared memory
  const int slot = tid % (6 * CIT);
  for (int k = 1; k < KS; ++k) {
    if (ks == k)
#pragma unroll
      for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int t = 0; t < 9; ++t) wg_smem[(c * 9 + t) * (6 * CIT) + slot] = s[c][t];
    __syncthreads();
    if (ks == 0)
#pragma unroll
      for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int t = 0; t < 9; ++t) s[c][t] += wg_smem[(c * 9 + t) * (6 * CIT) + slot];
    __syncthreads();
  }
  if (ks == 0 && ci0 + ci < Ci) {
    float* po = part + (size_t)blockIdx.x * Co * Ci * 27;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int co = co0 + cog * 8 + c;
      if (co < Co)
#pragma unroll
        for (int t = 0; t < 9; ++t) po[((size_t)co * Ci + ci0 + ci) * 27 + dz * 9 + t] = s[c][t];
    }
  }
  if (bias) {
    wg_smem[tid] = bsum;
    __syncthreads();
    if (tid < 16 && co0 + tid < Co) {
      float t = 0.f;
      for (int k = 0; k < WG_NT / 16; ++k) t += wg_smem[k * 16 + tid];
      partb[(size_t)blockIdx.x * Co + co0 + tid] = t;
    }
  }
}

// Weight gradient of a 1^3 convolution (the head): a thread walks voxels with 4 x 16 sums in
// registers (4 output, 16 input channels per block), one coalesced load per channel; bound by
// reading x and dy once.  The sums meet by a fixed shuffle tree, then over the warps in order.
__global__ void __launch_bounds__(256) k_wgrad1(const float* __restrict__ x,
                                                const float* __restrict__ dy,
                                                float* __restrict__ part, float* __restrict__ partb,
                                                int B, int Ci, int Co, int n, int G) {
  __shared__ float red[8][68];
  const int nci = (Ci + 15) / 16;
  const int ci0 = (blockIdx.y % nci) * 16, co0 = (blockIdx.y / nci) * 4;
  const int64_t nv = (int64_t)n * n * n;
  const int64_t per = (nv * B + G - 1) / G;
  const int64_t lo = blockIdx.x * per, hi = min(lo + per, nv * B);
  float s[4][16], sb[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    sb[c] = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) s[c][k] = 0.f;
  }
  for (int64_t i = lo + threadIdx.x; i < hi; i += 256) {
    const int64_t b = i / nv, v = i - b * nv;
    float g[4], xv[16];
#pragma unroll
    for (int c = 0; c < 4; ++c) g[c] = co0 + c < Co ? __ldg(dy + (b * Co + co0 + c) * nv + v) : 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) xv[k] = ci0 + k < Ci ? __ldg(x + (b * Ci + ci0 + k) * nv + v) : 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      sb[c] += g[c];
#pragma unroll
      for (int k = 0; k < 16; ++k) s[c][k] = fmaf(g[c], xv[k], s[c][k]);
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float t = warp_sum_f(s[c][k]);
      if (lane == 0) red[warp][c * 16 + k] = t;
    }
    const float t = warp_sum_f(sb[c]);
    if (lane == 0) red[warp][64 + c] = t;
  }
  __syncthreads();
  if (threadIdx.x < 68) {
    float t = 0.f;
    for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
    if (threadIdx.x < 64) {
      const int co = co0 + threadIdx.x / 16, ci = ci0 + threadIdx.x % 16;
      if (co < Co && ci < Ci) part[((size_t)blockIdx.x * Co + co) * Ci + ci] = t;
    } else if (partb && ci0 == 0 && co0 + (int)threadIdx.x - 64 < Co) {
      partb[(size_t)blockIdx.x * Co + co0 + threadIdx.x - 64] = t;
    }
  }
}

// dw[i] += sum_g part[g][i] (and db from partb): a block adds 32 values, its 8 warps the groups
// g = w, w + 8, ..., then the warps' sums in order.
__global__ void __launch_bounds__(256) k_wgrad_reduce(const float* __restrict__ part,
                                                      float* __restrict__ dw, int64_t count,
                                                      const float* __restrict__ partb,
                                                      float* __restrict__ db, int Co, int G) {
  __shared__ float red[8][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t nb = (count + 31) / 32;
  const bool isb = blockIdx.x >= nb;
  const int64_t i = (isb ? blockIdx.x - nb : blockIdx.x) * 32 + lane, m = isb ? Co : count;
  const float* p = isb ? partb : part;
  float s = 0.f;
  if (i < m) {
#pragma unroll 4
    for (int g = warp; g < G; g += 8) s += __ldg(p + (size_t)g * m + i);
  }
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && i < m) {
    float t = 0.f;
    for (int w = 0; w < 8; ++w) t += red[w][lane];
    (isb ? db : dw)[i] += t;
  }
}

// ---------------------------------------------------------------------------------------------
// elementwise and resampling kernels (n = size of the finer grid where it matters)
__global__ void k_relu_bwd(float* __restrict__ dy, const float* __restrict__ y, int64_t count) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (; i < count; i += st)
    if (y[i] <= 0.f) dy[i] = 0.f;
}

// avg pool 2x: x [BC][n^3] -> y [BC][(n/2)^3]
__global__ void k_pool_fwd(const float* __restrict__ x, float* __restrict__ y, int64_t BC, int n) {
  const int m = n / 2;
  const int64_t total = BC * m * m * m;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (; i < total; i += st) {
    const int X = i % m, Y = (i / m) % m, Z = (i / ((int64_t)m * m)) % m;
    const int64_t c = i / ((int64_t)m * m * m);
    const float* p = x + c * n * n * n;
    float s = 0.f;
    for (int dz = 0; dz < 2; ++dz)
      for (int dyy = 0; dyy < 2; ++dyy)
        for (int dx = 0; dx < 2; ++dx) s += p[((int64_t)(2 * Z + dz) * n + 2 * Y + dyy) * n + 2 * X + dx];
    y[i] = 0.125f * s;
  }
}

// dx[fine] = dy[coarse] / 8
__global__ void k_pool_bwd(const float* __restrict__ dy, float* __restrict__ dx, int64_t BC, int n) {
  const int m = n / 2;
  const int64_t total = BC * n * n * n;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (; i < total; i += st) {
    const int X = i % n, Y = (i / n) % n, Z = (i / ((int64_t)n * n)) % n;
    const int64_t c = i / ((int64_t)n * n * n);
    dx[i] = 0.125f * dy[c * m * m * m + ((int64_t)(Z / 2) * m + Y / 2) * m + X / 2];
  }
}

// nearest upsample 2x: x [B][C][m^3] -> y[b][coff + c][n^3] inside a buffer of Cy channels
__global__ void k_up_fwd(const float* __restrict__ x, float* __restrict__ y, int B, int C, int m,
                         int Cy, int coff) {
  const int n = 2 * m;
  const int64_t total = (int64_t)B * C * n * n * n;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (; i < total; i += st) {
    const int X = i % n, Y = (i / n) % n, Z = (i / ((int64_t)n * n)) % n;
    const int64_t bc = i / ((int64_t)n * n * n);
    const int c = (int)(bc % C), b = (int)(bc / C);
    y[((int64_t)b * Cy + coff + c) * n * n * n + ((int64_t)Z * n + Y) * n + X] =
        x[bc * m * m * m + ((int64_t)(Z / 2) * m + Y / 2) * m + X / 2];
  }
}

// dx[b][c][m^3] = sum of the 8 children of dy[b][coff + c][n^3] (Cy channels in dy)
__global__ void k_up_bwd(const float* __restrict__ dy, float* __restrict__ dx, int B, int C, int m,
                         int Cy, int coff) {
  const int n = 2 * m;
  const int64_t total = (int64_t)B * C * m * m * m;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (; i < total; i += st) {
    const int X = i % m, Y = (i / m) % m, Z = (i / ((int64_t)m * m)) % m;
    const int64_t bc = i / ((int64_t)m * m * m);
    const int c = (int)(bc % C), b = (int)(bc / C);
    const float* p = dy + ((int64_t)b * Cy + coff + c) * n * n * n;
    float s = 0.f;
    for (int dz = 0; dz < 2; ++dz)
      for (int dyy = 0; dyy < 2; ++dyy)
        for (int dx2 = 0; dx2 < 2; ++dx2) s += p[((int64_t)(2 * Z + dz) * n + 2 * Y + dyy) * n + 2 * X + dx2];
    dx[i] = s;
  }
}

// copy channels: dst[b][doff + c][v] = src[b][soff + c][v] for c < C (accumulate optional)
__global__ void k_copy_ch(const float* __restrict__ src, float* __restrict__ dst, int B, int C,
                          int64_t nv, int Cs, int soff, int Cd, int doff, int accumulate) {
  const int64_t total = (int64_t)B * C * nv;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (; i < total; i += st) {
    const int64_t v = i % nv;
    const int64_t bc = i / nv;
    const int c = (int)(bc % C), b = (int)(bc / C);
    const float s = src[((int64_t)b * Cs + soff + c) * nv + v];
    float* d = dst + ((int64_t)b * Cd + doff + c) * nv + v;
    *d = accumulate ? *d + s : s;
  }
}

// MSE: loss = mean (p - t)^2 (FP64 sum); grad = 2 (p - t) / count
__global__ void k_mse(const float* __restrict__ p, const float* __restrict__ t, float* __restrict__ g,
                      int64_t count, double* loss) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  float s = 0.f;
  const float sc = 2.f / (float)count;
  for (; i < count; i += st) {
    const float d = p[i] - t[i];
    s = fmaf(d, d, s);
    if (g) g[i] = sc * d;
  }
  block_sum_f_atomic(s, loss);
}

// Adam on FP32 master weights, with the bf16 copy used by the products refreshed in place.
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, __nv_bfloat16* __restrict__ wb, int64_t count,
                       float lr, float b1, float b2, float eps, float c1, float c2) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (; i < count; i += st) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    if (wb) wb[i] = __float2bfloat16_rn(wi);
  }
}

__global__ void k_cast_bf16(const float* __restrict__ a, __nv_bfloat16* __restrict__ b, int64_t count) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (; i < count; i += st) b[i] = __float2bfloat16_rn(a[i]);
}

// ---------------------------------------------------------------------------------------------
static inline int gs(int64_t n) {
  const int64_t b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

static int tiles_of(int n) { return ((n + BX - 1) / BX) * ((n + BY - 1) / BY) * ((n + BZ - 1) / BZ); }

bool conv_tc_supported(int Ci, int Co);
cudaError_t conv_tc_fwd(const float* x, const void* w, const float* bias, float* y, int B, int Ci,
                        int Co, int n, int ks, int relu, int accumulate, cudaStream_t s);

cudaError_t net_conv_fwd(const float* x, const void* w, const float* bias, float* y, int B, int Ci,
                         int Co, int n, int ks, int relu, int accumulate, cudaStream_t s) {
  // input channels in groups of 16: the tensor-core implicit GEMM (kernels_conv_tc.cu)
  if (conv_tc_supported(Ci, Co))
    return conv_tc_fwd(x, w, bias, y, B, Ci, Co, n, ks, relu, accumulate, s);
  dim3 grid(tiles_of(n), (Co + CT - 1) / CT, B);
  k_conv_fwd<<<grid, NTV, 0, s>>>(x, (const __nv_bfloat16*)w, bias, y, Ci, Co, n, ks, relu,
                                  accumulate);
  return cudaGetLastError();
}

cudaError_t net_conv_dgrad(const float* dy, const void* w, void* wT_scratch, float* dx, int B,
                           int Ci, int Co, int n, int ks, cudaStream_t s) {
  const int taps = ks * ks * ks;
  const int cnt = Ci * Co * taps;
  k_transpose_flip<<<(cnt + 255) / 256, 256, 0, s>>>((const __nv_bfloat16*)w,
                                                     (__nv_bfloat16*)wT_scratch, Ci, Co, taps);
  return net_conv_fwd(dy, wT_scratch, nullptr, dx, B, Co, Ci, n, ks, 0, 0, s);
}

// Partition of the weight gradient: input channels per block (16, or the next power of two of
// fewer), the voxel tile of a unit (rows of up to 32 voxels, split evenly so that 40 or 56 leave
// no ragged end; ty grows while the tile has room, so that short rows keep a small halo), and the
// number of groups G: one block per SM on 152 SMs (three for the 1^3 kernel, which waits on
// memory), evened out over the units.
struct WgPlan {
  int cit, G;
  WgTile tl;
};
static WgPlan wgrad_plan(int B, int Ci, int Co, int n, int ks) {
  WgPlan p{};
  const int64_t slots = 152 * (ks == 1 ? 3 : 1);
  if (ks == 1) {
    const int64_t nblk = (int64_t)((Ci + 15) / 16) * ((Co + 3) / 4);
    const int64_t units = ((int64_t)B * n * n * n + 2047) / 2048;
    const int64_t g = slots / nblk;
    p.G = (int)(g < 1 ? 1 : (g > units ? units : g));
    return p;
  }
  p.cit = Ci > 8 ? 16 : Ci > 4 ? 8 : Ci > 2 ? 4 : 2;
  const auto even = [](int len, int most) {
    const int k = (len + most - 1) / most;
    return (len + k - 1) / k;
  };
  WgTile& t = p.tl;
  t.tx = even(n, 32);
  t.ty = even(n, t.tx > 16 ? 4 : t.tx > 8 ? 4 : 8);
  const int room = WG_TV / (t.tx * t.ty);
  t.tz = even(n, room < 1 ? 1 : (room > 4 ? 4 : room));
  t.ntx = (n + t.tx - 1) / t.tx;
  t.nty = (n + t.ty - 1) / t.ty;
  t.ntz = (n + t.tz - 1) / t.tz;
  const int64_t nblk = (int64_t)((Ci + p.cit - 1) / p.cit) * ((Co + 15) / 16);
  const int64_t units = (int64_t)t.ntx * t.nty * t.ntz * B;
  int64_t g = slots / nblk;
  g = g < 1 ? 1 : (g > units ? units : g);
  const int64_t rounds = (units + g - 1) / g;
  p.G = (int)((units + rounds - 1) / rounds);
  return p;
}

int64_t net_conv_wgrad_scratch(int B, int Ci, int Co, int n, int ks) {
  const WgPlan p = wgrad_plan(B, Ci, Co, n, ks);
  return (int64_t)p.G * Co * Ci * ks * ks * ks + (int64_t)p.G * Co;
}

template <int CIT>
static cudaError_t launch_wgrad3(const float* x, const float* dy, float* part, float* partb, int B,
                                 int Ci, int Co, int n, const WgPlan& p, cudaStream_t s) {
  // two staging buffers, or the row slices' sums at the end
  const auto words = [](int halo) { return 2 * ((WG_TV * 16 + halo * (CIT + 1) + 3) & ~3); };
  const int fl = words((p.tl.tx + 2) * (p.tl.ty + 2) * (p.tl.tz + 2)), fe = 72 * 6 * CIT;
  const int smem = 4 * (fl > fe ? fl : fe);
  const int kMost = 4 * words(34 * 6 * 4);   // the largest tile's
  static const cudaError_t set = cudaFuncSetAttribute(
      k_wgrad3<CIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
  if (set != cudaSuccess) return set;
  if (smem > kMost) return cudaErrorInvalidValue;
  const dim3 grid(p.G, ((Ci + CIT - 1) / CIT) * ((Co + 15) / 16));
  k_wgrad3<CIT><<<grid, WG_NT, smem, s>>>(x, dy, part, partb, B, Ci, Co, n, p.tl, p.G);
  return cudaGetLastError();
}

cudaError_t net_conv_wgrad(const float* x, const float* dy, float* dw, float* db, float* scratch,
                           int B, int Ci, int Co, int n, int ks, cudaStream_t s) {
  const WgPlan p = wgrad_plan(B, Ci, Co, n, ks);
  const int64_t count = (int64_t)Co * Ci * ks * ks * ks;
  float* partb = db ? scratch + (size_t)p.G * count : nullptr;
  cudaError_t e;
  if (ks == 1) {
    const dim3 grid(p.G, ((Ci + 15) / 16) * ((Co + 3) / 4));
    k_wgrad1<<<grid, 256, 0, s>>>(x, dy, scratch, partb, B, Ci, Co, n, p.G);
    e = cudaGetLastError();
  } else if (p.cit == 16) {
    e = launch_wgrad3<16>(x, dy, scratch, partb, B, Ci, Co, n, p, s);
  } else if (p.cit == 8) {
    e = launch_wgrad3<8>(x, dy, scratch, partb, B, Ci, Co, n, p, s);
  } else if (p.cit == 4) {
    e = launch_wgrad3<4>(x, dy, scratch, partb, B, Ci, Co, n, p, s);
  } else {
    e = launch_wgrad3<2>(x, dy, scratch, partb, B, Ci, Co, n, p, s);
  }
  if (e != cudaSuccess) return e;
  const unsigned nb = (unsigned)((count + 31) / 32 + (db ? (Co + 31) / 32 : 0));
  k_wgrad_reduce<<<nb, 256, 0, s>>>(scratch, dw, count, partb, db, Co, p.G);
  return cudaGetLastError();
}

cudaError_t net_relu_bwd(float* dy, const float* y, int64_t count, cudaStream_t s) {
  k_relu_bwd<<<gs(count), 256, 0, s>>>(dy, y, count);
  return cudaGetLastError();
}
cudaError_t net_pool_fwd(const float* x, float* y, int64_t BC, int n, cudaStream_t s) {
  k_pool_fwd<<<gs(BC * n * n * n / 8), 256, 0, s>>>(x, y, BC, n);
  return cudaGetLastError();
}
cudaError_t net_pool_bwd(const float* dy, float* dx, int64_t BC, int n, cudaStream_t s) {
  k_pool_bwd<<<gs(BC * n * n * n), 256, 0, s>>>(dy, dx, BC, n);
  return cudaGetLastError();
}
cudaError_t net_up_fwd(const float* x, float* y, int B, int C, int m, int Cy, int coff,
                       cudaStream_t s) {
  k_up_fwd<<<gs((int64_t)B * C * 8 * m * m * m), 256, 0, s>>>(x, y, B, C, m, Cy, coff);
  return cudaGetLastError();
}
cudaError_t net_up_bwd(const float* dy, float* dx, int B, int C, int m, int Cy, int coff,
                       cudaStream_t s) {
  k_up_bwd<<<gs((int64_t)B * C * m * m * m), 256, 0, s>>>(dy, dx, B, C, m, Cy, coff);
  return cudaGetLastError();
}
cudaError_t net_copy_ch(const float* src, float* dst, int B, int C, int64_t nv, int Cs, int soff,
                        int Cd, int doff, int accumulate, cudaStream_t s) {
  k_copy_ch<<<gs((int64_t)B * C * nv), 256, 0, s>>>(src, dst, B, C, nv, Cs, soff, Cd, doff,
                                                    accumulate);
  return cudaGetLastError();
}
cudaError_t net_mse(const float* p, const float* t, float* g, int64_t count, double* loss,
                    cudaStream_t s) {
  k_mse<<<gs(count), 256, 0, s>>>(p, t, g, count, loss);
  return cudaGetLastError();
}
cudaError_t net_adam(float* w, const float* g, float* m, float* v, void* wb, int64_t count,
                     float lr, float b1, float b2, float eps, int step, cudaStream_t s) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_adam<<<gs(count), 256, 0, s>>>(w, g, m, v, (__nv_bfloat16*)wb, count, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}
cudaError_t net_cast_bf16(const float* a, void* b, int64_t count, cudaStream_t s) {
  k_cast_bf16<<<gs(count), 256, 0, s>>>(a, (__nv_bfloat16*)b, count);
  return cudaGetLastError();
}

}  // namespace lddmm
