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

// Weight gradient, deterministic: dw[co][ci][t] is summed voxel by voxel in a fixed order.  Units
// (batch, 8x8x4 tile) g, g + G, .. make one chain of FMAs per group g (x fastest, then y, z inside a
// tile); part[g][co][ci][t] holds its end, and k_wgrad_reduce adds the groups in order.  No
// floating-point atomics, the same bits on every run and for every shape of the block.
// It is a product of Co x B n^3 by B n^3 x 27 Ci in FP32 (274 GFLOP in a training step at 64^3,
// batch 8: 3.4 ms), so the FP32 pipes bound it and everything else has to stay off their issue
// slots.  A block owns 16 output channels x CIT input channels of one group; it stages a unit's x
// (with halo, [voxel][ci], rows of CIT + 1 words: conflict free both ways) and dy ([channel pair]
// [voxel][2]) by 4-byte asynchronous copies into two buffers, the next unit's under the products of
// this one.  A thread owns one input channel, one dz and 2 output channels: it walks the tile's rows
// with three rows of x in registers, so a voxel costs 1.6 + 0.5 shared loads at constant offsets for
// 18 FMAs.  The step's 14 such gradients take 6.3 ms: 6.8 with all positions decoded for every unit
// and dy read a voxel at a time, 8.3 with 3 loads of x per voxel, 57 with one (co, tap) per thread
// and two shared loads per FMA.  What is left: the partition leaves up to 24 SMs without a block,
// and a sixth of the issue slots stage.
constexpr int WG_DS = NTV * 2 + 4, WG_DY = CT / 2 * WG_DS;   // words of a channel pair of dy, of all
constexpr int WG_CPT = 2, WG_HX = BX + 2, WG_HXY = (BX + 2) * (BY + 2), WG_HV = WG_HXY * (BZ + 2);
__host__ __device__ constexpr int wg_threads(int cit) { return (cit * 3 * (CT / WG_CPT) + 31) / 32 * 32; }
__host__ __device__ constexpr int wg_words(int cit) { return WG_DY + WG_HV * (cit + 1); }

// 4 bytes to shared memory, asynchronously; zeros when len = 0 (the address is then not read)
__device__ __forceinline__ void cp4(float* dst, const float* src, int len) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(len)
               : "memory");
}

template <int CIT>
__global__ void __launch_bounds__(wg_threads(CIT), 1) k_wgrad3(const float* __restrict__ x,
                                                               const float* __restrict__ dy,
                                                               float* __restrict__ part, int B,
                                                               int Ci, int Co, int n, int G) {
  constexpr int NT = wg_threads(CIT), NW = NT / 32, XS = CIT + 1, COG = CT / WG_CPT;
  extern __shared__ __align__(16) float wg_smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ci = tid % CIT, cog = (tid / CIT) % COG, dz = tid / (CIT * COG);
  const int nci = (Ci + CIT - 1) / CIT;
  const int ci0 = (blockIdx.y % nci) * CIT, co0 = (blockIdx.y / nci) * CT;
  const int ntx = (n + BX - 1) / BX, nty = (n + BY - 1) / BY, ntz = (n + BZ - 1) / BZ;
  const int tiles = ntx * nty * ntz;
  const size_t nv = (size_t)n * n * n;
  float s[WG_CPT][9];
#pragma unroll
  for (int c = 0; c < WG_CPT; ++c)
#pragma unroll
    for (int t = 0; t < 9; ++t) s[c][t] = 0.f;
  // Staging.  A warp takes the channels w % CG, + CG, .. of the positions of its lanes.  What only
  // depends on the thread is kept: a position's offset from the tile's first voxel, and a bit for its
  // place along each axis, which the unit's mask of places outside the grid is tested against.
  // Addresses are clamped into the tensor, what lies outside the grid arrives as zero.
  constexpr int CG = NW < 4 ? 1 : NW % 4 == 0 ? 4 : 2, PG = NW / CG, XP = (WG_HV + PG * 32 - 1) / (PG * 32);
  constexpr int DP = (NTV + PG * 32 - 1) / (PG * 32);
  static_assert(NW % CG == 0 && CIT % CG == 0, "every warp stages");
  const int cw = warp % CG, cmax = Ci - 1 - ci0, omax = Co - 1 - co0;
  const int e0 = (warp / CG) * 32 + lane;
  int xrel[XP], drel[DP];
  unsigned xbit[XP], dbit[DP];
  auto place = [&](int hx, int hy, int hz, int& rel, unsigned& bit) {
    rel = ((hz - 1) * n + hy - 1) * n + hx - 1;
    bit = 1u << hx | 1u << (WG_HX + hy) | 1u << (WG_HX + BY + 2 + hz);
  };
#pragma unroll
  for (int k = 0; k < XP; ++k) {
    const int e = e0 + k * PG * 32, r = e % WG_HXY;
    place(r % WG_HX, r / WG_HX, min(e / WG_HXY, BZ + 1), xrel[k], xbit[k]);
  }
#pragma unroll
  for (int k = 0; k < DP; ++k) {
    const int v = e0 + k * PG * 32;
    place(v % BX + 1, v / BX % BY + 1, min(v / (BX * BY), BZ - 1) + 1, drel[k], dbit[k]);
  }
  const int units = tiles * B;
  // tile of the next unit to stage, and the step to the one after
  int tx = blockIdx.x % ntx, ty = blockIdx.x / ntx % nty, tz = blockIdx.x / (ntx * nty) % ntz, b = blockIdx.x / tiles;
  const int gx = G % ntx, gy = G / ntx % nty, gz = G / (ntx * nty) % ntz, gb = G / tiles;
  auto stage = [&](float* dys) {
    float* const xs = dys + WG_DY;
    const int x0 = tx * BX, y0 = ty * BY, z0 = tz * BZ;
    // places with no voxel: the first along an axis at its near face, those past n at the far one
    auto outside = [&](int o, int len) {
      const unsigned far = n - o + 1 < len ? ~0u << (n - o + 1) & ((1u << len) - 1) : 0u;
      return far | (o == 0 ? 1u : 0u);
    };
    const unsigned mask = outside(x0, WG_HX) | outside(y0, BY + 2) << WG_HX |
                          outside(z0, BZ + 2) << (WG_HX + BY + 2);
    const size_t o = ((size_t)z0 * n + y0) * n + x0;
    const float* const xb = x + ((size_t)b * Ci + ci0) * nv + o;
    const float* const db = dy + ((size_t)b * Co + co0) * nv + o;
    int off[XP], len[XP];
#pragma unroll
    for (int k = 0; k < XP; ++k) {
      const bool in = !(xbit[k] & mask);
      off[k] = in ? xrel[k] : 0;
      len[k] = in ? 4 : 0;
    }
#pragma unroll
    for (int j = 0; j < CIT / CG; ++j) {
      const int c = cw + j * CG;
      const float* const p = xb + (size_t)min(c, cmax) * nv;
#pragma unroll
      for (int k = 0; k < XP; ++k)
        if (k < XP - 1 || e0 + k * PG * 32 < WG_HV)
          cp4(xs + (e0 + k * PG * 32) * XS + c, p + off[k], c <= cmax ? len[k] : 0);
    }
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const bool in = !(dbit[k] & mask);
      off[k] = in ? drel[k] : 0;
      len[k] = in ? 4 : 0;
    }
#pragma unroll
    for (int j = 0; j < CT / CG; ++j) {
      const int c = cw + j * CG;
      const float* const p = db + (size_t)min(c, omax) * nv;
#pragma unroll
      for (int k = 0; k < DP; ++k)
        if (k < DP - 1 || e0 + k * PG * 32 < NTV)
          cp4(dys + (c >> 1) * WG_DS + (e0 + k * PG * 32) * 2 + (c & 1), p + off[k], c <= omax ? len[k] : 0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    tx += gx;
    ty += gy;
    tz += gz;
    b += gb;
    if (tx >= ntx) { tx -= ntx; ++ty; }
    if (ty >= nty) { ty -= nty; ++tz; }
    if (tz >= ntz) { tz -= ntz; ++b; }
  };
  int buf = 0;
  if ((int)blockIdx.x < units) stage(wg_smem);
  for (int u = blockIdx.x; u < units; u += G, buf ^= 1) {
    const float* dys = wg_smem + buf * wg_words(CIT);
    const float* xs = dys + WG_DY;
    if (u + G < units) {
      stage(wg_smem + (buf ^ 1) * wg_words(CIT));
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    if (dz < 3) {
      // rows of x stay in registers while they are in reach: row y + 1 is read in place of row y - 2
      for (int lz = 0; lz < BZ; ++lz) {
        const float* xr = xs + (lz + dz) * WG_HXY * XS + ci;
        const float* dr = dys + cog * WG_DS + lz * BY * BX * 2;
        float w[3][WG_HX];
#pragma unroll
        for (int d = 0; d < 2; ++d)
#pragma unroll
          for (int e = 0; e < WG_HX; ++e) w[d][e] = xr[(d * WG_HX + e) * XS];
#pragma unroll
        for (int ly = 0; ly < BY; ++ly) {
#pragma unroll
          for (int e = 0; e < WG_HX; ++e) w[(ly + 2) % 3][e] = xr[((ly + 2) * WG_HX + e) * XS];
#pragma unroll
          for (int lx = 0; lx < BX; lx += 2) {
            const float4 g = *reinterpret_cast<const float4*>(dr + (ly * BX + lx) * 2);
#pragma unroll
            for (int d = 0; d < 3; ++d)
#pragma unroll
              for (int e = 0; e < 3; ++e) {
                s[0][d * 3 + e] = fmaf(g.x, w[(ly + d) % 3][lx + e], s[0][d * 3 + e]);
                s[1][d * 3 + e] = fmaf(g.y, w[(ly + d) % 3][lx + e], s[1][d * 3 + e]);
              }
#pragma unroll
            for (int d = 0; d < 3; ++d)
#pragma unroll
              for (int e = 0; e < 3; ++e) {
                s[0][d * 3 + e] = fmaf(g.z, w[(ly + d) % 3][lx + 1 + e], s[0][d * 3 + e]);
                s[1][d * 3 + e] = fmaf(g.w, w[(ly + d) % 3][lx + 1 + e], s[1][d * 3 + e]);
              }
          }
        }
      }
    }
    __syncthreads();
  }
  if (dz < 3 && ci0 + ci < Ci) {
    float* po = part + (size_t)blockIdx.x * Co * Ci * 27;
#pragma unroll
    for (int c = 0; c < WG_CPT; ++c) {
      const int co = co0 + cog * WG_CPT + c;
      if (co < Co)
#pragma unroll
        for (int t = 0; t < 9; ++t) po[((size_t)co * Ci + ci0 + ci) * 27 + dz * 9 + t] = s[c][t];
    }
  }
}

// The same for a 1^3 convolution (the head): a block owns 16 x 16 channels of one group, a thread one
// pair of them; x and dy of a unit lie in shared memory as [voxel][16 channels] (17 words), the next
// unit's copies run under this one's chain.
__global__ void __launch_bounds__(256, 1) k_wgrad1(const float* __restrict__ x,
                                                   const float* __restrict__ dy,
                                                   float* __restrict__ part, int B, int Ci, int Co,
                                                   int n, int G) {
  extern __shared__ __align__(16) float wg_smem[];
  constexpr int S1 = CT + 1, HALF = NTV * S1, W1 = 2 * HALF;
  const int tid = threadIdx.x;
  const int nci = (Ci + 15) / 16;
  const int ci0 = (blockIdx.y % nci) * 16, co0 = (blockIdx.y / nci) * CT;
  const int ntx = (n + BX - 1) / BX, nty = (n + BY - 1) / BY, ntz = (n + BZ - 1) / BZ;
  const int tiles = ntx * nty * ntz, units = tiles * B;
  const size_t nv = (size_t)n * n * n;
  const int ni = min(16, Ci - ci0), no = min(CT, Co - co0);
  auto stage = [&](int u, float* xs) {
    const int b = u / tiles, tile = u - b * tiles;
    const int gx = (tile % ntx) * BX + tid % BX, gy = ((tile / ntx) % nty) * BY + tid / BX % BY,
              gz = (tile / (ntx * nty)) * BZ + tid / (BX * BY);
    const bool in = gx < n && gy < n && gz < n;
    const size_t o = in ? ((size_t)gz * n + gy) * n + gx : 0;
    const float* xb = x + ((size_t)b * Ci + ci0) * nv + o;
    const float* db = dy + ((size_t)b * Co + co0) * nv + o;
    for (int c = 0; c < ni; ++c) cp4(xs + tid * S1 + c, xb + (size_t)c * nv, in ? 4 : 0);
    for (int c = 0; c < no; ++c) cp4(xs + HALF + tid * S1 + c, db + (size_t)c * nv, in ? 4 : 0);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int ci = tid & 15, co = tid >> 4;
  float s = 0.f;
  int buf = 0;
  if ((int)blockIdx.x < units) stage(blockIdx.x, wg_smem);
  for (int u = blockIdx.x; u < units; u += G, buf ^= 1) {
    if (u + G < units) {
      stage(u + G, wg_smem + (buf ^ 1) * W1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    if (ci < ni && co < no) {
      const float* xs = wg_smem + buf * W1 + ci;
      const float* ds = wg_smem + buf * W1 + HALF + co;
#pragma unroll 16
      for (int v = 0; v < NTV; ++v) s = fmaf(ds[v * S1], xs[v * S1], s);
    }
    __syncthreads();
  }
  if (ci < ni && co < no) part[((size_t)blockIdx.x * Co + co0 + co) * Ci + ci0 + ci] = s;
}

// dw[i] += sum_{g = 0..G-1} part[g][i], in that order; 16 loads in flight.
__global__ void __launch_bounds__(64) k_wgrad_reduce(const float* __restrict__ part,
                                                     float* __restrict__ dw, int64_t count, int G) {
  const int64_t i = (int64_t)blockIdx.x * 64 + threadIdx.x;
  if (i >= count) return;
  const float* p = part + i;
  float s = 0.f;
  int g = 0;
  for (; g + 16 <= G; g += 16) {
    float v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __ldg(p + (size_t)(g + k) * count);
#pragma unroll
    for (int k = 0; k < 16; ++k) s += v[k];
  }
  for (; g < G; ++g) s += __ldg(p + (size_t)g * count);
  dw[i] += s;
}

// Bias gradient, deterministic: block (co, g) sums the fixed chunk g of the B * n^3 values of
// channel co (a thread every 256th value, eight loads in flight; then a tree of fixed shape) into
// partb[co][g]; k_bias_reduce adds them in order.
__global__ void __launch_bounds__(256) k_bias_partial(const float* __restrict__ dy,
                                                      float* __restrict__ partb, int B, int Co,
                                                      int n, int GB) {
  const int co = blockIdx.x, g = blockIdx.y;
  const size_t nv = (size_t)n * n * n;
  const size_t total = (size_t)B * nv, chunk = (total + GB - 1) / GB;
  const size_t lo = (size_t)g * chunk, hi = lo + chunk < total ? lo + chunk : total;
  float s = 0.f;
  // value i of the channel lies at (b Co + co) nv + v, i = b nv + v; b steps up as i passes it
  size_t i = lo + threadIdx.x, b = i / nv, end = (b + 1) * nv;
  const float* p = dy + (b * Co + co) * nv - b * nv;
  auto at = [&](size_t k) {
    while (k >= end) {
      ++b;
      end += nv;
      p += (size_t)(Co - 1) * nv;
    }
    return __ldg(p + k);
  };
  while (i < hi) {
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = i + 256 * k < hi ? at(i + 256 * k) : 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i + 256 * k < hi) s += v[k];
    i += 2048;
  }
  __shared__ float red[32];
  s = warp_sum_f(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    float t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    t = warp_sum_f(t);
    if (threadIdx.x == 0) partb[(size_t)co * GB + g] = t;
  }
}

__global__ void k_bias_reduce(const float* __restrict__ partb, float* __restrict__ db, int Co, int GB) {
  const int co = blockIdx.x * blockDim.x + threadIdx.x;
  if (co >= Co) return;
  float s = 0.f;
  for (int g = 0; g < GB; ++g) s += partb[(size_t)co * GB + g];
  db[co] += s;
}

// ---------------------------------------------------------------------------------------------
// Elementwise and resampling kernels: bound by memory, so a thread decodes its voxel once and then
// takes it through the channels (with a 64-bit division or three per element the four kernels of a
// 64^3 step took 1.77 ms, now 0.71).

// a / d for a >= 0, by the 32-bit division unless a needs more
__device__ __forceinline__ int64_t quot64(int64_t a, int64_t d) {
  return ((a | d) >> 32) ? a / d : (int64_t)((uint32_t)a / (uint32_t)d);
}

// Threads over `vox` voxels (blockIdx.x) and the channels (blockIdx.y): a block smaller than its 256
// threads takes several channels at once.  About four channels a thread, fewer while the chip is
// not full.
struct VoxGrid {
  dim3 grid;
  int cpb;              // channels a block takes at once
};
static VoxGrid vox_grid(int64_t vox, int64_t BC) {
  VoxGrid v;
  v.cpb = vox < 256 ? (int)(256 / vox) : 1;
  const int64_t gx = (vox + 255) / 256, steps = (BC + v.cpb - 1) / v.cpb;
  int64_t gy = (steps + 3) / 4, full = (152 * 16 + gx - 1) / gx;
  if (gy < full) gy = full;
  if (gy > steps) gy = steps;
  v.grid = dim3((unsigned)gx, (unsigned)(gy < 65535 ? gy : 65535));
  return v;
}
// the voxel and first channel of this thread; false: none
__device__ __forceinline__ bool vox_of(int64_t vox, int cpb, int64_t& j, int64_t& bc) {
  const int sub = cpb > 1 ? (int)(threadIdx.x / (unsigned)vox) : 0;
  j = cpb > 1 ? (int64_t)(threadIdx.x - sub * (unsigned)vox) : (int64_t)blockIdx.x * 256 + threadIdx.x;
  bc = (int64_t)blockIdx.y * cpb + sub;
  return j < vox && sub < cpb;
}

// 8 children of a coarse voxel, in rows of two (n is even: a row's pair is 8-byte aligned when the
// tensor is).  The thread of a coarse voxel j of an m^3 grid; first child of the fine one.
__device__ __forceinline__ int64_t first_child(int64_t j, int m) {
  const int64_t r = quot64(j, m), X = j - r * m, Z = quot64(r, m), Y = r - Z * m;
  return ((2 * Z) * (2 * m) + 2 * Y) * (2 * m) + 2 * X;
}

// Every child takes its parent's value: nearest upsampling x [B][C][m^3] -> y[b][coff + c][n^3]
// inside Cy channels, or (MEAN: an eighth of it) the average pooling's backward.
template <bool MEAN>
__global__ void __launch_bounds__(256) k_spread(const float* __restrict__ x, float* __restrict__ y,
                                                int64_t BC, int C, int m, int Cy, int coff, int cpb,
                                                int pairs) {
  const int64_t m3 = (int64_t)m * m * m, n = 2 * m;
  int64_t j, bc;
  if (!vox_of(m3, cpb, j, bc)) return;
  float* const q = y + first_child(j, m);
  for (; bc < BC; bc += (int64_t)gridDim.y * cpb) {
    const float s = __ldg(x + bc * m3 + j), v = MEAN ? 0.125f * s : s;
    const int64_t b = MEAN ? 0 : quot64(bc, C);
    float* const p = q + (MEAN ? bc : b * Cy + coff + (bc - b * C)) * 8 * m3;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float* d = p + (r >> 1) * n * n + (r & 1) * n;
      if (pairs) {
        *reinterpret_cast<float2*>(d) = make_float2(v, v);
      } else {
        d[0] = v;
        d[1] = v;
      }
    }
  }
}

// A coarse voxel takes the sum of its children, z slowest: the upsampling's backward (Cy channels
// in x), or (MEAN: an eighth of it) average pooling.
template <bool MEAN>
__global__ void __launch_bounds__(256) k_gather(const float* __restrict__ x, float* __restrict__ y,
                                                int64_t BC, int C, int m, int Cy, int coff, int cpb,
                                                int pairs) {
  const int64_t m3 = (int64_t)m * m * m, n = 2 * m;
  int64_t j, bc;
  if (!vox_of(m3, cpb, j, bc)) return;
  const float* const q = x + first_child(j, m);
  for (; bc < BC; bc += (int64_t)gridDim.y * cpb) {
    const int64_t b = MEAN ? 0 : quot64(bc, C);
    const float* const p = q + (MEAN ? bc : b * Cy + coff + (bc - b * C)) * 8 * m3;
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float* d = p + (r >> 1) * n * n + (r & 1) * n;
      const float2 v = pairs ? __ldg(reinterpret_cast<const float2*>(d)) : make_float2(__ldg(d), __ldg(d + 1));
      s += v.x;
      s += v.y;
    }
    y[bc * m3 + j] = MEAN ? 0.125f * s : s;
  }
}

__device__ __forceinline__ float sum(float a, float b) { return a + b; }
__device__ __forceinline__ float4 sum(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// copy channels: dst[b][doff + c][v] = src[b][soff + c][v] for c < C (accumulate optional); T is
// float4 where nv and both tensors allow, nv counts T
template <typename T>
__global__ void __launch_bounds__(256) k_copy_ch(const T* __restrict__ src, T* __restrict__ dst,
                                                 int64_t BC, int C, int64_t nv, int Cs, int soff, int Cd,
                                                 int doff, int accumulate, int cpb) {
  int64_t j, bc;
  if (!vox_of(nv, cpb, j, bc)) return;
  for (; bc < BC; bc += (int64_t)gridDim.y * cpb) {
    const int64_t b = quot64(bc, C), c = bc - b * C;
    T s = __ldg(src + (b * Cs + soff + c) * nv + j);
    T* d = dst + (b * Cd + doff + c) * nv + j;
    if (accumulate) s = sum(*d, s);
    *d = s;
  }
}

// dy = 0 where y <= 0; `quads` of four with 16-byte accesses, then the rest
__global__ void __launch_bounds__(256) k_relu_bwd(float* __restrict__ dy, const float* __restrict__ y,
                                                  int64_t count, int64_t quads) {
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = i0; i < quads; i += st) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(y) + i);
    float4 d = reinterpret_cast<float4*>(dy)[i];
    d.x = v.x <= 0.f ? 0.f : d.x;
    d.y = v.y <= 0.f ? 0.f : d.y;
    d.z = v.z <= 0.f ? 0.f : d.z;
    d.w = v.w <= 0.f ? 0.f : d.w;
    reinterpret_cast<float4*>(dy)[i] = d;
  }
  for (int64_t i = 4 * quads + i0; i < count; i += st)
    if (y[i] <= 0.f) dy[i] = 0.f;
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

bool conv_tc_supported(int Ci, int Co, int n);
cudaError_t conv_tc_fwd(const float* x, const void* w, const float* bias, float* y, int B, int Ci,
                        int Co, int n, int ks, int relu, int accumulate, cudaStream_t s);

cudaError_t net_conv_fwd(const float* x, const void* w, const float* bias, float* y, int B, int Ci,
                         int Co, int n, int ks, int relu, int accumulate, cudaStream_t s) {
  // input channels in groups of 16: the tensor-core implicit GEMM (kernels_conv_tc.cu)
  if (conv_tc_supported(Ci, Co, n))
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

// Partition of the weight-gradient sums: G voxel groups (about 2048 chains of units per 16 output
// channels and tap, at most one group per (batch, tile) unit), GB chunks per bias channel.
static void wgrad_groups(int B, int Ci, int Co, int n, int* G, int* GB) {
  const int units = tiles_of(n) * B;
  const int cb = Ci * ((Co + CT - 1) / CT);
  int g = (2048 + cb - 1) / cb;
  *G = g < 1 ? 1 : (g > units ? units : g);
  const int64_t total = (int64_t)B * n * n * n;
  int64_t gb = (total + 8191) / 8192;
  *GB = (int)(gb < 1 ? 1 : (gb > 64 ? 64 : gb));
}

int64_t net_conv_wgrad_scratch(int B, int Ci, int Co, int n, int ks) {
  int G, GB;
  wgrad_groups(B, Ci, Co, n, &G, &GB);
  return (int64_t)G * Co * Ci * ks * ks * ks + (int64_t)Co * GB;
}

template <int CIT>
static cudaError_t launch_wgrad3(const float* x, const float* dy, float* part, int B, int Ci, int Co,
                                 int n, int G, cudaStream_t s) {
  constexpr int smem = 2 * 4 * wg_words(CIT);
  static PerDevice<bool> set;
  const cudaError_t e = raise_smem_limit(set, k_wgrad3<CIT>, smem);
  if (e != cudaSuccess) return e;
  const dim3 grid(G, ((Ci + CIT - 1) / CIT) * ((Co + CT - 1) / CT));
  k_wgrad3<CIT><<<grid, wg_threads(CIT), smem, s>>>(x, dy, part, B, Ci, Co, n, G);
  return cudaGetLastError();
}

cudaError_t net_conv_wgrad(const float* x, const float* dy, float* dw, float* db, float* scratch,
                           int B, int Ci, int Co, int n, int ks, cudaStream_t s) {
  int G, GB;
  wgrad_groups(B, Ci, Co, n, &G, &GB);
  const int64_t count = (int64_t)Co * Ci * ks * ks * ks;
  cudaError_t e;
  if (ks == 1) {
    constexpr int smem = 2 * 4 * 2 * NTV * (CT + 1);
    static PerDevice<bool> set;
    if ((e = raise_smem_limit(set, k_wgrad1, smem)) != cudaSuccess) return e;
    const dim3 grid(G, ((Ci + 15) / 16) * ((Co + CT - 1) / CT));
    k_wgrad1<<<grid, 256, smem, s>>>(x, dy, scratch, B, Ci, Co, n, G);
    e = cudaGetLastError();
  } else if (Ci > 8) {
    e = launch_wgrad3<16>(x, dy, scratch, B, Ci, Co, n, G, s);
  } else if (Ci > 4) {
    e = launch_wgrad3<8>(x, dy, scratch, B, Ci, Co, n, G, s);
  } else if (Ci > 2) {
    e = launch_wgrad3<4>(x, dy, scratch, B, Ci, Co, n, G, s);
  } else {
    e = launch_wgrad3<2>(x, dy, scratch, B, Ci, Co, n, G, s);
  }
  if (e != cudaSuccess) return e;
  k_wgrad_reduce<<<(unsigned)((count + 63) / 64), 64, 0, s>>>(scratch, dw, count, G);
  if (db) {
    float* partb = scratch + (size_t)G * count;
    k_bias_partial<<<dim3(Co, GB), 256, 0, s>>>(dy, partb, B, Co, n, GB);
    k_bias_reduce<<<(Co + 127) / 128, 128, 0, s>>>(partb, db, Co, GB);
  }
  return cudaGetLastError();
}

static bool aligned(const void* a, const void* b, size_t bytes) {
  return (((uintptr_t)a | (uintptr_t)b) & (bytes - 1)) == 0;
}

cudaError_t net_relu_bwd(float* dy, const float* y, int64_t count, cudaStream_t s) {
  const int64_t quads = aligned(dy, y, 16) ? count / 4 : 0;
  k_relu_bwd<<<gs(quads ? quads : count), 256, 0, s>>>(dy, y, count, quads);
  return cudaGetLastError();
}
cudaError_t net_pool_fwd(const float* x, float* y, int64_t BC, int n, cudaStream_t s) {
  const int m = n / 2;
  const VoxGrid g = vox_grid((int64_t)m * m * m, BC);
  k_gather<true><<<g.grid, 256, 0, s>>>(x, y, BC, 1, m, 1, 0, g.cpb, aligned(x, x, 8));
  return cudaGetLastError();
}
cudaError_t net_pool_bwd(const float* dy, float* dx, int64_t BC, int n, cudaStream_t s) {
  const int m = n / 2;
  const VoxGrid g = vox_grid((int64_t)m * m * m, BC);
  k_spread<true><<<g.grid, 256, 0, s>>>(dy, dx, BC, 1, m, 1, 0, g.cpb, aligned(dx, dx, 8));
  return cudaGetLastError();
}
cudaError_t net_up_fwd(const float* x, float* y, int B, int C, int m, int Cy, int coff,
                       cudaStream_t s) {
  const VoxGrid g = vox_grid((int64_t)m * m * m, (int64_t)B * C);
  k_spread<false><<<g.grid, 256, 0, s>>>(x, y, (int64_t)B * C, C, m, Cy, coff, g.cpb, aligned(y, y, 8));
  return cudaGetLastError();
}
cudaError_t net_up_bwd(const float* dy, float* dx, int B, int C, int m, int Cy, int coff,
                       cudaStream_t s) {
  const VoxGrid g = vox_grid((int64_t)m * m * m, (int64_t)B * C);
  k_gather<false><<<g.grid, 256, 0, s>>>(dy, dx, (int64_t)B * C, C, m, Cy, coff, g.cpb, aligned(dy, dy, 8));
  return cudaGetLastError();
}
cudaError_t net_copy_ch(const float* src, float* dst, int B, int C, int64_t nv, int Cs, int soff,
                        int Cd, int doff, int accumulate, cudaStream_t s) {
  const int64_t BC = (int64_t)B * C;
  if (nv % 4 == 0 && aligned(src, dst, 16)) {
    const VoxGrid g = vox_grid(nv / 4, BC);
    k_copy_ch<<<g.grid, 256, 0, s>>>((const float4*)src, (float4*)dst, BC, C, nv / 4, Cs, soff, Cd, doff,
                                     accumulate, g.cpb);
  } else {
    const VoxGrid g = vox_grid(nv, BC);
    k_copy_ch<<<g.grid, 256, 0, s>>>(src, dst, BC, C, nv, Cs, soff, Cd, doff, accumulate, g.cpb);
  }
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
