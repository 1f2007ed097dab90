// Warm-start support: resampling fields between grids of the same box, and scaling a field.
//
// The learned warm start runs its network on a coarse n^3 grid that covers the whole box
// (an anisotropic resample of the registration grid), so the masks go down to n^3 and the
// predicted velocity comes back up to the registration grid.  Both use trilinear interpolation
// at cell-centred coordinates (voxel i of a grid of size d covers [i, i + 1) in units of the box
// divided by d): q = (i + 0.5) s / d - 0.5 in source voxels, clamped to the source grid.
// A velocity in voxels of the coarse grid becomes one in voxels of the fine grid by the ratio of
// the sizes along its own axis, so component c of a vector field is multiplied by scale[c].
#include "../../include/lddmm.h"
#include "kernels.h"

namespace lddmm {

namespace {

// The sample coordinate is formed in double precision (the ratio s/d is not a float), so the
// interpolation weight carries no error beyond its final rounding to float.
__device__ __forceinline__ void axis_weight(double q, int n, int& i0, float& t) {
  q = fmin(fmax(q, 0.0), (double)(n - 1));
  int i = (int)floor(q);
  if (i > n - 2) i = n - 2;
  if (i < 0) i = 0;
  i0 = i;
  t = n > 1 ? (float)(q - (double)i) : 0.f;
}

// A block makes a tile of W x H destination columns (W H = 256, W a power of two) and `zstep` of
// their planes, of one field of [nfields][dz][dy][dx].  FP64 runs at 2 FMAs a clock and SM here, so
// the double coordinates are formed once per axis position and block and read from shared memory
// (the ratios rx, ry, rz of the sizes once per call); a thread then walks up z and keeps the two
// bilinear values its sample lies between, so going up in size it reads the source only when it
// enters a new pair of planes.  32^3 -> 264x160x228 with 3 components takes 45 us, 17 of them for
// the stores alone (1500 us with all coordinates per voxel); going down to 32^3, where eight loads
// in a row are all there is, 7 us.  Each value comes from the same operations in the same order as
// a voxel by itself would take.
constexpr int RS_THREADS = 256, RS_ZMAX = 16;
__global__ void __launch_bounds__(RS_THREADS) k_resample(const float* __restrict__ src, int sx, int sy,
                                                         int sz, float* __restrict__ dst, int dx,
                                                         int dy, int dz, int ncomp, float s0, float s1,
                                                         float s2, double rx, double ry, double rz,
                                                         int lw, int zstep, int tx_n, long long txy,
                                                         long long tiles_f, long long tiles) {
  __shared__ int ib[RS_THREADS + 1 + RS_ZMAX];         // W + H <= 257
  __shared__ float tb[RS_THREADS + 1 + RS_ZMAX];
  const int W = 1 << lw, H = RS_THREADS >> lw, tid = threadIdx.x;
  const int lx = tid & (W - 1), ly = tid >> lw;
  const long long sp = (long long)sx * sy, dp = (long long)dx * dy;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    const long long f = t / tiles_f, r = t - f * tiles_f, zi = r / txy;
    const long long q = r - zi * txy, yi = q / tx_n;
    const int x0 = (int)(q - yi * tx_n) << lw, y0 = (int)yi * H, z0 = (int)zi * zstep;
    const int nz = min(zstep, dz - z0);
    // W + H + zstep axis positions: [x | y | z]
    for (int i = tid; i < W + H + zstep; i += RS_THREADS) {
      if (i < W)
        axis_weight(((double)x0 + i + 0.5) * rx - 0.5, sx, ib[i], tb[i]);
      else if (i < W + H)
        axis_weight(((double)y0 + (i - W) + 0.5) * ry - 0.5, sy, ib[i], tb[i]);
      else
        axis_weight(((double)z0 + (i - W - H) + 0.5) * rz - 0.5, sz, ib[i], tb[i]);
    }
    __syncthreads();
    const int x = x0 + lx, y = y0 + ly;
    if (x < dx && y < dy) {
      const int jx = ib[lx], jy = ib[W + ly];
      const float tx = tb[lx], ty = tb[W + ly];
      const float* s = src + f * sp * sz + (long long)jy * sx + jx;
      const int ox = sx > 1 ? 1 : 0;
      const long long oy = sy > 1 ? sx : 0;
      const int comp = (int)(f % ncomp);
      const float sc = comp == 0 ? s0 : comp == 1 ? s1 : s2;
      float* d = dst + (f * dz + z0) * dp + (long long)y * dx + x;
      auto plane = [&](int z) {
        const float* p = s + z * sp;
        const float a0 = __ldg(p), a1 = __ldg(p + ox), b0 = __ldg(p + oy), b1 = __ldg(p + oy + ox);
        const float c0 = a0 + tx * (a1 - a0), c1 = b0 + tx * (b1 - b0);
        return c0 + ty * (c1 - c0);
      };
      int zc = -2;                      // lower plane of the pair (c0, c1)
      float c0 = 0.f, c1 = 0.f;
      for (int k = 0; k < nz; ++k, d += dp) {
        const int jz = ib[W + H + k];
        const float tz = tb[W + H + k];
        if (jz != zc) {
          c0 = jz == zc + 1 ? c1 : plane(jz);
          c1 = sz > 1 ? plane(jz + 1) : c0;
          zc = jz;
        }
        *d = sc * (c0 + tz * (c1 - c0));
      }
    }
    __syncthreads();
  }
}

__global__ void k_scale(float* __restrict__ x, long long n, float c) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    x[i] *= c;
}

int grid_for(long long n) {
  const long long b = (n + 255) / 256;
  return (int)(b < 152 * 32 ? (b > 0 ? b : 1) : 152 * 32);
}

}  // namespace

}  // namespace lddmm

using namespace lddmm;

extern "C" {

int lddmm_resample(const float* src, int sx, int sy, int sz, float* dst, int dx, int dy, int dz,
                   int nfields, int ncomp, float s0, float s1, float s2, void* stream) {
  if (!src || !dst || sx < 1 || sy < 1 || sz < 1 || dx < 1 || dy < 1 || dz < 1 || nfields < 1 ||
      (ncomp != 1 && ncomp != 3) || nfields % ncomp)
    return LDDMM_ERR_INVALID_ARG;
  if ((long long)dx * dy * dz * nfields > (1LL << 40)) return LDDMM_ERR_INVALID_ARG;
  // tiles 32 x 8 columns, wider or taller where an axis is shorter than that; 16 planes a block, fewer
  // until there are eight blocks for every SM (going down to 32^3 there is little but latency)
  int lw = 5;
  while (lw < 8 && dy <= (RS_THREADS >> (lw + 1))) ++lw;
  while (lw > 0 && dx <= (1 << (lw - 1))) --lw;
  const int tx_n = (int)(((long long)dx + (1 << lw) - 1) >> lw), h = RS_THREADS >> lw;
  const long long txy = tx_n * (((long long)dy + h - 1) / h);
  int zstep = RS_ZMAX;
  const auto tiles_of = [&](int step) { return txy * (((long long)dz + step - 1) / step); };
  while (zstep > 1 && (zstep >= 2LL * dz || tiles_of(zstep) * nfields < 152 * 8)) zstep /= 2;
  const long long tiles_f = tiles_of(zstep), tiles = tiles_f * nfields;
  const unsigned grid = (unsigned)(tiles < (1 << 30) ? tiles : 1 << 30);
  k_resample<<<grid, RS_THREADS, 0, (cudaStream_t)stream>>>(src, sx, sy, sz, dst, dx, dy, dz, ncomp, s0,
                                                            s1, s2, (double)sx / dx, (double)sy / dy,
                                                            (double)sz / dz, lw, zstep, tx_n, txy,
                                                            tiles_f, tiles);
  return cudaGetLastError() == cudaSuccess ? LDDMM_OK : LDDMM_ERR_CUDA;
}

int lddmm_scale(float* x, int64_t count, float c, void* stream) {
  if (!x || count < 0) return LDDMM_ERR_INVALID_ARG;
  if (count == 0) return LDDMM_OK;
  k_scale<<<grid_for(count), 256, 0, (cudaStream_t)stream>>>(x, count, c);
  return cudaGetLastError() == cudaSuccess ? LDDMM_OK : LDDMM_ERR_CUDA;
}

}  // extern "C"
