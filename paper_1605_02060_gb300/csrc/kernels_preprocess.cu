// Preprocessing of §2.2 on the GPU.
//
// Image-LDDMM: the masks are applied to I0 and I1, and the masked I0 is histogram-matched to the
// masked I1.  Both images get a `bins`-bin histogram of their in-mask voxels over [min, max];
// `points` quantiles at k / (points + 1) are read off the cumulative counts (interpolated inside
// the bin that reaches the fraction); min maps to min, max to max, each quantile of I0 to the
// same quantile of I1, linearly in between and along the end segments beyond.
//
// Mask generation: [I > threshold], opened with a ball of radius r_open (erosion, then
// dilation), then closed with a ball of radius r_close (dilation, then erosion); voxels beyond
// the grid count as background.
//
// The histogram counts are integers (exact), and every floating-point step of the quantiles and
// of the map is FP64 with explicitly rounded operations, in the order of the definition above.
#include "kernels.h"

namespace lddmm {

namespace {

__device__ __forceinline__ int ord_of(float f) {
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float float_of(int i) {
  return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff);
}
// Range of an image over its mask in unsigned order (0 = no voxel yet): inv_min is the complement
// of the minimum's code, so that zeroed memory starts both.
struct Range {
  unsigned inv_min, max, count, pad;
};
__device__ __forceinline__ unsigned code_of(float f) { return (unsigned)ord_of(f) ^ 0x80000000u; }
__device__ __forceinline__ double lo_of(const Range& r) {
  return (double)float_of((int)(~r.inv_min ^ 0x80000000u));
}
__device__ __forceinline__ double hi_of(const Range& r) {
  return (double)float_of((int)(r.max ^ 0x80000000u));
}

struct Pair2 {
  const float* I[2];
  const float* M[2];
};

// Calls f(value) for the in-mask voxels of this thread's share: 16-byte loads, four per array
// requested before the first value is used, when both arrays are aligned.
template <typename F>
__device__ __forceinline__ void each_masked(const float* I, const float* M, int64_t n, F f) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x,
                st = (int64_t)gridDim.x * blockDim.x;
  int64_t done = 0;
  if ((((uintptr_t)I | (uintptr_t)M) & 15) == 0) {
    const int64_t n4 = n / 4;
    const float4* I4 = reinterpret_cast<const float4*>(I);
    const float4* M4 = reinterpret_cast<const float4*>(M);
    for (int64_t i = t; i < n4; i += 4 * st) {
      float4 m[4], v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const bool in = i + k * st < n4;
        m[k] = in ? __ldg(M4 + i + k * st) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[k] = in ? __ldg(I4 + i + k * st) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (m[k].x > 0.5f) f(v[k].x);
        if (m[k].y > 0.5f) f(v[k].y);
        if (m[k].z > 0.5f) f(v[k].z);
        if (m[k].w > 0.5f) f(v[k].w);
      }
    }
    done = n4 * 4;
  }
  for (int64_t i = done + t; i < n; i += st)
    if (M[i] > 0.5f) f(I[i]);
}

__global__ void __launch_bounds__(512) k_masked_range(Pair2 p, int64_t n, Range* rg) {
  __shared__ Range red[16];
  Range* out = rg + blockIdx.y;
  unsigned a = 0, b = 0, c = 0;
  each_masked(p.I[blockIdx.y], p.M[blockIdx.y], n, [&](float v) {
    const unsigned u = code_of(v);
    a = max(a, ~u);
    b = max(b, u);
    ++c;
  });
  for (int o = 16; o; o >>= 1) {
    a = max(a, __shfl_xor_sync(0xffffffffu, a, o));
    b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = Range{a, b, c, 0u};
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 16; ++w) {
      a = max(a, red[w].inv_min);
      b = max(b, red[w].max);
      c += red[w].count;
    }
    if (c) {
      atomicMax(&out->inv_min, a);
      atomicMax(&out->max, b);
      atomicAdd(&out->count, c);
    }
  }
}

__device__ __forceinline__ int bin_of(double v, double lo, double w, int bins) {
  if (w <= 0.0) return 0;
  const int b = (int)floor(__ddiv_rn(__dsub_rn(v, lo), w));
  return min(max(b, 0), bins - 1);
}

// counts[image][bins].  The bin is floor((v - lo) / w) of the FP64 quotient; FP64 division sets the
// pace when every voxel takes it (68 us per image at 264x160x228, 48 us for both this way), so the
// quotient is first formed in FP32 (three roundings, off by less than 1.8e-7 of itself), and only a
// voxel whose FP32 quotient lies within 2.5e-7 bins of a whole number (or is not a small finite
// one) takes the FP64 form.  Neighbouring voxels often share a bin: a thread adds runs.
__global__ void __launch_bounds__(512) k_masked_hist(Pair2 p, int64_t n, const Range* rg, int bins,
                                                     unsigned long long* counts) {
  extern __shared__ unsigned int sh[];
  if (rg[0].count == 0 || rg[1].count == 0) return;
  for (int b = threadIdx.x; b < bins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const Range r = rg[blockIdx.y];
  const double lo = lo_of(r), hi = hi_of(r);
  const double w = __ddiv_rn(__dsub_rn(hi, lo), (double)bins);
  const float lof = (float)lo, iw = (float)(1.0 / w);
  // (no short cut where the width or its reciprocal could be subnormal or overflow)
  const float tol = w > 1e-30 && w < 1e30 ? 2.5e-7f * (float)bins : 2.f;
  int cur = 0;
  unsigned run = 0;
  each_masked(p.I[blockIdx.y], p.M[blockIdx.y], n, [&](float v) {
    const float q = (v - lof) * iw, f = floorf(q), d = q - f;
    int b;
    if (d > tol && d < 1.f - tol && q > 0.f && q < 1.5f * (float)bins) b = min(max((int)f, 0), bins - 1);
    else b = bin_of((double)v, lo, w, bins);
    if (b != cur) {
      if (run) atomicAdd(&sh[cur], run);
      cur = b;
      run = 0;
    }
    ++run;
  });
  if (run) atomicAdd(&sh[cur], run);
  __syncthreads();
  for (int b = threadIdx.x; b < bins; b += blockDim.x)
    if (sh[b]) atomicAdd(&counts[(size_t)blockIdx.y * bins + b], (unsigned long long)sh[b]);
}

__device__ double quantile(const unsigned long long* c, int bins, double lo, double hi, double n,
                           double f) {
  const double w = __ddiv_rn(__dsub_rn(hi, lo), (double)bins);
  if (w <= 0.0) return lo;
  const double t = __dmul_rn(f, n);
  double C = 0.0, prev = 0.0;
  int k = bins - 1;
  for (int b = 0; b < bins; ++b) {
    prev = C;
    C = __dadd_rn(C, (double)c[b]);
    if (C >= t) {
      k = b;
      break;
    }
  }
  if (k == bins - 1 && C < t) {            // not reached (rounding): the last bin
    prev = __dsub_rn(C, (double)c[bins - 1]);
  }
  if (c[k] == 0) return __dadd_rn(lo, __dmul_rn(w, (double)k));
  return __dadd_rn(lo, __dmul_rn(w, __dadd_rn((double)k, __ddiv_rn(__dsub_rn(t, prev), (double)c[k]))));
}

// nodes[0..P+1] = x (source), nodes[P+2..2P+3] = y (reference), P = points.  A thread per quantile.
__global__ void __launch_bounds__(160) k_match_nodes(const Range* rg,
                                                     const unsigned long long* counts, int bins,
                                                     int points, double* nodes) {
  extern __shared__ unsigned long long cs[];
  if (rg[0].count == 0 || rg[1].count == 0) return;
  for (int b = threadIdx.x; b < 2 * bins; b += blockDim.x) cs[b] = counts[b];
  __syncthreads();
  const int m = points + 2;
  for (int k = threadIdx.x; k < 2 * m; k += blockDim.x) {
    const int im = k / m, q = k - im * m;
    const Range r = rg[im];
    const double lo = lo_of(r), hi = hi_of(r);
    nodes[k] = q == 0       ? lo
               : q == m - 1 ? hi
                            : quantile(cs + (size_t)im * bins, bins, lo, hi, (double)r.count,
                                       __ddiv_rn((double)q, (double)(points + 1)));
  }
}

// The map is FP64: y_k + (v - x_k) * slope_k.  The node search is exact in FP32 (v is a float, so
// x_k <= v just when the smallest float not below x_k is), the slopes are formed once per block,
// and only in-mask voxels reach the three FP64 operations (264x160x228: 103 -> 43 us).
__global__ void __launch_bounds__(256) k_apply_match(const float* I0, const float* __restrict__ M0,
                                                     int64_t n, const Range* rg,
                                                     const double* __restrict__ nodes, int m,
                                                     float* out) {
  __shared__ double xs[66], ys[66], sl[66];
  __shared__ float xf[66];
  if (rg[0].count == 0 || rg[1].count == 0) return;    // an empty mask: out stays as it was
  for (int k = threadIdx.x; k < m; k += blockDim.x) {
    xs[k] = nodes[k];
    ys[k] = nodes[m + k];
    xf[k] = __double2float_ru(xs[k]);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < m - 1; k += blockDim.x) {
    const double dx = __dsub_rn(xs[k + 1], xs[k]);
    sl[k] = dx > 0.0 ? __ddiv_rn(__dsub_rn(ys[k + 1], ys[k]), dx) : 0.0;
  }
  __syncthreads();
  auto map = [&](float v) {
    int k = 0;                                // last node with x <= v, kept inside [0, m-2]
    for (int j = 1; j < m - 1; ++j)
      if (xf[j] <= v) k = j;
    return (float)__dadd_rn(ys[k], __dmul_rn(__dsub_rn((double)v, xs[k]), sl[k]));
  };
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x,
                st = (int64_t)gridDim.x * blockDim.x;
  int64_t done = 0;
  if ((((uintptr_t)I0 | (uintptr_t)M0 | (uintptr_t)out) & 15) == 0) {
    const int64_t n4 = n / 4;
    for (int64_t i = t; i < n4; i += 2 * st) {
      float4 g[2], v[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const bool in = i + k * st < n4;
        g[k] = in ? __ldg(reinterpret_cast<const float4*>(M0) + i + k * st) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[k] = in ? reinterpret_cast<const float4*>(I0)[i + k * st] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
        if (g[k].x > 0.5f) r.x = map(v[k].x);
        if (g[k].y > 0.5f) r.y = map(v[k].y);
        if (g[k].z > 0.5f) r.z = map(v[k].z);
        if (g[k].w > 0.5f) r.w = map(v[k].w);
        if (i + k * st < n4) reinterpret_cast<float4*>(out)[i + k * st] = r;
      }
    }
    done = n4 * 4;
  }
  for (int64_t i = done + t; i < n; i += st) out[i] = M0[i] > 0.5f ? map(I0[i]) : 0.f;
}

// ---- masks as bits: row (z, y) of the grid is W = ceil(nx / 32) words, bit i of word j is voxel
// 32 j + i, the bits past nx are 0.  A ball's row at (dz, dy) is a run of 2 w + 1 voxels: the rows
// of one half width w are ORed first (three loads and ORs a row, whatever the radius), then
// spread by w once.  An erosion is the complement of a dilation of the complement, in which
// everything beyond the grid is set.  32 voxels cost what one did: the four operations of an
// opening by 1 and a closing by 3 at 264x160x228 take 47 us instead of 2411 us on bytes (74 us
// when every row was spread).
__global__ void __launch_bounds__(256) k_threshold_bits(const float* __restrict__ I, int nx, int W,
                                                        int64_t rows, float t,
                                                        uint32_t* __restrict__ out) {
  // a warp takes 8 consecutive words: their loads are in flight together
  const int64_t i0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 8, n = rows * W;
  const int lane = threadIdx.x & 31;
  if (i0 >= n) return;
  int64_t row = i0 / W;
  int j = (int)(i0 - row * W);
  float v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int x = j * 32 + lane;
    // what lies beyond the row or the grid compares false
    v[k] = i0 + k < n && x < nx ? __ldg(I + row * nx + x) : __int_as_float(0x7fc00000);
    if (++j == W) {
      j = 0;
      ++row;
    }
  }
  uint32_t mine = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const unsigned b = __ballot_sync(0xffffffffu, v[k] > t);
    if (lane == k) mine = b;
  }
  if (lane < 8 && i0 + lane < n) out[i0 + lane] = mine;
}

struct BallRows {
  uint16_t end[18];            // rows of half width w end at end[w + 1], begin at end[w]
  int8_t dz[33 * 33], dy[33 * 33];
};

// bit i of the result = OR of bits i - w .. i + w of the row, w <= 16 (l, c, r: the words to the
// left, at and to the right)
__device__ __forceinline__ uint32_t spread(uint32_t l, uint32_t c, uint32_t r, int w) {
  // bits -16 .. 47 of the row, then an OR over runs of 2 w + 1 bits by doubling
  uint64_t e = (uint64_t)(l >> 16) | (uint64_t)c << 16 | (uint64_t)r << 48;
  const int len = 2 * w + 1;
  int k = 1;
  for (; 2 * k <= len; k *= 2) e |= e >> k;
  e |= e >> (len - k);
  return (uint32_t)(e >> (16 - w));
}

template <bool ERODE>
__global__ void __launch_bounds__(256) k_ball_bits(const uint32_t* __restrict__ in, int nx, int ny,
                                                   int nz, int W, int r,
                                                   const __grid_constant__ BallRows br,
                                                   uint32_t* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)ny * nz * W) return;
  const int64_t row = i / W;
  const int j = (int)(i - row * W), z = (int)(row / ny), y = (int)(row - (int64_t)z * ny);
  uint32_t acc = 0;
  for (int w = 0; w <= r; ++w) {
    uint32_t l = 0, c = 0, g = 0;
#pragma unroll 4
    for (int k = br.end[w]; k < br.end[w + 1]; ++k) {
      const int zz = z + br.dz[k], yy = y + br.dy[k];
      const bool in_grid = zz >= 0 && zz < nz && yy >= 0 && yy < ny;
      const uint32_t* p = in + (in_grid ? (int64_t)zz * ny + yy : row) * W + j;
      const uint32_t pc = __ldg(p), pl = j > 0 ? __ldg(p - 1) : 0u, pr = j + 1 < W ? __ldg(p + 1) : 0u;
      if (ERODE) {
        // complements are set beyond the grid: past both ends of a row the stored bits are 0
        l |= in_grid ? ~pl : ~0u;
        c |= in_grid ? ~pc : ~0u;
        g |= in_grid ? ~pr : ~0u;
      } else if (in_grid) {
        l |= pl;
        c |= pc;
        g |= pr;
      }
    }
    if (l | c | g) acc |= spread(l, c, g, w);
    if (acc == ~0u) break;
  }
  const int left = nx - 32 * j;
  const uint32_t valid = left >= 32 ? ~0u : (1u << left) - 1u;
  out[i] = (ERODE ? ~acc : acc) & valid;
}

// bits -> bytes 0 / 1: four voxels per thread where rows and out allow 4-byte stores
__global__ void __launch_bounds__(256) k_unpack_bits(const uint32_t* __restrict__ in, int nx, int W,
                                                     int64_t rows, int vec, uint8_t* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (vec) {
    const int q = nx / 4;
    if (i >= rows * q) return;
    const int64_t row = i / q;
    const int x = (int)(i - row * q) * 4;
    const uint32_t nib = (__ldg(in + row * W + (x >> 5)) >> (x & 31)) & 15u;
    reinterpret_cast<uint32_t*>(out)[i] = (nib * 0x00204081u) & 0x01010101u;
  } else {
    if (i >= rows * nx) return;
    const int64_t row = i / nx;
    const int x = (int)(i - row * nx);
    out[i] = (uint8_t)((__ldg(in + row * W + (x >> 5)) >> (x & 31)) & 1u);
  }
}

int grid_1d(int64_t n) {
  const int64_t b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

}  // namespace

size_t match_scratch_bytes(int bins) {
  return 2 * sizeof(Range) + 2 * (size_t)bins * sizeof(unsigned long long) + 2 * 66 * sizeof(double);
}

cudaError_t histogram_match(const float* I0, const float* M0, const float* I1, const float* M1,
                            int64_t n, int bins, int points, void* scratch, float* out,
                            cudaStream_t s) {
  Range* rg = reinterpret_cast<Range*>(scratch);
  unsigned long long* counts = reinterpret_cast<unsigned long long*>(rg + 2);
  double* nodes = reinterpret_cast<double*>(counts + 2 * (size_t)bins);
  cudaError_t e = cudaMemsetAsync(scratch, 0, match_scratch_bytes(bins), s);
  if (e != cudaSuccess) return e;
  const Pair2 p{{I0, I1}, {M0, M1}};
  const int64_t nb = (n + 2047) / 2048;        // 512 threads x 4 voxels
  const dim3 grid((unsigned)(nb < 152 * 2 ? nb : 152 * 2), 2);   // one wave of 4 blocks per SM
  k_masked_range<<<grid, 512, 0, s>>>(p, n, rg);
  k_masked_hist<<<grid, 512, (size_t)bins * sizeof(unsigned int), s>>>(p, n, rg, bins, counts);
  k_match_nodes<<<1, 160, 2 * (size_t)bins * sizeof(unsigned long long), s>>>(rg, counts, bins,
                                                                              points, nodes);
  k_apply_match<<<grid_1d((n + 3) / 4), 256, 0, s>>>(I0, M0, n, rg, nodes, points + 2, out);
  return cudaGetLastError();
}

int64_t mask_bits_words(int nx, int ny, int nz) { return (int64_t)ny * nz * ((nx + 31) / 32); }

cudaError_t threshold_bits(const float* I, int nx, int ny, int nz, float t, uint32_t* out,
                           cudaStream_t s) {
  const int W = (nx + 31) / 32;
  const int64_t rows = (int64_t)ny * nz;
  k_threshold_bits<<<(unsigned)((rows * W + 63) / 64), 256, 0, s>>>(I, nx, W, rows, t, out);
  return cudaGetLastError();
}

cudaError_t ball_bits(int nx, int ny, int nz, const uint32_t* in, int r, bool erode, uint32_t* out,
                      cudaStream_t s) {
  const int W = (nx + 31) / 32;
  const int64_t words = mask_bits_words(nx, ny, nz);
  BallRows br;
  int k = 0;
  br.end[0] = 0;
  for (int w = 0; w <= r; ++w) {
    for (int dz = -r; dz <= r; ++dz)
      for (int dy = -r; dy <= r; ++dy) {
        const int d = r * r - dz * dz - dy * dy;       // half width w: w^2 <= d < (w + 1)^2
        if (w * w <= d && d < (w + 1) * (w + 1)) {
          br.dz[k] = (int8_t)dz;
          br.dy[k++] = (int8_t)dy;
        }
      }
    br.end[w + 1] = (uint16_t)k;
  }
  const unsigned nb = (unsigned)((words + 255) / 256);
  if (erode) k_ball_bits<true><<<nb, 256, 0, s>>>(in, nx, ny, nz, W, r, br, out);
  else k_ball_bits<false><<<nb, 256, 0, s>>>(in, nx, ny, nz, W, r, br, out);
  return cudaGetLastError();
}

cudaError_t unpack_bits(int nx, int ny, int nz, const uint32_t* in, uint8_t* out, cudaStream_t s) {
  const int W = (nx + 31) / 32;
  const int64_t rows = (int64_t)ny * nz;
  const int vec = nx % 4 == 0 && ((uintptr_t)out & 3) == 0;
  const int64_t t = vec ? rows * (nx / 4) : rows * nx;
  k_unpack_bits<<<(unsigned)((t + 255) / 256), 256, 0, s>>>(in, nx, W, rows, vec, out);
  return cudaGetLastError();
}

}  // namespace lddmm
