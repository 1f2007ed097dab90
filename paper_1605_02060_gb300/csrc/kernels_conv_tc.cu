// 3D convolution of the warm-start network on the tensor cores (tcgen05, sm_103a), as an
// implicit GEMM:
//     Y[b, co, v] = bias[co] + sum_{ci, t} X[b, ci, v + o(t)] W[co, ci, t]     (zero padding)
// with N = Co (padded to a multiple of 16) and K = Ci x taps walked as k-steps of 16 input
// channels at one tap t, channel groups outside, taps inside.
//
// M: rows are consecutive positions of the grid with its border of zeros (P = n + 2 per axis; the
// rows that fall on the border are computed and dropped, 6% at 64^3).  In that order a tap is a
// constant shift, so a CTA stages the R + 2 P + 2 positions that its R rows reach in each of the
// three z planes once per channel group, and a tap's A operand is the same shared memory from
// another start: in the K-major layout without swizzle a row of 8 channels is 16 bytes, rows lie
// 16 bytes apart, and a descriptor may start at any 16-byte address.  A voxel is then loaded,
// split and stored about 5 times per channel group, not 27 times (once per tap): the 27
// convolutions of a 64^3, batch 8 training step take 4.7 ms instead of 17.0 ms.
//
// The activations stay float32 [B][C][n^3]; the weights are bf16 [Co][Ci][taps].  A value is split
// into a bf16 hi and lo part (x = hi + lo to 16 mantissa bits), so the two products hi*W + lo*W
// give the FP32 activations times the bf16 weights to ~2^-17; accumulation is FP32 in TMEM.  A
// product of M = 128, K = 16 and N <= 32 takes 40 cycles (it is bound by reading A), 54 of them per
// row tile and channel group.
//
// One CTA: 256 threads stage, one of them issues the MMAs of a channel group, all wait for them
// (one buffer), and read the accumulators at the end.  Two CTAs per SM where shared memory allows:
// one stages while the other's products run.  (Weights fetched one 2-byte element at a time and
// positions decoded by division, 8 loads in flight: 10.4 ms.)
// Every wait is bounded: a timeout sets *err, marks the CTA's outputs NaN and returns.
#include <cuda_bf16.h>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace lddmm {

namespace {

constexpr int CV_THREADS = 256;
constexpr int CV_SMEM_CAP = 225 * 1024;

struct ConvArgs {
  const float* x;
  const __nv_bfloat16* w;
  const float* bias;
  float* y;
  int Ci, Co, Np, n;
  int taps, nph;        // filter taps; steps a channel group takes (1, or 3: a z plane each)
  int pad, P;           // border, n + 2 border
  int T, L;             // row tiles of 128 per CTA; positions staged per plane
  int nrb, nblk;        // blocks of T tiles in a sample, in all samples
  int wres;             // 1: the weights of all channel groups stay in shared memory
  int p_lo, p_hi;       // first and last position of a voxel
  int relu, accumulate, tcols;
  unsigned mP, mL;      // reciprocals of P and L (0: divide)
  int* err;
};

// bytes: positions of `planes` z planes, weights of `taps` taps (of all resident groups together)
inline int64_t cv_smem(int planes, int L, int64_t taps, int Np) {
  return 64 * (int64_t)planes * L + taps * Np * 32;
}

__device__ __forceinline__ uint32_t pack_bf2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// TPS taps a step: 27 (three z planes), 9 (one of the three) or 1 (a 1^3 filter).
template <int TPS>
__global__ void __launch_bounds__(CV_THREADS, 2) k_conv_tc(ConvArgs a) {
  constexpr int PL = TPS == 27 ? 3 : 1;
  extern __shared__ __align__(128) uint8_t cv_sm[];
  __shared__ __align__(8) uint64_t b_done;
  __shared__ uint32_t tmem_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = a.n, P = a.P;
  const size_t nv = (size_t)n * n * n;
  const int span = PL * a.L;                              // positions of a step's planes
  uint8_t* const bsm = cv_sm + 64 * span;

  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(&tmem_sh), (uint32_t)a.tcols);
    ptx::tmem_relinquish();
  }
  if (tid == 0) {
    ptx::mbar_init(ptx::smem_u32(&b_done), 1);
    ptx::fence_mbar_init();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = tmem_sh;

  // quotient by a divisor d with m = ceil(2^32 / d), exact while q d < 2^32 (the launch sees to it)
  auto quot = [](int q, int d, unsigned m) {
    return m ? (int)__umulhi((unsigned)q, m) : q / d;
  };
  // voxel offset of position p, -1 on the border or beyond
  auto voxel_at = [&](int p) -> int {
    if (p < 0) return -1;
    const int row = quot(p, P, a.mP), x = p - row * P - a.pad, zz = quot(row, P, a.mP);
    const int y = row - zz * P - a.pad, z = zz - a.pad;
    if (x < 0 || x >= n || y < 0 || y >= n || z < 0 || z >= n) return -1;
    return (z * n + y) * n + x;
  };

  // B: per tap [Np][16] in K-major core matrices (row co: 8 channels of half h at h 128 +
  // (co / 8) 256 + (co % 8) 16).  A thread collects 16-byte rows, the 8 loads of two in flight;
  // consecutive lanes take consecutive taps, which are contiguous in w.
  auto stage_weights = [&](int kc, int ph, uint8_t* wb) {
    for (int i0 = tid; i0 < a.Np * (2 * TPS); i0 += 2 * CV_THREADS) {
      uint16_t e[2][8];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = i0 + u * CV_THREADS, t = i % TPS, ch = i / TPS, co = ch >> 1;
        const bool in = co < a.Co && i < a.Np * (2 * TPS);
        const uint16_t* p = reinterpret_cast<const uint16_t*>(a.w) +
                            (in ? ((size_t)co * a.Ci + kc * 16 + (ch & 1) * 8) * a.taps + ph * TPS + t : 0);
#pragma unroll
        for (int j = 0; j < 8; ++j) e[u][j] = in ? __ldg(p + j * a.taps) : (uint16_t)0;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = i0 + u * CV_THREADS, t = i % TPS, ch = i / TPS, co = ch >> 1;
        if (i < a.Np * (2 * TPS))
          *reinterpret_cast<uint4*>(wb + (size_t)t * a.Np * 32 + (ch & 1) * 128 + (co >> 3) * 256 +
                                    (co & 7) * 16) =
              make_uint4(e[u][0] | (uint32_t)e[u][1] << 16, e[u][2] | (uint32_t)e[u][3] << 16,
                         e[u][4] | (uint32_t)e[u][5] << 16, e[u][6] | (uint32_t)e[u][7] << 16);
      }
    }
  };
  const int nst = a.Ci / 16 * a.nph, wbytes = TPS * a.Np * 32;
  bool ok = true;
  uint32_t step = 0;
  if (a.wres)
    for (int st = 0; st < nst; ++st) stage_weights(st / a.nph, st % a.nph, bsm + (size_t)st * wbytes);
  for (int blk = blockIdx.x; blk < a.nblk; blk += gridDim.x) {
    const int b = blk / a.nrb, p0 = a.p_lo + (blk - b * a.nrb) * (a.T * 128);   // position of row 0
    for (int st = 0; st < nst && ok; ++st, ++step) {
      const int kc = a.nph == 1 ? st : st / 3, ph = st - kc * a.nph;
      const int first = p0 + (a.taps > 1 ? (ph - 1) * P * P - P - 1 : 0);
      uint8_t* const wb = bsm + (a.wres ? (size_t)st * wbytes : 0);
      // ------------------------------------------------------------ staging
      if (!a.wres) stage_weights(kc, ph, wb);
      // A: [hi, lo][8-channel half][plane][position] of 16 bytes; a thread takes all 16 channels of a
      // position, 16 loads in flight
      const float* xb = a.x + ((size_t)b * a.Ci + kc * 16) * nv;
      for (int i = tid; i < span; i += CV_THREADS) {
        const int sp = PL == 1 ? 0 : quot(i, a.L, a.mL);
        const int o = voxel_at(first + sp * P * P + (i - sp * a.L));
        const float* p = xb + (o < 0 ? 0 : o);
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = o >= 0 ? __ldg(p + (size_t)j * nv) : 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t hw[4], lw[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float f0 = v[8 * h + 2 * j], f1 = v[8 * h + 2 * j + 1];
            hw[j] = pack_bf2(f0, f1);
            lw[j] = pack_bf2(f0 - __uint_as_float(hw[j] << 16), f1 - __uint_as_float(hw[j] & 0xffff0000u));
          }
          *reinterpret_cast<uint4*>(cv_sm + (size_t)(h * span + i) * 16) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
          *reinterpret_cast<uint4*>(cv_sm + (size_t)((2 + h) * span + i) * 16) =
              make_uint4(lw[0], lw[1], lw[2], lw[3]);
        }
      }
      ptx::fence_proxy_async_smem();
      __syncthreads();
      // ------------------------------------------------------------ products of the channel group
      if (tid == 0) {
        ptx::tc_fence_after();
        const uint32_t id = ptx::idesc_bf16(128, a.Np);
        const uint32_t sa = ptx::smem_u32(cv_sm), sb = ptx::smem_u32(wb);
        const uint64_t dA = ptx::smem_desc(sa, (uint32_t)span * 16u, 128);
        const uint64_t dB = ptx::smem_desc(sb, 128, 256);
        const uint32_t lo = 2u * (uint32_t)span;            // 16-byte units to the lo halves
        for (int t = 0; t < TPS; ++t) {
          // the tap's first row and its weights, in 16-byte units
          const int ox = t % 3, oy = t / 3 % 3, oz = t / 9;
          const uint64_t at = dA + (uint32_t)(oz * a.L + oy * P + ox), bt = dB + (uint32_t)(t * 2 * a.Np);
          for (int m = 0; m < a.T; ++m) {
            const uint32_t d = tmem + (uint32_t)(m * a.Np);
            const uint64_t am = at + 128u * (uint32_t)m;
            ptx::mma_bf16(d, am, bt, id, (st | t) ? 1u : 0u);
            ptx::mma_bf16(d, am + lo, bt, id, 1u);
          }
        }
        ptx::mma_commit(ptx::smem_u32(&b_done));
      }
      ok = ptx::mbar_wait(ptx::smem_u32(&b_done), step & 1u);
      ok = __syncthreads_and(ok);
    }
    ptx::tc_fence_after();
    // ------------------------------------------------------------ epilogue
    // warp w reads TMEM lanes 32 (w % 4)..; the two halves of the warps take alternate 16-column chunks
    const int q = warp & 3, half = warp >> 2, nch = a.Np / 16;
    for (int m = 0; m < a.T; ++m) {
      const int p = p0 + m * 128 + q * 32 + lane;
      const int vo = p <= a.p_hi ? voxel_at(p) : -1;
      for (int c = half; c < nch; c += 2) {
        float acc[16];
        if (ok) {
          ptx::tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(m * a.Np + c * 16), acc);
        } else {
          // a wait gave up: the outputs are marked invalid besides the error flag
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[j] = __int_as_float(0x7fc00000);
        }
        if (vo < 0) continue;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int co = c * 16 + j;
          if (co < a.Co) {
            float* o = a.y + ((size_t)b * a.Co + co) * nv + vo;
            float r = acc[j] + (a.bias ? __ldg(a.bias + co) : 0.f);
            if (a.accumulate) r += *o;
            if (a.relu && ok) r = fmaxf(r, 0.f);
            *o = r;
          }
        }
      }
    }
    // the accumulators are read before the next block's products write them
    ptx::tc_fence_before();
    __syncthreads();
  }
  // the products of an abandoned wait have finished (or are given another bounded wait) before TMEM
  // is freed
  if (warp == 0) {
    if (!ok && lane == 0) {
      ptx::mbar_wait(ptx::smem_u32(&b_done), (step - 1u) & 1u);
      if (a.err) atomicExch(a.err, 3);
    }
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, (uint32_t)a.tcols);
  }
}

}  // namespace

// (positions with the border are 32-bit: n up to 1288)
bool conv_tc_supported(int Ci, int Co, int n) {
  return Ci % 16 == 0 && Co >= 1 && Co <= 256 && n <= 1280;
}

// Device flag a tensor-core convolution sets when one of its bounded waits gave up (its tile's
// outputs are then NaN); allocated once per process.
static int* conv_err_flag() {
  static int* f = nullptr;
  if (!f && cudaMalloc((void**)&f, sizeof(int)) == cudaSuccess) cudaMemset(f, 0, sizeof(int));
  else cudaGetLastError();
  return f;
}

template <int TPS>
static cudaError_t launch_conv(const ConvArgs& a, int B, cudaStream_t s) {
  static const cudaError_t set = cudaFuncSetAttribute(
      k_conv_tc<TPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, CV_SMEM_CAP);
  if (set != cudaSuccess) return set;
  // persistent: two CTAs per SM share the blocks (the weights are staged once per CTA)
  const int smem = (int)cv_smem(TPS == 27 ? 3 : 1, a.L, TPS * (a.wres ? a.Ci / 16 * a.nph : 1), a.Np);
  const int grid = a.nblk < 304 ? a.nblk : 304;
  k_conv_tc<TPS><<<grid, CV_THREADS, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t conv_tc_fwd(const float* x, const void* w, const float* bias, float* y, int B, int Ci,
                        int Co, int n, int ks, int relu, int accumulate, cudaStream_t s) {
  ConvArgs a{};
  a.x = x; a.w = (const __nv_bfloat16*)w; a.bias = bias; a.y = y;
  a.Ci = Ci; a.Co = Co; a.n = n;
  a.Np = (Co + 15) / 16 * 16;
  a.taps = ks * ks * ks;
  a.pad = ks / 2;
  a.P = n + 2 * a.pad;
  a.relu = relu; a.accumulate = accumulate;
  a.err = conv_err_flag();
  a.p_lo = a.pad * (a.P * a.P + a.P + 1);
  a.p_hi = (n - 1 + a.pad) * (a.P * a.P + a.P + 1);
  const int halo = a.pad ? 2 * a.P + 2 : 0;
  // Row tiles per CTA: the more, the fewer border positions are staged twice (1.35 a row with three
  // at 64^3, 2.05 with one), as long as two CTAs fit an SM (115,000 bytes, 256 TMEM columns each)
  // and there are two for every SM; all taps of a channel group in one step, else plane by plane
  // (wide layers, and grids past 380^3).
  const int64_t rows = (int64_t)(a.p_hi - a.p_lo + 1) * B;
  const int nkc = Ci / 16;
  const auto fits = [&](int T, int nph, int64_t groups, int cap) {
    const int L = 128 * T + halo;
    return T * a.Np <= 256 &&
           cv_smem(ks == 1 ? 1 : 3 / nph, L, ks == 1 ? groups : 27 / nph * groups, a.Np) <= cap;
  };
  a.T = 1;
  a.nph = 1;
  bool found = false;
  for (int T = 3; T >= 1 && !found; --T) {
    if (T > 1 && rows < (int64_t)128 * T * 304) continue;
    for (int res = 1; res >= 0 && !found; --res)
      if (fits(T, 1, res ? nkc : 1, 115000)) {
        a.T = T;
        a.wres = res;
        found = true;
      }
  }
  if (!found && !fits(1, 1, 1, CV_SMEM_CAP)) {
    a.nph = 3;
    if (ks == 1 || !fits(1, 3, 1, CV_SMEM_CAP)) return cudaErrorInvalidValue;
  }
  a.L = 128 * a.T + halo;
  a.nrb = (a.p_hi - a.p_lo + 128 * a.T) / (128 * a.T);
  a.nblk = a.nrb * B;
  // positions stay below 2 P^3 and staged ones below 2^16: where the reciprocals are exact
  const auto recip = [](unsigned d) { return (unsigned)(((1ull << 32) + d - 1) / d); };
  a.mP = a.P > 1 && a.P <= 200 ? recip(a.P) : 0u;
  a.mL = recip(a.L);
  a.tcols = 32;
  while (a.tcols < a.T * a.Np) a.tcols <<= 1;
  if (ks == 1) return launch_conv<1>(a, B, s);
  return a.nph == 1 ? launch_conv<27>(a, B, s) : launch_conv<9>(a, B, s);
}

}  // namespace lddmm
