// 3D convolution of the warm-start network on the tensor cores (tcgen05, sm_103a), as an
// implicit GEMM:
//     Y[b, co, v] = bias[co] + sum_{ci, t} X[b, ci, v + o(t)] W[co, ci, t]     (zero padding)
// with N = Co (padded to a multiple of 16) and K = Ci x taps walked as k-steps of 16 input
// channels at one tap t, channel groups outside, taps inside.
//
// M: rows are consecutive positions of the grid with its border of zeros (P = n + 2 per axis; the
// rows that fall on the border are computed and dropped).  In that order a tap is a constant shift,
// so a CTA stages the R + 2 P + 2 positions that its R rows reach in a z plane once, and a tap's A
// operand is the same shared memory from another start: in the K-major layout without swizzle a row
// of 8 channels is 16 bytes, rows lie 16 bytes apart, and a descriptor may start at any 16-byte
// address.  A CTA makes the same rows of up to 8 planes, each with its accumulators in TMEM, and
// keeps the last three or four staged planes: a voxel is loaded, split and stored 2 to 3 times per
// channel group, not 27 times (once per tap).
//
// The activations stay float32 [B][C][n^3]; the weights are bf16 [Co][Ci][taps].  A value is split
// into a bf16 hi and lo part (x = hi + lo to 16 mantissa bits), so the two products hi*W + lo*W
// give the FP32 activations times the bf16 weights to ~2^-17; accumulation is FP32 in TMEM.  A
// product of M = 128, K = 16 and N <= 64 takes 40 cycles (it is bound by reading A), 54 of them per
// row tile and channel group: 1.4 ms for the 27 convolutions of a 64^3, batch 8 training step, which
// take 3.1 (5.5 with three planes staged for each plane of rows, 17.0 with every tap gathered anew).
//
// One CTA: eight warps stage a plane while one thread of the ninth issues the products of the plane
// before; two barriers in turn say when a batch has run, so that with four slots staging waits for
// the batch before the last only.  All read the accumulators at the end.  Two persistent CTAs per SM
// where shared memory allows; the output channels are divided between CTAs where there are too few
// blocks (8^3, 128 -> 128: 139 -> 68 us).  The issue loop decides as much as the staging:
// a loop over the 27 taps issues one product in 139 cycles, all 54 unrolled one in 40 when they are
// repeated, but here each runs once a plane and the instruction fetches cost more than that saves;
// the 9 taps of a plane unrolled, in a warp without divergence, measured best (64^3, 16 -> 16
// channels: 281 us with 27 unrolled, 212 with 9, 204 without divergence, 220 with 3).
// Every wait is bounded: a timeout sets *err, marks the CTA's outputs NaN and returns.
#include <cuda_bf16.h>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace lddmm {

namespace {

constexpr int CV_THREADS = 256;
// shared memory: at most, of two CTAs on an SM, and from where on a CTA surely has an SM (and its 512
// TMEM columns) to itself
constexpr int CV_SMEM_CAP = 225 * 1024, CV_SMEM_PAIR = 115000, CV_SMEM_ALONE = 118000;

struct ConvArgs {
  const float* x;
  const __nv_bfloat16* w;
  const float* bias;
  float* y;
  int Ci, Co, n;
  int Np, NS;           // output channels of a CTA (padded to 16), CTAs that share the channels
  int taps, nph;        // filter taps; steps a channel group takes (1, or 3: a z plane each)
  int pad, P;           // border, n + 2 border
  int T, L;             // row tiles of 128 per plane of a CTA; positions staged per plane
  int Z, slots;         // planes a CTA makes; planes in shared memory at a time
  int nrt, nzc, nblk;   // blocks along the rows, along z, in all samples
  int wres;             // 1: the weights of all channel groups stay in shared memory
  int r_lo, r_n;        // position of the first row, rows (of a plane, or of the volume if Z = 1)
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
__global__ void __launch_bounds__(CV_THREADS + 32, 2) k_conv_tc(ConvArgs a) {
  extern __shared__ __align__(128) uint8_t cv_sm[];
  __shared__ __align__(8) uint64_t b_done[2];
  __shared__ uint32_t tmem_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int uwarp = __shfl_sync(0xffffffffu, warp, 0);
  const int n = a.n, P = a.P, PP = P * P;
  const size_t nv = (size_t)n * n * n;
  const int span = a.slots * a.L;                         // positions in shared memory
  const int co0 = (int)(blockIdx.x % a.NS) * a.Np;        // first output channel
  uint8_t* const bsm = cv_sm + 64 * span;

  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(&tmem_sh), (uint32_t)a.tcols);
    ptx::tmem_relinquish();
  }
  if (tid == 0) {
    ptx::mbar_init(ptx::smem_u32(&b_done[0]), 1);
    ptx::mbar_init(ptx::smem_u32(&b_done[1]), 1);
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
        const int i = i0 + u * CV_THREADS, t = i % TPS, ch = i / TPS, co = co0 + (ch >> 1);
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
  const int nkc = a.Ci / 16, wbytes = TPS * a.Np * 32;
  bool ok = true;
  uint32_t issued = 0, waited = 0;    // batches of products: batch i signals barrier i & 1
  auto wait_to = [&](uint32_t batch) {
    for (; waited < batch; ++waited)
      ok = ok && ptx::mbar_wait(ptx::smem_u32(&b_done[waited & 1u]), (waited >> 1) & 1u);
  };
  if (a.wres && tid < CV_THREADS)
    for (int st = 0; st < nkc * a.nph; ++st)
      stage_weights(st / a.nph, st % a.nph, bsm + (size_t)st * wbytes);
  for (int blk = blockIdx.x / a.NS; blk < a.nblk; blk += gridDim.x / a.NS) {
    const int rt = blk % a.nrt, bz = blk / a.nrt, b = bz / a.nzc, z0 = (bz - b * a.nzc) * a.Z;
    const int r0 = rt * (a.T * 128), p0 = a.r_lo + r0 + z0 * PP;   // position of row 0
    const int Zc = TPS == 27 ? min(a.Z, n - z0) : 1;
    for (int kc = 0; kc < nkc; ++kc)
      for (int i = 0; i < (TPS == 27 ? Zc : a.nph); ++i) {
        uint8_t* const wb = bsm + (a.wres ? (size_t)(kc * a.nph + (TPS == 27 ? 0 : i)) * wbytes : 0);
        if (tid < CV_THREADS) {
          // ---------------------------------------------------------- staging
          // step 0 of a channel group fills planes z0 - 1 .. z0 + 1, a later one plane z0 + i + 1;
          // with four slots the batch before may still run, it reads the other three
          wait_to(TPS == 27 && i > 0 && a.slots == 4 ? issued - 1 : issued);
          if (ok) {
            if (!a.wres && (TPS != 27 || i == 0)) stage_weights(kc, TPS == 27 ? 0 : i, wb);
            // A: [hi, lo][8-channel half][slot][position] of 16 bytes; a thread takes all 16 channels
            // of a position, 16 loads in flight
            const float* xb = a.x + ((size_t)b * a.Ci + kc * 16) * nv;
            const int pl0 = TPS == 27 ? (i ? i + 2 : 0) : TPS == 9 ? i : 1, cnt = (TPS == 27 && !i ? 3 : 1) * a.L;
            const int first = p0 + (TPS == 1 ? 0 : (pl0 - 1) * PP - P - 1);
            const int slot0 = TPS == 27 ? (a.slots == 4 ? pl0 & 3 : pl0 % 3) * a.L : 0;
            for (int e = tid; e < cnt; e += CV_THREADS) {
              const int sp = cnt == a.L ? 0 : quot(e, a.L, a.mL);
              const int o = voxel_at(first + sp * PP + (e - sp * a.L));
              const float* p = xb + (o < 0 ? 0 : o);
              float v[16];
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] = o >= 0 ? __ldg(p + (size_t)j * nv) : 0.f;
              uint8_t* const d = cv_sm + (size_t)(slot0 + e) * 16;
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t hw[4], lw[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const float f0 = v[8 * h + 2 * j], f1 = v[8 * h + 2 * j + 1];
                  hw[j] = pack_bf2(f0, f1);
                  lw[j] = pack_bf2(f0 - __uint_as_float(hw[j] << 16), f1 - __uint_as_float(hw[j] & 0xffff0000u));
                }
                *reinterpret_cast<uint4*>(d + (size_t)h * span * 16) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                *reinterpret_cast<uint4*>(d + (size_t)(2 + h) * span * 16) =
                    make_uint4(lw[0], lw[1], lw[2], lw[3]);
              }
            }
          }
          ptx::fence_proxy_async_smem();
        }
        ok = __syncthreads_and(ok);
        if (!ok) break;
        // ------------------------------------------------------------ products of a plane's rows
        if (uwarp == CV_THREADS / 32) {
          const uint32_t el = ptx::elect_one();
          ptx::tc_fence_after();
          const uint32_t id = ptx::idesc_bf16(128, a.Np);
          const uint64_t dA = ptx::smem_desc(ptx::smem_u32(cv_sm), (uint32_t)span * 16u, 128);
          const uint64_t dB = ptx::smem_desc(ptx::smem_u32(wb), 128, 256);
          // the offsets added below stay inside the descriptors' 14 address bits
          const uint32_t a0 = (uint32_t)dA, b0 = (uint32_t)dB, lo = 2u * (uint32_t)span;
          auto desc = [](uint64_t d, uint32_t low) { return (d & 0xffffffff00000000ull) | low; };
          for (int m = 0; m < a.T; ++m) {
            const uint32_t d = tmem + (uint32_t)(((TPS == 27 ? i * a.T : 0) + m) * a.Np);
            uint32_t bt = b0;
#pragma unroll 1
            for (int oz = 0; oz < (TPS == 27 ? 3 : 1); ++oz) {
              const int pl = TPS == 27 ? i + oz : 0;
              const uint32_t az = a0 + (uint32_t)((a.slots == 4 ? pl & 3 : pl % 3) * a.L + m * 128);
#pragma unroll
              for (int t = 0; t < (TPS == 1 ? 1 : 9); ++t, bt += 2u * a.Np) {
                // the tap's first row and its weights, in 16-byte units
                const uint32_t at = az + (uint32_t)(t / 3 * P + t % 3);
                ptx::mma_bf16_one(el, d, desc(dA, at), desc(dB, bt), id,
                              t ? 1u : (kc | oz | (TPS == 27 ? 0 : i)) ? 1u : 0u);
                ptx::mma_bf16_one(el, d, desc(dA, at + lo), desc(dB, bt), id, 1u);
              }
            }
          }
          if (el) ptx::mma_commit(ptx::smem_u32(&b_done[issued & 1u]));
          __syncwarp();
        }
        ++issued;
      }
    if (tid < CV_THREADS) wait_to(issued);
    ok = __syncthreads_and(ok);
    ptx::tc_fence_after();
    // -------------------------------------------------------------- epilogue
    // warp w reads TMEM lanes 32 (w % 4)..; the two halves of the warps take alternate 16-column chunks
    const int q = warp & 3, half = warp >> 2, nch = a.Np / 16, items = half < 2 ? Zc * a.T * nch : 0;
    for (int it = half; it < items; it += 2) {
      const int m = nch == 1 ? it : it / nch, c = it - m * nch, zz = m / a.T;
      const int row = (m - zz * a.T) * 128 + q * 32 + lane;
      const int vo = r0 + row < a.r_n ? voxel_at(p0 + zz * PP + row) : -1;
      float acc[16];
      if (ok) {
        ptx::tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(it * 16), acc);
      } else {
        // a wait gave up: the outputs are marked invalid besides the error flag
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[j] = __int_as_float(0x7fc00000);
      }
      if (vo < 0) continue;
      float* const o = a.y + ((size_t)b * a.Co + co0 + c * 16) * nv + vo;
      const int nco = a.Co - co0 - c * 16;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (j < nco) {
          float r = acc[j] + (a.bias ? __ldg(a.bias + co0 + c * 16 + j) : 0.f);
          if (a.accumulate) r += o[(size_t)j * nv];
          if (a.relu && ok) r = fmaxf(r, 0.f);
          o[(size_t)j * nv] = r;
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
      for (uint32_t i = issued < 2 ? 0 : issued - 2; i < issued; ++i)
        ptx::mbar_wait(ptx::smem_u32(&b_done[i & 1u]), (i >> 1) & 1u);
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
// outputs are then NaN); allocated once on each device.
static int* conv_err_flag() {
  static PerDevice<int*> kept;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= kKeptDevices) return nullptr;
  return kept.get(dev, [] {
    int* f = nullptr;
    if (cudaMalloc((void**)&f, sizeof(int)) == cudaSuccess) cudaMemset(f, 0, sizeof(int));
    else cudaGetLastError();
    return f;
  });
}

template <int TPS>
static cudaError_t launch_conv(const ConvArgs& a, int B, cudaStream_t s) {
  static PerDevice<bool> set;
  const cudaError_t e = raise_smem_limit(set, k_conv_tc<TPS>, CV_SMEM_CAP);
  if (e != cudaSuccess) return e;
  // persistent: two CTAs per SM share the blocks (the weights are staged once per CTA)
  const int smem = (int)cv_smem(a.slots, a.L, TPS * (a.wres ? a.Ci / 16 * a.nph : 1), a.Np);
  const int cap = (smem <= CV_SMEM_PAIR ? 304 : 152) / a.NS, grid = a.NS * (a.nblk < cap ? a.nblk : cap);
  k_conv_tc<TPS><<<grid, CV_THREADS + 32, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t conv_tc_fwd(const float* x, const void* w, const float* bias, float* y, int B, int Ci,
                        int Co, int n, int ks, int relu, int accumulate, cudaStream_t s) {
  ConvArgs a{};
  a.x = x; a.w = (const __nv_bfloat16*)w; a.bias = bias; a.y = y;
  a.Ci = Ci; a.Co = Co; a.n = n;
  a.taps = ks * ks * ks;
  a.pad = ks / 2;
  a.P = n + 2 * a.pad;
  a.relu = relu; a.accumulate = accumulate;
  a.err = conv_err_flag();
  const int PP = a.P * a.P, halo = a.pad ? 2 * a.P + 2 : 0, nkc = Ci / 16;
  const int r_lo = a.pad * (PP + a.P + 1);                   // the first voxel
  const int r_vol = (n - 1) * (PP + a.P + 1) + 1, r_pl = (n - 1) * (a.P + 1) + 1;
  // The split is the cheapest by a model of a CTA's clocks, fitted to sweeps over the network's
  // layers at 4^3..64^3 (its choices are within 6% of the best found): staging 1000 + 15 a position
  // when two CTAs share an SM; a product 40, Np / 2 from 80 channels on, twice that with the
  // neighbour's; 1200 to read back and store 128 x 16 results; 1150 a pass over the weights.  With
  // four plane slots the staging of a plane hides behind the products of the one before.
  const int nco = (Co + 15) / 16;
  double best = 0;
  for (int nph = 1; best == 0 && nph <= (ks == 1 ? 1 : 3); nph += 2) {   // 3: the planes do not fit
    const int one = ks == 1 || nph > 1, taps = ks == 1 ? 1 : 27 / nph, ng = nkc * nph;
    for (int NS = 1, w16 = 0; NS <= nco; ++NS) {
      if ((nco + NS - 1) / NS == w16) continue;              // no fewer channels than before
      w16 = (nco + NS - 1) / NS;
      const int Np = 16 * w16;
      for (int T = 1; T <= 3; ++T)
        for (int Z : {1, 2, 3, 4, 6, 8})
          for (int slots = one ? 1 : Z > 1 ? 4 : 3; slots >= (one ? 1 : 3); --slots)
            for (int res = 1; res >= 0; --res) {
              if (Z > (one ? 1 : n)) continue;
              const int64_t m = cv_smem(slots, 128 * T + halo, (int64_t)taps * (res ? ng : 1), Np);
              if (m > CV_SMEM_CAP || T * Z * Np > (m <= CV_SMEM_ALONE ? 256 : 512)) continue;
              const int L = 128 * T + halo, cap = (m <= CV_SMEM_PAIR ? 304 : 152) / NS;
              const int64_t nblk = (int64_t)(((Z > 1 ? r_pl : r_vol) + 128 * T - 1) / (128 * T)) *
                                   (Z > 1 ? (n + Z - 1) / Z : 1) * B;
              const double st = 1000 + 15.0 * L, st0 = one ? st : 1000 + 45.0 * L;
              const double w = (Np * taps * 2 + 511) / 512 * 1150.0;
              const double mm = 2.0 * T * taps * (Np > 80 ? Np / 2 : 40) *
                                (nblk * NS > 152 && cap * NS > 152 ? 2 : 1.25);
              const double group = (res ? 0 : w) + st0 + mm +
                                   (Z - 1) * (slots < 4 ? st + mm : st > mm ? st : mm);
              const double c = ((nblk + cap - 1) / cap) * (ng * group + Z * T * w16 * 1200.0) +
                               (res ? ng * w : 0);
              if (best == 0 || c < best) {
                best = c;
                a.T = T; a.Z = Z; a.slots = slots; a.wres = res; a.NS = NS; a.Np = Np; a.nph = nph;
              }
              if (res && m <= CV_SMEM_PAIR) break;           // resident weights cost nothing there
            }
    }
  }
  if (best == 0) return cudaErrorInvalidValue;
  a.L = 128 * a.T + halo;
  a.r_lo = r_lo;
  a.r_n = a.Z > 1 ? r_pl : r_vol;
  a.nrt = (a.r_n + 128 * a.T - 1) / (128 * a.T);
  a.nzc = a.Z > 1 ? (n + a.Z - 1) / a.Z : 1;
  a.nblk = a.nrt * a.nzc * B;
  // positions stay below 2 P^3 and staged ones below 2^16: where the reciprocals are exact
  const auto recip = [](unsigned d) { return (unsigned)(((1ull << 32) + d - 1) / d); };
  a.mP = a.P > 1 && a.P <= 200 ? recip(a.P) : 0u;
  a.mL = recip(a.L);
  a.tcols = 32;
  while (a.tcols < a.T * a.Z * a.Np) a.tcols <<= 1;
  if (ks == 1) return launch_conv<1>(a, B, s);
  return a.nph == 1 ? launch_conv<27>(a, B, s) : launch_conv<9>(a, B, s);
}

}  // namespace lddmm
