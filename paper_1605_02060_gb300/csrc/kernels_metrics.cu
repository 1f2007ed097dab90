// Registration-quality measures of §2.7 on the GPU:
//   Hausdorff distance  d_H = max{ sup_{x in S(1)} inf_{y in S1} d(x, y), sup_{y in S1} inf_{x in S(1)} d(x, y) }
//   median distance     d_M = median of the union of both sets of directed distances
//   landmark error      e_k = | phi(x_k) - y_k |
// S(1) and S1 are the surfaces of two binary masks: mask voxels with a face neighbour outside
// the mask (a neighbour beyond the grid counts as outside).  d is the Euclidean distance between
// voxel centres in physical units.
//
// The surface voxels are listed by 8x8x8 cells (a block per cell counts its voxels, a scan places
// the cells, a second pass writes each voxel's position within its cell as 9 bits), and a query
// visits the other surface's cells in shells around its own until the next shell cannot hold
// anything nearer, or, further away, the cells that its cell cannot rule out.  Registered surfaces
// lie a few voxels apart, so a query meets a few hundred candidates.  Distances are compared in FP32 (every rounding in them is monotone in |dx|, |dy|,
// |dz|, so a cell whose nearest corner is no nearer than the best holds nothing nearer) and the
// winner's distance is recomputed in FP64.  The order statistics are found by radix selection on
// the bit patterns of the (non-negative) FP64 distances.
#include "kernels.h"

namespace lddmm {

namespace {

constexpr int kCell = 8;

struct CellGrid {
  int ncx, ncy, ncz, ncell;
};

// One warp per cell, mask blockIdx.y.  FILL = false: start[mask][cell] = the number of surface
// voxels; FILL = true: their positions in the cell, x | y << 3 | z << 6, from
// list[start[mask][cell]] on (the second mask's list starts at nA).  A lane takes two columns
// (x, y) and (x, y + 4) and marches up z with the planes below, at and above in registers, so a
// voxel is loaded once and only mask voxels load their x and y neighbours.  (A thread per voxel
// and a block per cell: 93 us to count both masks of 264x160x228; this way 28 us.)
template <bool FILL>
__global__ void __launch_bounds__(256) k_surface_cells(Grid g, CellGrid cg,
                                                       const uint8_t* __restrict__ A,
                                                       const uint8_t* __restrict__ B,
                                                       unsigned* __restrict__ start,
                                                       uint16_t* __restrict__ list, unsigned nA) {
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= cg.ncell) return;
  const int cx = c % cg.ncx, cy = (c / cg.ncx) % cg.ncy, cz = c / (cg.ncx * cg.ncy);
  unsigned* st = start + blockIdx.y * (size_t)(cg.ncell + 1);
  unsigned at = 0;
  if (FILL) {
    at = st[c];
    if (at == st[c + 1]) return;
    if (blockIdx.y) at += nA;
  }
  const uint8_t* m = blockIdx.y ? B : A;
  const int64_t sy = g.nx, sz = (int64_t)g.nx * g.ny;
  const int x = cx * kCell + (lane & 7), z0 = cz * kCell;
  unsigned cnt = 0;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int ly = (lane >> 3) + 4 * half, y = cy * kCell + ly;
    const bool in = x < g.nx && y < g.ny;
    const int64_t i0 = in ? z0 * sz + y * sy + x : 0;
    const bool edge = x == 0 || x == g.nx - 1 || y == 0 || y == g.ny - 1;
    uint8_t col[kCell + 2];
#pragma unroll
    for (int k = 0; k < kCell + 2; ++k) {
      const int z = z0 + k - 1;
      col[k] = in && z >= 0 && z < g.nz ? __ldg(m + i0 + (k - 1) * sz) : 0;
    }
#pragma unroll
    for (int k = 0; k < kCell; ++k) {
      // a neighbour beyond the grid reads as outside the mask
      bool s = col[k + 1] != 0;
      if (s && !edge && col[k] && col[k + 2]) {
        const uint8_t* q = m + i0 + k * sz;
        s = !q[-1] || !q[1] || !q[-sy] || !q[sy];
      }
      const unsigned b = __ballot_sync(0xffffffffu, s);
      if (FILL && s)
        list[at + cnt + __popc(b & ((1u << lane) - 1u))] = (uint16_t)((lane & 7) | ly << 3 | k << 6);
      cnt += __popc(b);
    }
  }
  if (!FILL && lane == 0) st[c] = cnt;
}

// start[mask][0..ncell): counts -> exclusive prefix sums, start[mask][ncell] = the total.
__global__ void __launch_bounds__(1024) k_cell_scan(unsigned* __restrict__ start, int ncell) {
  __shared__ unsigned wsum[32];
  unsigned* st = start + blockIdx.x * (size_t)(ncell + 1);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned base = 0;
  for (int c0 = 0; c0 < ncell; c0 += 1024) {
    const int c = c0 + threadIdx.x;
    const unsigned v = c < ncell ? st[c] : 0u;
    unsigned p = v;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned q = __shfl_up_sync(0xffffffffu, p, o);
      if (lane >= o) p += q;
    }
    if (lane == 31) wsum[wid] = p;
    __syncthreads();
    if (wid == 0) {
      unsigned w = wsum[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned q = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += q;
      }
      wsum[lane] = w;
    }
    __syncthreads();
    if (c < ncell) st[c] = base + (wid ? wsum[wid - 1] : 0u) + p - v;
    base += wsum[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) st[ncell] = base;
}

// d[mask][i] = distance (physical units, FP64) from surface voxel i of the mask (blockIdx.y, in
// list order) to the nearest surface voxel of the other.  One block per cell; a thread takes a
// voxel of the cell.  It looks in the cells around its own, shell by shell; what that costs is the
// candidates' FP32 arithmetic: at 264x160x228 (6e4 voxels each, a few voxels apart) both directions
// take 34 us, against 5.1 ms for comparing every pair.  Past kNearShells the empty cells of the shells
// would be most of the work: there the block passes over all cells once, for the least distance at
// which some cell is sure to hold a voxel, and again for the cells that may hold a nearer one, and its
// voxels look in those only.  Surfaces far apart at 264x160x228 (us a call; every pair / all shells /
// this way): ellipsoids at opposite ends 1329 / 6147 / 453, the first face against the last 3701 /
// 7987 / 2156, a voxel in either corner 264 / 3610 / 211, an ellipsoid and a corner 4733 / 7333 / 343.
// (20 blocks on an SM: registers and candidates as three coordinates, 6 KB, cost the near search 1 us.)
constexpr int kNearShells = 2, kCand = 512, kFewOpen = 4;

__device__ __forceinline__ float dist2(int ix, int iy, int iz, float hx, float hy, float hz) {
  const float x = (float)ix * hx, y = (float)iy * hy, z = (float)iz * hz;
  return fmaf(x, x, fmaf(y, y, z * z));
}

__global__ void __launch_bounds__(64, 20) k_nearest(Grid g, CellGrid cg,
                                                const unsigned* __restrict__ start,
                                                const uint16_t* __restrict__ list, unsigned nA,
                                                float hx, float hy, float hz,
                                                double* __restrict__ dA, double* __restrict__ dB) {
  __shared__ int cand[kCand];          // cells that may hold the nearest voxel of some query
  __shared__ unsigned wcnt[2];
  __shared__ float wmin[2];
  const int c = blockIdx.x, side = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
  const unsigned* sq = start + side * (size_t)(cg.ncell + 1);
  const unsigned* so = start + (side ^ 1) * (size_t)(cg.ncell + 1);
  const uint16_t* lq = list + (side ? nA : 0u);
  const uint16_t* lo = list + (side ? 0u : nA);
  double* d = side ? dB : dA;
  const unsigned q0 = sq[c], q1 = sq[c + 1];
  if (q0 == q1) return;
  const int cx = c % cg.ncx, cy = (c / cg.ncx) % cg.ncy, cz = c / (cg.ncx * cg.ncy);
  const int rmax = max(max(max(cx, cg.ncx - 1 - cx), max(cy, cg.ncy - 1 - cy)),
                       max(cz, cg.ncz - 1 - cz));
  float ub = -1.f;                     // far cells: the bound (once it is known),
  int ncand = -1;                      // and the cells within it, when cand holds all of them
  for (unsigned base = q0; base < q1; base += 64) {
    const unsigned i = base + tid;
    const bool on = i < q1;
    const unsigned code = on ? lq[i] : 0u;
    const int px = cx * kCell + (code & 7), py = cy * kCell + ((code >> 3) & 7),
              pz = cz * kCell + (code >> 6);
    // the nearest voxel so far of the query at (x, y, z)
    struct Near {
      float best;
      int x, y, z;
    };
    // the voxels p0 .. p1 - 1 of the list, of cell (x, y, z)
    auto scan = [&](Near& w, int qx, int qy, int qz, unsigned p0, unsigned p1, int x, int y, int z) {
      for (unsigned k = p0; k < p1; ++k) {
        const unsigned oq = __ldg(lo + k);
        const int ox = x * kCell + (oq & 7), oy = y * kCell + ((oq >> 3) & 7),
                  oz = z * kCell + (oq >> 6);
        const float d2 = dist2(qx - ox, qy - oy, qz - oz, hx, hy, hz);
        if (d2 < w.best) w = Near{d2, ox, oy, oz};
      }
    };
    // cell oc at (x, y, z), unless nothing in it can be nearer
    auto look = [&](Near& w, int qx, int qy, int qz, int oc, int x, int y, int z) {
      const int bx = max(max(x * kCell - qx, qx - (x * kCell + kCell - 1)), 0),
                by = max(max(y * kCell - qy, qy - (y * kCell + kCell - 1)), 0),
                bz = max(max(z * kCell - qz, qz - (z * kCell + kCell - 1)), 0);
      if (dist2(bx, by, bz, hx, hy, hz) < w.best) scan(w, qx, qy, qz, so[oc], so[oc + 1], x, y, z);
    };
    Near w{3.0e38f, 0, 0, 0};
    bool open = on;                    // a nearer voxel may lie beyond the shells
    for (int r = 0; open; ++r) {
      if (r > rmax) {
        open = false;
        break;
      }
      if (r > 0) {
        // the nearest a voxel of shell r or beyond can lie: past one of the faces of shell r - 1
        const int e = (r - 1) * kCell;
        const float fx = (float)min(px - (cx * kCell - e) + 1, cx * kCell + kCell + e - px) * hx;
        const float fy = (float)min(py - (cy * kCell - e) + 1, cy * kCell + kCell + e - py) * hy;
        const float fz = (float)min(pz - (cz * kCell - e) + 1, cz * kCell + kCell + e - pz) * hz;
        const float b = fminf(fx, fminf(fy, fz));
        if (b * b >= w.best) {
          open = false;
          break;
        }
      }
      if (r > kNearShells) break;
      const int z0 = max(cz - r, 0), z1 = min(cz + r, cg.ncz - 1);
      const int y0 = max(cy - r, 0), y1 = min(cy + r, cg.ncy - 1);
      for (int z = z0; z <= z1; ++z) {
        const int bz = max(max(z * kCell - pz, pz - (z * kCell + kCell - 1)), 0);
        const float gz = (float)bz * hz;
        for (int y = y0; y <= y1; ++y) {
          const int by = max(max(y * kCell - py, py - (y * kCell + kCell - 1)), 0);
          const float gy = (float)by * hy, gyz = fmaf(gy, gy, gz * gz);
          if (gyz >= w.best) continue;
          const bool face = z - cz == r || cz - z == r || y - cy == r || cy - y == r;
          const int step = face || r == 0 ? 1 : 2 * r;
          for (int x = cx - r; x <= cx + r; x += step) {
            if (x < 0 || x >= cg.ncx) continue;
            const int oc = (z * cg.ncy + y) * cg.ncx + x;
            const unsigned p0 = so[oc], p1 = so[oc + 1];
            if (p0 == p1) continue;
            const int bx = max(max(x * kCell - px, px - (x * kCell + kCell - 1)), 0);
            const float gx = (float)bx * hx;
            if (fmaf(gx, gx, gyz) < w.best) scan(w, px, py, pz, p0, p1, x, y, z);
          }
        }
      }
    }
    if (__syncthreads_or(open)) {
      // of cell o (o >= ncell: none): has it voxels?
      auto some = [&](int o) { return o < cg.ncell && so[o] != so[o + 1]; };
      auto decode = [&](int o, int& x, int& y, int& z) {
        const int t = o / cg.ncx;
        x = o - t * cg.ncx;
        z = t / cg.ncy;
        y = t - z * cg.ncy;
      };
      if (ub < 0.f) {
        float u = 3.0e38f;
        for (int o0 = tid; o0 < cg.ncell; o0 += 4 * 64) {
          bool has[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) has[k] = some(o0 + k * 64);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (has[k]) {
              int x, y, z;
              decode(o0 + k * 64, x, y, z);
              // no voxel of the one cell is further from one of the other than their far corners
              u = fminf(u, dist2(kCell * abs(x - cx) + kCell - 1, kCell * abs(y - cy) + kCell - 1,
                                 kCell * abs(z - cz) + kCell - 1, hx, hy, hz));
            }
        }
        for (int o = 16; o; o >>= 1) u = fminf(u, __shfl_xor_sync(0xffffffffu, u, o));
        if (lane == 0) wmin[tid >> 5] = u;
        __syncthreads();
        ub = fminf(wmin[0], wmin[1]);
      }
      // some voxel lies within the bound: a query that knows none looks for any up to it
      if (open && w.best > ub) w.best = __uint_as_float(__float_as_uint(ub) + 1u);
      auto look_in = [&](int n) {      // the first n candidates, by the open queries
        unsigned mine = __ballot_sync(0xffffffffu, open);
        if (__popc(mine) > kFewOpen) {
          for (int k = 0; k < n; ++k) {
            int x, y, z;
            decode(cand[k], x, y, z);
            if (open) look(w, px, py, pz, cand[k], x, y, z);
          }
          return;
        }
        // a warp with few open queries takes them one by one, a lane every 32nd cell
        for (; mine; mine &= mine - 1) {
          const int src = __ffs(mine) - 1;
          const int qx = __shfl_sync(0xffffffffu, px, src), qy = __shfl_sync(0xffffffffu, py, src),
                    qz = __shfl_sync(0xffffffffu, pz, src);
          Near t{__shfl_sync(0xffffffffu, w.best, src), 0, 0, 0};
          const float had = t.best;
          for (int k = lane; k < n; k += 32) {
            int x, y, z;
            decode(cand[k], x, y, z);
            look(t, qx, qy, qz, cand[k], x, y, z);
          }
          const unsigned m = __reduce_min_sync(0xffffffffu, __float_as_uint(t.best));
          const int from = __ffs(__ballot_sync(0xffffffffu, __float_as_uint(t.best) == m)) - 1;
          const Near f{__uint_as_float(m), __shfl_sync(0xffffffffu, t.x, from),
                       __shfl_sync(0xffffffffu, t.y, from), __shfl_sync(0xffffffffu, t.z, from)};
          if (lane == src && f.best < had) w = f;
        }
      };
      if (ncand >= 0) {
        look_in(ncand);
      } else {
        int n = 0;
        bool all = true;
        for (int o0 = 0; o0 < cg.ncell; o0 += 4 * 64) {
          bool in[4];
          unsigned b[4], m = 0;
#pragma unroll
          for (int k = 0; k < 4; ++k) in[k] = some(o0 + k * 64 + tid);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (in[k]) {
              int x, y, z;
              decode(o0 + k * 64 + tid, x, y, z);
              in[k] = dist2(max(kCell * abs(x - cx) - (kCell - 1), 0), max(kCell * abs(y - cy) - (kCell - 1), 0),
                            max(kCell * abs(z - cz) - (kCell - 1), 0), hx, hy, hz) <= ub;
            }
            b[k] = __ballot_sync(0xffffffffu, in[k]);
            m += __popc(b[k]);
          }
          if (lane == 0) wcnt[tid >> 5] = m;
          __syncthreads();
          int at = n + (tid >= 32 ? (int)wcnt[0] : 0);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (in[k]) cand[at + __popc(b[k] & ((1u << lane) - 1u))] = o0 + k * 64 + tid;
            at += __popc(b[k]);
          }
          n += (int)(wcnt[0] + wcnt[1]);
          __syncthreads();
          if (n > kCand - 4 * 64) {
            look_in(n);
            __syncthreads();
            n = 0;
            all = false;
          }
        }
        look_in(n);
        if (all) ncand = n;
      }
    }
    if (on) {
      const double dx = (double)(px - w.x) * hx, dy = (double)(py - w.y) * hy,
                   dz = (double)(pz - w.z) * hz;
      d[i] = sqrt(dx * dx + dy * dy + dz * dz);
    }
  }
}

// Order statistics of the n = na + nb distances in dA and dB: out[0] = max, out[1] = k1-th and
// out[2] = k2-th smallest (0-based, k1 <= k2 <= k1 + 1).  Non-negative doubles order like their
// bit patterns, so the k1-th is found digit by digit: pass p counts the digits of the values that
// share the digits found so far (equal digits of a warp counted once: most distances of a
// registration are among a few values), and the last block to finish picks the digit that holds
// the k1-th.  Pass 6 counts the values up to it and finds the next above.  Every pass reads the
// list once from L2: 7 short launches, 46 us for 1.1e5 distances.  (One block halving the bit
// range 2 x 64 times took 2.5 ms, one block doing these passes 267 us.)
typedef unsigned long long u64;
struct Select {          // zeroed before pass 0
  u64 prefix, mx, cnt, inv_next;   // inv_next: the complement of the next value above
  unsigned k, ticket;
  unsigned hist[2048];
};

__global__ void __launch_bounds__(512) k_select(const double* __restrict__ dA, unsigned na,
                                                const double* __restrict__ dB, unsigned nb,
                                                unsigned k1, unsigned k2, int pass, Select* sel,
                                                double* out) {
  __shared__ unsigned hist[2048];
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned n = na + nb, stride = gridDim.x * 512, i0 = blockIdx.x * 512 + tid;
  const unsigned nround = (n + 31u) & ~31u;      // whole warps
  auto at = [&](unsigned i) {
    return (u64)__double_as_longlong(i < na ? __ldg(dA + i) : __ldg(dB + (i - na)));
  };
  // digits: bits 53..63, 42..52, 31..41, 20..30, 9..19, 0..8
  const int shift = pass == 5 ? 0 : 53 - 11 * pass;
  const unsigned nbin = pass == 5 ? 512u : 2048u;
  const u64 prefix = sel->prefix;
  if (pass < 6) {
    const u64 above = pass == 0 ? 0ull : ~0ull << (pass == 5 ? 9 : shift + 11);
    for (unsigned b = tid; b < nbin; b += 512) hist[b] = 0;
    __syncthreads();
    u64 mx = 0;
    for (unsigned i = i0; i < nround; i += stride) {
      const u64 v = i < n ? at(i) : 0ull;
      const bool on = i < n && (v & above) == prefix;
      if (i < n) mx = max(mx, v);
      const unsigned digit = on ? (unsigned)(v >> shift) & (nbin - 1u) : 0xffffffffu;
      const unsigned peers = __match_any_sync(0xffffffffu, digit);
      if (on && lane == __ffs(peers) - 1) atomicAdd(&hist[digit], (unsigned)__popc(peers));
    }
    if (pass == 0) {
      for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (lane == 0) atomicMax(&sel->mx, mx);
    }
    __syncthreads();
    for (unsigned b = tid; b < nbin; b += 512)
      if (hist[b]) atomicAdd(&sel->hist[b], hist[b]);
  } else {
    u64 cnt = 0, inv = 0;
    for (unsigned i = i0; i < n; i += stride) {
      const u64 v = at(i);
      if (v <= prefix) ++cnt;
      else inv = max(inv, ~v);
    }
    for (int o = 16; o; o >>= 1) {
      cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
      inv = max(inv, __shfl_xor_sync(0xffffffffu, inv, o));
    }
    if (lane == 0) {
      atomicAdd(&sel->cnt, cnt);
      atomicMax(&sel->inv_next, inv);
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(&sel->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  volatile Select* vs = sel;
  if (pass == 6) {
    if (tid == 0) {
      out[0] = __longlong_as_double((long long)vs->mx);
      out[1] = __longlong_as_double((long long)prefix);
      out[2] = __longlong_as_double((long long)(k2 < vs->cnt ? prefix : ~vs->inv_next));
    }
    return;
  }
  for (unsigned b = tid; b < nbin; b += 512) {
    hist[b] = vs->hist[b];
    vs->hist[b] = 0;
  }
  __syncthreads();
  if (tid < 32) {
    // 64 (or 16) bins per lane: their sum, the lanes' prefix, then the bin that reaches k
    const unsigned k = pass == 0 ? k1 : vs->k, per = nbin / 32u;
    unsigned sum = 0;
    for (unsigned b = 0; b < per; ++b) sum += hist[lane * per + b];
    unsigned p = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned q = __shfl_up_sync(0xffffffffu, p, o);
      if (lane >= o) p += q;
    }
    __syncwarp();
    if (k >= p - sum && k < p) {
      unsigned c = p - sum, b = lane * per;
      while (k >= c + hist[b]) c += hist[b++];
      vs->prefix = prefix | (u64)b << shift;
      vs->k = k - c;
      vs->ticket = 0;
    }
  }
}

// e_k = |(x_k + u01(x_k) - y_k) h| with u01 (3 components of N, voxel units) interpolated
// trilinearly with clamp-to-edge coordinates.
__global__ void k_landmarks(Grid g, const float* __restrict__ u01, const float* __restrict__ xk,
                            const float* __restrict__ yk, int n, float hx, float hy, float hz,
                            double* __restrict__ e) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float x = xk[3 * k], y = xk[3 * k + 1], z = xk[3 * k + 2];
  const Tri w = tri_setup(g, x, y, z);
  const double px = (double)x + tri_apply(u01, w), py = (double)y + tri_apply(u01 + g.N, w),
               pz = (double)z + tri_apply(u01 + 2 * g.N, w);
  const double dx = (px - yk[3 * k]) * hx, dy = (py - yk[3 * k + 1]) * hy,
               dz = (pz - yk[3 * k + 2]) * hz;
  e[k] = sqrt(dx * dx + dy * dy + dz * dz);
}

}  // namespace

static CellGrid cells_of(const Grid& g) {
  CellGrid c;
  c.ncx = (g.nx + kCell - 1) / kCell;
  c.ncy = (g.ny + kCell - 1) / kCell;
  c.ncz = (g.nz + kCell - 1) / kCell;
  c.ncell = c.ncx * c.ncy * c.ncz;
  return c;
}

int64_t surface_cells(const Grid& g) { return cells_of(g).ncell; }
int64_t surface_select_bytes() { return sizeof(Select); }

cudaError_t surface_count(const Grid& g, const uint8_t* A, const uint8_t* B, unsigned* start,
                          cudaStream_t s) {
  const CellGrid c = cells_of(g);
  k_surface_cells<false><<<dim3((c.ncell + 7) / 8, 2), 256, 0, s>>>(g, c, A, B, start, nullptr, 0u);
  k_cell_scan<<<2, 1024, 0, s>>>(start, c.ncell);
  return cudaGetLastError();
}

cudaError_t surface_distances(const Grid& g, const uint8_t* A, const uint8_t* B, unsigned* start,
                              uint16_t* list, unsigned na, unsigned nb, float hx, float hy,
                              float hz, double* dA, double* dB, void* sel, double* out,
                              cudaStream_t s) {
  const CellGrid c = cells_of(g);
  cudaError_t e = cudaMemsetAsync(sel, 0, sizeof(Select), s);
  if (e != cudaSuccess) return e;
  k_surface_cells<true><<<dim3((c.ncell + 7) / 8, 2), 256, 0, s>>>(g, c, A, B, start, list, na);
  k_nearest<<<dim3(c.ncell, 2), 64, 0, s>>>(g, c, start, list, na, hx, hy, hz, dA, dB);
  const unsigned n = na + nb, nb512 = (n + 511) / 512;
  for (int pass = 0; pass < 7; ++pass)
    k_select<<<nb512 < 128u ? nb512 : 128u, 512, 0, s>>>(dA, na, dB, nb, (n - 1) / 2, n / 2, pass,
                                                        reinterpret_cast<Select*>(sel), out);
  return cudaGetLastError();
}

cudaError_t landmark_errors(const Grid& g, const float* u01, const float* xk, const float* yk,
                            int n, float hx, float hy, float hz, double* e, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_landmarks<<<(n + 127) / 128, 128, 0, s>>>(g, u01, xk, yk, n, hx, hy, hz, e);
  return cudaGetLastError();
}

}  // namespace lddmm
