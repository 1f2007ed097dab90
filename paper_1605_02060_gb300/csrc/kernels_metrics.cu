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
// anything nearer.  Registered surfaces lie a few voxels apart, so a query meets a few hundred
// candidates.  Distances are compared in FP32 (every rounding in them is monotone in |dx|, |dy|,
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
// voxel of the cell.  What it costs is the candidates' FP32 arithmetic: at 264x160x228 (6e4
// voxels each) both directions take 34 us, against 5.1 ms for comparing every pair.
__global__ void __launch_bounds__(64) k_nearest(Grid g, CellGrid cg,
                                                const unsigned* __restrict__ start,
                                                const uint16_t* __restrict__ list, unsigned nA,
                                                float hx, float hy, float hz,
                                                double* __restrict__ dA, double* __restrict__ dB) {
  const int c = blockIdx.x, side = blockIdx.y;
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
  for (unsigned i = q0 + threadIdx.x; i < q1; i += blockDim.x) {
    const unsigned code = lq[i];
    const int px = cx * kCell + (code & 7), py = cy * kCell + ((code >> 3) & 7),
              pz = cz * kCell + (code >> 6);
    float best = 3.0e38f;
    int wx = 0, wy = 0, wz = 0;
    for (int r = 0; r <= rmax; ++r) {
      if (r > 0) {
        // the nearest a voxel of shell r or beyond can lie: past one of the faces of shell r - 1
        const int e = (r - 1) * kCell;
        float b = 3.0e38f;
        const float fx = (float)min(px - (cx * kCell - e) + 1, cx * kCell + kCell + e - px) * hx;
        const float fy = (float)min(py - (cy * kCell - e) + 1, cy * kCell + kCell + e - py) * hy;
        const float fz = (float)min(pz - (cz * kCell - e) + 1, cz * kCell + kCell + e - pz) * hz;
        b = fminf(fx, fminf(fy, fz));
        if (b * b >= best) break;
      }
      const int z0 = max(cz - r, 0), z1 = min(cz + r, cg.ncz - 1);
      const int y0 = max(cy - r, 0), y1 = min(cy + r, cg.ncy - 1);
      for (int z = z0; z <= z1; ++z) {
        const int bz = max(max(z * kCell - pz, pz - (z * kCell + kCell - 1)), 0);
        const float gz = (float)bz * hz;
        for (int y = y0; y <= y1; ++y) {
          const int by = max(max(y * kCell - py, py - (y * kCell + kCell - 1)), 0);
          const float gy = (float)by * hy;
          const float gyz = fmaf(gy, gy, gz * gz);
          if (gyz >= best) continue;
          const bool face = z - cz == r || cz - z == r || y - cy == r || cy - y == r;
          const int step = face || r == 0 ? 1 : 2 * r;
          for (int x = cx - r; x <= cx + r; x += step) {
            if (x < 0 || x >= cg.ncx) continue;
            const int oc = (z * cg.ncy + y) * cg.ncx + x;
            const unsigned p0 = so[oc], p1 = so[oc + 1];
            if (p0 == p1) continue;
            const int bx = max(max(x * kCell - px, px - (x * kCell + kCell - 1)), 0);
            const float gx = (float)bx * hx;
            if (fmaf(gx, gx, gyz) >= best) continue;
            for (unsigned k = p0; k < p1; ++k) {
              const unsigned oq = __ldg(lo + k);
              const int qx = x * kCell + (oq & 7), qy = y * kCell + ((oq >> 3) & 7),
                        qz = z * kCell + (oq >> 6);
              const float dx = (float)(px - qx) * hx, dy = (float)(py - qy) * hy,
                          dz = (float)(pz - qz) * hz;
              const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
              if (d2 < best) {
                best = d2;
                wx = qx;
                wy = qy;
                wz = qz;
              }
            }
          }
        }
      }
    }
    const double dx = (double)(px - wx) * hx, dy = (double)(py - wy) * hy,
                 dz = (double)(pz - wz) * hz;
    d[i] = sqrt(dx * dx + dy * dy + dz * dz);
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
