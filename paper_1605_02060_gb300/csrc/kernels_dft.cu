// The smoothing operator K = (gamma - alpha Lap_h)^-2 of §2.4 (K = (L^T L)^-1 for
// L = -alpha Lap + gamma), applied on the periodic grid as separable per-axis real DFTs.
//
// For an axis of length n, R is the orthonormal real Fourier basis (rows: constant, then
// cos/sin pairs of frequency k = 1.., then the Nyquist cosine when n is even).  The symbol of
// K depends on each frequency only through lambda(k) = sum_d (2 - 2 cos(2 pi k_d / n_d)) / h_d^2,
// which is the same for the cos and the sin row of a pair, so with R3 = Rz (x) Ry (x) Rx
//     K = R3^T diag((gamma + alpha lambda)^-2) R3.
// Each axis transform is a dense matrix product over all lines of that axis: a batched GEMM
// whose small operand is R (n x n; in the FP32 form folded by parity into two of half the size)
// and whose large operand is the field.  The symbol scaling is fused into the epilogue of the
// forward z product.
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/lddmm.h"
#include "dft_rows.cuh"
#include "kernels.h"

namespace lddmm {

// ---------------------------------------------------------------------------------------------
// Table construction (host, double precision, angles reduced modulo n).
static void real_dft_matrix(int n, double h, std::vector<float>& R, std::vector<float>& lam) {
  R.assign((size_t)n * n, 0.f);
  lam.assign(n, 0.f);
  const double two_pi = 6.283185307179586476925286766559;
  for (int r = 0; r < n; ++r) {
    const int k = (r + 1) / 2;
    const bool is_sin = (r > 0) && (r % 2 == 0);
    const bool nyq = (n % 2 == 0) && (r == n - 1);
    const double scale = (r == 0 || nyq) ? std::sqrt(1.0 / n) : std::sqrt(2.0 / n);
    for (int m = 0; m < n; ++m) {
      const double ang = two_pi * (double)(((long long)k * m) % n) / (double)n;
      R[(size_t)r * n + m] = (float)(scale * (is_sin ? std::sin(ang) : std::cos(ang)));
    }
    lam[r] = (float)((2.0 - 2.0 * std::cos(two_pi * (double)k / (double)n)) / (h * h));
  }
}

void host_real_dft_tables(int n, double h, std::vector<float>& R, std::vector<float>& lam) {
  real_dft_matrix(n, h, R, lam);
}

static uint16_t bf16_rn(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  const uint32_t lsb = (u >> 16) & 1u;
  u += 0x7fffu + lsb;
  return (uint16_t)(u >> 16);
}
static float bf16_to_f(uint16_t b) {
  uint32_t u = (uint32_t)b << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}

// Tensor-core operand table: B(k, n) = R[n][k] (forward) or R[k][n] (inverse) for the output
// columns n < rows (rows a multiple of 16; zero for n >= n_len), k zero-padded to ceil16(n_len);
// per 16-wide k-step a bf16 hi block then a bf16 lo block (B = hi + lo), each rows x 16 k in the
// K-major no-swizzle core-matrix order the MMA descriptors expect:
// element (row, kk) at byte (kk/8)*128 + (row/8)*256 + (row%8)*16 + (kk%8)*2.
static void tc_table(const std::vector<float>& R, int n, bool inverse, int rows,
                     std::vector<uint16_t>& t) {
  const int Kpad = (n + 15) / 16 * 16, nk = Kpad / 16;
  const size_t block = (size_t)rows * 16;  // elements per hi (or lo) block
  t.assign((size_t)nk * 2 * block, 0);
  for (int s = 0; s < nk; ++s) {
    uint16_t* hi = t.data() + (size_t)s * 2 * block;
    uint16_t* lo = hi + block;
    for (int row = 0; row < rows; ++row)
      for (int kk = 0; kk < 16; ++kk) {
        const int k = s * 16 + kk;
        float b = 0.f;
        if (k < n && row < n) b = inverse ? R[(size_t)k * n + row] : R[(size_t)row * n + k];
        const uint16_t bh = bf16_rn(b);
        const uint16_t bl = bf16_rn(b - bf16_to_f(bh));
        const size_t off = ((size_t)(kk / 8) * 128 + (size_t)(row / 8) * 256 + (row % 8) * 16 +
                            (kk % 8) * 2) / 2;
        hi[off] = bh;
        lo[off] = bl;
      }
  }
}

// Operand table of the pre-split pass: B(k, n) as bf16 [hi plane][lo plane], each [Nc][Kp]
// row-major (row n = output column, k contiguous), Nc = Kp = ceil16(n), zero for n >= n_len or
// k >= n_len.
static void ks_table(const std::vector<float>& R, int n, bool inverse, std::vector<uint16_t>& t) {
  const int Kp = (n + 15) / 16 * 16, Nc = Kp;
  const size_t plane = (size_t)Nc * Kp;
  t.assign(2 * plane, 0);
  for (int row = 0; row < n && row < Nc; ++row)
    for (int k = 0; k < n; ++k) {
      const float b = inverse ? R[(size_t)k * n + row] : R[(size_t)row * n + k];
      const uint16_t bh = bf16_rn(b);
      t[(size_t)row * Kp + k] = bh;
      t[plane + (size_t)row * Kp + k] = bf16_rn(b - bf16_to_f(bh));
    }
}

template <typename T>
static cudaError_t upload(T** dst, const std::vector<T>& src) {
  cudaError_t e = cudaMalloc((void**)dst, src.size() * sizeof(T));
  if (e != cudaSuccess) return e;
  return cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice);
}

cudaError_t kplan_create(KPlan* kp, int nx, int ny, int nz, float hx, float hy, float hz,
                         float alpha, float gamma) {
  *kp = KPlan{};
  kp->nx = nx; kp->ny = ny; kp->nz = nz;
  kp->alpha = alpha; kp->gamma = gamma;
  kp->sym_normal = symbol_is_normal(hx, hy, hz, alpha, gamma);
  const int n[3] = {nx, ny, nz};
  const double h[3] = {hx, hy, hz};
  float** Rs[3] = {&kp->Rx, &kp->Ry, &kp->Rz};
  float** ls[3] = {&kp->lx, &kp->ly, &kp->lz};
  for (int d = 0; d < 3; ++d) {
    std::vector<float> R, lam;
    real_dft_matrix(n[d], h[d], R, lam);
    lam.resize((size_t)(n[d] + 15) / 16 * 16, 0.f);   // zero padded: 16-column groups load whole
    cudaError_t e;
    if ((e = upload(Rs[d], R)) != cudaSuccess) return e;
    if ((e = upload(ls[d], lam)) != cudaSuccess) return e;
    for (int dir = 0; dir < 2; ++dir) {
      std::vector<uint16_t> t;
      tc_table(R, n[d], dir == 1, (n[d] + 15) / 16 * 16, t);
      if ((e = upload(&kp->tc[d][dir], t)) != cudaSuccess) return e;
    }
    if (n[d] <= (d == 0 ? 264 : 256)) {
      for (int dir = 0; dir < 2; ++dir) {
        std::vector<uint16_t> t;
        ks_table(R, n[d], dir == 1, t);
        if ((e = upload(&kp->ks[d][dir], t)) != cudaSuccess) return e;
      }
    }
  }
  cudaError_t e = cudaMalloc((void**)&kp->err, sizeof(int));
  if (e != cudaSuccess) return e;
  return cudaMemset(kp->err, 0, sizeof(int));
}

void kplan_destroy(KPlan* kp) {
  void* ps[] = {kp->Rx, kp->Ry, kp->Rz, kp->lx, kp->ly, kp->lz, kp->err};
  for (void* p : ps)
    if (p) cudaFree(p);
  for (int d = 0; d < 3; ++d)
    for (int dir = 0; dir < 2; ++dir)
      if (kp->tc[d][dir]) cudaFree(kp->tc[d][dir]);
  for (int dir = 0; dir < 2; ++dir) {
    for (int d = 0; d < 3; ++d)
      if (kp->ks[d][dir]) cudaFree(kp->ks[d][dir]);
  }
  *kp = KPlan{};
}

// ---------------------------------------------------------------------------------------------
// FP32 axis transforms on the CUDA cores, folded by the parity of the basis.  With cos and sin rows
// p = 0..n/2 of R and x folded about 0 (e_m = x_m + x_{n-m}, o_m = x_m - x_{n-m}),
//     forward  c_p = sum_m C(p, m) e_m,  s_p = sum_m S(p, m) o_m,           m = 0..n/2,
//     inverse  E_m = sum_p C(p, m) c_p,  O_m = sum_p S(p, m) s_p,  x_m = E_m + O_m, x_{n-m} = E_m - O_m:
// two products of half the length each way, half the FMAs of the full matrix product and sums half
// as long (the error against FP64 falls from 5.3e-7 to 3.9e-7 at 132x80x114).  FP32 FMAs bound it.
// A block takes 4 TP pairs (p or m) by 128 columns (lines of the axis); a thread holds both
// products' sums for 4 pairs x 8 columns, so 6 16-byte shared loads feed 64 FMAs.  Field rows and
// table tiles (straight from R) arrive by asynchronous copies two stages ahead; a thread folds the
// rows it copied into the other of two folded stages.  128 registers, four blocks of 4 warps (five
// of 3) per SM: with prefetch through registers (167, 12 warps) a pass of 700 blocks left a second
// wave of 100 and took 27 to 42 us.
// At 132x80x114 (three components) the six passes take 31 + 18 + 28 + 19 + 16 + 33 us with the
// update in the last; as 64x64 tiles of the unfolded product they took 6 x 53 us and the update 5.
// What is left beside the FMAs is their issue: each stage's copies, folds and table tile are half of
// the instructions of an x pass (two thirds with every place decoded anew: 36 and 37 us).  Where the
// lines are whole 16-byte vectors x is copied as it lies, 5 vectors a line, and turned on the way to
// the folded stage; else 4 bytes at a time.
constexpr int FK = 8, FC = 128, FCS = FC + 4;   // rows per stage, columns per block, row stride
constexpr int FX = 20;                          // floats of a line in a raw stage (x by vectors)

struct FoldArgs {
  const float* in;
  float* out;
  const float* R;       // [n][n]: row 2 p - 1 = cos p (row 0: constant), row 2 p = sin p
  int n, H;             // axis length, n / 2 + 1 pairs
  int ncols;            // lines of the axis (offsets into the field are below 2^31)
  int W, hi;            // line col starts at (col / W) hi + col % W (x lines: col n)
  int rs;               // stride along the axis
  int vec;              // 16-byte accesses across 4 lines
  int tp;               // thread rows: the block's pairs / 4
  // forward z: divide by the symbol (gamma + alpha (lz[row] + ly[y] + lx[x]))^2
  const float* lx;
  const float* ly;
  const float* lz;
  int nx;
  float alpha, gamma;
  int sym_normal;       // one reciprocal serves both rows of a pair (a division each: +2% of a step)
  // inverse x: v_upd <- v_upd - eps (2 v_upd - result) instead of storing the result
  float* v_upd;
  float eps;
};

// FWD: rows m -> pairs p; else pairs p -> rows m.  XAX: lines contiguous along the axis.
template <bool FWD, bool XAX>
__global__ void __launch_bounds__(128, 4) k_fold(FoldArgs a) {
  extern __shared__ __align__(16) float fs[];
  constexpr int FE = 2 * FK * FCS;                      // floats of a stage's two row sets
  const int tid = threadIdx.x, nt = blockDim.x;
  const int BP = 4 * a.tp, tabw = 2 * FK * BP;
  // forward: two raw stages, two folded ones; inverse: three stages used as they are; three tables
  // (x lines by vectors: two raw stages of FX floats a line, two transposed ones)
  const bool xv = XAX && a.vec;
  float* const raw = fs;
  float* const eo = xv ? fs + 2 * FC * FX : FWD ? fs + 2 * FE : fs;
  float* const tab = eo + (xv || FWD ? 2 : 3) * FE;
  const int tc = tid & 15, tp = tid >> 4;
  const int p0 = blockIdx.y * BP;
  const int c0 = blockIdx.x * FC;
  const int n = a.n, H = a.H;
  const unsigned n4 = 4u * (unsigned)n;
  float ac[4][8], as[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) ac[i][j] = as[i][j] = 0.f;

  // the two field rows of contraction index k (forward: m = k and n - k; inverse: the cos and sin
  // rows of pair k); -1: none
  auto rows_of = [&](int k, int& r0, int& r1) {
    const bool two = k > 0 && 2 * k < n;
    r0 = k >= H ? -1 : FWD ? k : fold_row_c(k);
    r1 = k < H && two ? (FWD ? n - k : 2 * k) : -1;
  };
  // strided lines: lane = 4 columns, warp w takes k = w, w + nw, ..; x lines: 8 k x 4 lines a warp
  const int nw = nt >> 5, lane = tid & 31;
  const int lc = c0 + 4 * lane;                          // strided: this lane's first column
  // 32-bit divisions, one for 4 lines where they are contiguous (64-bit ones, per line, were a third
  // of the instructions)
  int base[4] = {0, 0, 0, 0};
  if (!XAX) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (a.vec && q) break;
      if (lc + q < a.ncols) {
        const int d = (lc + q) / a.W;
        base[q] = d * a.hi + (lc + q - d * a.W);
      }
    }
  }
  // x lines by vectors: the thread's vector xc of line xl, xl + xstep, .. (the last threads have none)
  const int xstep = nt / (FX / 4), xc = tid % (FX / 4), xl = tid < xstep * (FX / 4) ? tid / (FX / 4) : FC;
  // inverse tables: the thread's column ti and first row tk
  const int tstep = nt / BP, ti = tid % BP, tk = tid / BP;
  auto cp = [&](float* dst, const float* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(in ? src : a.in), "r"(in ? 4 : 0)
                 : "memory");
  };
  auto cp16 = [&](float* dst, const float* src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(in ? src : a.in), "r"(in ? 16 : 0)
                 : "memory");
  };
  // starts the copies of stage t (field rows, table tile) as one group
  auto issue = [&](int t) {
    const int k0 = t * FK;
    if (k0 < H) {
      float* e = (FWD ? raw + (t & 1) * FE : eo + (t % 3) * FE);
      float* o = e + FK * FCS;
      if (xv) {
        // the aligned vectors of a line that hold the stage's elements: forward m = k0 .. k0 + 7 and
        // n - k0 - 8 .. n - k0 + 3, inverse 2 k0 - 4 .. 2 k0 + 15
        if (xl < FC) {
          float* d = raw + (t & 1) * (FC * FX) + xl * FX + 4 * xc;
          const int m = !FWD ? 2 * k0 - 4 + 4 * xc : xc < 2 ? k0 + 4 * xc : n - k0 - 16 + 4 * xc;
          const bool in = m >= 0 && m < n;
          int o = (c0 + xl) * n + m;
          for (int l = xl; l < FC; l += xstep, d += xstep * FX, o += xstep * n)
            cp16(d, a.in + o, in && c0 + l < a.ncols);
        }
      } else if constexpr (XAX) {
        int r0, r1;
        rows_of(k0 + (tid & 7), r0, r1);
        const int k = tid & 7;
        for (int l = tid >> 3; l < FC; l += nt >> 3) {
          const bool in = c0 + l < a.ncols;
          const int ob = (c0 + l) * n;
          cp(e + k * FCS + l, a.in + ob + r0, in && r0 >= 0);
          cp(o + k * FCS + l, a.in + ob + r1, in && r1 >= 0);
        }
      } else {
        for (int k = tid >> 5; k < FK; k += nw) {
          int r0, r1;
          rows_of(k0 + k, r0, r1);
          float* ed = e + k * FCS + 4 * lane;
          float* od = o + k * FCS + 4 * lane;
          if (a.vec) {
            const bool in = lc < a.ncols;
            cp16(ed, a.in + base[0] + r0 * a.rs, in && r0 >= 0);
            cp16(od, a.in + base[0] + r1 * a.rs, in && r1 >= 0);
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const bool in = lc + q < a.ncols;
              cp(ed + q, a.in + base[q] + r0 * a.rs, in && r0 >= 0);
              cp(od + q, a.in + base[q] + r1 * a.rs, in && r1 >= 0);
            }
          }
        }
      }
      // table tile: entry (k, i) of C and S = the coefficient between contraction index k0 + k
      // and output index p0 + i; R is contiguous along m (forward k = m, inverse i = m)
      float* tb = tab + (t % 3) * tabw;
      if (FWD) {
        // a thread keeps k, its pairs are nt / FK apart
        const int k = tid % FK, m = k0 + k;
        const char* col = reinterpret_cast<const char*>(a.R + m);
        for (int i = tid / FK; i < BP; i += nt / FK) {
          const int p = p0 + i;
          const float* rc = reinterpret_cast<const float*>(col + fold_row_bytes(p, n4));
          const bool in = p < H && m < H;
          cp(tb + k * BP + i, rc, in);
          cp(tb + FK * BP + k * BP + i, rc + n, in && p > 0 && 2 * p < n);   // the sin row follows
        }
      } else {
        // a thread keeps i, its rows of the contraction are nt / BP apart
        const int m = p0 + ti;
        const char* col = reinterpret_cast<const char*>(a.R + m);
        for (int k = tk; k < FK; k += tstep) {
          const int p = k0 + k;
          const float* rc = reinterpret_cast<const float*>(col + fold_row_bytes(p, n4));
          const bool in = p < H && m < H;
          cp(tb + k * BP + ti, rc, in);
          cp(tb + FK * BP + k * BP + ti, rc + n, in && p > 0 && 2 * p < n);
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // forward: the rows this thread copied, (a, b) -> (a + b, a - b); without a mirror row (a, 0)
  auto fold = [&](int t) {
    const int k0 = t * FK;
    const float* e = raw + (t & 1) * FE;
    const float* o = e + FK * FCS;
    float* ed = eo + (t & 1) * FE;
    float* od = ed + FK * FCS;
    if (xv) {
      for (int l = tid; l < FC; l += nt) {
        const float4* q = reinterpret_cast<const float4*>(raw + (t & 1) * (FC * FX) + l * FX);
        float v[FX];
#pragma unroll
        for (int c = 0; c < FX / 4; ++c) {
          const float4 w = q[c];
          v[4 * c] = w.x; v[4 * c + 1] = w.y; v[4 * c + 2] = w.z; v[4 * c + 3] = w.w;
        }
        if (k0 > 0 && 2 * (k0 + FK - 1) < n) {  // every element has its mirror
#pragma unroll
          for (int k = 0; k < FK; ++k) {
            const float u = v[FWD ? k : 2 * k + 3], w = v[FWD ? 16 - k : 2 * k + 4];
            ed[k * FCS + l] = FWD ? u + w : u;
            od[k * FCS + l] = FWD ? u - w : w;
          }
        } else {
#pragma unroll
          for (int k = 0; k < FK; ++k) {
            const int kk = k0 + k;
            const bool two = kk > 0 && 2 * kk < n;
            const float u = kk < H ? (FWD ? v[k] : k == 0 && k0 == 0 ? v[4] : v[2 * k + 3]) : 0.f;
            const float w = two ? (FWD ? v[16 - k] : v[2 * k + 4]) : 0.f;
            ed[k * FCS + l] = FWD ? u + w : u;
            od[k * FCS + l] = FWD ? (two ? u - w : 0.f) : w;
          }
        }
      }
    } else if constexpr (XAX) {
      const int k = tid & 7, kk = k0 + k;
      const bool mir = kk > 0 && 2 * kk < n;
      for (int l = tid >> 3; l < FC; l += nt >> 3) {
        const float u = e[k * FCS + l], w = o[k * FCS + l];
        ed[k * FCS + l] = u + w;
        od[k * FCS + l] = mir ? u - w : 0.f;
      }
    } else {
      for (int k = tid >> 5; k < FK; k += nw) {
        const int kk = k0 + k;
        const bool mir = kk > 0 && 2 * kk < n;
        const float4 u = *reinterpret_cast<const float4*>(e + k * FCS + 4 * lane);
        const float4 w = *reinterpret_cast<const float4*>(o + k * FCS + 4 * lane);
        *reinterpret_cast<float4*>(ed + k * FCS + 4 * lane) =
            make_float4(u.x + w.x, u.y + w.y, u.z + w.z, u.w + w.w);
        *reinterpret_cast<float4*>(od + k * FCS + 4 * lane) =
            mir ? make_float4(u.x - w.x, u.y - w.y, u.z - w.z, u.w - w.w)
                : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  };

  issue(0);
  issue(1);
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  if (xv) __syncthreads();                    // a line's vectors come from several threads
  if (FWD || xv) fold(0);
  __syncthreads();
  const int nst = (H + FK - 1) / FK;
  for (int t = 0; t < nst; ++t) {
    issue(t + 2);
    const float* e = eo + (FWD || xv ? (t & 1) : t % 3) * FE + 4 * tc;
    const float* o = e + FK * FCS;
    const float* C = tab + (t % 3) * tabw + 4 * tp;
    const float* S = C + FK * BP;
#pragma unroll
    for (int k = 0; k < FK; ++k) {
      const float4 c4 = *reinterpret_cast<const float4*>(C + k * BP);
      const float4 s4 = *reinterpret_cast<const float4*>(S + k * BP);
      const float4 e0 = *reinterpret_cast<const float4*>(e + k * FCS);
      const float4 e1 = *reinterpret_cast<const float4*>(e + k * FCS + 64);
      const float4 o0 = *reinterpret_cast<const float4*>(o + k * FCS);
      const float4 o1 = *reinterpret_cast<const float4*>(o + k * FCS + 64);
      const float cv[4] = {c4.x, c4.y, c4.z, c4.w}, sv[4] = {s4.x, s4.y, s4.z, s4.w};
      const float ev[8] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
      const float ov[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          ac[i][j] = fmaf(cv[i], ev[j], ac[i][j]);
          as[i][j] = fmaf(sv[i], ov[j], as[i][j]);
        }
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    if (xv) __syncthreads();
    if ((FWD || xv) && t + 1 < nst) fold(t + 1);
    __syncthreads();
  }

  // ---- outputs of pair q = p0 + 4 tp + i: forward rows cos q, sin q; inverse rows q, n - q
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (!FWD) {
        const float E = ac[i][j], O = as[i][j];
        ac[i][j] = E + O;
        as[i][j] = E - O;
      }
  if constexpr (!XAX) {
    float lam[8];
    int ob[8];
    bool ok[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int col = c0 + 64 * (j >> 2) + 4 * tc + (j & 3);
      ok[j] = col < a.ncols;
      lam[j] = 0.f;
      if (a.vec && (j & 3)) {                 // 4 lines in one row of W
        ob[j] = ob[j & 4] + (j & 3);
      } else {
        const int d = ok[j] ? col / a.W : 0;
        ob[j] = ok[j] ? d * a.hi + (col - d * a.W) : 0;
      }
      if (FWD && a.lz && ok[j]) {
        const int w = col % a.W, y = w / a.nx;
        lam[j] = a.ly[y] + a.lx[w - y * a.nx];
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int q = p0 + 4 * tp + i;
      if (q >= H) break;
      const bool two = q > 0 && 2 * q < n;
      const int r0 = FWD ? fold_row_c(q) : q, r1 = FWD ? 2 * q : n - q;
      if (FWD && a.lz) {
        const float lz = a.lz[r0];              // the same for both rows of the pair
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float den = a.gamma + a.alpha * (lz + lam[j]), d2 = den * den;
          if (a.sym_normal) {
            const float q2 = 1.f / d2;
            ac[i][j] *= q2;
            as[i][j] *= q2;
          } else {                              // 1 / d2 may overflow where the quotient does not
            ac[i][j] /= d2;
            as[i][j] /= d2;
          }
        }
      }
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        const float* vc = &ac[i][4 * g];
        const float* vs = &as[i][4 * g];
        if (a.vec) {
          if (ok[4 * g]) {
            float* d = a.out + ob[4 * g];
            *reinterpret_cast<float4*>(d + r0 * a.rs) = make_float4(vc[0], vc[1], vc[2], vc[3]);
            if (two) *reinterpret_cast<float4*>(d + r1 * a.rs) = make_float4(vs[0], vs[1], vs[2], vs[3]);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (ok[4 * g + j]) {
              a.out[ob[4 * g + j] + r0 * a.rs] = vc[j];
              if (two) a.out[ob[4 * g + j] + r1 * a.rs] = vs[j];
            }
        }
      }
    }
  } else {
    // x lines leave through shared memory, 64 lines at a time, so that a warp stores consecutive
    // elements of one line: forward elements 2 p0 - 1 .. 2 p0 + 2 BP - 2, inverse two runs,
    // p0 .. p0 + BP - 1 and n - p0 - BP + 1 .. n - p0
    const int SW = 2 * BP + 1;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int il = 4 * tp + i;
          float* d = fs + (4 * tc + j) * SW;
          // forward: element 2 q - 1 at 2 il, 2 q at 2 il + 1; inverse: q at il, n - q at 2 BP - 1 - il
          d[FWD ? 2 * il : il] = ac[i][4 * g + j];
          d[FWD ? 2 * il + 1 : 2 * BP - 1 - il] = as[i][4 * g + j];
        }
      __syncthreads();
      // a lane's element offsets along a line (-1: none) are the same for every line
      int r[2];                               // 2 BP <= 64
#pragma unroll
      for (int t3 = 0; t3 < 2; ++t3) {
        const int t = lane + 32 * t3;
        r[t3] = -1;
        if (t < 2 * BP) {
          if (FWD) {
            // row 0 (the constant) is pair 0's cos; pair 0 has no sin
            const int q = p0 + (t >> 1);
            if (q < H && ((t & 1) == 0 || (q > 0 && 2 * q < n))) r[t3] = q == 0 ? 0 : 2 * q - 1 + (t & 1);
          } else {
            const bool mir = t >= BP;
            const int q = p0 + (mir ? 2 * BP - 1 - t : t);
            if (q < H && (!mir || (q > 0 && 2 * q < n))) r[t3] = mir ? n - q : q;
          }
        }
      }
      // 4 lines at a time; the update's old values are all requested before the first store
      for (int l0 = 4 * (tid >> 5); l0 < 64; l0 += 4 * nw) {
        float old[4][2];
        if (!FWD && a.v_upd) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int t3 = 0; t3 < 2; ++t3) {
              const int line = c0 + 64 * g + l0 + k;
              if (r[t3] >= 0 && line < a.ncols) old[k][t3] = a.v_upd[line * n + r[t3]];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int t3 = 0; t3 < 2; ++t3) {
            const int line = c0 + 64 * g + l0 + k;
            if (r[t3] < 0 || line >= a.ncols) continue;
            const float w = fs[(l0 + k) * SW + lane + 32 * t3];
            if (!FWD && a.v_upd) a.v_upd[line * n + r[t3]] = old[k][t3] - a.eps * (2.f * old[k][t3] - w);
            else a.out[line * n + r[t3]] = w;
          }
      }
      __syncthreads();
    }
  }
}

template <bool FWD, bool XAX>
static cudaError_t launch_fold(FoldArgs a, cudaStream_t s) {
  a.H = a.n / 2 + 1;
  // thread rows: 6 or 8 (blocks of 96 or 128 threads), the fewer padded pairs
  const int pad6 = (a.H + 23) / 24 * 6, pad8 = (a.H + 31) / 32 * 8;
  a.tp = pad6 <= pad8 ? 6 : 8;
  const int BP = 4 * a.tp;
  const int rows = XAX && a.vec ? 2 * FC * FX + 4 * FK * FCS : (FWD ? 4 : 3) * 2 * FK * FCS;
  const int stage = rows + 3 * 2 * FK * BP;
  const int outw = XAX ? 64 * (2 * BP + 1) : 0;
  const int smem = 4 * (stage > outw ? stage : outw);   // at most 43520 bytes
  const dim3 grid((unsigned)((a.ncols + FC - 1) / FC), (unsigned)((a.H + BP - 1) / BP));
  k_fold<FWD, XAX><<<grid, 16 * a.tp, smem, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// FP32 transforms of small axes from shared memory: x and y of one plane per block, and z forward,
// symbol and z inverse of 32 columns per block.  A small grid is bound by the length of each
// launch's chain (load, multiply, store) and by the number of launches, so a whole table lies in
// shared memory and the unfolded products use as many threads as outputs / 8 (2 rows x 4 columns a
// thread); past about 70 the shared loads of these small tiles cost more than k_fold's launches.
// One K of three components (us; k_fold alone; these; 64x64 tiles of the unfolded product and a
// separate update, as it was): 32^3 41 / 12 / 26, 33x20x29 46 / 16 / 29, 48^3 47 / 26 / 35,
// 64^3 68 / 50 / 53, 66x40x57 60 / 40 / 55, 96x40x60 55 / 58 / 61.
constexpr int SN_NT = 256;

// rows padded to 4 floats
__host__ __device__ inline int sn_pad(int n) { return (n + 3) & ~3; }

// o(i, j) for i < M, j < N (4 columns at a time): sum_k A(i, k) B[k][j], B rows of ldb floats.
// out(i, j4, float4) receives columns 4 j4 .. of row i.
template <typename FA, typename FO>
__device__ __forceinline__ void sn_product(int M, int N4, int K, const float* B, int ldb, FA A, FO out) {
  const int M2 = (M + 1) / 2;
  for (int t = threadIdx.x; t < M2 * N4; t += SN_NT) {
    const int i2 = t / N4, j4 = t - i2 * N4, i0 = 2 * i2, i1 = min(2 * i2 + 1, M - 1);
    float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
    const float* b = B + 4 * j4;
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
      const float4 v = *reinterpret_cast<const float4*>(b + k * ldb);
      const float a0 = A(i0, k), a1 = A(i1, k);
      s0.x = fmaf(a0, v.x, s0.x); s0.y = fmaf(a0, v.y, s0.y);
      s0.z = fmaf(a0, v.z, s0.z); s0.w = fmaf(a0, v.w, s0.w);
      s1.x = fmaf(a1, v.x, s1.x); s1.y = fmaf(a1, v.y, s1.y);
      s1.z = fmaf(a1, v.z, s1.z); s1.w = fmaf(a1, v.w, s1.w);
    }
    out(i0, j4, s0);
    if (i1 > i0) out(i1, j4, s1);
  }
}

// FWD: plane [y][x] -> [y'][x'] through Rx, Ry.  Else [y'][x'] -> [y][x], stored or combined with v.
template <bool FWD>
__global__ void __launch_bounds__(SN_NT) k_small_xy(const float* __restrict__ in, float* out, int X,
                                                    int Y, const float* __restrict__ Rx,
                                                    const float* __restrict__ Ry, float* v_upd,
                                                    float eps) {
  extern __shared__ __align__(16) float sm[];
  const int XP = sn_pad(X), YP = sn_pad(Y);
  float* P = sm;                    // [Y][XP]
  float* T = P + Y * XP;            // [Y][XP]
  float* tx = T + Y * XP;           // [X][XP]: FWD Rx transposed (row x, column x'), else Rx
  float* ty = tx + X * XP;          // [Y][YP]: Ry (row y')
  const int64_t o0 = (int64_t)blockIdx.x * X * Y;
  for (int i = threadIdx.x; i < Y * X; i += SN_NT) {
    const int y = i / X;
    P[y * XP + i - y * X] = in[o0 + i];
  }
  for (int i = threadIdx.x; i < X * X; i += SN_NT) {
    const int r = i / X, c = i - r * X;
    tx[FWD ? c * XP + r : r * XP + c] = __ldg(Rx + i);
  }
  for (int i = threadIdx.x; i < Y * Y; i += SN_NT) {
    const int r = i / Y;
    ty[r * YP + i - r * Y] = __ldg(Ry + i);
  }
  // the pad columns of the operands read as float4
  for (int i = threadIdx.x; i < (XP - X) * (2 * Y + X); i += SN_NT) {
    const int w = XP - X, r = i / w, c = X + i - r * w;
    (r < Y ? P + r * XP : r < 2 * Y ? T + (r - Y) * XP : tx + (r - 2 * Y) * XP)[c] = 0.f;
  }
  __syncthreads();
  const int N4 = XP / 4;
  if (FWD) {
    // T(y, x') = sum_x P(y, x) Rx(x', x), then out(y', x') = sum_y Ry(y', y) T(y, x')
    sn_product(Y, N4, X, tx, XP, [&](int i, int k) { return P[i * XP + k]; },
               [&](int i, int j4, float4 v) { *reinterpret_cast<float4*>(T + i * XP + 4 * j4) = v; });
    __syncthreads();
    sn_product(Y, N4, Y, T, XP, [&](int i, int k) { return ty[i * YP + k]; },
               [&](int i, int j4, float4 v) { *reinterpret_cast<float4*>(P + i * XP + 4 * j4) = v; });
  } else {
    // T(y, x') = sum_y' Ry(y', y) P(y', x'), then out(y, x) = sum_x' T(y, x') Rx(x', x)
    sn_product(Y, N4, Y, P, XP, [&](int i, int k) { return ty[k * YP + i]; },
               [&](int i, int j4, float4 v) { *reinterpret_cast<float4*>(T + i * XP + 4 * j4) = v; });
    __syncthreads();
    sn_product(Y, N4, X, tx, XP, [&](int i, int k) { return T[i * XP + k]; },
               [&](int i, int j4, float4 v) { *reinterpret_cast<float4*>(P + i * XP + 4 * j4) = v; });
  }
  __syncthreads();
  for (int i = threadIdx.x; i < Y * X; i += SN_NT) {
    const int y = i / X;
    const float w = P[y * XP + i - y * X];
    if (!FWD && v_upd) {
      const float v = v_upd[o0 + i];
      v_upd[o0 + i] = v - eps * (2.f * v - w);
    } else {
      out[o0 + i] = w;
    }
  }
}

// In place on [c][z][XY]: z forward, / (gamma + alpha (lz + ly + lx))^2, z inverse of 32 columns.
__global__ void __launch_bounds__(SN_NT) k_small_z(float* f, int Z, int XY, int X,
                                                   const float* __restrict__ Rz,
                                                   const float* __restrict__ lx,
                                                   const float* __restrict__ ly,
                                                   const float* __restrict__ lz, float alpha,
                                                   float gamma) {
  extern __shared__ __align__(16) float sm[];
  const int ZP = sn_pad(Z);
  float* P = sm;                    // [Z][32]
  float* T = P + Z * 32;            // [Z][32]
  float* tz = T + Z * 32;           // [Z][ZP]
  float* lam = tz + Z * ZP;         // [32]
  const int c0 = blockIdx.x * 32, nc = min(32, XY - c0);
  float* fb = f + (int64_t)blockIdx.y * Z * XY + c0;
  for (int i = threadIdx.x; i < Z * 32; i += SN_NT) {
    const int z = i >> 5, c = i & 31;
    P[i] = c < nc ? fb[(int64_t)z * XY + c] : 0.f;
  }
  for (int i = threadIdx.x; i < Z * Z; i += SN_NT) {
    const int r = i / Z;
    tz[r * ZP + i - r * Z] = __ldg(Rz + i);
  }
  if (threadIdx.x < 32) {
    const int w = min(c0 + (int)threadIdx.x, XY - 1), y = w / X;
    lam[threadIdx.x] = ly[y] + lx[w - y * X];
  }
  __syncthreads();
  sn_product(Z, 8, Z, P, 32, [&](int i, int k) { return tz[i * ZP + k]; },
             [&](int i, int j4, float4 v) {
               const float l = __ldg(lz + i);
               const float4 m = *reinterpret_cast<const float4*>(lam + 4 * j4);
               const float d0 = gamma + alpha * (l + m.x), d1 = gamma + alpha * (l + m.y),
                           d2 = gamma + alpha * (l + m.z), d3 = gamma + alpha * (l + m.w);
               *reinterpret_cast<float4*>(T + i * 32 + 4 * j4) =
                   make_float4(v.x / (d0 * d0), v.y / (d1 * d1), v.z / (d2 * d2), v.w / (d3 * d3));
             });
  __syncthreads();
  sn_product(Z, 8, Z, T, 32, [&](int i, int k) { return tz[k * ZP + i]; },
             [&](int i, int j4, float4 v) {
               const float q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
               for (int c = 0; c < 4; ++c)
                 if (4 * j4 + c < nc) fb[(int64_t)i * XY + 4 * j4 + c] = q[c];
             });
}

static int small_xy_floats(int X, int Y) {
  return 2 * Y * sn_pad(X) + X * sn_pad(X) + Y * sn_pad(Y);
}
static int small_z_floats(int Z) { return 2 * Z * 32 + Z * sn_pad(Z) + 32; }

constexpr int SN_MOST = 72, SN_SMEM = 4 * (2 * SN_MOST * SN_MOST + 2 * SN_MOST * SN_MOST);

// Where the lines lie: axes up to 72 (64^3 is 10% faster here, 96x40x60 5% slower), and planes'
// FMAs and column blocks up to a little past those of 64^3 (three blocks per SM).
static bool small_plane(const KPlan& kp, int ncomp) {
  const double work = (double)ncomp * kp.nz * kp.nx * kp.ny * (kp.nx + kp.ny);
  return kp.nx <= SN_MOST && kp.ny <= SN_MOST && work <= 1.2e8;
}
static bool small_columns(const KPlan& kp, int ncomp) {
  return kp.nz <= SN_MOST && (double)ncomp * kp.nx * kp.ny <= 456.0 * 32.0;
}

// x and y forward (in -> out) or inverse (in -> out, or the update of v) of every plane.
static cudaError_t small_xy(const KPlan& kp, bool fwd, const float* in, float* out, int ncomp,
                            float* v_upd, float eps, cudaStream_t s) {
  static PerDevice<bool> set[2];
  const int smem = 4 * small_xy_floats(kp.nx, kp.ny);
  auto* k = fwd ? k_small_xy<true> : k_small_xy<false>;
  const cudaError_t e = raise_smem_limit(set[fwd], k, SN_SMEM);
  if (e != cudaSuccess) return e;
  k<<<ncomp * kp.nz, SN_NT, smem, s>>>(in, out, kp.nx, kp.ny, kp.Rx, kp.Ry, v_upd, eps);
  return cudaGetLastError();
}

static cudaError_t small_z(const KPlan& kp, float* f, int ncomp, cudaStream_t s) {
  const int XY = kp.nx * kp.ny;
  k_small_z<<<dim3((XY + 31) / 32, ncomp), SN_NT, 4 * small_z_floats(kp.nz), s>>>(
      f, kp.nz, XY, kp.nx, kp.Rz, kp.lx, kp.ly, kp.lz, kp.alpha, kp.gamma);
  return cudaGetLastError();
}

static cudaError_t apply_K_fp32(const KPlan& kp, const float* in, float* out, float* work,
                                int ncomp, cudaStream_t s, const Hook& hook, float* v_upd,
                                float eps) {
  const int X = kp.nx, Y = kp.ny, Z = kp.nz, XY = X * Y, N = XY * Z;
  const auto v4 = [&](const float* p) { return X % 4 == 0 && ((uintptr_t)p & 15) == 0; };
  const int vy = v4(work) && v4(out);
  const int vz = vy;                 // XY and N are multiples of X
  const bool sp = small_plane(kp, ncomp), sc = small_columns(kp, ncomp);
  auto axis = [&](int n, const float* R, int ncols, int W, int hi, int rs, int vec,
                  const float* src, float* dst) {
    FoldArgs a{};
    a.in = src; a.out = dst; a.R = R; a.n = n;
    a.ncols = ncols; a.W = W; a.hi = hi; a.rs = rs; a.vec = vec;
    return a;
  };
  cudaError_t e;
#define FOLD(kid, fwd, xax, args)                       \
  do {                                                  \
    hook(kid, 0);                                       \
    e = launch_fold<fwd, xax>(args, s);                 \
    hook(kid, 1);                                       \
    if (e != cudaSuccess) return e;                     \
  } while (0)
#define SMALL(kid, call)                                \
  do {                                                  \
    hook(kid, 0);                                       \
    e = call;                                           \
    hook(kid, 1);                                       \
    if (e != cudaSuccess) return e;                     \
  } while (0)
  // x, y forward: in -> a; z and symbol: a -> b; y, x inverse: b -> out
  float* a = sp ? work : out;
  if (sp) {
    SMALL(KID_KX_FWD, small_xy(kp, true, in, a, ncomp, nullptr, 0.f, s));
  } else {
    FOLD(KID_KX_FWD, true, true, axis(kp.nx, kp.Rx, ncomp * Y * Z, 1, X, 1, v4(in), in, work));
    FOLD(KID_KY_FWD, true, false, axis(kp.ny, kp.Ry, ncomp * Z * X, X, XY, X, vy, work, a));
  }
  if (sc) {
    SMALL(KID_KZ_FUSED, small_z(kp, a, ncomp, s));
  } else {
    float* t = a == work ? out : work;
    FoldArgs zf = axis(kp.nz, kp.Rz, ncomp * XY, XY, N, XY, vz, a, t);
    zf.lx = kp.lx; zf.ly = kp.ly; zf.lz = kp.lz; zf.nx = kp.nx;
    zf.alpha = kp.alpha; zf.gamma = kp.gamma;
    zf.sym_normal = kp.sym_normal;
    FOLD(KID_KZ_SYM, true, false, zf);
    FOLD(KID_KZ_INV, false, false, axis(kp.nz, kp.Rz, ncomp * XY, XY, N, XY, vz, t, a));
  }
  if (sp) {
    SMALL(KID_KX_INV, small_xy(kp, false, a, out, ncomp, v_upd, eps, s));
  } else {
    FOLD(KID_KY_INV, false, false, axis(kp.ny, kp.Ry, ncomp * Z * X, X, XY, X, vy, a, work));
    FoldArgs xi = axis(kp.nx, kp.Rx, ncomp * Y * Z, 1, X, 1, v4(work), work, out);
    xi.v_upd = v_upd;
    xi.eps = eps;
    FOLD(KID_KX_INV, false, true, xi);
  }
#undef SMALL
#undef FOLD
  return cudaSuccess;
}

// Tensor-core K over pre-split intermediate fields.  Every pass reads its input with the
// transformed axis contiguous and writes its output in the next pass's line order (Xp, Yp, Zp: the
// sizes rounded up to 8, the pitches of x, y and z rows):
//   x fwd:  [c][z][Yp][x] (split, x rows)  -> [c][x'][Zp][y]   (split, y rows)
//   y fwd:                                  -> [c][x'][Yp][z]   (split, z rows)
//   z fwd + symbol + z inv (one pass):      -> [c][z][Xp][y']   (split, y rows)
//   y inv:                                  -> [c][z][y][x']    (split, x rows)
//   x inv:                                  -> fp32 [c][z][y][x], or the update of v
// The buffers alternate between work and out (in may alias out).  A plain fp32 input is first
// split into work; without the update the result then lands in work and is copied to out.
// Each pass runs over whole groups of 8 lines in its output rows (Yp, Zp, Yp and Xp lines a row), so
// that its 8-line output pieces start 16-byte aligned and stay within a row at any grid size.  The
// lines past an axis's end are written by no pass and read whatever the buffer holds; the rows of
// a product are independent, and their results land in the pitch padding of the next field, which
// its pass does not read (the TMA maps end at the line length).
static cudaError_t apply_K_ks(const KPlan& kp, int split, const float* in, float* out,
                              float* work, int ncomp, cudaStream_t s, const Hook& hook,
                              void* v_upd, float eps, bool in_split, int upd_kind = KS_OUT_UPD) {
  const long long X = kp.nx, Y = kp.ny, Z = kp.nz, C = ncomp;
  const long long Xp = ks_pitch(kp.nx), Yp = ks_pitch(kp.ny), Zp = ks_pitch(kp.nz);
  cudaError_t e;
  float* bA = work;   // receives the x forward product
  float* bB = out;
  const void* src = in;
  if (!in_split) {
    const KsOut o0{KS_OUT_SPLIT, work, C * Z * Yp * Xp, Y, 1, Yp, Xp, 1};
    if ((e = ks_split_rows(in, C * Z * Y, kp.nx, split, o0, s)) != cudaSuccess) return e;
    src = work;
    bA = out;
    bB = work;
  }
  struct Pass2 {
    int kid, axis;
    bool inv, zz;
    long long nlines;
    KsOut o;
  };
  const Pass2 ps[4] = {
      {KID_KX_FWD, 0, false, false, C * Z * Yp, {KS_OUT_SPLIT, bA, C * X * Zp * Yp, Z, Yp, X * Zp, Yp, Zp * Yp}},
      {KID_KY_FWD, 1, false, false, C * X * Zp, {KS_OUT_SPLIT, bB, C * X * Yp * Zp, 1, Zp, Yp, Zp, Zp}},
      {KID_KZ_FUSED, 2, true, true, C * X * Yp, {KS_OUT_SPLIT, bA, C * Z * Xp * Yp, X, Yp, Z * Xp, Yp, Xp * Yp}},
      {KID_KY_INV, 1, true, false, C * Z * Xp, {KS_OUT_SPLIT, bB, C * Z * Y * Xp, 1, Xp, Y, Xp, Xp}}};
  for (const Pass2& p : ps) {
    hook(p.kid, 0);
    e = ks_axis_pass(kp, p.axis, p.inv, split, src, p.nlines, p.o, 0.f, s, p.zz);
    hook(p.kid, 1);
    if (e != cudaSuccess) return e;
    src = p.o.out;
  }
  // x inverse: from the last output into v_upd (update) or fp32 rows in the other buffer
  void* dst = v_upd ? v_upd : (void*)bA;
  const KsOut o5{v_upd ? upd_kind : KS_OUT_F32, dst, 0, 1, 1, 1, X, 1};
  hook(KID_KX_INV, 0);
  e = ks_axis_pass(kp, 0, true, split, src, C * Z * Y, o5, eps, s);
  hook(KID_KX_INV, 1);
  if (e != cudaSuccess) return e;
  if (!v_upd && dst != out)
    e = cudaMemcpyAsync(out, dst, (size_t)C * X * Y * Z * sizeof(float), cudaMemcpyDeviceToDevice, s);
  return e;
}

cudaError_t apply_K_update_bf16(const KPlan& kp, int mode, const float* in, float* work,
                                cudaStream_t s, const Hook& hook, void* v_bf16, float eps,
                                long long cap, bool in_split) {
  if (!ks_path(kp, mode, 3, cap)) return cudaErrorNotSupported;
  return apply_K_ks(kp, mode == LDDMM_K_BF16X3 ? 1 : 0, in, const_cast<float*>(in), work, 3, s,
                    hook, v_bf16, eps, in_split, KS_OUT_UPD_BF16);
}

bool ks_path(const KPlan& kp, int mode, int ncomp, long long cap) {
  if (mode != LDDMM_K_BF16X3 && mode != LDDMM_K_BF16) return false;
  const long long N = (long long)kp.nx * kp.ny * kp.nz;
  if (cap <= 0) cap = (long long)ncomp * N;
  return ks_supported(kp) && cap >= ks_field_floats(kp.nx, kp.ny, kp.nz, ncomp);
}

static cudaError_t apply_K_tc(const KPlan& kp, int split, const float* in, float* out,
                              float* work, int ncomp, cudaStream_t s, const Hook& hook,
                              float* v_upd, float eps, long long cap, bool in_split) {
  if (ks_path(kp, split ? LDDMM_K_BF16X3 : LDDMM_K_BF16, ncomp, cap))
    return apply_K_ks(kp, split, in, out, work, ncomp, s, hook, v_upd, eps, in_split);
  if (in_split) return cudaErrorInvalidValue;
  cudaError_t e;
#define TC_PASS(kid, axis, inv, src, dst, epi)                                         \
  do {                                                                                 \
    hook(kid, 0);                                                                      \
    e = tc_axis_pass(kp, axis, inv, split, src, dst, ncomp, epi, eps, s);              \
    hook(kid, 1);                                                                      \
    if (e != cudaSuccess) return e;                                                    \
  } while (0)
  TC_PASS(KID_KX_FWD, 0, false, in, work, 0);
  TC_PASS(KID_KY_FWD, 1, false, work, out, 0);
  TC_PASS(KID_KZ_SYM, 2, false, out, work, 1);
  TC_PASS(KID_KZ_INV, 2, true, work, out, 0);
  TC_PASS(KID_KY_INV, 1, true, out, work, 0);
  if (v_upd) TC_PASS(KID_KX_INV, 0, true, work, v_upd, 2);
  else TC_PASS(KID_KX_INV, 0, true, work, out, 0);
#undef TC_PASS
  return cudaSuccess;
}

cudaError_t apply_K(const KPlan& kp, int mode, const float* in, float* out, float* work,
                    int ncomp, cudaStream_t s, const Hook& hook, float* v_upd, float eps,
                    long long cap, bool in_split) {
  switch (mode) {
    case LDDMM_K_FP32: {
      if (in_split) return cudaErrorInvalidValue;
      return apply_K_fp32(kp, in, out, work, ncomp, s, hook, v_upd, eps);
    }
    case LDDMM_K_BF16X3:
      return apply_K_tc(kp, 1, in, out, work, ncomp, s, hook, v_upd, eps, cap, in_split);
    case LDDMM_K_BF16:
      return apply_K_tc(kp, 0, in, out, work, ncomp, s, hook, v_upd, eps, cap, in_split);
    default:
      return cudaErrorNotSupported;
  }
}

}  // namespace lddmm
