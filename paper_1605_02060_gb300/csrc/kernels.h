// Host-side launch wrappers for the liblddmm kernels (one translation unit per kernel family).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "per_device.h"

namespace lddmm {

// Raises a kernel's dynamic shared memory limit to `bytes`, once on each device; `set` is the
// kernel's own record.  The limit is the most the kernel is ever launched with, not one launch's
// need: a lower value would undo what an earlier launch (a recorded graph node) counts on.
template <typename Kernel>
cudaError_t raise_smem_limit(PerDevice<bool>& set, Kernel* kernel, int bytes) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  set.get(dev, [&] {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e == cudaSuccess;
  });
  return e;
}

// SMs of the current device.
inline int sm_count() {
  static PerDevice<int> kept;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
  const int n = kept.get(dev, [&] {
    int m = 0;
    return cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? m : 0;
  });
  return n > 0 ? n : 148;
}

// Accumulators written by the reduction kernels (device memory, reset per iteration).
struct Acc {
  double e_reg;       // sum_j sum_x |(gamma - alpha Lap_h) v_j|^2   (unscaled)
  double e_data;      // sum_x M (J0_T - I1)^2                       (unscaled)
  int min_det_ord;    // ordered-int encoding of min det D phi_{j,1}
  int nonfinite;      // set when a reduction saw NaN/Inf
};

// Optional timing hook: mark(user, kernel_id, 0) before and mark(user, kernel_id, 1) after
// every kernel launch (the host records CUDA events on the launching stream).
struct Hook {
  void (*mark)(void* user, int kernel_id, int phase) = nullptr;
  void* user = nullptr;
  void operator()(int id, int phase) const {
    if (mark) mark(user, id, phase);
  }
};

enum KernelId {
  KID_BACK_DISP = 0, KID_BACK_TERMS, KID_FWD_TERMS, KID_FWD_FLOW, KID_KX_FWD, KID_KY_FWD,
  KID_KZ_SYM, KID_KZ_INV, KID_KY_INV, KID_KX_INV, KID_UPDATE, KID_EREG, KID_KZ_FUSED,
  KID_FWD_FUSED, KID_J0_EDATA, KID_BACK_FUSED, KID_COUNT
};

// ---- flows (kernels_flow.cu) ----
// Velocity fields and images (vj, I0, I1, M) are stored as float (st = 0) or bf16 (st = 1);
// displacements, J1, W, b and all arithmetic are float.  Maps (displacements) are planar,
// [3][N], or, with quad = 1, [N] x (u_x, u_y, u_z, 0) (16 bytes a voxel): the iteration's
// backward sweep (launch_flow_back), the map phi_{0,1} it leaves and the steps of a forward sweep
// without the residual use the quad layout, the iteration's forward sweep (launch_fwd_fused) and
// phi_{1,0} the planar one.
// Backward sweep step j (quad maps): u_cur = dt v_j / h + u_next(x + dt v_j / h) (u_next ==
// nullptr: id) and, unless u_next is null, the terms of u_next = phi_{j+1,1} - id: J1 = I1 o phi,
// W = (M o phi) det(I + Du_next), min det into acc.  launch_back_last: the terms of
// u = phi_{0,1} - id.  IM holds I1 and M interleaved as pairs (launch_interleave).
void launch_flow_back(const Grid& g, const void* vj, const float* u_next, float* u_cur,
                      const void* IM, float* J1, float* W, float dtx, float dty, float dtz,
                      Acc* acc, cudaStream_t s, const Hook& hook, int st, int rk = 0);
void launch_back_last(const Grid& g, const float* u, const void* IM, float* J1, float* W, Acc* acc,
                      cudaStream_t s, const Hook& hook, int st);
// out[i] = (a[i], b[i]) as storage-type pairs.
void launch_interleave(const void* a, const void* b, void* out, int64_t n, cudaStream_t s,
                       int st);
// Forward sweep step j: u_next = -dt v_j / h + u_cur(x - dt v_j / h) (u_cur == nullptr: id);
// if last, J0_T = I0 o (id + u_next) and E_data.  quad: u_cur and u_next in the quad layout, but
// the last u_next planar; else all planar, for float fields and one lookup a step only.
void launch_fwd_flow(const Grid& g, const void* vj, const float* u_cur, float* u_next,
                     float dtx, float dty, float dtz, bool last, const void* I0, const void* I1,
                     const void* M, float* J0T, Acc* acc, cudaStream_t s, int st, int rk = 0,
                     int quad = 0);
// Forward sweep step j (planar maps) in one pass over u_cur = phi_{j,0} - id (nullptr: id): the
// residual b = c W_j (J0_j - J1_j) grad J0_j / h with J0_j = I0 o (id + u_cur) (bsplit 0: b as 3
// fp32 fields; 1 / 2: b split for the pre-split K, bf16 hi plane / hi and lo planes, rows of pitch
// px), and u_next as launch_fwd_flow (without J0_T and E_data: launch_j0_edata gives them).
void launch_fwd_fused(const Grid& g, const void* vj, const float* u_cur, float* u_next,
                      float dtx, float dty, float dtz, const void* I0, const float* J1j,
                      const float* Wj, float* b, float c, float ihx, float ihy, float ihz,
                      int bsplit, int px, int py, cudaStream_t s, int st, int rk = 0);
// J0_T = I0 o (id + u) and E_data = sum M (J0_T - I1)^2 into acc, from the planar map u = u_T.
void launch_j0_edata(const Grid& g, const float* u, const void* I0, const void* I1,
                     const void* M, float* J0T, Acc* acc, cudaStream_t s, int st);
// E_reg of all T fields v[T][3][N] into acc->e_reg (unscaled sum of |(gamma - alpha Lap_h) v|^2).
void launch_ereg(const Grid& g, const void* v, int T, float alpha, float gamma, float ihx2,
                 float ihy2, float ihz2, Acc* acc, cudaStream_t s, int st);
// v_j <- v_j - eps (2 v_j - Kb), 3 components.
void launch_update(const Grid& g, void* vj, const float* Kb, float eps, cudaStream_t s, int st);
// Displacement of phi_{1,0} (planar) / phi_{0,1} (quad) only: flows without the residual, to
// recompute or refresh maps.  rk = 1: RK4 along each step (v_j held over the step) instead of one
// lookup.
void launch_flow_only_fwd(const Grid& g, const float* vj, const float* u_cur, float* u_next,
                          float dtx, float dty, float dtz, cudaStream_t s);
void launch_flow_only_back(const Grid& g, const void* vj, const float* u_next, float* u_cur,
                           float dtx, float dty, float dtz, cudaStream_t s, int st, int rk = 0);
// A map in the quad layout ([N] x (u_x, u_y, u_z, 0), the iteration's sweeps) to the planar one
// ([3][N]).
void launch_quad_to_planar(const float* quad, float* planar, int64_t n, cudaStream_t s);
// dst = src o (id + u), u planar or (quad = 1) in the quad layout; labels by nearest neighbour.
void launch_warp(const Grid& g, const float* src, const float* u, float* dst, cudaStream_t s,
                 int quad = 0);
void launch_labels(const Grid& g, const uint16_t* L0, const float* u, uint16_t* dst,
                   cudaStream_t s);
void launch_downsample(const Grid& fine, const Grid& coarse, int factor, const float* src,
                       void* dst, cudaStream_t s, int st);
void launch_upsample(const Grid& coarse, const Grid& fine, float ratio, const void* src,
                     void* dst, int nfields, cudaStream_t s, int st);
void launch_to_storage(const float* src, void* dst, int64_t n, cudaStream_t s, int st);
// launch_to_storage that also sets *flag when src holds NaN or Inf (both float: a checked copy).
void launch_store_checked(const float* src, void* dst, int64_t n, int* flag, cudaStream_t s,
                          int st);
void launch_from_storage(const void* src, float* dst, int64_t n, cudaStream_t s, int st);
// *flag |= bit when a[0..n) holds a NaN or an infinity.
void launch_check_finite(const float* a, int64_t n, int* flag, cudaStream_t s, int bit = 1);
void launch_fill(float* a, int64_t n, float value, cudaStream_t s);
// hist (kDiceWords, the first kDiceZero of them zeroed): voxels per label of A, of B and of both at
// once, 65536 each, and the mean's scratch; out = mean Dice over the labels > 0 present in either
// (1 when there are none).
constexpr int kDiceBlocks = 64, kDiceZero = 3 * 65536 + 2, kDiceWords = kDiceZero + 2 * kDiceBlocks;
void launch_dice(const uint16_t* A, const uint16_t* B, int64_t n, unsigned long long* hist,
                 double* out, cudaStream_t s);

// ---- registration-quality measures of §2.7 (kernels_metrics.cu) ----
// 8x8x8-voxel cells of a grid.
int64_t surface_cells(const Grid& g);
int64_t surface_select_bytes();
// start[0..cells) and start[cells + 1 ..]: where each cell's surface voxels of mask A, of mask B
// begin; start[cells], start[2 cells + 1]: their numbers.
cudaError_t surface_count(const Grid& g, const uint8_t* A, const uint8_t* B, unsigned* start,
                          cudaStream_t s);
// After surface_count: list (na + nb entries), the directed distances dA (na) and dB (nb), sel
// (surface_select_bytes() of scratch) and out[0] = their maximum, out[1], out[2] = the two middle
// values (equal for an odd number).
cudaError_t surface_distances(const Grid& g, const uint8_t* A, const uint8_t* B, unsigned* start,
                              uint16_t* list, unsigned na, unsigned nb, float hx, float hy,
                              float hz, double* dA, double* dB, void* sel, double* out,
                              cudaStream_t s);
// e[k] = |(x_k + u01(x_k) - y_k) h| for n points (float [n][3], voxel coordinates).
cudaError_t landmark_errors(const Grid& g, const float* u01, const float* xk, const float* yk,
                            int n, float hx, float hy, float hz, double* e, cudaStream_t s);

// ---- preprocessing of §2.2 (kernels_preprocess.cu) ----
// Image-LDDMM histogram matching into out; scratch: match_scratch_bytes(bins), whose first 32
// bytes then hold the two ranges (int 2 and int 6: the masks' voxel counts).  Where a mask is
// empty, out is not written.
size_t match_scratch_bytes(int bins);
cudaError_t histogram_match(const float* I0, const float* M0, const float* I1, const float* M1,
                            int64_t n, int bins, int points, void* scratch, float* out,
                            cudaStream_t s);
// Masks as bits, rows of ceil(nx / 32) words (the bits past nx are 0): I > t; erosion or dilation
// by the ball of radius r <= 16 (beyond the grid is background); back to bytes 0 / 1.
int64_t mask_bits_words(int nx, int ny, int nz);
cudaError_t threshold_bits(const float* I, int nx, int ny, int nz, float t, uint32_t* out,
                           cudaStream_t s);
cudaError_t ball_bits(int nx, int ny, int nz, const uint32_t* in, int r, bool erode, uint32_t* out,
                      cudaStream_t s);
cudaError_t unpack_bits(int nx, int ny, int nz, const uint32_t* in, uint8_t* out, cudaStream_t s);

// ---- geodesic shooting (kernels_shoot.cu) ----
// m = |D phi| (D phi)^T (m0 o phi), phi = id + u (u in voxels), 3 components of N each.
cudaError_t transport_momentum(const Grid& g, const float* m0, const float* u, float hx,
                               float hy, float hz, float* m, cudaStream_t s);

// ---- exact gradient of the discrete energy (kernels_adjoint.cu) ----
void launch_adj_init(const Grid& g, const float* uT, const float* I0, const float* I1,
                     const float* M, float* gT, float scale, cudaStream_t s);
void launch_adj_step(const Grid& g, const float* vj, const float* uj, const float* gnext,
                     float* gcur, float* gradj, float dtx, float dty, float dtz, cudaStream_t s);
void launch_apply_L3(const Grid& g, const float* src, float* dst, float* clear, float alpha,
                     float gamma, float ihx2, float ihy2, float ihz2, float scale, bool accumulate,
                     cudaStream_t s);

// ---- smoothing operator K (kernels_dft.cu) ----
struct KPlan {
  int nx, ny, nz;
  float alpha, gamma;
  // per-axis orthonormal real DFT matrices R (row k = frequency basis vector), row-major
  float* Rx; float* Ry; float* Rz;
  // per-axis discrete-Laplacian eigenvalue of each row, lambda_d(row) / h_d^2 folded in
  float* lx; float* ly; float* lz;
  // tensor-core operand tables per axis (x, y, z) and direction (0 forward, 1 inverse):
  // nk = Npad/16 k-steps, each [hi | lo] bf16 blocks of Npad x 16 in K-major core-matrix order
  uint16_t* tc[3][2];
  // operand tables of the pre-split pass (kernels_ks.cu) per axis and direction: bf16
  // [2][Nc][Kp] (hi plane, lo plane), row n = output column, k contiguous (Nc = Kp =
  // ceil16(n)), zero beyond the axis length
  uint16_t* ks[3][2];
  int* err;  // device flag set by a tensor-core kernel whose bounded wait timed out
  // probes per pipeline wait in the pre-split tensor-core pass (0: the default, 2^22)
  uint32_t poll_limit;
  bool sym_normal;   // symbol_is_normal of the grid (false: nothing is known)
};
// Whether every value of the symbol's square (gamma + alpha lambda)^2 on a grid of this spacing is
// a normal number with a normal reciprocal, so that a product with the reciprocal may take the
// division's place.  lambda lies in [0, 4 (hx^-2 + hy^-2 + hz^-2)]; the bounds leave a factor of 4.
inline bool symbol_is_normal(double hx, double hy, double hz, double alpha, double gamma) {
  const double top = gamma + alpha * 4.0 * (1.0 / (hx * hx) + 1.0 / (hy * hy) + 1.0 / (hz * hz));
  return gamma >= 0x1p-62 && top <= 0x1p62;
}
// Build device tables for one grid (allocates; free with kplan_destroy).
cudaError_t kplan_create(KPlan* kp, int nx, int ny, int nz, float hx, float hy, float hz,
                         float alpha, float gamma);
void kplan_destroy(KPlan* kp);
// out = K in for `ncomp` scalar fields stored back to back (each nx*ny*nz); work needs
// ncomp*N floats.  in and out may alias.  mode: LDDMM_K_*.
// If v_upd != nullptr the result is not stored: instead v_upd <- v_upd - eps (2 v_upd - K in)
// (the gradient-descent update, fused into the last pass on the tensor-core path).
// cap: floats available in out and in work (0: ncomp*N); the tensor-core modes take the
// pre-split path when cap >= ks_field_floats (intermediate fields with padded rows).
cudaError_t apply_K(const KPlan& kp, int mode, const float* in, float* out, float* work,
                    int ncomp, cudaStream_t s, const Hook& hook = Hook(),
                    float* v_upd = nullptr, float eps = 0.f, long long cap = 0,
                    bool in_split = false);
// Output addressing of a pre-split pass: line l = (a D + b) E + e is written at column n to
// element (a F + b) P + e + n G, as bf16 hi/lo planes `plane` elements apart (KS_OUT_SPLIT), as
// fp32 (KS_OUT_F32), or as the update out <- out - eps (2 out - C) of fp32 rows (KS_OUT_UPD) or
// of bf16 rows (KS_OUT_UPD_BF16, arithmetic in FP32, one rounding).
enum { KS_OUT_SPLIT = 0, KS_OUT_F32 = 1, KS_OUT_UPD = 2, KS_OUT_UPD_BF16 = 3 };
struct KsOut {
  int kind;
  void* out;
  long long plane;
  long long D, E, F, P, G;
};
// cuTensorMapEncodeTiled from the driver, as void* (nullptr when unavailable).
void* tma_encode_fn();
// The pre-split path (all six products on k_dft_ks).  Row pitch of a split line (elements),
// the sizes it takes, whether it applies, and the floats a buffer needs for any intermediate field
// of ncomp components.
int ks_pitch(int L);
bool ks_shape(int nx, int ny, int nz);
bool ks_supported(const KPlan& kp);
long long ks_field_floats(int nx, int ny, int nz, int ncomp);
cudaError_t ks_axis_pass(const KPlan& kp, int axis, bool inverse, int split, const void* in,
                         long long nlines, const KsOut& o, float eps, cudaStream_t s,
                         bool zz = false);
// True when apply_K(kp, mode, ..., ncomp, cap) takes the pre-split path; its input may then be
// given already split (in_split): bf16 hi/lo planes [ncomp][nz][ks_pitch(ny)][ks_pitch(nx)].
bool ks_path(const KPlan& kp, int mode, int ncomp, long long cap);
// The pre-split K of `in` (3 components, on the pre-split path only) with the update fused into
// its last product for a velocity stored in bf16: v <- bf16(v - eps (2 v - K in)), the
// arithmetic in FP32.  cudaErrorNotSupported when the pre-split path does not apply.
cudaError_t apply_K_update_bf16(const KPlan& kp, int mode, const float* in, float* work,
                                cudaStream_t s, const Hook& hook, void* v_bf16, float eps,
                                long long cap, bool in_split);
// fp32 rows [nrows][L] -> split field at the addresses `o` gives (line = row, column = n).
cudaError_t ks_split_rows(const float* in, long long nrows, int L, int split, const KsOut& o,
                          cudaStream_t s);
// One tensor-core axis pass (kernels_tc.cu): epi 0 plain, 1 times the K symbol, 2 update.
cudaError_t tc_axis_pass(const KPlan& kp, int axis, bool inverse, int split, const float* in,
                         float* out, int ncomp, int epi, float eps, cudaStream_t s);

}  // namespace lddmm
