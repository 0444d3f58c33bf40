// Host-side launch wrappers shared by the translation units of the library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "firls_common.cuh"

namespace firls {

// Launch, if chained with a programmatic dependency on the kernel before it in the
// stream: the CTAs are set up while that one drains and wait in chained_start, which
// every kernel launched so calls first, in every thread.  For the short kernels
// of a macro step on little data (chains() in firls_api.cu has the figures).
template <typename... P, typename... A>
inline void launch_chained(bool chained, void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                           A... args) {
  if (!chained) {
    k<<<grid, block, smem, s>>>(static_cast<P>(args)...);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);  // a failure stays with cudaGetLastError
}

struct FftArgs {
  int batch = 0;
  cudaStream_t stream = 0;
  const float2* tw = nullptr;     // twiddles exp(-2 pi i j / n), j < n
  const SliceState* st = nullptr;
  double* part = nullptr;
  const float2* z = nullptr;
  float2* d = nullptr;
  float2* t = nullptr;
  const float2* b = nullptr;
  const uint8_t* mask = nullptr;
  float2* atb = nullptr;
  float2* x = nullptr;
  const float2* u = nullptr;
  const float* wtv = nullptr;
  const float* wtv2 = nullptr;  // l1 TV: the vertical weights W2 (wtv then holds W1)
  float2* q = nullptr;
  const float2* xs = nullptr;   // row FFT, per-slice mode: x^k of slices starting an outer step
  // row FFT: z, row IFFT: q in the ILU's skewed layout (k_ilu.cu); q of a
  // slice starting an outer step is then its first residual atb - S x^k
  int skew = 0;
  float2* dx = nullptr;         // row FFT: dx += alpha d of the PCG step before
  int mode = 0;
  int real = 0;
  bool chained = false;  // column mask and row IFFT: launch_chained
};

bool fft_size_supported(int n);
int fft_row_ctas(int n);
int fft_col_ctas(int n);
void fft_row_fwd(int n, const FftArgs& a);
void fft_row_ahb(int n, const FftArgs& a);
void fft_col_mask(int n, const FftArgs& a);
void fft_col_inv(int n, const FftArgs& a);
void fft_row_inv(int n, const FftArgs& a);
// partial ||R F x - b||^2 (t = rowFFT(x), a.b, a.mask) into slot a.mode
void fft_col_resid(int n, const FftArgs& a);
// t = colIFFT((1 - R) colFFT(t) + R n b)  (data consistency, column part)
void fft_col_dc(int n, const FftArgs& a);
void fft_prepare(int n);  // set shared-memory limits (call outside capture)

// ---- wavelet (lifting) ----
enum WavMode { WAV_RAW = 0, WAV_MUL_W = 1, WAV_MUL_PINV = 2, WAV_SINGLETON_W = 3 };

struct WavArgs {
  int batch = 0, n = 0, levels = 0, kind = 0;
  cudaStream_t stream = 0;
  const SliceState* st = nullptr;   // slices not running are skipped (may be null)
  float2* tmpA = nullptr;           // [batch][n/2 * n/2] ping-pong LL buffers
  float2* tmpB = nullptr;
  double* part = nullptr;
  int rb = 0;          // rows per CTA of the tiled levels (0: default 8)
  int coarse_max = 0;  // largest side kept in shared memory (0: default 64)
  bool chained = false;  // the one-launch form: launch_chained
  // the one-launch form with r, where wavelet_updates: the residual update on the
  // way in (axpy_step's work with these arguments; ||r||^2 partials, one per CTA, in
  // SLOT_RR)
  const float2* upd_q = nullptr;
  const float2* upd_atb = nullptr;
  int upd_mode = 0;
};
// c = Phi x (Mallat, stride n) with the final store scaled per `mode`:
// RAW: c; MUL_W: w*c; MUL_PINV: c / (abar + lam w); SINGLETON_W: writes
// w = (|c|^2 + eps)^-1/2 into `w` instead of c.
void wavelet_forward(const WavArgs& a, const float2* x, float2* c, float* w, int mode);
// x = Phi^T c; if r != null also partial Re<r, x> into SLOT_RZ.
void wavelet_inverse(const WavArgs& a, const float2* c, float2* x, const float2* r, int real);
// u = Phi^T (s o Phi x), s = w (MUL_W) or 1/(abar + lam w) (MUL_PINV).
// Where a slice fits the shared memory of one thread-block cluster (rb 0, 1
// or 2; above 256^2 only rb 0) every level runs in one launch and c is not
// touched; otherwise
// (rb 4, 8, 16, or no fit) the fine levels are tiled, a launch per level,
// their scaled details going through c, and the levels that fit one CTA's
// shared memory are fused.  Optional partial Re<r, u>.
void wavelet_apply(const WavArgs& a, const float2* x, float2* c, float* w, int mode, float2* u,
                   const float2* r, int real);
int wavelet_cluster_ctas(int n, int levels, int kind, int rb);
bool wavelet_updates(int n, int levels, int kind, int rb);
int wavelet_apply_ctas(int n, int levels, int kind, int rb, int coarse_max);
int wavelet_apply_launches(int n, int levels, int kind, int rb, int coarse_max);
void wav_prepare();

// ---- TV, preconditioner, groups, PCG scalars ----
// wtv2 null: isotropic TV weights into wtv; else l1 TV: W1 into wtv, W2 into wtv2.
// channels C > 1: joint TV weights of each image of C consecutive slices
// (isotropic only), the same W into every contrast.
void tv_weights(int batch, int n, cudaStream_t s, const SliceState* st, const float2* x, float* wtv, float* wtv2,
                int channels = 1);
// Joint wavelet-sparsity weights from the raw coefficients cw of every slice:
// ww = (sum over the C contrasts of |c_j|^2 + eps)^(-1/2) for every contrast.
void joint_wavelet_weights(int batch, int n, int channels, cudaStream_t s, const SliceState* st, const float2* cw,
                           float* ww);
void wavelet_diag(int batch, int n, int levels, int kind, cudaStream_t s, const SliceState* st, const float* w,
                  float* out, const float* sqtab, const int* sqlen);
void penta_setup(int batch, int n, cudaStream_t s, const SliceState* st, const float* wtv, const float* wtv2,
                 const float* wdiag, float* ia);
// ---- the TV preconditioner's sweeps (k_ilu.cu), on arrays in a skewed layout ----
size_t ilu_slice_elems(int n);  // float2 per slice of a skewed array
bool ilu_prepare();
// 1/a of P in ia, wa = (lam W, 1/a) skewed, and for l1 TV w2s = lam W2 skewed, of the
// slices st shows running; before a sweep with new weights
void penta_pack(int batch, int n, cudaStream_t s, const SliceState* st, const float* wtv, const float* wtv2,
                const float* wdiag, float* ia, float4* wa, float2* w2s);
// wa and w2s of every slice from an ia that is there already
void ilu_pack(int batch, int n, cudaStream_t s, const SliceState* st, const float* wtv, const float* wtv2,
              const float* ia, float4* wa, float2* w2s);
// 1/a -> 1/d, the ILU(0) pivots (updated pivots, zero fill), in wa and ia
void ilu0_pivots(int batch, int n, cudaStream_t s, SliceState* st, const SliceState* view, float4* wa,
                 const float2* w2s, float* ia);
// a complex array between the natural layout (stride n n) and the skewed one
void ilu_skew(int batch, int n, cudaStream_t s, bool to_skewed, const float2* src, float2* dst);

// The outer step's update dx = sum_j alpha_j d_j is kept one step behind: the
// row FFT, which reads d anyway, adds alpha d of the step before, and
// outer_apply the last one.
enum IluMode { ILU_INIT = 0, ILU_STEP = 1, ILU_PER_SLICE = -1 };
// all arrays skewed.  INIT: r = q (the first residual); STEP: r -= alpha q.
// w2s null: isotropic TV.
// shape: the sweeps' chunks (0: ilu_default_shape)
// fuse_scalars: the CTA finishes the PCG scalars itself from its sums (rho
// at ILU_INIT; rr, the residual test against pcg_tol, beta and rho at ILU_STEP)
// alpha_np > 0 (ILU_PER_SLICE): the CTA of a slice in PCG first forms alpha
// from the S apply's alpha_np partial sums of <d, S d> (pcg_alpha's work)
void ilu_step(int batch, int n, cudaStream_t s, SliceState* st, double* part, int mode, float2* r, const float2* q,
              float2* y, float2* z, const float4* wa, const float2* w2s, int shape, int fuse_scalars = 0,
              PcgSched ps = PcgSched{0.f, 0, 1 << 30, 0, 0}, int wait_test = 0, int alpha_np = 0,
              bool chained = false);
int ilu_default_shape(int n, int batch);
bool ilu_shape_fits(int n, int shape, bool aniso = false);

// AXPY_PER_SLICE (and ILU_PER_SLICE, SCALARS_PER_SLICE, mode < 0 of the row
// FFT): each slice's own phase picks the first residual (PH_BOUNDARY) or a
// PCG step (PH_PCG).
enum AxpyMode { AXPY_INIT = 0, AXPY_STEP = 1, AXPY_PER_SLICE = -1 };
// Residual update (INIT: r = A^H b - q; STEP: r -= alpha q) with a diagonal preconditioner z = sdiag o r (sdiag null: z = r), partial
// Re<r, z> into SLOT_RZ and ||r||^2 into SLOT_RR (axpy_ctas parts).
void axpy_diag_step(int batch, int n, cudaStream_t s, const SliceState* st, double* part, int mode, float2* r,
                    const float2* q, const float2* atb, const float* sdiag, float2* z, bool chained = false);
// Jacobi scale of a wavelet-only system: ia = 1 / (abar + lam diag(Phi^T W Phi)).
void jacobi_wavelet_setup(int batch, int n, cudaStream_t s, const SliceState* st, const float* wdiag, float* ia);
void axpy_step(int batch, int n, cudaStream_t s, const SliceState* st, double* part, int mode, float2* r,
               const float2* q, const float2* atb, bool chained = false);
int axpy_ctas(int n);

void group_norms(int batch, int n, int n_groups, cudaStream_t s, const SliceState* st,
                 const int* gidx, const int* goff, int gsize, const float2* c, float* wg, float eps_unused);
void group_gather(int batch, int n, int n_groups, cudaStream_t s, const SliceState* st,
                  const int* inv_off, const int* inv_ids, const float* wg, float* w);
// Build the inverse map; returns via err (device int) 1 on bad index/offsets.
void group_inverse_build(int n, int n_groups, int gsize, cudaStream_t s, const int* gidx, const int* goff,
                         int* counts, int* inv_off, int* inv_ids, int* cursor, int* err);

void mask_popcount(int batch, int n, cudaStream_t s, const uint8_t* mask, int* counts);

// Partial sums of the regularisers of F_eps (one slot each, axpy_ctas parts):
// sum_j sqrt(|c_j|^2 + eps) (singleton groups) or sum_g sqrt(||c_g||^2 + eps),
// and sum_i sqrt(|D1 x|_i^2 + |D2 x|_i^2 + eps).  channels C > 1: the joint
// sums of each image in its first slice (the other slices' parts are 0).
void l21_sum(int batch, int n, cudaStream_t s, const float2* c, const int* gidx, const int* goff, int n_groups,
             int gsize, float eps, double* part, int slot, int channels = 1);
void tv_sum(int batch, int n, cudaStream_t s, const float2* x, float eps, double* part, int slot, int aniso,
            int channels = 1);
// f[s] = F_eps of slice s from the partial sums of its terms (nd and nr of them)
void objective_sum(int batch, cudaStream_t s, const double* part, int nd, int nr, bool wavelet, bool tv,
                   const float* lam, const float* lam_tv, double* f, int channels);
// whether a slice keeps the warm start x1 of objective f1, f0 that of A^H b
__host__ __device__ inline bool guard_keeps(double f1, double f0) { return f1 - f1 == 0.0 && f1 <= f0; }
// x0 = x1 or A^H b per slice; x1 and x0 16-byte aligned
void guard_pick(int batch, int n, cudaStream_t s, const double* f1, const double* f0, const void* x1,
                const float2* atb, void* x0);

// PCG scalar updates (a warp per slice).  channels C > 1: the inner
// products are summed over the C consecutive slices of a multi-contrast
// image, whose slices then carry the same scalars (here, in outer_end and in
// state_init's ||A^H b||^2).
void pcg_alpha(int batch, cudaStream_t s, SliceState* st, const double* part, int nparts, int channels = 1,
               bool chained = false);
enum ScalarsMode { SCALARS_INIT = 0, SCALARS_STEP = 1, SCALARS_PER_SLICE = -1 };
void pcg_scalars(int batch, cudaStream_t s, SliceState* st, const double* part, int nparts_rz, int nparts_rr,
                 int mode, const PcgSched& ps, int channels = 1, bool chained = false, const float2* r = nullptr,
                 int n = 0);
// view = st with every slice not at the start of its outer step marked done
// (and the slices whose outer step is due move to PH_START)
void boundary_view(int batch, cudaStream_t s, SliceState* st, SliceState* view);
// x += dx + alpha d (the outer step's accumulated update and its last step)
// with partial norms squared of that update and of x before it, for the
// relative change; dx cleared.
void outer_apply(int batch, int n, cudaStream_t s, const SliceState* st, float2* x, float2* dx, const float2* d,
                 double* part);
// plateau_after: first outer step at which kind 1 also stops on a plateau
void outer_end(int batch, cudaStream_t s, SliceState* st, const double* part, int nparts,
               float outer_tol, int tol_kind, float stall_tol, int plateau_after, int channels = 1);
// phase: PH_BOUNDARY for a solve (its first outer step is due), PH_START for
// the single operator applications (no outer step)
void state_init(int batch, cudaStream_t s, SliceState* st, const double* part, int nparts_rhs,
                const int* counts, int n, const float* lam, const float* lam_tv, float eps, int outer_max,
                int phase, int channels = 1);

}  // namespace firls
