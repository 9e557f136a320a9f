// launch.h -- size-dispatching launchers for the kernels in kernels.cuh.
// Every launcher picks the template instance for its transform length and
// returns the launch status (cudaGetLastError after the launch).
#pragma once

#include <cuda_runtime.h>

namespace pce {

struct Box;
struct SepTerms;
struct SecGeom;

// Columns of a CTA of the block column kernels, and such CTAs resident on an SM (at most 4).
int cols_columns_per_cta(int ny);
int cols_ctas_per_sm(int ny);
// Rows handled per CTA of the row kernels (two rows per FFT).
int rows_pairs_per_cta(int nx);
// Row pairs per CTA of the window-gradient row kernel.
int rows_grad_pairs_per_cta(int nx);
// Items (row pairs) handled per CTA of the R2C row kernel.
int rows_r2c_items_per_cta(int nx);
// Raise the dynamic shared-memory limit of every kernel that needs it (once per device).
cudaError_t prepare_kernels();

// Storage-precision arguments: `lowp` selects bfloat16 windows (wbox) and
// half2 spectra scaled by hscale[k]; otherwise float windows and float2 spectra.
cudaError_t launch_rows_r2c(int nx, bool window, dim3 grid, cudaStream_t s,
                            const float* src, long long src_bstride, int nrows,
                            const void* wbox, bool lowp, const Box* box, const int2* items, int nitems,
                            float2* dst, long long dst_bstride, long long dst_kstride,
                            const float2* tw, const float2* tw1024);

// F1 by row pairs (k_rows_r2c_pairs): the same output as launch_rows_r2c with a
// window, the terms (or slots) of each row pair from the CSR lists kptr/klist.
cudaError_t launch_rows_r2c_pairs(int nx, int nb, cudaStream_t s, const float* src, long long src_bstride,
                                  int nrows, const void* wbox, bool lowp, const Box* box, const int* kptr,
                                  const int* klist, float2* dst, long long dst_bstride, long long dst_kstride,
                                  const float2* tw);

cudaError_t launch_rows_c2r(int nx, dim3 grid, cudaStream_t s, const float2* src,
                            long long src_bstride, int nrows, float* dst, long long dst_bstride,
                            float scale, const float2* tw, const float2* tw1024);

cudaError_t launch_rows_adj(int nx, dim3 grid, cudaStream_t s, const float2* Q, long long q_bstride,
                            long long q_kstride, int nrows, const void* wbox, bool lowp, const Box* box,
                            const int* kptr, const int* klist, float* dst, long long dst_bstride,
                            float scale, const float2* tw, const float2* tw1024, int rv = 0, int kmin = 0,
                            int kmax = 1 << 30, int accumulate = 0);

// One-warp plain row transforms for Nx = 1024 or 512 (wrows.cuh): the same results
// and layouts as launch_rows_r2c without a window (row pairs of every row) and
// launch_rows_c2r; one warp per row pair, grids derived from nrows.
cudaError_t launch_wrows_r2c(int nx, int nb, cudaStream_t s, const float* src, long long src_bstride, int nrows,
                             float2* dst, long long dst_bstride, const float2* tw1024);
cudaError_t launch_wrows_c2r(int nx, int nb, cudaStream_t s, const float2* src, long long src_bstride, int nrows, float* dst,
                             long long dst_bstride, float scale, const float2* tw1024);

// What the column passes of a plan (not its separable fast path) read: nb right-hand
// sides of a launch, the spectra in both layouts (hh [m][ny][nxh], hhT per column; the
// Nyquist column hN, hN2 split by parity for ny = 2048; half2 with hscale when lowp),
// twiddles, the plan's status word.  warp: the one-warp column kernels where they
// exist (ny = 512, 1024, 2048), else block Stockham.  frame_rows: col_frame_rows(), tab
// the phased twiddles.  split: CTAs that share a column tile's terms (forward:
// cols_fwd_split()).
struct ColArgs {
    int ny = 0, nxh = 0, nb = 1, m = 0;
    unsigned split = 1;
    bool lowp = false, warp = true;
    const void *hh = nullptr, *hN = nullptr, *hhT = nullptr, *hN2 = nullptr;
    const float* hscale = nullptr;
    const Box* box = nullptr;   // device
    int frame_rows = 0;
    const float2 *tw = nullptr, *tw1024 = nullptr, *tab = nullptr, *tw2048l = nullptr;
    int* status = nullptr;
    long long wait_limit = 0;
    int skip_copy = 0;
};
// Frame rows the windows need in the column kernels of ny = 512, 1024 or 2048 rows
// (ckernels.cuh; at most 512 or 1024), 0 where those kernels do not serve them.
// box: host.
int col_frame_rows(int ny, const Box* box, int m);
// float2 of the phased twiddle tables of ny rows, both directions (0: none).
long long col_table_size(int ny);

cudaError_t launch_cols_fwd(const ColArgs& c, cudaStream_t s, const float2* Z, long long z_bstride,
                            long long z_kstride, float2* A, long long a_bstride);
cudaError_t launch_cols_adj(const ColArgs& c, cudaStream_t s, const float2* V, long long v_bstride, float2* Q,
                            long long q_bstride, long long q_kstride);
// The forward over clusters of CTAs (colsplit.cu): dense plans cols_fwd_split() (c.split; 8, 4
// or none) for a grid of ctas column CTAs, separable ones with tensor-memory columns kSepSplit
// (grid.z).
constexpr int kSepSplit = 4;
int cols_fwd_split(int ny, int m, long long ctas);
cudaError_t launch_cols_fwd_split(const ColArgs& c, cudaStream_t s, const float2* Z, long long z_bstride,
                                  long long z_kstride, float2* A, long long a_bstride);
cudaError_t launch_cols_fwd_sep_split(int ny, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                                      long long z_kstride, const float2* hhT, const float2* hN, const Box* box, int nxh,
                                      float2* A, long long a_bstride, const float2* tw1024, const SepTerms& sep);
// every row of Q (the window gradient); FP32 storage
cudaError_t launch_cols_adj_full(const ColArgs& c, cudaStream_t s, const float2* V, long long v_bstride, float2* Q,
                                 long long q_bstride, long long q_kstride);

cudaError_t launch_cols_spec(int ny, dim3 grid, cudaStream_t s, const float2* S, int nxh,
                             float2* hh, float2* hN, const float2* tw);

cudaError_t launch_plain_cols_inv(int ny, dim3 grid, cudaStream_t s, const float2* acc,
                                  const float2* accN, int nxh, float2* A, const float2* tw);

// Sectioned apply (section.cuh)
int sec_rows_per_cta(int lc);
cudaError_t prepare_sec();
// wbox: float or bfloat16 (lowp) box copies; hsT / hsN: float2 or half2 (lowp)
// section spectra with per-term scales hscale (lowp only).
cudaError_t launch_sec_r2c(int lc, bool win, dim3 grid, cudaStream_t s, const float* src, long long src_bstride,
                           int nyg, int nxg, const void* wbox, bool lowp, const SecGeom* geo, const int2* items,
                           int nitems, float2* dst, long long dst_bstride, long long dst_kstride, const float2* tw);
cudaError_t launch_sec_cols(bool conj, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                            long long z_kstride, int nb, const void* hsT, const void* hsN, const float* hscale,
                            bool lowp, const SecGeom* geo, int nxh, float2* A, long long a_bstride,
                            long long a_kstride, const float2* tw1024, int* status, long long wait_limit,
                            int skip_copy);
cudaError_t launch_sec_c2r(int lc, bool win, dim3 grid, cudaStream_t s, const float2* src, long long src_bstride,
                           long long src_kstride, const SecGeom* geo, const int2* items, int nitems,
                           const void* wbox, bool lowp, float* dst, long long dst_bstride, int nyg, int nxg,
                           float scale, const float2* tw);

// Separable windows, Ny = 1024 or 512 (one-warp column kernels): Z / Q hold
// one slot per column factor, box[] is indexed by slot.
cudaError_t launch_cols_fwd_sep(int ny, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                                long long z_kstride, const float2* hhT, const float2* hN,
                                const Box* box, int nxh, float2* A, long long a_bstride,
                                const float2* tw1024, int* status, long long wait_limit, int skip_copy,
                                const SepTerms& sep);
cudaError_t launch_cols_adj_sep(int ny, dim3 grid, cudaStream_t s, const float2* V, long long v_bstride,
                                const float2* hhT, const float2* hN, const Box* box, int nxh,
                                float2* Q, long long q_bstride, long long q_kstride,
                                const float2* tw1024, int* status, long long wait_limit, int skip_copy,
                                const SepTerms& sep);

// The same with the per-warp state in tensor memory (tkernels.cuh), Ny = 1024 or
// 512.  With sep.kq0 set (Ny = 1024 only), the pruned kernels run and hhT / hN
// must be the rotated spectra hhat_k[f] W1024^{32 f kq0[k]}.
cudaError_t launch_cols_fwd_sep_tm(int ny, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                                   long long z_kstride, const float2* hhT, const float2* hN, const Box* box,
                                   int nxh, float2* A, long long a_bstride, const float2* tw1024, int* status,
                                   long long wait_limit, int skip_copy, const SepTerms& sep);
cudaError_t launch_cols_adj_sep_tm(int ny, dim3 grid, cudaStream_t s, float2* V, long long v_bstride,
                                   const float2* hhT, const float2* hN, const Box* box, int nxh, float2* Q,
                                   long long q_bstride, long long q_kstride, const float2* tw1024, int* status,
                                   long long wait_limit, int skip_copy, const SepTerms& sep);

cudaError_t launch_cols_grad_h(int ny, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                               long long z_kstride, int nb, const float2* Rh, const float2* RhN,
                               const Box* box, int nxh, float2* dhh, float scale, int accumulate,
                               const float2* tw);

cudaError_t launch_rows_grad_w(int nx, dim3 grid, cudaStream_t s, const float2* Qf, long long q_bstride,
                               long long q_kstride, int nrows, int nb, const float* u,
                               long long u_bstride, float* dw, float scale, int accumulate,
                               const float2* tw);

cudaError_t launch_grad_1d(int n, int m, cudaStream_t s, const float* u, const float* r,
                           const float* w, const float2* hp, int nb, float2* dh, float* dw,
                           float scale, int accumulate, const float2* tw);

// 1D apply (adjoint or forward), N <= 8192.  tw1024 (may be NULL): the four-step
// table of the one-warp 1024-point FFT; with it, N = 1024 and fewer than 304
// right-hand sides run the one-warp kernels
cudaError_t launch_1d(bool adjoint, int n, int batch, cudaStream_t s, const float* in, const void* w, const void* hp,
                      const float* hscale, bool lowp, int m, float* out, float scale, const float2* tw,
                      const float2* tw1024);

cudaError_t launch_spec_1d(int n, int m, cudaStream_t s, const float* h, float2* hp,
                           const float2* tw);

// 1D transforms of N = ny * nx > 8192 points (four-step, k1d_large.cuh).
int l1_cols_per_cta(int ny);
int l1_row_items(int nx);
cudaError_t launch_l1_cols(int ny, int mode, dim3 grid, cudaStream_t s, const float* src,
                           long long src_bstride, const float* w, int m, int nx, const float2* twN,
                           float2* G, const float2* tw);
cudaError_t launch_l1_rows_fwd(int nx, int nb, cudaStream_t s, const float2* G, int npairs,
                               const float2* hh4, int m, int ny, const float2* twN, float2* A,
                               const float2* tw);
cudaError_t launch_l1_cols_inv(int ny, dim3 grid, cudaStream_t s, const float2* A, int nx, float* y,
                               float scale, const float2* tw);
// alone: no other apply runs beside this one (the pairs may be split over CTAs)
cudaError_t launch_l1_rows_adj(int nx, int nb, bool alone, cudaStream_t s, const float2* V, int npairs,
                               const float2* hh4, int m, int ny, const float2* twN, float2* Q,
                               const float2* tw);
cudaError_t launch_l1_cols_adj(int ny, dim3 grid, cudaStream_t s, const float2* Q, int npairs,
                               const float* w, int m, int nx, float* x, float scale, const float2* tw);
cudaError_t launch_l1_rows_spec(int nx, dim3 grid, cudaStream_t s, const float2* G, int npairs, int m,
                                int ny, float2* hh4, const float2* tw);

}  // namespace pce
