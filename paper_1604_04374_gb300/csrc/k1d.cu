// k1d.cu -- instances of the single-CTA 1D kernels for N = 16 .. 8192.
#include "kernels.cuh"
#include "k1d_large.cuh"
#include "wk1d.cuh"
#include "launch.h"

namespace pce {

#define PCE_1D_SIZES(X) X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096) X(8192)

cudaError_t prepare_cols();

#define PCE_L1_SIZES(X) X(128) X(256) X(512)

cudaError_t prepare_l1() {
    cudaError_t e = cudaSuccess;
#define X(N)                                                                                   \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k4_cols<N, kL1Win>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                 ColCfg<N>::SMEM);                                             \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k4_cols<N, kL1Pair>,                                          \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, ColCfg<N>::SMEM); \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k4_cols<N, kL1One>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                 ColCfg<N>::SMEM);                                             \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k4_cols_inv<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                 ColCfg<N>::SMEM);                                             \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k4_cols_adj<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                 ColCfg<N>::SMEM);                                             \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k4_rows_fwd<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                 L1Rows<N>::SMEM);                                             \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k4_rows_adj<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                 L1Rows<N>::SMEM);                                             \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k4_rows_spec<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                 L1Rows<N>::SMEM);
    PCE_L1_SIZES(X)
#undef X
    return e;
}

int l1_cols_per_cta(int ny) { return cols_columns_per_cta(ny); }
int l1_row_items(int nx) {
    switch (nx) {
#define X(N) case N: return L1Rows<N>::ITEMS;
        PCE_L1_SIZES(X)
#undef X
    }
    return 0;
}

cudaError_t launch_l1_cols(int ny, int mode, dim3 grid, cudaStream_t s, const float* src,
                           long long src_bstride, const float* w, int m, int nx, const float2* twN,
                           float2* G, const float2* tw) {
    switch (ny) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        if (mode == kL1Win)                                                                    \
            k4_cols<N, kL1Win><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(src, src_bstride, w, m, \
                                                                           nx, twN, G, tw);   \
        else if (mode == kL1Pair)                                                              \
            k4_cols<N, kL1Pair><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(src, src_bstride, w,  \
                                                                            m, nx, twN, G, tw); \
        else                                                                                   \
            k4_cols<N, kL1One><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(src, src_bstride, w, m, \
                                                                           nx, twN, G, tw);   \
        break;
        PCE_L1_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

namespace {

// The kernels for few right-hand sides: while nb right-hand sides' one-pair CTAs, at most
// 128 registers a thread, fit the GPU at once (N = 65536: up to 9, N = 16384: up to 37;
// forward and adjoint there still 1.1 and 1.4 times as fast).  Not for rows or columns of
// 512: N = 262144, m = 32, one right-hand side, adjoint 111 -> 121 us.
template <int N>
bool l1_few(int ny, int nb) {
    return N <= 256 && ny <= 256 && (long long)(ny / 2 + 1) * nb <= (long long)kSms * (512 / L1Few<N>::NT);
}

template <int N>
void l1_rows_fwd(int nb, cudaStream_t s, const float2* G, int npairs, const float2* hh4, int m, int ny,
                 const float2* twN, float2* A, const float2* tw) {
    constexpr int IT = L1Rows<N>::ITEMS;
    if constexpr (N <= 256) {
        if (l1_few<N>(ny, nb)) {
            k4_rows_fwd_few<N><<<dim3(ny / 2 + 1, nb), L1Few<N>::NT, L1Few<N>::SMEM, s>>>(G, npairs, hh4, m, ny, twN, A,
                                                                                          tw);
            return;
        }
    }
    k4_rows_fwd<N><<<dim3((ny / 2 + IT) / IT, nb), L1Rows<N>::NT, L1Rows<N>::SMEM, s>>>(G, npairs, hh4, m, ny, twN, A,
                                                                                        tw);
}

// alone: the pairs may go to several CTAs
template <int N>
void l1_rows_adj(int nb, bool alone, cudaStream_t s, const float2* V, int npairs, const float2* hh4, int m, int ny,
                 const float2* twN, float2* Q, const float2* tw) {
    constexpr int R = 2 * L1Rows<N>::ITEMS;
    if constexpr (N <= 256) {
        if (l1_few<N>(ny, nb)) {
            int split = 1;
            while (alone && 2 * split <= npairs && l1_few<N>(ny, 2 * split * nb)) split *= 2;
            k4_rows_adj_few<N><<<dim3(ny / 2, nb, split), L1Few<N>::NT, L1Few<N>::SMEM, s>>>(V, npairs, hh4, m, ny, twN,
                                                                                             Q, tw);
            return;
        }
    }
    k4_rows_adj<N><<<dim3((ny + R - 1) / R, nb), L1Rows<N>::NT, L1Rows<N>::SMEM, s>>>(V, npairs, hh4, m, ny, twN, Q,
                                                                                      tw);
}

template <int N>
void l1_cols_adj(dim3 grid, cudaStream_t s, const float2* Q, int npairs, const float* w, int m, int nx, float* x,
                 float scale, const float2* tw) {
    if constexpr (N <= 256) {
        if (nx <= 256 && grid.x * grid.y <= 2 * kSms) {   // about two CTAs an SM
            k4_cols_adj_few<N><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(Q, npairs, w, m, nx, x, scale, tw);
            return;
        }
    }
    k4_cols_adj<N><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(Q, npairs, w, m, nx, x, scale, tw);
}

}  // namespace

cudaError_t launch_l1_rows_fwd(int nx, int nb, cudaStream_t s, const float2* G, int npairs,
                               const float2* hh4, int m, int ny, const float2* twN, float2* A,
                               const float2* tw) {
    switch (nx) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        l1_rows_fwd<N>(nb, s, G, npairs, hh4, m, ny, twN, A, tw);                              \
        break;
        PCE_L1_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_l1_cols_inv(int ny, dim3 grid, cudaStream_t s, const float2* A, int nx, float* y,
                               float scale, const float2* tw) {
    switch (ny) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        k4_cols_inv<N><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(A, nx, y, scale, tw);      \
        break;
        PCE_L1_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_l1_rows_adj(int nx, int nb, bool alone, cudaStream_t s, const float2* V, int npairs,
                               const float2* hh4, int m, int ny, const float2* twN, float2* Q,
                               const float2* tw) {
    switch (nx) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        l1_rows_adj<N>(nb, alone, s, V, npairs, hh4, m, ny, twN, Q, tw);                       \
        break;
        PCE_L1_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_l1_cols_adj(int ny, dim3 grid, cudaStream_t s, const float2* Q, int npairs,
                               const float* w, int m, int nx, float* x, float scale, const float2* tw) {
    switch (ny) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        l1_cols_adj<N>(grid, s, Q, npairs, w, m, nx, x, scale, tw);                            \
        break;
        PCE_L1_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_l1_rows_spec(int nx, dim3 grid, cudaStream_t s, const float2* G, int npairs, int m,
                                int ny, float2* hh4, const float2* tw) {
    switch (nx) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        k4_rows_spec<N><<<grid, L1Rows<N>::NT, L1Rows<N>::SMEM, s>>>(G, npairs, m, ny, hh4, tw); \
        break;
        PCE_L1_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

namespace {

// Few right-hand sides (a batch that leaves most SMs idle) take wide CTAs, which hold more
// slots, at 512 to 4096 points (1024: wk1d.cuh), by shares (Sum1d).  At 8192 every CTA holds
// one slot, by shares for any batch.  Below 512 the narrow CTA's slots hold so many pairs that
// wide CTAs add none and clusters little (N = 256, m = 40, one right-hand side, adjoint: 8.9 us
// with clusters, 10.5 without, 12.3 before the slots had barriers of their own).
template <int N>
constexpr bool has_wide() { return N >= 512 && N <= 4096 && N != kWarpN; }
template <int N>
constexpr bool has_shares() { return has_wide<N>() || N == 8192; }

template <int N, int WIDE, int MODE>
constexpr int smem_1d() { return MODE == kShares ? Cfg1d<N, WIDE>::SMEM_SHARES : Cfg1d<N, WIDE>::SMEM; }

template <int N, int WIDE, int MODE, typename WT, typename HT>
cudaError_t prepare_1d_as() {
    const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(k_fwd_1d<N, WT, HT, WIDE, MODE>, at, smem_1d<N, WIDE, MODE>());
    return e != cudaSuccess ? e : cudaFuncSetAttribute(k_adj_1d<N, WT, HT, WIDE, MODE>, at, smem_1d<N, WIDE, MODE>());
}

template <int N, typename WT, typename HT>
cudaError_t prepare_1d_of() {
    cudaError_t e = cudaSuccess;
    if constexpr (N != 8192) e = prepare_1d_as<N, 0, kOneSum, WT, HT>();
    if constexpr (has_shares<N>()) {
        if (e == cudaSuccess) e = prepare_1d_as<N, has_wide<N>(), kShares, WT, HT>();
        if (e == cudaSuccess) e = prepare_1d_as<N, has_wide<N>(), kCluster, WT, HT>();
    }
    return e;
}

}  // namespace

cudaError_t prepare_kernels() {
    cudaError_t e = prepare_cols();
    if (e == cudaSuccess) e = prepare_l1();
    if (e == cudaSuccess) e = prepare_sec();
#define X(N)                                                                                   \
    if (e == cudaSuccess) e = prepare_1d_of<N, float, float2>();                               \
    if (e == cudaSuccess) e = prepare_1d_of<N, __nv_bfloat16, __half2>();                      \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_spec_1d<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,    \
                                 Cfg1d<N>::SMEM);                                              \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_grad_1d<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,    \
                                 Cfg1d<N>::SMEM);
    PCE_1D_SIZES(X)
#undef X
    return e;
}

// Wide CTAs (more slots per right-hand side) when the batch leaves most SMs
// idle and the terms need more than one round of the narrow CTA's slots.
template <int N>
bool wide_1d(int batch, int m) {
    const int npairs = (m + 1) / 2;
    return has_wide<N>() && npairs > Cfg1d<N>::G && batch < 2 * 152;
}

// CTAs per right-hand side: one cluster whose CTAs share the rounds of term pairs
// that one CTA would run one after another (an SM each), doubled while the batch
// leaves SMs for them and a CTA has more than one round.  (Three rounds take four CTAs, one
// of them idle: one round long, where two CTAs would run two.)  N = 8192, m = 32, three
// right-hand sides, adjoint: 94.7 -> 28.9 us (three clusters of eight).  In the lanes of a
// batch too, where other tasks could use the SMs: 64 tasks of N = 8192, m = 32 on 16 lanes
// 408 -> 142 us, 256 of N = 4096 552 -> 259, 256 of all sizes 2769 -> 2800.
int cluster_1d(int batch, int rounds) {
    int cl = 1;
    while (cl < kMaxCluster && cl < rounds && (long long)batch * 2 * cl <= kSms) cl *= 2;
    return cl;
}

// Shares of the rounds (Sum1d): as many as the most CTAs, whatever the batch.
int shares_1d(int rounds) { return cluster_1d(1, rounds); }

// N = 1024 with few right-hand sides: the one-warp kernels (wk1d.cuh)
bool warp_1d(int n, int batch, const float2* tw1024) { return n == kWarpN && tw1024 && batch < 2 * 152; }

namespace {

template <int N, int WIDE, int MODE, typename WT, typename HT>
cudaError_t run_1d(bool adjoint, int batch, cudaStream_t s, const float* in, const WT* w, const HT* hp,
                   const float* hscale, int m, float* out, float scale, const float2* tw, int cl, int shares) {
    using CF = Cfg1d<N, WIDE>;
    return launch_cluster(adjoint ? k_adj_1d<N, WT, HT, WIDE, MODE> : k_fwd_1d<N, WT, HT, WIDE, MODE>, batch * cl, cl,
                          CF::NT, smem_1d<N, WIDE, MODE>(), s, in, w, hp, hscale, m, out, scale, tw, cl, shares);
}

template <int N, typename WT, typename HT>
cudaError_t run_1d_of(bool adjoint, int batch, cudaStream_t s, const float* in, const WT* w, const HT* hp,
                      const float* hscale, int m, float* out, float scale, const float2* tw) {
    if constexpr (has_shares<N>()) {
        constexpr int W = has_wide<N>();
        if (!W || wide_1d<N>(batch, m)) {
            const int rounds = ((m + 1) / 2 + Cfg1d<N, W>::G - 1) / Cfg1d<N, W>::G;
            const int cl = cluster_1d(batch, rounds), shares = shares_1d(rounds);
            if (cl > 1)
                return run_1d<N, W, kCluster>(adjoint, batch, s, in, w, hp, hscale, m, out, scale, tw, cl, shares);
            return run_1d<N, W, kShares>(adjoint, batch, s, in, w, hp, hscale, m, out, scale, tw, 1, shares);
        }
    }
    if constexpr (N != 8192)
        return run_1d<N, 0, kOneSum>(adjoint, batch, s, in, w, hp, hscale, m, out, scale, tw, 1, 1);
    return cudaErrorInvalidValue;   // not reached
}

template <typename WT, typename HT>
cudaError_t run_warp_1d(bool adjoint, int batch, cudaStream_t s, const float* in, const WT* w, const HT* hp,
                        const float* hscale, int m, float* out, float scale, const float2* tw1024) {
    const int rounds = ((m + 1) / 2 + kW1dWarps - 1) / kW1dWarps, shares = shares_1d(rounds);
    // one share a rank, or no cluster: m = 24, 70 right-hand sides 16.6 us with two, 14.5 alone
    const int cl = cluster_1d(batch, rounds) == shares ? shares : 1;
    if (cl > 1)
        return launch_cluster(adjoint ? kw_adj_1d<WT, HT, kCluster> : kw_fwd_1d<WT, HT, kCluster>, batch * cl, cl,
                              kW1dWarps * 32, 0, s, in, w, hp, hscale, m, out, scale, tw1024, cl, shares);
    return launch_cluster(adjoint ? kw_adj_1d<WT, HT, kShares> : kw_fwd_1d<WT, HT, kShares>, batch, 1, kW1dWarps * 32,
                          0, s, in, w, hp, hscale, m, out, scale, tw1024, 1, shares);
}

template <typename WT, typename HT>
cudaError_t apply_1d(bool adjoint, int n, int batch, cudaStream_t s, const float* in, const WT* w, const HT* hp,
                     const float* hscale, int m, float* out, float scale, const float2* tw, const float2* tw1024) {
    if (warp_1d(n, batch, tw1024)) return run_warp_1d(adjoint, batch, s, in, w, hp, hscale, m, out, scale, tw1024);
    switch (n) {
#define X(N) \
    case N: return run_1d_of<N>(adjoint, batch, s, in, w, hp, hscale, m, out, scale, tw);
        PCE_1D_SIZES(X)
#undef X
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_1d(bool adjoint, int n, int batch, cudaStream_t s, const float* in, const void* w, const void* hp,
                      const float* hscale, bool lowp, int m, float* out, float scale, const float2* tw,
                      const float2* tw1024) {
    if (lowp)
        return apply_1d(adjoint, n, batch, s, in, static_cast<const __nv_bfloat16*>(w),
                        static_cast<const __half2*>(hp), hscale, m, out, scale, tw, tw1024);
    return apply_1d(adjoint, n, batch, s, in, static_cast<const float*>(w), static_cast<const float2*>(hp), hscale, m,
                    out, scale, tw, tw1024);
}

cudaError_t launch_spec_1d(int n, int m, cudaStream_t s, const float* h, float2* hp,
                           const float2* tw) {
    switch (n) {
#define X(N)                                                                                   \
    case N: {                                                                                  \
        const int npairs = (m + 1) / 2;                                                        \
        const int grid = (npairs + Cfg1d<N>::G - 1) / Cfg1d<N>::G;                              \
        k_spec_1d<N><<<grid, Cfg1d<N>::NT, Cfg1d<N>::SMEM, s>>>(h, m, hp, tw);                 \
        break;                                                                                 \
    }
        PCE_1D_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_grad_1d(int n, int m, cudaStream_t s, const float* u, const float* r,
                           const float* w, const float2* hp, int nb, float2* dh, float* dw,
                           float scale, int accumulate, const float2* tw) {
    switch (n) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        k_grad_1d<N><<<m, Cfg1d<N>::NT, Cfg1d<N>::SMEM, s>>>(u, r, w, hp, nb, dh, dw, scale,   \
                                                             accumulate, tw);                  \
        break;
        PCE_1D_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace pce
