// cols.cu -- instances of the column-pass kernels for NY = 16 .. 2048 (one-warp
// kernels for NY = 512, 1024 and, two warps per column, 2048).
#include <algorithm>

#include "kernels.cuh"
#include "wkernels.cuh"
#include "wkernels2.cuh"
#include "ckernels.cuh"
#include "tkernels.cuh"
#include "launch.h"

namespace pce {

#define PCE_COL_SIZES(X) X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048)

int cols_columns_per_cta(int ny) {
    switch (ny) {
#define X(N) case N: return ColCfg<N>::C;
        PCE_COL_SIZES(X)
#undef X
    }
    return 0;
}
int cols_ctas_per_sm(int ny) {
    constexpr int kSmSmem = 228 * 1024, kCtaReserve = 1024;   // shared memory of an SM, taken by every CTA
    switch (ny) {
#define X(N) case N: return std::min({4, 2048 / ColCfg<N>::NT, kSmSmem / (ColCfg<N>::SMEM + kCtaReserve)});
        PCE_COL_SIZES(X)
#undef X
    }
    return 1;
}

template <int NF, int PAR, typename HT>
cudaError_t prepare_ccols_of() {
    const void* fns[] = {(const void*)kc_cols_fwd<NF, PAR, false, HT>, (const void*)kc_cols_fwd<NF, PAR, true, HT>,
                         (const void*)kc_cols_adj<NF, PAR, false, false, HT>,
                         (const void*)kc_cols_adj<NF, PAR, false, true, HT>,
                         (const void*)kc_cols_adj<NF, PAR, true, false, HT>};
    for (const void* f : fns) {
        const cudaError_t e =
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kc_smem<NF, PAR>(NF));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t prepare_ccols() {
    cudaError_t e = prepare_ccols_of<512, 1, float2>();
    if (e == cudaSuccess) e = prepare_ccols_of<512, 1, __half2>();
    if (e == cudaSuccess) e = prepare_ccols_of<1024, 1, float2>();
    if (e == cudaSuccess) e = prepare_ccols_of<1024, 1, __half2>();
    if (e == cudaSuccess) e = prepare_ccols_of<1024, 2, float2>();
    if (e == cudaSuccess) e = prepare_ccols_of<1024, 2, __half2>();
    return e;
}

// Every row of Q (the window gradient): block kernels up to 256 rows, kc_cols_adj above.
template <int N>
constexpr bool full_block() { return N <= 256; }
template <int N>
cudaError_t prepare_full() {
    if constexpr (full_block<N>())
        return cudaFuncSetAttribute(k_cols_adj<N, true, float2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    ColCfg<N>::SMEM);
    return cudaSuccess;
}

cudaError_t prepare_cols() {
    cudaError_t e = prepare_ccols();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kt_cols_fwd<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTColSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kt_cols_adj<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTColSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kt_cols_fwd<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTColSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kt_cols_adj<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTColSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kw2_cols_fwd<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kW2Smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kw2_cols_fwd<__half2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kW2Smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kw_cols_fwd<kWarpN>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWColSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kw_cols_adj<kWarpN>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWColSmem);
#define X(N)                                                                                   \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_cols_fwd<N, float2>,                                        \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, ColCfg<N>::SMEM); \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_cols_fwd<N, __half2>,                                       \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, ColCfg<N>::SMEM); \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_cols_adj<N, false, float2>,                                 \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, ColCfg<N>::SMEM); \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_cols_adj<N, false, __half2>,                                \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, ColCfg<N>::SMEM); \
    if (e == cudaSuccess) e = prepare_full<N>();                                               \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_cols_grad_h<N>,                                             \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, ColCfg<N>::SMEM); \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_cols_spec<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                 ColCfg<N>::SMEM);                                             \
    if (e == cudaSuccess)                                                                      \
        e = cudaFuncSetAttribute(k_plain_cols_inv<N>,                                          \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, ColCfg<N>::SMEM);
    PCE_COL_SIZES(X)
#undef X
    return e;
}

int col_frame_rows(int ny, const Box* box, int m) {
    if (ny != 512 && ny != 1024 && ny != 2048) return 0;
    const int nf = ny == 512 ? 512 : 1024;
    int rows = 1;
    for (int k = 0; k < m; ++k) {
        const int need = (box[k].r0 & 31) + box[k].nr;
        if (box[k].nr == 0 || need <= rows) continue;
        if (need > nf && ny == 2048) return 0;
        rows = need < nf ? need : nf;
    }
    return rows;
}

long long col_table_size(int ny) {
    return 2ll * (ny == 512    ? col_table_len<512, 1>()
                  : ny == 1024 ? col_table_len<1024, 1>()
                  : ny == 2048 ? col_table_len<1024, 2>()
                               : 0);
}

namespace {

dim3 ccols_grid(int nb, int nxh, unsigned split) { return dim3(nb, (nxh + kCCols - 1) / kCCols, split); }

template <int NF, int PAR, typename HT>
cudaError_t ccols_fwd(const ColArgs& c, cudaStream_t s, const float2* Z, long long z_bstride, long long z_kstride,
                      float2* A, long long a_bstride) {
    const bool half = c.frame_rows <= NF / 2;
    auto kernel = half ? kc_cols_fwd<NF, PAR, true, HT> : kc_cols_fwd<NF, PAR, false, HT>;
    kernel<<<ccols_grid(c.nb, c.nxh, 1), kCCols * PAR * 32, kc_smem<NF, PAR>(half ? NF / 2 : NF), s>>>(
        Z, z_bstride, z_kstride, static_cast<const HT*>(c.hhT), static_cast<const HT*>(PAR == 2 ? c.hN2 : c.hN),
        c.hscale, c.m, c.box, c.nxh, A, a_bstride, c.tw1024, c.tab, c.tw2048l, c.status, c.wait_limit, c.skip_copy);
    return cudaGetLastError();
}

template <int NF, int PAR, typename HT>
cudaError_t ccols_adj(const ColArgs& c, bool full, cudaStream_t s, const float2* V, long long v_bstride, float2* Q,
                      long long q_bstride, long long q_kstride) {
    auto kernel = full || c.frame_rows == 0     ? kc_cols_adj<NF, PAR, true, false, HT>
                  : c.frame_rows <= NF / 2 ? kc_cols_adj<NF, PAR, false, true, HT>
                                           : kc_cols_adj<NF, PAR, false, false, HT>;
    kernel<<<ccols_grid(c.nb, c.nxh, c.split), kCCols * PAR * 32, kc_smem<NF, PAR>(0), s>>>(
        V, v_bstride, static_cast<const HT*>(c.hhT), static_cast<const HT*>(PAR == 2 ? c.hN2 : c.hN), c.hscale, c.m,
        c.box, c.nxh, Q, q_bstride, q_kstride, c.tw1024, c.tab, c.tw2048l, full ? 1 : 0);
    return cudaGetLastError();
}

template <typename HT>
cudaError_t cols_fwd(const ColArgs& c, cudaStream_t s, const float2* Z, long long z_bstride, long long z_kstride,
                     float2* A, long long a_bstride) {
    if (c.warp && c.ny == 512) return ccols_fwd<512, 1, HT>(c, s, Z, z_bstride, z_kstride, A, a_bstride);
    if (c.warp && c.ny == 1024) return ccols_fwd<1024, 1, HT>(c, s, Z, z_bstride, z_kstride, A, a_bstride);
    if (c.warp && c.ny == 2048 && c.frame_rows > 0)
        return ccols_fwd<1024, 2, HT>(c, s, Z, z_bstride, z_kstride, A, a_bstride);
    if (c.warp && c.ny == 2048) {
        kw2_cols_fwd<HT><<<dim3(c.nb, (c.nxh + kW2Cols - 1) / kW2Cols), 128, kW2Smem, s>>>(
            Z, z_bstride, z_kstride, static_cast<const HT*>(c.hhT), static_cast<const HT*>(c.hN2), c.hscale, c.m,
            c.box, c.nxh, A, a_bstride, c.tw1024, c.tw2048l, c.status, c.wait_limit, c.skip_copy);
        return cudaGetLastError();
    }
    switch (c.ny) {
#define X(N)                                                                                                     \
    case N:                                                                                                      \
        k_cols_fwd<N, HT><<<dim3(c.nb, (c.nxh + ColCfg<N>::C - 1) / ColCfg<N>::C), ColCfg<N>::NT,                \
                            ColCfg<N>::SMEM, s>>>(Z, z_bstride, z_kstride, static_cast<const HT*>(c.hh),         \
                                                  static_cast<const HT*>(c.hN), c.hscale, c.m, c.box, c.nxh, A,  \
                                                  a_bstride, c.tw);                                              \
        return cudaGetLastError();
        PCE_COL_SIZES(X)
#undef X
    }
    return cudaErrorInvalidValue;
}

template <int N, bool FULL, typename HT>
cudaError_t block_adj(const ColArgs& c, cudaStream_t s, const float2* V, long long v_bstride, float2* Q,
                      long long q_bstride, long long q_kstride) {
    if constexpr (FULL && !full_block<N>()) {
        return cudaErrorInvalidValue;
    } else {
        k_cols_adj<N, FULL, HT><<<dim3(c.nb, (c.nxh + ColCfg<N>::C - 1) / ColCfg<N>::C, c.split), ColCfg<N>::NT,
                                  ColCfg<N>::SMEM, s>>>(V, v_bstride, static_cast<const HT*>(c.hh),
                                                        static_cast<const HT*>(c.hN), c.hscale, c.m, c.box, c.nxh, Q,
                                                        q_bstride, q_kstride, c.tw);
        return cudaGetLastError();
    }
}

template <bool FULL, typename HT>
cudaError_t cols_adj(const ColArgs& c, cudaStream_t s, const float2* V, long long v_bstride, float2* Q,
                     long long q_bstride, long long q_kstride) {
    if (c.warp && c.ny == 512) return ccols_adj<512, 1, HT>(c, FULL, s, V, v_bstride, Q, q_bstride, q_kstride);
    if (c.warp && c.ny == 1024) return ccols_adj<1024, 1, HT>(c, FULL, s, V, v_bstride, Q, q_bstride, q_kstride);
    if (c.warp && c.ny == 2048) return ccols_adj<1024, 2, HT>(c, FULL, s, V, v_bstride, Q, q_bstride, q_kstride);
    switch (c.ny) {
#define X(N) \
    case N: return block_adj<N, FULL, HT>(c, s, V, v_bstride, Q, q_bstride, q_kstride);
        PCE_COL_SIZES(X)
#undef X
    }
    return cudaErrorInvalidValue;
}

// the one-warp column kernels index these tables: refuse to launch without them
bool tables_missing(const ColArgs& c) {
    const bool warp_size = c.ny == 512 || c.ny == 1024 || c.ny == 2048;
    return warp_size && c.warp && (!c.tw1024 || !c.tab || !c.hhT || (c.ny == 2048 && (!c.tw2048l || !c.hN2)));
}

}  // namespace

cudaError_t launch_cols_fwd(const ColArgs& c, cudaStream_t s, const float2* Z, long long z_bstride,
                            long long z_kstride, float2* A, long long a_bstride) {
    if (tables_missing(c)) return cudaErrorInvalidValue;
    if (c.split > 1) return launch_cols_fwd_split(c, s, Z, z_bstride, z_kstride, A, a_bstride);
    return c.lowp ? cols_fwd<__half2>(c, s, Z, z_bstride, z_kstride, A, a_bstride)
                  : cols_fwd<float2>(c, s, Z, z_bstride, z_kstride, A, a_bstride);
}

cudaError_t launch_cols_adj(const ColArgs& c, cudaStream_t s, const float2* V, long long v_bstride, float2* Q,
                            long long q_bstride, long long q_kstride) {
    if (tables_missing(c)) return cudaErrorInvalidValue;
    return c.lowp ? cols_adj<false, __half2>(c, s, V, v_bstride, Q, q_bstride, q_kstride)
                  : cols_adj<false, float2>(c, s, V, v_bstride, Q, q_bstride, q_kstride);
}

cudaError_t launch_cols_adj_full(const ColArgs& c, cudaStream_t s, const float2* V, long long v_bstride, float2* Q,
                                 long long q_bstride, long long q_kstride) {
    if (tables_missing(c) || c.lowp) return cudaErrorInvalidValue;
    return cols_adj<true, float2>(c, s, V, v_bstride, Q, q_bstride, q_kstride);
}

cudaError_t launch_cols_spec(int ny, dim3 grid, cudaStream_t s, const float2* S, int nxh,
                             float2* hh, float2* hN, const float2* tw) {
    switch (ny) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        k_cols_spec<N><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(S, nxh, hh, hN, tw);        \
        break;
        PCE_COL_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_plain_cols_inv(int ny, dim3 grid, cudaStream_t s, const float2* acc,
                                  const float2* accN, int nxh, float2* A, const float2* tw) {
    switch (ny) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        k_plain_cols_inv<N><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(acc, accN, nxh, A, tw); \
        break;
        PCE_COL_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_cols_fwd_sep(int ny, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                                long long z_kstride, const float2* hhT, const float2* hN,
                                const Box* box, int nxh, float2* A, long long a_bstride,
                                const float2* tw1024, int* status, long long wait_limit, int skip_copy,
                                const SepTerms& sep) {
    if (!tw1024 || !hhT) return cudaErrorInvalidValue;
    if (ny == kWarpN)
        kw_cols_fwd<kWarpN><<<grid, kWColWarps * 32, kWColSmem, s>>>(
            Z, z_bstride, z_kstride, hhT, hN, box, nxh, A, a_bstride, tw1024, status, wait_limit,
            skip_copy, sep);
    else if (ny == 512)
        kw_cols_fwd<512><<<grid, kWColWarps * 32, kw_col_smem<512>(), s>>>(
            Z, z_bstride, z_kstride, hhT, hN, box, nxh, A, a_bstride, tw1024, status, wait_limit,
            skip_copy, sep);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_cols_adj_sep(int ny, dim3 grid, cudaStream_t s, const float2* V, long long v_bstride,
                                const float2* hhT, const float2* hN, const Box* box, int nxh,
                                float2* Q, long long q_bstride, long long q_kstride,
                                const float2* tw1024, int* status, long long wait_limit, int skip_copy,
                                const SepTerms& sep) {
    if (!tw1024 || !hhT) return cudaErrorInvalidValue;
    if (ny == kWarpN)
        kw_cols_adj<kWarpN><<<grid, kWColWarps * 32, kWColSmem, s>>>(
            V, v_bstride, hhT, hN, box, nxh, Q, q_bstride, q_kstride, tw1024, status, wait_limit,
            skip_copy, sep);
    else if (ny == 512)
        kw_cols_adj<512><<<grid, kWColWarps * 32, kw_col_smem<512>(), s>>>(
            V, v_bstride, hhT, hN, box, nxh, Q, q_bstride, q_kstride, tw1024, status, wait_limit,
            skip_copy, sep);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_cols_fwd_sep_tm(int ny, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                                   long long z_kstride, const float2* hhT, const float2* hN, const Box* box,
                                   int nxh, float2* A, long long a_bstride, const float2* tw1024, int* status,
                                   long long wait_limit, int skip_copy, const SepTerms& sep) {
    if (!tw1024 || !hhT || (grid.z > 1 && (sep.kq0 || sep.t1 >= 0))) return cudaErrorInvalidValue;
    if (grid.z > 1)
        return launch_cols_fwd_sep_split(ny, grid, s, Z, z_bstride, z_kstride, hhT, hN, box, nxh, A, a_bstride, tw1024,
                                         sep);
    if (ny == 512 && !sep.kq0) {   // 512-point columns: no pruned form
        kt_cols_fwd<false, 512><<<grid, kWColWarps * 32, kt_smem<512>(), s>>>(
            Z, z_bstride, z_kstride, hhT, hN, box, nxh, A, a_bstride, tw1024, status, wait_limit, skip_copy, sep);
        return cudaGetLastError();
    }
    if (ny != kWarpN) return cudaErrorInvalidValue;
    if (sep.kq0)
        kt_cols_fwd<true><<<grid, kWColWarps * 32, kTColSmem, s>>>(Z, z_bstride, z_kstride, hhT, hN, box, nxh, A,
                                                                   a_bstride, tw1024, status, wait_limit, skip_copy,
                                                                   sep);
    else
        kt_cols_fwd<false><<<grid, kWColWarps * 32, kTColSmem, s>>>(Z, z_bstride, z_kstride, hhT, hN, box, nxh, A,
                                                                    a_bstride, tw1024, status, wait_limit,
                                                                    skip_copy, sep);
    return cudaGetLastError();
}

cudaError_t launch_cols_adj_sep_tm(int ny, dim3 grid, cudaStream_t s, float2* V, long long v_bstride,
                                   const float2* hhT, const float2* hN, const Box* box, int nxh, float2* Q,
                                   long long q_bstride, long long q_kstride, const float2* tw1024, int* status,
                                   long long wait_limit, int skip_copy, const SepTerms& sep) {
    if (!tw1024 || !hhT) return cudaErrorInvalidValue;
    if (ny == 512 && !sep.kq0) {
        kt_cols_adj<false, 512><<<grid, kWColWarps * 32, kt_smem<512>(), s>>>(
            V, v_bstride, hhT, hN, box, nxh, Q, q_bstride, q_kstride, tw1024, status, wait_limit, skip_copy, sep);
        return cudaGetLastError();
    }
    if (ny != kWarpN) return cudaErrorInvalidValue;
    if (sep.kq0)
        kt_cols_adj<true><<<grid, kWColWarps * 32, kTColSmem, s>>>(V, v_bstride, hhT, hN, box, nxh, Q, q_bstride,
                                                                   q_kstride, tw1024, status, wait_limit, skip_copy,
                                                                   sep);
    else
        kt_cols_adj<false><<<grid, kWColWarps * 32, kTColSmem, s>>>(V, v_bstride, hhT, hN, box, nxh, Q, q_bstride,
                                                                    q_kstride, tw1024, status, wait_limit,
                                                                    skip_copy, sep);
    return cudaGetLastError();
}

cudaError_t launch_cols_grad_h(int ny, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                               long long z_kstride, int nb, const float2* Rh, const float2* RhN,
                               const Box* box, int nxh, float2* dhh, float scale, int accumulate,
                               const float2* tw) {
    switch (ny) {
#define X(N)                                                                                   \
    case N:                                                                                    \
        k_cols_grad_h<N><<<grid, ColCfg<N>::NT, ColCfg<N>::SMEM, s>>>(                          \
            Z, z_bstride, z_kstride, nb, Rh, RhN, box, nxh, dhh, scale, accumulate, tw);       \
        break;
        PCE_COL_SIZES(X)
#undef X
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace pce
