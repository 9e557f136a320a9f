// colsplit.cu -- forward column passes whose terms are shared by a cluster: few
// right-hand sides.
//
// The kernels of kernels.cuh and tkernels.cuh give a column tile's terms to one CTA, one
// after the other; with a few right-hand sides the tiles leave most SMs idle and the
// chain of a tile's terms is the time.  Here a cluster of S CTAs (blockIdx.z, the rank)
// takes a tile.  In a round each rank transforms one term's columns into its shared
// memory; then every rank owns 1 / S of the frequencies and adds, for these, the products
// of the round's S terms in term order, reading the other ranks' transforms through
// distributed shared memory.  So each frequency's sum is formed by the same operations
// in the same order as by one CTA: the same bits for any S, hence for any number of
// right-hand sides a launch.  (Adding the ranks' partial sums instead needs one
// exchange, not one a round, but makes the result depend on the batch.)  At the end rank 0
// collects the sums, runs the inverse transform and stores.
// What bounds them is latency: the chain of a round's reads, FFT and exchange.  Whole
// forward applies, m = 16, one right-hand side: 1024^2 separable 93 -> 81 us (unsplit ->
// split); 512^2 separable 52 -> 39; 256^2 dense 33 -> 27; 64^2 dense 31 -> 23.  Four CTAs at
// least: two repeat the exchange for half the rounds (256^2 dense, 8 right-hand sides 41 ->
// 51 us; 1024^2 separable, 2 right-hand sides 129 -> 160).
#include "kernels.cuh"
#include "tkernels.cuh"
#include "ckernels.cuh"
#include "launch.h"

namespace pce {

namespace {

// Shared memory of k_cols_fwd_split: the FFT buffers and two rounds' transforms.
template <int NY>
constexpr int split_smem() { return (ColCfg<NY>::C * ColCfg<NY>::CS + 2 * kR * ColCfg<NY>::NT) * (int)sizeof(float2); }

// k_cols_fwd over a cluster.  Grid (batch, NXh / C, S), clusters of (1, 1, S).  A rank
// owns kR / S of each thread's frequencies.  The round's transforms are double
// buffered, so one cluster barrier a round orders writes and reads.
template <int NY, int S, typename HT>
__global__ void __launch_bounds__(ColCfg<NY>::NT, 4)
k_cols_fwd_split(const float2* __restrict__ Z, long long z_bstride, long long z_kstride, const HT* __restrict__ hh,
                 const HT* __restrict__ hN, const float* __restrict__ hscale, int m, const Box* __restrict__ box,
                 int NXh, float2* __restrict__ A, long long a_bstride, const float2* __restrict__ tw) {
    using CC = ColCfg<NY>;
    constexpr int T = CC::T, C = CC::C, NT = CC::NT, VP = kR / S;
    extern __shared__ __align__(16) float2 smem[];
    const int c = threadIdx.x % C, j = threadIdx.x / C;
    float2* b0 = smem + c * CC::CS;
    float2* b1 = b0 + pad_len(NY);
    float2* X = smem + C * CC::CS;
    const int b = blockIdx.x, rank = blockIdx.z;
    const int col = blockIdx.y * C + c;
    const bool cv = col < NXh;
    const bool dcn = col == 0;
    const float2* Zb = Z + b * z_bstride;
    // the terms with a nonempty box in order, 32 boxes read at a time (a box after the
    // other, each read waits for the one before); m: none left
    int kb = -32;
    unsigned live = 0;
    auto next_term = [&] {
        while (live == 0) {
            kb += 32;
            if (kb >= m) return m;
            const int k = kb + (threadIdx.x & 31);
            live = __ballot_sync(0xffffffffu, k < m && box[k].nr > 0);
        }
        const int k = kb + __ffs(live) - 1;
        live &= live - 1;
        return k;
    };
    float2 acc[VP];
#pragma unroll
    for (int i = 0; i < VP; ++i) acc[i] = make_float2(0.f, 0.f);
    for (;; X = X == smem + C * CC::CS ? X + kR * NT : X - kR * NT) {
        int kk[S], mine = m;   // the round's terms (m: none)
#pragma unroll
        for (int g = 0; g < S; ++g) {
            kk[g] = next_term();
            if (g == rank) mine = kk[g];
        }
        if (kk[0] >= m) break;
        float2 hv[S][VP];
#pragma unroll
        for (int g = 0; g < S; ++g) {
            const float sk = kk[g] < m ? hscale_of<HT>(hscale, kk[g]) : 0.f;
#pragma unroll
            for (int i = 0; i < VP; ++i)
                hv[g][i] = cv && kk[g] < m
                               ? ldh(&hh[((long long)kk[g] * NY + j + (rank * VP + i) * T) * NXh + col], sk)
                               : make_float2(0.f, 0.f);
        }
        if (mine < m) {
            float2 v[kR];
            load_col<NY>(v, Zb + mine * z_kstride, box[mine], j, col, NXh, cv);
            fft<NY, false, kColLayout>(v, j, b0, b1, tw);
#pragma unroll
            for (int r = 0; r < kR; ++r) X[r * NT + threadIdx.x] = v[r];
        }
        cluster_sync();
#pragma unroll
        for (int g = 0; g < S; ++g) {
            if (kk[g] >= m) break;
            const unsigned a = cluster_map(X, g);
            float2 x[VP];
#pragma unroll
            for (int i = 0; i < VP; ++i) x[i] = cluster_ld2(a + ((rank * VP + i) * NT + threadIdx.x) * 8u);
            if (dcn) {
                const float sk = hscale_of<HT>(hscale, kk[g]);
#pragma unroll
                for (int i = 0; i < VP; ++i) {
                    const int f = j + (rank * VP + i) * T, fm = (NY - f) & (NY - 1);
                    float2 y, z;
                    split_dc_nyq(x[i], cluster_ld2(a + ((fm / T) * NT + (fm % T) * C) * 8u), y, z);
                    acc[i] = cfma(hv[g][i], y, acc[i]);
                    const float2 t = cmul(ldh(&hN[(long long)kk[g] * NY + f], sk), z);
                    acc[i].x -= t.y;
                    acc[i].y += t.x;
                }
            } else {
#pragma unroll
                for (int i = 0; i < VP; ++i) acc[i] = cfma(hv[g][i], x[i], acc[i]);
            }
        }
    }
    // this buffer's last readers have passed the last round's barrier
#pragma unroll
    for (int i = 0; i < VP; ++i) X[(rank * VP + i) * NT + threadIdx.x] = acc[i];
    cluster_sync();
    float2 v[kR];
    if (rank == 0) {
#pragma unroll
        for (int r = 0; r < kR; ++r) v[r] = cluster_ld2(cluster_map(X, r / VP) + (r * NT + threadIdx.x) * 8u);
    }
    cluster_sync();   // rank 0 has read the others' sums
    if (rank != 0) return;
    fft<NY, true, kColLayout>(v, j, b0, b1, tw);
    if (cv) {
        float2* Ab = A + b * a_bstride;
#pragma unroll
        for (int r = 0; r < kR; ++r) Ab[(long long)(j + r * T) * NXh + col] = v[r];
    }
}

// Shared memory of kt_cols_fwd_split: the transpose tiles and a rank's sums.
template <int NY, int S>
constexpr int tsplit_smem() { return kWColWarps * (fft_tile<NY>() + NY / S) * (int)sizeof(float2); }

// kt_cols_fwd<false, NY> over a cluster.  Grid (batch, NXh / 4, S), clusters of
// (1, 1, S), 128 threads.  Rank r owns frequencies lane + 32 q, q in its 1 / S of
// [0, NY / 32); its sums live in shared memory, a round's transforms in the transpose tiles.
template <int NY, int S>
__global__ void __launch_bounds__(kWColWarps * 32, NY == kWarpN ? 4 : 6)
kt_cols_fwd_split(const float2* __restrict__ Z, long long z_bstride, long long z_kstride,
                  const float2* __restrict__ hhT, const float2* __restrict__ hN, const Box* __restrict__ box, int NXh,
                  float2* __restrict__ A, long long a_bstride, const float2* __restrict__ tw, SepTerms sep) {
    constexpr int QN = NY / 32, QS = QN / S;
    extern __shared__ __align__(16) float2 smem[];
    float2* tile = smem;   // staging tile [NY][4] (swizzled), over the transpose tiles
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float2* tr = smem + warp * fft_tile<NY>();
    float2* sums = smem + kWColWarps * fft_tile<NY>() + warp * QS * 32 + lane;
    const int b = blockIdx.x, rank = blockIdx.z;
    const int col0 = blockIdx.y * kWColWarps, col = col0 + warp;   // NXh is a multiple of 8
    const bool dcn = col == 0;
    const float2* Zb = Z + b * z_bstride;
#pragma unroll
    for (int i = 0; i < QS; ++i) sums[32 * i] = make_float2(0.f, 0.f);
    auto prefetch = [&](int t) {
        if (lane == 0 && t < sep.nterms)
            bulk_prefetch_l2(hhT + ((long long)__ldg(&sep.korder[t]) * NXh + col) * NY, NY * sizeof(float2));
    };
    prefetch(rank);
    // this rank's term of a round, its slot and rows: three dependent reads, a round ahead
    int k = 0, sl = 0, r0 = 0, nr = 0;
    auto next_term = [&](int t) {
        if (t >= sep.nterms) return;
        k = __ldg(&sep.korder[t]);
        sl = __ldg(&sep.kslot[k]);
        r0 = box[sl].r0;
        nr = box[sl].nr;
    };
    next_term(rank);
    for (int t0 = 0; t0 < sep.nterms; t0 += S) {
        const int t = t0 + rank;
        if (t < sep.nterms) {   // uniform over the CTA
            tile_load(tile, Zb + sl * z_kstride, nr, NXh, col0);
            prefetch(t + S);
            const float* wr = sep.wrow + (long long)k * NY;
            float2 v[QN];
            cp_async_wait_all();
            __syncthreads();
#pragma unroll
            for (int q = 0; q < QN; ++q) {
                const int i = wrap(lane + 32 * q - r0, NY);
                v[q] = i < nr ? tile[tix(i, warp)] : make_float2(0.f, 0.f);
            }
            __syncthreads();   // the staging tile is read: the transpose tiles are free
            next_term(t + S);
            // right before the FFT, as in kt_cols_fwd: the compiler fuses these products
            // with the first butterflies' sums, and the bits have to be the same
#pragma unroll
            for (int q = 0; q < QN; ++q) v[q] = cscale(v[q], __ldg(&wr[lane + 32 * q]));
            warp_fft<NY, false, kTmSplit>(v, tr, tw);
            __syncwarp();
#pragma unroll
            for (int q = 0; q < QN; ++q) tr[lane + 32 * q] = v[q];
        }
        // this rank's frequencies of the round's spectra
        float2 h[S][QS];
#pragma unroll
        for (int g = 0; g < S; ++g) {
            if (t0 + g >= sep.nterms) break;
            const float2* hk = hhT + ((long long)__ldg(&sep.korder[t0 + g]) * NXh + col) * NY + lane + 32 * rank * QS;
#pragma unroll
            for (int i = 0; i < QS; ++i) h[g][i] = __ldg(&hk[32 * i]);
        }
        cluster_sync();
        float2 acc[QS];
#pragma unroll
        for (int i = 0; i < QS; ++i) acc[i] = sums[32 * i];
#pragma unroll
        for (int g = 0; g < S; ++g) {
            if (t0 + g >= sep.nterms) break;
            const unsigned a = cluster_map(tr, g);
            if (dcn) {
                const float2* hn = hN + (long long)__ldg(&sep.korder[t0 + g]) * NY;
#pragma unroll
                for (int i = 0; i < QS; ++i) {
                    const int f = lane + 32 * (rank * QS + i);
                    float2 x, y;
                    split_dc_nyq(cluster_ld2(a + 8u * f), cluster_ld2(a + 8u * ((NY - f) & (NY - 1))), x, y);
                    acc[i] = cfma(h[g][i], x, acc[i]);
                    const float2 s = cmul(__ldg(&hn[f]), y);
                    acc[i].x -= s.y;
                    acc[i].y += s.x;
                }
            } else {
                float2 x[QS];
#pragma unroll
                for (int i = 0; i < QS; ++i) x[i] = cluster_ld2(a + 8u * (lane + 32 * (rank * QS + i)));
#pragma unroll
                for (int i = 0; i < QS; ++i) acc[i] = cfma(h[g][i], x[i], acc[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < QS; ++i) sums[32 * i] = acc[i];
        cluster_sync();   // the round's transforms are read, the sums visible to rank 0
    }
    float2 acc[QN];
    if (rank == 0) {
#pragma unroll
        for (int q = 0; q < QN; ++q) acc[q] = cluster_ld2(cluster_map(sums, q / QS) + 256u * (q % QS));
    }
    cluster_sync();   // rank 0 has read the others' sums
    if (rank != 0) return;
    warp_fft<NY, true, kTmSplit>(acc, tr, tw);
    __syncthreads();   // every warp is done with its transpose tile: stage the four columns
#pragma unroll
    for (int q = 0; q < QN; ++q) tile[4 * (lane + 32 * q) + tix_sw(lane, warp)] = acc[q];
    __syncthreads();
    store_cols<NY>(A + b * a_bstride, tile, 0, NY, NXh, col0);
}

#define PCE_SPLIT_SIZES(X) X(16) X(32) X(64) X(128) X(256)

template <int NY, int S, typename HT>
cudaError_t split_fwd(const ColArgs& c, cudaStream_t s, const float2* Z, long long z_bstride, long long z_kstride,
                      float2* A, long long a_bstride) {
    return launch_cluster(k_cols_fwd_split<NY, S, HT>, dim3(c.nb, (c.nxh + ColCfg<NY>::C - 1) / ColCfg<NY>::C, S),
                          dim3(1, 1, S), ColCfg<NY>::NT, split_smem<NY>(), s, Z, z_bstride, z_kstride,
                          static_cast<const HT*>(c.hh), static_cast<const HT*>(c.hN), c.hscale, c.m, c.box, c.nxh, A,
                          a_bstride, c.tw);
}

template <int NY, typename HT>
cudaError_t split_fwd_of(const ColArgs& c, cudaStream_t s, const float2* Z, long long z_bstride, long long z_kstride,
                         float2* A, long long a_bstride) {
    switch (c.split) {
        case 4: return split_fwd<NY, 4, HT>(c, s, Z, z_bstride, z_kstride, A, a_bstride);
        case 8: return split_fwd<NY, 8, HT>(c, s, Z, z_bstride, z_kstride, A, a_bstride);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// Eight CTAs a tile, else four, while all are resident at once (four an SM), and only where they
// repay the exchange.  Eight: from 8 terms on, at 256 points with five terms a round (256^2, one
// right-hand side: 8 terms 23.6 -> 20.6 us, 16 terms 32.8 -> 26.7; two: 9 terms 24.6 -> 27.5;
// fewer terms, so of four CTAs: 5 terms 20.5 -> 24.6; 64 x 128, reduced storage, 10 terms, 18
// right-hand sides, both directions 61.4 -> 57.4).  Four: where the rounds are three quarters full and
// the chain is long, at 256 points from 28 terms on (4 right-hand sides: 16 terms 32.8 ->
// 34.6, 28 terms 47.2 -> 45.6, 64 terms 94.1 -> 85.8), at 64 from 40 on (64 x 2048, 2
// right-hand sides: 32 terms 57.6 -> 59.0, 48 terms 77.0 -> 75.4), at the other lengths,
// whose terms take longer one after another, from 8 on (128 x 256, 8 right-hand sides:
// 8 terms 28.7 -> 25.1, 32 terms 73.7 -> 54.9).
int cols_fwd_split(int ny, int m, long long ctas) {
    if (ny > 256) return 1;
    const int r8 = (m + 7) / 8, r4 = (m + 3) / 4;   // rounds
    if (m >= 8 && (ny < 256 || m >= 5 * r8) && ctas * 8 <= 4LL * kSms) return 8;
    if (m >= (ny == 256 ? 28 : ny == 64 ? 40 : 8) && m >= 3 * r4 && ctas * 4 <= 4LL * kSms) return 4;
    return 1;
}

cudaError_t launch_cols_fwd_split(const ColArgs& c, cudaStream_t s, const float2* Z, long long z_bstride,
                                  long long z_kstride, float2* A, long long a_bstride) {
    switch (c.ny) {
#define X(N)                                                                                                    \
    case N:                                                                                                     \
        return c.lowp ? split_fwd_of<N, __half2>(c, s, Z, z_bstride, z_kstride, A, a_bstride)                   \
                      : split_fwd_of<N, float2>(c, s, Z, z_bstride, z_kstride, A, a_bstride);
        PCE_SPLIT_SIZES(X)
#undef X
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_cols_fwd_sep_split(int ny, dim3 grid, cudaStream_t s, const float2* Z, long long z_bstride,
                                      long long z_kstride, const float2* hhT, const float2* hN, const Box* box, int nxh,
                                      float2* A, long long a_bstride, const float2* tw1024, const SepTerms& sep) {
    if (!tw1024 || !hhT || nxh % kWColWarps) return cudaErrorInvalidValue;
    auto go = [&](auto kernel, int smem) {
        return launch_cluster(kernel, grid, dim3(1, 1, grid.z), kWColWarps * 32, smem, s, Z, z_bstride, z_kstride, hhT,
                              hN, box, nxh, A, a_bstride, tw1024, sep);
    };
    if (ny == kWarpN && grid.z == 4) return go(kt_cols_fwd_split<kWarpN, 4>, tsplit_smem<kWarpN, 4>());
    if (ny == 512 && grid.z == 4) return go(kt_cols_fwd_split<512, 4>, tsplit_smem<512, 4>());
    return cudaErrorInvalidValue;
}

// every kernel above fits the shared memory that needs no attribute
static_assert(split_smem<256>() <= 48 * 1024 && split_smem<16>() <= 48 * 1024 && split_smem<64>() <= 48 * 1024 &&
                  tsplit_smem<kWarpN, 4>() <= 48 * 1024 && tsplit_smem<512, 4>() <= 48 * 1024,
              "column kernels over clusters: shared memory");

}  // namespace pce
