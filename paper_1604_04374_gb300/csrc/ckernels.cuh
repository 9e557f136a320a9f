// ckernels.cuh -- column kernels of dense (not separable) plans for columns of
// NY = NF PAR points: 512 and 1024 (PAR = 1) and 2048 (NF = 1024, PAR = 2).
//
// Every column is transformed by PAR warps with the one-warp FFT of NF points
// (warpfft.cuh).  PAR = 2 splits the 2048-point DFT by decimation in frequency:
//   X[2k]     = DFT1024( x[n] + x[n + 1024] )[k]
//   X[2k + 1] = DFT1024( (x[n] - x[n + 1024]) W2048^n )[k]
// and warp `par` of a column takes the even (0) or the odd (1) frequencies; the
// inverse runs the two halves backwards, a = IDFT(even), b = W2048^-n IDFT(odd),
// x[n] = a + b, x[n + 1024] = a - b, combined when the column is stored.  Spectra:
// hhT [m][NXh][PAR][NF] (column 0: the DC column), hN [m][PAR][NF] (Nyquist column).
//
// A CTA takes four columns (4 PAR warps).  What bounds these kernels is latency
// (a term's rows and spectrum come from L2 or DRAM) and the instructions around
// the FFT, so:
//  - the state a warp carries from term to term (forward: the spectral accumulator,
//    adjoint: the column spectrum of V) lives in tensor memory (tmem.cuh), which
//    leaves 128 registers a thread and 16 warps an SM (20 and more at 512 points);
//  - a term's rows are staged for the CTA by cp.async while the previous term's FFT
//    runs, on a frame that starts at a multiple of 32 rows, 32 s (the box's first row
//    rounded down), zeros around the box.  The warps transform the frame's rows in
//    place, x'[i] = x[32 s + i], i < NF: no index or bounds arithmetic a value, for
//    PAR = 2 no second half (i < 1024), and where every frame holds at most NF / 2
//    rows (HALF; Lemma 3.2) an FFT without the butterflies of its zero half, an
//    inverse without the outputs outside the frame.  The shift costs nothing:
//    FFT(x)[f] = W^(32 s f) FFT(x')[f], and with f = PAR (p + 32 j) + par the phase is
//    W^(32 s (PAR p + par)), independent of j, so it is folded into the twiddles of
//    the four-step FFT, which the first transform leaves at register p (forward) or
//    lane p (inverse): one table a value of (s, par) and direction (col_tables);
//  - the next term's spectrum is started towards L2 a term ahead (one bulk prefetch
//    a warp); the forward brings it into the warp's transpose tile during the second
//    half of the FFT, the adjoint loads it straight into registers;
//    The twiddle tables cost 2 MB a plan of 2048 rows (0.5 and 0.1 MB at 1024 and 512);
//  - the power-of-two scale of a term's reduced spectrum is applied where the fewest
//    values pass (exact): to the staged rows (forward), to the stored rows (adjoint).
//
// 2048^2, m = 64, 4 right-hand sides, reduced storage, forward, whole apply: 3742 us
// with the register kernels, 2286 with tensor memory and frames read behind uniform
// branches, 1907 with the shifted transforms.  At 2048^2, m = 16, 2 right-hand sides
// the forward / adjoint kernels execute 123 / 115 M warp instructions (164 / 132 M
// before the shift) at 57 % of the issue slots: 192 / 185 us.
#pragma once

#include "tkernels.cuh"

namespace pce {

constexpr int kCCols = 4;   // columns per CTA

// cos(2 pi j / 64) on [0, 16] (FP32, rounded from FP64; exact at 0 and 16)
__host__ __device__ constexpr float cos64q(int j) {
    return j == 0 ? 1.0f : j == 1 ? 0.9951847f : j == 2 ? 0.98078525f : j == 3 ? 0.95694035f
         : j == 4 ? 0.9238795f : j == 5 ? 0.8819213f : j == 6 ? 0.8314696f : j == 7 ? 0.77301043f
         : j == 8 ? 0.70710677f : j == 9 ? 0.6343933f : j == 10 ? 0.55557024f : j == 11 ? 0.47139674f
         : j == 12 ? 0.38268343f : j == 13 ? 0.29028466f : j == 14 ? 0.19509032f : j == 15 ? 0.09801714f
         : 0.0f;
}
__host__ __device__ constexpr float cos64(int j) {
    return (j & 63) <= 16 ? cos64q(j & 63)
         : (j & 63) <= 32 ? -cos64q(32 - (j & 63))
         : (j & 63) <= 48 ? -cos64q((j & 63) - 32)
         : cos64q(64 - (j & 63));
}
// W64^q = exp(-2 pi i q / 64)
__host__ __device__ constexpr float2 w64(int q) { return float2{cos64(q), -cos64((q + 48) & 63)}; }

// tensor-memory columns of a CTA: 2 NF / 32 a warp, four warps side by side
template <int NF, int PAR>
__host__ __device__ constexpr int kc_tm_cols() { return PAR * 2 * (NF / 32); }
// CTAs per SM the kernels are compiled for (128 registers; 80 at 512 points)
template <int NF, int PAR>
__host__ __device__ constexpr int kc_min_ctas() { return NF == 512 ? 6 : PAR == 1 ? 4 : 2; }
// shared memory: the transpose tiles, and in the forward a term's frame rows
template <int NF, int PAR>
__host__ __device__ constexpr int kc_smem(int rows) {
    return (kCCols * PAR * warp_tile(NF) + rows * kCCols) * (int)sizeof(float2);
}

// Frame of a term's rows: frame row i is row 32 s + i of the column (mod NY), the
// box's row r is frame row (a + r) mod NY.  Boxes that do not fit a frame of NF rows
// take the whole period (PAR = 1; columns of 2048 with such boxes use wkernels2.cuh).
struct CFrame {
    int s, a;
};
template <int NF>
__host__ __device__ __forceinline__ CFrame col_frame(const Box& b) {
    const int a = b.r0 & 31;
    return a + b.nr > NF ? CFrame{0, b.r0} : CFrame{b.r0 >> 5, a};
}

// Phased twiddles: tab[dir][s][par][p * 32 + l] = W_NF^(l p) W_NY^(32 s (PAR k + par)),
// k = p for dir 0 (forward), k = l for dir 1 (inverse, used conjugated).
template <int NF, int PAR>
__host__ __device__ constexpr int col_table_len() { return NF * PAR * (NF * PAR / 32); }
template <int NF, int PAR>
__device__ __forceinline__ const float2* col_table(const float2* tab, int dir, int s, int par) {
    return tab + (long long)dir * col_table_len<NF, PAR>() + (s * PAR + par) * NF;
}

__device__ __forceinline__ void bulk_prefetch_l2(const void* p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}

// Cooperative async copy of a term's box rows (src [nr][nxh], columns col0 ..
// col0 + 3) to ROWS rows of its frame in the swizzled tile, zeros outside the box.
template <int NY, int ROWS, int NT>
__device__ __forceinline__ void frame_load(float2* tile, const float2* __restrict__ src, const Box& b, CFrame f,
                                           int nxh, int col0) {
#pragma unroll 4
    for (int e = threadIdx.x; e < ROWS * kCCols; e += NT) {
        const int i = e >> 2, c = e & 3;
        const int r = wrap(i - f.a, NY);
        const bool ok = r < b.nr && col0 + c < nxh;
        cp_async8(tile + tix(i, c), src + (ok ? (long long)r * nxh + col0 + c : 0), ok);
    }
    cp_async_commit();
}

// X[NY - f] of a packed DC/Nyquist column from the transpose tile holding this
// warp's half: index NF - f' (even half) or NF - 1 - f' (odd half).
template <int NF>
__device__ __forceinline__ float2 half_partner(const float2* tr, int f, int par) {
    return tr[par ? NF - 1 - f : (NF - f) & (NF - 1)];
}

// The four columns' inverse transforms (transpose tiles of the CTA, element n of
// column c, half p at (c PAR + p) warp_tile(NF) + ((n + 4 c) mod NF)) combined and stored:
// rows i < nr of dst ([rows][nxh], columns col0 ..) from rows r0 + i (mod NY),
// times sc.  Two columns a 16-byte store where dst allows it.
template <int NF, int PAR, int NT>
__device__ __forceinline__ void store_halves(float2* __restrict__ dst, const float2* tiles, int r0, int nr, int nxh,
                                             int col0, float sc) {
    constexpr int NY = NF * PAR;
    auto get = [&](int g, int c) {
        const int n = (g + 4 * c) & (NF - 1);
        const float2* t = tiles + c * PAR * warp_tile(NF);
        float2 x = t[n];
        if constexpr (PAR == 2) {
            const float2 y = t[warp_tile(NF) + n];
            x = g < NF ? cadd(x, y) : csub(x, y);
        }
        return cscale(x, sc);
    };
    if ((reinterpret_cast<unsigned long long>(dst) & 15) == 0 && (nxh & 3) == 0) {
        for (int e = threadIdx.x; e < nr * 2; e += NT) {
            const int i = e >> 1, c = (e & 1) * 2;
            const int g = wrap(r0 + i, NY);
            const float2 x0 = get(g, c), x1 = get(g, c + 1);
            *reinterpret_cast<float4*>(dst + (long long)i * nxh + col0 + c) = make_float4(x0.x, x0.y, x1.x, x1.y);
        }
    } else {
        for (int e = threadIdx.x; e < nr * kCCols; e += NT) {
            const int i = e >> 2, c = e & 3;
            if (col0 + c < nxh) dst[(long long)i * nxh + col0 + c] = get(wrap(r0 + i, NY), c);
        }
    }
}

// F2.  Grid (batch, ceil(NXh / 4)), 128 PAR threads, kc_smem<NF, PAR>(frame rows)
// bytes.  tab: the phased twiddles (forward part), tw: the plain ones.
template <int NF, int PAR, bool HALF, typename HT>
__global__ void __launch_bounds__(kCCols * PAR * 32, (kc_min_ctas<NF, PAR>()))
kc_cols_fwd(const float2* __restrict__ Z, long long z_bstride, long long z_kstride, const HT* __restrict__ hhT,
            const HT* __restrict__ hN, const float* __restrict__ hscale, int m, const Box* __restrict__ box, int NXh,
            float2* __restrict__ A, long long a_bstride, const float2* __restrict__ tw,
            const float2* __restrict__ tab, const float2* __restrict__ tw2048l, int* __restrict__ status,
            long long wait_limit, int skip_copy) {
    constexpr int ROWS = HALF ? NF / 2 : NF;
    constexpr int NY = NF * PAR, QN = NF / 32, NQ = QN / 8, NT = kCCols * PAR * 32;
    extern __shared__ __align__(16) float2 smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cl = warp / PAR, par = warp % PAR;
    float2* tr = smem + warp * warp_tile(NF);           // this warp's transpose tile
    float2* tile = smem + kCCols * PAR * warp_tile(NF);   // the term's rows
    __shared__ unsigned long long bars[kCCols * PAR];
    __shared__ unsigned tm_slot;
    const int b = blockIdx.x;
    const int col0 = blockIdx.y * kCCols, col = col0 + cl;
    const bool cv = col < NXh;
    const bool dcn = col == 0;
    const float2* Zb = Z + b * z_bstride;
    unsigned long long* bar = &bars[warp];
    if (lane == 0) mbar_init(bar);
    if (warp == 0) tm_alloc(&tm_slot, kc_tm_cols<NF, PAR>());
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const unsigned t_acc = tm_slot + ((unsigned)(32 * (warp & 3)) << 16) + (warp >> 2) * 2 * QN;
    {
        float2 z[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) z[j] = make_float2(0.f, 0.f);
#pragma unroll
        for (int qq = 0; qq < NQ; ++qq) tm_store8c(t_acc + 16 * qq, z);
        tm_wait_st();
    }
    unsigned parity = 0;
    bool failed = false;
    const float2 wl = PAR == 2 ? __ldg(&tw2048l[lane]) : make_float2(1.f, 0.f);
    const HT* hcol = hhT + ((long long)(cv ? col : 0) * PAR + par) * NF;   // + k NXh PAR NF
    const long long hstride = (long long)NXh * PAR * NF;
    const int sw = tix_sw(lane, cl);

    const int kend = m;
    // The terms with a nonempty box in order.  512 points in reduced storage, the shortest chain
    // a term: 32 boxes looked at at a time, and the next term's box and scale read before
    // this one's rows are waited for (512 x 64, m = 9, forward apply 45.2 -> 41.0 us).  The
    // longer chains lose by it (2048 x 256, m = 16, 4 right-hand sides 154 -> 174 us).
    constexpr bool kAhead = NF == 512 && sizeof(HT) != sizeof(float2);
    int kb = -32;
    unsigned live = 0;
    auto next_k = [&](int k) {
        if constexpr (kAhead) {
            while (live == 0) {
                kb += 32;
                if (kb >= m) return m;
                const int i = kb + lane;
                live = __ballot_sync(0xffffffffu, i < m && box[i].nr > 0);
            }
            k = kb + __ffs(live) - 1;
            live &= live - 1;
        } else {
            while (k < kend && box[k].nr == 0) ++k;
        }
        return k;
    };
    int k = next_k(0), fs = 0;
    float sk = 1.f;
    if (k < kend) {
        const Box bx = box[k];
        fs = col_frame<NF>(bx).s;
        if constexpr (kAhead) sk = hscale_of<HT>(hscale, k);
        frame_load<NY, ROWS, NT>(tile, Zb + k * z_kstride, bx, col_frame<NF>(bx), NXh, col0);
        if (lane == 0 && cv) bulk_prefetch_l2(hcol + k * hstride, NF * sizeof(HT));
    }
    while (k < kend) {
        const float2* twk = col_table<NF, PAR>(tab, 0, kAhead ? fs : col_frame<NF>(box[k]).s, par);
        const int kn = next_k(k + 1);
        Box bn;
        float skn = 1.f;
        if constexpr (kAhead) {
            bn = box[kn < kend ? kn : k];
            skn = hscale_of<HT>(hscale, kn < kend ? kn : k);
        }
        cp_async_wait_all();
        __syncthreads();   // the term's rows have landed
        float2 v[QN];
        if constexpr (!kAhead) sk = hscale_of<HT>(hscale, k);
        const float2* tb = tile + 4 * lane + sw;
        const float2 wls = cscale(wl, sk);
#pragma unroll
        for (int q = 0; q < ROWS / 32; ++q) {
            float2 x = tb[128 * q];
            if (PAR == 2 && par) x = cmul(cmul(x, wls), w64(q));   // W2048^i of the odd half
            else if (sizeof(HT) != sizeof(float2)) x = cscale(x, sk);
            v[q] = x;
        }
        __syncthreads();   // every warp has read its rows: the next term's may come
        if (kn < kend) {
            if constexpr (!kAhead) bn = box[kn];
            frame_load<NY, ROWS, NT>(tile, Zb + kn * z_kstride, bn, col_frame<NF>(bn), NXh, col0);
            if (lane == 0 && cv) bulk_prefetch_l2(hcol + kn * hstride, NF * sizeof(HT));
        }
        const bool bulk = !dcn && cv && !failed;
        auto hook = [&] {
            if (bulk && lane == 0) bulk_load(tr, hcol + k * hstride, NF * sizeof(HT), bar, skip_copy);
        };
        warp_fft_phased<NF, false, HALF, false, decltype(hook)>(v, tr, twk, hook);
        if (bulk) {
            if (!mbar_wait(bar, parity, wait_limit)) {
                failed = true;
                if (lane == 0) atomicOr(status, kStatusTimeout);
                // a copy may still be in flight into the tile: wait for it once more
                // (bounded); no further copies are issued, the products are skipped
                mbar_wait(bar, parity, wait_limit);
            }
            parity ^= 1;
        }
        if (dcn) {
            const HT* h0 = hcol + k * hstride;
            const HT* hn = hN + ((long long)k * PAR + par) * NF;
            __syncwarp();
#pragma unroll
            for (int mm = 0; mm < QN; ++mm) tr[lane + 32 * mm] = v[mm];
            __syncwarp();
#pragma unroll
            for (int qq = 0; qq < NQ; ++qq)
                tm_update8(t_acc, qq, [&](int mm, float2 a) {
                    const int fr = lane + 32 * mm;
                    float2 x, y;
                    split_dc_nyq(v[mm], half_partner<NF>(tr, fr, par), x, y);
                    a = cfma(ldh(&h0[fr], 1.f), x, a);
                    const float2 s = cmul(ldh(&hn[fr], 1.f), y);
                    a.x -= s.y;
                    a.y += s.x;
                    return a;
                });
            tm_wait_st();
            __syncwarp();
        } else if (cv && !failed) {
            const HT* th = reinterpret_cast<const HT*>(tr);
#pragma unroll
            for (int qq = 0; qq < NQ; ++qq)
                tm_update8(t_acc, qq, [&](int mm, float2 a) { return cfma(lds_h(&th[lane + 32 * mm], 1.f), v[mm], a); });
            tm_wait_st();
        }
        k = kn;
        if constexpr (kAhead) {
            fs = col_frame<NF>(bn).s;
            sk = skn;
        }
    }
    float2 acc[QN];
    tm_loadq<QN>(t_acc, acc);
    warp_fft<NF, true, kTmSplit, NoHook, true>(acc, tr, tw);
    if constexpr (PAR == 2) {
        if (par) {
#pragma unroll
            for (int q = 0; q < QN; ++q) acc[q] = cmulc(cmulc(acc[q], wl), w64(q));
        }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < QN; ++q) tr[(lane + 32 * q + 4 * cl) & (NF - 1)] = acc[q];
    __syncthreads();
    store_halves<NF, PAR, NT>(A + b * a_bstride, smem, 0, NY, NXh, col0, 1.f);
    tm_end(&tm_slot, kc_tm_cols<NF, PAR>());
}

// G1b + G2.  Grid (batch, ceil(NXh / 4), split), 128 PAR threads,
// kc_smem<NF, PAR>(0) bytes.  WHOLE: the inverse transforms give the whole column (not
// HALF), for boxes that no frame holds and for full (every row of Q: the window gradient).  split:
// CTA z of a column tile takes its share of the terms and forms the FFT of V itself.
template <int NF, int PAR, bool WHOLE, bool HALF, typename HT>
__global__ void __launch_bounds__(kCCols * PAR * 32, (kc_min_ctas<NF, PAR>()))
kc_cols_adj(const float2* __restrict__ V, long long v_bstride, const HT* __restrict__ hhT, const HT* __restrict__ hN,
            const float* __restrict__ hscale, int m, const Box* __restrict__ box, int NXh, float2* __restrict__ Q,
            long long q_bstride, long long q_kstride, const float2* __restrict__ tw,
            const float2* __restrict__ tab, const float2* __restrict__ tw2048l, int full) {
    constexpr int QS = HALF ? NF / 64 : NF / 32;   // output values a lane needs
    constexpr int NY = NF * PAR, QN = NF / 32, NQ = QN / 8, NT = kCCols * PAR * 32;
    extern __shared__ __align__(16) float2 smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cl = warp / PAR, par = warp % PAR;
    float2* tr = smem + warp * warp_tile(NF);
    __shared__ unsigned tm_slot;
    const int b = blockIdx.x;
    const int col0 = blockIdx.y * kCCols, col = col0 + cl;
    const bool cv = col < NXh;
    const bool dcn = col == 0;
    if (warp == 0) tm_alloc(&tm_slot, kc_tm_cols<NF, PAR>());
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const unsigned t_hold = tm_slot + ((unsigned)(32 * (warp & 3)) << 16) + (warp >> 2) * 2 * QN;
    const float2 wl = PAR == 2 ? __ldg(&tw2048l[lane]) : make_float2(1.f, 0.f);
    const HT* hcol = hhT + ((long long)(cv ? col : 0) * PAR + par) * NF;
    const long long hstride = (long long)NXh * PAR * NF;
    const int kend = share_beg(m, blockIdx.z + 1, gridDim.z);
    auto next_k = [&](int k) {
        while (!full && k < kend && box[k].nr == 0) ++k;
        return k;
    };
    int k = next_k(share_beg(m, blockIdx.z, gridDim.z));
    if (lane == 0 && k < kend && cv) bulk_prefetch_l2(hcol + k * hstride, NF * sizeof(HT));
    {
        // the four columns of V through the transpose tiles, [NY][4] swizzled
        for (int e = threadIdx.x; e < NY * kCCols; e += NT) {
            const int i = e >> 2, c = e & 3;
            const bool ok = col0 + c < NXh;
            cp_async8(smem + tix(i, c), V + b * v_bstride + (long long)i * NXh + (ok ? col0 + c : 0), ok);
        }
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        float2 v[QN];
        const float2* tb = smem + 4 * lane + tix_sw(lane, cl);
#pragma unroll
        for (int q = 0; q < QN; ++q) {
            v[q] = tb[128 * q];
            if constexpr (PAR == 2) {
                const float2 hi = tb[128 * q + 4 * NF];
                v[q] = par ? cmul(cmul(csub(v[q], hi), wl), w64(q)) : cadd(v[q], hi);
            }
        }
        __syncthreads();   // every warp has read its column: the transpose tiles are free
        warp_fft<NF, false, kTmSplit, NoHook, true>(v, tr, tw);
        tm_storeq<QN>(t_hold, v);
        tm_wait_st();
    }
    while (k < kend) {
        const int kn = next_k(k + 1);
        if (lane == 0 && kn < kend && cv) bulk_prefetch_l2(hcol + kn * hstride, NF * sizeof(HT));
        const float sk = hscale_of<HT>(hscale, k);
        const HT* hk = hcol + k * hstride;
        float2 p[QN];
        if (dcn) {
            tm_loadq<QN>(t_hold, p);
            const HT* hn = hN + ((long long)k * PAR + par) * NF;
            __syncwarp();
#pragma unroll
            for (int mm = 0; mm < QN; ++mm) tr[lane + 32 * mm] = p[mm];
            __syncwarp();
#pragma unroll
            for (int mm = 0; mm < QN; ++mm) {
                const int fr = lane + 32 * mm;
                float2 x, y;
                split_dc_nyq(p[mm], half_partner<NF>(tr, fr, par), x, y);
                float2 r = cmulc(x, ldh(&hk[fr], 1.f));
                const float2 s = cmulc(y, ldh(&hn[fr], 1.f));
                r.x -= s.y;
                r.y += s.x;
                p[mm] = r;
            }
            __syncwarp();
        } else {
#pragma unroll
            for (int mm = 0; mm < QN; ++mm) p[mm] = ldh(&hk[lane + 32 * mm], 1.f);
#pragma unroll
            for (int qq = 0; qq < NQ; ++qq) {
                float2 x[8];
                tm_load8c(t_hold + 16 * qq, x);
#pragma unroll
                for (int j = 0; j < 8; ++j) p[8 * qq + j] = cmulc(x[j], p[8 * qq + j]);
            }
        }
        // frame rows lane + 32 q of the inverse (WHOLE: rows of the column)
        const Box bx = box[k];
        const CFrame f = col_frame<NF>(bx);
        if constexpr (WHOLE) warp_fft<NF, true, kTmSplit, NoHook, true>(p, tr, tw);
        else warp_fft_phased<NF, true, false, HALF>(p, tr, col_table<NF, PAR>(tab, 1, f.s, par));
        if constexpr (PAR == 2) {
            if (par) {
#pragma unroll
                for (int q = 0; q < QS; ++q) p[q] = cmulc(cmulc(p[q], wl), w64(q));
            }
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < QS; ++q) tr[(lane + 32 * q + 4 * cl) & (NF - 1)] = p[q];
        __syncthreads();
        store_halves<NF, PAR, NT>(Q + b * q_bstride + k * q_kstride, smem,
                                  full ? 0 : WHOLE ? bx.r0 : f.a, full ? NY : bx.nr, NXh, col0, sk);
        __syncthreads();   // the transpose tiles are free again
        k = kn;
    }
    tm_end(&tm_slot, kc_tm_cols<NF, PAR>());
}

}  // namespace pce
