// Fold of a segment longer than 4096 samples onto the 4096 positions of the lag grid's coset
// transforms (Sec. III B 4 with a segment longer than the on-chip transform).  The grid has
// G = C x 4096 frequencies with C = 2 F cosets for F = ceil(N_s / 4096) folds (G >= 2 N_s);
// coset c takes the 4096-point transform of Z_c[p] W_G^(c p) with
//   Z_c[p] = sum_f x[p + 4096 f] W_C^(c f),
// a C-point DFT over the fold index, done here once per (template, detector, weight, segment)
// for every c and stored in FP32; corr_kernel streams the rows.
//
// C = 2 F splits into two F-point DFTs: c = 2 u takes a_f, c = 2 u + 1 takes a_f W_C^f.  Each
// F-point DFT combines a_f +- a_(F-f) (half the products of the direct sum); its constants
// are kernel parameters, read as immediate operands.  Bound by the write of Z (2 x the bytes
// of the segment) for F up to about ten: 150 us per template of the 120-day band at a ten-hour lag
// (F = 9, 0.93 GB read and written, 6.2 TB/s); the whole search 0.74 ms per template in FP32, 6.4
// when every coset read and twiddled the whole segment.
#include <algorithm>

#include "corr.cuh"

namespace cc {

namespace {

constexpr int FOLD_L = 4096;
constexpr int FOLD_MAX_F = 16;

struct FoldTab {
    float2 w[2 * FOLD_MAX_F];   // exp(-2 pi i n / (2 F))
};

// X_u = sum_f a_f W_F^(u f), u < F
template <int F>
__device__ __forceinline__ void dft_f(const float2 (&a)[F], float2 (&X)[F], const FoldTab& tb) {
    constexpr int H = (F - 1) / 2;
    float2 s[H + 1], d[H + 1], sum = a[0];
#pragma unroll
    for (int f = 1; f <= H; ++f) {
        s[f] = cadd(a[f], a[F - f]);
        d[f] = csub(a[f], a[F - f]);
        sum = cadd(sum, s[f]);
    }
    X[0] = F % 2 == 0 ? cadd(sum, a[F / 2]) : sum;
    if constexpr (F % 2 == 0) {
        float2 alt = (F / 2) % 2 ? csub(a[0], a[F / 2]) : cadd(a[0], a[F / 2]);
#pragma unroll
        for (int f = 1; f <= H; ++f) alt = f % 2 ? csub(alt, s[f]) : cadd(alt, s[f]);
        X[F / 2] = alt;
    }
#pragma unroll
    for (int u = 1; u <= H; ++u) {
        float2 re = a[0], im = make_float2(0.f, 0.f);
        if (F % 2 == 0) re = u % 2 ? csub(a[0], a[F / 2]) : cadd(a[0], a[F / 2]);
#pragma unroll
        for (int f = 1; f <= H; ++f) {
            const float2 w = tb.w[2 * ((u * f) % F)];   // cos, -sin of 2 pi u f / F
            re.x = fmaf(w.x, s[f].x, re.x);
            re.y = fmaf(w.x, s[f].y, re.y);
            im.x = fmaf(w.y, d[f].x, im.x);
            im.y = fmaf(w.y, d[f].y, im.y);
        }
        X[u] = make_float2(re.x - im.y, re.y + im.x);   // re + i im
        X[F - u] = make_float2(re.x + im.y, re.y - im.x);
    }
}

template <bool BF16>
__device__ __forceinline__ float2 load_row(const void* ab, size_t i) {
    if constexpr (BF16) return __bfloat1622float2(((const __nv_bfloat162*)ab)[i]);
    else return __ldg((const float2*)ab + i);
}

// grid: x = segment K, y = detector X * 2 + weight w, z = template of the batch.
// ab: [n_t][Q][2][N_tau] in the storage type, z: [n_t][Q][2][M][C][4096], act as in
// CorrArgs: a row without weight is never read, and not written.
template <int F, bool BF16>
__global__ void __launch_bounds__(CORR_THREADS)
fold_kernel(const void* __restrict__ ab, const uint8_t* __restrict__ act, int t_pad, int Q, int64_t N_s, int64_t N_tau,
            float2* __restrict__ z, FoldTab tb) {
    constexpr int C = 2 * F;
    const int64_t K = blockIdx.x, M = gridDim.x;
    const int X = blockIdx.y >> 1, w = blockIdx.y & 1;
    const int64_t t = blockIdx.z;
    if (!__ldg(act + ((size_t)X * M + K) * t_pad + t)) return;
    const size_t row = (((size_t)t * Q + X) * 2 + w) * N_tau + (size_t)(K * N_s);
    const size_t zrow = ((((size_t)t * Q + X) * 2 + w) * M + K) * C * FOLD_L;
    for (int pp = threadIdx.x; pp < FOLD_L; pp += CORR_THREADS) {
        float2 a[F], x[F];
#pragma unroll
        for (int f = 0; f < F; ++f) {
            const int64_t s = pp + (int64_t)f * FOLD_L;
            a[f] = f < F - 1 || s < N_s ? load_row<BF16>(ab, row + s) : make_float2(0.f, 0.f);
        }
        auto put = [&](int c, float2 v) { z[zrow + (size_t)c * FOLD_L + pp] = v; };
        dft_f<F>(a, x, tb);
#pragma unroll
        for (int u = 0; u < F; ++u) put(2 * u, x[u]);
#pragma unroll
        for (int f = 1; f < F; ++f) a[f] = cmul(a[f], tb.w[f]);
        dft_f<F>(a, x, tb);
#pragma unroll
        for (int u = 0; u < F; ++u) put(2 * u + 1, x[u]);
    }
}

// Any number of folds (segments longer than 16 x 4096 samples): the direct sum.
template <bool BF16>
__global__ void __launch_bounds__(CORR_THREADS)
fold_any_kernel(const void* __restrict__ ab, const uint8_t* __restrict__ act, int t_pad, int Q, int64_t N_s,
                int64_t N_tau, float2* __restrict__ z, int F) {
    const int C = 2 * F;
    const int64_t K = blockIdx.x, M = gridDim.x;
    const int X = blockIdx.y >> 1, w = blockIdx.y & 1;
    const int64_t t = blockIdx.z;
    if (!__ldg(act + ((size_t)X * M + K) * t_pad + t)) return;
    const size_t row = (((size_t)t * Q + X) * 2 + w) * N_tau + (size_t)(K * N_s);
    const size_t zrow = ((((size_t)t * Q + X) * 2 + w) * M + K) * C * FOLD_L;
    for (int c = 0; c < C; ++c)
        for (int pp = threadIdx.x; pp < FOLD_L; pp += CORR_THREADS) {
            float2 acc = make_float2(0.f, 0.f);
            for (int f = 0; f < F; ++f) {
                const int64_t s = pp + (int64_t)f * FOLD_L;
                if (s < N_s) acc = cadd(acc, cmul(load_row<BF16>(ab, row + s), unit_root((int64_t)c * f, C)));
            }
            z[zrow + (size_t)c * FOLD_L + pp] = acc;
        }
}

}  // namespace

int64_t fold_count(const cc_plan* plan) { return (plan->N_s + FOLD_L - 1) / FOLD_L; }

cc_status launch_fold(cc_plan* plan, int64_t n_t, const void* ab, const uint8_t* act, int t_pad, float2* z,
                      cudaStream_t st) {
    const int64_t F = fold_count(plan);
    if (n_t > 65535 || plan->M > 0x7fffffff) return fail(CC_ERR_UNSUPPORTED, "fold launch size");
    const dim3 grid((unsigned)plan->M, (unsigned)(2 * plan->Q), (unsigned)n_t);
    const bool bf16 = plan->cfg.store == CC_STORE_BF16;
    if (F > FOLD_MAX_F) {
        if (bf16)
            fold_any_kernel<true><<<grid, CORR_THREADS, 0, st>>>(ab, act, t_pad, plan->Q, plan->N_s, plan->N_tau, z, (int)F);
        else
            fold_any_kernel<false><<<grid, CORR_THREADS, 0, st>>>(ab, act, t_pad, plan->Q, plan->N_s, plan->N_tau, z, (int)F);
    } else {
        FoldTab tb;
        for (int64_t n = 0; n < 2 * F; ++n) {
            const double a = -M_PI * (double)n / (double)F;
            tb.w[n] = make_float2((float)cos(a), (float)sin(a));
        }
        switch (F) {
#define CC_FOLD(FV)                                                                                                     \
    case FV:                                                                                                            \
        if (bf16) fold_kernel<FV, true><<<grid, CORR_THREADS, 0, st>>>(ab, act, t_pad, plan->Q, plan->N_s, plan->N_tau, z, tb); \
        else fold_kernel<FV, false><<<grid, CORR_THREADS, 0, st>>>(ab, act, t_pad, plan->Q, plan->N_s, plan->N_tau, z, tb);     \
        break;
            CC_FOLD(2) CC_FOLD(3) CC_FOLD(4) CC_FOLD(5) CC_FOLD(6) CC_FOLD(7) CC_FOLD(8) CC_FOLD(9)
            CC_FOLD(10) CC_FOLD(11) CC_FOLD(12) CC_FOLD(13) CC_FOLD(14) CC_FOLD(15) CC_FOLD(16)
#undef CC_FOLD
            default: return fail(CC_ERR_UNSUPPORTED, "fold count");
        }
    }
    count_launch();
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? CC_OK : cuda_fail(e, "fold launch");
}

}  // namespace cc
