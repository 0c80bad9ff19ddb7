// Resampling and weighting (Sec. III A), several templates per block: FP32 storage, and BF16
// storage of segments too long for one staged window.
//
// A block owns one (segment, detector) and a group of templates.  The templates of a batch
// see the same detector samples to within a few of them, so the block stages, once for the
// group, the window of x and of the antenna functions at the integer samples and the inverse
// noise variance of each sample's block (0 in gaps); a warp then walks one template's
// 128-sample knot intervals, four source samples a lane per knot record.  Per sample there
// remain the cubic between knots, the taps from shared memory, the phase and two
// interpolations: about 170 instructions, where a block per template spent about 410 on them,
// half of that on integer divisions, table look-ups and record loads that the group shares now.
//
// Windowed sinc: with g_k = (-1)^k w_k / (delta^2 - k^2) the taps j* -+ k add
//   s g_k [delta (x_-k + x_k) + k (x_k - x_-k)],  s = sin(pi delta) / pi,
// (the coefficients s (-1)^k w_k / (delta +- k) over a common denominator): one reciprocal,
// one product and four multiply-adds per pair of taps.
//
// Weights at t = floor(t) + u: a and b linear between integer samples, which is their table's
// linear interpolation (its nodes lie on integer samples); the noise block is floor(t)'s, since
// block boundaries lie on integer samples too.
//
// BF16 storage: the values are rounded twice on their way (here and when a long segment is
// folded), so they keep the arithmetic of resample_kernel (stages.cu) to the bit -- taps one by
// one, weights from the tables -- and only x is staged.  120-day band, ten-hour segments:
// 173 us per template of 16, 315 with a block per template that read its 17 taps from L1.
//
// What bounds it: instruction issue (72 % of the slots; shared-memory wavefronts 61 %; sharing the
// taps of two neighbouring samples by 16-byte loads took half of those away and no time).  FP32,
// 120-day band: 98 us per template of 72, 176 with a block per template.
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace cc {

namespace {

constexpr int RG_MAX_WARPS = 12;      // 56 registers a thread at three blocks per SM (40 spill)
constexpr int RG_TILE = 3616;         // samples of a staged tile: three blocks of 73 KB per SM
constexpr int RG_TILE_BF16 = 9024;    // x alone

// 1 / x in one MUFU for x far from denormals
__device__ __forceinline__ float rcp_normal(float x) {
    float g;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(g) : "f"(x));
    return g;
}

template <int DT>
struct SincTab {
    float ca[DT > 0 ? DT : 1], cb[DT > 0 ? DT : 1];   // g_k = 1 / (ca[k-1] delta^2 + cb[k-1])
};

template <int DT>
__device__ __forceinline__ float2 sinc_pairs(const SincTab<DT>& tb, const float2* __restrict__ xc, float delta) {
    const float sc = sinc_pi(delta), s = delta * sc, d2 = delta * delta;
    float2 E = make_float2(0.f, 0.f), O = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 1; k <= DT; ++k) {
        // the argument is between 0.75 and 13 k^2 in size
        const float g = rcp_normal(fmaf(d2, tb.ca[k - 1], tb.cb[k - 1]));
        const float h = g * (float)k;
        const float2 xm = xc[-k], xp = xc[k];
        const float2 e = cadd(xp, xm), o = csub(xp, xm);
        E.x = fmaf(g, e.x, E.x);
        E.y = fmaf(g, e.y, E.y);
        O.x = fmaf(h, o.x, O.x);
        O.y = fmaf(h, o.y, O.y);
    }
    // (a sample that falls on one of the series is that one, whatever lies beside it: not 0 x inf)
    const float2 x0 = xc[0];
    return delta == 0.f ? x0 : make_float2(fmaf(s, fmaf(delta, E.x, O.x), sc * x0.x), fmaf(s, fmaf(delta, E.y, O.y), sc * x0.y));
}

// sinc_taps (common.cuh) with the half width at compile time for DT > 0, value for value: its
// quotients s / (delta - n) are s times the approximate reciprocal, as PTX defines the
// approximate division, here without that one's care for denormal divisors (delta is zero, which
// takes another branch, or a multiple of 2^-25).
template <int DT>
__device__ __forceinline__ float2 sinc_taps_each(const DevParams& p, const float2* __restrict__ xp, float delta) {
    if constexpr (DT == 0) return sinc_taps(p, xp, delta);
    const float s = delta * sinc_pi(delta);
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int n = 0; n <= 2 * DT; ++n) {
        const float q = s * rcp_normal(delta - (float)(n - DT));
        const float c = p.ham[n] * (((n - DT) & 1) ? -q : q);
        const float2 xv = xp[n];
        acc.x = fmaf(c, xv.x, acc.x);
        acc.y = fmaf(c, xv.y, acc.y);
    }
    return acc;
}

__device__ __forceinline__ void put_sample(float2* p, int r, float2 v) { p[r] = v; }
__device__ __forceinline__ void put_sample(__nv_bfloat162* p, int r, float2 v) { p[r] = __float22bfloat162_rn(v); }

// grid: x = segment K, y = detector X, z = template group.  blockDim = 32 tg wpt: wpt warps
// per template.  Outputs as resample_kernel's (stages.cu); kn: the knot records of the
// pre-pass.
template <int DT, bool LEARNED, bool BF16>
__global__ void __launch_bounds__(32 * RG_MAX_WARPS, 3)
resample_group_kernel(void* __restrict__ ab, float4* __restrict__ norm, const KnotRec* __restrict__ kn, int64_t nkn,
                      int n_t, int tg, int wpt, int tile, int cap, int write_inactive, uint8_t* __restrict__ act,
                      int t_pad, SincTab<DT> tb, DevParams p) {
    extern __shared__ __align__(16) float2 sm[];
    float2* xs = sm;                     // [cap] samples of x, zero outside the series
    float2* abs_ = sm + cap;             // FP32: [cap] (a, b) at the integer samples
    float* inv = (float*)(sm + 2 * cap); // FP32: [cap] 1 / sigma^2, 0 in gaps
    __shared__ int s_lo[RG_MAX_WARPS], s_hi[RG_MAX_WARPS], s_on[RG_MAX_WARPS];
    __shared__ float red[RG_MAX_WARPS][3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
    const int tl = warp / wpt, sub = warp - tl * wpt;
    const int K = blockIdx.x, X = blockIdx.y;
    const int t0 = blockIdx.z * tg, t = t0 + tl;
    const int N_s = (int)p.N_s, seg0 = K * N_s;
    const int Dm = LEARNED ? 4 : (DT > 0 ? DT : p.D);   // the taps lie in [j* - Dm, j* + Dm]
    const float2* __restrict__ x = p.x[X];
    const KnotRec* __restrict__ knX = kn + ((size_t)t * p.Q + X) * nkn;

    // detector times of the segment lie within [seg0 - max d - 2, seg1 + 2 - min d] (d from the
    // segment's knots; the cubic between knots stays within 1e-4 samples of them); weight only
    // if a noise block there is locked
    bool on = false;
    if (t < n_t) {
        const int ka = seg0 >> 7, kb = min(((seg0 + N_s - 1) >> 7) + 1, (int)nkn - 1);
        float dmin = 3.0e38f, dmax = -3.0e38f;
        for (int k = ka + lane; k <= kb; k += 32) {
            const KnotRec kr = load_knot(knX + k);
            const float d = (float)kr.N + kr.f;
            dmin = fminf(dmin, d);
            dmax = fmaxf(dmax, d);
        }
        for (int o = 16; o > 0; o >>= 1) {
            dmin = fminf(dmin, __shfl_xor_sync(0xffffffffu, dmin, o));
            dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
        }
        const int lo = seg0 - (int)ceilf(dmax) - 2, hi = seg0 + N_s - (int)floorf(dmin) + 2;
        const int ns = (int)p.n_sig[X];
        const int blo = max(floor_div32(lo, p.nsft), 0), bhi = min(floor_div32(hi, p.nsft), ns - 1);
        on = blo <= bhi && __ldg(p.lockc[X] + bhi + 1) - __ldg(p.lockc[X] + blo) > 0;
        if (lane == 0 && sub == 0) {
            // stencil centres lie in [lo + 1, hi - 1]; taps reach Dm + 1 beyond
            s_lo[tl] = lo - Dm - 2;
            s_hi[tl] = hi + Dm + 2;
        }
    }
    if (lane == 0 && sub == 0) {
        s_on[tl] = on;
        if (t < n_t && act) act[((size_t)X * p.M + K) * t_pad + t] = on;
    }
    __syncthreads();
    int lo = 0x7fffffff, hi = -0x7fffffff;
    for (int i = 0; i < tg; ++i)
        if (s_on[i]) {
            lo = min(lo, s_lo[i]);
            hi = max(hi, s_hi[i]);
        }
    const size_t sa = t < n_t ? (((size_t)t * p.Q + X) * 2) * p.N_tau : 0;
    using E = std::conditional_t<BF16, __nv_bfloat162, float2>;
    E* __restrict__ pa = (E*)ab + sa;
    E* __restrict__ pb = pa + p.N_tau;
    if (t < n_t && !on) {
        if (lane == 0 && sub == 0) norm[((size_t)t * p.Q + X) * p.M + K] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (write_inactive)
            for (int r = seg0 + sub * 32 + lane; r < seg0 + N_s; r += 32 * wpt) {
                put_sample(pa, r, make_float2(0.f, 0.f));
                put_sample(pb, r, make_float2(0.f, 0.f));
            }
    }
    if (hi < lo) return;   // no template of the group has weight here

    float A = 0.f, B = 0.f, Cn = 0.f;
    for (int ta = 0; ta < N_s; ta += tile) {
        const int tb_ = min(N_s, ta + tile);
        const int w0 = lo + ta, nw = min(hi - (N_s - tb_) - w0, cap);
        if (ta > 0) __syncthreads();
        {
            const int N = (int)p.N_t, nab = (int)p.n_ab[X], ns = (int)p.n_sig[X];
            const float step_inv = 1.0f / (float)p.n_ab_step;
            for (int i = tid; i < nw; i += nthr) {
                const int jj = w0 + i;
                xs[i] = (jj >= 0 && jj < N) ? __ldg(x + jj) : make_float2(0.f, 0.f);
                if constexpr (BF16) continue;
                const int ja = jj - (int)p.ab_j0;
                const int ia = floor_div_magic(ja, p.n_ab_step, p.ab_m, p.ab_s);
                const int ic = ia < 0 ? 0 : (ia > nab - 2 ? nab - 2 : ia);
                const float fr = (float)(ja - ic * p.n_ab_step) * step_inv;
                const float a0 = __ldg(p.atab[X] + ic), a1 = __ldg(p.atab[X] + ic + 1);
                const float b0 = __ldg(p.btab[X] + ic), b1 = __ldg(p.btab[X] + ic + 1);
                abs_[i] = make_float2(fmaf(fr, a1 - a0, a0), fmaf(fr, b1 - b0, b0));
                const int blk = floor_div_magic(jj, p.nsft, p.nsft_m, p.nsft_s);
                inv[i] = (blk >= 0 && blk < ns) ? __ldg(p.sigw[X] + blk).y : 0.f;
            }
        }
        __syncthreads();
        if (!on) continue;
        const int ra = seg0 + ta, rb = seg0 + tb_;
        const unsigned lim = nw > 2 * Dm + 1 ? (unsigned)(nw - 2 * Dm - 1) : 0u;
        for (int k = (ra >> 7) + sub; k <= (rb - 1) >> 7; k += wpt) {
            const KnotRec kr = load_knot(knX + k);
#pragma unroll 1
            for (int i = 0; i < KNOT; i += 32) {
                const int r0 = k * KNOT + i;
                if (r0 + 31 < ra || r0 >= rb) continue;
                const int r = r0 + lane;
                const SampleTiming st = sample_timing(p, kr, r, k * KNOT);
                const bool neg = st.delta < 0.f;
                const float u = neg ? st.delta + 1.0f : st.delta;
                const int ci = st.jstar - w0;
                float2 va = make_float2(0.f, 0.f), vb = va;
                if ((unsigned)(ci - Dm) < lim) {
                    const int fi = neg ? ci - 1 : ci;
                    SampleWeights w{};
                    if constexpr (BF16) w = sample_weights(p, X, st.jstar, st.delta);
                    else w.s2 = inv[fi];
                    if (w.s2 > 0.f && r >= ra && r < rb) {
                        float2 xv;
                        if constexpr (LEARNED) {
                            float c[LEARNED_TAPS];
                            learned_coeffs(p, u, c);
                            const float2* xp = xs + fi - LEARNED_TAP_OFFSET;
                            xv = make_float2(0.f, 0.f);
#pragma unroll
                            for (int n = 0; n < LEARNED_TAPS; ++n) {
                                xv.x = fmaf(c[n], xp[n].x, xv.x);
                                xv.y = fmaf(c[n], xp[n].y, xv.y);
                            }
                        } else if constexpr (BF16) {
                            xv = st.delta == 0.0f ? xs[ci] : sinc_taps_each<DT>(p, xs + ci - Dm, st.delta);
                        } else if constexpr (DT > 0) {
                            xv = sinc_pairs<DT>(tb, xs + ci, st.delta);
                        } else {
                            xv = st.delta == 0.0f ? xs[ci] : sinc_taps(p, xs + ci - Dm, st.delta);
                        }
                        const float2 xr = cmul(xv, phase_rot(st.psi));
                        if constexpr (BF16) {
                            va = cscale(xr, w.alpha);
                            vb = cscale(xr, w.beta);
                            A = fmaf(w.alpha * w.alpha, w.s2, A);
                            B = fmaf(w.beta * w.beta, w.s2, B);
                            Cn = fmaf(w.alpha * w.beta, w.s2, Cn);
                        } else {
                            const float2 f0 = abs_[fi], f1 = abs_[fi + 1];
                            const float a = fmaf(u, f1.x - f0.x, f0.x), b = fmaf(u, f1.y - f0.y, f0.y);
                            const float al = a * w.s2, be = b * w.s2;   // (w.s2: 1 / sigma^2)
                            va = cscale(xr, al);
                            vb = cscale(xr, be);
                            A = fmaf(a, al, A);
                            B = fmaf(b, be, B);
                            Cn = fmaf(a, be, Cn);
                        }
                    }
                } else if (r >= ra && r < rb) {   // outside the staged window: straight from the tables
                    const float2 xr = cmul(interp_sample(p, x, st.jstar, st.delta), phase_rot(st.psi));
                    const SampleWeights w = sample_weights(p, X, st.jstar, st.delta);
                    va = cscale(xr, w.alpha);
                    vb = cscale(xr, w.beta);
                    A = fmaf(w.alpha * w.alpha, w.s2, A);
                    B = fmaf(w.beta * w.beta, w.s2, B);
                    Cn = fmaf(w.alpha * w.beta, w.s2, Cn);
                }
                if (r >= ra && r < rb) {
                    put_sample(pa, r, va);
                    put_sample(pb, r, vb);
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        A += __shfl_xor_sync(0xffffffffu, A, o);
        B += __shfl_xor_sync(0xffffffffu, B, o);
        Cn += __shfl_xor_sync(0xffffffffu, Cn, o);
    }
    if (lane == 0) {
        red[warp][0] = A;
        red[warp][1] = B;
        red[warp][2] = Cn;
    }
    __syncthreads();
    if (on && lane == 0 && sub == 0) {
        for (int i = 1; i < wpt; ++i) {
            A += red[warp + i][0];
            B += red[warp + i][1];
            Cn += red[warp + i][2];
        }
        norm[((size_t)t * p.Q + X) * p.M + K] = make_float4(A, B, Cn, 0.f);
    }
}

template <int DT, bool LEARNED, bool BF16>
cudaError_t launch_group(dim3 grid, int threads, size_t smem, cudaStream_t st, void* ab, float4* norm, const KnotRec* kn,
                         int64_t nkn, int n_t, int tg, int wpt, int tile, int cap, int write_inactive, uint8_t* act,
                         int t_pad, const DevParams& p) {
    SincTab<DT> tb;
    for (int k = 1; k <= (DT > 0 ? DT : 1); ++k) {
        const double ca = (k & 1 ? -1.0 : 1.0) / (double)p.ham[(DT > 0 ? DT : 1) - k];
        tb.ca[k - 1] = (float)ca;
        tb.cb[k - 1] = (float)(-(double)(k * k) * ca);
    }
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(resample_group_kernel<DT, LEARNED, BF16>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    resample_group_kernel<DT, LEARNED, BF16><<<grid, threads, smem, st>>>(ab, norm, kn, nkn, n_t, tg, wpt, tile, cap,
                                                                    write_inactive, act, t_pad, tb, p);
    return cudaGetLastError();
}

}  // namespace

template <bool BF16>
static cudaError_t launch_group_any(const DevParams& p, dim3 grid, int threads, size_t smem, cudaStream_t st, void* ab,
                                    float4* norm, const KnotRec* kn, int64_t nkn, int n_t, int tg, int wpt, int tile, int cap,
                                    int write_inactive, uint8_t* act, int t_pad) {
    auto go = [&](auto launch) {
        return launch(grid, threads, smem, st, ab, norm, kn, nkn, n_t, tg, wpt, tile, cap, write_inactive, act, t_pad, p);
    };
    if (p.interp == CC_INTERP_LEARNED) return go(launch_group<0, true, BF16>);
    return p.D == 8 ? go(launch_group<8, false, BF16>) : p.D == 16 ? go(launch_group<16, false, BF16>)
                                                                   : go(launch_group<0, false, BF16>);
}

// a_r, b_r (the storage type) and segment norms of n_t templates with the knot records kn; act
// (nullable) as in resample_kernel.
cc_status launch_resample_group(cc_plan* plan, int64_t n_t, void* ab, float* norm, cudaStream_t st, const KnotRec* kn,
                                int64_t nkn, int write_inactive, uint8_t* act, int t_pad) {
    const DevParams& p = plan->dp;
    const bool bf16 = p.store == CC_STORE_BF16;
    // warps per block by the segment's knot intervals; templates per block: up to eight (the
    // window is staged once for them), fewer while there are less than two blocks per SM
    const int warps = p.N_s <= 512 ? 4 : p.N_s <= 1536 ? 8 : RG_MAX_WARPS;
    static const int groups[] = {12, 6, 3, 2, 1, 0}, groups8[] = {8, 4, 2, 1, 0};
    const int* gp = warps == 12 ? groups : warps == 8 ? groups8 : groups8 + 1;
    if (warps == 12) ++gp;
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    while (gp[1] && (gp[0] >= 2 * n_t || p.M * p.Q * ((n_t + gp[0] - 1) / gp[0]) < 2 * sms)) ++gp;
    const int tg = gp[0];
    const int64_t most = bf16 ? RG_TILE_BF16 : RG_TILE, tiles = (p.N_s + most - 1) / most;
    const int tile = (int)(((p.N_s + tiles - 1) / tiles + 31) & ~(int64_t)31);
    // the window of a tile: its samples, the drift of the delay over the segment
    // (|d'| < 2.5e-4 for the Earth and a binary orbit), the taps, and slack for the templates
    // of a group (a wider spread of them takes the samples it misses straight from the tables)
    // (at most what a block's shared memory holds: segments of millions of samples)
    const size_t elem = bf16 ? 8 : 20;
    const int cap = (int)std::min<int64_t>(std::min<int64_t>(tile, p.N_s) + p.N_s / 512 + 2 * std::max(p.D, 4) + 48,
                                           (int64_t)(220 * 1024 / elem));
    const size_t smem = (size_t)cap * elem;
    const int64_t step = (int64_t)65535 * tg;
    for (int64_t t0 = 0; t0 < n_t; t0 += step) {
        const int64_t nt = std::min(step, n_t - t0);
        const dim3 grid((unsigned)p.M, (unsigned)p.Q, (unsigned)((nt + tg - 1) / tg));
        void* a = (char*)ab + (size_t)t0 * p.Q * 2 * p.N_tau * (bf16 ? 4 : 8);
        float4* nm = (float4*)norm + (size_t)t0 * p.Q * p.M;
        const KnotRec* k = kn + (size_t)t0 * p.Q * nkn;
        uint8_t* ac = act ? act + t0 : nullptr;
        auto launch = bf16 ? launch_group_any<true> : launch_group_any<false>;
        const cudaError_t e = launch(p, grid, 32 * warps, smem, st, a, nm, k, nkn, (int)nt, tg, warps / tg, tile, cap,
                                     write_inactive, ac, t_pad);
        count_launch();
        if (e != cudaSuccess) return cuda_fail(e, "resample launch");
    }
    return CC_OK;
}

}  // namespace cc
