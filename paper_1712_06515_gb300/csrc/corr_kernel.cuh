// Spectra and pair products of the two-pass search on the lag grid.
//
// The pair sum rho_raw(f) = Re sum_P conj(F_K(f)) F_L(f) (Sec. III B 1, Eq.
// final-formatted-rho) is the Fourier transform of a correlation that lives on a bounded
// set of lags: a product of two N_s-sample segments has 2 N_s - 1 of them.  So the products
// need only be known at G >= 2 N_s - 1 equally spaced frequencies omega_j = 2 pi j / G;
// their sums over segments, an inverse transform to lags and one transform per template to
// the N_FFT-point output grid (corr.cu) give rho at every output bin, the same value as
// products taken bin by bin (an exact identity; the rounding differs).  Per segment that is
// a transform of G = 8192 points for N_s = 3600 instead of the N_FFT = 32768 output grid.
//
// With T_K(j) the transform of segment K from its own first sample on, S_K the sum over
// detectors, the kernel accumulates over segments, per template and weight,
//   A(j) = sum_K sum_(X<Y) Re(conj(T_YK) T_XK)   (|S_K|^2 with every ordered pair), real,
//   B(j) = sum_K conj(S_K) S_(K-1)     (R = 1), complex,
// each compensated at every segment, and left as two floats: the value and what it rounds off
// (the sums after it carry those, corr.cu; a line just outside the band leaves in rho what sums
// at the output bins leave there, five times that with plain runs of 16 segments).
//
// A CTA of 256 threads holds 4096 points, 16 per thread: T = 4096 / L transforms of L
// points, each one (template, weight) series (L = 4096: one).  G = L for N_s <= 2048
// (HALF: the upper half of the transform's input is zero); G = C L with cosets c (frequency
// j = C m + c, one work unit each) for longer segments, C = 2 up to 4096 samples, folded
// rows beyond that.
//
//   * persistent CTAs, two per SM, take units (series group, chunk of segments, coset) from
//     one counter; the cosets of a unit are neighbours, so their CTAs read the same rows
//     from L2.  A unit is computed by one CTA in a fixed order: repeated runs give the same
//     bits;
//   * the rows of the next (detector, segment) arrive by cp.async.bulk (TMA) on an mbarrier
//     under the current transform's later passes (16-byte rows; otherwise by 8- or 4-byte
//     cp.async);
//   * the running sums, their compensations and S_(K-1) -- 128 words per thread -- live in
//     tensor memory, 32 columns per group of four bins (8 without a lag), read and written by
//     tcgen05.ld/st once per segment: registers hold only the transform (16 points) and detector
//     0's spectrum (MULTI, three or four detectors: the sum of the earlier ones), so two CTAs of
//     128 registers fit an SM;
//   * twiddles as in the staged kernel: the coset factor of sample s = t + 256 r is split
//     between a factor per r (first pass) and the table of the second and the powers of the
//     last pass.  The coset's tables (10 KB) are kept in shared memory: read through L1, whose
//     share beside 2 x 110 KB is 8 KB, they cost 8 % of the kernel;
//   * one CTA barrier per transform: the second pass's outputs that a last-pass butterfly needs
//     come from one column of threads, which share a half-warp and exchange them in place.
//
// What bounds it (L = 4096): instruction issue (64 to 70 % of the slots with 16 warps per SM), the
// FP32 pipe (54 %) and the shared-memory exchanges (55 %) together.  120-day band (N_s = 3600,
// 2880 segments, two detectors), 72 templates at once, per template: 151 us; 161 with XOR-swizzled
// exchanges, 174 with three barriers a transform, 640 at the output bins (8 transforms of 4096
// points a row instead of 2).  (Plain FP32 runs of 16 segments take 144 us and lose precision.)
//
// Waits are bounded (about one second): a wait that runs out sets bit 0 of the plan's error
// word; the CTA agrees on it at the next barrier, waits for its copies in flight, frees its
// tensor memory and returns.
#pragma once

#include <type_traits>

#include "corr.cuh"
#include "tma.cuh"
#include "tmem.cuh"

namespace cc {

// Shape of the transforms of L points.
template <int LT>
struct CorrShape {
    static constexpr int L = LT;
    static constexpr int T = CORR_POINTS / L;            // transforms per CTA
    static constexpr int GT = L / 16;                    // threads per transform
    static constexpr bool PASS2 = L >= 512;              // a radix-16 pass with NS = 16
    static constexpr int RL = PASS2 ? L / 256 : L / 16;  // radix of the last pass
    static constexpr int NSL = L / RL;                   // its butterflies
    static constexpr int BPT = 16 / RL;                  // of them per thread
    static constexpr int NP = RL == 16 ? 4 : RL == 8 ? 3 : RL == 4 ? 2 : 1;   // twiddle powers of one: 1, 2, 4, 8
    static constexpr int TA = T > 1 ? T / 2 : 1;         // templates of a series group
    static_assert(T * GT == CORR_THREADS && NSL == GT * BPT, "16 points per thread in every pass");
};

// x[r] *= w^r, r < R, from the powers 1, 2, 4, 8 of w (as many as R needs).
template <int R>
__device__ __forceinline__ void twiddle_powers(float2 (&x)[16], const float2 (&w)[4]) {
    x[1] = cmul(x[1], w[0]);
    if constexpr (R >= 4) {
        const float2 w3 = cmul(w[1], w[0]);
        x[2] = cmul(x[2], w[1]);
        x[3] = cmul(x[3], w3);
        if constexpr (R >= 8) {
            x[4] = cmul(x[4], w[2]);
            x[5] = cmul(x[5], cmul(w[2], w[0]));
            x[6] = cmul(x[6], cmul(w[2], w[1]));
            x[7] = cmul(x[7], cmul(w[2], w3));
            if constexpr (R == 16) {
                const float2 w12 = cmul(w[3], w[2]);
                x[8] = cmul(x[8], w[3]);
                x[9] = cmul(x[9], cmul(w[3], w[0]));
                x[10] = cmul(x[10], cmul(w[3], w[1]));
                x[11] = cmul(x[11], cmul(w[3], w3));
                x[12] = cmul(x[12], w12);
                x[13] = cmul(x[13], cmul(w12, w[0]));
                x[14] = cmul(x[14], cmul(w12, w[1]));
                x[15] = cmul(x[15], cmul(w12, w3));
            }
        }
    }
}

// Compensated sums of two FP32 values in paired operations (the same rounding as kahan_add
// on each): y = v - c, t = s + y, c = (t - s) - y.
__device__ __forceinline__ void kahan2(float2& s, float2& c, float2 v) {
    const float2 y = csub(v, c), t = cadd(s, y);
    c = csub(csub(t, s), y);
    s = t;
}

// The TA activity bytes (0 or 1) at p, aligned to TA, of which the first `valid` count, as bits.
template <int TA>
__device__ __forceinline__ uint32_t act_bits(const uint8_t* p, int valid) {
    uint32_t b = 0;
#pragma unroll
    for (int i = 0; i < TA; ++i)
        if (i < valid) b |= (uint32_t)__ldg(p + i) << i;
    return b;
}

template <int LT, bool BF16, bool LAG, bool HALF, bool MULTI>
__global__ void __launch_bounds__(CORR_THREADS, CORR_CTAS_PER_SM)
corr_kernel(const CorrArgs q) {
    using S = CorrShape<LT>;
    constexpr int L = S::L, T = S::T, GT = S::GT, RL = S::RL, NSL = S::NSL, BPT = S::BPT, TA = S::TA, NP = S::NP;
    // tensor-memory words per group of four bins: A [4], its compensations [4]; LAG: per bin B re im,
    // its compensations, S of the segment before
    constexpr int W = LAG ? 32 : 8;
    constexpr uint32_t COLS = 8 * W;                 // two warps of a lane quarter, four groups each
    constexpr uint32_t ESZ = BF16 ? 4 : 8;
    constexpr int PLANES = LAG ? 3 : 1;
    constexpr int SH = corr_act_bits(T, MULTI);      // activity bits of a detector in a segment's word
    using AW = std::conditional_t<T == 1, uint8_t, uint32_t>;
    constexpr bool PAD = T == 1;                     // exchange buffers padded instead of swizzled
    static_assert(TA <= SH, "one activity bit per template of the group");
    extern __shared__ __align__(128) unsigned char sm[];
    unsigned char* stage = sm;
    uint64_t* bar = (uint64_t*)(sm + q.off_bar);
    __shared__ int s_unit;
    __shared__ uint32_t s_tmem;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = tid / GT, j = tid % GT;
    // Exchange buffers: element p of a transform lies at 16 (p >> 4) + ((p ^ (p >> 4)) & 15), so
    // that 16 lanes reach 16 different banks down a column as well as along a row (8-point last
    // passes of neighbouring groups also take different halves).  PAD: row R of 16 elements at
    // 17 R + (R >> 4), conflict-free alike and at constant offsets in r (4 % fewer instructions).
    float2* const ex = (float2*)(sm + q.off_y);
    const int gsw = GT == 8 ? 8 * (g & 1) : 0;
    // second and last pass: thread j takes column k, rows i + RL r (see below)
    const int hw = j >> 4, i0 = S::PASS2 ? (j & 15) % RL : 0, k = S::PASS2 ? hw + RL * ((j & 15) / RL) : 0;
    const int wr1 = PAD ? 17 * j + hw : g * L + 16 * j + ((j & 15) ^ gsw);   // ^ r (PAD: + r): pass 1's output r
    const int rd2 = PAD ? 17 * i0 + k : g * L + 16 * i0 + (k ^ i0);          // pass 2's row i0, column k
    const int rd3 = PAD ? 273 * i0 + k : g * L + 16 * RL * i0 + 16 * i0 + (k ^ i0 ^ ((RL * i0) & 15));
    AW* aw = (AW*)(sm + q.off_act);      // per segment of the chunk: activity bits
    float2* const twk = (float2*)(sm + q.off_tw);    // the coset's first- and second-pass twiddles,
    float2* const twp = twk + 272;                   // and the last pass's powers
    int c_held = -1;
    const int C = q.C, M = q.M;
    const size_t act_x = (size_t)M * q.t_pad;        // bytes of one detector's activity

    if (warp == 0) tmem_alloc(&s_tmem, COLS);
    if (tid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    // the stage's rows end in zeros up to the transform's input length; no copy reaches them
    for (int s = q.n_in + j; s < (HALF ? L / 2 : L); s += GT) {
        if constexpr (BF16) ((uint32_t*)(stage + g * q.row_stride))[s] = 0u;
        else ((float2*)(stage + g * q.row_stride))[s] = make_float2(0.f, 0.f);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm_base = s_tmem;
    const uint32_t tm = tm_base + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * (COLS / 2);
    const uint32_t own_bit = T > 1 ? 1u << (g >> 1) : 1u;
    uint32_t phase = 0;
    bool first_unit = true;
    bool failed = false;

    for (;;) {
        if (tid == 0) s_unit = atomicAdd(q.ctr, 1);
        __syncthreads();
        const int u = s_unit;
        if (u >= q.units) break;
        const int c = u % C, v0 = u / C;
        const int chunk = v0 % q.n_chunks, sg = v0 / q.n_chunks;
        const int Ka = chunk * q.chunk_len;
        const int Kb = min(M, Ka + q.chunk_len);
        const int Kl = LAG ? max(0, Ka - 1) : Ka;
        // this thread's series: template t, weight w
        const int ser = sg * T + g;
        const int t = ser >> 1, w = ser & 1;
        // the coset's tables, when it changes
        if (c != c_held) {
            for (int i = tid; i < 272; i += CORR_THREADS) twk[i] = __ldg(q.twk + (size_t)c * 272 + i);
            for (int i = tid; i < BPT * NP * GT; i += CORR_THREADS) twp[i] = __ldg(q.twp + (size_t)c * BPT * NP * GT + i);
            c_held = c;
        }
        // activity of the chunk's segments: bit X SH + i, template i of the group has weight of
        // detector X
        {
            const int t0 = (sg * T) >> 1, nvalid = min(TA, q.n_t - t0);
            for (int K = Kl + tid; K < Kb; K += CORR_THREADS) {
                const uint8_t* p = q.act + (size_t)K * q.t_pad + t0;
                uint32_t b = act_bits<TA>(p, nvalid);
                for (int X = 1; X < q.Q; ++X) b |= act_bits<TA>(p + X * act_x, nvalid) << (X * SH);
                aw[K - Kl] = (AW)b;
            }
        }
        __syncthreads();
        // the transform after (K, X) in unit order; X = -1 starts at segment K
        auto next_after = [&](int K, int X, int& nK, int& nX) -> bool {
            uint32_t b = X + 1 < q.Q ? aw[K - Kl] >> ((X + 1) * SH) : 0u;
            if (b) {
                nK = K;
                nX = X + 1 + (__ffs(b) - 1) / SH;
                return true;
            }
            for (int k = K + 1; k < Kb; ++k) {
                b = aw[k - Kl];
                if (b) {
                    nK = k;
                    nX = (__ffs(b) - 1) / SH;
                    return true;
                }
            }
            return false;
        };
        auto row = [&](int K, int X, int tt, int ww) -> const char* {
            const size_t el = q.folded ? (((((size_t)tt * q.Q + X) * 2 + ww) * M + K) * C + c) * L
                                       : (((size_t)tt * q.Q + X) * 2 + ww) * q.N_tau + (size_t)K * q.N_s;
            return (const char*)q.src + el * ESZ;
        };
        // copy of the group's rows of the transform after (K, X) into the stage, after a
        // barrier that ends every read of it.  Rows of a template without weight there are
        // not copied (nor read).
        auto issue_after = [&](int K, int X) {
            int nK, nX;
            if (q.tma) {
                if (T == 1) {
                    if (tid == 0 && next_after(K, X, nK, nX)) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        mbar_arrive_expect_tx(bar, q.row_bytes);
                        tma_load_1d(stage, row(nK, nX, t, w), q.row_bytes, bar);
                    }
                } else if (warp == 0 && next_after(K, X, nK, nX)) {
                    const int s2 = sg * T + lane, tt = s2 >> 1;
                    const uint32_t b = aw[nK - Kl] >> (nX * SH);
                    const bool on = lane < T && ((b >> (lane >> 1)) & 1u);
                    const int n = __popc(__ballot_sync(0xffffffffu, on));
                    if (lane == 0) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        mbar_arrive_expect_tx(bar, (uint32_t)n * q.row_bytes);
                    }
                    __syncwarp();
                    if (on) tma_load_1d(stage + lane * q.row_stride, row(nK, nX, tt, s2 & 1), q.row_bytes, bar);
                }
            } else {
                if (next_after(K, X, nK, nX) && ((aw[nK - Kl] >> (nX * SH)) & own_bit)) {
                    const char* src = row(nK, nX, t, w);
                    unsigned char* dst = stage + g * q.row_stride;
                    for (int s = j; s < q.n_in; s += GT) cp_async<ESZ>(dst + s * ESZ, src + s * ESZ);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
        };

        {   // zero sums
            float z[W];
#pragma unroll
            for (int i = 0; i < W; ++i) z[i] = 0.f;
#pragma unroll
            for (int gi = 0; gi < 4; ++gi) tmem_st(tm + gi * W, z);
        }
        if (!(q.wait_test && first_unit)) issue_after(Kl, -1);
        first_unit = false;
        bool prev_zero = true;
        int parity = 0;

        for (int K = Kl; K < Kb; ++K) {
            const uint32_t bits = aw[K - Kl];
            if (!bits) {
                prev_zero = true;
                continue;
            }
            const bool acc_on = !LAG || K >= Ka;
            float2 v[16], f0[16];   // f0: detector 0's spectrum, MULTI: the earlier ones' sum
            bool have = false;      // f0 holds something
#pragma unroll
            for (int e = 0; e < 16; ++e) f0[e] = make_float2(0.f, 0.f);
#pragma unroll 1
            for (int X = 0; X < q.Q; ++X) {
                const uint32_t xbits = (bits >> (X * SH)) & ((1u << SH) - 1u);
                if (!xbits) continue;
                bool ok = true;
                if (q.tma) {
                    ok = mbar_wait(bar, phase);
                    phase ^= 1;
                } else {
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    __syncthreads();
                }
                // first pass: sample s = j + r GT of the segment
                const unsigned char* st = stage + g * q.row_stride;
#pragma unroll
                for (int r = 0; r < (HALF ? 8 : 16); ++r) {
                    if constexpr (BF16) v[r] = __bfloat1622float2(((const __nv_bfloat162*)st)[j + r * GT]);
                    else v[r] = ((const float2*)st)[j + r * GT];
                }
                if (T > 1 && !(xbits & own_bit)) {   // no weight: the row was not copied
#pragma unroll
                    for (int r = 0; r < 8; ++r) v[r] = make_float2(0.f, 0.f);
                }
                // buffers alternate between transforms: one CTA barrier each
                float2* buf = ex + (parity ? corr_buffer(T) : 0);
                parity ^= 1;
                if constexpr (HALF) {
                    dft16_in8(v);
                } else {
                    if (c > 0) {
#pragma unroll
                        for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], twk[r]);
                    }
                    dft16(v);
                }
#pragma unroll
                for (int r = 0; r < 16; ++r) buf[PAD ? wr1 + r : wr1 ^ r] = v[r];
                // every thread has read the stage and written its outputs; all agree on a failed wait
                if (__syncthreads_or(!ok)) {
                    failed = true;
                    break;
                }
                issue_after(K, X);
                // last pass: butterfly (i) of this thread leaves outputs m = b + NSL r in v[i RL + r]
                if constexpr (S::PASS2) {
                    // second pass on column k = j' mod 16 of the rows j' >> 4 + RL r (j' the Stockham
                    // index): the last pass needs the outputs of the RL threads of that column only,
                    // which sit in one half-warp and exchange them in place, without a CTA barrier
#pragma unroll
                    for (int r = 0; r < 16; ++r) v[r] = buf[PAD ? rd2 + 273 * r : (rd2 ^ ((RL * r) & 15)) + 16 * RL * r];
#pragma unroll
                    for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], twk[16 + r * 16 + k]);
                    dft16(v);
                    __syncwarp();
#pragma unroll
                    for (int r = 0; r < 16; ++r) {
                        const int cx = r & (RL - 1);
                        buf[PAD ? rd2 + 273 * r : (rd2 ^ (16 * cx + (cx ^ ((RL * r) & 15)))) + 16 * RL * r] = v[r];
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < BPT; ++i)
#pragma unroll
                        for (int r = 0; r < RL; ++r)
                            v[i * RL + r] = buf[PAD ? rd3 + 17 * r : (rd3 ^ (17 * r) ^ ((RL * RL * i) & 15)) + 16 * RL * RL * i];
                } else {
#pragma unroll
                    for (int i = 0; i < BPT; ++i)
#pragma unroll
                        for (int r = 0; r < RL; ++r)
                            v[i * RL + r] = buf[g * L + 16 * r + (((j + GT * i) ^ r ^ gsw) & 15)];
                }
#pragma unroll
                for (int i = 0; i < BPT; ++i) {
                    float2 x[16];
#pragma unroll
                    for (int r = 0; r < RL; ++r) x[r] = v[i * RL + r];
                    float2 pw[4];
#pragma unroll
                    for (int n = 0; n < NP; ++n) pw[n] = twp[(i * NP + n) * GT + j];
                    twiddle_powers<RL>(x, pw);
                    dft_r<RL>(x);
#pragma unroll
                    for (int r = 0; r < RL; ++r) v[i * RL + r] = x[r];
                }
                if constexpr (MULTI) {
                    // this detector's pairs with the earlier ones, then their sum
                    if (have && acc_on && !q.all_ordered) {
                        tmem_wait_st();
#pragma unroll
                        for (int gi = 0; gi < 4; ++gi) {
                            float z[8];
                            tmem_ld(z, tm + gi * W);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const int e = 4 * gi + 2 * h;
                                float2 s = make_float2(z[2 * h], z[2 * h + 1]), cp = make_float2(z[4 + 2 * h], z[5 + 2 * h]);
                                kahan2(s, cp, make_float2(redot(v[e], f0[e]), redot(v[e + 1], f0[e + 1])));
                                z[2 * h] = s.x;
                                z[2 * h + 1] = s.y;
                                z[4 + 2 * h] = cp.x;
                                z[5 + 2 * h] = cp.y;
                            }
                            tmem_st(tm + gi * W, z);
                        }
                    }
                    have = true;
#pragma unroll
                    for (int e = 0; e < 16; ++e) f0[e] = cadd(f0[e], v[e]);
                } else if (X + 1 < q.Q && (bits >> SH) != 0) {   // the second detector pairs with this one
#pragma unroll
                    for (int e = 0; e < 16; ++e) f0[e] = v[e];
                    have = true;
                }
            }
            if (failed) break;
            // pair terms of segment K
            const bool same = acc_on && (q.all_ordered || (!MULTI && have));   // terms of A
            if (LAG || same) {
                tmem_wait_st();
#pragma unroll
                for (int gi = 0; gi < 4; ++gi) {
                    float z[W];
                    tmem_ld(z, tm + gi * W);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int e = 4 * gi + 2 * h;
                        float2 Sk[2];
#pragma unroll
                        for (int i = 0; i < 2; ++i) Sk[i] = MULTI ? f0[e + i] : cadd(f0[e + i], v[e + i]);
                        if (same) {
                            const float2 d = q.all_ordered ? make_float2(redot(Sk[0], Sk[0]), redot(Sk[1], Sk[1]))
                                                           : make_float2(redot(v[e], f0[e]), redot(v[e + 1], f0[e + 1]));
                            float2 s = make_float2(z[2 * h], z[2 * h + 1]), cp = make_float2(z[4 + 2 * h], z[5 + 2 * h]);
                            kahan2(s, cp, d);
                            z[2 * h] = s.x;
                            z[2 * h + 1] = s.y;
                            z[4 + 2 * h] = cp.x;
                            z[5 + 2 * h] = cp.y;
                        }
                        if constexpr (LAG) {
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                float* const B = z + 8 + 6 * (2 * h + i);
                                if (acc_on && !prev_zero) {
                                    const float2 d = make_float2(redot(Sk[i], make_float2(B[4], B[5])),
                                                                 fmaf(Sk[i].x, B[5], -Sk[i].y * B[4]));
                                    float2 s = make_float2(B[0], B[1]), cp = make_float2(B[2], B[3]);
                                    kahan2(s, cp, d);
                                    B[0] = s.x;
                                    B[1] = s.y;
                                    B[2] = cp.x;
                                    B[3] = cp.y;
                                }
                                B[4] = Sk[i].x;
                                B[5] = Sk[i].y;
                            }
                        }
                    }
                    tmem_st(tm + gi * W, z);
                }
            }
            prev_zero = false;
        }
        if (failed) break;
        // the unit's sums to its row, through the exchange buffers (padded) for whole lines: the
        // values, then what they round off
        float* const fl = (float*)ex;
        constexpr int FP = CORR_POINTS + CORR_POINTS / 16;
        tmem_wait_st();
#pragma unroll 1
        for (int part = 0; part < 2; ++part) {
            __syncthreads();   // every thread has left the last transform's buffers (read the part before)
#pragma unroll
            for (int gi = 0; gi < 4; ++gi) {
                float z[W];
                tmem_ld(z, tm + gi * W);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int e = 4 * gi + i, b = e / RL;
                    const int m = g * L + (S::PASS2 ? 16 * (i0 + RL * b) + k : j + GT * b) + NSL * (e % RL), o = m + (m >> 4);
                    fl[o] = part ? -z[4 + i] : z[i];
                    if constexpr (LAG) {
                        const float* const B = z + 8 + 6 * i;
                        fl[FP + o] = part ? -B[2] : B[0];
                        fl[2 * FP + o] = part ? -B[3] : B[1];
                    }
                }
            }
            __syncthreads();
#pragma unroll
            for (int pl = 0; pl < PLANES; ++pl)
                for (int o = tid; o < CORR_POINTS; o += CORR_THREADS) {
                    const int so = sg * T + o / L, to = so >> 1;
                    if (to < q.n_t)
                        q.raw[((((size_t)to * 2 * q.n_chunks + (size_t)(so & 1) * q.n_chunks + chunk) * 2 * PLANES + 2 * pl + part) * C + c) * L + o % L] =
                            fl[pl * FP + o + (o >> 4)];
                }
        }
        __syncthreads();   // the next unit's first pass rewrites the buffers
    }
    // a failed wait leaves stores under way: every warp's are complete before tensor memory is freed
    tmem_wait_st();
    if (failed && tid == 0) {
        atomicOr(q.err, 1u);
        mbar_wait(bar, phase ^ 1);   // the copy still in flight, bounded
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) tmem_free(tm_base, COLS);
}

template <int LT, bool BF16, bool LAG, bool HALF, bool MULTI>
cudaError_t launch_corr_t(const CorrArgs& a, int sms, cudaStream_t st) {
    auto kern = corr_kernel<LT, BF16, LAG, HALF, MULTI>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)a.smem);
    if (e != cudaSuccess) return e;
    const int grid = a.units < CORR_CTAS_PER_SM * sms ? a.units : CORR_CTAS_PER_SM * sms;
    kern<<<grid, CORR_THREADS, a.smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace cc
