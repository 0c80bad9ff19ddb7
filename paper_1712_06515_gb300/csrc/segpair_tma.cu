// Spectra and pair sums at the output bins on 4096-point cosets: a persistent kernel whose
// segment samples arrive by TMA bulk copies.  It serves the two-pass search of segments longer
// than 4096 samples stored in BF16 (the long-lag band: N_FFT = 2^18 = 64 cosets of 4096): the
// folded rows are rounded to BF16 per output coset, so the products belong to these cosets'
// bins; every other two-pass search sums its products on the lag grid (corr_kernel.cuh), about a
// quarter of the transform work.
//
// Per (template, weight, chunk of segments, coset) unit a CTA of 256 threads walks the chunk's
// segments; per segment it transforms detector 0's and detector 1's folded row (the N_FFT-point
// DFT restricted to coset c, Sec. III B 4: a 4096-point transform of Z_q[p] times
// exp(-2 pi i (b0 + c) p / N_FFT)) and folds the two spectra into the pair sum of Eq.
// final-formatted-rho:
//
//   * staging: rows arrive in two stages by cp.async.bulk (TMA, completion on an mbarrier each),
//     the copy of the row after the next issued as soon as the current transform's first pass
//     has read its stage.  Rows are read once, from HBM;
//   * scheduling: two persistent CTAs per SM, units handed out by one atomic counter,
//     neighbouring cosets in turn (neighbouring rows of Z); results never depend on placement;
//   * segment-relative positions: sample s of a segment sits at transform position s, so its
//     transform T_K(m) lacks the segment-start phase W_N^(k seg0_K) of bin k = b0 + c + C m.  In
//     a pair of consecutive segments that phase leaves theta(m) = W_N^(-k N_s), one constant per
//     bin: Re(conj(F_K) F_(K-1)) = Re(conj(T_K) T_(K-1) theta(m)), and the same-segment terms
//     carry no phase.  theta(m + 256) = theta(m) psi with psi = exp(2 pi i N_s / 16), so each
//     thread keeps theta of its first bin and steps by psi through its eight bins m = b + 256 r
//     (psi = 1 when 16 divides N_s);
//   * the passes are corr_kernel's: one CTA barrier per transform, the second pass's outputs
//     exchanged inside half-warps through padded buffers, the coset's twiddles in shared
//     memory; the last pass computes only the 8 outputs m < 2048 that hold output bins;
//   * the previous segment's detector sum (times theta) and detector 0's spectrum -- 32 words a
//     thread -- live in tensor memory, read and written once per segment, the Kahan sums in
//     registers.
//
// What bounds it: instruction issue (71 % of the slots, about 970 instructions a warp and
// transform, 16 warps per SM), the FP32 pipe (59 %) and the shared-memory exchanges (58 %); Z
// leaves HBM at 1.8 TB/s.  The 120-day band at a ten-hour lag, per template of two: 667 us; 684 with
// XOR-swizzled exchanges, 842 with two more barriers a transform, twiddles read through L1 and
// one stage.  (16 at once: 600.)
//
// Waits on the mbarriers are bounded (about one second of clock): a wait that runs out sets bit
// 0 of the plan's device error word, every thread of the CTA agrees on it at the next barrier,
// the CTA waits (bounded again) for the copies still in flight, frees its tensor memory and
// returns; crosscorr_plan_check reports CC_ERR_TIMEOUT.
#include <algorithm>

#include "segpair.cuh"
#include "tma.cuh"
#include "tmem.cuh"

namespace cc {

namespace {

constexpr int TT_THREADS = 256;
constexpr int TT_L = 4096;
constexpr int TT_EX = 17 * 256 + 16;  // elements of an exchange buffer
constexpr int TT_BINS = TT_L / 2;    // kept positions m < 2048 of a coset, eight a thread
constexpr int TT_MAX_CHUNK = 1023;   // segments of a chunk (its activity, and one before, is kept on chip)
constexpr int FOLD_MAX_F = 16;       // folds of a long segment onto the 4096 positions
constexpr int FOLD_MAX_C = 1024;     // cosets of a folded plan
constexpr uint32_t TT_ROW = TT_L * 4;   // bytes of a folded row (bf16 pairs)

// shared memory: two stages, two exchange buffers, the coset's twiddles (272 and 4 x 256), a
// byte of activity a segment, two mbarriers
constexpr size_t TT_OFF_EX = 2 * TT_ROW;
constexpr size_t TT_OFF_TW = TT_OFF_EX + 2 * (size_t)TT_EX * sizeof(float2);
constexpr size_t TT_OFF_ACT = TT_OFF_TW + (272 + 4 * TT_THREADS) * sizeof(float2);
constexpr size_t TT_OFF_BAR = TT_OFF_ACT + TT_MAX_CHUNK + 1;
constexpr size_t TT_SMEM = TT_OFF_BAR + 16;
static_assert(TT_OFF_BAR % 8 == 0 && 2 * (TT_SMEM + 1024) <= 228 * 1024, "two CTAs per SM");

struct PairArgs {
    const char* z;          // folded rows [n_t][Q][2][M][C][4096], bf16 pairs
    const float4* norm;     // [n_t][Q][M] (hat-A, hat-B, hat-C, 0)
    float* raw;             // [n_t][2 n_chunks][N_f] partial pair sums
    int* ctr;               // unit counter, zero at launch
    unsigned* err;          // the plan's device error word
    const float2* twk;      // DevParams::twk
    const int *coset_off, *coset_k, *coset_m;   // the cosets' output bins and their positions
    int64_t N_FFT, b0, N_s, N_f, units;
    int M, Q, C, n_chunks, chunk_len, lag, all_ordered, wait_test;
};

__global__ void __launch_bounds__(TT_THREADS, 2)
segpair_tma_kernel(const PairArgs q) {
    constexpr int W = 32;   // tensor-memory words of a thread: S_(K-1) theta [8], detector 0's spectrum [8]
    constexpr uint32_t COLS = 2 * W;
    extern __shared__ __align__(128) unsigned char sm[];
    float2* const ex = (float2*)(sm + TT_OFF_EX);
    float2* const twk = (float2*)(sm + TT_OFF_TW);
    float2* const twp = twk + 272;
    uint8_t* const act = sm + TT_OFF_ACT;   // bit 0: detector 0, bit Q - 1: the last one has weight in the segment
    uint64_t* const bar = (uint64_t*)(sm + TT_OFF_BAR);
    __shared__ int s_unit;
    __shared__ uint32_t s_tmem;

    const int tid = threadIdx.x, warp = tid >> 5, Q = q.Q, C = q.C, M = q.M;
    // Exchange buffers: row R of 16 elements starts at 17 R + (R >> 4), so that 16 lanes reach 16
    // different banks down a column, along a row and from block to block, at constant offsets in
    // r.  Second and last pass: thread j takes column k2, rows i0 + 16 r, then butterfly b
    const int k2 = tid >> 4, i0 = tid & 15, b = 16 * i0 + k2;
    const int wr1 = 17 * tid + k2, rd2 = 17 * i0 + k2, rd3 = 273 * i0 + k2;
    const uint64_t N = (uint64_t)q.N_FFT, mask = N - 1;
    const bool psi_one = (q.N_s & 15) == 0;
    float2 psi;
    sincospif(0.125f * (float)(q.N_s & 15), &psi.y, &psi.x);   // exp(2 pi i (N_s mod 16) / 16)

    if (warp == 0) tmem_alloc(&s_tmem, COLS);
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm_base = s_tmem;
    const uint32_t tm = tm_base + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * W;
    uint32_t phase = 0, in_flight = 0;   // bit per stage (in_flight: thread 0's)
    int slot = 0, parity = 0;
    bool first_unit = true, failed = false;

    for (;;) {
        if (tid == 0) s_unit = atomicAdd(q.ctr, 1);
        __syncthreads();
        const int u = s_unit;
        if (u >= q.units) break;
        const int c = u % C, v0 = u / C, chunk = v0 % q.n_chunks, tw = v0 / q.n_chunks;
        const int t = tw >> 1;
        const int Ka = chunk * q.chunk_len, Kb = min(M, Ka + q.chunk_len), Kl = max(0, Ka - q.lag);
        const uint64_t bc = ((uint64_t)q.b0 + (uint64_t)c) & mask, ct = bc + (uint64_t)C * b;
        // pair phase of this thread's first bin
        const float2 theta = twiddle_N((N - (ct * (uint64_t)q.N_s & mask)) & mask, N);
        // last pass: element r of butterfly b takes W_L^(b r) W_N^(bc r) = W_N^(ct r), formed
        // from powers 1, 2, 4, 8
#pragma unroll
        for (int n = 0; n < 4; ++n) twp[n * TT_THREADS + tid] = twiddle_N((ct << n) & mask, N);
        for (int i = tid; i < 272; i += TT_THREADS) twk[i] = __ldg(q.twk + (size_t)c * 272 + i);
        for (int K = Kl + tid; K < Kb; K += TT_THREADS) {
            uint32_t a = 0;
            for (int X = 0; X < Q; ++X) {
                const float4 n = __ldg(q.norm + ((size_t)t * Q + X) * M + K);
                a |= (n.x + n.y > 0.f ? 1u : 0u) << X;
            }
            act[K - Kl] = (uint8_t)a;
        }
        __syncthreads();
        // row Z_q of coset c: q = (b0 + c) mod C
        const char* const src = q.z + (((size_t)tw + (size_t)t * 2 * (Q - 1)) * M * C + (size_t)(bc & (uint64_t)(C - 1))) * TT_ROW;
        // thread 0: the copy of the transform after (pK, pX) in unit order into stage s, after a
        // barrier that ends every read of it
        int pK = Kl, pX = -1;
        auto issue = [&](int s) {
            if (pK >= Kb) return;
            uint32_t a = pX + 1 < Q ? (uint32_t)act[pK - Kl] >> (pX + 1) << (pX + 1) : 0u;
            while (!a) {
                if (++pK >= Kb) return;
                a = act[pK - Kl];
            }
            pX = __ffs(a) - 1;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive_expect_tx(bar + s, TT_ROW);
            tma_load_1d(sm + s * TT_ROW, src + ((size_t)pX * 2 * M + pK) * C * TT_ROW, TT_ROW, bar + s);
            in_flight |= 1u << s;
        };
        // (the wait test leaves the CTA's first copies unissued: its bounded wait runs out)
        if (tid == 0 && !(q.wait_test && first_unit)) {
            issue(slot);
            issue(slot ^ 1);
        }
        first_unit = false;

        float accP[8], cmpP[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) accP[r] = cmpP[r] = 0.f;
        bool prev_zero = true;

        for (int K = Kl; K < Kb; ++K) {
            const uint32_t bits = act[K - Kl];
            if (!bits) {
                prev_zero = true;
                continue;
            }
            const bool a0 = Q > 1 && (bits & 1u), al = (bits >> (Q - 1)) & 1u;
            float2 v[16];
#pragma unroll 1
            for (int X = a0 ? 0 : Q - 1; X < (al ? Q : 1); ++X) {
                const bool ok = mbar_wait(bar + slot, (phase >> slot) & 1u);
                if (ok) in_flight &= ~(1u << slot);
                const __nv_bfloat162* st = (const __nv_bfloat162*)(sm + slot * TT_ROW);
                float2* const buf = ex + (parity ? TT_EX : 0);   // buffers alternate: one CTA barrier a transform
                parity ^= 1;
                // first pass: position p = tid + 256 r times the coset factor W_N^(256 bc r)
#pragma unroll
                for (int r = 0; r < 16; ++r) v[r] = __bfloat1622float2(st[tid + 256 * r]);
#pragma unroll
                for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], twk[r]);
                dft16(v);
#pragma unroll
                for (int r = 0; r < 16; ++r) buf[wr1 + r] = v[r];
                // every thread has read the stage and written its outputs; all agree on a failed wait
                if (__syncthreads_or(!ok)) {
                    failed = true;
                    break;
                }
                if (tid == 0) issue(slot);
                phase ^= 1u << slot;
                slot ^= 1;
                // second pass: twiddles W_L^(16 k r) W_N^(16 bc r)
#pragma unroll
                for (int r = 0; r < 16; ++r) v[r] = buf[rd2 + 273 * r];
#pragma unroll
                for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], twk[16 + r * 16 + k2]);
                dft16(v);
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 16; ++r) buf[rd2 + 273 * r] = v[r];
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 16; ++r) v[r] = buf[rd3 + 17 * r];
                {
                    const float2 b1 = twp[tid], b2 = twp[TT_THREADS + tid], b4 = twp[2 * TT_THREADS + tid];
                    const float2 b8 = twp[3 * TT_THREADS + tid], b3 = cmul(b2, b1), b12 = cmul(b8, b4);
                    v[1] = cmul(v[1], b1);
                    v[2] = cmul(v[2], b2);
                    v[3] = cmul(v[3], b3);
                    v[4] = cmul(v[4], b4);
                    v[5] = cmul(v[5], cmul(b4, b1));
                    v[6] = cmul(v[6], cmul(b4, b2));
                    v[7] = cmul(v[7], cmul(b4, b3));
                    v[8] = cmul(v[8], b8);
                    v[9] = cmul(v[9], cmul(b8, b1));
                    v[10] = cmul(v[10], cmul(b8, b2));
                    v[11] = cmul(v[11], cmul(b8, b3));
                    v[12] = cmul(v[12], b12);
                    v[13] = cmul(v[13], cmul(b12, b1));
                    v[14] = cmul(v[14], cmul(b12, b2));
                    v[15] = cmul(v[15], cmul(b12, b3));
                }
                dft16_lo8(v);
                if (X + 1 < Q) {
                    float z[16];
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        z[2 * r] = v[r].x;
                        z[2 * r + 1] = v[r].y;
                    }
                    tmem_st(tm + 16, z);
                }
            }
            if (failed) break;
            // pair terms of segment K (zero for a detector with no weight in it)
            const bool acc_on = K >= Ka;
            float z[W], s[16];
            tmem_wait_st();
            tmem_ld(z, tm);
            float2 th = theta;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float2 zero = make_float2(0.f, 0.f);
                const float2 F1 = al ? v[r] : zero, F0 = a0 ? make_float2(z[16 + 2 * r], z[17 + 2 * r]) : zero;
                const float2 S = Q > 1 ? cadd(F0, F1) : F1;
                const float2 P = prev_zero ? zero : make_float2(z[2 * r], z[2 * r + 1]);
                const float term = q.all_ordered ? fmaf(2.f, redot(S, P), redot(S, S)) : redot(S, P) + redot(F1, F0);
                if (acc_on) kahan_add(accP[r], cmpP[r], term);
                const float2 n = cmul(S, th);
                s[2 * r] = n.x;
                s[2 * r + 1] = n.y;
                if (!psi_one) th = cmul(th, psi);
            }
            if (q.lag) tmem_st(tm, s);
            prev_zero = !q.lag;
        }
        if (failed) break;
        // partial sums of this (template, weight, chunk) row for the coset's bins, staged through
        // an exchange buffer
        __syncthreads();
        float* const accm = (float*)ex;
#pragma unroll
        for (int r = 0; r < 8; ++r) accm[b + 256 * r] = accP[r];
        __syncthreads();
        const int o = __ldg(q.coset_off + c), nbc = __ldg(q.coset_off + c + 1) - o;
        float* const out = q.raw + ((size_t)tw * q.n_chunks + chunk) * q.N_f;
        for (int i = tid; i < nbc; i += TT_THREADS) out[__ldg(q.coset_k + o + i)] = accm[__ldg(q.coset_m + o + i)];
        // the next unit's first pass rewrites the buffer: the unit fetch's barrier orders it
    }
    // a failed wait leaves stores under way: every warp's are complete before tensor memory is freed
    tmem_wait_st();
    if (failed && tid == 0) {
        atomicOr(q.err, 1u);
        for (int s = 0; s < 2; ++s)   // copies still in flight, bounded
            if (in_flight & (1u << s)) mbar_wait(bar + s, (phase >> s) & 1u);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) tmem_free(tm_base, COLS);
}

// Fold of a long segment (N_s > L) onto the L = 4096 positions of the coset transforms
// (Sec. III B 4 with a segment longer than the on-chip transform): position p of coset c
// takes sum_f x[p + f L] W_N^((b0+c)(p + f L)) = W_N^((b0+c) p) Z_q[p] with
// Z_q[p] = sum_f x[p + f L] W_C^(q f) and q = (b0 + c) mod C (W_N^L = W_C), a C-point
// DFT over the fold index f computed once per (template, detector, weight, segment) for
// every q, instead of each coset re-reading and re-twiddling the whole segment.  The
// persistent kernel applies W_N^((b0+c) p) as it does for whole segments.
// grid: x = segment K, y = detector X * 2 + weight w, z = template of the batch.
// ab: [n_t][Q][2][N_tau], z: [n_t][Q][2][M][C][L], bf16 pairs.
__global__ void __launch_bounds__(TT_THREADS)
fold_cosets_kernel(DevParams p, const void* __restrict__ ab, const float4* __restrict__ norm, void* __restrict__ z) {
    __shared__ float2 wc[FOLD_MAX_C];   // W_C^n
    constexpr int L = TT_L;
    const int64_t K = blockIdx.x;
    const int X = blockIdx.y >> 1, w = blockIdx.y & 1;
    const int64_t t = blockIdx.z;
    const int Q = p.Q, C = p.C4, tid = threadIdx.x;
    const int64_t N_s = p.N_s, M = p.M;
    const float4 nm = norm[((size_t)t * Q + X) * M + K];
    if (!(nm.x + nm.y > 0.f)) return;   // no weight in the segment: the row is never read
    for (int n = tid; n < C; n += TT_THREADS) {
        float sn, cs;
        sincospif(-2.0f * (float)n / (float)C, &sn, &cs);
        wc[n] = make_float2(cs, sn);
    }
    __syncthreads();
    const int F = (int)((N_s + L - 1) / L);
    const size_t row = (((size_t)t * Q + X) * 2 + w) * p.N_tau + (size_t)(K * N_s);
    const size_t zrow = ((((size_t)t * Q + X) * 2 + w) * M + K) * C * L;
    for (int i = 0; i < L / TT_THREADS; ++i) {
        const int pp = tid + TT_THREADS * i;
        float2 a[FOLD_MAX_F];
#pragma unroll
        for (int f = 0; f < FOLD_MAX_F; ++f) {
            const int64_t sidx = pp + (int64_t)f * L;
            a[f] = make_float2(0.f, 0.f);
            if (f < F && sidx < N_s) {
                a[f] = __bfloat1622float2(((const __nv_bfloat162*)ab)[row + sidx]);
            }
        }
        for (int qq = 0; qq < C; ++qq) {
            float2 acc = a[0];
#pragma unroll
            for (int f = 1; f < FOLD_MAX_F; ++f)
                if (f < F) acc = cadd(acc, cmul(a[f], wc[(qq * f) & (C - 1)]));
            const size_t o = zrow + (size_t)qq * L + pp;
            ((__nv_bfloat162*)z)[o] = __float22bfloat162_rn(acc);
        }
    }
}

// fold_cosets_kernel for C = 64 cosets (the long-lag band: N_FFT = 2^18 = 64 x 4096) and at most
// 16 folds, by a radix-8 split of the 64-point DFT over the fold index: with q = u + 8 v
// and f = f1 + 8 f2, W_64^(q f) = W_8^(v f1) W_64^(u f1) W_8^(u f2), so
// Z_(u+8v) = DFT8_v[ W_64^(u f1) (a_(f1) + a_(f1+8) W_8^u) ]: per residue u a twiddle and
// one register 8-point DFT instead of 64 x F products.
template <int MAXF>
__global__ void __launch_bounds__(TT_THREADS, 3)
fold64_kernel(DevParams p, const void* __restrict__ ab, const float4* __restrict__ norm, void* __restrict__ z) {
    static_assert(MAXF > 8 && MAXF <= 16, "folds f = f1 + 8 f2 with f2 < 2");
    __shared__ float2 w64[64];   // W_64^n = W_4096^(64 n)
    constexpr int L = TT_L, C = 64;
    const int64_t K = blockIdx.x;
    const int X = blockIdx.y >> 1, w = blockIdx.y & 1;
    const int64_t t = blockIdx.z;
    const int Q = p.Q, tid = threadIdx.x;
    const int64_t N_s = p.N_s, M = p.M;
    const float4 nm = norm[((size_t)t * Q + X) * M + K];
    if (!(nm.x + nm.y > 0.f)) return;   // no weight in the segment: the row is never read
    if (tid < C) w64[tid] = __ldg(p.twL + 64 * tid);
    __syncthreads();
    const int F = (int)((N_s + L - 1) / L);
    const size_t row = (((size_t)t * Q + X) * 2 + w) * p.N_tau + (size_t)(K * N_s);
    const size_t zrow = ((((size_t)t * Q + X) * 2 + w) * M + K) * C * L;
    for (int i = 0; i < L / TT_THREADS; ++i) {
        const int pp = tid + TT_THREADS * i;
        float2 a[MAXF];
#pragma unroll
        for (int f = 0; f < MAXF; ++f) {
            const int64_t sidx = pp + (int64_t)f * L;
            a[f] = make_float2(0.f, 0.f);
            if (f < F && sidx < N_s) {
                a[f] = __bfloat1622float2(((const __nv_bfloat162*)ab)[row + sidx]);
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            float2 v[16];
#pragma unroll
            for (int f1 = 0; f1 < 8; ++f1) {
                float2 b = a[f1];
                if (f1 + 8 < MAXF && f1 + 8 < F) b = cadd(b, u == 0 ? a[f1 + 8] : cmul(a[f1 + 8], w64[8 * u]));
                v[f1] = (u == 0 || f1 == 0) ? b : cmul(b, w64[(u * f1) & 63]);
            }
            dft8(v);   // v[j] = sum_f1 W_8^(j f1) (...): Z_(u + 8 j)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const size_t o = zrow + (size_t)(u + 8 * j) * L + pp;
                ((__nv_bfloat162*)z)[o] = __float22bfloat162_rn(v[j]);
            }
        }
    }
}

}  // namespace

// Folded segments in BF16: more than 4096 samples, a multiple of 4 (rows then start on 16-byte
// boundaries for the bulk copies), at most FOLD_MAX_F folds and FOLD_MAX_C cosets, Q <= 2,
// R <= 1, the output bins in the lower half of each coset transform.
bool segpair_tma_supported(const cc_plan* plan) {
    const DevParams& p = plan->dp;
    if (p.store != CC_STORE_BF16 || p.N_s <= TT_L || p.L != TT_L || p.Q > 2 || p.R > 1 ||
        p.pair_mode == CC_PAIRS_CROSS_ONLY || plan->N_f < 1)
        return false;
    if (p.C4 > FOLD_MAX_C || (p.N_s + TT_L - 1) / TT_L > FOLD_MAX_F || p.N_s % 4) return false;
    return p.C4 > 0 && plan->kbar_span4 < TT_BINS;
}

// Segment chunks per (template, weight) for a batch of n_t templates: about
// `units per CTA` (the tuning's chunk_waves, default 24) units per persistent CTA, each
// chunk at least 4R + 1 segments and at most TT_MAX_CHUNK.
int segpair_tma_chunks(const cc_plan* plan, int64_t n_t) {
    const DevParams& p = plan->dp;
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t per_cta = plan->tuning.chunk_waves > 0 ? plan->tuning.chunk_waves : 24;
    const int64_t ctas_per_coset = std::max<int64_t>(1, 2 * (int64_t)sms / p.C4);
    const int64_t want = (per_cta * ctas_per_coset + 2 * n_t - 1) / (2 * n_t);
    const int64_t maxch = std::max<int64_t>(1, p.M / (4 * p.R + 1));
    const int64_t least = (p.M + TT_MAX_CHUNK - 1) / TT_MAX_CHUNK;
    return (int)std::max<int64_t>(least, std::min<int64_t>({want, maxch, 32767}));
}

// Bytes of the fold kernel's output per template.
size_t segpair_tma_fold_bytes(const cc_plan* plan) {
    const DevParams& p = plan->dp;
    return (size_t)p.Q * 2 * p.M * p.C4 * TT_L * 4;
}

cc_status launch_fold_bf16(cc_plan* plan, int64_t n_t, const void* ab, const float4* norm, void* z, cudaStream_t st) {
    const DevParams& p = plan->dp;
    if (n_t > 65535 || p.M > 0x7fffffff) return fail(CC_ERR_UNSUPPORTED, "fold launch size");
    const dim3 grid((unsigned)p.M, (unsigned)(2 * p.Q), (unsigned)n_t);
    const int64_t F = (p.N_s + TT_L - 1) / TT_L;
    if (p.C4 == 64 && F <= 9)   // the long-lag band: nine folds
        fold64_kernel<9><<<grid, TT_THREADS, 0, st>>>(p, ab, norm, z);
    else if (p.C4 == 64)
        fold64_kernel<16><<<grid, TT_THREADS, 0, st>>>(p, ab, norm, z);
    else
        fold_cosets_kernel<<<grid, TT_THREADS, 0, st>>>(p, ab, norm, z);
    count_launch();
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? CC_OK : cuda_fail(e, "fold launch");
}

cc_status launch_segpair_tma(cc_plan* plan, int n_chunks, int64_t chunk_len, int64_t n_t, const void* z,
                             const float4* norm, float* raw, int* counter, cudaStream_t st) {
    const DevParams& p = plan->dp;
    PairArgs q;
    q.z = (const char*)z;
    q.norm = norm;
    q.raw = raw;
    q.ctr = counter;
    q.err = p.err;
    q.twk = p.twk;
    q.coset_off = p.coset4_off;
    q.coset_k = p.coset4_k;
    q.coset_m = p.coset4_m;
    q.N_FFT = p.N_FFT;
    q.b0 = p.b0;
    q.N_s = p.N_s;
    q.N_f = p.N_f;
    q.M = (int)p.M;
    q.Q = p.Q;
    q.C = p.C4;
    q.n_chunks = n_chunks;
    q.chunk_len = (int)chunk_len;
    q.lag = (int)p.R;
    q.all_ordered = p.pair_mode == CC_PAIRS_ALL_ORDERED;
    q.wait_test = p.wait_test;
    q.units = n_t * 2 * n_chunks * p.C4;
    if (q.units > 0x7fffffff - 65536) return fail(CC_ERR_UNSUPPORTED, "too many work units in one launch");
    int dev = 0, sms = 152;
    cudaError_t e = cudaFuncSetAttribute(segpair_tma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TT_SMEM);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return cuda_fail(e, "segment pair set-up");
    segpair_tma_kernel<<<(unsigned)std::min<int64_t>(2 * (int64_t)sms, q.units), TT_THREADS, TT_SMEM, st>>>(q);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "segpair_tma launch");
    return CC_OK;
}

}  // namespace cc
