// The staged segment-FFT stage for whole segments of up to 4096 samples (the 120-day single
// band: N_FFT = 32768 = 8 cosets of 4096, N_s = 3600): one persistent CTA per SM computes whole
// output rows F[t][X][K][w][0 .. N_f).
//
// Each coset transform is the zero-padded N_FFT-point DFT restricted to bins k = b0 + c (mod C)
// (Sec. III B 4: a 4096-point transform of the samples times exp(-2 pi i (b0 + c) s / N_FFT)),
// times the segment-start phase.  Neighbouring output bins belong to different cosets: a CTA per
// coset wrote 8 bytes into every sector of the row in turn, eight CTAs the row, four times the
// L2 transactions of the row's bytes, which took most of the stage's time.  Here two groups of
// 256 threads take a coset each, C / 2 rounds, the samples staged once per row by a TMA bulk
// copy; the outputs gather in a row buffer in shared memory, which leaves by one bulk copy under
// the next row's first pass (an odd number of bins: by plain stores).  The
// exchanges are the pair kernels' (padded buffers, the last one inside half-warps).  A row of zeros (a
// gapped segment, as the resampling stage writes it) is written without transforms.
//
// What bounds it: shared memory (65 % of its wavefronts) and issue, with the 16 warps per SM that
// registers and 200 KB of buffers allow, and the barriers between a row's rounds.  20 days, three
// templates (N_FFT = 32768, N_f = 12356): 433 us, 470 with plain stores of the row, about 650
// with a CTA per coset; 510 MB leave.
//
// Waits on the mbarrier are bounded (about one second): a wait that runs out sets bit 0 of the
// plan's error word, the CTA waits (bounded again) for the copy in flight and returns.
#include <algorithm>

#include "segpair.cuh"
#include "tma.cuh"

namespace cc {

namespace {

constexpr int SR_THREADS = 512;
constexpr int SR_L = 4096;
constexpr int SR_EX = 17 * 256 + 16;   // elements of an exchange buffer

struct RowsArgs {
    const void* ab;          // [n_t][Q][2][N_tau]
    float2* F;               // [n_t][Q][M][2][N_f]
    int* ctr;                // row counter, zero at launch
    unsigned* err;
    const float2* twk;       // [C][272] first- and second-pass twiddles (DevParams::twk)
    const float2* twp;       // [C][4][256] last-pass powers, or null: computed
    const int* kmap;         // [C][2048] output bin of position m, or -1
    int64_t N_FFT, b0, N_tau, M, N_s, N_f;
    int64_t rows;
    int Q, C, wait_test;
    int bulk;                // rows of F are whole 16-byte pieces: they leave by bulk copies
    uint32_t row_bytes, off_ex, off_row, off_bar;
};

// A bulk copy shared -> global (16-byte pieces) as a group of its own, and the wait until the
// thread's copies have read their source.
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_store_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

__device__ __forceinline__ void group_sync(int grp) {
    asm volatile("bar.sync %0, 256;" ::"r"(grp + 1) : "memory");
}

// DIRECT: a row too long for the buffers beside it goes to F from the registers.
template <bool BF16, bool DIRECT>
__global__ void __launch_bounds__(SR_THREADS, 1)
segfft_rows_kernel(RowsArgs q) {
    constexpr uint32_t ESZ = BF16 ? 4 : 8;
    extern __shared__ __align__(128) unsigned char sm[];
    unsigned char* stage = sm;
    float2* row = (float2*)(sm + q.off_row);
    uint64_t* bar = (uint64_t*)(sm + q.off_bar);
    __shared__ int64_t s_next;
    __shared__ int s_nz[2];   // a nonzero sample in the row (two rows in turn)
    const int tid = threadIdx.x, grp = tid >> 8, j = tid & 255;
    float2* ex = (float2*)(sm + q.off_ex) + grp * SR_EX;
    const int C = q.C;
    const uint64_t N = (uint64_t)q.N_FFT, mask = N - 1;
    // second and last pass: thread j takes column k, rows i + 16 r (see corr_kernel.cuh)
    const int k2 = j >> 4, i0 = j & 15;
    const int wr1 = 17 * j + k2, rd2 = 17 * i0 + k2, rd3 = 273 * i0 + k2;   // rows at 17 R + (R >> 4), see segpair_tma.cu
    const int b = 16 * i0 + k2;                  // last-pass butterfly: outputs m = b + 256 r

    if (tid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        s_next = atomicAdd(q.ctr, 1);
        s_nz[0] = s_nz[1] = 0;
    }
    for (int s = (int)q.N_s + tid; s < SR_L; s += SR_THREADS) {   // zeros beyond the samples; no copy reaches them
        if constexpr (BF16) ((uint32_t*)stage)[s] = 0u;
        else ((float2*)stage)[s] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    auto issue = [&](int64_t r) {   // thread 0, after a barrier that ends every read of the stage
        const int w = (int)(r & 1);
        const int64_t tX = (r >> 1) / q.M, K = (r >> 1) - tX * q.M;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect_tx(bar, q.row_bytes);
        tma_load_1d(stage, (const char*)q.ab + ((size_t)(2 * tX + w) * q.N_tau + (size_t)K * q.N_s) * ESZ, q.row_bytes, bar);
    };
    int64_t cur = s_next;
    if (tid == 0 && cur < q.rows && !q.wait_test) issue(cur);
    __syncthreads();
    uint32_t phase = 0;   // also which of s_nz the row uses
    while (cur < q.rows) {
        if (tid == 0) s_next = atomicAdd(q.ctr, 1);
        const int64_t tX = (cur >> 1) / q.M, K = (cur >> 1) - tX * q.M;
        const uint64_t s0 = (uint64_t)(K * q.N_s) & mask;
        float2* Fo = q.F + (size_t)cur * q.N_f;
        const bool ok = mbar_wait(bar, phase);
        int* const nzp = &s_nz[phase];
        phase ^= 1;
        bool zero = false;
        // the segment-start phase W_N^(k seg0) of bin k = bc + C m, m = b + 256 r, steps by this
        const float2 phs = twiddle_N(((256 * (uint64_t)C) * s0) & mask, N);
#pragma unroll 1
        for (int c0 = 0; c0 < C; c0 += 2) {
            const int c = c0 + grp;
            const bool on = c < C;
            const bool last = c0 + 2 >= C;
            float2 v[16];
            if (on) {
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    if constexpr (BF16) v[r] = __bfloat1622float2(((const __nv_bfloat162*)stage)[j + 256 * r]);
                    else v[r] = ((const float2*)stage)[j + 256 * r];
                }
                if (c0 == 0 && grp == 0) {   // group 0 sees every sample
                    bool nz = false;
#pragma unroll
                    for (int r = 0; r < 16; ++r) nz |= v[r].x != 0.f || v[r].y != 0.f;
                    if (__any_sync(0xffffffffu, nz) && (tid & 31) == 0) *nzp = 1;
                }
                const float2* __restrict__ tw = q.twk + (size_t)c * 272;
#pragma unroll
                for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], __ldg(tw + r));
                dft16(v);
#pragma unroll
                for (int r = 0; r < 16; ++r) ex[wr1 + r] = v[r];
            }
            if (c0 == 0) {
                if (tid == 0) bulk_store_read();   // the row before has left its buffer
                if (__syncthreads_or(!ok)) {
                    if (tid == 0) {
                        atomicOr(q.err, 1u);
                        mbar_wait(bar, phase ^ 1);   // the copy still in flight, bounded
                    }
                    __syncthreads();
                    return;
                }
                zero = *nzp == 0;
                if (tid == 0) s_nz[phase] = 0;   // the next row's word (every thread is past reading it)
            } else if (last) {
                __syncthreads();
            } else {
                group_sync(grp);
            }
            if ((last || zero) && tid == 0 && s_next < q.rows) issue(s_next);   // every read of the stage is done
            if (zero) break;
            if (on) {
                const float2* __restrict__ tw = q.twk + (size_t)c * 272 + 16;
#pragma unroll
                for (int r = 0; r < 16; ++r) v[r] = ex[rd2 + 273 * r];
#pragma unroll
                for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], __ldg(tw + r * 16 + k2));
                dft16(v);
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 16; ++r) ex[rd2 + 273 * r] = v[r];
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 16; ++r) v[r] = ex[rd3 + 17 * r];
                const uint64_t ct = ((uint64_t)q.b0 + (uint64_t)c + (uint64_t)C * b) & mask;
                float2 b1, b2, b4, b8;
                if (q.twp) {
                    const float2* __restrict__ pw = q.twp + (size_t)c * 1024 + j;
                    b1 = __ldg(pw), b2 = __ldg(pw + 256), b4 = __ldg(pw + 512), b8 = __ldg(pw + 768);
                } else {
                    b1 = twiddle_N(ct, N), b2 = twiddle_N((2 * ct) & mask, N);
                    b4 = twiddle_N((4 * ct) & mask, N), b8 = twiddle_N((8 * ct) & mask, N);
                }
                const float2 b3 = cmul(b2, b1), b12 = cmul(b8, b4);
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
                dft16_lo8(v);
                float2 ph = twiddle_N((ct * s0) & mask, N);
                const int* __restrict__ km = q.kmap + (size_t)c * 2048 + b;
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int k = __ldg(km + 256 * r);
                    if (k >= 0) (DIRECT ? Fo : row)[k] = cmul(v[r], ph);
                    ph = cmul(ph, phs);
                }
            }
            if (!last) group_sync(grp);   // the next round's first pass rewrites the exchange buffer
        }
        if (zero) {
            for (int i = tid; i < (int)q.N_f; i += SR_THREADS) Fo[i] = make_float2(0.f, 0.f);
        } else if constexpr (!DIRECT) {
            if (q.bulk) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (!q.bulk) {
                for (int i = tid; i < (int)q.N_f; i += SR_THREADS) Fo[i] = row[i];
            } else if (tid == 0) {
                bulk_store(Fo, row, (uint32_t)q.N_f * 8u);
            }
        }
        cur = s_next;
        __syncthreads();   // the row buffer (or its copy is under way), the exchange buffers and s_next are free
    }
    if (tid == 0) bulk_store_read();
}

constexpr size_t SR_SMEM = 226 * 1024;

size_t rows_layout(const cc_plan* plan, RowsArgs* q, bool direct) {
    const DevParams& p = plan->dp;
    const int esz = p.store == CC_STORE_BF16 ? 4 : 8;
    auto al = [](size_t b) { return (b + 127) & ~(size_t)127; };
    q->row_bytes = (uint32_t)(p.N_s * esz);
    size_t o = (size_t)SR_L * esz;
    q->off_ex = (uint32_t)o;
    o += (size_t)2 * SR_EX * sizeof(float2);
    q->off_row = (uint32_t)o;
    if (!direct) o = al(o + (size_t)p.N_f * sizeof(float2));
    q->off_bar = (uint32_t)o;
    return o + 16;
}

}  // namespace

// Whole segments (N_s <= 4096) on 4096-point cosets (the plan's own, or zero-padded when the plan
// is tuned to transform_len 4096), Q <= 2, output bins in the lower half of each coset transform
// (the plan's tables exist where these hold, plan.cu); rows of whole 16-byte pieces from a
// 16-byte boundary for the bulk copies.
bool segfft_rows_supported(const cc_plan* plan, const void* ab) {
    const DevParams& p = plan->dp;
    const bool padded = p.L < SR_L && plan->tuning.transform_len == SR_L && p.C4 > 0;
    if ((p.L != SR_L && !padded) || !plan->rows_kmap) return false;
    return p.N_s % (p.store == CC_STORE_BF16 ? 4 : 2) == 0 && ((uintptr_t)ab & 15) == 0;
}

cc_status launch_segfft_rows(cc_plan* plan, int64_t n_t, const void* ab, float2* F, int* counter, cudaStream_t st) {
    const DevParams& p = plan->dp;
    RowsArgs q;
    const bool direct = rows_layout(plan, &q, false) > SR_SMEM;
    const size_t smem = rows_layout(plan, &q, direct);
    q.ab = ab;
    q.F = F;
    q.ctr = counter;
    q.err = p.err;
    q.twk = p.twk;
    q.twp = plan->rows_twp;
    q.kmap = plan->rows_kmap;
    q.N_FFT = p.N_FFT;
    q.b0 = p.b0;
    q.N_tau = p.N_tau;
    q.M = p.M;
    q.N_s = p.N_s;
    q.N_f = p.N_f;
    q.rows = n_t * p.Q * p.M * 2;
    q.Q = p.Q;
    q.C = p.C4;
    q.wait_test = p.wait_test;
    if (q.rows > 0x7fffffff - 65536) return fail(CC_ERR_UNSUPPORTED, "too many segment transforms in one launch");
    q.bulk = q.N_f % 2 == 0 && ((uintptr_t)F & 15) == 0;
    const bool bf16 = p.store == CC_STORE_BF16;
    void (*const kern)(RowsArgs) = bf16 ? (direct ? segfft_rows_kernel<true, true> : segfft_rows_kernel<true, false>)
                                        : (direct ? segfft_rows_kernel<false, true> : segfft_rows_kernel<false, false>);
    int dev = 0, sms = 152;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return cuda_fail(e, "segment FFT set-up");
    const unsigned grid = (unsigned)std::min<int64_t>(sms, q.rows);
    kern<<<grid, SR_THREADS, smem, st>>>(q);
    count_launch();
    e = cudaGetLastError();
    return e == cudaSuccess ? CC_OK : cuda_fail(e, "segment FFT (rows) launch");
}

}  // namespace cc
