// Two-pass search: the resampling kernel writes the weighted source-frame series a_r, b_r of
// a template batch to HBM; corr_kernel forms every segment's spectrum on the lag grid and
// sums the pair products there (corr_kernel.cuh says why that grid is enough); this file
// turns those sums into rho at the output bins:
//
//   corr_lags_kernel   sums the partial rows of a template, inverse transform per coset to
//                      lags, and the template's normalisation;
//   corr_merge_kernel  the lag sequence from the cosets (more than one);
//   corr_rho_kernel    one coset of the N_FFT-point output transform of the lag sequence,
//                      normalised at the output bins.
//
// With a(l) and b(l) the inverse transforms of A and B, the pair sum at bin k is
//   rho_raw(k) = Re sum_(n = 0)^(2 N_s - 1) h(n) W_N^(k n),
//   h(0) = a(0), h(n) = 2 a(n) [n < N_s] + conj(b(N_s - n)) [n >= 1]
// (a(-l) = conj(a(l)) because A is real; a pair of consecutive segments carries the phase
// W_N^(-k N_s) of their distance; b counts twice with every ordered pair).
//
// These three work on numbers of two floats (twofloat.cuh).  A and B hold the power of every
// frequency of the series, in the searched band or not, and a transform spreads the rounding of
// the loudest of them over all lags and from there over all output bins: in FP32 a line of three
// times the noise outside the band left errors of 0.08 in rho, where sums at the output bins
// leave 1e-5, because there the rounding is relative to the spectra's amplitude.  Bound by the
// FP32 pipe (about twelve operations for one of FP64, whose rate here is 1/64) and, for few
// templates, by latency.  A pass with them in two floats against FP32: 144 templates of the 120-day
// band 40.6 against 40.3 ms, 4 templates of an hour 59 against 56 us.
#include <algorithm>

#include "corr.cuh"
#include "segpair.cuh"
#include "tma.cuh"
#include "twofloat.cuh"

namespace cc {

cc_status launch_resample(cc_plan* plan, const cc_template* t_dev, int64_t n_t, void* ab, float* norm,
                          cudaStream_t st, const KnotRec* kn = nullptr, int64_t nkn = 0, int write_inactive = 0,
                          uint8_t* act = nullptr, int t_pad = 0);
cc_status launch_knots(cc_plan* plan, const cc_template* t_dev, int64_t n_t, KnotRec* kn, cudaStream_t st,
                       int* zero_word = nullptr);
cc_status launch_norm(cc_plan* plan, const float* norm, int64_t n_t, double* Dws, cudaStream_t st);
cc_status launch_pair_finalize(cc_plan* plan, const float* raw, const double* Dws, int n_rows, int64_t n_t,
                               float* rho, cudaStream_t st);
int64_t fold_count(const cc_plan* plan);
cc_status launch_fold(cc_plan* plan, int64_t n_t, const void* ab, const uint8_t* act, int t_pad, float2* z,
                      cudaStream_t st);

CC_CORR_INST(extern, 128)
CC_CORR_INST(extern, 256)
CC_CORR_INST(extern, 512)
CC_CORR_INST(extern, 1024)
CC_CORR_INST(extern, 2048)
CC_CORR_INST(extern, 4096)
CC_CORR_INST_FULL(extern)
CC_CORR_INST_MULTI(extern, 256)
CC_CORR_INST_MULTI(extern, 512)
CC_CORR_INST_MULTI(extern, 1024)
CC_CORR_INST_MULTI(extern, 2048)
CC_CORR_INST_MULTI(extern, 4096)
CC_CORR_INST_MULTI_FULL(extern)

constexpr size_t TWO_PASS_WS_BUDGET = (size_t)24 << 30;   // a_r, b_r (and folded rows) of one template batch
constexpr size_t SHARED_WS_BUDGET = (size_t)4 << 30;      // the same for plans that the cluster or stage kernels serve too
constexpr int LAG_THREADS = 256;
constexpr int LAG_MAX_THREADS = 1024;   // the two-float transforms: a radix-4 butterfly a thread, at least LAG_THREADS
constexpr int ROW_BLOCK = 32;        // partial rows summed by one block of corr_rows_kernel

// What the kernels after corr_kernel need.
struct LagArgs {
    const float* raw;       // [n_t][n_rows][planes][2][G]: partial sums and what they round off
    ffc* U;                 // [n_t][planes > 1 ? 2 : 1][C][L]: per coset the inverse transform of A and B
    ffc* h;                 // [n_t][n_lags] (C > 1)
    const ffc* root;        // exp(-2 pi i j / L)
    const ffc *g_lo, *g_hi; // powers of exp(-2 pi i / G) (C > 1), see ffc_power
    const float4* norm;     // [n_t][Q][M]
    double* D;              // [n_t] sqrt(2 / normalisation), 0 without weight
    int64_t M;
    int L, log2L, C, planes, n_rows, n_lags, N_s, Q, R, pair_mode;
};

// One partial row's value at p, its second word G further on
__device__ __forceinline__ ff row_value(const float* __restrict__ p, size_t G) { return make_float2(__ldg(p), __ldg(p + G)); }

// Sum of ROW_BLOCK partial rows (few templates have many): out [n_t][gridDim.y][planes][2][G], four
// neighbouring values a thread.
__global__ void __launch_bounds__(LAG_THREADS)
corr_rows_kernel(const float* __restrict__ raw, int n_rows, int planes, int G, float* __restrict__ out) {
    const int i = 4 * (blockIdx.x * LAG_THREADS + threadIdx.x);
    const size_t t = blockIdx.z;
    if (i >= planes * G) return;
    const int pl = i / G, m = i - pl * G;
    const int r0 = blockIdx.y * ROW_BLOCK, r1 = min(n_rows, r0 + ROW_BLOCK);
    const size_t stride = (size_t)planes * 2 * G;
    const float* p = raw + t * n_rows * stride + (size_t)pl * 2 * G + m;
    ff s[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int r = r0; r < r1; ++r) {
        const float4 h = __ldg((const float4*)(p + r * stride)), l = __ldg((const float4*)(p + r * stride + G));
        s[0] = ff_add(s[0], make_float2(h.x, l.x));
        s[1] = ff_add(s[1], make_float2(h.y, l.y));
        s[2] = ff_add(s[2], make_float2(h.z, l.z));
        s[3] = ff_add(s[3], make_float2(h.w, l.w));
    }
    float* const o = out + ((t * gridDim.y + blockIdx.y) * planes + pl) * 2 * (size_t)G + m;
    *(float4*)o = make_float4(s[0].x, s[1].x, s[2].x, s[3].x);
    *(float4*)(o + G) = make_float4(s[0].y, s[1].y, s[2].y, s[3].y);
}

// The L roots of a block's transform into shared memory, under the loads of its input, and the
// barrier before both are read.
__device__ __forceinline__ void stage_roots(ffc* dst, const ffc* __restrict__ root, int L) {
    for (int j = threadIdx.x; j < L; j += blockDim.x) cp_async<16>(dst + j, root + j);
}
__device__ __forceinline__ void roots_staged() {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

__device__ __forceinline__ double norm_pair(float4 a, float4 b) {
    return (double)a.x * b.x + (double)a.y * b.y + 2.0 * (double)a.z * b.z;
}

// grid: x = coset c (x = C, y = 0: the normalisation factor of template z), y = A or B, z = template.
__global__ void __launch_bounds__(LAG_MAX_THREADS)
corr_lags_kernel(const LagArgs q) {
    extern __shared__ __align__(16) ffc buf[];
    const int c = blockIdx.x, ser = blockIdx.y;
    const size_t t = blockIdx.z;
    if (c == q.C) {   // sum over the pair set of A_i A_j + B_i B_j + 2 C_i C_j
        if (ser) return;
        __shared__ double red[LAG_MAX_THREADS / 32];
        const float4* nt = q.norm + t * q.Q * q.M;
        double acc = 0.0;
        for (int64_t idx = threadIdx.x; idx < q.Q * q.M; idx += blockDim.x) {
            const int Y = (int)(idx / q.M);
            const int64_t K = idx - Y * q.M;
            const float4 nY = nt[Y * q.M + K];
            double s = 0.0;
            for (int X = 0; X < Y; ++X) s += norm_pair(nt[X * q.M + K], nY);
            if (q.R > 0 && K > 0)
                for (int X = 0; X < q.Q; ++X) s += norm_pair(nt[X * q.M + K - 1], nY);
            if (q.pair_mode == CC_PAIRS_ALL_ORDERED) s = 2.0 * s + norm_pair(nY, nY);
            acc += s;
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < (int)blockDim.x / 32; ++w) s += red[w];
            q.D[t] = s > 0.0 ? 1.4142135623730951 / sqrt(s) : 0.0;
        }
        return;
    }
    const size_t G = (size_t)q.C * q.L, plane = 2 * G, stride = q.planes * plane;
    const float* p0 = q.raw + t * q.n_rows * stride + (size_t)c * q.L;
    stage_roots(buf + 2 * q.L, q.root, q.L);
    // the inverse transform as the conjugate of the forward one of the conjugate
    for (int m = threadIdx.x; m < q.L; m += blockDim.x) {
        const float* p = p0 + m + (ser ? plane : 0);
        ff re = make_float2(0.f, 0.f), im = re;
        if (ser == 0) {
#pragma unroll 8
            for (int r = 0; r < q.n_rows; ++r) re = ff_add(re, row_value(p + r * stride, G));
        } else {
#pragma unroll 4
            for (int r = 0; r < q.n_rows; ++r) {
                re = ff_add(re, row_value(p + r * stride, G));
                im = ff_add(im, row_value(p + r * stride + plane, G));
            }
        }
        buf[m] = ffc_make(re, ff_neg(im));
    }
    roots_staged();
    const ffc* res = ffc_stockham(buf, buf + q.L, q.L, q.log2L, buf + 2 * q.L);
    // times 1 / G = 1 / (C L): C is not a power of two for folded segments
    const float inv_l = 1.0f / (float)q.L;
    const ff inv_c = ff_from(1.0 / (double)q.C);
    ffc* o = q.U + ((t * (q.planes > 1 ? 2 : 1) + ser) * q.C + c) * q.L;
    for (int m = threadIdx.x; m < q.L; m += blockDim.x) {
        const ffc v = ffc_scale2(ffc_conj(res[m]), inv_l);
        o[m] = q.C == 1 ? v : ffc_make(ff_mul(ffc_re(v), inv_c), ff_mul(ffc_im(v), inv_c));
    }
}

// sum_c W_G^(-c l) u_c(l mod L): the inverse transform at lag l from those of the cosets
__device__ __forceinline__ ffc lag_value(const LagArgs& q, const ffc* __restrict__ u, int l) {
    ffc v = __ldg(u + (l & (q.L - 1)));
    for (int c = 1; c < q.C; ++c) {
        const ffc w = ffc_conj(ffc_power(q.g_lo, q.g_hi, (uint64_t)c * (uint64_t)l % ((uint64_t)q.C * q.L)));
        v = ffc_add(v, ffc_mul(__ldg(u + (size_t)c * q.L + (l & (q.L - 1))), w));
    }
    return v;
}

__device__ __forceinline__ ffc lag_h(const LagArgs& q, size_t t, int n) {
    const int G = q.C * q.L;
    const ffc* u = q.U + t * (q.planes > 1 ? 2 : 1) * G;
    ffc h = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n < q.N_s) {
        const ffc a = lag_value(q, u, n);
        h = n > 0 ? ffc_scale2(a, 2.f) : a;
    }
    if (q.planes > 1 && n > 0) {
        const int l = q.N_s - n;
        const ffc b = ffc_conj(lag_value(q, u + G, l < 0 ? l + G : l));
        h = ffc_add(h, q.pair_mode == CC_PAIRS_ALL_ORDERED ? ffc_scale2(b, 2.f) : b);
    }
    return h;
}

__global__ void __launch_bounds__(LAG_THREADS)
corr_merge_kernel(const LagArgs q) {
    const int n = blockIdx.x * LAG_THREADS + threadIdx.x;
    const size_t t = blockIdx.y;
    if (n < q.n_lags) q.h[t * q.n_lags + n] = lag_h(q, t, n);
}

// Output bins b0 + c + C m (the plan's coset lists), one coset per block: position p takes
// sum_f h(p + f L) W_N^((b0 + c)(p + f L)), an L-point transform gives the bins.  L and root are
// the plan's; n_lo, n_hi: powers of exp(-2 pi i / N).
// grid: x = coset, y = template.
__global__ void __launch_bounds__(LAG_MAX_THREADS)
corr_rho_kernel(const LagArgs q, int L, int log2L, const ffc* __restrict__ root, const ffc* __restrict__ n_lo,
                const ffc* __restrict__ n_hi, int64_t N_FFT, int64_t b0, const int* __restrict__ off,
                const int* __restrict__ ck, const int* __restrict__ cm, int64_t N_f, float* __restrict__ rho) {
    extern __shared__ __align__(16) ffc buf[];
    const int c = blockIdx.x;
    const size_t t = blockIdx.y;
    stage_roots(buf + 2 * L, root, L);
    const uint64_t mask = (uint64_t)N_FFT - 1;
    const uint64_t bc = ((uint64_t)b0 + (uint64_t)c) & mask;
    for (int pos = threadIdx.x; pos < L; pos += blockDim.x) {
        ffc acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
        for (int n = pos; n < q.n_lags; n += L) {
            const ffc h = q.h ? __ldg(q.h + t * q.n_lags + n) : lag_h(q, t, n);
            acc = ffc_add(acc, ffc_mul(h, ffc_power(n_lo, n_hi, (bc * (uint64_t)n) & mask)));
        }
        buf[pos] = acc;
    }
    roots_staged();
    const ffc* res = ffc_stockham(buf, buf + L, L, log2L, buf + 2 * L);
    const double sc = q.D[t];
    const int e = __ldg(off + c + 1);
    for (int i = __ldg(off + c) + threadIdx.x; i < e; i += blockDim.x) {
        const ffc v = res[__ldg(cm + i)];
        rho[t * N_f + __ldg(ck + i)] = sc > 0.0 ? (float)(((double)v.x + (double)v.y) * sc) : 0.f;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }
static size_t al128(size_t b) { return (b + 127) & ~(size_t)127; }

struct CorrLayout {
    int L, C, T, half, padded, folded, bf16_rows, planes, n_rows, n_blocks, n_lags;
    int64_t G, t_pad;
    CorrArgs a;
    // workspace pieces of a batch, bytes
    size_t ab, z, norm, act, D, raw, rows2, U, h, kn, total;
};

std::vector<float2> corr_powers(int64_t L, int64_t C) {
    if (L < 16) return {};   // no pass of 16 points a thread
    const int64_t GT = L / 16, RL = L >= 512 ? L / 256 : L / 16, nb = 16 / RL, G = C * L;
    int np = 0;
    while ((1 << np) < RL) ++np;
    std::vector<float2> v((size_t)(C * nb * np * GT));
    for (int64_t c = 0; c < C; ++c)
        for (int64_t i = 0; i < nb; ++i)
            for (int n = 0; n < np; ++n)
                for (int64_t j = 0; j < GT; ++j) {
                    // the thread's butterfly: column k, row i0 + RL i of the second pass's outputs
                    const int64_t b = L >= 512 ? 16 * ((j & 15) % RL + RL * i) + (j >> 4) + RL * ((j & 15) / RL) : j + GT * i;
                    const double a = -2.0 * M_PI * (double)(((c + C * b) << n) % G) / (double)G;
                    v[(size_t)(((c * nb + i) * np + n) * GT + j)] = make_float2((float)cos(a), (float)sin(a));
                }
    return v;
}

// Whether the plan takes the two-pass kernels by name (CC_PATH_TWO_PASS): Q <= 2, R <= 1, no
// cross-only pair set, coset length 64..4096, every bin in the lower half of its coset.
bool two_pass_supported(const cc_plan* plan) {
    const DevParams& p = plan->dp;
    if (p.Q > 2 || p.R > 1 || p.pair_mode == CC_PAIRS_CROSS_ONLY) return false;
    if (p.L < 64 || p.L > 4096 || plan->N_f < 1) return false;
    return 2 * ((plan->kbar.back() - plan->k0) / p.C) < p.L;
}

// Whether the lag grid serves the plan: the conditions of two_pass_supported but any output bins
// (the last transform reaches all of them); with three or four detectors FP32 storage and at
// least 256-point transforms (one activity bit per detector and template of a series group).
// Asked at plan creation too, before the kernel parameters are filled.
bool lag_grid_supported(const cc_plan* plan) {
    if (plan->R > 1 || plan->cfg.pair_mode == CC_PAIRS_CROSS_ONLY || plan->L < 64 || plan->L > 4096 || plan->N_f < 1) return false;
    return plan->Q <= 2 || (plan->cfg.store == CC_STORE_FP32 && plan->L >= 128);
}

static int sm_count() {
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// The fewest segment chunks a search can be split into.
static int64_t least_chunks(const cc_plan* plan) { return (plan->M + CORR_MAX_CHUNK - 1) / CORR_MAX_CHUNK; }

// Grid, shared memory, chunk split (of at most max_chunks chunks, where the kernel can do with as
// few) and workspace of a batch of n_t templates.
static void corr_layout(const cc_plan* plan, int64_t n_t, int64_t max_chunks, CorrLayout* y) {
    const DevParams& p = plan->dp;
    const bool padded = plan->tuning.transform_len == CORR_POINTS && p.L < CORR_POINTS;
    y->padded = padded;
    y->folded = p.N_s > CORR_POINTS;
    y->half = 2 * p.N_s <= CORR_POINTS;
    y->L = y->half && !padded ? 2 * p.L : CORR_POINTS;
    y->C = y->folded ? 2 * (int)fold_count(plan) : y->half ? 1 : 2;
    y->T = CORR_POINTS / y->L;
    y->G = (int64_t)y->C * y->L;
    y->planes = p.R > 0 ? 3 : 1;
    y->n_lags = (int)(p.R > 0 ? 2 * p.N_s : p.N_s);
    y->bf16_rows = !y->folded && p.store == CC_STORE_BF16;
    y->t_pad = (n_t + 15) & ~(int64_t)15;
    const int esz = y->bf16_rows ? 4 : 8;
    CorrArgs& a = y->a;
    a = CorrArgs{};
    a.n_in = y->folded ? CORR_POINTS : (int)p.N_s;
    a.row_bytes = (uint32_t)(a.n_in * esz);
    a.row_stride = (uint32_t)((y->half ? y->L / 2 : y->L) * esz);   // whole inputs, zero beyond the samples
    a.tma = a.row_bytes % 16 == 0;   // bulk copies: rows of whole 16-byte pieces start on 16-byte boundaries
    size_t o = al128((size_t)y->T * a.row_stride);
    a.off_y = (uint32_t)o;
    o = al128(o + (size_t)2 * corr_buffer(y->T) * sizeof(float2));
    a.off_tw = (uint32_t)o;
    o += (272 + 1024) * sizeof(float2);
    a.off_act = (uint32_t)o;
    o += (CORR_MAX_CHUNK + 1) * corr_act_bytes(y->T);
    a.off_bar = (uint32_t)o;
    a.smem = (uint32_t)(o + 16);
    // Chunks of segments: units are equal, handed out one by one to two CTAs per SM, each
    // rereads its first segment's predecessor (R = 1) and writes one row (98 KB with a lag, written
    // and read again: about the time of four segments): the count with the least
    // ceil(units / slots) (length + overhead); with cc_tuning.chunk_waves, that many units per
    // slot, at most M / (4 R + 1) chunks.
    const int64_t slots = (int64_t)CORR_CTAS_PER_SM * sm_count();
    const int64_t per_chunk = (2 * n_t + y->T - 1) / y->T * y->C;
    // rows beyond ROW_BLOCK are summed first (a launch, about three segments' time) where the blocks
    // of corr_lags_kernel do not fill the chip
    const bool pre_sum = n_t * y->C * (y->planes > 1 ? 2 : 1) < sm_count();
    const int64_t minch = least_chunks(plan);
    const int64_t maxch = std::max<int64_t>(minch, p.M);
    int64_t nch = minch;
    if (plan->tuning.chunk_waves > 0) {
        nch = std::max(minch, std::min<int64_t>(std::max<int64_t>(1, p.M / (4 * p.R + 1)), (plan->tuning.chunk_waves * slots + per_chunk - 1) / per_chunk));
    } else {
        const int64_t most = std::max(minch, std::min<int64_t>(maxch, (32 * slots + per_chunk - 1) / per_chunk));
        int64_t best = -1;
        for (int64_t n = minch; n <= most; n += 1 + n / 16) {
            const int64_t len = (p.M + n - 1) / n, waves = (per_chunk * ((p.M + len - 1) / len) + slots - 1) / slots;
            const int64_t cost = waves * (len + p.R + (y->planes > 1 ? 4 : 2)) + (2 * n > ROW_BLOCK && pre_sum ? 3 : 0);
            if (best < 0 || cost < best) {
                best = cost;
                nch = n;
            }
        }
    }
    nch = std::max(minch, std::min(nch, max_chunks));
    a.chunk_len = (int)((p.M + nch - 1) / nch);
    a.n_chunks = (int)((p.M + a.chunk_len - 1) / a.chunk_len);
    y->n_rows = 2 * a.n_chunks;
    const size_t b = (size_t)n_t;
    y->ab = al256(b * plan->Q * 2 * plan->N_tau * (plan->cfg.store == CC_STORE_BF16 ? 4 : 8));
    y->z = y->folded ? al256(b * plan->Q * 2 * plan->M * y->G * esz) : 0;
    y->norm = al256(b * plan->Q * plan->M * sizeof(float4));
    y->act = al256((size_t)plan->Q * plan->M * y->t_pad);
    y->D = al256(b * sizeof(double));
    y->raw = al256(b * y->n_rows * y->planes * 2 * y->G * sizeof(float));
    // (held for any batch of that many rows, so that the bytes of a chunk split grow with the batch)
    const int blocks = y->n_rows > ROW_BLOCK ? (y->n_rows + ROW_BLOCK - 1) / ROW_BLOCK : 0;
    y->n_blocks = pre_sum ? blocks : 0;
    y->rows2 = al256(b * blocks * y->planes * 2 * y->G * sizeof(float));
    y->U = al256(b * (y->planes > 1 ? 2 : 1) * y->G * sizeof(ffc));
    y->h = y->C > 1 ? al256(b * y->n_lags * sizeof(ffc)) : 0;
    y->kn = al256(b * plan->Q * knot_rows(plan) * sizeof(KnotRec));
    y->total = y->ab + y->z + y->norm + y->act + y->D + y->raw + y->rows2 + y->U + y->h + y->kn + 256;
}

// Templates per batch: as many as the budget of a_r, b_r and folded rows holds.
static int64_t two_pass_batch(const cc_plan* plan, int64_t n_t) {
    const size_t ab = (size_t)plan->Q * 2 * plan->N_tau * (plan->cfg.store == CC_STORE_BF16 ? 4 : 8);
    const size_t z = segpair_tma_supported(plan) ? segpair_tma_fold_bytes(plan)
                     : plan->N_s > CORR_POINTS   ? (size_t)plan->Q * 2 * plan->M * 2 * fold_count(plan) * CORR_POINTS * 8
                                                 : 0;
    const int64_t b = plan->tuning.batch_templates > 0
                          ? plan->tuning.batch_templates
                          : (int64_t)std::max<size_t>(1, (two_pass_supported(plan) ? TWO_PASS_WS_BUDGET : SHARED_WS_BUDGET) / (ab + z));
    return std::max<int64_t>(1, std::min<int64_t>({b, n_t, 65535}));
}

// Folded segments in BF16 (segpair_tma.cu): batch, chunks and workspace.
struct FoldedLayout {
    int64_t batch, chunk_len;
    int n_chunks;
    size_t ab, z, norm, D, raw, kn, total;
};

static void folded_chunks(const cc_plan* plan, int64_t n_t, int64_t max_chunks, FoldedLayout* y) {
    const int64_t nch = std::max<int64_t>(least_chunks(plan), std::min<int64_t>(segpair_tma_chunks(plan, n_t), max_chunks));
    y->chunk_len = (plan->M + nch - 1) / nch;
    y->n_chunks = (int)((plan->M + y->chunk_len - 1) / y->chunk_len);
}

static void folded_layout(const cc_plan* plan, int64_t batch, int64_t max_chunks, FoldedLayout* y) {
    y->batch = batch;
    folded_chunks(plan, batch, max_chunks, y);
    const size_t b = (size_t)batch;
    y->ab = al256((size_t)plan->Q * 2 * plan->N_tau * 4 * b);
    y->z = al256(segpair_tma_fold_bytes(plan) * b);
    y->norm = al256(b * plan->Q * plan->M * sizeof(float4));
    y->D = al256(b * sizeof(double));
    y->raw = al256(b * 2 * y->n_chunks * plan->N_f * sizeof(float));
    y->kn = al256(b * plan->Q * knot_rows(plan) * sizeof(KnotRec));
    y->total = y->ab + y->z + y->norm + y->D + y->raw + y->kn + al256((size_t)plan->dp.C4 * sizeof(int));
}

// How a search is split: templates per batch and the largest number of segment chunks.
struct Split {
    int64_t batch, chunks;
};

static size_t split_bytes(const cc_plan* plan, int64_t n_t, Split f) {
    if (segpair_tma_supported(plan)) {
        FoldedLayout y;
        folded_layout(plan, f.batch, f.chunks, &y);
        return y.total;
    }
    CorrLayout y;
    corr_layout(plan, f.batch, f.chunks, &y);
    size_t bytes = y.total;
    if (n_t % f.batch) {   // the last batch may split its segments into more chunks
        corr_layout(plan, n_t % f.batch, f.chunks, &y);
        bytes = std::max(bytes, y.total);
    }
    return bytes;
}

// The split of a search of n_t templates: the fastest one, or, with less memory than that takes,
// fewer chunks (the partial rows of a search of few templates can be most of its bytes).  With the
// fewest chunks the bytes grow with the templates, so memory that holds n of them in some split
// holds any smaller number.  Plans that other kernels serve in little memory (more than two
// detectors, bands over both coset halves) then take fewer templates at once, down to one: the
// cluster kernel needs a few MB for any search, at 20 to 30 times the time on large ones.  batch 0:
// does not fit.
static Split fit_split(const cc_plan* plan, int64_t n_t, size_t avail) {
    Split f{two_pass_batch(plan, n_t), plan->M};   // as many chunks as pay
    if (split_bytes(plan, n_t, f) <= avail) return f;
    const int64_t least = least_chunks(plan);
    while (f.chunks > least) {
        f.chunks = std::max(least, f.chunks * 3 / 4);
        if (split_bytes(plan, n_t, f) <= avail) return f;
    }
    int64_t fits = 0, over = f.batch;
    while (!two_pass_supported(plan) && over - fits > 1) {
        f.batch = fits + (over - fits) / 2;
        (split_bytes(plan, f.batch, f) <= avail ? fits : over) = f.batch;
    }
    return Split{fits, least};
}

// The split to search n_t templates with, and its workspace: the plan's own memory grows to the
// fastest split's; the caller's, and the plan's while its stream is captured (when nothing can be
// allocated), is taken as it is.
static cc_status claim_split(cc_plan* plan, int64_t n_t, cudaStream_t st, Split* f) {
    *f = Split{two_pass_batch(plan, n_t), plan->M};
    const size_t need = split_bytes(plan, n_t, *f);
    if (plan->ws_bytes >= need) return CC_OK;
    bool fixed = plan->ws_external;
    if (!fixed && plan->ws_bytes > 0) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) cudaGetLastError();
        fixed = cap == cudaStreamCaptureStatusActive;
    }
    if (!fixed) return ensure_workspace(plan, need);
    const Split g = fit_split(plan, n_t, plan->ws_bytes);
    if (g.batch < 1)
        return fail(CC_ERR_OOM, "workspace of " + std::to_string(plan->ws_bytes) + " bytes; this call needs " + std::to_string(need));
    *f = g;
    return CC_OK;
}

// Whether the two-pass kernels can search n_t templates of a plan that other kernels serve too, with
// the memory they need claimed.
bool two_pass_claim(cc_plan* plan, int64_t n_t, cudaStream_t st) {
    Split f;
    return claim_split(plan, n_t, st, &f) == CC_OK;
}

static cc_status search_folded_bf16(cc_plan* plan, const cc_template* t_dev, int64_t n_t, float* rho, cudaStream_t st) {
    Split f;
    cc_status s = claim_split(plan, n_t, st, &f);
    if (s != CC_OK) return s;
    FoldedLayout y;
    folded_layout(plan, f.batch, f.chunks, &y);
    char* w = (char*)plan->ws;
    void* ab = w;
    void* z = w += y.ab;
    float* norm = (float*)(w += y.z);
    double* D = (double*)(w += y.norm);
    float* raw = (float*)(w += y.D);
    KnotRec* kn = (KnotRec*)(w += y.raw);
    int* counters = (int*)(w += y.kn);
    for (int64_t t0 = 0; t0 < n_t; t0 += y.batch) {
        const int64_t nb = std::min(y.batch, n_t - t0);
        FoldedLayout b = y;
        folded_chunks(plan, nb, f.chunks, &b);   // chunking for this batch size (workspace sized for the largest)
        if (b.n_chunks > y.n_chunks) b = y;
        if ((s = launch_knots(plan, t_dev + t0, nb, kn, st)) != CC_OK) return s;
        if ((s = launch_resample(plan, t_dev + t0, nb, ab, norm, st, kn, knot_rows(plan))) != CC_OK) return s;
        if ((s = launch_norm(plan, norm, nb, D, st)) != CC_OK) return s;
        cudaEvent_t ev0, ev1;
        timing_pair(plan, &ev0, &ev1);
        if (ev0) cudaEventRecord(ev0, st);
        s = launch_fold_bf16(plan, nb, ab, (const float4*)norm, z, st);
        if (s == CC_OK) s = launch_segpair_tma(plan, b.n_chunks, b.chunk_len, nb, z, (const float4*)norm, raw, counters, st);
        if (ev1) cudaEventRecord(ev1, st);
        if (s != CC_OK) return s;
        if ((s = launch_pair_finalize(plan, raw, D, 2 * b.n_chunks, nb, rho + t0 * plan->N_f, st)) != CC_OK) return s;
    }
    return CC_OK;
}

size_t two_pass_workspace_bytes(const cc_plan* plan, int64_t n_t) {
    return n_t < 1 ? 0 : split_bytes(plan, n_t, Split{two_pass_batch(plan, n_t), plan->M});
}

template <bool BF16, bool LAG>
static cudaError_t launch_corr_l(const CorrLayout& y, int sms, cudaStream_t st) {
    if (!y.half) return launch_corr_t<4096, BF16, LAG, false, false>(y.a, sms, st);
    switch (y.L) {
        case 128: return launch_corr_t<128, BF16, LAG, true, false>(y.a, sms, st);
        case 256: return launch_corr_t<256, BF16, LAG, true, false>(y.a, sms, st);
        case 512: return launch_corr_t<512, BF16, LAG, true, false>(y.a, sms, st);
        case 1024: return launch_corr_t<1024, BF16, LAG, true, false>(y.a, sms, st);
        case 2048: return launch_corr_t<2048, BF16, LAG, true, false>(y.a, sms, st);
        case 4096: return launch_corr_t<4096, BF16, LAG, true, false>(y.a, sms, st);
    }
    return cudaErrorInvalidValue;
}

template <bool LAG>
static cudaError_t launch_corr_multi(const CorrLayout& y, int sms, cudaStream_t st) {
    if (!y.half) return launch_corr_t<4096, false, LAG, false, true>(y.a, sms, st);
    switch (y.L) {
        case 256: return launch_corr_t<256, false, LAG, true, true>(y.a, sms, st);
        case 512: return launch_corr_t<512, false, LAG, true, true>(y.a, sms, st);
        case 1024: return launch_corr_t<1024, false, LAG, true, true>(y.a, sms, st);
        case 2048: return launch_corr_t<2048, false, LAG, true, true>(y.a, sms, st);
        case 4096: return launch_corr_t<4096, false, LAG, true, true>(y.a, sms, st);
    }
    return cudaErrorInvalidValue;
}

static cudaError_t launch_corr(const CorrLayout& y, cudaStream_t st) {
    const int sms = sm_count();
    if (y.a.Q > 2) return y.planes > 1 ? launch_corr_multi<true>(y, sms, st) : launch_corr_multi<false>(y, sms, st);
    if (y.bf16_rows) return y.planes > 1 ? launch_corr_l<true, true>(y, sms, st) : launch_corr_l<true, false>(y, sms, st);
    return y.planes > 1 ? launch_corr_l<false, true>(y, sms, st) : launch_corr_l<false, false>(y, sms, st);
}

cc_status search_two_pass(cc_plan* plan, const cc_template* t_dev, int64_t n_t, float* rho, cudaStream_t st) {
    if (segpair_tma_supported(plan)) return search_folded_bf16(plan, t_dev, n_t, rho, st);
    const DevParams& p = plan->dp;
    Split f;
    cc_status s = claim_split(plan, n_t, st, &f);
    if (s != CC_OK) return s;
    cudaError_t e;
    for (int64_t t0 = 0; t0 < n_t; t0 += f.batch) {
        const int64_t nb = std::min(f.batch, n_t - t0);
        CorrLayout y;
        corr_layout(plan, nb, f.chunks, &y);
        const int64_t units = (2 * nb + y.T - 1) / y.T * y.C * y.a.n_chunks;
        if (units > 0x7fffffff) return fail(CC_ERR_UNSUPPORTED, "too many work units in one launch");
        char* w = (char*)plan->ws;
        auto take = [&](size_t bytes) {
            char* r = w;
            w += bytes;
            return r;
        };
        void* ab = take(y.ab);
        void* z = take(y.z);
        float* norm = (float*)take(y.norm);
        uint8_t* act = (uint8_t*)take(y.act);
        double* D = (double*)take(y.D);
        float* raw = (float*)take(y.raw);
        float* rows2 = (float*)take(y.rows2);
        ffc* U = (ffc*)take(y.U);
        ffc* h = (ffc*)take(y.h);
        KnotRec* kn = (KnotRec*)take(y.kn);
        int* ctr = (int*)take(256);
        if ((s = launch_knots(plan, t_dev + t0, nb, kn, st, ctr)) != CC_OK) return s;
        if ((s = launch_resample(plan, t_dev + t0, nb, ab, norm, st, kn, knot_rows(plan), 0, act, (int)y.t_pad)) != CC_OK)
            return s;
        cudaEvent_t ev0, ev1;
        timing_pair(plan, &ev0, &ev1);
        if (ev0) cudaEventRecord(ev0, st);
        if (y.folded && (s = launch_fold(plan, nb, ab, act, (int)y.t_pad, (float2*)z, st)) != CC_OK) {
            if (ev1) cudaEventRecord(ev1, st);
            return s;
        }
        CorrArgs& a = y.a;
        a.src = y.folded ? z : ab;
        a.act = act;
        a.raw = raw;
        a.ctr = ctr;
        a.err = p.err;
        a.twk = plan->corr_twk;
        a.twp = y.padded ? plan->corr_twp4096 : plan->corr_twp;
        a.N_s = p.N_s;
        a.M = (int)p.M;
        a.N_tau = p.N_tau;
        a.n_t = (int)nb;
        a.t_pad = (int)y.t_pad;
        a.Q = p.Q;
        a.C = y.C;
        a.units = (int)units;
        a.folded = y.folded;
        a.all_ordered = p.pair_mode == CC_PAIRS_ALL_ORDERED;
        a.wait_test = p.wait_test;
        e = launch_corr(y, st);
        count_launch();
        if (ev1) cudaEventRecord(ev1, st);
        if (e != cudaSuccess) return cuda_fail(e, "pair products launch");
        LagArgs q;
        q.raw = raw;
        q.n_rows = y.n_rows;
        if (y.n_blocks) {
            corr_rows_kernel<<<dim3((unsigned)launch_blocks_for(y.planes * y.G, 4 * LAG_THREADS), (unsigned)y.n_blocks, (unsigned)nb),
                               LAG_THREADS, 0, st>>>(raw, y.n_rows, y.planes, (int)y.G, rows2);
            count_launch();
            q.raw = rows2;
            q.n_rows = y.n_blocks;
        }
        q.U = U;
        q.h = y.C > 1 ? h : nullptr;
        q.root = y.padded ? plan->corr_root4096 : plan->corr_root;
        q.g_lo = plan->corr_glo;
        q.g_hi = plan->corr_ghi;
        q.norm = (const float4*)norm;
        q.D = D;
        q.M = p.M;
        q.L = y.L;
        q.log2L = 0;
        while ((1 << q.log2L) < y.L) ++q.log2L;
        q.C = y.C;
        q.planes = y.planes;
        q.n_lags = y.n_lags;
        q.N_s = (int)p.N_s;
        q.Q = p.Q;
        q.R = (int)p.R;
        q.pair_mode = p.pair_mode;
        const size_t sm1 = (size_t)3 * y.L * sizeof(ffc), sm2 = (size_t)3 * p.L * sizeof(ffc);
        const int thr1 = std::max(LAG_THREADS, y.L / 4), thr2 = std::max(LAG_THREADS, p.L / 4);
        const int big = (int)(3 * CORR_POINTS * sizeof(ffc));
        if ((sm1 > 32 * 1024 && (e = cudaFuncSetAttribute(corr_lags_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, big)) != cudaSuccess) ||
            (sm2 > 32 * 1024 && (e = cudaFuncSetAttribute(corr_rho_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, big)) != cudaSuccess))
            return cuda_fail(e, "lag kernels smem attribute");
        corr_lags_kernel<<<dim3((unsigned)(y.C + 1), y.planes > 1 ? 2u : 1u, (unsigned)nb), thr1, sm1, st>>>(q);
        count_launch();
        if (y.C > 1) {
            corr_merge_kernel<<<dim3((unsigned)launch_blocks_for(y.n_lags, LAG_THREADS), (unsigned)nb), LAG_THREADS, 0, st>>>(q);
            count_launch();
        }
        corr_rho_kernel<<<dim3((unsigned)p.C, (unsigned)nb), thr2, sm2, st>>>(
            q, p.L, p.log2L, plan->corr_rootL, plan->corr_nlo, plan->corr_nhi, p.N_FFT, p.b0, p.coset_off, p.coset_k, p.coset_m,
            p.N_f, rho + t0 * plan->N_f);
        count_launch();
        if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "lag kernels launch");
    }
    return CC_OK;
}

}  // namespace cc
