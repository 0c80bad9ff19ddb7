// Top-k of rho over (template, bin): descending rho, ties by flat index ascending.
//
// Pass 1: each block scans a contiguous slice, keeps its best KP entries in shared
// memory and admits a new element only if it beats the current KP-th best, merging
// the admitted candidates by a bitonic sort when the candidate buffer fills.
// Pass 2: one block merges the per-block lists the same way.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "common.cuh"

namespace cc {

constexpr int TOPK_THREADS = 512;
constexpr int TOPK_MAX = 4096;
constexpr int TOPK_BLOCKS = 304;   // pass-1 blocks (two per SM)

// per-block lists of TOPK_MAX candidates plus the merged list, values and indices
static size_t topk_buffer_bytes() {
    return ((size_t)TOPK_BLOCKS + 1) * TOPK_MAX * (sizeof(float) + sizeof(long long)) + 64;
}

struct __align__(16) Cand {
    float v;
    int pad;
    long long idx;
};

__device__ __forceinline__ bool better(const Cand& a, const Cand& b) {
    return a.v > b.v || (a.v == b.v && a.idx < b.idx);
}

// Bitonic sort of n (power of two) entries in shared memory, best first.
__device__ void bitonic_sort(Cand* s, int n) {
    for (int size = 2; size <= n; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int i = threadIdx.x; i < (n >> 1); i += blockDim.x) {
                int lo = 2 * stride * (i / stride) + (i % stride);
                int hi = lo + stride;
                bool desc_block = ((lo & size) == 0);
                Cand a = s[lo], b = s[hi];
                bool swap = desc_block ? better(b, a) : better(a, b);
                if (swap) {
                    s[lo] = b;
                    s[hi] = a;
                }
            }
        }
    }
    __syncthreads();
}

__device__ __forceinline__ Cand worst_cand() {
    Cand c;
    c.v = -INFINITY;
    c.pad = 0;
    c.idx = 0x7fffffffffffffffLL;
    return c;
}

// s holds 2*KP entries: [0, KP) the current best (sorted), [KP, 2KP) candidates.
// After the call [0, KP) holds the best KP of the union, sorted.
__device__ void merge_best(Cand* s, int KP, int ncand) {
    for (int i = KP + ncand + threadIdx.x; i < 2 * KP; i += blockDim.x) s[i] = worst_cand();
    bitonic_sort(s, 2 * KP);
}

__device__ void scan_slice(const float* __restrict__ src, const long long* __restrict__ src_idx,
                           long long begin, long long end, Cand* s, int KP, int* ncand) {
    for (int i = threadIdx.x; i < 2 * KP; i += blockDim.x) s[i] = worst_cand();
    if (threadIdx.x == 0) *ncand = 0;
    __syncthreads();
    for (long long base = begin; base < end; base += blockDim.x) {
        long long i = base + threadIdx.x;
        if (i < end) {
            Cand c;
            float v = src[i];
            c.v = isnan(v) ? -INFINITY : v;
            c.pad = 0;
            c.idx = src_idx ? src_idx[i] : i;
            if (better(c, s[KP - 1])) {
                int pos = atomicAdd(ncand, 1);
                s[KP + pos] = c;
            }
        }
        __syncthreads();
        const int n = *ncand;
        // every thread has read the count before any thread admits the next tile's
        // candidates: otherwise a fast warp's atomicAdd reaches a slow warp's read and the
        // warps disagree on whether to merge (divergent barriers, overfull buffer)
        __syncthreads();
        if (n > KP - (int)blockDim.x || base + blockDim.x >= end) {
            if (n > 0) merge_best(s, KP, n);
            if (threadIdx.x == 0) *ncand = 0;
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(TOPK_THREADS)
topk_pass1(const float* __restrict__ rho, long long n, int KP, float* out_v, long long* out_i) {
    extern __shared__ __align__(16) unsigned char smem[];
    Cand* s = (Cand*)smem;
    __shared__ int ncand;
    long long per = (n + gridDim.x - 1) / gridDim.x;
    long long b = per * blockIdx.x, e = b + per < n ? b + per : n;
    scan_slice(rho, nullptr, b, e > b ? e : b, s, KP, &ncand);
    for (int i = threadIdx.x; i < KP; i += blockDim.x) {
        out_v[(long long)blockIdx.x * KP + i] = s[i].v;
        out_i[(long long)blockIdx.x * KP + i] = s[i].idx;
    }
}

__global__ void __launch_bounds__(TOPK_THREADS)
topk_pass2(const float* __restrict__ cv, const long long* __restrict__ ci, long long n, int KP,
           float* out_v, long long* out_i) {
    extern __shared__ __align__(16) unsigned char smem[];
    Cand* s = (Cand*)smem;
    __shared__ int ncand;
    scan_slice(cv, ci, 0, n, s, KP, &ncand);
    for (int i = threadIdx.x; i < KP; i += blockDim.x) {
        out_v[i] = s[i].v;
        out_i[i] = s[i].idx;
    }
}

// ---------------------------------------------------------------------------
// One pass over rho for the usual case (k well below the number of groups): every warp takes
// groups of contiguous values and notes each group's maximum; the last block to finish takes a
// threshold that k of those maxima reach, and few more -- so at least k values reach it --,
// rereads the groups that reach it, collects their values above it and sorts those.  Values
// are compared by an unsigned key that orders as `better` does (NaN as -inf, -0 as +0); ties end
// in the sort by index.  When the collection overflows (values bunched into few groups, or many
// equal ones) the count says so and the caller takes the block-list passes above.
//
// What bounds it: the read of rho, then the one block's chain of latencies (24.7 M values,
// k = 100: about 8 us to reread 119 groups, 3 us for the threshold, 2 us for the ranks).  The
// whole call, with its synchronisation, 69 us (74 with a copy of the list); 2140 us by the block
// lists alone.
// ---------------------------------------------------------------------------
constexpr int SEL_THREADS = 1024;
constexpr int SEL_BLOCKS = 152;        // one per SM
constexpr int SEL_GROUPS = 16384;      // maxima
constexpr int SEL_CAP = 8192;          // collected candidates
constexpr int SEL_BATCH = 8;           // 16-byte loads a lane has in flight while it rereads

struct SelHead {                       // on the device: blocks done; the maxima follow
    unsigned done, pad[3];
};
struct SelOut {                        // in pinned host memory, followed by the hits' indices [k] and values [k]
    unsigned count, err, pad[2];
};

__device__ __forceinline__ unsigned sel_key(float v) {
    v = isnan(v) ? -INFINITY : v + 0.0f;
    const unsigned u = __float_as_uint(v);
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}

// Largest key of values [b, e) over the warp (aligned: b and rho allow 16-byte loads).  fmaxf
// passes over NaN, as the key's order does.
__device__ __forceinline__ unsigned group_max(const float* __restrict__ rho, long long b, long long e, bool aligned) {
    const int lane = threadIdx.x & 31;
    float m = -INFINITY;
    if (aligned) {
        const float4* p = (const float4*)(rho + b);
        const long long n4 = (e - b) >> 2;
#pragma unroll 8
        for (long long i = lane; i < n4; i += 32) {
            const float4 v = __ldg(p + i);
            m = fmaxf(fmaxf(m, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
        }
        b += n4 << 2;
    }
    for (long long i = b + lane; i < e; i += 32) m = fmaxf(m, __ldg(rho + i));
    return __reduce_max_sync(0xffffffffu, sel_key(m));
}

__global__ void __launch_bounds__(SEL_THREADS)
topk_select(const float* __restrict__ rho, long long n, int gsize, int n_groups, int k, int aligned,
            unsigned* __restrict__ maxima, SelHead* head, SelOut* out, long long* __restrict__ out_i, float* __restrict__ out_v,
            const unsigned* __restrict__ err) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ bool last;
    __shared__ int cnt[32], ncand, n_list;
    __shared__ unsigned range[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nw = gridDim.x * (SEL_THREADS / 32);
    for (int g = blockIdx.x * (SEL_THREADS / 32) + warp; g < n_groups; g += nw) {
        const long long b = (long long)g * gsize, e = b + gsize < n ? b + gsize : n;
        const unsigned m = group_max(rho, b, e, aligned);
        if (lane == 0) maxima[g] = m;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&head->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the threshold, bit by bit from above: the largest value so far that k maxima reach, until
    // not many more than k do (a histogram of them would serialise: they share their leading
    // bits).  A trial value outside the maxima's range needs no count.
    unsigned mine[SEL_GROUPS / SEL_THREADS], lo = 0xffffffffu, hi = 0;
#pragma unroll
    for (int i = 0; i < SEL_GROUPS / SEL_THREADS; ++i) {
        const int g = i * SEL_THREADS + tid;
        mine[i] = g < n_groups ? __ldcg(maxima + g) : 0u;
        hi = max(hi, mine[i]);
        if (g < n_groups) lo = min(lo, mine[i]);
    }
    if (tid < 32) cnt[tid] = 0;
    if (tid == 0) {
        ncand = n_list = 0;
        range[0] = 0xffffffffu;
        range[1] = 0;
    }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        atomicMin(&range[0], lo);
        atomicMax(&range[1], hi);
    }
    __syncthreads();
    lo = range[0];
    hi = range[1];
    unsigned thr = 0;
    for (int bit = 31; bit >= 0; --bit) {
        const unsigned c = thr | (1u << bit);
        if (c <= lo) thr = c;   // all of them, at least 2 k
        if (c <= lo || c > hi) continue;
        int n_ge = 0;
#pragma unroll
        for (int i = 0; i < SEL_GROUPS / SEL_THREADS; ++i) n_ge += mine[i] >= c;
        n_ge = __reduce_add_sync(0xffffffffu, n_ge);
        if (lane == 0 && n_ge) atomicAdd(&cnt[bit], n_ge);
        __syncthreads();
        const int reach = cnt[bit];
        if (reach >= k) thr = c;
        if (reach >= k && reach <= k + k / 8 + 32) break;
    }
    Cand* s = (Cand*)smem;
    unsigned short* list = (unsigned short*)(s + SEL_CAP);   // the groups that reach it
#pragma unroll
    for (int i = 0; i < SEL_GROUPS / SEL_THREADS; ++i) {
        const int g = i * SEL_THREADS + tid;
        if (g < n_groups && mine[i] >= thr) list[atomicAdd(&n_list, 1)] = (unsigned short)g;
    }
    __syncthreads();
    // the threshold as a value: v >= floor_v where key(v) >= thr, but for one that every key
    // reaches (-inf, and NaN with it)
    const bool all = thr <= sel_key(-INFINITY);
    const float floor_v = __uint_as_float(thr & 0x80000000u ? thr ^ 0x80000000u : ~thr);
    for (int li = warp; li < n_list; li += SEL_THREADS / 32) {
        const int g = list[li];
        const long long b = (long long)g * gsize, e = b + gsize < n ? b + gsize : n;
        auto take = [&](float v, long long i) {
            if (all || v >= floor_v) {
                const int pos = atomicAdd(&ncand, 1);
                if (pos < SEL_CAP) {
                    Cand c;
                    c.v = isnan(v) ? -INFINITY : v;
                    c.pad = 0;
                    c.idx = i;
                    s[pos] = c;
                }
            }
        };
        long long i0 = b;
        if (aligned) {
            const float4* p = (const float4*)(rho + b);
            const int n4 = (int)((e - b) >> 2);
            for (int i = lane; i < n4; i += 32 * SEL_BATCH) {   // the loads of a batch before its tests
                float4 v[SEL_BATCH];
#pragma unroll
                for (int j = 0; j < SEL_BATCH; ++j)
                    v[j] = i + 32 * j < n4 ? __ldg(p + i + 32 * j) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
#pragma unroll
                for (int j = 0; j < SEL_BATCH; ++j) {
                    if (!(all ? i + 32 * j < n4 : fmaxf(fmaxf(v[j].x, v[j].y), fmaxf(v[j].z, v[j].w)) >= floor_v)) continue;
                    const long long at = b + 4 * (i + 32 * j);
                    take(v[j].x, at);
                    take(v[j].y, at + 1);
                    take(v[j].z, at + 2);
                    take(v[j].w, at + 3);
                }
            }
            i0 += (long long)n4 << 2;
        }
        for (long long i = i0 + lane; i < e; i += 32) take(__ldg(rho + i), i);
    }
    __syncthreads();
    const int m = ncand;
    if (m <= SEL_THREADS / 2) {   // few: each one's rank, counted by `per` neighbouring threads
        const int per = m <= SEL_THREADS / 8 ? 8 : m <= SEL_THREADS / 4 ? 4 : 2;
        const int ci = tid / per, part = tid & (per - 1);
        Cand c = ci < m ? s[ci] : worst_cand();
        int rank = 0;
        for (int i = part; i < m; i += per) rank += better(s[i], c);
        for (int o = 1; o < per; o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        if (ci < m && part == 0 && rank < k) {
            out_i[rank] = c.idx;
            out_v[rank] = c.v;
        }
    } else if (m <= SEL_CAP) {
        int size = 2;
        while (size < m) size <<= 1;
        for (int i = m + tid; i < size; i += SEL_THREADS) s[i] = worst_cand();
        bitonic_sort(s, size);
        for (int i = tid; i < k; i += SEL_THREADS) {
            out_i[i] = s[i].idx;
            out_v[i] = s[i].v;
        }
    }
    if (tid == 0) {
        out->count = (unsigned)m;
        out->err = __ldcg(err);
    }
}

static void fill_hits(const cc_plan* plan, int nk, const long long* idx, const float* val, cc_hit* out) {
    for (int i = 0; i < nk; ++i) {
        cc_hit h;
        memset(&h, 0, sizeof(h));
        h.tmpl = idx[i] / plan->N_f;
        h.bin = (int32_t)(idx[i] % plan->N_f);
        h.freq = plan->freq[h.bin];
        h.rho = val[i];
        out[i] = h;
    }
}

}  // namespace cc

extern "C" cc_status crosscorr_rho_topk(cc_plan* plan, const float* rho_dev, int64_t n_t, int k,
                                        cc_hit* hits_host, void* stream) {
    CC_NVTX_RANGE("crosscorr_rho_topk");
    using namespace cc;
    if (!plan) return fail(CC_ERR_INVALID, "plan is null");
    if (n_t < 0 || k < 1 || k > TOPK_MAX) return fail(CC_ERR_INVALID, "need n_t >= 0 and 1 <= k <= 4096");
    if (!hits_host) return fail(CC_ERR_INVALID, "hits_host is null");
    const long long n = (long long)n_t * plan->N_f;
    if (n == 0) return CC_OK;
    if (!rho_dev) return fail(CC_ERR_INVALID, "rho_dev is null");
    cudaStream_t st = (cudaStream_t)stream;
    // Group maxima and candidate lists live in a buffer of their own, sized once for the
    // largest k and block count, so top-k never touches (or grows) the search workspace: a search
    // queued on another stream for this plan keeps its workspace intact.
    if (!plan->topk_ws) {
        cudaError_t ea = cudaMalloc(&plan->topk_ws, topk_buffer_bytes());
        if (ea != cudaSuccess) {
            plan->topk_ws = nullptr;
            return cuda_fail(ea, "top-k candidate buffer");
        }
    }
    const int nk = (int)std::min<long long>(k, n);
    // Groups of at least 256 values, at most three for each of the grid's warps (full rounds); the
    // threshold needs k groups and is close to the k-th value while there are several times more.
    const long long most = 3 * SEL_BLOCKS * (SEL_THREADS / 32);
    static_assert(3 * SEL_BLOCKS * (SEL_THREADS / 32) <= SEL_GROUPS, "one maximum per group");
    const long long gsize = std::max<long long>(256, ((n + most - 1) / most + 127) / 128 * 128);
    const long long n_groups = (n + gsize - 1) / gsize;
    if (n_groups >= 2 * (long long)nk) {
        // the list goes straight to pinned host memory (50 KB, allocated by the first call): a copy
        // to pageable memory after the kernel cost 5 us
        if (!plan->topk_host) {
            const cudaError_t ea = cudaHostAlloc(&plan->topk_host, sizeof(SelOut) + (size_t)TOPK_MAX * 12,
                                                 cudaHostAllocMapped | cudaHostAllocPortable);
            if (ea != cudaSuccess) {
                plan->topk_host = nullptr;
                return cuda_fail(ea, "top-k result buffer");
            }
        }
        SelHead* head = (SelHead*)plan->topk_ws;
        unsigned* maxima = (unsigned*)(head + 1);
        SelOut* out = nullptr;
        const size_t sm = (size_t)SEL_CAP * sizeof(Cand) + SEL_GROUPS * sizeof(unsigned short);
        cudaError_t e = cudaFuncSetAttribute(topk_select, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&out, plan->topk_host, 0);
        if (e == cudaSuccess) e = cudaMemsetAsync(head, 0, sizeof(SelHead), st);
        if (e != cudaSuccess) return cuda_fail(e, "top-k selection set-up");
        long long* oi = (long long*)(out + 1);
        float* ov = (float*)(oi + nk);
        const int aligned = ((uintptr_t)rho_dev & 15) == 0;
        const int blocks = (int)std::min<long long>(SEL_BLOCKS, (n_groups + SEL_THREADS / 32 - 1) / (SEL_THREADS / 32));
        topk_select<<<blocks, SEL_THREADS, sm, st>>>(rho_dev, n, (int)gsize, (int)n_groups, nk, aligned, maxima, head, out, oi,
                                                     ov, plan->dp.err);
        count_launch();
        if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "topk launch");
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_fail(e, "topk");
        const SelOut* h = (const SelOut*)plan->topk_host;
        if (h->err) return crosscorr_plan_check(plan, stream);   // a failed bounded wait of the searches before
        if (h->count <= (unsigned)SEL_CAP) {
            const long long* hi = (const long long*)(h + 1);
            fill_hits(plan, nk, hi, (const float*)(hi + nk), hits_host);
            return CC_OK;
        }
    }
    int KP = 1;
    while (KP < k) KP <<= 1;
    KP = std::max(KP, 2 * TOPK_THREADS);   // candidate buffer must exceed one tile
    int nb = (int)std::min<long long>(TOPK_BLOCKS, (n + 65535) / 65536);
    nb = std::max(nb, 1);
    size_t cand = (size_t)nb * KP;
    char* w = (char*)plan->topk_ws;
    long long* ci = (long long*)w;
    long long* fi = ci + cand;
    float* cv = (float*)(fi + KP);
    float* fv = cv + cand;
    const size_t sm = (size_t)2 * KP * sizeof(Cand);
    cudaError_t e = cudaFuncSetAttribute(topk_pass1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(topk_pass2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return cuda_fail(e, "topk smem attribute");
    topk_pass1<<<nb, TOPK_THREADS, sm, st>>>(rho_dev, n, KP, cv, ci);
    count_launch();
    topk_pass2<<<1, TOPK_THREADS, sm, st>>>(cv, ci, (long long)cand, KP, fv, fi);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "topk launch");
    std::vector<float> hv(KP);
    std::vector<long long> hi(KP);
    e = cudaMemcpyAsync(hv.data(), fv, sizeof(float) * KP, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hi.data(), fi, sizeof(long long) * KP, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "topk copy");
    // the stream is synchronised: report a failed bounded wait of the searches before it
    unsigned err_word = 0;
    e = cudaMemcpy(&err_word, plan->dp.err, sizeof(err_word), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "reading the device error word");
    if (err_word) return crosscorr_plan_check(plan, stream);
    fill_hits(plan, nk, hi.data(), hv.data(), hits_host);
    return CC_OK;
}
