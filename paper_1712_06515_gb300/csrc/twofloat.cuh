// Numbers as unevaluated sums of two floats (x the value rounded to FP32, y the rest: 48 bits), for
// the short transforms whose rounding must not reach the sums' own (corr.cu).  FP64 has 1/64 of the
// FP32 rate here: a radix-4 butterfly takes 28 FP64 operations or about 340 FP32 ones, a fifth of
// the time.  Sums by Knuth's and Dekker's error-free additions, products with the error of the
// leading product from a fused multiply-add; relative error of an operation about 2^-46 of its
// operands' size.
#pragma once

#include "common.cuh"

namespace cc {

// a complex number: real part (x, y), imaginary part (z, w)
using ff = float2;
using ffc = float4;

__host__ __device__ inline ff ff_from(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}

// s + e = a + b for |a| >= |b|
__device__ __forceinline__ ff ff_renorm(float a, float b) {
    const float s = __fadd_rn(a, b);
    return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ ff ff_add(ff a, ff b) {
    const float s = __fadd_rn(a.x, b.x), t = __fsub_rn(s, a.x);
    const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, t)), __fsub_rn(b.x, t));
    return ff_renorm(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}

__device__ __forceinline__ ff ff_neg(ff a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }

__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    const float p = __fmul_rn(a.x, b.x);
    return ff_renorm(p, __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.y, __fmaf_rn(a.x, b.x, -p))));
}

__device__ __forceinline__ ff ffc_re(ffc a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ ff ffc_im(ffc a) { return make_float2(a.z, a.w); }
__device__ __forceinline__ ffc ffc_make(ff re, ff im) { return make_float4(re.x, re.y, im.x, im.y); }

__device__ __forceinline__ ffc ffc_add(ffc a, ffc b) {
    return ffc_make(ff_add(ffc_re(a), ffc_re(b)), ff_add(ffc_im(a), ffc_im(b)));
}
__device__ __forceinline__ ffc ffc_sub(ffc a, ffc b) {
    return ffc_make(ff_sub(ffc_re(a), ffc_re(b)), ff_sub(ffc_im(a), ffc_im(b)));
}
__device__ __forceinline__ ffc ffc_negi(ffc a) { return make_float4(a.z, a.w, -a.x, -a.y); }   // -i a
__device__ __forceinline__ ffc ffc_conj(ffc a) { return make_float4(a.x, a.y, -a.z, -a.w); }
__device__ __forceinline__ ffc ffc_scale2(ffc a, float s) { return make_float4(a.x * s, a.y * s, a.z * s, a.w * s); }   // s a power of two
__device__ __forceinline__ ffc ffc_mul(ffc a, ffc b) {
    const ff ar = ffc_re(a), ai = ffc_im(a), br = ffc_re(b), bi = ffc_im(b);
    return ffc_make(ff_sub(ff_mul(ar, br), ff_mul(ai, bi)), ff_add(ff_mul(ar, bi), ff_mul(ai, br)));
}

// W^e, 0 <= e, from the tables lo[e mod 4096] and hi[e / 4096] of the root's powers
__device__ __forceinline__ ffc ffc_power(const ffc* __restrict__ lo, const ffc* __restrict__ hi, uint64_t e) {
    const ffc w = __ldg(lo + (e & 4095));
    return e >> 12 ? ffc_mul(w, __ldg(hi + (e >> 12))) : w;
}

// fft_stockham (common.cuh) on two-float numbers; tw: exp(-2 pi i j / L), j < L, in shared memory.
__device__ __forceinline__ ffc* ffc_stockham(ffc* a, ffc* b, int L, int log2L, const ffc* tw) {
    ffc *in = a, *out = b;
    int Ns = 1;
    const int quarter = L >> 2;
    for (int ps = 0; ps < (log2L >> 1); ++ps) {
        const int stride = L / (Ns * 4);
        for (int j = threadIdx.x; j < quarter; j += blockDim.x) {
            const int k = j & (Ns - 1);
            ffc v0 = in[j], v1 = in[j + quarter], v2 = in[j + 2 * quarter], v3 = in[j + 3 * quarter];
            if (Ns > 1) {
                v1 = ffc_mul(v1, tw[k * stride]);
                v2 = ffc_mul(v2, tw[2 * k * stride]);
                v3 = ffc_mul(v3, tw[3 * k * stride]);
            }
            const ffc a0 = ffc_add(v0, v2), a1 = ffc_sub(v0, v2), a2 = ffc_add(v1, v3), a3 = ffc_negi(ffc_sub(v1, v3));
            ffc* const o = out + ((j - k) << 2) + k;
            o[0] = ffc_add(a0, a2);
            o[Ns] = ffc_add(a1, a3);
            o[2 * Ns] = ffc_sub(a0, a2);
            o[3 * Ns] = ffc_sub(a1, a3);
        }
        __syncthreads();
        ffc* t = in;
        in = out;
        out = t;
        Ns <<= 2;
    }
    if (log2L & 1) {
        const int half = L >> 1, stride = L / (Ns * 2);
        for (int j = threadIdx.x; j < half; j += blockDim.x) {
            const int k = j & (Ns - 1);
            const ffc v0 = in[j];
            ffc v1 = in[j + half];
            if (Ns > 1) v1 = ffc_mul(v1, tw[k * stride]);
            ffc* const o = out + ((j - k) << 1) + k;
            o[0] = ffc_add(v0, v1);
            o[Ns] = ffc_sub(v0, v1);
        }
        __syncthreads();
        ffc* t = in;
        in = out;
        out = t;
    }
    return in;
}

}  // namespace cc
