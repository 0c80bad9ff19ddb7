// Shared declarations of the two-pass search's kernels on the lag grid (corr_kernel.cuh,
// corr.cu).
#pragma once

#include "common.cuh"
#include "fft_reg.cuh"

namespace cc {

constexpr int CORR_THREADS = 256;
constexpr int CORR_MAX_CHUNK = 1023;    // segments of a chunk (its activity words, and one before, are kept on chip)
constexpr int CORR_POINTS = 4096;   // points of one CTA's transforms: 4096 / L of L points each

// T transforms a CTA: elements of an exchange buffer (T = 1: padded), activity bits of a detector
// in a segment's word (a byte for T = 1) and the word's bytes.
__host__ __device__ constexpr int corr_buffer(int T) { return T == 1 ? 17 * 256 + 16 : CORR_POINTS; }
__host__ __device__ constexpr int corr_act_bits(int T, bool multi) { return T == 1 ? 1 : multi ? 8 : 16; }
__host__ __device__ constexpr int corr_act_bytes(int T) { return T == 1 ? 1 : 4; }

// Everything corr_kernel needs.
struct CorrArgs {
    const void* src;        // a_r, b_r [n_t][Q][2][N_tau], or folded rows Z [n_t][Q][2][M][C][4096]
    const uint8_t* act;     // [Q][M][t_pad]: the detector has weight in (segment, template)
    float* raw;             // [n_t][2 n_chunks][planes][2][C][L] partial sums and what they round off (planes: A, and Re B, Im B with a lag)
    int* ctr;               // unit counter, zero at launch
    unsigned* err;          // the plan's device error word
    const float2* twk;      // [C][272] coset and second-pass twiddles on the grid of G = C L points
    const float2* twp;      // [C][butterflies][powers][L / 16] last-pass twiddle powers per thread (corr_powers)
    int64_t N_s, N_tau;
    int M, chunk_len, n_t, t_pad, Q, C, n_chunks, units;
    int n_in;               // samples of a staged row: N_s, or 4096 positions of a folded row
    int folded, tma, all_ordered, wait_test;
    uint32_t row_bytes, row_stride, off_y, off_tw, off_act, off_bar, smem;
};

template <int LT, bool BF16, bool LAG, bool HALF, bool MULTI>
cudaError_t launch_corr_t(const CorrArgs& a, int sms, cudaStream_t st);

#define CC_CORR_ONE(KW, L, B, G, H, MU) KW template cudaError_t launch_corr_t<L, B, G, H, MU>(const CorrArgs&, int, cudaStream_t);
#define CC_CORR_INST(KW, L) \
    CC_CORR_ONE(KW, L, false, false, true, false) CC_CORR_ONE(KW, L, false, true, true, false) \
    CC_CORR_ONE(KW, L, true, false, true, false) CC_CORR_ONE(KW, L, true, true, true, false)
#define CC_CORR_INST_FULL(KW) \
    CC_CORR_ONE(KW, 4096, false, false, false, false) CC_CORR_ONE(KW, 4096, false, true, false, false) \
    CC_CORR_ONE(KW, 4096, true, false, false, false) CC_CORR_ONE(KW, 4096, true, true, false, false)
// three or four detectors (FP32 rows)
#define CC_CORR_INST_MULTI(KW, L) CC_CORR_ONE(KW, L, false, false, true, true) CC_CORR_ONE(KW, L, false, true, true, true)
#define CC_CORR_INST_MULTI_FULL(KW) CC_CORR_ONE(KW, 4096, false, false, false, true) CC_CORR_ONE(KW, 4096, false, true, false, true)

// Threads' last-pass twiddle powers for C cosets of L points (host, at plan creation): thread j
// of a transform, butterfly i, power 2^n of W_G^(c + C b), G = C L, at ((c nb + i) np + n) L/16 + j.
std::vector<float2> corr_powers(int64_t L, int64_t C);

// Whether the lag grid serves the plan (corr.cu): its tables are made for such plans only.
bool lag_grid_supported(const cc_plan* plan);

// Work units per resident CTA slot (2 per SM), shared by the layout and the launch.
constexpr int CORR_CTAS_PER_SM = 2;

}  // namespace cc
