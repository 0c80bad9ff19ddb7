// Shared declarations of the two-pass search's kernels on the lag grid (corr_kernel.cuh,
// corr.cu).
#pragma once

#include "common.cuh"
#include "fft_reg.cuh"

namespace cc {

constexpr int CORR_THREADS = 256;
constexpr int CORR_MAX_CHUNK = 1023;    // segments of a chunk (its activity words, and one before, are kept on chip)
constexpr int CORR_POINTS = 4096;   // points of one CTA's transforms: 4096 / L of L points each

// Everything corr_kernel needs.
struct CorrArgs {
    const void* src;        // a_r, b_r [n_t][Q][2][N_tau], or folded rows Z [n_t][Q][2][M][C][4096]
    const uint8_t* act;     // [2][M][t_pad]: detector 0 / the last detector has weight in (segment, template)
    float* raw;             // [n_t][2 n_chunks][planes][C][L] partial sums (planes: A, and Re B, Im B with a lag)
    int* ctr;               // unit counter, zero at launch
    unsigned* err;          // the plan's device error word
    const float2* twk;      // [C][272] coset and second-pass twiddles on the grid of G = C L points
    const float4* tw8;      // [C][256][2] powers 1, 2, 4, 8 of W_G^(c + C j), G = 4096 C (last pass of L = 4096)
    const float2* twL;      // exp(-2 pi i j / L)
    int64_t N_s, N_tau;
    int M, chunk_len, n_t, t_pad, Q, C, n_chunks, units;
    int n_in;               // samples of a staged row: N_s, or 4096 positions of a folded row
    int folded, tma, all_ordered, wait_test;
    uint32_t row_bytes, row_stride, off_y, off_z, off_act, off_bar, smem;
};

template <int LT, bool BF16, bool LAG, bool HALF>
cudaError_t launch_corr_t(const CorrArgs& a, int sms, cudaStream_t st);

#define CC_CORR_INST(KW, L)                                                                    \
    KW template cudaError_t launch_corr_t<L, false, false, true>(const CorrArgs&, int, cudaStream_t);  \
    KW template cudaError_t launch_corr_t<L, false, true, true>(const CorrArgs&, int, cudaStream_t);   \
    KW template cudaError_t launch_corr_t<L, true, false, true>(const CorrArgs&, int, cudaStream_t);   \
    KW template cudaError_t launch_corr_t<L, true, true, true>(const CorrArgs&, int, cudaStream_t);
#define CC_CORR_INST_FULL(KW)                                                                  \
    KW template cudaError_t launch_corr_t<4096, false, false, false>(const CorrArgs&, int, cudaStream_t); \
    KW template cudaError_t launch_corr_t<4096, false, true, false>(const CorrArgs&, int, cudaStream_t);  \
    KW template cudaError_t launch_corr_t<4096, true, false, false>(const CorrArgs&, int, cudaStream_t);  \
    KW template cudaError_t launch_corr_t<4096, true, true, false>(const CorrArgs&, int, cudaStream_t);

// Work units per resident CTA slot (2 per SM), shared by the layout and the launch.
constexpr int CORR_CTAS_PER_SM = 2;

}  // namespace cc
