// Shared declarations of the kernels on 4096-point output cosets (segpair_tma.cu,
// segfft_rows.cu).
#pragma once

#include "common.cuh"
#include "fft_reg.cuh"

namespace cc {

// Two-pass search of folded segments in BF16: whether the plan takes it, the segment chunks
// per (template, weight), the folded rows' bytes per template, the fold and one launch of the
// spectrum + pair-sum kernel over a template batch.
bool segpair_tma_supported(const cc_plan* plan);
int segpair_tma_chunks(const cc_plan* plan, int64_t n_t);
size_t segpair_tma_fold_bytes(const cc_plan* plan);
cc_status launch_fold_bf16(cc_plan* plan, int64_t n_t, const void* ab, const float4* norm, void* z, cudaStream_t st);
cc_status launch_segpair_tma(cc_plan* plan, int n_chunks, int64_t chunk_len, int64_t n_t, const void* z,
                             const float4* norm, float* raw, int* counter, cudaStream_t st);
// The staged segment-FFT stage by whole output rows: whether plan and input fit it, and one launch
// writing F [n_t][Q][M][2][N_f] (counter: one int).
bool segfft_rows_supported(const cc_plan* plan, const void* ab);
cc_status launch_segfft_rows(cc_plan* plan, int64_t n_t, const void* ab, float2* F, int* counter, cudaStream_t st);

}  // namespace cc
