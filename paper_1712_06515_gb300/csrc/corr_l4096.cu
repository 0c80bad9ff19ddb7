// corr_kernel for transforms of 4096 points: segments of up to 2048 samples (upper half of the
// input zero), and the cosets of longer ones.
#include "corr_kernel.cuh"
namespace cc {
CC_CORR_INST(, 4096)
CC_CORR_INST_FULL()
}  // namespace cc
