// corr_kernel for transforms of 128, 256 and 512 points.
#include "corr_kernel.cuh"
namespace cc {
CC_CORR_INST(, 128)
CC_CORR_INST(, 256)
CC_CORR_INST(, 512)
}  // namespace cc
