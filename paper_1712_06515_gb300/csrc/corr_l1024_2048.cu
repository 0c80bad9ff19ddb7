// corr_kernel for transforms of 1024 and 2048 points.
#include "corr_kernel.cuh"
namespace cc {
CC_CORR_INST(, 1024)
CC_CORR_INST(, 2048)
}  // namespace cc
