// corr_kernel for three and four detectors.
#include "corr_kernel.cuh"
namespace cc {
CC_CORR_INST_MULTI(, 256)
CC_CORR_INST_MULTI(, 512)
CC_CORR_INST_MULTI(, 1024)
CC_CORR_INST_MULTI(, 2048)
CC_CORR_INST_MULTI(, 4096)
CC_CORR_INST_MULTI_FULL()
}  // namespace cc
