// The batched step with blocks of 512 threads, half sweeps only.
#include "batch_step.cuh"

namespace fld {
FLD_BATCH_DEFINE(512, false)
}  // namespace fld
