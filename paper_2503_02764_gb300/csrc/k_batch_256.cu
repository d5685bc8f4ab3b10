// The batched step with blocks of 256 threads, half sweeps only.
#include "batch_step.cuh"

namespace fld {
FLD_BATCH_DEFINE(256, false)
}  // namespace fld
