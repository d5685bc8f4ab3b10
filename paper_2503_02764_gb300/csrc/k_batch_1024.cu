// The batched step with blocks of 1024 threads.
#include "batch_step.cuh"

namespace fld {
FLD_BATCH_DEFINE(1024, false)
}  // namespace fld
