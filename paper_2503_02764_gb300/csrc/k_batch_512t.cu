// The batched step with blocks of 512 threads and tiles.
#include "batch_step.cuh"

namespace fld {
FLD_BATCH_DEFINE(512, true)
}  // namespace fld
