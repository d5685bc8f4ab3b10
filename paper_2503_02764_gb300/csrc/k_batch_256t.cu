// The batched step with blocks of 256 threads and tiles.
#include "batch_step.cuh"

namespace fld {
FLD_BATCH_DEFINE(256, true)
}  // namespace fld
