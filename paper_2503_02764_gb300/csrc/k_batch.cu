// The batched step's kernels by block size (batch_step.cuh; one translation unit each).
#include "fld_batch.cuh"

namespace fld {

int batch_threads_supported(int nt) { return nt == 256 || nt == 512 || nt == 1024; }
int batch_cluster_supported(int cs) { return cs == 1 || cs == 2 || cs == 4 || cs == 8; }

int batch_max_groups(int nt, int cs, const BatchParams& prm) {
    if (nt == 1024) return batch_groups<1024, false>(cs);
    if (nt == 256) return prm.tiles ? batch_groups<256, true>(cs) : batch_groups<256, false>(cs);
    return prm.tiles ? batch_groups<512, true>(cs) : batch_groups<512, false>(cs);
}

void launch_batch_step(int nt, int cs, int ngroups, const BProb* probs, const BDyn* dyn,
                       const int* order, int nprob, int* queue, const BatchParams& prm,
                       const double* rho, double* T, double* E, const double* Ebc, double* wsd,
                       float* wsf, BatchStat* stats, unsigned* err, cudaStream_t s) {
    auto* launch = nt == 1024  ? batch_launch<1024, false>
                   : nt == 256 ? (prm.tiles ? batch_launch<256, true> : batch_launch<256, false>)
                               : (prm.tiles ? batch_launch<512, true> : batch_launch<512, false>);
    launch(cs, ngroups, probs, dyn, order, nprob, queue, prm, rho, T, E, Ebc, wsd, wsf, stats, err,
           s);
}

}  // namespace fld
