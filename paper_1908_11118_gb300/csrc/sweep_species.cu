// sweep_species.cu -- the sweep of one system's replicas with two mobile
// species (a cluster, or two grand-canonical species) or with delayed
// acceptance (sm_103a).  See walker.cuh.
#include "sweep_launch.cuh"

namespace regc {

cudaError_t launch_sweep_species(const SweepParams& P, cudaStream_t s) {
    const bool cl = P.n_cluster > 0 || P.gc2;
    if (P.delayed) return cl ? launch_k<1, true, true, false>(P, s) : launch_k<1, true, false, false>(P, s);
    return sweep_direct(P) ? launch_k<1, false, true, true>(P, s) : launch_k<1, false, true, false>(P, s);
}

}  // namespace regc
