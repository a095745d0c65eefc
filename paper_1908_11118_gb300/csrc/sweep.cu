// sweep.cu -- the sweep of one system's replicas: one grand-canonical species,
// plain acceptance (sm_103a).  See walker.cuh.
#include "sweep_launch.cuh"

namespace regc {

size_t sweep_smem(const SweepParams& P, int warps_per_walker) {
    return smem_bytes(P.nmax, P.cg.ncell, P.cg.cap, warps_per_walker, sweep_direct(P));
}

// The sizes of Nmax and of the cell grid that handles are created for: what a
// walker with 128 bytes of statistics, 72 bytes of result and 1792 bytes of
// stencil and scratch per warp beside its positions, moves and cell list takes
// of one CTA's shared memory.  The layouts in use need less; the bound stays,
// so that a problem refused once stays refused.
size_t sweep_smem_admitted(int nmax, int ncell, int cap, int warps_per_walker) {
    const size_t K = (size_t)warps_per_walker;
    return align16(size_t(nmax) * 16) + 16 + 128 + 32 + 2048 + align16(K * 72) + K * 1792 + align16(size_t(ncell) * 2) +
           align16(size_t(ncell) * cap * 2);
}

cudaError_t launch_sweep(const SweepParams& P, cudaStream_t s) {
    if (P.n_sweeps <= 0) return cudaSuccess;
    // delayed acceptance and two mobile species: one warp per walker
    if (P.delayed || P.n_cluster > 0 || P.gc2) return launch_sweep_species(P, s);
    const bool direct = sweep_direct(P);
    switch (P.warps_per_walker) {
        case 1: return direct ? launch_k<1, false, false, true>(P, s) : launch_k<1, false, false, false>(P, s);
        case 2: return direct ? launch_k<2, false, false, true>(P, s) : launch_k<2, false, false, false>(P, s);
        case 4: return direct ? launch_k<4, false, false, true>(P, s) : launch_k<4, false, false, false>(P, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace regc
