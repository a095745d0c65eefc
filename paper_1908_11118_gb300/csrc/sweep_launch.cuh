// sweep_launch.cuh -- the sweep kernel of one system and its launch (internal).
#pragma once

#include "walker.cuh"

namespace regc {
namespace {

// Registers per thread are bounded so that every walker that fits in shared
// memory is resident: a direct walker takes 3-5 KB, so up to 28 one-warp CTAs
// share an SM (a launch of 4096 walkers, 27 per SM: 24 resident 444 us on
// fcc(100) and 571 us of clusters, 28 resident 366 and 507 us, the spills of 72
// registers included); four warps per walker run at a few walkers per SM.
template <int K, bool DA, bool CL, bool DIRECT>
constexpr int min_ctas() {
    return DIRECT && K == 1 ? 28 : (K == 4 ? 3 : 1);
}

template <int K, bool TRACE, bool DA, bool CL, bool DIRECT, int GEO>
__global__ void __launch_bounds__(32 * K, min_ctas<K, DA, CL, DIRECT>())
    sweep_kernel(const __grid_constant__ SweepParams P) {
    extern __shared__ __align__(16) char smem[];
    const int w = P.w_begin + (int)blockIdx.x;
    if (w >= P.w_end) return;
    walker_sweep<K, TRACE, DA, CL, DIRECT, GEO>(P, w, smem, threadIdx.x, 0);
}

template <int K, bool TRACE, bool DA, bool CL, bool DIRECT, int GEO>
cudaError_t launch_one(const SweepParams& P, int n_walkers, cudaStream_t s) {
    const size_t smem = smem_bytes(P.nmax, P.cg.ncell, P.cg.cap, K, DIRECT);
    const cudaError_t err = cudaFuncSetAttribute(sweep_kernel<K, TRACE, DA, CL, DIRECT, GEO>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    sweep_kernel<K, TRACE, DA, CL, DIRECT, GEO><<<n_walkers, 32 * K, smem, s>>>(P);
    return cudaGetLastError();
}

template <int K, bool DA, bool CL, bool DIRECT>
cudaError_t launch_k(const SweepParams& P, cudaStream_t s) {
    const int n_walkers = P.w_end - P.w_begin;   // one CTA per walker of the shard
    if (n_walkers <= 0) return cudaSuccess;
    // (traced launches are for comparisons: the general form alone; delayed
    // acceptance meets no sheared cell often enough for one of its own)
    if (P.trace) return launch_one<K, true, DA, CL, DIRECT, 0>(P, n_walkers, s);
    switch (sweep_geo(P)) {
        case 1: return launch_one<K, false, DA, CL, DIRECT, 1>(P, n_walkers, s);
        case 2: return launch_one<K, false, DA, CL, DIRECT, DA ? 0 : 2>(P, n_walkers, s);
        case 3: return launch_one<K, false, DA, CL, DIRECT, 3>(P, n_walkers, s);
    }
    return launch_one<K, false, DA, CL, DIRECT, 0>(P, n_walkers, s);
}

}  // namespace
}  // namespace regc
