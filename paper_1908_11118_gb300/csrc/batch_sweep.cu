// batch_sweep.cu -- the persistent sweep of a batch of uneven systems (sm_103a).
// See walker.cuh.
#include "walker.cuh"

namespace regc {
namespace {

// Persistent sweep of a batch of walkers from several systems.  Every group
// of K warps of the CTA is one walker at a time: its first thread takes the
// next (system, walker) item from the queue, the group copies that system's
// parameters to the head of its shared-memory region of `region` bytes and runs
// the walker's sweeps in the rest of it (K > 1: the speculative
// walker, synchronised by the group's named barrier 1 + group); items are
// listed largest first, so the queue balances the uneven costs.  DA: the
// systems of the launch sample with delayed acceptance (their networks'
// fragments take ~240 registers per thread, so at most kBatchMaxWarpsDA
// walkers per CTA); CL: every system of the launch carries a cluster species;
// DIRECT: its walkers enumerate all particles instead of a cell list; SLAB:
// every system of the launch is a rectangular slab (sweep_geo 1).
constexpr int kBatchMaxWarps = 16;
constexpr int kBatchMaxWarpsDA = 4;
constexpr int kBatchHead = (int)((sizeof(SweepParams) + sizeof(int) + 15) / 16 * 16);   // parameters and item

template <bool DA, bool CL, bool DIRECT, bool SLAB, int K>
__global__ void __launch_bounds__(32 * (DA ? kBatchMaxWarpsDA : kBatchMaxWarps))
    batch_sweep_kernel(const SweepParams* __restrict__ sys, const int2* __restrict__ items, int n_items,
                       int* counter, int region) {
    extern __shared__ __align__(16) char smem[];
    const int tid = threadIdx.x % (32 * K), grp = threadIdx.x / (32 * K);
    const int bar = K == 1 ? 0 : 1 + grp;
    char* mine = smem + (size_t)grp * region;
    SweepParams& Psh = *reinterpret_cast<SweepParams*>(mine);
    int& item_sh = *reinterpret_cast<int*>(mine + sizeof(SweepParams));
    for (;;) {
        int item = 0;
        if (K == 1) {
            if (tid == 0) item = atomicAdd(counter, 1);
            item = __shfl_sync(FULL, item, 0);
        } else {
            if (tid == 0) item_sh = atomicAdd(counter, 1);
            group_sync<K>(bar);
            item = item_sh;
        }
        if (item >= n_items) break;
        const int2 mw = items[item];
        const int* src = reinterpret_cast<const int*>(sys + mw.x);
        int* dst = reinterpret_cast<int*>(mine);
        for (int k = tid; k < (int)(sizeof(SweepParams) / sizeof(int)); k += 32 * K) dst[k] = src[k];
        group_sync<K>(bar);
        walker_sweep<K, false, DA, CL, DIRECT, SLAB ? 1 : 0>(Psh, mw.y, mine + kBatchHead, tid, bar);
        group_sync<K>(bar);   // the slot and the item are rewritten for the next walker
    }
}

}  // namespace

size_t batch_head() { return kBatchHead; }

// A system joins a batch where its walker was admitted beside the parameter
// blocks (756 bytes each) of a CTA's most walkers; the regions in use need less.
bool batch_admits(const SweepParams& P) {
    const int groups = P.delayed ? kBatchMaxWarpsDA : kBatchMaxWarps;
    return align16(sweep_smem_admitted(P.nmax, P.cg.ncell, P.cg.cap, 1)) + (size_t)756 * groups <= 232448;
}

int batch_max_warps(bool da) { return da ? kBatchMaxWarpsDA : kBatchMaxWarps; }

namespace {

struct Launch {
    const SweepParams* sys;
    const int2* items;
    int n_items;
    int* counter;
    int walkers_per_cta, grid, region;
    cudaStream_t s;
    cudaError_t err = cudaErrorInvalidValue;
    template <bool DA, bool CL, bool DIRECT, bool SLAB, int K>
    void run() {
        const size_t smem = (size_t)walkers_per_cta * region;
        batch_sweep_kernel<DA, CL, DIRECT, SLAB, K>
            <<<grid, 32 * K * walkers_per_cta, smem, s>>>(sys, items, n_items, counter, region);
        err = cudaGetLastError();
    }
};

struct Prepare {
    int max_smem;
    cudaError_t err = cudaSuccess;
    template <bool DA, bool CL, bool DIRECT, bool SLAB, int K>
    void run() {
        if (err == cudaSuccess)
            err = cudaFuncSetAttribute(batch_sweep_kernel<DA, CL, DIRECT, SLAB, K>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       max_smem);
    }
};

struct Occupancy {
    int walkers_per_cta;
    size_t smem;
    int n = 0;
    template <bool DA, bool CL, bool DIRECT, bool SLAB, int K>
    void run() {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_sweep_kernel<DA, CL, DIRECT, SLAB, K>,
                                                          32 * K * walkers_per_cta, smem) != cudaSuccess)
            n = 0;
    }
};

// f.run<DA, CL, DIRECT, SLAB, K>() of a class; false where there is no such
// kernel: delayed acceptance follows the cell list, more than one warp per
// walker is for plain one-species walkers, and so is the slab's own form.
template <int K, class F>
void dispatch_plain(const BatchClass& c, F& f) {
    if (c.direct && c.slab) f.template run<false, false, true, true, K>();
    else if (c.direct) f.template run<false, false, true, false, K>();
    else if (c.slab) f.template run<false, false, false, true, K>();
    else f.template run<false, false, false, false, K>();
}

template <class F>
bool dispatch(const BatchClass& c, int K, F& f) {
    if ((c.da && c.direct) || ((c.da || c.cl) && (c.slab || K != 1))) return false;
    if (c.da && c.cl) f.template run<true, true, false, false, 1>();
    else if (c.da) f.template run<true, false, false, false, 1>();
    else if (c.cl && c.direct) f.template run<false, true, true, false, 1>();
    else if (c.cl) f.template run<false, true, false, false, 1>();
    else if (K == 1) dispatch_plain<1>(c, f);
    else if (K == 2) dispatch_plain<2>(c, f);
    else if (K == 4) dispatch_plain<4>(c, f);
    else return false;
    return true;
}

}  // namespace

cudaError_t launch_batch_sweep(const SweepParams* sys, const int2* items, int n_items, int* counter,
                               int walkers_per_cta, int warps_per_walker, int grid, int region, BatchClass c,
                               cudaStream_t s) {
    if (n_items <= 0) return cudaSuccess;
    if (walkers_per_cta < 1 || warps_per_walker * walkers_per_cta > batch_max_warps(c.da) || grid < 1)
        return cudaErrorInvalidValue;
    Launch f{sys, items, n_items, counter, walkers_per_cta, grid, region, s};
    if (!dispatch(c, warps_per_walker, f)) return cudaErrorInvalidValue;
    return f.err;
}

cudaError_t batch_prepare(int max_smem) {
    Prepare f{max_smem};
    for (int bits = 0; bits < 16; ++bits)
        for (int K = 1; K <= 4; K *= 2)
            dispatch(BatchClass{(bits & 1) != 0, (bits & 2) != 0, (bits & 4) != 0, (bits & 8) != 0}, K, f);
    return f.err;
}

int batch_occupancy(int walkers_per_cta, int warps_per_walker, int region, BatchClass c) {
    Occupancy f{walkers_per_cta, (size_t)walkers_per_cta * region};   // within the limit batch_prepare set
    return dispatch(c, warps_per_walker, f) ? f.n : 0;
}

}  // namespace regc
