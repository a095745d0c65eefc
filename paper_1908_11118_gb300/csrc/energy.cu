// energy.cu -- from-scratch energies of every walker (sm_103a).
#include "cells.cuh"
#include "launch.h"

namespace regc {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// Displacement q - p with the exact minimum image on periodic axes (cell
// frame), x made Cartesian.
__device__ __forceinline__ void disp_exact(const Geometry& g, float4 q, float4 p, float& dx, float& dy, float& dz) {
    dy = min_image_exact(q.y, p.y, g.Ly, g.hLy);
    dx = cart_dx(g, min_image_exact(q.x, p.x, g.Lx, g.hLx), dy);
    dz = g.periodic_z ? min_image_exact(q.z, p.z, g.Lz, g.hLz) : __fsub_rn(q.z, p.z);
}

// From-scratch energy of every walker: every unordered pair of particles and
// every particle-surface pair, with the nearest periodic image.  A walker gets
// kEnergySplit CTAs of kEnergyThreads threads; its positions are staged in
// shared memory.  Two enumerations of the mobile pairs:
//
// * cells (the cell grid of the sweep has at least three cells along every
//   periodic axis, so the 27 cells around a cell are distinct): every CTA
//   builds the walker's cell list (shared-memory atomics; the order inside a
//   cell does not matter) and takes items (i, o) -- particle i against the
//   o-th cell of the forward half of its stencil (o = 0: its own cell, partners
//   j > i; o = 1..13: the 13 offsets after (0, 0, 0) in (z, y, x) order) --
//   which lists every pair within rc once;
// * all pairs (small periodic boxes, or a cell over capacity): the circulant
//   order (i, i + d mod N), d = 1 .. floor(N / 2) (for even N the offset N / 2
//   only from i < N / 2), which lists each unordered pair once and gives every
//   particle the same number of partners.
//
// Consecutive threads take consecutive items.  The displacement is
// antisymmetric under exchange of the pair (min_image_exact and cart_dx round
// -x to -fl(x)), so r^2, hence every pair term, is the one the sweep computes
// for that pair.  The surface partners of a particle come from its column of
// the surface table, one warp per particle, exactly as in the sweep.  Partial
// sums are folded to 64 bits before the int32 parts of a Fix3 can overflow and
// added to the walker's total with a 64-bit integer atomic: fixed-point sums do
// not depend on the order, so the result is deterministic and equals the
// sweep's running total exactly.
//
// What bounds it is the latency of a thread's candidates: two are taken at a
// time without branches, and a particle's surface terms are folded only when
// needed.  Setting 1024 fcc(111) walkers, a sweep launch and reading them back:
// 441 -> 431 us; ten MD steps with the energies after them 1153 -> 1121 us.  Two
// CTAs per walker are slower (440 us, one: 466), eight no faster (434).
constexpr int kEnergyThreads = 256;
constexpr int kEnergySplit = 4;
constexpr int kEnergyTeam = kEnergySplit * kEnergyThreads;
constexpr int kFoldEvery = 256;   // pair terms per thread between folds (|lo| < 2^21 per term)

struct EnergyAcc {
    Fix3 acc;
    long long total;
    int folds, n_in, overlap;
    __device__ __forceinline__ void add(float phi) {
        fix_add(acc, phi, 1);
        if (++folds == kFoldEvery) fold();
    }
    __device__ __forceinline__ void fold() {
        total += fix_value(acc.big, acc.hi, acc.lo);
        acc = Fix3{0, 0, 0};
        folds = 0;
    }
};

// One candidate of a cell item, without branches: a pair left out or out of
// range enters as 0.
template <bool CL>
__device__ __forceinline__ void energy_term(const SweepParams& P, float4 p, float4 q, bool iA, bool jA, bool use,
                                            EnergyAcc& a) {
    const PairTab& tp = CL ? (iA ? (jA ? P.gA : P.gAB) : (jA ? P.gAB : P.gg)) : P.gg;
    float dx, dy, dz;
    disp_exact(P.g, p, q, dx, dy, dz);
    const float r2 = r2_of(dx, dy, dz);
    const float phi = phi_of_r2(r2, tp);   // (r2 = 0: the particle itself, dropped)
    const bool in = use && r2 < P.g.rc2;
    a.n_in += in;
    a.overlap |= in && r2 < tp.rhc2;
    fix_add(a.acc, in ? phi : 0.f, 1);
}

template <bool CL>
__device__ __forceinline__ void energy_pair(const SweepParams& P, const float4* sp, int i, int j, int split,
                                            EnergyAcc& a) {
    const bool iA = CL && i < split, jA = CL && j < split;
    const PairTab& tp = iA ? (jA ? P.gA : P.gAB) : (jA ? P.gAB : P.gg);
    float dx, dy, dz;
    disp_exact(P.g, sp[i], sp[j], dx, dy, dz);
    a.add(pair_phi(dx, dy, dz, P.g.rc2, tp, a.n_in, a.overlap));
}

// Fixed-point energy of a particle against the images of frozen surface atoms
// listed for its column (the sweep's terms).
template <bool CL>
__device__ __forceinline__ void surface_pass(const SweepParams& P, int col, float4 q, EnergyAcc& e, int lane,
                                             bool mA) {
    const int beg = col * P.st.stride, end = beg + P.st.stride;
    for (int j = beg + lane; j < end; j += 32) {
        const float4 a = __ldg(&P.st.atoms[j]);
        const unsigned bits = __float_as_uint(a.w);
        const PairTab& t = (CL && mA) ? P.gsA[bits & 3u] : surf_tab(P, (int)(bits & 3u));
        const float sx = (bits & 4u) ? P.g.Lx : 0.f, sy = (bits & 8u) ? P.g.Ly : 0.f;
        const float sz = (bits & 16u) ? P.g.Lz : 0.f;
        const float dy = __fsub_rn(__fsub_rn(q.y, sy), a.y);
        fix_add(e.acc, pair_phi(cart_dx(P.g, __fsub_rn(__fsub_rn(q.x, sx), a.x), dy), dy,
                                __fsub_rn(__fsub_rn(q.z, sz), a.z), P.g.rc2, t, e.n_in, e.overlap), 1);
    }
}

template <bool CL>
__global__ void __launch_bounds__(kEnergyThreads) energy_kernel(const __grid_constant__ SweepParams P,
                                                                unsigned long long* out, int check_overlap,
                                                                int use_cells) {
    extern __shared__ float4 sp[];   // [nmax] positions (w: packed cell), then cnt [ncell], slots [ncell][cap]
    int* cnt = reinterpret_cast<int*>(sp + P.nmax);
    uint16_t* slots = reinterpret_cast<uint16_t*>(cnt + ((P.cg.ncell + 3) & ~3));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int w = blockIdx.x / kEnergySplit, c = blockIdx.x % kEnergySplit;
    const int N = P.n[w];
    const int split = CL ? (P.gc2 ? P.nb[w] : P.n_cluster) : 0;   // two mobile species: the boundary
    const int t = c * kEnergyThreads + threadIdx.x;
    const float4* pos = P.pos + size_t(w) * P.nmax;
    if (use_cells)
        for (int k = threadIdx.x; k < P.cg.ncell; k += kEnergyThreads) cnt[k] = 0;
    for (int i = threadIdx.x; i < N; i += kEnergyThreads) {
        float4 q = pos[i];
        if (use_cells) {
            const Cell3 cc = cell3_of(P, q.x, q.y, q.z);
            q.w = __uint_as_float((unsigned)cc.x | ((unsigned)cc.y << 10) | ((unsigned)cc.z << 20));
        }
        sp[i] = q;
    }
    __syncthreads();
    bool cells = false;
    if (use_cells) {
        int full = 0;
        for (int i = threadIdx.x; i < N; i += kEnergyThreads) {
            const unsigned b = __float_as_uint(sp[i].w);
            const int cell = (int)(((b >> 20) * P.cg.ncy + ((b >> 10) & 1023u)) * P.cg.ncx + (b & 1023u));
            const int k = atomicAdd(cnt + cell, 1);
            if (k < P.cg.cap) slots[cell * P.cg.cap + k] = (uint16_t)i;
            else full = 1;
        }
        cells = !__syncthreads_or(full);   // identical in every CTA of the walker (counts are)
    }
    EnergyAcc a{{0, 0, 0}, 0, 0, 0, 0};
    if (cells) {
        // item k = 14 i + o; this thread takes k = t, t + T, ... (one division)
        int i = t / 14, o = t % 14;
        constexpr int qT = kEnergyTeam / 14, rT = kEnergyTeam % 14;
        while (i < N) {
            const unsigned b = __float_as_uint(sp[i].w);
            const int idx = 13 + o;   // offset (ox, oy, oz) = (idx % 3, idx / 3 % 3, idx / 9) - 1
            int nx = (int)(b & 1023u) + idx % 3 - 1;
            int ny = (int)((b >> 10) & 1023u) + (idx / 3) % 3 - 1;
            int nz = (int)(b >> 20) + idx / 9 - 1;
            if (nx < 0) nx += P.cg.ncx;
            else if (nx >= P.cg.ncx) nx -= P.cg.ncx;
            if (ny < 0) ny += P.cg.ncy;
            else if (ny >= P.cg.ncy) ny -= P.cg.ncy;
            bool ok = true;
            if (nz >= P.cg.ncz) {
                if (P.g.periodic_z) nz -= P.cg.ncz;
                else ok = false;
            }
            if (ok) {
                const int cell = (nz * P.cg.ncy + ny) * P.cg.ncx + nx;
                const int n_c = cnt[cell];
                const uint16_t* sl = slots + cell * P.cg.cap;
                const float4 p = sp[i];
                const bool iA = CL && i < split;
#pragma unroll 1
                for (int m = 0; m < n_c; m += 2) {   // two partners at a time
                    const bool two = m + 1 < n_c;
                    const int j0 = sl[m], j1 = sl[two ? m + 1 : m];
                    const float4 q0 = sp[j0], q1 = sp[j1];
                    energy_term<CL>(P, p, q0, iA, CL && j0 < split, o != 0 || j0 > i, a);
                    energy_term<CL>(P, p, q1, iA, CL && j1 < split, two && (o != 0 || j1 > i), a);
                    if ((a.folds += 2) >= kFoldEvery) a.fold();
                }
            }
            o += rT;
            i += qT;
            if (o >= 14) {
                o -= 14;
                i += 1;
            }
        }
    } else if (N >= 2) {
        // item k = (d - 1) N + i, d = 1 .. D
        const int D = N >> 1;
        int i = t % N, d = t / N + 1;
        const int qT = kEnergyTeam / N, rT = kEnergyTeam % N;
        const bool even = (N & 1) == 0;
        while (d <= D) {
            if (!(even && d == D && i >= D)) {
                int j = i + d;
                if (j >= N) j -= N;
                energy_pair<CL>(P, sp, i, j, split, a);
            }
            i += rT;
            d += qT;
            if (i >= N) {
                i -= N;
                d += 1;
            }
        }
    }
    a.fold();
    // surface partners: one warp per particle
    for (int i = c * (kEnergyThreads / 32) + warp; i < N; i += kEnergyTeam / 32) {
        const float4 pi = sp[i];
        if (near_surface(P, pi.z)) {
            const int terms = P.st.stride / 32;
            if (a.folds + terms > kFoldEvery) a.fold();
            a.folds += terms;
            surface_pass<CL>(P, surface_col(P, pi.x, pi.y), pi, a, lane, CL && i < split);
        }
    }
    // each warp adds its share (two's complement: exact, in any order) and
    // leaves; no barrier after the items, so a warp that finished early exits
    a.fold();
    const long long total = warp_sum_ll(a.total);
    const int overlap = __any_sync(FULL, a.overlap);
    if (lane == 0) {
        if (total != 0) atomicAdd(out + w, (unsigned long long)total);
        if (overlap && check_overlap) atomicOr(P.error, check_overlap == 2 ? ERR_NUMERIC : ERR_OVERLAP);
    }
}

}  // namespace

cudaError_t launch_energy(const SweepParams& P, long long* out, int check_overlap, cudaStream_t s) {
    constexpr size_t kMaxSmem = 232448;   // 227 KB per block
    const size_t base = size_t(P.nmax) * sizeof(float4);
    const size_t with_cells = base + size_t((P.cg.ncell + 3) & ~3) * 4 + size_t(P.cg.ncell) * P.cg.cap * 2;
    // cells: 27 distinct stencil cells, cell coordinates packed in 10 bits each
    const int use_cells = P.cg.ncx >= 3 && P.cg.ncy >= 3 && (!P.g.periodic_z || P.cg.ncz >= 3) &&
                          P.cg.ncx < 1024 && P.cg.ncy < 1024 && P.cg.ncz < 1024 && with_cells + 1024 <= kMaxSmem;
    const size_t smem = use_cells ? with_cells : base;
    // the pair tables of a second species only where the walkers hold a cluster
    auto kernel = (P.n_cluster > 0 || P.gc2) ? energy_kernel<true> : energy_kernel<false>;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaMemsetAsync(out, 0, size_t(P.S) * sizeof(long long), s);
    if (e != cudaSuccess) return e;
    kernel<<<P.S * kEnergySplit, kEnergyThreads, smem, s>>>(P, reinterpret_cast<unsigned long long*>(out),
                                                            check_overlap, use_cells);
    return cudaGetLastError();
}

}  // namespace regc
