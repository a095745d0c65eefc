// md.cu -- molecular-dynamics segments of every walker (REGCMD), sm_103a.
//
// Sec. II.A.3: the canonical sampling between grand-canonical and exchange
// moves may be done by MD instead of Metropolis displacements; Appendix:
// velocity Verlet with the stochastic velocity rescaling thermostat.  One CTA
// of kMdWarps warps per walker; thread t owns particles t, t + 128, ...
// Per segment:
//   - velocities drawn from the Maxwell-Boltzmann distribution at the
//     walker's kT (particle i: Philox counter (i, seg, w, 8), Box-Muller);
//   - every step: the thermostat of Bussi, Donadio & Parrinello (2007) with
//     time constant tau over all 3N degrees of freedom (normals from counters
//     (k, seg * n_steps + step, w, 9)), then velocity Verlet
//     (v += f dt/2, r += v dt, cells rebuilt, f = F(r), v += f dt/2);
//   - forces from the distinct neighbour cells (nearest image) and the
//     particle's surface column, FP32; per-particle sums in a fixed order (cells
//     in (z, y, x) order, particles of a cell by index, then the column), so a
//     segment is reproducible;
//   - x, y periodic (z too in a periodic box), else walls at z_lo and z_hi
//     reflect;
//   - positions and (optionally) kinetic energies back to HBM; the caller
//     recomputes the exact energies.
#include "cells.cuh"
#include "launch.h"

namespace regc {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kMdWarps = 4;
constexpr int kMdThreads = 32 * kMdWarps;

__host__ __device__ inline size_t md_align16(size_t v) { return (v + 15) & ~size_t(15); }

__host__ __device__ inline size_t md_smem_bytes(int nmax, int ncell, int cap) {
    return 3 * md_align16(size_t(nmax) * 16) + md_align16(size_t(ncell) * 2) + md_align16(size_t(ncell) * cap * 2);
}

// Four standard normals from one Philox block (Box-Muller on words 0-1, 2-3;
// uniforms from the top 24 bits, offset by half a step so that none is 0).
__device__ __forceinline__ void normals4(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                         uint32_t k1, float g[4]) {
    const U4 u = philox(c0, c1, c2, c3, k0, k1);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float u1 = ((float)(w[2 * h] >> 8) + 0.5f) * (1.0f / 16777216.0f);
        const float u2 = ((float)(w[2 * h + 1] >> 8) + 0.5f) * (1.0f / 16777216.0f);
        const float r = sqrtf(-2.0f * logf(u1));
        g[2 * h] = r * cospif(2.0f * u2);
        g[2 * h + 1] = r * sinpif(2.0f * u2);
    }
}

// Sum of one float per thread over the CTA in a fixed order; every thread
// receives the sum.
__device__ __forceinline__ float cta_sum(float v, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    const int warp = threadIdx.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[warp] = v;
    __syncthreads();
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kMdWarps; ++k) s += red[k];
    return s;
}

// Three such sums at once.
__device__ __forceinline__ void cta_sum3(float (&v)[3], float (*red)[kMdWarps]) {
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(FULL, v[q], o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int q = 0; q < 3; ++q) red[q][threadIdx.x >> 5] = v[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        v[q] = 0.f;
#pragma unroll
        for (int k = 0; k < kMdWarps; ++k) v[q] += red[q][k];
    }
}

// Drift of a particle at p with velocity (vx, vy, vz), wrapped or reflected.
__device__ __forceinline__ void md_drift(const SweepParams& P, float dt, float vx, float vy, float& vz, float4& p) {
    p.x = fmaf(dt, fmaf(-P.g.shear, vy, vx), p.x);   // u = x - shear y
    p.y = fmaf(dt, vy, p.y);
    p.z = fmaf(dt, vz, p.z);
    if (p.x < 0.f) p.x += P.g.Lx;
    if (p.x >= P.g.Lx) p.x -= P.g.Lx;
    if (p.y < 0.f) p.y += P.g.Ly;
    if (p.y >= P.g.Ly) p.y -= P.g.Ly;
    if (P.g.periodic_z) {
        if (p.z < 0.f) p.z += P.g.Lz;
        if (p.z >= P.g.Lz) p.z -= P.g.Lz;
    } else {
        if (p.z < P.g.z_lo) { p.z = 2.0f * P.g.z_lo - p.z; vz = -vz; }
        if (p.z > P.g.z_hi) { p.z = 2.0f * P.g.z_hi - p.z; vz = -vz; }
        p.z = fminf(fmaxf(p.z, P.g.z_lo), P.g.z_hi);
    }
    if (!(p.x >= 0.f && p.x < P.g.Lx)) p.x = 0.f;   // rounding at the boundary
    if (!(p.y >= 0.f && p.y < P.g.Ly)) p.y = 0.f;
    if (P.g.periodic_z && !(p.z >= 0.f && p.z < P.g.Lz)) p.z = 0.f;
}

// The range of distinct cell offsets along one axis of n cells: periodic
// -1..1 while those are distinct cells (0..1 for two cells, 0 for one),
// otherwise the offsets that stay inside the grid.  With nearest-image
// displacements a cell visited twice would count its pairs twice.
__device__ __forceinline__ void axis_range(int c, int n, bool periodic, int& lo, int& hi) {
    if (periodic) {
        lo = n >= 3 ? -1 : 0;
        hi = n >= 2 ? 1 : 0;
    } else {
        lo = c > 0 ? -1 : 0;
        hi = c < n - 1 ? 1 : 0;
    }
}

__device__ __forceinline__ void lj_force_add(const PairTab& t, float r2, float dx, float dy, float dz, float& fx,
                                             float& fy, float& fz) {
    const float inv = __fdividef(1.0f, r2);
    const float s2 = t.sig2 * inv;
    const float s6 = s2 * s2 * s2;
    const float g = 6.0f * t.eps4 * (2.0f * s6 * s6 - s6) * inv;   // 24 eps (2 s^12 - s^6) / r^2
    fx = fmaf(g, dx, fx);
    fy = fmaf(g, dy, fy);
    fz = fmaf(g, dz, fz);
}

// The pair of particles i at p and j at q: add the force on i if within rc.
template <bool CL>
__device__ __forceinline__ void md_pair(const SweepParams& P, float4 p, float4 q, bool iA, int j, float& fx,
                                        float& fy, float& fz) {
    const float dy = min_image_exact(p.y, q.y, P.g.Ly, P.g.hLy);
    const float dx = cart_dx(P.g, min_image_exact(p.x, q.x, P.g.Lx, P.g.hLx), dy);
    const float dz = P.g.periodic_z ? min_image_exact(p.z, q.z, P.g.Lz, P.g.hLz) : p.z - q.z;
    const float r2 = r2_of(dx, dy, dz);
    if (r2 < P.g.rc2) {
        const bool jA = CL && j < P.n_cluster;
        const PairTab& t = CL ? (iA ? (jA ? P.gA : P.gAB) : (jA ? P.gAB : P.gg)) : P.gg;
        lj_force_add(t, r2, dx, dy, dz, fx, fy, fz);
    }
}

// The force on a particle at p from its surface column.
template <bool CL>
__device__ __forceinline__ void md_surface(const SweepParams& P, float4 p, bool iA, float& fx, float& fy, float& fz) {
    if (near_surface(P, p.z)) {
        const int beg = surface_col(P, p.x, p.y) * P.st.stride;
        for (int k = beg; k < beg + P.st.stride; ++k) {
            const float4 at = __ldg(&P.st.atoms[k]);
            const unsigned bits = __float_as_uint(at.w);
            if (bits & 32u) break;   // padding: the column's images are listed first
            const PairTab& t = (CL && iA) ? P.gsA[bits & 3u] : P.gs[bits & 3u];
            const float sx = (bits & 4u) ? P.g.Lx : 0.f, sy = (bits & 8u) ? P.g.Ly : 0.f;
            const float sz = (bits & 16u) ? P.g.Lz : 0.f;
            const float dy = (p.y - sy) - at.y, dz = (p.z - sz) - at.z;
            const float dx = cart_dx(P.g, (p.x - sx) - at.x, dy);
            const float r2 = r2_of(dx, dy, dz);
            if (r2 < P.g.rc2) lj_force_add(t, r2, dx, dy, dz, fx, fy, fz);
        }
    }
}

// Force on particle i at p through the cell list.
template <bool CL>
__device__ __forceinline__ float3 md_force(const SweepParams& P, const float4* pos, const uint16_t* cnt,
                                           const uint16_t* slots, int i, float4 p) {
    float fx = 0.f, fy = 0.f, fz = 0.f;
    const bool iA = CL && i < P.n_cluster;
    const Cell3 c = cell3_of(P, p.x, p.y, p.z);
    int xlo, xhi, ylo, yhi, zlo, zhi;
    axis_range(c.x, P.cg.ncx, true, xlo, xhi);
    axis_range(c.y, P.cg.ncy, true, ylo, yhi);
    axis_range(c.z, P.cg.ncz, P.g.periodic_z != 0, zlo, zhi);
    for (int a = zlo; a <= zhi; ++a)
        for (int b = ylo; b <= yhi; ++b)
            for (int d = xlo; d <= xhi; ++d) {
                int cz = c.z + a, cy = c.y + b, cx = c.x + d;   // wrapped into the grid
                if (cz < 0) cz += P.cg.ncz;
                if (cz >= P.cg.ncz) cz -= P.cg.ncz;
                if (cy < 0) cy += P.cg.ncy;
                if (cy >= P.cg.ncy) cy -= P.cg.ncy;
                if (cx < 0) cx += P.cg.ncx;
                if (cx >= P.cg.ncx) cx -= P.cg.ncx;
                const int cell = (cz * P.cg.ncy + cy) * P.cg.ncx + cx;
                const int m = cnt[cell];
                for (int s = 0; s < m; ++s) {
                    const int j = slots[cell * P.cg.cap + s];
                    if (j == i) continue;
                    const float4 q = pos[j];
                    md_pair<CL>(P, p, q, iA, j, fx, fy, fz);
                }
            }
    md_surface<CL>(P, p, iA, fx, fy, fz);
    return make_float3(fx, fy, fz);
}

template <bool CL>
__device__ __forceinline__ void forces_all(const SweepParams& P, const float4* pos, const uint16_t* cnt,
                                           const uint16_t* slots, float4* frc, float4* vel, int N, float half_dt,
                                           bool kick) {
    for (int i = threadIdx.x; i < N; i += kMdThreads) {
        const float3 f = md_force<CL>(P, pos, cnt, slots, i, pos[i]);
        frc[i] = make_float4(f.x, f.y, f.z, 0.f);
        if (kick) {
            float4 v = vel[i];
            v.x = fmaf(half_dt, f.x, v.x);
            v.y = fmaf(half_dt, f.y, v.y);
            v.z = fmaf(half_dt, f.z, v.z);
            vel[i] = v;
        }
    }
}

template <bool CL>
__global__ void __launch_bounds__(kMdThreads) md_kernel(const __grid_constant__ SweepParams P, int n_steps, float dt,
                                                        double c_tau, uint32_t seg, float* kin_out) {
    extern __shared__ __align__(16) char smem[];
    __shared__ float red[kMdWarps];
    __shared__ float alpha_sh;
    const int w = blockIdx.x;
    if (w >= P.S) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float4* pos = reinterpret_cast<float4*>(smem);
    float4* vel = reinterpret_cast<float4*>(smem + md_align16(size_t(P.nmax) * 16));
    float4* frc = reinterpret_cast<float4*>(smem + 2 * md_align16(size_t(P.nmax) * 16));
    uint16_t* cnt = reinterpret_cast<uint16_t*>(smem + 3 * md_align16(size_t(P.nmax) * 16));
    uint16_t* slots = cnt + md_align16(size_t(P.cg.ncell) * 2) / 2;
    const int N = P.n[w];
    const int s = P.state_of_walker[w];
    const float kT = (float)(1.0 / P.beta[s]);
    float4* gpos = P.pos + size_t(w) * P.nmax;

    for (int i = tid; i < N; i += kMdThreads) {
        pos[i] = gpos[i];
        float g[4];
        normals4((uint32_t)i, seg, (uint32_t)w, 8u, P.key0, P.key1, g);
        const float sk = sqrtf(kT);
        vel[i] = make_float4(sk * g[0], sk * g[1], sk * g[2], 0.f);
    }
    __syncthreads();
    if (warp == 0) build_cell_list(P, pos, N, cnt, slots, lane);
    __syncthreads();
    forces_all<CL>(P, pos, cnt, slots, frc, vel, N, 0.5f * dt, false);
    __syncthreads();

    const int nf = 3 * N;
    const double Kt = 0.5 * nf * (double)kT;
    for (int step = 0; step < n_steps && N > 0; ++step) {
        // thermostat: kinetic energy and the normals of this step
        float kp = 0.f, chi = 0.f, r1 = 0.f;
        for (int i = tid; i < N; i += kMdThreads) {
            const float4 v = vel[i];
            kp += 0.5f * (v.x * v.x + v.y * v.y + v.z * v.z);
        }
        const uint32_t gstep = seg * (uint32_t)n_steps + (uint32_t)step;
        for (int k = tid; 4 * k < nf; k += kMdThreads) {
            float g[4];
            normals4((uint32_t)k, gstep, (uint32_t)w, 9u, P.key0, P.key1, g);
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int idx = 4 * k + h;
                if (idx == 0) r1 = g[h];
                else if (idx < nf) chi += g[h] * g[h];
            }
        }
        const float K = cta_sum(kp, red);
        const float CHI = cta_sum(chi, red);
        const float R1 = cta_sum(r1, red);   // only thread 0 contributes
        if (tid == 0) {
            double a = 1.0;
            if (K > 0.f) {
                const double k_new = c_tau * K + (1.0 - c_tau) * Kt * ((double)R1 * R1 + CHI) / nf +
                                     2.0 * R1 * sqrt(c_tau * (1.0 - c_tau) * K * Kt / nf);
                a = sqrt(fmax(k_new, 0.0) / K);
                if (R1 + sqrt(c_tau * nf * K / ((1.0 - c_tau) * Kt)) < 0.0) a = -a;
            }
            alpha_sh = (float)a;
        }
        __syncthreads();
        const float alpha = alpha_sh;
        // half kick, drift, walls
        for (int i = tid; i < N; i += kMdThreads) {
            float4 v = vel[i];
            const float4 f = frc[i];
            v.x = fmaf(0.5f * dt, f.x, alpha * v.x);
            v.y = fmaf(0.5f * dt, f.y, alpha * v.y);
            v.z = fmaf(0.5f * dt, f.z, alpha * v.z);
            float4 p = pos[i];
            md_drift(P, dt, v.x, v.y, v.z, p);
            pos[i] = p;
            vel[i] = v;
        }
        __syncthreads();
        if (warp == 0) build_cell_list(P, pos, N, cnt, slots, lane);
        __syncthreads();
        forces_all<CL>(P, pos, cnt, slots, frc, vel, N, 0.5f * dt, true);
        __syncthreads();
    }
    float kp = 0.f;
    for (int i = tid; i < N; i += kMdThreads) {
        const float4 v = vel[i];
        kp += 0.5f * (v.x * v.x + v.y * v.y + v.z * v.z);
        const float4 p = pos[i];
        gpos[i] = make_float4(p.x, p.y, p.z, 0.f);
    }
    const float K = cta_sum(kp, red);
    if (tid == 0 && kin_out) kin_out[w] = K;
}

// ---- up to kMdRegs kMdThreads particles: the same segment with velocities in
// registers (thread t owns particles t, t + 128, ..) and, instead of cells of
// fixed capacity, the particles sorted by cell: a row of neighbour cells is then
// one contiguous run of positions (two where it wraps), read without an index
// in between.  Per particle the partners come in the order of the cell list, so
// the force sums are the same bit for bit.
//
// What bounds it: the warps' instructions.  A warp runs as long as the lane with
// the most partners; over 27 cells one by one that was some four times the mean
// (the largest of 32 Poisson counts, 27 times over).  Forces are therefore
// computed in sorted order -- the lanes of a warp stand in neighbouring cells,
// walk rows of nearly equal length, often the same addresses, and reach the
// surface together -- and handed to the owners through shared memory.  That
// memory falls from 39 to 27 KB at Nmax 512, so seven walkers share an SM
// instead of five and the 1024 walkers of the fcc(111) grid run in one wave.
// That launch then takes as long as its densest walker, whose few warps wait for
// their own results (ncu: 31 % of the issue slots used, 10 cycles an instruction,
// 3.4 of them for a fixed latency, 1.2 for shared memory, 1.0 for a branch): a
// lane takes two partners at a time, without branches, and adds their terms in
// order.  Ten steps: 1250 -> 790 us.  (Eight warps per walker for the forces,
// four walkers per SM: 900 us.)
constexpr int kMdRegs = 4;

__host__ __device__ inline size_t md_regs_smem(int nmax, int ncell) {
    return 3 * md_align16(size_t(nmax) * 16) + md_align16(size_t(nmax) * 2) + md_align16(size_t(ncell + 1) * 4) +
           md_align16(size_t(ncell) * 4);
}

struct MdSorted {
    float4* pos;      // [nmax] by particle
    float4* srt;      // [nmax] by cell, w: the particle's index
    float4* frc;      // [nmax] by particle
    uint16_t* order;  // [nmax] particles by cell, by index within one
    int* start;       // [ncell + 1]
    int* fill;        // [ncell]
};

// Sort the particles by cell, by index within a cell (every thread of the CTA).
// A cell beyond the cell list's capacity sets ERR_CAPACITY.
// The counts are scanned by one warp: 32 cells at a time, or (WIDE) a run of cells
// per lane, so that it exchanges sums once.  A large and nearly empty box waits for
// that scan: ten steps of 10 particles in 1728 cells, 16 walkers, 323 / 273 us (in
// the kernel with a list of fixed capacity 273), of 30 in 1000 cells, 1024 walkers, 351
// / 306, of 30 in 512 cells, 16 walkers, 291 / 269; the fcc(111) grid's 168 cells
// 4782 / 4838 us a pass.
constexpr int kWideCells = 256;
template <bool WIDE>
__device__ __forceinline__ void md_sort(const SweepParams& P, const MdSorted& S, int N) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int ncell = P.cg.ncell;
    for (int c = tid; c < ncell; c += kMdThreads) S.fill[c] = 0;
    __syncthreads();
    for (int i = tid; i < N; i += kMdThreads) {
        const float4 p = S.pos[i];
        atomicAdd(S.fill + cell_of(P, p.x, p.y, p.z), 1);
    }
    __syncthreads();
    if (WIDE && tid < 32) {   // exclusive scan
        const int per = ((ncell + 31) / 32) | 1;   // odd: the lanes stand in different banks
        const int c0 = min(ncell, lane * per), c1 = min(ncell, c0 + per);
        int mine = 0;
#pragma unroll 4
        for (int c = c0; c < c1; ++c) mine += S.fill[c];
        int v = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, v, o);
            if (lane >= o) v += u;
        }
        int run = v - mine;
        bool full = false;
#pragma unroll 4
        for (int c = c0; c < c1; ++c) {
            const int n = S.fill[c];
            S.start[c] = S.fill[c] = run;
            full |= n > P.cg.cap;
            run += n;
        }
        if (full) atomicOr(P.error, ERR_CAPACITY);
        if (lane == 31) S.start[ncell] = run;
    }
    if (!WIDE && tid < 32) {
        int run = 0;
        for (int c0 = 0; c0 < ncell; c0 += 32) {
            const int c = c0 + lane;
            const int n = c < ncell ? S.fill[c] : 0;
            int v = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(FULL, v, o);
                if (lane >= o) v += u;
            }
            if (c < ncell) {
                S.start[c] = run + v - n;
                S.fill[c] = run + v - n;
                if (n > P.cg.cap) atomicOr(P.error, ERR_CAPACITY);
            }
            run += __shfl_sync(FULL, v, 31);
        }
        if (lane == 0) S.start[ncell] = run;
    }
    __syncthreads();
    for (int i = tid; i < N; i += kMdThreads) {
        const float4 p = S.pos[i];
        S.order[atomicAdd(S.fill + cell_of(P, p.x, p.y, p.z), 1)] = (uint16_t)i;
    }
    __syncthreads();
    for (int c = tid; c < ncell; c += kMdThreads) {   // into index order
        const int b0 = S.start[c], b1 = S.start[c + 1];
        for (int k = b0 + 1; k < b1; ++k) {
            const uint16_t x = S.order[k];
            int q = k;
            for (; q > b0 && S.order[q - 1] > x; --q) S.order[q] = S.order[q - 1];
            S.order[q] = x;
        }
    }
    __syncthreads();
    for (int k = tid; k < N; k += kMdThreads) {
        const int i = S.order[k];
        const float4 p = S.pos[i];
        S.srt[k] = make_float4(p.x, p.y, p.z, __int_as_float(i));
    }
    __syncthreads();
}

// The force of one partner without a branch: g (dx, dy, dz), g = 0 where `use` does
// not hold, the partner is the particle itself or lies beyond rc.
struct MdTerm {
    float g, dx, dy, dz;
};
__device__ __forceinline__ float lj_force_g(const PairTab& t, float r2) {
    const float inv = __fdividef(1.0f, r2);
    const float s2 = t.sig2 * inv;
    const float s6 = s2 * s2 * s2;
    return 6.0f * t.eps4 * (2.0f * s6 * s6 - s6) * inv;
}
template <bool CL>
__device__ __forceinline__ MdTerm md_term(const SweepParams& P, float4 p, float4 q, bool iA, int i, bool use) {
    MdTerm m;
    const int j = __float_as_int(q.w);
    m.dy = min_image_exact(p.y, q.y, P.g.Ly, P.g.hLy);
    m.dx = cart_dx(P.g, min_image_exact(p.x, q.x, P.g.Lx, P.g.hLx), m.dy);
    m.dz = P.g.periodic_z ? min_image_exact(p.z, q.z, P.g.Lz, P.g.hLz) : p.z - q.z;
    const float r2 = r2_of(m.dx, m.dy, m.dz);
    const bool jA = CL && j < P.n_cluster;
    const float g = lj_force_g(CL ? (iA ? (jA ? P.gA : P.gAB) : (jA ? P.gAB : P.gg)) : P.gg, r2);
    m.g = use && j != i && r2 < P.g.rc2 ? g : 0.f;
    return m;
}
__device__ __forceinline__ void md_add(const MdTerm& m, float& fx, float& fy, float& fz) {
    fx = fmaf(m.g, m.dx, fx);
    fy = fmaf(m.g, m.dy, fy);
    fz = fmaf(m.g, m.dz, fz);
}

template <bool CL>
__device__ __forceinline__ float3 md_force_sorted(const SweepParams& P, const MdSorted& S, int i, float4 p) {
    float fx = 0.f, fy = 0.f, fz = 0.f;
    const bool iA = CL && i < P.n_cluster;
    const Cell3 c = cell3_of(P, p.x, p.y, p.z);
    int xlo, xhi, ylo, yhi, zlo, zhi;
    axis_range(c.x, P.cg.ncx, true, xlo, xhi);
    axis_range(c.y, P.cg.ncy, true, ylo, yhi);
    axis_range(c.z, P.cg.ncz, P.g.periodic_z != 0, zlo, zhi);
    // the row's cells xlo .. xhi, wrapped: cells a0 .. a1 - 1, then 0 .. b1 - 1
    int a0 = c.x + xlo, a1 = c.x + xhi + 1, b1 = 0;
    if (a0 < 0) {
        b1 = a1;
        a0 += P.cg.ncx;
        a1 = P.cg.ncx;
    } else if (a1 > P.cg.ncx) {
        b1 = a1 - P.cg.ncx;
        a1 = P.cg.ncx;
    }
    for (int a = zlo; a <= zhi; ++a)
        for (int b = ylo; b <= yhi; ++b) {
            int cz = c.z + a, cy = c.y + b;
            if (cz < 0) cz += P.cg.ncz;
            if (cz >= P.cg.ncz) cz -= P.cg.ncz;
            if (cy < 0) cy += P.cg.ncy;
            if (cy >= P.cg.ncy) cy -= P.cg.ncy;
            const int* row = S.start + (cz * P.cg.ncy + cy) * P.cg.ncx;
            const int k = row[a0], n1 = row[a1] - k;
            const int n = n1 + row[b1] - row[0], k2 = row[0] - n1;
            // one loop over both runs, two partners at a time
#pragma unroll 1
            for (int q = 0; q < n; q += 2) {
                const int q1 = min(q + 1, n - 1);
                const float4 x0 = S.srt[q + (q < n1 ? k : k2)], x1 = S.srt[q1 + (q1 < n1 ? k : k2)];
                const MdTerm t0 = md_term<CL>(P, p, x0, iA, i, true), t1 = md_term<CL>(P, p, x1, iA, i, q + 1 < n);
                md_add(t0, fx, fy, fz);
                md_add(t1, fx, fy, fz);
            }
        }
    md_surface<CL>(P, p, iA, fx, fy, fz);
    return make_float3(fx, fy, fz);
}

template <bool CL, bool WIDE>
__global__ void __launch_bounds__(kMdThreads, 7) md_regs_kernel(const __grid_constant__ SweepParams P, int n_steps,
                                                                float dt, double c_tau, uint32_t seg,
                                                                float* kin_out) {
    extern __shared__ __align__(16) char smem[];
    __shared__ float red[3][kMdWarps];
    __shared__ float alpha_sh;
    const int w = blockIdx.x;
    if (w >= P.S) return;
    const int tid = threadIdx.x;
    MdSorted S;
    char* at = smem;
    S.pos = reinterpret_cast<float4*>(at);
    at += md_align16(size_t(P.nmax) * 16);
    S.srt = reinterpret_cast<float4*>(at);
    at += md_align16(size_t(P.nmax) * 16);
    S.frc = reinterpret_cast<float4*>(at);
    at += md_align16(size_t(P.nmax) * 16);
    S.order = reinterpret_cast<uint16_t*>(at);
    at += md_align16(size_t(P.nmax) * 2);
    S.start = reinterpret_cast<int*>(at);
    at += md_align16(size_t(P.cg.ncell + 1) * 4);
    S.fill = reinterpret_cast<int*>(at);
    const int N = P.n[w];
    const int s = P.state_of_walker[w];
    const float kT = (float)(1.0 / P.beta[s]);
    float4* gpos = P.pos + size_t(w) * P.nmax;
    float3 vel[kMdRegs];

#pragma unroll
    for (int r = 0; r < kMdRegs; ++r) {
        const int i = tid + r * kMdThreads;
        vel[r] = make_float3(0.f, 0.f, 0.f);
        if (i < N) {
            S.pos[i] = gpos[i];
            float g[4];
            normals4((uint32_t)i, seg, (uint32_t)w, 8u, P.key0, P.key1, g);
            const float sk = sqrtf(kT);
            vel[r] = make_float3(sk * g[0], sk * g[1], sk * g[2]);
        }
    }
    __syncthreads();
    md_sort<WIDE>(P, S, N);
#pragma unroll 1
    for (int step = -1; step < n_steps && N > 0; ++step) {
        const bool first = step < 0;   // the forces at the start
        if (!first) {
            // thermostat: kinetic energy and the normals of this step
            const int nf = 3 * N;
            float kp = 0.f, chi = 0.f, r1 = 0.f;
#pragma unroll
            for (int r = 0; r < kMdRegs; ++r)
                if (tid + r * kMdThreads < N) {
                    const float3 v = vel[r];
                    kp += 0.5f * (v.x * v.x + v.y * v.y + v.z * v.z);
                }
            const uint32_t gstep = seg * (uint32_t)n_steps + (uint32_t)step;
            for (int k = tid; 4 * k < nf; k += kMdThreads) {
                float g[4];
                normals4((uint32_t)k, gstep, (uint32_t)w, 9u, P.key0, P.key1, g);
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int idx = 4 * k + h;
                    if (idx == 0) r1 = g[h];
                    else if (idx < nf) chi += g[h] * g[h];
                }
            }
            float sum[3] = {kp, chi, r1};   // only thread 0 contributes to r1
            cta_sum3(sum, red);
            if (tid == 0) {
                const float K = sum[0], CHI = sum[1], R1 = sum[2];
                const double Kt = 0.5 * nf * (double)kT;
                double a = 1.0;
                if (K > 0.f) {
                    const double k_new = c_tau * K + (1.0 - c_tau) * Kt * ((double)R1 * R1 + CHI) / nf +
                                         2.0 * R1 * sqrt(c_tau * (1.0 - c_tau) * K * Kt / nf);
                    a = sqrt(fmax(k_new, 0.0) / K);
                    if (R1 + sqrt(c_tau * nf * K / ((1.0 - c_tau) * Kt)) < 0.0) a = -a;
                }
                alpha_sh = (float)a;
            }
            __syncthreads();
            const float alpha = alpha_sh;
            // half kick, drift, walls
#pragma unroll
            for (int r = 0; r < kMdRegs; ++r) {
                const int i = tid + r * kMdThreads;
                if (i < N) {
                    float3 v = vel[r];
                    const float4 f = S.frc[i];
                    v.x = fmaf(0.5f * dt, f.x, alpha * v.x);
                    v.y = fmaf(0.5f * dt, f.y, alpha * v.y);
                    v.z = fmaf(0.5f * dt, f.z, alpha * v.z);
                    float4 p = S.pos[i];
                    md_drift(P, dt, v.x, v.y, v.z, p);
                    S.pos[i] = p;
                    vel[r] = v;
                }
            }
            __syncthreads();
            md_sort<WIDE>(P, S, N);
        }
#pragma unroll 1
        for (int k = tid; k < N; k += kMdThreads) {
            const float4 p = S.srt[k];
            const int i = __float_as_int(p.w);
            const float3 f = md_force_sorted<CL>(P, S, i, p);
            S.frc[i] = make_float4(f.x, f.y, f.z, 0.f);
        }
        __syncthreads();
        if (!first) {
#pragma unroll
            for (int r = 0; r < kMdRegs; ++r) {
                const int i = tid + r * kMdThreads;
                if (i < N) {
                    const float4 f = S.frc[i];
                    vel[r].x = fmaf(0.5f * dt, f.x, vel[r].x);
                    vel[r].y = fmaf(0.5f * dt, f.y, vel[r].y);
                    vel[r].z = fmaf(0.5f * dt, f.z, vel[r].z);
                }
            }
        }
    }
    float kp = 0.f;
#pragma unroll
    for (int r = 0; r < kMdRegs; ++r) {
        const int i = tid + r * kMdThreads;
        if (i < N) {
            const float3 v = vel[r];
            kp += 0.5f * (v.x * v.x + v.y * v.y + v.z * v.z);
            const float4 p = S.pos[i];
            gpos[i] = make_float4(p.x, p.y, p.z, 0.f);
        }
    }
    float sum[3] = {kp, 0.f, 0.f};
    cta_sum3(sum, red);
    if (tid == 0 && kin_out) kin_out[w] = sum[0];
}

}  // namespace

size_t md_smem(int nmax, int ncell, int cap) { return md_smem_bytes(nmax, ncell, cap); }

namespace {

template <class Kernel>
cudaError_t launch_md_kernel(Kernel kernel, size_t smem, const SweepParams& P, int n_steps, float dt, double c_tau,
                             uint32_t seg, float* kin_out, cudaStream_t s) {
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    kernel<<<P.S, kMdThreads, smem, s>>>(P, n_steps, dt, c_tau, seg, kin_out);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_md(const SweepParams& P, int n_steps, float dt, float tau, uint32_t seg, float* kin_out,
                      cudaStream_t s) {
    const double c_tau = exp(-(double)dt / (double)tau);   // thermostat decay per step
    // the sorted form where a thread's particles fit its registers
    const size_t smem_regs = md_regs_smem(P.nmax, P.cg.ncell);
    if (P.nmax <= kMdRegs * kMdThreads && smem_regs <= 232448) {   // 227 KB
        auto run = [&](auto kernel) { return launch_md_kernel(kernel, smem_regs, P, n_steps, dt, c_tau, seg, kin_out, s); };
        if (P.cg.ncell > kWideCells)
            return P.n_cluster > 0 ? run(md_regs_kernel<true, true>) : run(md_regs_kernel<false, true>);
        return P.n_cluster > 0 ? run(md_regs_kernel<true, false>) : run(md_regs_kernel<false, false>);
    }
    const size_t smem = md_smem_bytes(P.nmax, P.cg.ncell, P.cg.cap);
    return P.n_cluster > 0 ? launch_md_kernel(md_kernel<true>, smem, P, n_steps, dt, c_tau, seg, kin_out, s)
                           : launch_md_kernel(md_kernel<false>, smem, P, n_steps, dt, c_tau, seg, kin_out, s);
}

}  // namespace regc
