// walker.cuh -- the grand-canonical Monte Carlo walk of one replica (sm_103a).
//
// K warps (K = 1, 2 or 4) own one walker (replica configuration) for a whole
// launch:
//   1. its positions are staged from HBM into shared memory by a bulk TMA
//      copy (cp.async.bulk, completion on an mbarrier with a bounded wait);
//   2. the Philox blocks of 32 moves are drawn at a time, one move per lane,
//      and reduced to what does not depend on the configuration: the kind of
//      move, its displacement or insertion point, ln u of its acceptance;
//   3. one warp evaluates one move against the current configuration: the
//      truncated-LJ energy change of the moved particle against the other
//      mobile particles and the frozen surface atoms listed for its column,
//      each pair term added in exact fixed point and reduced with redux.sync.
//      The mobile partners come from one of two enumerations (below);
//   4. the committing warp decides and applies the move.  With K > 1 the warps
//      evaluate K moves of the walker's sequence at once and the first warp
//      commits them in order: move m0 + j keeps its evaluated energy change if
//      no earlier move of the round that was accepted changed anything it
//      depends on (N, for a move that picks a particle by index; any position
//      within rc of its query points); otherwise the round stops there and the
//      move is evaluated again.  Fixed-point sums do not depend on the order of
//      the pairs, so a kept energy change is bit-identical to the one a
//      strictly sequential evaluation would compute, and the chain is exactly
//      the sequential Markov chain.  The acceptance test ln u < ln alpha is
//      decided in binary32 when the two sides differ by more than 1e-3, and in
//      FP64 otherwise, which gives the FP64 decision in every case;
//   5. after each sweep the walker is observed into its state's histograms;
//   6. positions, N and the running energy go back to HBM.
//
// What bounds it: a walker's moves form one dependent chain, so the time of a
// launch is the latency of a move times the moves.  Everything below serves
// that latency: all lanes hold the walk's state and decide together (no result
// goes through shared memory with one warp per walker), the surface column is
// requested before the mobile partners are evaluated, and the parameters used
// in the loop are held in registers.  A move took 645 warp instructions at 5.3
// cycles each on the 1024-replica fcc(111) grid with a committing thread fed
// through shared memory and the draws made one move at a time; it took 572 at
// 4.9 (ncu: 1.9 of them waiting for a fixed latency, 1.0 for shared memory or a
// shuffle, 0.4 for a branch, 0.3 for the instruction fetch) without them, and
// 513 at 4.8 with the geometry compiled in (make_hot) and cells out of reach
// left out (stencil_list).  Steps of ten sweeps, before / after all of it: 16
// fcc(100) replicas 406 / 184 us with the walkers read back, a hundred REGC steps
// of 160 A18 replicas 2.2 / 0.85 ms, 4096 clusters 950 / 456 us, the 1024-replica
// grid 400 / 322 us.  With delayed acceptance the code of the features stands
// once instead of six times and the kernel is no longer bound by the instruction
// fetch: 1930 / 760 us.
#pragma once

#include "cells.cuh"
#include "launch.h"
#include "surrogate.cuh"

namespace regc {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr long long kWaitCycles = 2000000000LL;  // ~1 s at 2 GHz
constexpr double kLn2m32 = -22.18070977791825;   // ln 2^-32
constexpr int kRing = 64;                         // drawn moves kept ahead

// One drawn move: two 16-byte words of the ring.
struct Draw {
    float x, y, z;    // displacement (0 for a removal), or the insertion point
    unsigned kind;    // bits 0-1 the type (0 displacement, 1 insertion, 2 removal), bit 2 the second species
    unsigned b0;      // Philox word picking the particle
    unsigned b1;      // Philox word of the acceptance
    float lu;         // its ln u in binary32
    unsigned b3;      // Philox word of the surrogate stage
};
static_assert(sizeof(Draw) == 32, "two 16-byte words");

// The evaluation of one trial move.
struct Trial {
    float qx, qy, qz;   // new position (removal: the old one)
    int type;           // 0 displacement, 1 insertion, 2 removal
    float ox, oy, oz;   // old position of a displacement or removal
    float ow;           // its cell and slot (cells enumeration)
    int status;         // 0 evaluated, 1 at the N boundary, 2 displacement left the region
    int idx;            // particle picked (insertion: unused)
    int n_eval;         // N the move was evaluated with
    int c_new;          // cell of the new position (displacement, insertion)
    int big, hi, lo;    // fixed-point energy change
    int ovl;            // the new position overlaps a particle
    int pairs;          // pairs within rc
    int dec;            // decision with N = n_eval: 0 reject, 1 accept, 2 near tie (FP64 needed)
    int stage1;         // delayed acceptance: 1 if the surrogate stage accepted
    float dE_sur;       // delayed acceptance: surrogate energy change
    int gy;             // two mobile species: 0 if the moved (inserted, removed) particle is
                        // of the first (index < split), 1 of the second
    unsigned b1, b3;
    float lu;
};
static_assert(sizeof(Trial) == 96, "six 16-byte words");

// Constants of the walker's state for the binary32 pre-test of the acceptance.
struct StateF {
    float beta, c_ins, c_del;
    float c_ins2, c_del2;   // a second grand-canonical species
};

// The parameters of the move loop, copied to registers once per launch (in a
// batch the parameter block lives in shared memory).
struct Hot {
    Geometry g;
    CellGrid cg;
    SurfaceTab st;
    PairTab gg, gA, gAB, ts, tsA;   // ts, tsA: the surface tables where the surface has one type
    float max_disp;
    int nmax, mps;
    bool sheared;                   // false: x is Cartesian as it stands
    float inv_rc;                   // 1 / rc
    float wx, wy, wz, reach2;       // cell widths; squared distance beyond which a cell holds no partner
};

// GEO (sweep_geo): 0 any geometry; 1 a rectangular cell and 2 a sheared one over
// a surface of one type, walls along z; 3 a fully periodic box without a surface.
// What the general form needs beside it is then known at compile time and drops
// out.  A launch of ten sweeps, general form / this (with the cells out of reach
// left out too, stencil_list): 1024 fcc(111) replicas 332 / 285 us (form 1), 1024
// of two gases 308 / 271 (1), 160 A18 132 / 108 (2), 4096 clusters 508 / 416 (3).
template <int GEO>
__device__ __forceinline__ Hot make_hot(const SweepParams& P) {
    Hot H;
    H.g = P.g;
    H.cg = P.cg;
    H.st = P.st;
    H.gg = P.gg;
    H.gA = P.gA;
    H.gAB = P.gAB;
    H.ts = P.gs[P.st.one_type & 3];
    H.tsA = P.gsA[P.st.one_type & 3];
    H.max_disp = P.max_disp;
    H.nmax = P.nmax;
    H.mps = P.mps;
    H.sheared = GEO == 0 || GEO == 2;
    if (GEO == 1 || GEO == 2) {
        H.g.periodic_z = 0;
        H.st.one_type = 0;
        H.st.n_all = 1;
    }
    if (GEO == 3) {
        H.g.periodic_z = 1;
        H.st.n_all = 0;
    }
    H.inv_rc = 1.0f / H.g.rc;
    H.wx = 1.0f / H.cg.icx;
    H.wy = 1.0f / H.cg.icy;
    H.wz = 1.0f / H.cg.icz;
    // well beyond the rounding of a coordinate, a cell index or a width
    const float zs = H.g.periodic_z ? H.g.Lz : fabsf(H.g.z_lo) + fabsf(H.g.z_hi);
    const float reach = H.g.rc * 1.001f + 2e-6f * (H.g.Lx + H.g.Ly + zs);
    H.reach2 = reach * reach;
    return H;
}

// Cartesian x component of a displacement in the cell frame.
__device__ __forceinline__ float cart(const Hot& H, float du, float dv) {
    return H.sheared ? cart_dx(H.g, du, dv) : du;
}

// Pair tables of the moving particle's species against a partner of the first
// species (tA: index < split) and of the second (tB); mA: the moving particle
// is of the first.
struct MoveTabs {
    PairTab tA, tB;
    bool mA;
};

// Binary32 pair energy without branches: 0 unless `use` and r < rc.  An
// in-range term is computed with the same operations as pair_phi, hence is
// bit-identical to it; the branch-free form lets the candidate loop be one
// basic block, so independent loads and arithmetic overlap.
__device__ __forceinline__ float pair_phi_sel(float dx, float dy, float dz, float rc2, const PairTab& t, bool use,
                                              int& n_in, bool& overlap) {
    const float r2 = r2_of(dx, dy, dz);
    const bool in = use && r2 < rc2;
    const float s2 = __fdividef(t.sig2, r2);   // (what r2 out of range, or 0, makes of it is dropped)
    const float s6 = __fmul_rn(__fmul_rn(s2, s2), s2);
    const float phi = __fmul_rn(t.eps4, __fmaf_rn(s6, s6, -s6));
    n_in += in;
    overlap = overlap || (in && (r2 < t.rhc2));
    return in ? phi : 0.0f;
}

// Binary32 pre-test of ln u < ln alpha: c_f the constants and ln N terms, de_f
// the energy change.  0 reject, 1 accept, 2 the two sides are within 1e-3 and
// FP64 must decide.
__device__ __forceinline__ int pretest(float c_f, float beta, float de_f, float lu_f) {
    const float la_f = c_f - beta * de_f;
    if (la_f >= 0.f || lu_f < la_f - 1e-3f) return 1;
    if (lu_f > la_f + 1e-3f) return 0;
    return 2;
}

__device__ __forceinline__ float fix_to_f32(int big, int hi, int lo) {
    return __fmaf_rn((float)lo, 9.313225746154785e-10f, __fmaf_rn((float)hi, 0.00390625f, (float)big * 8192.0f));
}

// ln of the count factor of a grand-canonical move, in binary32, with its constant.
__device__ __forceinline__ float count_term(int type, int gcnt, float c_ins, float c_del) {
    if (type == 1) return c_ins - __logf((float)(gcnt + 1));
    if (type == 2) return c_del + __logf((float)gcnt);
    return 0.f;
}

// Round state broadcast by the committing warp (K > 1).
struct RoundHdr {
    int N;
    int committed;
    long long E;
    int split;   // two mobile species: the current boundary
    int pad;
};

struct WalkerSmem {
    float4* pos;        // [nmax]  x, y, z, (cell << 16 | slot) as bits (cells enumeration)
    uint64_t* bar;      // mbarrier of the position copy
    uint4* ring;        // [kRing][2] drawn moves
    RoundHdr* hdr;      // K > 1
    Trial* res;         // [K], K > 1
    float4* stencil;    // [K][32] the non-empty stencil cells (cells enumeration)
    uint16_t* cnt;      // [ncell] particles per cell
    uint16_t* slots;    // [ncell][cap] particle indices (cells enumeration)
};

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~size_t(15); }

// Bytes of the walker's region; direct: the enumeration over all particles
// (counts per cell are kept only where a cell can be over capacity).
__host__ __device__ inline size_t smem_bytes(int nmax, int ncell, int cap, int K, bool direct) {
    size_t b = align16(size_t(nmax) * 16) + 16 + size_t(kRing) * sizeof(Draw);
    if (K > 1) b += align16(sizeof(RoundHdr)) + size_t(K) * sizeof(Trial);
    if (direct) return b + (cap < nmax ? align16(size_t(ncell) * 2) : 0);
    return b + size_t(K) * 32 * sizeof(float4) + align16(size_t(ncell) * 2) + align16(size_t(ncell) * cap * 2);
}

template <int K, bool DIRECT>
__device__ inline WalkerSmem carve(char* base, const SweepParams& P) {
    WalkerSmem w;
    size_t off = 0;
    w.pos = reinterpret_cast<float4*>(base + off);
    off += align16(size_t(P.nmax) * 16);
    w.bar = reinterpret_cast<uint64_t*>(base + off);
    off += 16;
    w.ring = reinterpret_cast<uint4*>(base + off);
    off += size_t(kRing) * sizeof(Draw);
    w.hdr = nullptr;
    w.res = nullptr;
    if (K > 1) {
        w.hdr = reinterpret_cast<RoundHdr*>(base + off);
        off += align16(sizeof(RoundHdr));
        w.res = reinterpret_cast<Trial*>(base + off);
        off += size_t(K) * sizeof(Trial);
    }
    w.stencil = nullptr;
    w.slots = nullptr;
    if (!DIRECT) {
        w.stencil = reinterpret_cast<float4*>(base + off);
        off += size_t(K) * 32 * sizeof(float4);
    }
    w.cnt = reinterpret_cast<uint16_t*>(base + off);
    if (!DIRECT) {
        off += align16(size_t(P.cg.ncell) * 2);
        w.slots = reinterpret_cast<uint16_t*>(base + off);
    }
    return w;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------- bulk copy + mbarrier

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t phase) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}

// Wait for phase 0 of bar with a cycle budget.  Returns false on timeout.
__device__ bool mbar_wait_bounded(uint64_t* bar) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, 0)) {
        if (clock64() - t0 > kWaitCycles) return false;
    }
    return true;
}

// Synchronise the K warps of a walker group: a warp barrier for one warp,
// else named barrier bar over the group's 32 K threads (bar 0 with the whole
// CTA in the one-walker-per-CTA kernel, where it is __syncthreads()).
template <int K>
__device__ __forceinline__ void group_sync(int bar) {
    if (K == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(32 * K) : "memory");
}

// True in every thread of the group iff p holds in all of them (a barrier).
template <int K>
__device__ __forceinline__ bool group_all(int bar, bool p) {
    if (K == 1) return __all_sync(0xffffffffu, p) != 0;
    unsigned r;
    asm volatile(
        "{\n\t.reg .pred q, a;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.and.pred a, %2, %3, q;\n\t"
        "selp.u32 %0, 1, 0, a;\n\t}"
        : "=r"(r)
        : "r"((unsigned)p), "r"(bar), "r"(32 * K)
        : "memory");
    return r != 0;
}

// ------------------------------------------------------------------ drawing

// Draw moves first .. first + 31 of the launch (move m: sweep m / mps, move
// m % mps), one per lane.
template <bool CL>
__device__ __forceinline__ void draw_moves(const SweepParams& P, const Hot& H, uint4* ring, int w, int first,
                                           int total, int lane) {
    const int m = first + lane;
    if (m >= total) return;
    const int ts = m / H.mps, k = m - ts * H.mps;
    const U4 A = philox((uint32_t)k, P.t0 + (uint32_t)ts, (uint32_t)w, 0u, P.key0, P.key1);
    const U4 B = philox((uint32_t)k, P.t0 + (uint32_t)ts, (uint32_t)w, 1u, P.key0, P.key1);
    // the kind of move: drawn from A0 in a sweep, fixed by its place in a REGC
    // cycle step (move 0: the particle exchange, the others displacements)
    const unsigned gc_type = (B.z >> 31) == 0u ? 2u : 1u;
    const bool disp = P.cycle ? k != 0 : (unsigned long long)A.x < P.th_disp;
    const unsigned type = disp ? 0u : gc_type;
    Draw d;
    if (disp) {
        d.x = __fmul_rn(H.max_disp, __fsub_rn(__fmul_rn(2.0f, u24(A.y)), 1.0f));
        d.y = __fmul_rn(H.max_disp, __fsub_rn(__fmul_rn(2.0f, u24(A.z)), 1.0f));
        d.z = __fmul_rn(H.max_disp, __fsub_rn(__fmul_rn(2.0f, u24(A.w)), 1.0f));
    } else {
        d.x = __fmul_rn(H.g.Lx, u24(A.y));
        d.y = __fmul_rn(H.g.Ly, u24(A.z));
        d.z = __fadd_rn(H.g.z_lo, __fmul_rn(H.g.height, u24(A.w)));
        if (d.x >= H.g.Lx) d.x = __fsub_rn(d.x, H.g.Lx);
        if (d.y >= H.g.Ly) d.y = __fsub_rn(d.y, H.g.Ly);
        if (H.g.periodic_z && d.z >= H.g.Lz) d.z = __fsub_rn(d.z, H.g.Lz);
        if (type == 2u) d.x = d.y = d.z = 0.f;
    }
    // the species of a grand-canonical move: the second (the gas after a
    // cluster), or with two grand-canonical species the one bit 30 of B2 picks
    const unsigned gy = (CL && P.gc2) ? (B.z >> 30) & 1u : 1u;
    d.kind = type | (gy << 2);
    d.lu = __logf(((float)B.y + 0.5f) * 2.3283064365386963e-10f);
    uint4* out = ring + 2 * ((unsigned)m % kRing);
    out[0] = make_uint4(__float_as_uint(d.x), __float_as_uint(d.y), __float_as_uint(d.z), d.kind);
    out[1] = make_uint4(B.x, B.y, __float_as_uint(d.lu), B.w);
}

// ------------------------------------------------------- mobile partners
//
// Two enumerations of the partners of a query point:
// * cells: the particles of the query's 27-cell stencil, through the walker's
//   cell list.  Periodic axes always contribute three images (-1, 0, +1); with
//   fewer than three cells along an axis the same cell appears with different
//   shifts, which evaluates every periodic image of its particles (at most one
//   of them can be within rc, because every period is at least 2 rc);
// * direct: every particle with its nearest image.  No cell list is read or
//   kept up, so a move costs one batch of 32 distances per 32 particles and
//   little else, and a walker's shared memory falls from 20-30 KB to 3-5 KB.
// Both compute a displacement rounded once from the same exact operands, so an
// in-range pair term is the same bit for bit.

// This lane's place in the 3 x 3 x 3 stencil, and what wrapping its coordinate
// around the grid adds to it: to the cell, and as the entry's shift.
struct LaneCell {
    int x, y, z;
    bool in;
    int wx, wy, wz;
    float sx, sy, sz;
    float ax, ay, az, bx, by, bz;   // the gap to that cell from a point f beyond its own's lower corner: |b - a f| per axis
};

__device__ __forceinline__ LaneCell lane_cell(const Hot& H, int lane) {
    LaneCell l;
    l.x = lane % 3 - 1;
    l.y = (lane / 3) % 3 - 1;
    l.z = lane / 9 - 1;
    l.in = lane < 27;
    l.wx = l.x < 0 ? H.cg.ncx : -H.cg.ncx;
    l.wy = l.y < 0 ? H.cg.ncy : -H.cg.ncy;
    l.wz = l.z < 0 ? H.cg.ncz : -H.cg.ncz;
    l.sx = l.x < 0 ? -H.g.Lx : H.g.Lx;
    l.sy = l.y < 0 ? -H.g.Ly : H.g.Ly;
    l.sz = l.z < 0 ? -H.g.Lz : H.g.Lz;
    // (in a sheared cell the gap along x is not a Cartesian distance: left out)
    const bool x_gap = !H.sheared || H.g.shear == 0.f;
    l.ax = x_gap ? fabsf((float)l.x) : 0.f;
    l.bx = x_gap && l.x > 0 ? H.wx : 0.f;
    l.ay = fabsf((float)l.y);
    l.by = l.y > 0 ? H.wy : 0.f;
    l.az = fabsf((float)l.z);
    l.bz = l.z > 0 ? H.wz : 0.f;
    return l;
}

// The stencil of cell c as a list of its non-empty cells in st: {slot base,
// shift x, y, z}; the candidate list is the concatenation of their slots, and
// slot base + j is the slot of its j-th candidate while j stays in the entry.
// A shift s > 0 is taken off the query, s < 0 off the partner (every shifted
// operand is exact, Sterbenz, so a displacement is rounded once).  Returns the
// candidates; cnt and excl are this lane's own cell's.  NQ queries (0: every
// cell is listed): a cell beyond reach of all of them is left out -- a third of
// the candidates where cells are little wider than rc.
template <int NQ>
__device__ __forceinline__ int stencil_list(const Hot& H, const uint16_t* cnts, Cell3 c, LaneCell lc, int lane,
                                            float4* st, int& cnt, int& excl, float q0x, float q0y, float q0z,
                                            float q1x, float q1y, float q1z) {
    int ix = c.x + lc.x, iy = c.y + lc.y, iz = c.z + lc.z;
    const bool wx = (unsigned)ix >= (unsigned)H.cg.ncx, wy = (unsigned)iy >= (unsigned)H.cg.ncy;
    const bool wz = (unsigned)iz >= (unsigned)H.cg.ncz;
    ix = wx ? ix + lc.wx : ix;
    iy = wy ? iy + lc.wy : iy;
    const float sx = wx ? lc.sx : 0.f, sy = wy ? lc.sy : 0.f;
    float sz = 0.f;
    bool in = lc.in;
    if (H.g.periodic_z) {
        iz = wz ? iz + lc.wz : iz;
        sz = wz ? lc.sz : 0.f;
    } else {
        in = in && !wz;
    }
    if (NQ > 0) {
        const float x0 = (float)c.x * H.wx, y0 = (float)c.y * H.wy;
        const float z0 = fmaf((float)c.z, H.wz, H.g.periodic_z ? 0.f : H.g.z_lo);
        auto gap2 = [&](float x, float y, float z) {
            const float gx = fmaf(lc.ax, x0 - x, lc.bx), gy = fmaf(lc.ay, y0 - y, lc.by), gz = fmaf(lc.az, z0 - z, lc.bz);
            return fmaf(gx, gx, fmaf(gy, gy, gz * gz));
        };
        float d2 = gap2(q0x, q0y, q0z);
        if (NQ == 2) d2 = fminf(d2, gap2(q1x, q1y, q1z));
        in = in && d2 < H.reach2;
    }
    const int cell = (iz * H.cg.ncy + iy) * H.cg.ncx + ix;
    cnt = in ? (int)cnts[cell] : 0;
    const int total = (int)__reduce_add_sync(FULL, (unsigned)cnt);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)   // inclusive scan; the shuffle's predicate says which lanes have a source
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
            "shfl.sync.up.b32 t|p, %0, %1, 0, 0xffffffff;\n\t"
            "@p add.s32 %0, %0, t;\n\t}"
            : "+r"(incl)
            : "r"(o));
    excl = incl - cnt;
    const unsigned nonempty = __ballot_sync(FULL, cnt > 0);
    if (cnt > 0)
        st[__popc(nonempty & lanemask_lt(lane))] =
            make_float4(__int_as_float(cell * H.cg.cap - excl), sx, sy, sz);
    __syncwarp();
    return total;
}

// The stencil entry of candidate base + lane: `started` entries began in
// earlier batches; starts is the mask of those that begin in this one.  Every
// lane finds a valid entry (some entry starts at or below it).
__device__ __forceinline__ unsigned batch_starts(int cnt, int excl, int base) {
    const int at = excl - base;
    const unsigned bit = (cnt > 0 && at >= 0 && at < 32) ? (1u << at) : 0u;
    return __reduce_or_sync(FULL, bit);
}

// Fixed-point sum of the pair energies of NQ queries (sharing the stencil of
// cell c) with the stencil's particles except `skip`: query 0 minus query 1.
template <int NQ, bool CL>
__device__ __forceinline__ void mobile_cells(const Hot& H, const WalkerSmem& S, Cell3 c, LaneCell lc, float q0x,
                                             float q0y, float q0z, float q1x, float q1y, float q1z, int skip,
                                             Fix3& acc, int& n_in, int& n_cand, bool& overlap, int lane, int warp,
                                             int split, const MoveTabs& mt) {
    float4* st = S.stencil + warp * 32;
    int cnt, excl;
    const int total = stencil_list<NQ>(H, S.cnt, c, lc, lane, st, cnt, excl, q0x, q0y, q0z, q1x, q1y, q1z);
    bool ov = false, ov1 = false;
    int started = 0;
#pragma unroll 2   // two batches' independent chains may overlap
    for (int base = 0; base < total; base += 32) {
        const unsigned starts = batch_starts(cnt, excl, base);
        const int j = base + lane;
        const bool act = j < total;
        const float4 e = st[started + __popc(starts & lanemask_le(lane)) - 1];
        int pj = -1;
        if (act) pj = S.slots[__float_as_int(e.x) + j];
        const bool use = act && pj != skip;
        // lanes without a partner read particle 0 and discard the term
        const float4 p = S.pos[use ? pj : 0];
        const float bx = __fsub_rn(p.x, fmaxf(-e.y, 0.f)), by = __fsub_rn(p.y, fmaxf(-e.z, 0.f));
        const float ax = fmaxf(e.y, 0.f), ay = fmaxf(e.z, 0.f);
        const float bz = H.g.periodic_z ? __fsub_rn(p.z, fmaxf(-e.w, 0.f)) : p.z;
        const float az0 = H.g.periodic_z ? __fsub_rn(q0z, fmaxf(e.w, 0.f)) : q0z;
        n_cand += use ? NQ : 0;
        const PairTab& tp = CL ? (pj < split ? mt.tA : mt.tB) : H.gg;
        const float dy0 = __fsub_rn(__fsub_rn(q0y, ay), by);
        const float phi0 = pair_phi_sel(cart(H, __fsub_rn(__fsub_rn(q0x, ax), bx), dy0), dy0,
                                        __fsub_rn(az0, bz), H.g.rc2, tp, use, n_in, ov);
        fix_add(acc, phi0, 1);
        if (NQ == 2) {
            const float az1 = H.g.periodic_z ? __fsub_rn(q1z, fmaxf(e.w, 0.f)) : q1z;
            const float dy1 = __fsub_rn(__fsub_rn(q1y, ay), by);
            const float phi1 = pair_phi_sel(cart(H, __fsub_rn(__fsub_rn(q1x, ax), bx), dy1), dy1,
                                            __fsub_rn(az1, bz), H.g.rc2, tp, use, n_in, ov1);
            fix_add(acc, phi1, -1);
        }
        started += __popc(starts);
    }
    overlap = overlap || ov;
    __syncwarp();
}

// Displacement q - p with the nearest image along a period L: where |q - p|
// is half a period or more the operand in the upper half is shifted by -L
// (exact), so the result is rounded once.  An image left out by the comparison
// is at least half a period (>= rc) away along the axis, so the in-range terms
// are those of the stencil's images.
__device__ __forceinline__ float near_diff(float q, float p, float L, float hL) {
    const float e = __fsub_rn(q, p);
    const float qs = e >= hL ? __fsub_rn(q, L) : q;
    const float ps = e <= -hL ? __fsub_rn(p, L) : p;
    return __fsub_rn(qs, ps);
}

// The same sum over all N particles.
template <int NQ, bool CL>
__device__ __forceinline__ void mobile_direct(const Hot& H, const WalkerSmem& S, int N, float q0x, float q0y,
                                              float q0z, float q1x, float q1y, float q1z, int skip, Fix3& acc,
                                              int& n_in, int& n_cand, bool& overlap, int lane, int split,
                                              const MoveTabs& mt) {
    bool ov = false, ov1 = false;
#pragma unroll 2
    for (int j = lane; j - lane < N; j += 32) {
        const bool use = j < N && j != skip;
        const float4 p = S.pos[use ? j : 0];
        n_cand += use ? NQ : 0;
        const PairTab& tp = CL ? (j < split ? mt.tA : mt.tB) : H.gg;
        const float dy0 = near_diff(q0y, p.y, H.g.Ly, H.g.hLy);
        const float dz0 = H.g.periodic_z ? near_diff(q0z, p.z, H.g.Lz, H.g.hLz) : __fsub_rn(q0z, p.z);
        const float phi0 = pair_phi_sel(cart(H, near_diff(q0x, p.x, H.g.Lx, H.g.hLx), dy0), dy0, dz0, H.g.rc2,
                                        tp, use, n_in, ov);
        fix_add(acc, phi0, 1);
        if (NQ == 2) {
            const float dy1 = near_diff(q1y, p.y, H.g.Ly, H.g.hLy);
            const float dz1 = H.g.periodic_z ? near_diff(q1z, p.z, H.g.Lz, H.g.hLz) : __fsub_rn(q1z, p.z);
            const float phi1 = pair_phi_sel(cart(H, near_diff(q1x, p.x, H.g.Lx, H.g.hLx), dy1), dy1, dz1,
                                            H.g.rc2, tp, use, n_in, ov1);
            fix_add(acc, phi1, -1);
        }
    }
    overlap = overlap || ov;
}

// ----------------------------------------------------------- the surface

// Squared distance of a query from one listed image of a frozen atom and its
// pair table.  Each listed image holds its coordinate already shifted by minus
// the period where that is exact; flag bits ask for the query to be shifted by
// minus the period instead.
template <bool CL>
__device__ __forceinline__ PairTab surface_tab(const SweepParams& P, const Hot& H, unsigned bits, bool mA) {
    if (H.st.one_type >= 0) return (CL && mA) ? H.tsA : H.ts;
    return (CL && mA) ? P.gsA[bits & 3u] : P.gs[bits & 3u];
}

__device__ __forceinline__ void surface_diff(const Hot& H, float4 a, float qx, float qy, float qz, float& dx,
                                             float& dy, float& dz) {
    const unsigned bits = __float_as_uint(a.w);
    const float sx = (bits & 4u) ? H.g.Lx : 0.f, sy = (bits & 8u) ? H.g.Ly : 0.f;
    dy = __fsub_rn(__fsub_rn(qy, sy), a.y);
    dx = cart(H, __fsub_rn(__fsub_rn(qx, sx), a.x), dy);
    dz = __fsub_rn(H.g.periodic_z ? __fsub_rn(qz, (bits & 16u) ? H.g.Lz : 0.f) : qz, a.z);
}

template <bool CL>
__device__ __forceinline__ float surface_phi(const SweepParams& P, const Hot& H, float4 a, float qx, float qy,
                                             float qz, bool mA, int& n_in, int& n_cand, bool& overlap) {
    float dx, dy, dz;
    surface_diff(H, a, qx, qy, qz, dx, dy, dz);
    const unsigned bits = __float_as_uint(a.w);
    n_cand += (bits & 32u) ? 0 : 1;   // padding slots are not candidates
    return pair_phi_sel(dx, dy, dz, H.g.rc2, surface_tab<CL>(P, H, bits, mA), true, n_in, overlap);
}

__device__ __forceinline__ bool near_surf(const Hot& H, float z) {
    return H.st.n_all > 0 && (H.g.periodic_z || z < H.st.z_reach);
}

__device__ __forceinline__ int surf_slot(const Hot& H, float x, float y) {
    const int sx = min(H.st.nsx - 1, (int)(x * H.st.isx));
    const int sy = min(H.st.nsy - 1, (int)(y * H.st.isy));
    return (sy * H.st.nsx + sx) * H.st.stride;
}

__device__ __forceinline__ Cell3 cell3_hot(const Hot& H, float x, float y, float z) {
    Cell3 c;
    c.x = min(H.cg.ncx - 1, (int)(x * H.cg.icx));
    c.y = min(H.cg.ncy - 1, (int)(y * H.cg.icy));
    const float zz = H.g.periodic_z ? z : (z - H.g.z_lo);
    c.z = min(H.cg.ncz - 1, max(0, (int)(zz * H.cg.icz)));
    return c;
}

__device__ __forceinline__ int cell_lin(const Hot& H, Cell3 c) { return (c.z * H.cg.ncy + c.y) * H.cg.ncx + c.x; }

// ------------------------------------------------- the surrogate's features

// Surrogate features of one query from the mobile particles of its stencil
// except `skip` and from its surface column, accumulated per lane (candidates
// in list order, so the sums do not depend on which query is evaluated when).
template <bool CL>
__device__ __forceinline__ void query_features(const SweepParams& P, const Hot& H, const WalkerSmem& S, LaneCell lc,
                                               float qx, float qy, float qz, int skip, float (&F)[kNF], int lane,
                                               int warp, int split, const MoveTabs& mt) {
    float4* st = S.stencil + warp * 32;
    int cnt, excl;
    const int total = stencil_list<0>(H, S.cnt, cell3_hot(H, qx, qy, qz), lc, lane, st, cnt, excl, 0.f, 0.f, 0.f, 0.f,
                                      0.f, 0.f);
    const int n_mob = (total + 31) & ~31;
    const bool surf = near_surf(H, qz);
    const int n_all = n_mob + (surf ? H.st.stride : 0);
    const int slot0 = surf ? surf_slot(H, qx, qy) : 0;
    int started = 0;
    // the mobile batches, then the batches of the surface column: one loop, so
    // that the code of the Gaussians stands once in the kernel
#pragma unroll 1
    for (int base = 0; base < n_all; base += 32) {
        float r2 = INFINITY, wgt = 0.f;
        if (base < n_mob) {
            const unsigned starts = batch_starts(cnt, excl, base);
            const int j = base + lane;
            if (j < total) {
                const float4 e = st[started + __popc(starts & lanemask_le(lane)) - 1];
                const int pj = S.slots[__float_as_int(e.x) + j];
                if (pj != skip) {
                    const float4 p = S.pos[pj];
                    const float dy = __fsub_rn(__fsub_rn(qy, fmaxf(e.z, 0.f)), __fsub_rn(p.y, fmaxf(-e.z, 0.f)));
                    const float du = __fsub_rn(__fsub_rn(qx, fmaxf(e.y, 0.f)), __fsub_rn(p.x, fmaxf(-e.y, 0.f)));
                    const float dz = __fsub_rn(__fsub_rn(qz, fmaxf(e.w, 0.f)), __fsub_rn(p.z, fmaxf(-e.w, 0.f)));
                    r2 = r2_of(cart(H, du, dy), dy, dz);
                    wgt = CL ? (pj < split ? mt.tA.eps : mt.tB.eps) : H.gg.eps;
                }
            }
            started += __popc(starts);
        } else {
            const float4 a = __ldg(&H.st.atoms[slot0 + base - n_mob + lane]);
            float dx, dy, dz;
            surface_diff(H, a, qx, qy, qz, dx, dy, dz);
            r2 = r2_of(dx, dy, dz);
            wgt = surface_tab<CL>(P, H, __float_as_uint(a.w), mt.mA).eps;
        }
        if (r2 < H.g.rc2) add_features(F, r2, wgt, H.g.rc, H.inv_rc);
    }
    __syncwarp();
}

// ------------------------------------------------------------- evaluation

// Evaluate the drawn move m with one warp against the current configuration
// with N particles; every lane returns the same Trial.  s: the walker's state.
template <bool DA, bool CL, bool DIRECT>
__device__ __forceinline__ Trial evaluate_move(const SweepParams& P, const Hot& H, const WalkerSmem& S,
                                               const StateF& sf, int s, int m, int N, int split_in, int& n_cand,
                                               LaneCell lc, int lane, int warp, const NetFrag* nf) {
    // Two mobile species (CL): particles [0, split) are of the first, the
    // rest of the second -- a cluster (split = n_cluster, moved only by
    // displacement; insertion and removal act on the gas after it) or two
    // grand-canonical species B and C (split = N_B, gc2).
    const int split = CL ? split_in : 0;
    const uint4 d0 = S.ring[2 * ((unsigned)m % kRing)], d1 = S.ring[2 * ((unsigned)m % kRing) + 1];
    Trial r;
    const int type = (int)(d0.w & 3u);
    const int gy = CL ? (int)((d0.w >> 2) & 1u) : 1;
    const int gcnt = gy ? N - split : split;          // the species' count before the move
    const bool use2 = CL && P.gc2 && gy == 1;         // species C's constants
    const float cins_f = use2 ? sf.c_ins2 : sf.c_ins, cdel_f = use2 ? sf.c_del2 : sf.c_del;
    r.b1 = d1.y;
    r.lu = __uint_as_float(d1.z);
    r.b3 = d1.w;
    // One path for the three kinds, without branches: the new position is the
    // particle's (an insertion: 0) plus the drawn numbers; what a kind does not
    // need is read from particle 0 and dropped.
    const bool disp = type == 0, ins = type == 1;
    // the particle: any of N for a displacement, of the species for a removal
    const int pick_n = disp ? N : gcnt, pick_0 = (type == 2 && gy) ? split : 0;
    int status = (ins ? N == H.nmax : pick_n == 0) ? 1 : 0;
    const int idx = (ins || status) ? -1 : pick_0 + (int)__umulhi(d1.x, (unsigned)pick_n);
    float4 old = S.pos[max(idx, 0)];
    if (ins) old = make_float4(0.f, 0.f, 0.f, 0.f);
    // ln of the count factor with its constant, ready for the decision
    const float lg = __logf((float)(gcnt + (ins ? 1 : 0)));
    const float c_gc = disp ? 0.f : (ins ? cins_f - lg : cdel_f + lg);
    float qx = __fadd_rn(old.x, __uint_as_float(d0.x));
    float qy = __fadd_rn(old.y, __uint_as_float(d0.y));
    float qz = __fadd_rn(old.z, __uint_as_float(d0.z));
    // (an insertion's point and a removed particle's are inside already)
    qx = qx < 0.f ? __fadd_rn(qx, H.g.Lx) : qx;
    qx = qx >= H.g.Lx ? __fsub_rn(qx, H.g.Lx) : qx;
    qy = qy < 0.f ? __fadd_rn(qy, H.g.Ly) : qy;
    qy = qy >= H.g.Ly ? __fsub_rn(qy, H.g.Ly) : qy;
    if (H.g.periodic_z) {
        qz = qz < 0.f ? __fadd_rn(qz, H.g.Lz) : qz;
        qz = qz >= H.g.Lz ? __fsub_rn(qz, H.g.Lz) : qz;
    } else if (disp && status == 0 && (qz < H.g.z_lo || qz > H.g.z_hi)) {
        status = 2;
    }
    const bool two_q = type == 0;
    // pair tables of the moving species
    MoveTabs mt;
    mt.mA = CL && ((type != 1 && idx >= 0 && idx < split) || (type == 1 && gy == 0));
    if (CL) {
        mt.tA = mt.mA ? H.gA : H.gAB;
        mt.tB = mt.mA ? H.gAB : H.gg;
    }
    const int skip = idx;

    // delayed acceptance, stage 1: the surrogate energy change dE~
    int stage1 = 1;
    float dEs = 0.f;
    if (DA && status == 0) {
        float rq[2] = {0.f, 0.f};
#pragma unroll 1   // one copy of the feature code for both queries
        for (int q = 0; q < (two_q ? 2 : 1); ++q) {
            float F[kNF];
#pragma unroll
            for (int k = 0; k < kNF; ++k) F[k] = 0.f;
            query_features<CL>(P, H, S, lc, q ? old.x : qx, q ? old.y : qy, q ? old.z : qz, skip, F, lane, warp, split,
                               mt);
            const float v = warp_reduce16(F, lane);
            if (q) rq[1] = v;
            else rq[0] = v;
        }
        // both positions through the network at once: rows 0 and 1 of the tiles
        uint32_t a[4];
        features_to_frag(rq[0], rq[1], lane, a);
        float e1 = 0.f;
        const float e0 = net_mma(*nf, a, &e1);
        dEs = type == 1 ? e0 : (type == 2 ? -e0 : e0 - e1);
        // ln u1 < ln alpha with dE~ in place of dE (u1 from B3)
        const float la1 = c_gc - sf.beta * dEs;
        const float lu1 = __logf(((float)r.b3 + 0.5f) * 2.3283064365386963e-10f);
        if (la1 >= 0.f || lu1 < la1 - 1e-3f) stage1 = 1;
        else if (lu1 > la1 + 1e-3f) stage1 = 0;
        else {
            double c = 0.0;
            if (type == 1) c = (use2 ? P.c_ins2[s] : P.c_ins[s]) - P.ln_tab[gcnt + 1];
            else if (type == 2) c = (use2 ? P.c_del2[s] : P.c_del[s]) + P.ln_tab[gcnt];
            stage1 = (log((double)r.b3 + 0.5) + kLn2m32) < c - P.beta[s] * (double)dEs;
        }
    }

    Fix3 acc{0, 0, 0};
    int n_in = 0;
    bool overlap = false;
    int c_new = 0;
    if (status == 0 && stage1) {
        // the surface columns are requested first: they come from L2 while the
        // mobile partners are evaluated
        const bool s0 = near_surf(H, qz), s1 = two_q && near_surf(H, old.z);
        int col0 = 0, col1 = 0;
        float4 a0, a1;
        if (s0) {
            col0 = surf_slot(H, qx, qy);
            a0 = __ldg(&H.st.atoms[col0 + lane]);
        }
        if (s1) {
            col1 = surf_slot(H, old.x, old.y);
            a1 = __ldg(&H.st.atoms[col1 + lane]);
        }
        if (DIRECT) {
            if (H.cg.cap < H.nmax) c_new = cell_lin(H, cell3_hot(H, qx, qy, qz));
            if (two_q)
                mobile_direct<2, CL>(H, S, N, qx, qy, qz, old.x, old.y, old.z, skip, acc, n_in, n_cand, overlap, lane,
                                     split, mt);
            else
                mobile_direct<1, CL>(H, S, N, qx, qy, qz, qx, qy, qz, skip, acc, n_in, n_cand, overlap, lane, split,
                                     mt);
        } else {
            const Cell3 c0 = cell3_hot(H, qx, qy, qz);
            c_new = cell_lin(H, c0);
            const Cell3 c1 = two_q ? cell3_hot(H, old.x, old.y, old.z) : c0;
            const bool same = c0.x == c1.x && c0.y == c1.y && c0.z == c1.z;
            if (two_q && same) {
                mobile_cells<2, CL>(H, S, c0, lc, qx, qy, qz, old.x, old.y, old.z, skip, acc, n_in, n_cand, overlap,
                                    lane, warp, split, mt);
            } else {
                // one pass per query: query 0, then (a displacement across
                // cells) the old position, whose sum is taken off
#pragma unroll 1
                for (int pass = 0; pass < (two_q ? 2 : 1); ++pass) {
                    const float px = pass ? old.x : qx, py = pass ? old.y : qy, pz = pass ? old.z : qz;
                    bool ovp = false;
                    Fix3 part{0, 0, 0};
                    mobile_cells<1, CL>(H, S, pass ? c1 : c0, lc, px, py, pz, px, py, pz, skip, part, n_in, n_cand,
                                        ovp, lane, warp, split, mt);
                    const int sg = pass ? -1 : 1;
                    acc.big += sg * part.big;
                    acc.hi += sg * part.hi;
                    acc.lo += sg * part.lo;
                    if (pass == 0) overlap = ovp;
                }
            }
        }
        bool ov1 = false;
        if (s0) {
            fix_add(acc, surface_phi<CL>(P, H, a0, qx, qy, qz, mt.mA, n_in, n_cand, overlap), 1);
#pragma unroll 1   // a column longer than a warp
            for (int j = lane + 32; j < H.st.stride; j += 32)
                fix_add(acc, surface_phi<CL>(P, H, __ldg(&H.st.atoms[col0 + j]), qx, qy, qz, mt.mA, n_in, n_cand,
                                             overlap), 1);
        }
        if (s1) {
            fix_add(acc, surface_phi<CL>(P, H, a1, old.x, old.y, old.z, mt.mA, n_in, n_cand, ov1), -1);
#pragma unroll 1
            for (int j = lane + 32; j < H.st.stride; j += 32)
                fix_add(acc, surface_phi<CL>(P, H, __ldg(&H.st.atoms[col1 + j]), old.x, old.y, old.z, mt.mA, n_in,
                                             n_cand, ov1), -1);
        }
    }
    // a removal's sum enters with a minus, and the old position of a particle
    // never overlaps
    const int sg = type == 2 ? -1 : 1;
    const int big = sg * (int)__reduce_add_sync(FULL, (unsigned)acc.big);
    const int hi = sg * (int)__reduce_add_sync(FULL, (unsigned)acc.hi);
    const int lo = sg * (int)__reduce_add_sync(FULL, (unsigned)acc.lo);
    const unsigned both = __reduce_add_sync(FULL, (unsigned)n_in | (overlap ? 1u << 24 : 0u));
    const int ovl = type != 2 && (both >> 24) != 0u;
    r.qx = qx; r.qy = qy; r.qz = qz;
    r.type = type;
    r.ox = old.x; r.oy = old.y; r.oz = old.z; r.ow = old.w;
    r.status = status;
    r.idx = idx;
    r.n_eval = N;
    r.c_new = c_new;
    r.big = big;
    r.hi = hi;
    r.lo = lo;
    r.ovl = ovl;
    r.pairs = (int)(both & 0xffffffu);
    r.stage1 = stage1;
    r.dE_sur = dEs;
    r.gy = gy;
    r.dec = 0;
    if (status == 0 && !ovl) {
        const float de_f = fix_to_f32(big, hi, lo);
        if (!DA) {
            r.dec = pretest(c_gc, sf.beta, de_f, r.lu);
        } else if (stage1) {
            // stage 2: ln u2 < -beta (dE - dE~) (u2 from B1)
            const float la2 = -sf.beta * (de_f - dEs);
            if (la2 >= 0.f || r.lu < la2 - 1e-3f) r.dec = 1;
            else if (r.lu > la2 + 1e-3f) r.dec = 0;
            else
                r.dec = (log((double)r.b1 + 0.5) + kLn2m32) <
                        -P.beta[s] * ((double)fix_value(big, hi, lo) * kFixUnit - (double)dEs);
        }
    }
    return r;
}

// ------------------------------------------------------------------- commit

// floor(d / bin) for 0 <= d < 2^63 from the host's magic = floor((2^64 - 1) /
// bin): the high product is that quotient or one below it.
__device__ __forceinline__ long long floor_div(long long d, long long bin, unsigned long long magic) {
    const long long q = (long long)__umul64hi((unsigned long long)d, magic);
    return (q + 1) * bin <= d ? q + 1 : q;
}

// One observation of energy E (2^-30 units) into state s's own histogram:
// bin 0 below the window, k + 1 for window bin k, hE_bins + 1 at or beyond its end.
__device__ __forceinline__ void observe_state_energy(const SweepParams& P, int s, long long E) {
    const long long d = E - P.hE_lo_fix[s];
    const long long kb = d >= 0 ? floor_div(d, P.hE_bin_fix, P.hE_bin_magic) : -1;
    const int idx = kb < 0 ? 0 : (kb >= P.hE_bins ? P.hE_bins + 1 : (int)kb + 1);
    atomicAdd(&P.hE[size_t(s) * (P.hE_bins + 2) + idx], 1ull);
}

// Squared minimum-image distance in binary32 (periodic axes per geometry).
__device__ __forceinline__ float dist2(const Geometry& g, float ax, float ay, float az, float bx, float by,
                                       float bz) {
    const float dy = min_image_exact(ay, by, g.Ly, g.hLy);
    const float dx = cart_dx(g, min_image_exact(ax, bx, g.Lx, g.hLx), dy);
    const float dz = g.periodic_z ? min_image_exact(az, bz, g.Lz, g.hLz) : __fsub_rn(az, bz);
    return r2_of(dx, dy, dz);
}

// Remove a particle (whose packed w gives its cell and slot) from its cell.
__device__ __forceinline__ void cell_remove(const SweepParams& P, const Hot& H, const WalkerSmem& S, float wbits) {
    const int c = cell_bits(wbits), s = slot_bits(wbits);
    if (c >= H.cg.ncell || s >= H.cg.cap || s >= (int)S.cnt[c]) {
        // only reachable after a capacity overflow left a particle out of the list
        atomicOr(P.error, ERR_CAPACITY);
        return;
    }
    const int last = S.cnt[c] - 1;
    const int moved = S.slots[c * H.cg.cap + last];
    S.slots[c * H.cg.cap + s] = (uint16_t)moved;
    S.pos[moved].w = __uint_as_float(((unsigned)c << 16) | (unsigned)s);
    S.cnt[c] = (uint16_t)last;
}

// The per-cell counts alone (direct enumeration where a cell can be over
// capacity): as build_cell_list counts them, a cell beyond cap sets
// ERR_CAPACITY and stays at cap.
__device__ __forceinline__ void count_cells(const SweepParams& P, const Hot& H, const WalkerSmem& S, int N,
                                            int lane) {
    for (int c = lane; c < H.cg.ncell; c += 32) S.cnt[c] = 0;
    __syncwarp();
    for (int base = 0; base < N; base += 32) {
        const int j = base + lane;
        int c = -1;
        if (j < N) {
            const float4 p = S.pos[j];
            c = cell_lin(H, cell3_hot(H, p.x, p.y, p.z));
        }
        const unsigned grp = __match_any_sync(FULL, c);
        if (c >= 0 && lane == __ffs(grp) - 1) {
            const int n = S.cnt[c] + __popc(grp);
            if (n > H.cg.cap) atomicOr(P.error, ERR_CAPACITY);
            S.cnt[c] = (uint16_t)min(H.cg.cap, n);
        }
        __syncwarp();
    }
}

// The walk's running state, identical in every lane of the committing warp but
// for the statistics, which are spread over the lanes (one register instead of
// one per sum): `count` of lane l < 3 the trials of type l, of lane 3 + l the
// accepted ones, of lanes 6 and 7 the moves screened and passed; `sum` of lane
// l the sums of sum_lane, once per sweep.
struct Walk {
    int N, split;
    long long E;
    int k;                 // place of the next move in its sweep
    int count;
    unsigned pairs;        // pairs within rc since the last observation
    long long sum;
    double mE2;            // lane 0: sum of E^2
};

enum SumLane { kSumOmega, kSumOut, kSumN, kSumN2, kSumE, kSumC, kSumC2, kSumPairs, kSumLanes };

// Decide move m (evaluated as r) and apply it: executed by all lanes of the
// committing warp, which hold the same values; lane 0 writes.  Returns 1 if
// the move was accepted.
template <int K, bool TRACE, bool DA, bool CL, bool DIRECT>
__device__ __forceinline__ int commit_move(const SweepParams& P, const Hot& H, const WalkerSmem& S, const StateF& sf,
                                           const Trial& r, int w, int s, int m, Walk& W, int lane) {
    const bool two = CL && P.gc2;
    int status = r.status;
    if (K > 1 && r.type == 1 && W.N == H.nmax) status = 1;    // became full in this round
    const long long dfix = fix_value(r.big, r.hi, r.lo);
    // cell and slot of the particle now (with K > 1 an earlier move of the
    // round may have renumbered its slot)
    float ow = r.ow;
    int c_old = -1;
    const bool counted = !DIRECT || H.cg.cap < H.nmax;   // cells hold a count
    if (r.type != 1 && status != 1) {
        if (!DIRECT && K > 1) ow = S.pos[r.idx].w;
        if (!DIRECT) c_old = cell_bits(ow);
        else if (counted) c_old = cell_lin(H, cell3_hot(H, r.ox, r.oy, r.oz));
    }
    // capacity of the destination cell
    int n_new = 0;
    const bool stay = r.type == 0 && r.c_new == c_old;
    if (counted && status == 0 && r.type != 2 && !stay) {
        n_new = S.cnt[r.c_new];
        if (n_new >= H.cg.cap) {
            status = 3;
            if (lane == 0) atomicOr(P.error, ERR_CAPACITY);
        }
    }
    // acceptance: ln u < ln alpha (pre-tested by the evaluating warp when N is
    // still the one it saw)
    int accepted = 0;
    double la = 0.0;
    // the grand-canonical species of the move: its count and constants
    const int split = W.split;
    const int gcnt = (CL && r.gy == 0) ? split : W.N - split;
    const bool use2 = two && r.gy == 1;
    auto log_alpha = [&]() {
        double c = 0.0;
        if (r.type == 1) c = (use2 ? P.c_ins2 : P.c_ins)[s] - P.ln_tab[gcnt + 1];
        else if (r.type == 2) c = (use2 ? P.c_del2 : P.c_del)[s] + P.ln_tab[gcnt];
        return c - P.beta[s] * ((double)dfix * kFixUnit);
    };
    if (DA && status == 0) {
        // both stages were decided by the evaluation
        accepted = !r.ovl && r.dec == 1;
        W.count += (lane == 6) + (lane == 7 && r.stage1);
        if (TRACE) la = r.stage1 ? log_alpha() : (double)NAN;
    } else if (status == 0 && !r.ovl) {
        int dec = r.dec;
        if (K > 1 && W.N != r.n_eval)
            dec = pretest(count_term(r.type, gcnt, use2 ? sf.c_ins2 : sf.c_ins, use2 ? sf.c_del2 : sf.c_del), sf.beta,
                          fix_to_f32(r.big, r.hi, r.lo), r.lu);
        accepted = dec == 1;
        if (dec == 2 || TRACE) {
            la = log_alpha();
            if (dec == 2) accepted = (log((double)r.b1 + 0.5) + kLn2m32) < la;
        }
    }
    if (accepted) {
        const int N = W.N, cap = H.cg.cap;
        __syncwarp();   // every lane has read what lane 0 now writes
        if (lane == 0) {
            if (r.type == 0) {
                if (DIRECT) {
                    S.pos[r.idx] = make_float4(r.qx, r.qy, r.qz, 0.f);
                    if (counted && !stay) {
                        S.cnt[c_old] = (uint16_t)(S.cnt[c_old] - 1);
                        S.cnt[r.c_new] = (uint16_t)(n_new + 1);
                    }
                } else if (stay) {
                    S.pos[r.idx] = make_float4(r.qx, r.qy, r.qz, ow);
                } else {
                    // out of the old cell first: the slot swap may renumber the
                    // particle itself
                    cell_remove(P, H, S, ow);
                    S.slots[r.c_new * cap + n_new] = (uint16_t)r.idx;
                    S.cnt[r.c_new] = (uint16_t)(n_new + 1);
                    S.pos[r.idx] = packed(r.qx, r.qy, r.qz, r.c_new, n_new);
                }
            } else if (r.type == 1) {
                // a new particle goes to the end, or (species B of two
                // grand-canonical species) to index split, whose C moves to the end
                int at = N;
                if (two && r.gy == 0) {
                    at = split;
                    if (split < N) {
                        const float4 pc = S.pos[split];
                        S.pos[N] = pc;
                        if (!DIRECT) S.slots[cell_bits(pc.w) * cap + slot_bits(pc.w)] = (uint16_t)N;
                    }
                }
                if (counted) S.cnt[r.c_new] = (uint16_t)(n_new + 1);
                if (!DIRECT) S.slots[r.c_new * cap + n_new] = (uint16_t)at;
                S.pos[at] = DIRECT ? make_float4(r.qx, r.qy, r.qz, 0.f) : packed(r.qx, r.qy, r.qz, r.c_new, n_new);
            } else {
                if (!DIRECT) cell_remove(P, H, S, ow);
                else if (counted) S.cnt[c_old] = (uint16_t)(S.cnt[c_old] - 1);
                const int last = N - 1;
                // the gap is filled from the end of the particle's block; a
                // removed B's block end is then filled by the last C
                const int fill = (two && r.gy == 0) ? split - 1 : last;
                if (r.idx != fill) {
                    const float4 pl = S.pos[fill];
                    S.pos[r.idx] = pl;
                    if (!DIRECT) S.slots[cell_bits(pl.w) * cap + slot_bits(pl.w)] = (uint16_t)r.idx;
                }
                if (fill != last) {
                    const float4 pc = S.pos[last];
                    S.pos[fill] = pc;
                    if (!DIRECT) S.slots[cell_bits(pc.w) * cap + slot_bits(pc.w)] = (uint16_t)fill;
                }
            }
        }
        const int dn = (r.type == 1) - (r.type == 2);
        W.E += dfix;
        W.N += dn;
        if (two && r.gy == 0) W.split += dn;
        __syncwarp();   // the writes are seen by the next evaluation
    }
    W.count += (lane == r.type) + (accepted && lane == r.type + 3);
    // pairs that entered dE (a move that became impossible in this round,
    // status 1, has none, whatever its evaluation counted)
    if (status != 1) W.pairs += (unsigned)r.pairs;   // below 2^14 a move, at most 1024 moves a sweep
    const int k = W.k;
    W.k = k + 1 == H.mps ? 0 : k + 1;
    if (TRACE && lane == 0) {
        const int ts = m / H.mps;
        regc_move_record t;
        t.type = r.type;
        t.index = status == 1 ? 0
                              : (r.type == 1 ? ((two && r.gy == 0) ? split : W.N - accepted) : r.idx);
        t.accepted = accepted;
        t.status = status == 3 ? 0 : status;
        t.dE = (status == 0 || status == 3) ? (double)dfix * kFixUnit : 0.0;
        if (DA && status == 0 && !r.stage1) t.dE = (double)NAN;
        t.log_alpha = (status == 0 || status == 3) ? (r.ovl ? -INFINITY : la) : 0.0;
        t.ln_u = log((double)r.b1 + 0.5) + kLn2m32;
        t.sum_abs = 0.0;
        t.band = 0.0;
        t.n_pairs = r.pairs;
        t.stage1 = DA ? r.stage1 : 1;
        t.dE_sur = DA ? (double)r.dE_sur : 0.0;
        t.ln_u1 = log((double)r.b3 + 0.5) + kLn2m32;
        P.trace[(size_t(w) * P.trace_steps + ts) * H.mps + k] = t;
    }
    // observe once per sweep into the current state's histograms
    if (k == H.mps - 1) {
        // N_B: the grand-canonical count (with two species, species B's)
        const int NB = two ? W.split : W.N - W.split;
        const int NC = two ? W.N - W.split : 0;
        const long long d = W.E - P.e_lo_fix;
        const long long kb = d >= 0 ? floor_div(d, P.e_bin_fix, P.e_bin_magic) : -1;
        const bool in = kb >= 0 && kb < P.n_e_bins;
        long long v = lane == kSumOmega ? 1 : 0;
        if (lane == kSumOut) v = !in;
        if (lane == kSumN) v = NB;
        if (lane == kSumN2) v = (long long)NB * NB;
        if (lane == kSumE) v = W.E;
        if (CL && lane == kSumC) v = NC;
        if (CL && lane == kSumC2) v = (long long)NC * NC;
        if (lane == kSumPairs) v = W.pairs;
        W.sum += v;
        W.pairs = 0u;
        if (lane == 0) {
            const double e = (double)W.E * kFixUnit;
            W.mE2 = fma(e, e, W.mE2);
            atomicAdd(&P.hN[size_t(s) * (H.nmax + 1) + NB], 1ull);   // fire-and-forget reductions
            if (two) atomicAdd(&P.hN2[size_t(s) * (H.nmax + 1) + NC], 1ull);
            const size_t row = two ? size_t(NB) * (H.nmax + 1) + NC : size_t(NB);
            if (in) atomicAdd(&P.hNE[row * P.n_e_bins + (size_t)kb], 1ull);
            if (P.hE) observe_state_energy(P, s, W.E);
        }
    }
    return accepted;
}

// --------------------------------------------------------------- the walk

// n_sweeps sweeps of walker w by a group of K warps (tid: thread index in the
// group, smem: the group's shared-memory region, bar: the group's named
// barrier when K > 1).
template <int K, bool TRACE, bool DA, bool CL, bool DIRECT, int GEO>
__device__ __forceinline__ void walker_sweep(const SweepParams& P, int w, char* smem, int tid, int bar) {
    static_assert(!(DA && DIRECT), "the feature sums follow the cell list's order");
    const int lane = tid & 31, warp = tid >> 5;
    const WalkerSmem S = carve<K, DIRECT>(smem, P);
    const Hot H = make_hot<GEO>(P);

    Walk W;
    W.N = P.n[w];
    W.E = P.efix[w];
    const int s = P.state_of_walker[w];
    const bool two = CL && P.gc2;
    // two mobile species: particles [0, split) are the cluster, or species B
    // of two grand-canonical species (then split = N_B changes with the moves)
    W.split = CL ? (two ? P.nb[w] : P.n_cluster) : 0;
    const StateF sf{P.beta_f[s], P.c_ins_f[s], P.c_del_f[s], two ? P.c_ins2_f[s] : 0.f,
                    two ? P.c_del2_f[s] : 0.f};
    float4* gpos = P.pos + size_t(w) * H.nmax;

    // 1. stage positions with a bulk copy
    if (W.N > 0) {
        if (tid == 0) {
            mbar_init(S.bar);
            // the region may have been read and written by ordinary accesses
            // (a previous walker): order those before the asynchronous copy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (!P.expire_waits) bulk_load(S.pos, gpos, uint32_t(W.N) * 16u, S.bar);
        }
        group_sync<K>(bar);
        const bool ok = mbar_wait_bounded(S.bar);
        const bool all_ok = group_all<K>(bar, ok);
        if (!all_ok) {
            if (tid == 0) atomicOr(P.error, ERR_TIMEOUT);
            mbar_wait_bounded(S.bar);  // one more bounded chance for the copy in flight
            return;
        }
        group_sync<K>(bar);
        if (tid == 0) mbar_inval(S.bar);   // the barrier's memory is reused by the next walker
    }
    // 2. cell list (deterministic: in particle order), or the counts alone
    if (warp == 0) {
        if (!DIRECT) build_cell_list(P, S.pos, W.N, S.cnt, S.slots, lane);
        else if (H.cg.cap < H.nmax) count_cells(P, H, S, W.N, lane);
    }
    group_sync<K>(bar);

    const LaneCell lc = lane_cell(H, lane);
    int n_cand = 0;
    NetFrag nf;                       // the surrogate's weights in this lane's fragments
    if (DA) load_net(P.net, lane, nf);
    const int total_moves = P.n_sweeps * H.mps;
    const float rc_guard = H.g.rc2 * 1.0004f + 1e-6f;   // a little beyond rc, conservatively
    int filled = 0;   // moves drawn so far
    int m0 = P.m_first;   // first move of the round
    W.k = P.m_first % H.mps;
    W.count = 0;
    W.pairs = 0u;
    W.sum = 0;
    W.mE2 = 0.0;
    unsigned long long rounds = 0, evals = 0;

#pragma unroll 1
    while (m0 < total_moves) {
        // 3a. the next 32 moves, one per lane of the first warp
        if (m0 + K > filled) {
            if (warp == 0) draw_moves<CL>(P, H, S.ring, w, filled, total_moves, lane);
            filled += 32;
            group_sync<K>(bar);
        }
        if (K == 1) {
            const Trial r = evaluate_move<DA, CL, DIRECT>(P, H, S, sf, s, m0, W.N, W.split, n_cand, lc, lane, 0, &nf);
            commit_move<K, TRACE, DA, CL, DIRECT>(P, H, S, sf, r, w, s, m0, W, lane);
            m0 += 1;
            continue;
        }
        // 3b. evaluate moves m0 .. m0 + K - 1 in parallel, one warp each
        if (m0 + warp < total_moves) {
            const Trial r =
                evaluate_move<DA, CL, DIRECT>(P, H, S, sf, s, m0 + warp, W.N, W.split, n_cand, lc, lane, warp, &nf);
            if (lane == 0) S.res[warp] = r;
        }
        group_sync<K>(bar);
        // 4. commit in order (the first warp)
        if (warp == 0) {
            bool any_acc = false, n_changed = false;
            float chx = 0.f, chy = 0.f, chz = 0.f;   // lane c: the c-th position changed by an accepted move
            int nch = 0, committed = 0;
            // not unrolled: one copy of the commit keeps the kernel's code
            // small enough for the instruction caches
#pragma unroll 1
            for (int j = 0; j < K && m0 + j < total_moves; ++j) {
                const Trial r = S.res[j];
                // is the evaluation still the one the sequential chain would make?
                if (any_acc) {
                    bool valid = true;
                    if (n_changed && r.type != 1) valid = false;                      // index of N picked
                    if (r.type == 1 && r.status == 1 && W.N != H.nmax) valid = false;  // no longer full
                    // a changed position within rc of a query point: the energy
                    // change would differ; the old position of a displacement is
                    // checked whatever its status, since its particle may have moved
                    if (valid && (r.status == 0 || (r.type == 0 && r.status == 2))) {
                        bool hit = false;
                        if (lane < nch) {
                            hit = (r.status == 0 && dist2(H.g, chx, chy, chz, r.qx, r.qy, r.qz) < rc_guard) ||
                                  (r.type == 0 && dist2(H.g, chx, chy, chz, r.ox, r.oy, r.oz) < rc_guard);
                        }
                        valid = !__any_sync(FULL, hit);
                    }
                    if (!valid) break;
                }
                const int acc = commit_move<K, TRACE, DA, CL, DIRECT>(P, H, S, sf, r, w, s, m0 + j, W, lane);
                if (acc) {
                    any_acc = true;
                    if (lane == nch) { chx = r.qx; chy = r.qy; chz = r.qz; }
                    ++nch;
                    if (r.type == 0) {
                        if (lane == nch) { chx = r.ox; chy = r.oy; chz = r.oz; }
                        ++nch;
                    } else {
                        n_changed = true;
                    }
                }
                ++committed;
            }
            if (lane == 0) {
                S.hdr->N = W.N;
                S.hdr->E = W.E;
                S.hdr->split = W.split;
                S.hdr->committed = committed;
            }
            rounds += 1;
            evals += min(K, total_moves - m0);
        }
        // the header and the results are rewritten only after every warp has
        // passed the next round's barriers
        group_sync<K>(bar);
        W.N = S.hdr->N;
        W.E = S.hdr->E;
        W.split = S.hdr->split;
        m0 += S.hdr->committed;
    }
    if (K == 1) rounds = evals = (unsigned long long)max(0, total_moves - P.m_first);

    // 7. write back
    for (int j = tid; j < W.N; j += 32 * K) gpos[j] = S.pos[j];
    // candidate distances evaluated (all evaluations, kept or not)
    const unsigned sum_cand = __reduce_add_sync(FULL, (unsigned)n_cand);
    if (lane == 0) atomicAdd(&P.pair_counts[1], (unsigned long long)sum_cand);
    if (warp == 0) {
        if (lane == kSumPairs) W.sum += W.pairs;
        if (lane < 6) P.move_counts[size_t(w) * 6 + (lane < 3 ? 2 * lane : 2 * (lane - 3) + 1)] += W.count;
        if (DA && (lane == 6 || lane == 7))
            atomicAdd(&P.pair_counts[lane - 2], (unsigned long long)(unsigned)W.count);
        double* mm = P.moments + size_t(s) * 4;
        if (lane == kSumOmega) P.omega[s] += (unsigned long long)W.sum;
        if (lane == kSumOut) P.e_out[s] += (unsigned long long)W.sum;
        if (lane == kSumN || lane == kSumN2) mm[lane - kSumN] += (double)W.sum;
        if (lane == kSumE) mm[2] += (double)W.sum * kFixUnit;
        if (two && (lane == kSumC || lane == kSumC2)) P.moments2[size_t(s) * 2 + lane - kSumC] += (double)W.sum;
        if (lane == kSumPairs) atomicAdd(&P.pair_counts[0], (unsigned long long)W.sum);
        if (lane == 0) {
            mm[3] += W.mE2;
            atomicAdd(&P.pair_counts[2], rounds);
            atomicAdd(&P.pair_counts[3], evals);
            P.n[w] = W.N;
            P.efix[w] = W.E;
            if (two) P.nb[w] = W.split;
        }
    }
}

}  // namespace
}  // namespace regc
