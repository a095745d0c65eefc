// launch.h -- host-side launchers of the REGC kernels (internal to the library).
#pragma once

#include <cuda_runtime.h>

#include "regc_internal.cuh"

namespace regc {

// Nmax up to which a walker's moves enumerate every particle (walker.cuh).  A
// stencil of 27 of the ncell cells spares the share 1 - 27 / ncell of the
// distances and costs what about 96 of them do; with many walkers per SM the
// smaller region counts too (more of them resident), and the line lies higher.
// Microseconds of a ten-sweep launch, direct / cells, every walker nearly full:
//   fcc(111), 168 cells, 16 walkers:   136 / 152 at Nmax 64, 144 / 153 at 96, 148 / 157 at 128, 159 / 157 at 192
//   fcc(111), 1024 walkers (7 per SM):   184 / 207 at 64, 203 / 210 at 96, 218 / 212 at 128
//   periodic cube, 125 cells, 16 walkers:   160 / 165 at 68, 164 / 172 at 96, 178 / 176 at 128
//   periodic cube, 4096 walkers (27 per SM):   416 / 544 at 68, 475 / 551 at 128, 533 / 564 at 160, 593 / 583 at 192
//   A18, 40 cells, 160 walkers of 20 particles:   78 / 101
// Above kDirectMax every walker has cells, also in boxes of few cells, where the
// direct form would still be the faster one (N nearly Nmax, four and one warps):
//   A18, 40 cells, 160 walkers:   109 / 133 at 192, 125 / 143 at 256, 133 / 153 at 320
//   fcc(100), at most 27 cells, 16 and 4096 walkers:   175 / 255 and 780 / 1438 at 192
// Where that ends was not measured; a line beyond it is a change of its own.  The
// rule goes by Nmax, which is known when the shared memory is laid out; the cost goes
// by N, so a walker that stays far below a large Nmax keeps its cells although all
// its particles would cost less.
constexpr int kDirectMax = 160;

inline int direct_limit(int ncell, long long walkers, int sms) {
    const int line = walkers > 12LL * sms ? kDirectMax : 96;
    if (ncell <= 27) return kDirectMax;
    const long long n = (long long)line * ncell / (ncell - 27);
    return n < kDirectMax ? (int)n : kDirectMax;
}

// Whether the system's walkers enumerate all particles with their nearest
// images (walker.cuh) instead of a cell list; delayed acceptance follows the
// cell list.
inline bool sweep_direct(const SweepParams& P) { return P.direct && !P.delayed; }

// The geometry the walk is compiled for (walker.cuh: make_hot): 1 a rectangular
// cell and 2 a sheared one, not periodic in z, over a surface of one atom type;
// 3 a rectangular box, periodic in z, without a surface; 0 any.
inline int sweep_geo(const SweepParams& P) {
    const bool sheared = P.g.shear != 0.0f;
    if (!P.g.periodic_z && P.st.n_all > 0 && P.st.one_type >= 0) return sheared ? 2 : 1;
    return P.g.periodic_z && P.st.n_all == 0 && !sheared ? 3 : 0;
}

// Shared-memory bytes of one walker of the sweep kernel with W warps.
size_t sweep_smem(const SweepParams& P, int warps_per_walker);

// The bytes by which handles are admitted (at most 227 KB; never less than
// sweep_smem of the same sizes).
size_t sweep_smem_admitted(int nmax, int ncell, int cap, int warps_per_walker);

// P.n_sweeps sweeps of every walker with P.warps_per_walker warps per walker;
// P.trace may be null.
cudaError_t launch_sweep(const SweepParams& P, cudaStream_t s);
// launch_sweep of the systems with two mobile species or delayed acceptance.
cudaError_t launch_sweep_species(const SweepParams& P, cudaStream_t s);

// From-scratch fixed-point energy of every walker into out[S]; a pair inside
// the hard-core guard sets ERR_OVERLAP (check_overlap 1) or ERR_NUMERIC
// (check_overlap 2) in P.error.
cudaError_t launch_energy(const SweepParams& P, long long* out, int check_overlap,
                          cudaStream_t s);

// Caller positions xyz [S][nmax][3] -> pos [S][nmax] (zeros beyond n[w]);
// coordinates outside the region set ERR_INPUT in *error.
cudaError_t pack_walkers(const float* xyz, const int* n, int S, int nmax, const Geometry& g, float4* pos, int* error,
                         cudaStream_t s);

// What a read-back returns beside positions: arrays of 32-bit words (words[q]
// of them, 0: none), energies (null: none) and the error word, to host memory
// the device can write (page-locked).
struct ReadBack {
    static constexpr int kSegs = 3;
    const unsigned* src[kSegs];
    unsigned* dst[kSegs];
    long long words[kSegs];
    const long long* efix;   // [S] in units of 2^-30
    double* energy;          // [S]
    int S;
    const int* error;
    int* error_out;
};

// One launch: r, and (xyz given) pos [count] -> xyz [count][3] (count = S nmax);
// with n [S], only the first n[w] entries of each walker are written.
cudaError_t read_back(const float4* pos, long long count, int nmax, const int* n, float* xyz, const ReadBack& r,
                      cudaStream_t s);

// ---------------------------------------------------------------- batch
// Bytes at the head of a batch walker's region of shared memory (before
// sweep_smem's), whether a system's walkers are admitted to a batch, and the
// batch sweep kernel's warp limit per CTA (da: the delayed-acceptance
// instantiation).
size_t batch_head();
bool batch_admits(const SweepParams& P);
int batch_max_warps(bool da);

// What the systems of one batch launch have in common: da, sampling with
// delayed acceptance; cl, a cluster species; direct, sweep_direct; slab,
// sweep_geo 1 (only where it is used: without da and cl).
struct BatchClass {
    bool da, cl, direct, slab;
};

// Persistent sweep of items (system, walker) of the systems sys[] (device
// table; every system's n_sweeps and t0 are read from it), taken in order from
// the queue *counter (zero before the launch); walkers_per_cta walkers of
// warps_per_walker warps each per CTA (1, 2 or 4; more than one for plain
// one-species systems only), each with `region` bytes of dynamic shared
// memory.
cudaError_t launch_batch_sweep(const SweepParams* sys, const int2* items, int n_items, int* counter,
                               int walkers_per_cta, int warps_per_walker, int grid, int region, BatchClass c,
                               cudaStream_t s);

// Allow every batch sweep kernel up to max_smem bytes of shared memory in all
// (before any launch or capture that needs more than 48 KB).
cudaError_t batch_prepare(int max_smem);

// Resident CTAs per SM of the batch sweep kernel for this shape (0 if none fit).
int batch_occupancy(int walkers_per_cta, int warps_per_walker, int region, BatchClass c);

// out[m] = system m's error word (out: page-locked host memory).
cudaError_t batch_errors(const SweepParams* sys, int n_systems, int* out, cudaStream_t s);

// One exchange attempt of every system's grid (attempt numbers e_ctr[]), then
// e_ctr[m] += 1 and sys[m].t0 += n_sweeps on the device.
cudaError_t launch_batch_exchange(const ExchangeParams* xs, uint32_t* e_ctr, SweepParams* sys, int n_systems,
                                  int n_sweeps, cudaStream_t s);

// One MD segment of every walker (md.cu): n_steps velocity-Verlet steps of
// length dt with the stochastic velocity rescaling thermostat (time constant
// tau) from Maxwell-Boltzmann velocities (segment number seg); kinetic
// energies after the last step into kin_out[S] if not null.  Positions are
// written back; energies are not recomputed.
cudaError_t launch_md(const SweepParams& P, int n_steps, float dt, float tau, uint32_t seg, float* kin_out,
                      cudaStream_t s);
size_t md_smem(int nmax, int ncell, int cap);

// One collective exchange attempt number e.
cudaError_t launch_exchange(const ExchangeParams& X, uint32_t e, cudaStream_t s);

// ------------------------------------------------------------ surrogate
// Device buffers of the surrogate's BF16 inference copy.
struct SurrogateStore {
    __nv_bfloat16* w1;   // [64][16]
    float* b1;           // [64]
    __nv_bfloat16* w2;   // [64][64]
    float* b2;           // [64]
    __nv_bfloat16* w3;   // [64]
    float* b3;           // [1]
};

// FP32 master parameters theta[5313] -> the inference copy.
cudaError_t surrogate_pack(const float* theta, const SurrogateStore& st, cudaStream_t s);

// Surrogate energies e_out[Q] and features f_out[Q][16] of Q positions q
// (x, y, z) against every particle of walker w and the surface.
cudaError_t surrogate_eval(const SweepParams& P, int w, int Q, const float4* q, float* e_out, float* f_out,
                           cudaStream_t s);

// S * (parts + probes) training rows (features X[.][16], targets y = min(e, clip))
// written to the ring of cap rows starting at row base.
cudaError_t surrogate_harvest(const SweepParams& P, int parts, int probes, float clip, uint32_t round, float* X,
                              float* y, int base, int cap, cudaStream_t s);

// Floats of the per-CTA gradient scratch of surrogate_step for n rows.
size_t surrogate_partial_floats(int n);

// Gradient of the mean squared error of n rows (idx[t] or t) at theta_in into
// grad (may be null) and the sum of squared residuals into *loss; then, when
// adam_t > 0, Adam step number adam_t with learning rate lr on theta, m, v.
// tensor_cores: the matrix products in BF16 on mma.sync tiles (FP32
// accumulation); else everything in binary32 on the FP32 pipe.
cudaError_t surrogate_step(const float* theta_in, const float* X, const float* y, const int* idx, int n,
                           float* partial, float* grad, float* loss, float* theta, float* m, float* v, int adam_t,
                           float lr, bool tensor_cores, cudaStream_t s);

// Whether a mini-batch of this size trains in one cluster of CTAs, and `steps`
// training steps (rows drawn as surrogate_batch_index draws them for steps
// adam_t + 1 .., gradient and Adam as surrogate_step's on tensor cores, bit for
// bit) of such a mini-batch in one launch; loss [steps]: sums of squared residuals.
bool surrogate_train_fits(int batch);
cudaError_t surrogate_train_steps(float* theta, float* m, float* v, const float* X, const float* y, int count,
                                  int batch, int steps, int adam_t, float lr, uint32_t k0, uint32_t k1, float* loss,
                                  cudaStream_t s);

// Seeded initial parameters (normal weights of standard deviation
// scale / sqrt(fan-in), zero biases) into theta[5313].
cudaError_t surrogate_init(float* theta, float scale, uint32_t k0, uint32_t k1, cudaStream_t s);

// batch uniform row indices in [0, count) for training step `step`.
cudaError_t surrogate_batch_index(int* idx, int batch, int count, uint32_t step, uint32_t k0, uint32_t k1,
                                  cudaStream_t s);

}  // namespace regc
