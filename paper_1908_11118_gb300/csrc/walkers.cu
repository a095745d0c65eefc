// walkers.cu -- walker state in and out of the device (sm_103a).
//
// The caller's positions are [S][nmax][3] binary32; the device keeps
// float4 [S][nmax].  These kernels convert between the two on the device, so a
// state upload or download is one contiguous copy of the caller's buffer and
// one launch, with the coordinate checks of regc_set_walkers done on the GPU.
#include "launch.h"

namespace regc {
namespace {

__global__ void pack_walkers_kernel(const float* xyz, const int* n, int S, int nmax, Geometry g, float4* pos,
                                    int* error) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)S * nmax) return;
    const int w = (int)(k / nmax), i = (int)(k % nmax);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < n[w]) {
        const float x = xyz[3 * k], y = xyz[3 * k + 1], z = xyz[3 * k + 2];
        const bool okx = x >= 0.0f && x < g.Lx, oky = y >= 0.0f && y < g.Ly;
        const bool okz = g.periodic_z ? (z >= 0.0f && z < g.Lz) : (z >= g.z_lo && z <= g.z_hi);
        if (okx && oky && okz) v = make_float4(x, y, z, 0.0f);
        else atomicOr(error, ERR_INPUT);
    }
    pos[k] = v;
}

// One launch for everything a call reads back: positions (where xyz is given;
// with n only the first n[w] entries of each walker), energies, arrays copied
// word by word and the error word, written straight to page-locked host memory.
// Four copies and the error word's, one after the other on the copy engine,
// were most of the 50 us that reading sixteen walkers took.
__global__ void __launch_bounds__(256) read_back_kernel(const float4* pos, long long count, int nmax, const int* n,
                                                        float* xyz, const __grid_constant__ ReadBack r) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (xyz && k < count && !(n && (int)(k % nmax) >= n[k / nmax])) {
        const float4 v = pos[k];
        xyz[3 * k] = v.x;
        xyz[3 * k + 1] = v.y;
        xyz[3 * k + 2] = v.z;
    }
    for (int q = 0; q < ReadBack::kSegs; ++q)
        for (long long i = k; i < r.words[q]; i += stride) r.dst[q][i] = r.src[q][i];
    if (r.energy)
        for (long long i = k; i < r.S; i += stride) r.energy[i] = (double)r.efix[i] * kFixUnit;
    if (k == 0) *r.error_out = *r.error;
}

}  // namespace

cudaError_t pack_walkers(const float* xyz, const int* n, int S, int nmax, const Geometry& g, float4* pos, int* error,
                         cudaStream_t s) {
    const long long count = (long long)S * nmax;
    if (count == 0) return cudaSuccess;
    pack_walkers_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(xyz, n, S, nmax, g, pos, error);
    return cudaGetLastError();
}

cudaError_t read_back(const float4* pos, long long count, int nmax, const int* n, float* xyz, const ReadBack& r,
                      cudaStream_t s) {
    // a thread per position, or per word of a launch of at most 64 CTAs
    long long most = r.energy ? r.S : 1;
    for (int q = 0; q < ReadBack::kSegs; ++q) most = most > r.words[q] ? most : r.words[q];
    long long ctas = (most + 255) / 256 < 64 ? (most + 255) / 256 : 64;
    if (xyz && (count + 255) / 256 > ctas) ctas = (count + 255) / 256;
    read_back_kernel<<<(unsigned)ctas, 256, 0, s>>>(pos, count, nmax, n, xyz, r);
    return cudaGetLastError();
}

}  // namespace regc
