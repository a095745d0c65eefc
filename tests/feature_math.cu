// feature_math.cu -- how often the short forms of surrogate.cuh differ from CUDA's
// general ones (built by test_gpu_feature_math.py).
#include "surrogate.cuh"

namespace {

__device__ bool differs(int what, float x, float b, float y) {
    using namespace regc;
    float p = 0.f, q = 0.f;
    switch (what) {
        case 0: p = root(x); q = sqrtf(x); break;
        case 1: p = quotient(x, b, y); q = x / b; break;
        case 2: p = reciprocal(x); q = 1.0f / x; break;
        case 3: p = ex2(x); q = exp2f(x); break;
        case 4: p = ex2(-x); q = exp2f(-x); break;
    }
    return __float_as_uint(p) != __float_as_uint(q);
}

// the binary32 numbers of bit patterns lo .. hi - 1, against each divisor
__global__ void count_kernel(int what, unsigned lo, unsigned hi, const float* div, unsigned long long* count) {
    const float b = div[blockIdx.y], y = 1.0f / b;
    const unsigned end = what == 1 ? min(hi, __float_as_uint(3.14159265358979f * b)) : hi;   // arguments below pi rc
    unsigned n = 0;
    for (unsigned i = lo + blockIdx.x * blockDim.x + threadIdx.x; i < end; i += gridDim.x * blockDim.x)
        n += differs(what, __uint_as_float(i), b, y);
    if (n) atomicAdd(count, (unsigned long long)n);
}

}  // namespace

// Arguments from lo up to hi (0 < lo < hi < 2^127) that differ, over n divisors
// (what 1; else one, unused); -1: a CUDA call failed.
extern "C" __attribute__((visibility("default"))) long long feature_math_differences(int what, float lo, float hi, const float* divisors, int n) {
    float* d = nullptr;
    unsigned long long* c = nullptr;
    unsigned long long got = 0;
    unsigned a, b;
    memcpy(&a, &lo, 4);
    memcpy(&b, &hi, 4);
    cudaError_t e = cudaMalloc(&d, n * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&c, sizeof(got));
    if (e == cudaSuccess) e = cudaMemcpy(d, divisors, n * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(c, 0, sizeof(got));
    if (e == cudaSuccess) {
        count_kernel<<<dim3(1216, n), 256>>>(what, a, b, d, c);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&got, c, sizeof(got), cudaMemcpyDeviceToHost);
    cudaFree(d);
    cudaFree(c);
    return e == cudaSuccess ? (long long)got : -1;
}
