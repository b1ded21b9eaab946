// Largest errors of the self-written FP32 functions of project.cuh and common.cuh
// against CUDA's FP64 functions (built and run by test_gpu_math.py).
#include "common.cuh"
#include "project.cuh"

namespace {

__device__ unsigned hash(unsigned x) {
    x = (x ^ (x >> 16)) * 0x7feb352du;
    x = (x ^ (x >> 15)) * 0x846ca68bu;
    return x ^ (x >> 16);
}
__device__ float uniform(unsigned h) { return (h >> 8) * 0x1p-24f; }
__device__ double in_ulps(float got, double ref) { return fabs((double)got - ref) * ldexp(1.0, 23 - ilogb(ref)); }
__device__ double relative(float got, double ref) { return fabs((double)got - ref) / fabs(ref); }

// what: 0 arctangent of every float of [2^-31, 1], 1 quotient, 2 num / sqrt(x), 3 inv_sqrt
__global__ void k_errors(int what, unsigned long long n, unsigned long long *worst) {
    double e = 0.0;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned h = hash((unsigned)i), g = hash(h + 0x9e3779b9u);
        double d;
        if (what == 0) {
            const float x = __uint_as_float(0x30000000u + (unsigned)i), y = proj::atan_unit(x);
            d = proj::atan_unit(-x) == -y ? in_ulps(y, atan((double)x)) : 1e9;
        } else if (what == 1) {   // 2^-50 <= den < 1, 2^-60 den <= |num| <= den
            const float den = ldexpf(0.5f + 0.5f * uniform(h), -(int)(g % 50u));
            const float num = (g & 64u ? -1.f : 1.f) * ldexpf(den * (0.5f + 0.5f * uniform(hash(g))), -(int)((g >> 8) % 60u) * (int)(g >> 31));
            d = in_ulps(proj::recip_times(num, den), (double)num / (double)den);
        } else if (what == 2) {   // x = num (1 + z), 0 <= z <= 1, 1e-30 <= num <= 1
            const float num = ldexpf(0.5f + 0.5f * uniform(h), -(int)(g % 100u)), x = num * (1.f + uniform(hash(g)));
            d = relative(proj::rsqrt_times(num, x), (double)num / sqrt((double)x));
        } else {   // 2^-150 <= v < 2^150
            const double v = ldexp(0.5 + (double)h * 0x1p-33 + (double)g * 0x1p-65, (int)(hash(g) % 300u) - 149);
            const double ref = 1.0 / sqrt(v);
            d = ref < 0x1p126 && ref > 0x1p-126 ? in_ulps(inv_sqrt(v), ref) : 0.0;
        }
        e = d > e ? d : e;
    }
    atomicMax(worst, (unsigned long long)__double_as_longlong(e));   // non-negative doubles order as integers
}

}  // namespace

extern "C" int math_error(int what, unsigned long long n, double *worst) {
    unsigned long long *w = nullptr, r = 0;
    cudaError_t e = cudaMalloc(&w, sizeof r);
    if (e == cudaSuccess) e = cudaMemset(w, 0, sizeof r);
    if (e == cudaSuccess) {
        k_errors<<<1216, 256>>>(what, n, w);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&r, w, sizeof r, cudaMemcpyDeviceToHost);
    if (w) cudaFree(w);
    memcpy(worst, &r, sizeof r);
    return (int)e;
}
