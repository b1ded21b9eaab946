// All-pairs XCF search for 128 x 128 detectors (the hot loop of the indexer).
//
// Paper: Eqs. 3 and 6 (correlation surface r(s) = sum_k conj(S_t) S_p
// exp(+2 pi i k.s / N)), Fig. 1 B-C (best template by peak height), Fig. 5 /
// Discussion (one inverse FFT per pattern-template pair dominates the cost).
//
// One CTA (512 threads, one per SM) keeps one pattern's half spectrum in
// shared memory and streams the library's half spectra from L2/HBM.  Its two
// groups of 256 threads each correlate one template at a time, the even and the
// odd ones: the real surface of X = conj(S_t) S_p, whose 128 rows are
// transformed as 64 complex lines (rows y and y + 64 packed, Ra + i Rb), from 64
// complex columns (columns 0 and 64, real after the column transform, packed in
// one), 8,192 complex values in 64 KB of shared memory and 32 per thread.  Three
// register rounds with two shared-memory transposes:
//   round 1: thread (q, l): stored column q, rows u = l + 8 m: 16-point FFTs
//            over m for l and l + 4, twiddle W128^(l k2);
//   round 2: thread (k2, g): radix 8 over l completes rows k2 + 16 j of the
//            columns +-g mod 32, the rows are paired into lines, radix 4 over
//            the line's columns g + 32 i, twiddle W128^(g k3);
//   round 3: thread (line, k3): a 32-point FFT over g gives the columns k3 + 4 k4
//            of two rows; the maximum is kept per thread.
// Rounds 2 and 3 of a warp (two k2, all g; eight lines) exchange within the
// warp: three barriers of the group per template.
//
// What bounds it: the FP32 issue of the transforms (15 k warp instructions per
// template, 12 k of them FP32) and the shared-memory traffic of the exchanges
// (448 KB) take about the same time, so they have to overlap.  With one
// template pair per 512-thread CTA (Re and Im the two surfaces of one complex
// transform) all sixteen warps met at six barriers per pair and did either the
// one or the other: 168.0 ms for 2,000 patterns x 4,065 templates.  Two groups
// that share no barrier: 156.0 ms; rounds 2 and 3 within a warp and no exchange
// for the maximum: 152.8 ms = 33.2 TFLOP/s of algorithmic work, 41 % of the
// FP32 peak (issue active 65 %, shared-memory pipe 67 %).  Loading the templates
// straight into registers, without the staging copy, measured 201 ms (no
// registers left to cover the L2 latency).
// No surface is written to global memory; only the per-pattern best key (and
// optionally every per-pair peak) leave the kernel.
//
// Library spectra are read in a packed "search layout" (pack_search_layout):
// for each template, columns 0..63 as [l][m/2][q][m&1] with u = l + 8m (64 KB,
// so that the 16 rows a round-1 thread needs are 8 conflict-free 16-byte
// shared loads), then column 64.  A group's next template is copied from L2
// with cp.async into its buffer while round 3 computes.
#include "common.cuh"
#include "kernels.cuh"

#include "search128.cuh"

namespace {

using namespace s128;

template <bool ALL>
__global__ void __launch_bounds__(NT, 1)
k_search128(const float2 *__restrict__ Spk, int T, const float2 *__restrict__ Sp,
            const int *__restrict__ degen, int pairs_per_cta,
            unsigned long long *__restrict__ keys, float *__restrict__ peaks_all) {
    const int p = blockIdx.y;
    if (degen[p]) return;
    const int npairs = (T + 1) / 2;
    const int pb = blockIdx.x * pairs_per_cta;
    const int pe = min(npairs, pb + pairs_per_cta);
    if (pb >= pe) return;
    search_body<ALL>(Spk, T, Sp, p, pb, pe, keys, peaks_all);
}

// the same over each pattern's candidate list cand [P][kc]: 2,000 patterns x 32
// candidates 3.13 -> 1.49 ms (26.7 TFLOP/s), one pattern's 20 -> 14 us for one and 61
// -> 56 us for 32, against template pairs as warp lines on 1,024-thread CTAs
__global__ void __launch_bounds__(NT, 1)
k_search128_list(const float2 *__restrict__ Spk, const int *__restrict__ cand, int kc, const float2 *__restrict__ Sp,
                 const int *__restrict__ degen, int pairs_per_cta, unsigned long long *__restrict__ keys) {
    const int p = blockIdx.y;
    if (degen[p]) return;
    const int pb = blockIdx.x * pairs_per_cta, pe = min((kc + 1) / 2, pb + pairs_per_cta);
    if (pb >= pe) return;
    search_body<false, true>(Spk, kc, Sp, p, pb, pe, keys, nullptr, cand + (size_t)p * kc);
}

// standard half spectra [T][128][65] -> packed search layout [T][8320]
__global__ void k_pack_search_layout(const float2 *__restrict__ src, int T, float2 *__restrict__ dst) {
    const size_t total = (size_t)T * SPEC;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t t = i / SPEC;
        const int k = (int)(i % SPEC), u = k / HW, v = k % HW;
        dst[t * SPEC + (v < 64 ? pk(u, v) : COL64 + u)] = src[i];
    }
}

// one CTA per SM at a time: split the library into at most max(4, SMs / P)
// parts of at least 8 pairs each, taking the part count c that minimises
// waves(P c) x pairs per part (the split does not change the results: the
// key is an exact maximum, the lowest template winning ties)
int pairs_per_part(int npairs, int P, int num_sms) {
    const int cap = max(1, min(max(4, (num_sms + P - 1) / P), (npairs + 7) / 8));
    int chunks = 1;
    long best_cost = -1;
    for (int c = 1; c <= cap; ++c) {
        const long waves = ((long)P * c + num_sms - 1) / num_sms;
        const long cost = waves * ((npairs + c - 1) / c);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            chunks = c;
        }
    }
    return (npairs + chunks - 1) / chunks;
}

}  // namespace

cudaError_t launch_pack_search_layout(const float2 *spectra, int T, int N_, float2 *packed, cudaStream_t st) {
    if (N_ != N) return cudaErrorInvalidValue;
    if (T <= 0) return cudaSuccess;
    const size_t total = (size_t)T * SPEC;
    const int blocks = (int)((total + 255) / 256 < 65536 ? (total + 255) / 256 : 65536);
    k_pack_search_layout<<<blocks, 256, 0, st>>>(spectra, T, packed);
    return cudaGetLastError();
}

cudaError_t launch_search128(const float2 *Spk, int T, const float2 *Sp, const int *degen, int P,
                             unsigned long long *keys, float *peaks_all, int num_sms, cudaStream_t st) {
    auto *kern = peaks_all ? k_search128<true> : k_search128<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
    if (e != cudaSuccess) return e;
    const int ppc = pairs_per_part((T + 1) / 2, P, num_sms);
    const dim3 grid(((T + 1) / 2 + ppc - 1) / ppc, P);
    kern<<<grid, NT, SMEM_BYTES, st>>>(Spk, T, Sp, degen, ppc, keys, peaks_all);
    return cudaGetLastError();
}

cudaError_t launch_search128_list(const float2 *Spk, const int *cand, int kc, const float2 *Sp, const int *degen, int P,
                                  unsigned long long *keys, int num_sms, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_search128_list, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
    if (e != cudaSuccess) return e;
    const int ppc = pairs_per_part((kc + 1) / 2, P, num_sms);
    const dim3 grid(((kc + 1) / 2 + ppc - 1) / ppc, P);
    k_search128_list<<<grid, NT, SMEM_BYTES, st>>>(Spk, cand, kc, Sp, degen, ppc, keys);
    return cudaGetLastError();
}
