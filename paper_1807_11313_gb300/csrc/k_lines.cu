// All-pairs search for the native 160 and 200 px sides: one real correlation
// surface at a time as N / 2 packed complex lines in shared memory.
//
// Paper: the correlation surface of Eqs. 3/6 and its maximum (Fig. 1 B-C).
//
// The surface's rows y and y + N / 2 are one complex line of N values, its half
// spectrum N / 2 complex columns (columns 0 and N / 2, real after the column
// transform, packed in one): N^2 / 2 values, 102 KB at 160 and 160 KB at 200.
// With columns N = R1 R2 and lines N = S1 S2 the transform is four passes of
// small DFTs, each task reading and writing its own slots of the buffer L[line][v],
// so that a thread takes one task after another:
//   1: column q, l: products conj(S_t) S_p at rows l + R2 m straight from the
//      spectra in L2; R1 points over m, twiddle;
//   2: column q, k2: R2 points over l give the rows k2 + R1 j, paired into the
//      lines' columns q and N - q (the slots the inputs lay in);
//   3: line, g: S1 points over the columns g + S2 i, twiddle;
//   4: line, k3: S2 points over g; the maximum per thread.
// Four barriers per template.  At 160 two 320-thread CTAs share an SM and fill
// each other's waits; the pattern is read from L2 beside the template (its 104 KB
// beside two buffers do not fit).  Line slots of 16 are swizzled at 160 so that
// pass 4's 16-byte loads spread over every bank.
// Bound by instruction issue and the three exchanges.  301 patterns x 1,018
// templates at 160: 22.0 -> 14.0 ms (14.1 -> 22.2 TFLOP/s) against warp-line
// transforms of template pairs on one 1,024-thread CTA (256 to 512 threads here:
// 14.0 to 14.6; one CTA of 640: 16.1); 150 x 500 at 200: 16.2 -> 5.95 ms (7.6 ->
// 20.8 TFLOP/s) against Stockham passes of one warp per line.
#include "common.cuh"
#include "dft_small.cuh"
#include "kernels.cuh"

namespace {

template <int N_>
struct Plan;
template <>
struct Plan<160> {
    static constexpr int R1 = 16, R2 = 10, S1 = 10, S2 = 16, NT = 320, CTAS = 2;
};
template <>
struct Plan<200> {
    static constexpr int R1 = 20, R2 = 10, S1 = 10, S2 = 20, NT = 512, CTAS = 1;
};

template <int N>
struct Smem {
    float2 line[N * N / 2];
    float2 tw[N];      // e^{+2 pi i e / N}
    float2 p0[N];      // the packed column X[u][0] + i X[u][N / 2]
    float red[32];
};

// slot of column v of a line
template <int N>
__device__ __forceinline__ int slot(int pr, int v) {
    if constexpr (Plan<N>::S2 == 16) {
        const int b = v >> 4, sw = (pr * Plan<N>::S1 + b) & 7;
        return pr * N + (b << 4) + (((((v & 15) >> 1) ^ sw) << 1) | (v & 1));
    } else {
        return pr * N + v;
    }
}

template <int N, bool ALL>
__global__ void __launch_bounds__(Plan<N>::NT, Plan<N>::CTAS)
k_search_lines(const float2 *__restrict__ St, int T, const float2 *__restrict__ Sp, const int *__restrict__ degen,
               int per_cta, unsigned long long *__restrict__ keys, float *__restrict__ peaks_all,
               const int *__restrict__ cand, int kc) {
    using L = Plan<N>;
    constexpr int HW = N / 2 + 1, C = N / 2, R1 = L::R1, R2 = L::R2, S1 = L::S1, S2 = L::S2, NT = L::NT;
    const int p = blockIdx.y;
    if (degen[p]) return;
    const int n = cand ? kc : T;
    const int jb = blockIdx.x * per_cta, je = min(n, jb + per_cta);
    extern __shared__ float4 smem_raw[];
    Smem<N> &sm = *reinterpret_cast<Smem<N> *>(smem_raw);
    float2 *line = sm.line;
    const int tid = threadIdx.x;
    const float2 *sp = Sp + (size_t)p * N * HW;
    for (int e = tid; e < N; e += NT) {
        const int r = e < C ? e : e - C;
        const float2 w = make_float2(kTwTable<N>.re[r], kTwTable<N>.im[r]);
        sm.tw[e] = e < C ? w : make_float2(-w.x, -w.y);
    }
    float2 s0 = make_float2(0.f, 0.f), sh = s0;   // the pattern's columns 0 and N / 2 at row tid
    if (tid < N) {
        s0 = __ldg(sp + tid * HW);
        sh = __ldg(sp + tid * HW + C);
    }
    auto template_of = [&](int j) { return cand ? cand[(size_t)p * kc + j] : j; };
    auto next_used = [&](int j) {   // the next slot with a template (uniform over the CTA)
        while (j < je && template_of(j) < 0) {
            if (ALL && tid == 0) peaks_all[(size_t)p * n + j] = -INFINITY;
            ++j;
        }
        return j;
    };
    auto make_p0 = [&](const float2 *tp) {
        if (tid < N) {
            const float2 a = c_mulcj(__ldg(tp + tid * HW), s0), h = c_mulcj(__ldg(tp + tid * HW + C), sh);
            sm.p0[tid] = make_float2(a.x - h.y, a.y + h.x);
        }
    };
    float best_v = -INFINITY;
    int best_t = -1;
    int j = next_used(jb);
    if (j < je) make_p0(St + (size_t)template_of(j) * N * HW);
    __syncthreads();
    while (j < je) {
        const int t = template_of(j), jn = next_used(j + 1);
        const float2 *tp = St + (size_t)t * N * HW;
        // ---- 1
        for (int task = tid; task < C * R2; task += NT) {
            const int l = task / C, q = task - l * C;
            float2 x[R1];
            {
                float2 s[R1];
#pragma unroll
                for (int m = 0; m < R1; ++m) {
                    const int k = (l + R2 * m) * HW + q;
                    x[m] = __ldg(tp + k);
                    s[m] = __ldg(sp + k);
                }
#pragma unroll
                for (int m = 0; m < R1; ++m) x[m] = c_mulcj(x[m], s[m]);
            }
            if (q == 0) {
#pragma unroll
                for (int m = 0; m < R1; ++m) x[m] = sm.p0[l + R2 * m];
            }
            dft::inverse<R1>(x);
            const bool low = l < R2 / 2;
            const int base = R1 * (low ? l : l - R2 / 2), v = low ? q : q ? N - q : C;
            StaticFor<0, R1>::run([&](auto kk) {
                constexpr int k2 = decltype(kk)::value;
                const float2 y = x[dft::at<R1>(k2)];
                line[slot<N>(base + k2, v)] = k2 ? c_mul(y, sm.tw[l * k2]) : y;
            });
        }
        __syncthreads();
        // ---- 2
        for (int task = tid; task < C * R1; task += NT) {
            const int k2 = task / C, q = task - k2 * C, qm = q ? N - q : C;
            float2 x[R2];
#pragma unroll
            for (int i = 0; i < R2 / 2; ++i) {
                x[i] = line[slot<N>(k2 + R1 * i, q)];
                x[i + R2 / 2] = line[slot<N>(k2 + R1 * i, qm)];
            }
            dft::inverse<R2>(x);
            StaticFor<0, R2 / 2>::run([&](auto ii) {
                constexpr int i = decltype(ii)::value;
                const float2 ra = x[dft::at<R2>(i)], rb = x[dft::at<R2>(i + R2 / 2)];
                float2 z = make_float2(ra.x - rb.y, ra.y + rb.x), zm = make_float2(ra.x + rb.y, rb.x - ra.y);
                if (q == 0) {
                    z = make_float2(ra.x, rb.x);
                    zm = make_float2(ra.y, rb.y);
                }
                line[slot<N>(k2 + R1 * i, q)] = z;
                line[slot<N>(k2 + R1 * i, qm)] = zm;
            });
        }
        __syncthreads();
        // ---- 3
        for (int task = tid; task < C * S2; task += NT) {
            const int pr = task / S2, g = task - pr * S2;
            float2 x[S1];
#pragma unroll
            for (int i = 0; i < S1; ++i) x[i] = line[slot<N>(pr, g + S2 * i)];
            dft::inverse<S1>(x);
            StaticFor<0, S1>::run([&](auto kk) {
                constexpr int k3 = decltype(kk)::value;
                const float2 y = x[dft::at<S1>(k3)];
                line[slot<N>(pr, g + S2 * k3)] = k3 ? c_mul(y, sm.tw[g * k3]) : y;
            });
        }
        __syncthreads();
        // ---- 4; the next template's packed column meanwhile
        if (jn < je) make_p0(St + (size_t)template_of(jn) * N * HW);
        float m = -INFINITY;
        for (int task = tid; task < C * S1; task += NT) {
            const int pr = task / S1, k3 = task - pr * S1;
            float2 x[S2];
            const float4 *src = reinterpret_cast<const float4 *>(line + pr * N + S2 * k3);
#pragma unroll
            for (int i = 0; i < S2 / 2; ++i) {
                const float4 v = src[S2 == 16 ? i ^ (task & 7) : i];
                x[2 * i] = make_float2(v.x, v.y);
                x[2 * i + 1] = make_float2(v.z, v.w);
            }
            dft::inverse<S2>(x);
#pragma unroll
            for (int i = 0; i < S2; ++i) m = fmaxf(m, fmaxf(x[i].x, x[i].y));
        }
        if (m > best_v || (m == best_v && t < best_t)) {
            best_v = m;
            best_t = t;
        }
        if (ALL) {
#pragma unroll
            for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if ((tid & 31) == 0) sm.red[tid >> 5] = m;
        }
        __syncthreads();   // the lines have been read; the next packed column is in place
        if (ALL && tid == 0) {
            for (int w = 1; w < NT / 32; ++w) m = fmaxf(m, sm.red[w]);
            peaks_all[(size_t)p * n + j] = m;
        }
        j = jn;
    }
    unsigned long long key = best_t >= 0 ? pack_key(best_v, best_t) : 0ull;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long k = __shfl_xor_sync(0xffffffffu, key, o);
        key = k > key ? k : key;
    }
    if ((tid & 31) == 0 && key) atomicMax(keys + p, key);
}

template <int N>
cudaError_t run(const float2 *St, int T, const float2 *Sp, const int *degen, int P, unsigned long long *keys,
                float *peaks_all, int num_sms, cudaStream_t st, const int *cand, int kc) {
    using L = Plan<N>;
    const int n = cand ? kc : T;
    if (P <= 0 || n <= 0) return cudaSuccess;
    auto *kern = peaks_all ? k_search_lines<N, true> : k_search_lines<N, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem<N>));
    if (e != cudaSuccess) return e;
    // enough CTAs to fill the GPU a few times over, at least 8 templates each
    const long want = 8L * L::CTAS * num_sms;
    int chunks = (int)((want + P - 1) / P);
    chunks = max(1, min(chunks, (n + 7) / 8));
    const int per = (n + chunks - 1) / chunks;
    chunks = (n + per - 1) / per;
    kern<<<dim3(chunks, P), L::NT, sizeof(Smem<N>), st>>>(St, T, Sp, degen, per, keys, peaks_all, cand, kc);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_search_lines(int N, const float2 *St, int T, const float2 *Sp, const int *degen, int P,
                                unsigned long long *keys, float *peaks_all, int num_sms, cudaStream_t st,
                                const int *cand, int kc) {
    switch (N) {
        case 160: return run<160>(St, T, Sp, degen, P, keys, peaks_all, num_sms, st, cand, kc);
        case 200: return run<200>(St, T, Sp, degen, P, keys, peaks_all, num_sms, st, cand, kc);
        default: return cudaErrorInvalidValue;
    }
}
