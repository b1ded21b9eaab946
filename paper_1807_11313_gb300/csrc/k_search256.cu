// 256 x 256 all-pairs search on thread-block clusters of two CTAs.
//
// Paper: the cross-correlation of Eqs. 3/6 (conj(S_t) S_p, inverse FFT, peak)
// for every template of the library (Fig. 1 B-C), at the 256 x 256 detector.
//
// One real surface at a time (k_lines.cu's plan): rows y and y + 128 are one
// complex line of 256 values, the half spectrum 128 complex columns (columns 0
// and 128, real after the column transform, packed in one).  The 256 KB of
// values lie in the distributed shared memory of the pair: CTA c owns the
// columns 64 c .. 64 c + 63 in the column passes and the lines 64 c .. 64 c + 63
// in the line passes, 128 KB either way, 32 values per thread.  With 256 = 16 x
// 16 every pass is 16-point transforms, two per thread:
//   1: column q, l: products conj(S_t) S_p at rows l + 16 m straight from the
//      spectra in L2, 16 points over m, twiddle W256^(l k2);
//   2: column q, k2: 16 points over l in place give the rows k2 + 16 j, paired
//      into the lines' columns q and 256 - q;
//   3: line, g: gathers the columns g + 16 i from both CTAs (half of them
//      remote), 16 points over i, twiddle W256^(g k3);
//   4: line, k3: 16 points over g; the maximum per thread.
// Two cluster barriers per template: the lines are complete; they have been
// gathered.
//
// What bounds it: sixteen warps go through the passes together, and the load
// queue (64 global and 18 cluster loads per thread and template) fills in the
// first and third; issue is active 42 %.  300 patterns x 1,018 templates: 53.6 ->
// 39.5 ms (15.9 -> 21.8 TFLOP/s, 27 % of the FP32 peak) against template pairs on
// clusters of four; the 32-candidate rescore of 1,000 patterns 5.42 -> 4.54 ms.  The
// release after the gathers is 0.5 ms of the 39.5; a full one at the barrier between
// the column and line passes too would be 3 % more.
// Measured without gain (without the release after the gathers): 16-byte template loads from an aligned copy of the
// library with half of the pattern in shared memory (41.3), the next template's
// first values loaded a pass ahead (49.4: spills), 1,024 threads at 64 registers
// (42.2), all gathers as cluster loads (41.6); two clusters of four CTAs per four SMs
// (passes256.cuh) 40.3, the rescore 4.42.  The templates stay in the plain
// layout: no second copy of the library (5.5 GB at 20,000 templates).
#include <algorithm>

#include "cluster.cuh"
#include "common.cuh"
#include "kernels.cuh"

namespace {

constexpr int N = 256, HW = 129, NT = 512, NC = 2, OWN = 64;

struct Smem {
    float2 buf[N * N / 4];   // columns: [line][128] (column, mirror); lines: [64][256]
    float2 tw[256];          // W256^(a b) at [a][b]
    float2 p0[N];            // CTA 0: the packed column X[u][0] + i X[u][128]
    float red[NT / 32];
    float top[NC];           // CTA 0: the CTAs' maxima of a surface (every-peak mode)
};

// decimation-in-frequency stages 0 .. 2 of a 16-point inverse transform
__device__ __forceinline__ void dif16_head(float2 (&x)[16]) {
    StaticFor<0, 3>::run([&](auto stage) {
        constexpr int span = 16 >> (decltype(stage)::value + 1);
        StaticFor<0, 16 / (2 * span)>::run([&](auto blk) {
            StaticFor<0, span>::run([&](auto k) {
                constexpr int kk = decltype(k)::value, i0 = decltype(blk)::value * 2 * span + kk, i1 = i0 + span;
                const float2 a = x[i0], b = x[i1];
                x[i0] = c_add(a, b);
                x[i1] = tw_mul<kk, 2 * span, +1>(c_sub(a, b));
            });
        });
    });
}

// the values g + 16 i of lines l0 and l0 + 32 for CTA C: v < 64 and v > 192 (and 128,
// the packed column's mirror) lie with CTA 0, the others with CTA 1, mirrors at 64
// + their column.  Own values by plain shared loads: loads from the cluster queue
// with the global ones, and 32 of them per thread filled that queue.
template <int C>
__device__ __forceinline__ void gather(float2 (&z)[2][16], const float2 *buf, uint32_t base0, uint32_t base1, int l0,
                                       int g) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int line = (l0 + 32 * h) * 128;
        const uint32_t F = (uint32_t)sizeof(float2), at0 = base0 + line * F, at1 = base1 + line * F;
        StaticFor<0, 16>::run([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if constexpr (i == 8) {   // v = 128 + g: 256 - v with CTA 1, or 128
                z[h][i] = ld_cluster(g ? at1 + (128 - g) * F : at0 + 64 * F);
            } else if constexpr (i == 12) {   // v = 192 + g: 320 - v with CTA 0, or 192
                z[h][i] = ld_cluster(g ? at0 + (128 - g) * F : at1 + 64 * F);
            } else {
                constexpr int owner = i >= 4 && i < 12 ? 1 : 0;
                const int s = i < 4 ? g + 16 * i : i < 8 ? g + 16 * i - 64 : i < 12 ? 256 - 16 * i - g : 320 - 16 * i - g;
                if constexpr (owner == C) z[h][i] = buf[line + s];
                else z[h][i] = ld_cluster((owner ? at1 : at0) + s * F);
            }
        });
    }
}

template <bool ALL>
__global__ void __launch_bounds__(NT, 1)
k_search256(const float2 *__restrict__ St, int T, const float2 *__restrict__ Sp, const int *__restrict__ degen,
            int P, int per, int n_items, unsigned long long *__restrict__ keys, float *__restrict__ peaks_all,
            const int *__restrict__ cand, int kc) {
    extern __shared__ float4 smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    float2 *buf = sm.buf;
    const int tid = threadIdx.x, lane = tid & 31;
    const int c = (int)cluster_rank(), cid = blockIdx.x / NC, ncl = gridDim.x / NC;
    const int n = cand ? kc : T;
    for (int i = tid; i < 256; i += NT) {
        const int e = ((i >> 4) * (i & 15)) & 255, r = e & 127;
        const float2 w = make_float2(kTwTable<N>.re[r], kTwTable<N>.im[r]);
        sm.tw[i] = e & 128 ? make_float2(-w.x, -w.y) : w;
    }
    // passes 1 and 2: column q = 64 c + ql, l or k2 = a8 + 8 h
    const int ql = tid & 63, a8 = tid >> 6, q = OWN * c + ql;
    const bool packed = q == 0;
    // passes 3 and 4: line 64 c + lr + 32 h, g or k3 = b
    const int lr = tid >> 4, b = tid & 15;
    const uint32_t base0 = map_to_rank(buf, 0), base1 = map_to_rank(buf, 1);
    const uint32_t top0 = map_to_rank(&sm.top[c], 0);
    __syncthreads();

    auto template_of = [&](int p, int j) { return cand ? cand[(size_t)p * kc + j] : j; };
    // this CTA's half of a template into L2 ahead of the pass that reads it
    auto prefetch = [&](int t) {
        if (tid == 0 && t >= 0) {
            const char *s = reinterpret_cast<const char *>(St + (size_t)t * N * HW) + (size_t)c * (N * HW * sizeof(float2) / NC);
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(s), "r"((uint32_t)(N * HW * sizeof(float2) / NC)) : "memory");
        }
    };
    for (int item = cid; item < n_items; item += ncl) {
        // part by part: the clusters that run together read the same templates
        const int part = item / P, p = item - part * P, jb = part * per, je = min(n, jb + per);
        if (degen[p]) continue;   // uniform over the cluster, as every bound below
        const float2 *sp = Sp + (size_t)p * N * HW;
        float2 s0 = make_float2(0.f, 0.f), sh = s0;   // the pattern's columns 0 and 128 at row tid
        if (c == 0 && tid < N) {
            s0 = __ldg(sp + tid * HW);
            sh = __ldg(sp + tid * HW + 128);
        }
        auto make_p0 = [&](int t) {
            if (c == 0 && tid < N) {
                const float2 *tp = St + (size_t)t * N * HW + tid * HW;
                const float2 a = c_mulcj(__ldg(tp), s0), h = c_mulcj(__ldg(tp + 128), sh);
                sm.p0[tid] = make_float2(a.x - h.y, a.y + h.x);
            }
        };
        auto next_used = [&](int j) {
            while (j < je && template_of(p, j) < 0) {
                if (ALL && c == 0 && tid == 0) peaks_all[(size_t)p * n + j] = -INFINITY;
                ++j;
            }
            return j;
        };
        float best_v = -INFINITY;
        int best_t = -1;
        int j = next_used(jb);
        if (j < je) make_p0(template_of(p, j));
        __syncthreads();
        while (j < je) {
            const int t = template_of(p, j), jn = next_used(j + 1), tn = jn < je ? template_of(p, jn) : -1;
            prefetch(tn);
            const float2 *tp = St + (size_t)t * N * HW;
            // ---- 1
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int l = a8 + 8 * h;
                float2 x[16], s[16];
#pragma unroll
                for (int m = 0; m < 16; ++m) {
                    x[m] = __ldg(tp + (l + 16 * m) * HW + q);
                    s[m] = __ldg(sp + (l + 16 * m) * HW + q);
                }
#pragma unroll
                for (int m = 0; m < 16; ++m) x[m] = c_mulcj(x[m], s[m]);
                if (packed) {
#pragma unroll
                    for (int m = 0; m < 16; ++m) x[m] = sm.p0[l + 16 * m];
                }
                fft_reg_dif<16, +1>(x);
                float2 *dst = buf + (16 * a8) * 128 + 64 * h + ql;   // line k2 + 16 (l mod 8), the column or its mirror
                const float4 *w4 = reinterpret_cast<const float4 *>(sm.tw + l * 16);
                StaticFor<0, 8>::run([&](auto kk) {
                    constexpr int k2 = 2 * decltype(kk)::value, R0 = cx_bitrev(k2, 4), R1 = cx_bitrev(k2 + 1, 4);
                    const float4 w = w4[k2 >> 1];
                    dst[k2 * 128] = k2 ? c_mul(x[R0], make_float2(w.x, w.y)) : x[R0];
                    dst[(k2 + 1) * 128] = c_mul(x[R1], make_float2(w.z, w.w));
                });
            }
            __syncthreads();
            // ---- 2
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 *col = buf + (a8 + 8 * h) * 128 + ql;   // k2 = a8 + 8 h
                float2 x[16];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    x[i] = col[2048 * i];
                    x[8 + i] = col[2048 * i + 64];
                }
                fft_reg_dif<16, +1>(x);
                StaticFor<0, 8>::run([&](auto ii) {
                    constexpr int i = decltype(ii)::value;
                    const float2 ra = x[cx_bitrev(i, 4)], rb = x[cx_bitrev(i + 8, 4)];
                    float2 z = make_float2(ra.x - rb.y, ra.y + rb.x), zm = make_float2(ra.x + rb.y, rb.x - ra.y);
                    if (packed) {
                        z = make_float2(ra.x, rb.x);
                        zm = make_float2(ra.y, rb.y);
                    }
                    col[2048 * i] = z;
                    col[2048 * i + 64] = zm;
                });
            }
            cluster_arrive_shared();
            cluster_wait();   // both CTAs' columns are complete
            // ---- 3
            float2 z[2][16];
            if (c == 0) gather<0>(z, buf, base0, base1, OWN * c + lr, b);
            else gather<1>(z, buf, base0, base1, OWN * c + lr, b);
#pragma unroll
            for (int h = 0; h < 2; ++h) fft_reg_dif<16, +1>(z[h]);
            cluster_arrive();   // releases this thread's gathers
            cluster_wait();     // every thread of both CTAs has its values: the buffer takes the lines
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 *dst = buf + (lr + 32 * h) * 256 + (b & 1);
                const int g2 = b >> 1;
                StaticFor<0, 16>::run([&](auto kk) {
                    constexpr int k3 = decltype(kk)::value, R = cx_bitrev(k3, 4);
                    dst[16 * k3 + ((g2 ^ (k3 & 7)) << 1)] = k3 ? c_mul(z[h][R], sm.tw[k3 * 16 + b]) : z[h][R];
                });
            }
            __syncthreads();
            // ---- 4; the next template's packed column meanwhile
            if (tn >= 0) make_p0(tn);
            float m = -INFINITY;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 *src = reinterpret_cast<const float4 *>(buf + (lr + 32 * h) * 256 + 16 * b);
                float2 x[16];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 v = src[i ^ (b & 7)];
                    x[2 * i] = make_float2(v.x, v.y);
                    x[2 * i + 1] = make_float2(v.z, v.w);
                }
                dif16_head(x);
                // the last stage folded into the maximum: max(a + b, a - b) = a + |b|
#pragma unroll
                for (int i = 0; i < 16; i += 2)
                    m = fmaxf(m, fmaxf(x[i].x + fabsf(x[i + 1].x), x[i].y + fabsf(x[i + 1].y)));
            }
            if (m > best_v || (m == best_v && t < best_t)) {
                best_v = m;
                best_t = t;
            }
            if (ALL) {
#pragma unroll
                for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (lane == 0) sm.red[tid >> 5] = m;
            }
            __syncthreads();   // the lines have been read; the next packed column is in place
            if (ALL) {
                if (tid == 0) {
                    for (int w = 1; w < NT / 32; ++w) m = fmaxf(m, sm.red[w]);
                    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(top0), "f"(m) : "memory");
                }
                cluster_arrive();
                cluster_wait();
                if (c == 0 && tid == 0) peaks_all[(size_t)p * n + j] = fmaxf(sm.top[0], sm.top[1]);
            }
            j = jn;
        }
        unsigned long long key = best_t >= 0 ? pack_key(best_v, best_t) : 0ull;
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long k = __shfl_xor_sync(0xffffffffu, key, o);
            key = k > key ? k : key;
        }
        if (lane == 0 && key) atomicMax(keys + p, key);
    }
    cluster_arrive();   // no CTA leaves while the other may still read its shared memory
    cluster_wait();
}

}  // namespace

cudaError_t launch_search_c256(const float2 *St, int T, const float2 *Sp, const int *degen, int P,
                               unsigned long long *keys, float *peaks_all, const int *cand, int kc,
                               cudaStream_t st) {
    const int n = cand ? kc : T;
    if (P <= 0 || n <= 0) return cudaSuccess;
    auto *kern = peaks_all ? k_search256<true> : k_search256<false>;
    static std::atomic<int> resident[2] = {{0}, {0}};
    int ncl_max = 0;
    const cudaError_t e = resident_clusters(kern, NC, NT, sizeof(Smem), resident[peaks_all ? 1 : 0], &ncl_max);
    if (e != cudaSuccess) return e;
    // each pattern's templates in c parts, c minimising rounds of items over the resident
    // clusters x time of an item (a part starts with the pattern's columns 0 and 128 and
    // ends with a reduction: half a template's time).  Items go part by part: pattern by
    // pattern, the running clusters spread over the library and miss L2 (300 x 1,018:
    // 40.2 ms, part by part 38.9, whole items 39.7).  Against about four items per cluster
    // whatever the remainder, 2,000 templates: 10 patterns 3.25 -> 2.61 ms, 77: 24.6 ->
    // 19.9, 500: 136 -> 128; 32 candidates of 77 patterns 432 -> 402 us, of 1,000 4.65 ->
    // 4.49 ms (each side before the release after the gathers, 1 to 2 % on top).
    int nchunks = 1;
    long least = -1;
    const int most = (int)std::min<long>(n, std::max<long>(64, 4L * ncl_max / P));
    for (int c = 1; c <= most; ++c) {
        const int len = (n + c - 1) / c;
        const long rounds = ((long)P * ((n + len - 1) / len) + ncl_max - 1) / ncl_max, cost = rounds * (2L * len + 1);
        if (least < 0 || cost <= least) {
            least = cost;
            nchunks = c;
        }
    }
    const int per = (n + nchunks - 1) / nchunks;
    nchunks = (n + per - 1) / per;
    const long n_items = (long)P * nchunks;
    if (n_items > (1L << 30)) return cudaErrorInvalidValue;
    return launch_clusters(kern, NC, NT, sizeof(Smem), n_items < ncl_max ? n_items : ncl_max, st, St, T, Sp, degen,
                           P, per, (int)n_items, keys, peaks_all, cand, kc);
}
