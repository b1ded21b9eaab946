// 256 x 256 pre-processing (Eq. 4 and the filtering / normalisation of the FFT
// section) on thread-block clusters: standardise, window, transform, band-pass,
// normalise; optionally the filtered image back in space.
//
// One image at a time as 128 packed complex lines (rows y and y + 128 are one
// line of 256 values), its half spectrum as 128 complex columns (columns 0 and
// 128, real after the line transforms, packed in one).  CTA c of the NC holds the
// lines OWN c .. in the line passes and the columns OWN c .. in the column passes,
// 32 values per thread in registers either way, and every pass is two 16-point
// transforms per thread (256 = 16 x 16):
//   A: line, g: pixels x = g + 16 i from memory, statistics over the cluster,
//      standardised and windowed, 16 points over i, twiddle W256^-(g k1);
//   B: line, k1: 16 points over g in place (the same half warp: no barrier);
//   C: column q, l: gathers the lines l + 16 m at q and 256 - q from all CTAs,
//      splits them into rows y and y + 128, 16 points over m, twiddle;
//   D: column, k2: 16 points over l: rows k2 + 16 j of the spectrum; band-pass,
//      energy over the cluster, scaled and stored straight from registers.
// The filtered image goes back the same way (k_search256.cu's passes) from the
// registers of D.
//
// What bounds it: latency.  Every image passes two FP64 statistics and four to six
// cluster barriers; issue is active 34 %, the LSU 35 to 40 %, DRAM 25 %.  Two
// clusters of four interleave on their SMs (1,000 images with the filtered image
// and without, five launches: 1.88 ms; one cluster of two CTAs of 512 threads:
// 1.93).  Against row spectra [64][129] per CTA gathered column by column, one
// cluster of four with 256 threads per SM: 0.75 -> 0.36 us per image over those
// five launches (3.73 -> 1.81 ms), 0.263 without and 0.422 with the filtered image.
// The barriers that publish a CTA's own values release its shared memory only: a full
// release at each waits for the previous image's stores on their way to memory (0.271
// us without the filtered image).  At 128 registers (two CTAs per SM) 364 bytes per
// thread spill.  Separate kernels with and without the way back: no difference.
#include "kernels.cuh"
#include "passes256.cuh"

namespace {

using namespace p256;

struct Smem {
    float2 buf[OWN * N];     // lines: [OWN][256]; columns: [128][2 OWN] (column, mirror)
    float2 tw[256];          // W256^(a b) at [a][b]
    float2 band[N];          // (expm1(-f^2 / 2 s_h^2), exp(-f^2 / 2 s_l^2)) of a frequency index
    float2 p0[N];            // CTA 0: the packed column
    float2 sum[2][NT / 32];  // the warps' sums of two successive images
    float energy[NT / 32];
    float win[N];
    float stat[4];           // mean, 1 / deviation, degenerate; scale
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(NT, 2)
k_prep256(const float *__restrict__ img, int P, PrepArgs a, float2 *__restrict__ spec, float *__restrict__ spatial,
          int *__restrict__ degen, const int *__restrict__ active) {
    extern __shared__ float4 smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    float2 *buf = sm.buf;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = (int)cluster_rank(), cid = blockIdx.x / NC, ncl = gridDim.x / NC;
    for (int i = tid; i < N; i += NT) {
        sm.tw[i] = twiddle(i);
        const float f = (float)(i < N / 2 ? i : i - N), f2 = f * f;
        sm.band[i] = make_float2(expm1f(-f2 * a.inv2shp), expf(-f2 * a.inv2slp));
        sm.win[i] = a.window ? 0.5f * (1.f - cospif(2.f * i / N)) : 1.f;
    }
    // passes A and B: lines OWN c + lr + h OWN / 2, g or k1 = b
    const int lr = tid >> 4, b = tid & 15;
    // passes C and D: column q, l or k2 = a8 + 8 h
    const int ql = tid & (OWN - 1), a8 = tid / OWN, q = OWN * c + ql;
    const bool packed = q == 0;
    uint32_t base[NC];
#pragma unroll
    for (int r = 0; r < NC; ++r) base[r] = map_to_rank(buf, r);
    constexpr uint32_t F = (uint32_t)sizeof(float2);
    const bool hint = ((reinterpret_cast<uintptr_t>(img) | ((uintptr_t)a.W * 4) | ((uintptr_t)a.ox * 4) |
                        ((uintptr_t)a.W * a.H * 4)) & 15) == 0;
    auto next_active = [&](int p) {   // uniform over the cluster
        while (p < P && active && !active[p]) p += ncl;
        return p;
    };
    cluster_arrive();   // every CTA runs (its shared memory may be written) and its tables are filled
    cluster_wait();

    int par = 0;
    for (int p = next_active(cid), pn; p < P; p = pn, par ^= 1) {
        pn = next_active(p + ncl);
        const float *src = img + (size_t)p * a.W * a.H + (size_t)a.oy * a.W + a.ox;
        float2 *out = spec + (size_t)p * N * HW;
        // ---- A: pixels and statistics: FP32 sums of x - x0 over a warp (x0 the crop's first
        // pixel: a constant crop has exactly zero variance), the 32 warps' sums in FP64
        float2 z[2][16];
        const float x0 = __ldg(src);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float *row = src + (size_t)(OWN * c + lr + h * (OWN / 2)) * a.W + b;
#pragma unroll
            for (int i = 0; i < 16; ++i) z[h][i] = make_float2(__ldg(row + 16 * i), __ldg(row + (size_t)128 * a.W + 16 * i));
        }
        if (hint && pn < P && tid < 2 * OWN) {   // the next image's rows of this CTA into L2
            const float *row = img + (size_t)pn * a.W * a.H + a.ox +
                               (size_t)(a.oy + OWN * c + (tid < OWN ? tid : 128 + tid - OWN)) * a.W;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row), "r"((uint32_t)(N * sizeof(float))) : "memory");
        }
        float s = 0.f, s2 = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float d0 = z[h][i].x - x0, d1 = z[h][i].y - x0;
                s += d0 + d1;
                s2 = fmaf(d0, d0, fmaf(d1, d1, s2));
            }
        s = warp_sum(s);
        s2 = warp_sum(s2);
        if (lane == 0) sm.sum[par][warp] = make_float2(s, s2);
        cluster_arrive_shared();
        cluster_wait();
        if (warp == 0) {   // lane: one of the cluster's 32 warps
            const float2 v = ld_cluster(map_to_rank(&sm.sum[par][lane & (NT / 32 - 1)], lane / (NT / 32)));
            const double m1 = warp_sum((double)v.x) / ((double)N * N), m2 = warp_sum((double)v.y) / ((double)N * N);
            if (lane == 0) {
                const double mean = x0 + m1, var = fmax(m2 - m1 * m1, 0.0), least = 1e-12 * (1.0 + fabs(mean));
                const bool none = !(var > least * least);
                sm.stat[0] = (float)mean;
                sm.stat[1] = none ? 0.f : inv_sqrt(var);
                sm.stat[2] = none ? 1.f : 0.f;
            }
        }
        __syncthreads();
        bool bad = sm.stat[2] != 0.f;
        float sc = 0.f;
        float2 x[2][16], ca = make_float2(0.f, 0.f), cb = ca;
        if (!bad) {
            const float m = sm.stat[0], inv = sm.stat[1];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int y = OWN * c + lr + h * (OWN / 2);
                const float w0 = sm.win[y] * inv, w1 = sm.win[y + 128] * inv;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float wx = sm.win[b + 16 * i];
                    z[h][i] = make_float2((z[h][i].x - m) * wx * w0, (z[h][i].y - m) * wx * w1);
                }
                float2 *line = buf + (lr + h * (OWN / 2)) * N;
                fft_reg_dif<16, -1>(z[h]);
                line_store<-1>(z[h], line, sm.tw, b);
                __syncwarp();
                // ---- B
                line_load(z[h], line, b);
                fft_reg_dif<16, -1>(z[h]);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 16; ++k) line[b + 16 * cx_bitrev(k, 4)] = z[h][k];
            }
            cluster_arrive_shared();
            cluster_wait();   // the lines are complete
            // ---- C
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int l = a8 + 8 * h;
                StaticFor<0, 8>::run([&](auto mm) {
                    constexpr int m = decltype(mm)::value;
                    const uint32_t at = base[m / PER] + (uint32_t)((l + 16 * (m % PER)) * N) * F;
                    const float2 u = ld_cluster(at + q * F), v = ld_cluster(at + (packed ? N / 2 : N - q) * F);
                    x[h][m] = make_float2(0.5f * (u.x + v.x), 0.5f * (u.y - v.y));
                    x[h][m + 8] = make_float2(0.5f * (u.y + v.y), 0.5f * (v.x - u.x));
                    if (packed) {
                        x[h][m] = make_float2(u.x, v.x);
                        x[h][m + 8] = make_float2(u.y, v.y);
                    }
                });
                fft_reg_dif<16, -1>(x[h]);
            }
            cluster_arrive();   // releases this thread's gathers
            cluster_wait();     // every thread of the cluster has its values: the buffer takes the columns
#pragma unroll
            for (int h = 0; h < 2; ++h) column_store<-1>(x[h], buf, sm.tw, ql, a8, h);
            __syncthreads();
            // ---- D
            float e = 0.f;
            const float2 fv = sm.band[q];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k2 = a8 + 8 * h;
                column_load(x[h], buf + k2 * 2 * OWN + ql);
                fft_reg_dif<16, -1>(x[h]);
                if (packed) {
#pragma unroll
                    for (int k = 0; k < 16; ++k) sm.p0[k2 + 16 * cx_bitrev(k, 4)] = x[h][k];
                } else {
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const float2 fu = sm.band[k2 + 16 * cx_bitrev(k, 4)];
                        const float f = -(fu.x + fv.x + fu.x * fv.x) * (fu.y * fv.y);
                        x[h][k] = make_float2(x[h][k].x * f, x[h][k].y * f);
                        e = fmaf(2.f, x[h][k].x * x[h][k].x + x[h][k].y * x[h][k].y, e);
                    }
                }
            }
            if (c == 0) {   // columns 0 and 128 of row tid from the packed one: P = A + i B, A and B Hermitian
                __syncthreads();
                if (tid < N) {
                    const float2 u = sm.p0[tid], v = sm.p0[(N - tid) & (N - 1)], fu = sm.band[tid], fh = sm.band[N / 2],
                                 f0 = sm.band[0];
                    const float ga = -(fu.x + f0.x + fu.x * f0.x) * (fu.y * f0.y),
                                gb = -(fu.x + fh.x + fu.x * fh.x) * (fu.y * fh.y);
                    ca = make_float2(0.5f * (u.x + v.x) * ga, 0.5f * (u.y - v.y) * ga);
                    cb = make_float2(0.5f * (u.y + v.y) * gb, 0.5f * (v.x - u.x) * gb);
                    e += ca.x * ca.x + ca.y * ca.y + (cb.x * cb.x + cb.y * cb.y);
                }
            }
            e = warp_sum(e);
            if (lane == 0) sm.energy[warp] = e;
            cluster_arrive_shared();
            cluster_wait();
            if (warp == 0) {
                const double energy =
                    warp_sum((double)ld_cluster_f(map_to_rank(&sm.energy[lane & (NT / 32 - 1)], lane / (NT / 32))));
                if (lane == 0) sm.stat[3] = energy > 0.0 ? inv_sqrt(energy) : 0.f;
            }
            __syncthreads();
            sc = sm.stat[3];
            bad = !(sc > 0.f);
        }
        if (tid == 0 && c == 0 && degen) degen[p] = bad ? 1 : 0;
        if (bad) {   // uniform over the cluster: the decisions used cluster-wide sums
            for (int i = tid; i < 2 * OWN * HW; i += NT) out[(size_t)2 * OWN * c * HW + i] = make_float2(0.f, 0.f);
            if (spatial)
                for (int i = tid; i < 2 * OWN * N; i += NT) spatial[(size_t)p * N * N + (size_t)2 * OWN * c * N + i] = 0.f;
            cluster_arrive();   // releases the reads of the warps' sums, as the arrivals after the gathers do otherwise
            cluster_wait();
            continue;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                x[h][k] = make_float2(x[h][k].x * sc, x[h][k].y * sc);
                if (!packed) out[(a8 + 8 * h + 16 * cx_bitrev(k, 4)) * HW + q] = x[h][k];
            }
        if (c == 0 && tid < N) {
            ca = make_float2(ca.x * sc, ca.y * sc);
            cb = make_float2(cb.x * sc, cb.y * sc);
            out[tid * HW] = ca;
            out[tid * HW + 128] = cb;
        }
        if (!spatial) continue;
        // ---- back: columns
        if (c == 0) {
            if (tid < N) sm.p0[tid] = make_float2(ca.x - cb.y, ca.y + cb.x);
            __syncthreads();
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float2 t[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) t[j] = x[h][cx_bitrev(j, 4)];
            if (packed) {
#pragma unroll
                for (int j = 0; j < 16; ++j) t[j] = sm.p0[a8 + 8 * h + 16 * j];
            }
            fft_reg_dif<16, +1>(t);
            column_store<+1>(t, buf, sm.tw, ql, a8, h);
        }
        __syncthreads();
        columns_to_lines(buf, ql, a8, packed);
        cluster_arrive_shared();
        cluster_wait();   // the columns are complete
        gather_lines(z, base, OWN * c + lr, b);
        cluster_arrive();   // releases this thread's gathers
        cluster_wait();     // the buffer takes the lines
        const float inv_n = 1.f / N;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float2 *line = buf + (lr + h * (OWN / 2)) * N;
            line_store<+1>(z[h], line, sm.tw, b);
            __syncwarp();
            line_load(z[h], line, b);
            fft_reg_dif<16, +1>(z[h]);
            float *o = spatial + (size_t)p * N * N + (size_t)(OWN * c + lr + h * (OWN / 2)) * N + b;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                o[16 * cx_bitrev(k, 4)] = z[h][k].x * inv_n;
                o[128 * N + 16 * cx_bitrev(k, 4)] = z[h][k].y * inv_n;
            }
        }
        __syncwarp();   // the half warp's lines have been read: the next image's go there
    }
    cluster_arrive();   // no CTA leaves while another may still use its shared memory
    cluster_wait();
}

}  // namespace

cudaError_t launch_prep_c256(const float *img, int P, const PrepArgs &a, float2 *spec, float *spatial, int *degen,
                             const int *active, cudaStream_t st) {
    if (P <= 0) return cudaSuccess;
    if (a.N != N) return cudaErrorInvalidValue;
    static std::atomic<int> resident{0};
    int most = 0;
    const cudaError_t e = resident_clusters(k_prep256, NC, NT, sizeof(Smem), resident, &most);
    if (e != cudaSuccess) return e;
    return launch_clusters(k_prep256, NC, NT, sizeof(Smem), P < most ? P : most, st, img, P, a, spec, spatial, degen, active);
}
