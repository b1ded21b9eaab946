// Pre-processing at N = 128: real images (read, or projected from the master)
// to unit-norm filtered half spectra, and optionally back to filtered images.
//
// Paper: FFT section (zero mean and unit deviation, window, Eq. 4 transform,
// band-pass, normalisation by the autocorrelation).
//
// What bounds it: the earlier kernel walked the image through about ten
// shared-memory passes (80 k warp instructions per image with its filtered
// image) and let all of its 512 threads evaluate the FP64 statistics, whose
// square roots and divisions kept GB300's narrow FP64 pipe busy for about half
// of the 55 k cycles an image took (952 us for 4,999 patterns with their
// filtered images; 337 us = 43 % of the measured copy rate now; 2,000 projected
// templates 0.54 -> 0.27 ms).  Here one thread does the FP64 work and
// the transform is three rounds in registers, 32 complex values per thread,
// with two shared-memory transposes of 64 KB between them (the inverse runs
// the same rounds backwards):
//   round 1: thread (pr, n0): image rows pr and pr + 64 as one complex line, a
//            32-point transform over n1 of its columns n0 + 4 n1, the twiddle
//            W128^(n0 k1);
//   round 2: thread (y0, g): the 4-point transforms over n0 that finish the
//            lines pr = y0 + 16 j at columns = +-g mod 32, split by Hermitian
//            symmetry into the two rows' half spectra at columns g, 32 - g,
//            32 + g and 64 - g, then the radix-8 over the eight rows
//            y0 + 16 j that starts the columns, the twiddle W128^(y0 m);
//   round 3: thread (column, m): two 16-point transforms over y0 give rows
//            u = m + 8 q of the spectrum; band-pass, energy.
// Columns 0 and 64 hold real sequences before the column transforms and share
// one complex column, split by symmetry after it.  g = 0 takes columns 0, 64,
// 32, 16 and 48 and sits in the first half of warp 0, so that no other warp
// carries its selects.  Every shared access of a warp is free of bank
// conflicts (the swizzles below).
#include "common.cuh"
#include "fft128.cuh"
#include "kernels.cuh"
#include "project.cuh"

namespace {

using namespace fft128;

constexpr int N = 128, HW = 65, NT = 256, CTAS = 2;

// where the images come from: memory, or projected while they are loaded (by
// the lookup's options, or bilinearly from the master's 2 x 2 cells)
enum Source { kRead, kProject, kProjectQuad };

struct Smem {
    float2 buf[N * N / 2];       // the image [128][128] floats; A[k1][pr][n0]; C[m][column][y0]
    float2 tw1[4 * 34];          // e^{+2 pi i n0 k1 / 128} at [n0][k1] (rows of 34: no conflicts between n0)
    float2 twc[8 * 16];          // e^{+2 pi i m y0 / 128} at [m][y0]
    float2 band[HW + 1];         // per frequency: expm1(-f^2 / 2 s_h^2), exp(-f^2 / 2 s_l^2)
    float2 c0[N];                // columns 0 and 64 of the spectrum, packed
    float win[N];
    float2 part[NT / 32];        // per-warp partial sums
    float stat[4];               // mean, 1 / deviation, ok | scale, ok
};

// image pixel (r, c) as a float of buf: 16-byte pieces swizzled by the row so
// that eight rows' same columns lie in different banks
__device__ __forceinline__ int img_at(int r, int c) { return (r << 7) + ((((c >> 2) ^ (r & 7)) << 2) | (c & 3)); }
// C: one line of 16 y0 per (m, column), its 16-byte pieces swizzled by the column
__device__ __forceinline__ int c_at(int m, int col, int y0) {
    return (((m << 6) + col) << 4) + ((((y0 >> 1) ^ (col & 7)) << 1) | (y0 & 1));
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <Source SRC>
__global__ void __launch_bounds__(NT, CTAS)
k_prep128(const float *__restrict__ img, int P, PrepArgs a, float2 *__restrict__ spec, float *__restrict__ spatial,
          int *__restrict__ degen, const int *__restrict__ active, ProjSrc ps) {
    constexpr bool PROJ = SRC != kRead;
    extern __shared__ float4 smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    __shared__ proj::Frame fr;
    float2 *buf = sm.buf;
    float *imgs = reinterpret_cast<float *>(buf);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < N; i += NT) {
        sm.win[i] = a.window ? 0.5f * (1.f - cospif(2.f * i / N)) : 1.f;
        sm.twc[i] = w128((i >> 4) * (i & 15));
        sm.tw1[(i >> 5) * 34 + (i & 31)] = w128((i >> 5) * (i & 31));
    }
    for (int i = tid; i < HW; i += NT) {
        const float f2 = (float)(i * i);
        sm.band[i] = make_float2(expm1f(-f2 * a.inv2shp), expf(-f2 * a.inv2slp));
    }
    // round identities
    const int pr = tid >> 2, n0 = tid & 3;                  // 1: row pair, column residue mod 4
    const int y0 = lane & 15, g = 2 * warp + (lane >> 4);   // 2: row residue mod 16, column residue +-g mod 32
    const int gb = residue_b(g);                            //    its second residue
    const bool special = warp == 0 && g == 0;
    const int col = tid & 63, mq = tid >> 6;                // 3: column, u residues mq and mq + 4 mod 8
    // 16-byte copies where every crop row and the output allow them
    const bool vec_in = !PROJ && ((a.W | a.ox) & 3) == 0 && (reinterpret_cast<uintptr_t>(img) & 15) == 0 &&
                        (((size_t)a.W * a.H) & 3) == 0;
    const bool vec_out = (reinterpret_cast<uintptr_t>(spatial) & 15) == 0;

    for (int p = blockIdx.x; p < P; p += gridDim.x) {
        if (active && !active[p]) continue;   // uniform over the CTA
        __syncthreads();                      // the tables; the previous image's reads of buf
        if constexpr (PROJ) {
            if (tid == 0) proj::frame(ps.quats + 4 * (size_t)p, ps.pcs ? ps.pcs + 3 * (size_t)p : nullptr, ps.a, fr);
            __syncthreads();
            const proj::Frame f = fr;   // in registers: the loop's stores could alias shared memory
            const int c = tid & 127;    // one column per thread: its part of the direction once
            const proj::Col pcol = proj::column(f, ps.a, a.ox + c);
#pragma unroll 4
            for (int r = tid >> 7; r < N; r += 2)
                imgs[img_at(r, c)] = proj::pixel<SRC == kProjectQuad>(f, pcol, ps.master, ps.M, ps.a, a.oy + r);
        } else {
            const float *src = img + (size_t)p * a.W * a.H + (size_t)a.oy * a.W + a.ox;
            if (vec_in) {
#pragma unroll
                for (int k = 0; k < N * N / 4 / NT; ++k) {
                    const int i = tid + k * NT, r = i >> 5, c = (i & 31) << 2;
                    cp_async16(imgs + img_at(r, c), src + (size_t)r * a.W + c);
                }
            } else {
#pragma unroll 8
                for (int k = 0; k < N * N / NT; ++k) {
                    const int i = tid + k * NT, r = i >> 7, c = i & 127;
                    cp_async4(imgs + img_at(r, c), src + (size_t)r * a.W + c);
                }
            }
            cp_async_wait();
        }
        __syncthreads();
        float2 z[32];   // rows pr and pr + 64 at columns n0 + 4 n1
        {
            // FP32 sums of (x - x0), x0 the crop's first pixel (a constant crop has exactly zero
            // variance, and the sums stay well conditioned), the warps' sums added in FP64
            const float x0 = imgs[0];
            float s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                z[k] = make_float2(imgs[img_at(pr, n0 + 4 * k)], imgs[img_at(pr + 64, n0 + 4 * k)]);
                const float d0 = z[k].x - x0, d1 = z[k].y - x0;
                s1 += d0 + d1;
                s2 = fmaf(d0, d0, fmaf(d1, d1, s2));
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            }
            if (lane == 0) sm.part[warp] = make_float2(s1, s2);
            __syncthreads();
            if (tid == 0) {
                double t1 = 0.0, t2 = 0.0;
#pragma unroll
                for (int w = 0; w < NT / 32; ++w) {
                    t1 += (double)sm.part[w].x;
                    t2 += (double)sm.part[w].y;
                }
                const double m1 = t1 * (1.0 / (N * N)), mean = x0 + m1, var = t2 * (1.0 / (N * N)) - m1 * m1;
                const double lim = 1e-12 * (1.0 + fabs(mean));
                const bool ok = var > 0.0 && var > lim * lim;   // deviation above lim
                sm.stat[0] = (float)mean;
                sm.stat[1] = ok ? (float)rsqrt(var) : 0.f;
                sm.stat[2] = ok ? 1.f : 0.f;
            }
            __syncthreads();
        }
        bool bad = !(sm.stat[2] > 0.f);
        if (!bad) {
            // ---- round 1
            {
                const float mean = sm.stat[0], inv = sm.stat[1], wa = sm.win[pr], wb = sm.win[pr + 64];
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    const float wc = sm.win[n0 + 4 * k] * inv;
                    z[k] = make_float2((z[k].x - mean) * wc * wa, (z[k].y - mean) * wc * wb);
                }
            }
            fft_reg_dif<32, -1>(z);
            {
                const float4 *t4 = reinterpret_cast<const float4 *>(sm.tw1 + n0 * 34);
                StaticFor<0, 16>::run([&](auto kk) {
                    constexpr int k1 = 2 * decltype(kk)::value, R0 = cx_bitrev(k1, 5), R1 = cx_bitrev(k1 + 1, 5);
                    const float4 w = t4[k1 >> 1];
                    buf[a_at(k1, pr, n0)] = k1 ? c_mulcj(make_float2(w.x, w.y), z[R0]) : z[R0];
                    buf[a_at(k1 + 1, pr, n0)] = c_mulcj(make_float2(w.z, w.w), z[R1]);
                });
            }
            __syncthreads();
            // ---- round 2
            float2 x[4][8];   // [column][row y0 + 16 j]
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int q = y0 + 16 * j;
                const float4 *pa = reinterpret_cast<const float4 *>(buf), *pb = pa;
                const float4 u0 = pa[a_at(g, q, 0) >> 1], u1 = pa[a_at(g, q, 2) >> 1];
                const float4 v0 = pb[a_at(gb, q, 0) >> 1], v1 = pb[a_at(gb, q, 2) >> 1];
                float2 A[4] = {{u0.x, u0.y}, {u0.z, u0.w}, {u1.x, u1.y}, {u1.z, u1.w}};
                float2 B[4] = {{v0.x, v0.y}, {v0.z, v0.w}, {v1.x, v1.y}, {v1.z, v1.w}};
                dft4<-1>(A[0], A[1], A[2], A[3]);   // Z at columns g + 32 k
                dft4<-1>(B[0], B[1], B[2], B[3]);   // Z at columns gb + 32 k
                float2 ra[4], rb[4];
                split_rows(A, B, special, ra, rb);
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k][j] = ra[k], x[k][j + 4] = rb[k];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) fft_reg_dif<8, -1>(x[k]);
            __syncthreads();   // every thread has read A
            StaticFor<0, 8>::run([&](auto mm) {
                constexpr int m = decltype(mm)::value, R = cx_bitrev(m, 3);
                const float2 w = sm.twc[m * 16 + y0];
#pragma unroll
                for (int k = 0; k < 4; ++k) buf[c_at(m, col_of(g, k), y0)] = m ? c_mulcj(w, x[k][R]) : x[k][R];
            });
            __syncthreads();
            // ---- round 3: rows u = mq + 4 h + 8 q of this thread's column
            float2 s[2][16];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 *line = reinterpret_cast<const float4 *>(buf + c_at(mq + 4 * h, col, 0) -
                                                                      ((col & 7) << 1));
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 v = line[i ^ (col & 7)];
                    s[h][2 * i] = make_float2(v.x, v.y);
                    s[h][2 * i + 1] = make_float2(v.z, v.w);
                }
                fft_reg_dif<16, -1>(s[h]);   // s[h][bitrev(q)] = S[mq + 4 h + 8 q]
                if (col == 0)
                    StaticFor<0, 16>::run([&](auto qq) {
                        constexpr int q = decltype(qq)::value;
                        sm.c0[mq + 4 * h + 8 * q] = s[h][cx_bitrev(q, 4)];
                    });
            }
            __syncthreads();
            // band-pass h = -(e_u + e_v + e_u e_v) b_u b_v (1 - exp(-(a + b)) from expm1 of a and b: free of
            // cancellation near DC) and the filtered energy; columns 1..63 stand for their mirror images too
            float e = 0.f;
            {
                const float2 bv = sm.band[col];
                const float ev1 = 1.f + bv.x;
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    StaticFor<0, 16>::run([&](auto qq) {
                        constexpr int q = decltype(qq)::value, R = cx_bitrev(q, 4);
                        const int u = mq + 4 * h + 8 * q;
                        const float2 bu = sm.band[q < 8 ? u : N - u];
                        const float f = -fmaf(bu.x, ev1, bv.x) * (bu.y * bv.y);
                        s[h][R] = make_float2(s[h][R].x * f, s[h][R].y * f);
                        e = fmaf(s[h][R].x, s[h][R].x, fmaf(s[h][R].y, s[h][R].y, e));
                    });
                e = col ? 2.f * e : 0.f;
            }
            float2 S0 = make_float2(0.f, 0.f), SH = S0;   // columns 0 and 64 at row u = tid
            if (tid < N) {
                const float2 zu = sm.c0[tid], zn = sm.c0[(N - tid) & (N - 1)];
                const float2 bu = sm.band[tid <= 64 ? tid : N - tid], bh = sm.band[64];
                const float f0 = -bu.x * bu.y, fh = -fmaf(bu.x, 1.f + bh.x, bh.x) * (bu.y * bh.y);
                S0 = make_float2(f0 * (zu.x + zn.x), f0 * (zu.y - zn.y));
                SH = make_float2(fh * (zu.y + zn.y), fh * (zn.x - zu.x));
                e += S0.x * S0.x + S0.y * S0.y + SH.x * SH.x + SH.y * SH.y;
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (lane == 0) sm.part[warp].x = e;
            __syncthreads();   // also: c0 has been read
            if (tid == 0) {
                double t = 0.0;
#pragma unroll
                for (int w = 0; w < NT / 32; ++w) t += (double)sm.part[w].x;
                sm.stat[0] = t > 0.0 ? (float)rsqrt(t) : 0.f;
                sm.stat[1] = t > 0.0 ? 1.f : 0.f;
            }
            if (spatial && tid < N) sm.c0[tid] = make_float2(S0.x - SH.y, S0.y + SH.x);   // packed again
            __syncthreads();
            bad = !(sm.stat[1] > 0.f);
            if (!bad) {
                const float sc = sm.stat[0];
                float2 *out = spec + (size_t)p * N * HW;
                if (tid < N) {
                    out[tid * HW] = make_float2(S0.x * sc, S0.y * sc);
                    out[tid * HW + 64] = make_float2(SH.x * sc, SH.y * sc);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    StaticFor<0, 16>::run([&](auto qq) {
                        constexpr int q = decltype(qq)::value, R = cx_bitrev(q, 4);
                        s[h][R] = make_float2(s[h][R].x * sc, s[h][R].y * sc);
                        if (col) out[(mq + 4 * h + 8 * q) * HW + col] = s[h][R];
                    });
                if (spatial) {
                    // ---- round 3 backwards: 16-point inverse over q, the twiddle W128^(m y0)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float2 t[16];
                        StaticFor<0, 16>::run([&](auto qq) {
                            constexpr int q = decltype(qq)::value;
                            t[q] = s[h][cx_bitrev(q, 4)];
                            if (col == 0) {
                                const float2 c = sm.c0[mq + 4 * h + 8 * q];
                                t[q] = make_float2(c.x * sc, c.y * sc);
                            }
                        });
                        fft_reg_dif<16, +1>(t);
                        const int m = mq + 4 * h;
                        const float4 *w4 = reinterpret_cast<const float4 *>(sm.twc + m * 16);
                        float4 *line = reinterpret_cast<float4 *>(buf + c_at(m, col, 0) - ((col & 7) << 1));
                        StaticFor<0, 8>::run([&](auto ii) {
                            constexpr int i = decltype(ii)::value;
                            const float4 w = w4[i];
                            const float2 r0 = c_mul(t[cx_bitrev(2 * i, 4)], make_float2(w.x, w.y));
                            const float2 r1 = c_mul(t[cx_bitrev(2 * i + 1, 4)], make_float2(w.z, w.w));
                            line[i ^ (col & 7)] = make_float4(r0.x, r0.y, r1.x, r1.y);
                        });
                    }
                    __syncthreads();
                    // ---- round 2 backwards: radix 8 over m, the rows paired again, 4-point inverse over columns
                    StaticFor<0, 8>::run([&](auto mm) {
                        constexpr int m = decltype(mm)::value;
#pragma unroll
                        for (int k = 0; k < 4; ++k) x[k][m] = buf[c_at(m, col_of(g, k), y0)];
                    });
#pragma unroll
                    for (int k = 0; k < 4; ++k) fft_reg_dif<8, +1>(x[k]);   // x[k][bitrev(j)] = row y0 + 16 j
                    __syncthreads();   // every thread has read C
                    StaticFor<0, 4>::run([&](auto jj) {
                        constexpr int j = decltype(jj)::value, RA = cx_bitrev(j, 3), RB = cx_bitrev(j + 4, 3);
                        const float2 ra[4] = {x[0][RA], x[1][RA], x[2][RA], x[3][RA]};
                        const float2 rb[4] = {x[0][RB], x[1][RB], x[2][RB], x[3][RB]};
                        float2 A[4], B[4];
                        merge_rows(ra, rb, special, A, B);
                        dft4<+1>(A[0], A[1], A[2], A[3]);
                        dft4<+1>(B[0], B[1], B[2], B[3]);
                        const int q = y0 + 16 * j;
                        float4 *d = reinterpret_cast<float4 *>(buf);
                        d[a_at(g, q, 0) >> 1] = make_float4(A[0].x, A[0].y, A[1].x, A[1].y);
                        d[a_at(g, q, 2) >> 1] = make_float4(A[2].x, A[2].y, A[3].x, A[3].y);
                        d[a_at(gb, q, 0) >> 1] = make_float4(B[0].x, B[0].y, B[1].x, B[1].y);
                        d[a_at(gb, q, 2) >> 1] = make_float4(B[2].x, B[2].y, B[3].x, B[3].y);
                    });
                    __syncthreads();
                    // ---- round 1 backwards
                    {
                        const float4 *t4 = reinterpret_cast<const float4 *>(sm.tw1 + n0 * 34);
#pragma unroll
                        for (int k1 = 0; k1 < 32; k1 += 2) {
                            const float4 w = t4[k1 >> 1];
                            z[k1] = c_mul(buf[a_at(k1, pr, n0)], make_float2(w.x, w.y));
                            z[k1 + 1] = c_mul(buf[a_at(k1 + 1, pr, n0)], make_float2(w.z, w.w));
                        }
                    }
                    fft_reg_dif<32, +1>(z);
                    __syncthreads();   // every thread has read A
                    StaticFor<0, 32>::run([&](auto kk) {
                        constexpr int k = decltype(kk)::value, R = cx_bitrev(k, 5);
                        imgs[img_at(pr, n0 + 4 * k)] = z[R].x * (1.f / N);
                        imgs[img_at(pr + 64, n0 + 4 * k)] = z[R].y * (1.f / N);
                    });
                    __syncthreads();
                    float *dst = spatial + (size_t)p * N * N;
                    if (vec_out) {
#pragma unroll
                        for (int k = 0; k < N * N / 4 / NT; ++k) {
                            const int i = tid + k * NT, r = i >> 5, c = (i & 31) << 2;
                            reinterpret_cast<float4 *>(dst)[i] = *reinterpret_cast<const float4 *>(imgs + img_at(r, c));
                        }
                    } else {
                        for (int i = tid; i < N * N; i += NT) dst[i] = imgs[img_at(i >> 7, i & 127)];
                    }
                }
            }
        }
        if (tid == 0 && degen) degen[p] = bad ? 1 : 0;
        if (bad) {
            for (int i = tid; i < N * HW; i += NT) spec[(size_t)p * N * HW + i] = make_float2(0.f, 0.f);
            if (spatial)
                for (int i = tid; i < N * N; i += NT) spatial[(size_t)p * N * N + i] = 0.f;
        }
    }
}

template <Source SRC>
cudaError_t launch(const float *img, int P, const PrepArgs &a, float2 *spec, float *spatial, int *degen,
                   const int *active, const ProjSrc &src, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_prep128<SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(Smem));
    int dev = 0, num_sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int grid = P < CTAS * num_sms ? P : CTAS * num_sms;   // persistent: the tables once per CTA
    k_prep128<SRC><<<grid, NT, sizeof(Smem), st>>>(img, P, a, spec, spatial, degen, active, src);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_prep128(const float *img, int P, const PrepArgs &a, float2 *spec, float *spatial, int *degen,
                           const int *active, cudaStream_t st) {
    return launch<kRead>(img, P, a, spec, spatial, degen, active, ProjSrc{}, st);
}

cudaError_t launch_prep128_projected(const ProjSrc &src, int P, const PrepArgs &a, float2 *spec, float *spatial,
                                     int *degen, const int *active, cudaStream_t st) {
    return proj::use_quad(src.a) ? launch<kProjectQuad>(nullptr, P, a, spec, spatial, degen, active, src, st)
                                 : launch<kProject>(nullptr, P, a, spec, spatial, degen, active, src, st);
}
