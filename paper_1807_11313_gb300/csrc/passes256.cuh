// 256 x 256 transforms on thread-block clusters of four CTAs, two clusters per four
// SMs: a real image or surface as 128 packed complex lines (rows y and y + 128 are
// one line of 256 values), its half spectrum as 128 complex columns (columns 0 and
// 128 packed in one).  CTA c holds the lines OWN c .. as [OWN][256] in the line
// passes and the columns OWN c .. as [128][2 OWN] (a column, its mirror) in the
// column passes, 64 KB either way, 32 values per thread; every pass is two 16-point
// transforms per thread (256 = 16 x 16).  Line passes: thread lr = tid / 16, b = tid
// mod 16 has the lines lr and lr + OWN / 2; a line's sixteen threads are one half of
// a warp.  Column passes: thread ql = tid mod OWN, a8 = tid / OWN has the column
// OWN c + ql and the rows (or classes) a8 and a8 + 8.
#pragma once
#include "cluster.cuh"
#include "common.cuh"

namespace p256 {

constexpr int N = 256, HW = 129, NC = 4, OWN = 128 / NC, NT = 8 * OWN, PER = OWN / 16;

// W256^(a b) at [a][b] of the twiddle table
__device__ __forceinline__ float2 twiddle(int i) {
    const int e = ((i >> 4) * (i & 15)) & 255, r = e & 127;
    const float2 w = make_float2(kTwTable<N>.re[r], kTwTable<N>.im[r]);
    return e & 128 ? make_float2(-w.x, -w.y) : w;
}

// z[k3] times W256^(+-g k3) to the line's positions (g, k3), and back as the 16 values over g of k3 = b
template <int SIGN>
__device__ __forceinline__ void line_store(const float2 (&z)[16], float2 *line, const float2 *tw, int b) {
    StaticFor<0, 16>::run([&](auto kk) {
        constexpr int k = decltype(kk)::value, R = cx_bitrev(k, 4);
        const float2 w = tw[k * 16 + b];
        line[16 * k + (((b >> 1) ^ (k & 7)) << 1) + (b & 1)] = k == 0 ? z[R] : SIGN > 0 ? c_mul(z[R], w) : c_mulcj(w, z[R]);
    });
}
__device__ __forceinline__ void line_load(float2 (&x)[16], const float2 *line, int b) {
    const float4 *src = reinterpret_cast<const float4 *>(line + 16 * b);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float4 v = src[i ^ (b & 7)];
        x[2 * i] = make_float2(v.x, v.y);
        x[2 * i + 1] = make_float2(v.z, v.w);
    }
}
// the 16 values over k of l to the column's positions, and the 16 over l of k2
template <int SIGN>
__device__ __forceinline__ void column_store(const float2 (&x)[16], float2 *buf, const float2 *tw, int ql, int a8, int h) {
    float2 *dst = buf + 16 * a8 * 2 * OWN + OWN * h + ql;
    const float4 *w4 = reinterpret_cast<const float4 *>(tw + (a8 + 8 * h) * 16);
    StaticFor<0, 8>::run([&](auto kk) {
        constexpr int k = 2 * decltype(kk)::value, R0 = cx_bitrev(k, 4), R1 = cx_bitrev(k + 1, 4);
        const float4 w = w4[k >> 1];
        const float2 w0 = make_float2(w.x, w.y), w1 = make_float2(w.z, w.w);
        dst[k * 2 * OWN] = k == 0 ? x[R0] : SIGN > 0 ? c_mul(x[R0], w0) : c_mulcj(w0, x[R0]);
        dst[(k + 1) * 2 * OWN] = SIGN > 0 ? c_mul(x[R1], w1) : c_mulcj(w1, x[R1]);
    });
}
__device__ __forceinline__ void column_load(float2 (&x)[16], const float2 *col) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        x[i] = col[32 * OWN * i];
        x[8 + i] = col[32 * OWN * i + OWN];
    }
}

// the column pass after column_store<+1>: rows y0 + 16 j of the column, paired into
// the packed lines' values at q and 256 - q
__device__ __forceinline__ void columns_to_lines(float2 *buf, int ql, int a8, bool packed) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float2 *col = buf + (a8 + 8 * h) * 2 * OWN + ql;
        float2 t[16];
        column_load(t, col);
        fft_reg_dif<16, +1>(t);
        StaticFor<0, 8>::run([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            const float2 ra = t[cx_bitrev(i, 4)], rb = t[cx_bitrev(i + 8, 4)];
            float2 w = make_float2(ra.x - rb.y, ra.y + rb.x), wm = make_float2(ra.x + rb.y, rb.x - ra.y);
            if (packed) {
                w = make_float2(ra.x, rb.x);
                wm = make_float2(ra.y, rb.y);
            }
            col[32 * OWN * i] = w;
            col[32 * OWN * i + OWN] = wm;
        });
    }
}
// values b + 16 i of the lines L and L + OWN / 2 from all CTAs (the mirror of column
// 256 - v beyond 128), transformed over i
__device__ __forceinline__ void gather_lines(float2 (&z)[2][16], const uint32_t (&base)[NC], int L, int b) {
    constexpr uint32_t F = (uint32_t)sizeof(float2);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t line = (uint32_t)((L + h * (OWN / 2)) * 2 * OWN) * F;
        StaticFor<0, 16>::run([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if constexpr (i < 8) {
                z[h][i] = ld_cluster(base[i / PER] + line + (b + 16 * (i % PER)) * F);
            } else {
                constexpr int j = 15 - i, j0 = i == 8 ? 0 : 16 - i;   // column 16 j + 16 - b, or 16 j0 (0: packed) at b = 0
                z[h][i] = ld_cluster((b ? base[j / PER] + (OWN + 16 * (j % PER) + 16 - b) * F
                                        : base[j0 / PER] + (OWN + 16 * (j0 % PER)) * F) + line);
            }
        });
        fft_reg_dif<16, +1>(z[h]);
    }
}

}  // namespace p256
