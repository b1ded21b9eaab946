// Small DFTs in registers, V[p] = sum_q v[q] e^{SIGN 2 pi i p q / R}, used by the
// mixed-radix kernels.
#pragma once
#include "common.cuh"

namespace dft {

// radix 5 from the sums and differences of the conjugate-symmetric pairs
// (v1, v4) and (v2, v3): V_1,4 = v0 + c1 t1 + c2 t2 +- i SIGN (s1 t3 + s2 t4),
// V_2,3 = v0 + c2 t1 + c1 t2 +- i SIGN (s2 t3 - s1 t4)
template <int SIGN>
__device__ __forceinline__ void dft5(float2 &v0, float2 &v1, float2 &v2, float2 &v3, float2 &v4) {
    constexpr float c1 = Tw<1, 5, +1>::re, s1 = Tw<1, 5, +1>::im;
    constexpr float c2 = Tw<2, 5, +1>::re, s2 = Tw<2, 5, +1>::im;
    const float2 t1 = c_add(v1, v4), t2 = c_add(v2, v3);
    const float2 t3 = c_sub(v1, v4), t4 = c_sub(v2, v3);
    const float2 a1 = make_float2(fmaf(c1, t1.x, fmaf(c2, t2.x, v0.x)), fmaf(c1, t1.y, fmaf(c2, t2.y, v0.y)));
    const float2 a2 = make_float2(fmaf(c2, t1.x, fmaf(c1, t2.x, v0.x)), fmaf(c2, t1.y, fmaf(c1, t2.y, v0.y)));
    float2 b1 = make_float2(fmaf(s1, t3.x, s2 * t4.x), fmaf(s1, t3.y, s2 * t4.y));
    float2 b2 = make_float2(fmaf(s2, t3.x, -s1 * t4.x), fmaf(s2, t3.y, -s1 * t4.y));
    // i SIGN b
    b1 = SIGN > 0 ? c_mul_pi(b1) : c_mul_mi(b1);
    b2 = SIGN > 0 ? c_mul_pi(b2) : c_mul_mi(b2);
    v0 = c_add(v0, c_add(t1, t2));
    v1 = c_add(a1, b1);
    v4 = c_sub(a1, b1);
    v2 = c_add(a2, b2);
    v3 = c_sub(a2, b2);
}

// inverse transforms of R = 10, 16 and 20 points; output k is left at x[at<R>(k)].
// R = Q x 5: n = Q n1 + n2, k = k1 + 5 k2, X[k] at Q k1 + k2
template <int R>
__host__ __device__ constexpr int at(int k) {
    return R == 16 ? cx_bitrev(k, 4) : R / 5 * (k % 5) + k / 5;
}
template <int R>
__device__ __forceinline__ void inverse(float2 (&x)[R]) {
    if constexpr (R == 16) {
        fft_reg_dif<16, +1>(x);
    } else {
        constexpr int Q = R / 5;
        static_assert(R == 10 || R == 20, "10, 16 or 20 points");
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) dft5<+1>(x[n2], x[Q + n2], x[2 * Q + n2], x[3 * Q + n2], x[4 * Q + n2]);
        StaticFor<0, 5>::run([&](auto kk) {
            constexpr int k1 = decltype(kk)::value;
            StaticFor<1, Q>::run([&](auto nn) {
                constexpr int n2 = decltype(nn)::value;
                x[Q * k1 + n2] = tw_mul<k1 * n2, R, +1>(x[Q * k1 + n2]);
            });
            float2 *y = x + Q * k1;
            if constexpr (Q == 2) {
                const float2 a = y[0], b = y[1];
                y[0] = c_add(a, b);
                y[1] = c_sub(a, b);
            } else {
                const float2 s = c_add(y[0], y[2]), t = c_sub(y[0], y[2]), u = c_add(y[1], y[3]),
                             v = c_mul_pi(c_sub(y[1], y[3]));
                y[0] = c_add(s, u);
                y[1] = c_add(t, v);
                y[2] = c_sub(s, u);
                y[3] = c_sub(t, v);
            }
        });
    }
}

}  // namespace dft
