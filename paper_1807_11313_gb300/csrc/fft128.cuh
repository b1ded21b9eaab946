// Pieces of the 128 x 128 real-surface transforms shared by the
// pre-processing, the search and the single-surface peak: a real surface as 64
// complex lines (rows pr and pr + 64 packed), its half spectrum as 64 complex
// columns (columns 0 and 64, real before the column transforms, packed in
// one), 32 complex values per thread of a 256-thread unit.
//
// Column thread (y0, g): y0 = lane & 15, g = 2 warp + lane / 16.  It holds the
// columns +-g mod 32 up to 64 (g, 32 - g, 32 + g, 64 - g) of the rows y0 + 16 j;
// g = 0 holds the packed column, 16, 32 and 48.  All of g = 0 sits in the first
// half of warp 0, so that the other warps carry none of its selects.
#pragma once
#include "common.cuh"

namespace fft128 {

__device__ __forceinline__ float2 w128(int e) {   // e^{+2 pi i e / 128}, 0 <= e < 128
    const int r = e & 63;
    const float2 w = make_float2(kTwTable<128>.re[r], kTwTable<128>.im[r]);
    return e & 64 ? make_float2(-w.x, -w.y) : w;
}

// line layout [k1][pr][n0] of a 64 KB buffer (n0 pairs swizzled by pr so that
// 16-byte accesses of eight consecutive pr fill every bank)
__device__ __forceinline__ int a_at(int k1, int pr, int n0) {
    return (k1 << 8) + (pr << 2) + (n0 ^ (((pr >> 2) & 1) << 1));
}

// 4-point transform, SIGN -1 forward
template <int SIGN>
__device__ __forceinline__ void dft4(float2 &a, float2 &b, float2 &c, float2 &d) {
    const float2 s = c_add(a, c), t = c_sub(a, c), u = c_add(b, d);
    const float2 v = SIGN > 0 ? c_mul_pi(c_sub(b, d)) : c_mul_mi(c_sub(b, d));
    a = c_add(s, u);
    b = c_add(t, v);
    c = c_sub(s, u);
    d = c_sub(t, v);
}

// the k-th column of thread (y0, g), and its second residue mod 32
__device__ __forceinline__ int col_of(int g, int k) {
    return g ? (k == 0 ? g : k == 1 ? 32 - g : k == 2 ? 32 + g : 64 - g) : 16 * k;
}
__device__ __forceinline__ int residue_b(int g) { return g ? 32 - g : 16; }

// two rows ra, rb of the surface's column-transformed half spectrum at the
// thread's four columns -> the packed line Z = Ra + i Rb, Z[128 - v] = conj Ra +
// i conj Rb at the columns g + 32 k (A) and residue_b(g) + 32 k (B)
__device__ __forceinline__ void merge_rows(const float2 (&ra)[4], const float2 (&rb)[4], bool special, float2 (&A)[4],
                                           float2 (&B)[4]) {
    auto zv = [&](int k) { return make_float2(ra[k].x - rb[k].y, ra[k].y + rb[k].x); };
    auto zn = [&](int k) { return make_float2(ra[k].x + rb[k].y, rb[k].x - ra[k].y); };
    A[0] = zv(0), A[1] = zv(2), A[2] = zn(3), A[3] = zn(1);
    B[0] = zv(1), B[1] = zv(3), B[2] = zn(2), B[3] = zn(0);
    if (special) {   // (Ra[0], Ra[64]) and (Rb[0], Rb[64]) are packed; residue 16 pairs 16 with 112, 48 with 80
        A[0] = make_float2(ra[0].x, rb[0].x);
        A[2] = make_float2(ra[0].y, rb[0].y);
        A[3] = zn(2);
        B[2] = zn(3);
        B[3] = zn(1);
    }
}

// the reverse, without its factor 1/2: 2 Ra = Z[v] + conj Z[128 - v], 2 Rb =
// (Z[v] - conj Z[128 - v]) / i (the packed column comes out without the factor
// too, as the pair (2 Ra, 2 Rb) of its split does later)
__device__ __forceinline__ void split_rows(const float2 (&A)[4], const float2 (&B)[4], bool special, float2 (&ra)[4],
                                           float2 (&rb)[4]) {
    auto split = [&](float2 zv, float2 zn, int k) {
        ra[k] = make_float2(zv.x + zn.x, zv.y - zn.y);
        rb[k] = make_float2(zv.y + zn.y, zn.x - zv.x);
    };
    float2 n1 = A[3], n2 = B[2], n3 = A[2];   // mirrors of columns 32 - g, 32 + g, 64 - g
    if (special) {
        n1 = B[3];
        n2 = A[3];
        n3 = B[2];
    }
    split(A[0], B[3], 0);
    split(B[0], n1, 1);
    split(A[1], n2, 2);
    split(B[1], n3, 3);
    if (special) {
        ra[0] = make_float2(A[0].x, A[2].x);
        rb[0] = make_float2(A[0].y, A[2].y);
    }
}

}  // namespace fft128
