// Gnomonic reprojection of the master pattern, shared by the projection
// kernel and the pre-processing kernels that project their input images
// themselves (the same arithmetic: the same pixel values either way).
//
// Paper: "SO(3) Library Generation" (a template is the master pattern seen
// through the detector at an orientation and pattern centre).
#pragma once
#include "common.cuh"
#include "kernels.cuh"

namespace proj {

// ------------------------------------------------------ Lambert lookup
// Keys' cubic convolution weight, a = -1/2
__device__ __forceinline__ float keys_weight(float t) {
    t = fabsf(t);
    if (t <= 1.f) return (1.5f * t - 2.5f) * t * t + 1.f;
    if (t < 2.f) return ((-0.5f * t + 2.5f) * t - 4.f) * t + 2.f;
    return 0.f;
}

// num / den and num / sqrt(x) from the hardware approximations of 1 / den and
// 1 / sqrt(x) (1 ulp, 2^-22.9) and one Newton-Raphson step with the residual by FMA
// (the quotient's is Markstein's, IBM J. Res. Dev. 34, 1990), without the range
// handling of the IEEE operations.  For the normal values they get here the quotient is
// within 0.51 ulp (0.500 measured); the other rounds the product, the residual's x r and
// the sum once each, a relative error of at most 2.5 x 2^-24 (2.45 measured)
__device__ __forceinline__ float recip_times(float num, float den) {   // num / den
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(den));
    const float q = num * r;
    return fmaf(fmaf(-q, den, num), r, q);
}
__device__ __forceinline__ float rsqrt_times(float num, float x) {   // num / sqrt(x)
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    const float w = num * r;
    return fmaf(w, fmaf(-(x * r), 0.5f * r, 0.5f), w);
}
// arctangent on [-1, 1]: x + x s Q(s), s = x^2, Q the minimax fit (Remez
// exchange, relative error 2.4e-9 before rounding; 0.93 ulp in FP32 steps, over every float)
__device__ __forceinline__ float atan_unit(float x) {
    const float s = x * x;
    float q = -0.0017539305845275521f;
    q = fmaf(q, s, 0.010726945474743843f);
    q = fmaf(q, s, -0.030804598703980446f);
    q = fmaf(q, s, 0.05755210295319557f);
    q = fmaf(q, s, -0.0837731584906578f);
    q = fmaf(q, s, 0.1094203069806099f);
    q = fmaf(q, s, -0.142619326710701f);
    q = fmaf(q, s, 0.1999826580286026f);
    q = fmaf(q, s, -0.3333328366279602f);
    return fmaf(x * s, q, x);
}

// Rosca equal-area square of a hemisphere, then bilinear (interp 0) or
// bicubic (interp 1, Keys) interpolation of the M x M grid of cell centres,
// clamped at the edges.
//
// Four scattered 4-byte loads per pixel are bound by the L1's tag lookups: 7.65
// ps per pixel at 128 x 128 (4,000 projections) against 3.31 for the arithmetic
// alone.  With the master kept as 2 x 2 cells (quad, 16 bytes per cell) one
// load brings the pixel's four values from one sector: 3.98 ps.  (Learned form
// on 2,000 patterns 9.96 -> 8.95 ms, refinement of 1,999 3.71 -> 3.40 ms, the
// 4,065-template library 1.83 -> 1.67 ms, all at 128 x 128.)
//
// The map itself is one branch-free sequence.  With w = sqrt((x^2 + y^2) / (1 + |z|))
// = sqrt(1 - |z|) (free of cancellation) and den the larger of |x|, |y|, the
// square's coordinates in units of half its side are w sign(larger component)
// along that component's axis and w (4 / pi) atan(other / den) along the other.
// QUAD (compile time, so that no branch keeps one pixel's load from being issued
// beside another's arithmetic): bilinear from the 2 x 2 cells; else as interp says.
template <bool QUAD>
__device__ __forceinline__ float master_lookup(const float *__restrict__ master, int M, float x, float y,
                                               float z, int interp, const float4 *__restrict__ quad) {
    const float s2 = fmaf(x, x, y * y);
    const float c = 0.5f * M;
    float X = 0.f, Y = 0.f;   // from the square's centre, in cells
    if (s2 > 1e-30f) {        // below: the pole itself, to rounding (selects, not a branch)
        const float w = c * rsqrt_times(s2, s2 * (1.f + fabsf(z)));
        const bool xmaj = fabsf(y) <= fabsf(x);
        const float num = xmaj ? y : x, den = xmaj ? x : y;
        const float u = copysignf(w, den);
        const float t = w * (1.2732395447351627f * atan_unit(recip_times(num, fabsf(den))));
        X = xmaj ? u : t;
        Y = xmaj ? t : u;
    }
    const float fx = fminf(fmaxf(X + (c - 0.5f), 0.f), (float)(M - 1));
    const float fy = fminf(fmaxf(Y + (c - 0.5f), 0.f), (float)(M - 1));
    if (!QUAD && interp == 1) {
        const float *g = master + (z >= 0.f ? 0 : (size_t)M * M);
        const int i0 = (int)floorf(fx), j0 = (int)floorf(fy);
        float s = 0.f;
#pragma unroll
        for (int dj = -1; dj <= 2; ++dj) {
            const int j = min(max(j0 + dj, 0), M - 1);
            const float wy = keys_weight(fy - (float)(j0 + dj));
            float row = 0.f;
#pragma unroll
            for (int di = -1; di <= 2; ++di) {
                const int i = min(max(i0 + di, 0), M - 1);
                row = fmaf(keys_weight(fx - (float)(i0 + di)), __ldg(g + (size_t)j * M + i), row);
            }
            s = fmaf(wy, row, s);
        }
        return s;
    }
    // the cell's corner: f - 1/2 rounded to a whole number by adding 1.5 2^23 (a
    // coordinate on a cell boundary may take either cell: the weights 0 and 1
    // then pick the same value), at most M - 2
    const float big = 12582912.f, top = (float)(M - 2);
    const float kx = fminf(fx - 0.5f, top) + big, ky = fminf(fy - 0.5f, top) + big;
    const int i0 = __float_as_int(kx) - 0x4B400000, j0 = __float_as_int(ky) - 0x4B400000;
    const float tx = fx - (kx - big), ty = fy - (ky - big);
    const ptrdiff_t o = (z >= 0.f ? 0 : (ptrdiff_t)M * M) + ((ptrdiff_t)j0 * M + i0);
    float4 v;   // (i0, j0), (i0 + 1, j0), (i0, j0 + 1), (i0 + 1, j0 + 1)
    if constexpr (QUAD) {
        v = __ldg(quad + o);
    } else {
        const float *g = master + o;
        v = make_float4(__ldg(g), __ldg(g + 1), __ldg(g + M), __ldg(g + M + 1));
    }
    const float lo = fmaf(tx, v.y - v.x, v.x), hi = fmaf(tx, v.w - v.z, v.z);
    return fmaf(ty, hi - lo, lo);
}

// per-image frame: G = R(q) Rx(alpha) (detector direction -> crystal
// direction) and the pattern centre in pixels, in FP32 (FP64 here stalled
// the block on GB300's narrow FP64 pipe)
struct Frame {
    float G[9];
    float pc[3];
};
__device__ __forceinline__ void frame(const double *__restrict__ q4, const double *__restrict__ pc3,
                                      const ProjArgs &a, Frame &f) {
    float w = (float)q4[0], x = (float)q4[1], y = (float)q4[2], z = (float)q4[3];
    const float inv = rsqrtf(w * w + x * x + y * y + z * z);
    w *= inv; x *= inv; y *= inv; z *= inv;
    float R[9];
    R[0] = 1 - 2 * (y * y + z * z); R[1] = 2 * (x * y - w * z); R[2] = 2 * (x * z + w * y);
    R[3] = 2 * (x * y + w * z); R[4] = 1 - 2 * (x * x + z * z); R[5] = 2 * (y * z - w * x);
    R[6] = 2 * (x * z - w * y); R[7] = 2 * (y * z + w * x); R[8] = 1 - 2 * (x * x + y * y);
    const float sa = (float)a.sa, ca = (float)a.ca;
    for (int i = 0; i < 3; ++i) {
        f.G[3 * i + 0] = R[3 * i + 0];
        f.G[3 * i + 1] = R[3 * i + 1] * ca + R[3 * i + 2] * sa;
        f.G[3 * i + 2] = -R[3 * i + 1] * sa + R[3 * i + 2] * ca;
    }
    double px = a.pcx, py = a.pcy, pz = a.pcz;
    if (pc3) { px = pc3[0]; py = pc3[1]; pz = pc3[2]; }
    f.pc[0] = (float)px * (float)a.W;
    f.pc[1] = (float)py * (float)a.H;
    f.pc[2] = (float)pz * (float)a.W;
}
// the part of a pixel's detector direction that depends on its column j alone
// (detector column ox + j): the x offset from the pattern centre and the
// rotated contributions of the x and z components, G[:, 0] dx + G[:, 2] dz
struct Col {
    float dx, bx, by, bz;
};
__device__ __forceinline__ Col column(const Frame &f, const ProjArgs &a, int j) {
    const float dx = (float)(a.ox + j) + 0.5f - f.pc[0], dz = f.pc[2];
    return Col{dx, fmaf(f.G[0], dx, f.G[2] * dz), fmaf(f.G[3], dx, f.G[5] * dz), fmaf(f.G[6], dx, f.G[8] * dz)};
}
// the template's value at pixel (i, c) of the output region (detector pixel
// (oy + i, ox + j) for the column c = column(f, a, j), centre of the pixel):
// the crystal direction G d / |d| (G is a rotation, so the direction is
// rotated first and normalised after) looked up in the master pattern
template <bool QUAD>
__device__ __forceinline__ float pixel(const Frame &f, const Col &c, const float *__restrict__ master, int M,
                                       const ProjArgs &a, int i) {
    const float dy = f.pc[1] - ((float)(a.oy + i) + 0.5f), dz = f.pc[2];
    const float inv = rsqrtf(fmaf(dy, dy, fmaf(c.dx, c.dx, dz * dz)));
    const float cx = fmaf(f.G[1], dy, c.bx) * inv;
    const float cy = fmaf(f.G[4], dy, c.by) * inv;
    const float cz = fmaf(f.G[7], dy, c.bz) * inv;
    return master_lookup<QUAD>(master, M, cx, cy, cz, a.interp, a.quad);
}
template <bool QUAD>
__device__ __forceinline__ float pixel(const Frame &f, const float *__restrict__ master, int M, const ProjArgs &a,
                                       int i, int j) {
    return pixel<QUAD>(f, column(f, a, j), master, M, a, i);
}

// whether a launch reads the cells
inline bool use_quad(const ProjArgs &a) { return a.quad && a.interp == 0; }

}  // namespace proj
