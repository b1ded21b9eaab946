// FP32 convolutions of the proposal network: forward, gradient into the input
// and gradient into the weights of the 3 x 3 stride-2 layers (pad 1), as tiled
// matrix products that gather their operands from the activations.
//
// Network (see k_cnn.cu): channels 1 -> 32 -> 64 -> 64 -> 128 -> 128 on sides
// 128 -> 64 -> 32 -> 16 -> 8 -> 4.
//
// What bounds them: FP32 FMAs, once the gathers are cheap.  The products they
// replace (64 x 64 tiles, 4 x 4 outputs per thread, divisions per gathered
// element) ran at 8 % of the FP32 peak over a training step of 256 patterns:
// 8.48 ms, now 2.25 (forward layers 123 / 400 / 217 / 116 / 142 -> 37 / 213 /
// 132 / 80 / 86 us, input gradients 2,810 / 894 / 613 / 382 -> 309 / 170 / 83 /
// 58, weight gradients 517 / 740 / 336 / 171 / 81 -> 179 / 338 / 161 / 83 / 39).
//   * Tiles of 64 (or 32) x 128 (or 64) outputs, 8 x 8 (4 x 8, 8 x 4) per
//     thread, 16 deep, the next slice's elements fetched into registers while
//     the current one is multiplied (one barrier per slice).
//   * A thread gathers for one output position: its address and its border
//     bits are computed once, and each tap costs one table entry (offset and
//     border bits) shared by the whole warp.
//   * The input gradient runs by output parity: an input row 2 i meets the tap
//     ky = 1 alone, a row 2 i + 1 the taps 0 and 2 (likewise the columns), so
//     the four parity classes have 4, 2, 2 and 1 of the 9 taps and none of the
//     products with zeros that a gather over all nine spends 3/4 of its time on.
//   * Every sum runs over its terms in ascending order (input channel, tap),
//     so the forward pass and the input gradient keep their values bit for bit
//     (a skipped term was an exact zero).
//   * The weight gradient splits the sum over positions; the partials are
//     summed in a fixed order, so training is reproducible.  The bias gradient
//     (the row sums of its first operand) comes from the same pass.
#include "common.cuh"
#include "kernels.cuh"

namespace {

constexpr int BK = 16, NT = 128;

// thread layout of a BM x BN tile: BM / TM row groups x 16 column groups; a
// thread's TN columns in runs of 4, 64 apart
template <int BM, int BN>
struct Tile {
    static constexpr int TM = BM / (NT / 16), TN = BN / 16;
    static constexpr int LA = BM + 4, LB = BN + 4;   // row strides in shared memory (16-byte rows)
    float a[2][BK][LA], b[2][BK][LB];
};

template <int BM, int BN>
__device__ __forceinline__ void multiply(const Tile<BM, BN> &t, int s, float (&acc)[Tile<BM, BN>::TM][Tile<BM, BN>::TN]) {
    constexpr int TM = Tile<BM, BN>::TM, TN = Tile<BM, BN>::TN;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int k = 0; k < BK; ++k) {
        float a[TM], b[TN];
#pragma unroll
        for (int i = 0; i < TM; i += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(&t.a[s][k][ty * TM + i]);
            a[i] = v.x, a[i + 1] = v.y, a[i + 2] = v.z, a[i + 3] = v.w;
        }
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(&t.b[s][k][tx * 4 + 16 * j]);
            b[j] = v.x, b[j + 1] = v.y, b[j + 2] = v.z, b[j + 3] = v.w;
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
}

// ------------------------------------------------------------------ forward
// y[b][co][p] = relu(bias[co] + sum over (ci, ky, kx) of w[co][ci][ky][kx] x[b][ci][2 oy - 1 + ky][2 ox - 1 + kx])
template <int CI, int CO, int S, int BN>
__global__ void __launch_bounds__(NT) k_conv32_fwd(const float *__restrict__ x, const float *__restrict__ w,
                                                   const float *__restrict__ bias, int B, float *__restrict__ y) {
    constexpr int BM = 64, K = CI * 9, SO = S / 2, Q = SO * SO, PER = BK * BN / NT;
    constexpr int KSTEP = NT / BN;   // a thread gathers position tid % BN at depths tid / BN + KSTEP i
    static_assert(K % BK == 0 && CO % BM == 0, "whole slices and row tiles");
    __shared__ __align__(16) Tile<BM, BN> t;
    __shared__ int tap[K];   // (offset from the window's centre) * 4 + (ky == 0) * 2 + (kx == 0)
    const int tid = threadIdx.x;
    for (int k = tid; k < K; k += NT) {
        const int ci = k / 9, r = k - ci * 9, ky = r / 3, kx = r - ky * 3;
        tap[k] = (ci * S * S + (ky - 1) * S + (kx - 1)) * 4 + (ky == 0) * 2 + (kx == 0);
    }
    const int m0 = blockIdx.y * BM;
    const long n0 = (long)blockIdx.x * BN, N = (long)B * Q;
    const long n = n0 + tid % BN;
    const int kq = tid / BN;
    const bool in = n < N;
    const int p = (int)(n % Q), oy = p / SO, ox = p % SO;
    const float *src = x + (in ? (n / Q) * (long)CI * S * S + 2 * oy * S + 2 * ox : 0);
    const int border = in ? (oy == 0) * 2 + (ox == 0) : 3;
    const float *wrow = w + (long)(m0 + tid / 2) * K + (tid & 1) * 8;
    float4 wa, wb;
    float xb[PER];
    auto fetch = [&](int k0) {
        wa = *reinterpret_cast<const float4 *>(wrow + k0);
        wb = *reinterpret_cast<const float4 *>(wrow + k0 + 4);
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int e = tap[k0 + kq + KSTEP * i];
            xb[i] = in && !(e & border) ? src[e >> 2] : 0.f;
        }
    };
    auto put = [&](int s) {
        const float a[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) t.a[s][(tid & 1) * 8 + i][tid / 2] = a[i];
#pragma unroll
        for (int i = 0; i < PER; ++i) t.b[s][kq + KSTEP * i][tid % BN] = xb[i];
    };
    constexpr int TM = Tile<BM, BN>::TM, TN = Tile<BM, BN>::TN;
    float acc[TM][TN] = {};
    __syncthreads();   // the taps
    fetch(0);
    put(0);
    __syncthreads();
    for (int k0 = 0, s = 0; k0 < K; k0 += BK, s ^= 1) {
        if (k0 + BK < K) fetch(k0 + BK);
        multiply(t, s, acc);
        if (k0 + BK < K) put(s ^ 1);
        __syncthreads();
    }
    const int tx = tid & 15, ty = tid >> 4;
#pragma unroll
    for (int j = 0; j < TN; j += 4) {
        const long c = n0 + tx * 4 + 16 * j;   // four positions of one image (Q is a multiple of 16)
        if (c >= N) continue;
        float *dst = y + ((c / Q) * CO + m0 + ty * TM) * (long)Q + c % Q;
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const float bi = bias[m0 + ty * TM + i];
            *reinterpret_cast<float4 *>(dst + (long)i * Q) =
                make_float4(fmaxf(acc[i][j] + bi, 0.f), fmaxf(acc[i][j + 1] + bi, 0.f), fmaxf(acc[i][j + 2] + bi, 0.f),
                            fmaxf(acc[i][j + 3] + bi, 0.f));
        }
    }
}

// the first layer (one standardised input channel, 32 filters): one thread per
// output position, bound by the 128 MB it writes per 256 patterns
__global__ void __launch_bounds__(256) k_conv32_first(CnnInput in, const float2 *__restrict__ affine,
                                                      const float *__restrict__ w, const float *__restrict__ bias,
                                                      int B, float *__restrict__ y) {
    constexpr int S = 128, SO = 64, CO = 32, Q = SO * SO;
    __shared__ __align__(16) float ws[9 * CO];   // [tap][filter]
    __shared__ float bs[CO];
    for (int i = threadIdx.x; i < CO * 9; i += blockDim.x) ws[(i % 9) * CO + i / 9] = w[i];
    if (threadIdx.x < CO) bs[threadIdx.x] = bias[threadIdx.x];
    __syncthreads();
    const long n = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (long)B * Q) return;
    const int b = (int)(n / Q), p = (int)(n % Q), oy = p / SO, ox = p % SO;
    const float2 a = affine[b];
    const float *img = in.x + b * in.img_stride + (long)in.oy * in.row_stride + in.ox;
    float acc[CO] = {};
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const int iy = 2 * oy - 1 + r / 3, ix = 2 * ox - 1 + r % 3;
        const float v = iy >= 0 && ix >= 0 && iy < S && ix < S ? fmaf(img[(long)iy * in.row_stride + ix], a.x, a.y) : 0.f;
        const float4 *w4 = reinterpret_cast<const float4 *>(ws + r * CO);
#pragma unroll
        for (int c = 0; c < CO; c += 4) {
            const float4 q = w4[c / 4];
            acc[c] = fmaf(q.x, v, acc[c]);
            acc[c + 1] = fmaf(q.y, v, acc[c + 1]);
            acc[c + 2] = fmaf(q.z, v, acc[c + 2]);
            acc[c + 3] = fmaf(q.w, v, acc[c + 3]);
        }
    }
    float *dst = y + (long)b * CO * Q + p;
#pragma unroll
    for (int c = 0; c < CO; ++c) dst[(long)c * Q] = fmaxf(acc[c] + bs[c], 0.f);
}

// ------------------------------------------------- gradient into the input
// weights by parity class: class z = 2 (iy & 1) + (ix & 1) holds its taps t of
// every output channel, wt[class offset + (co ntaps + t)][ci]
__host__ __device__ constexpr int class_taps(int z) { return (z & 2 ? 2 : 1) * (z & 1 ? 2 : 1); }
__host__ __device__ constexpr int class_base(int z, int co) { return co * (z == 0 ? 0 : z == 1 ? 1 : z == 2 ? 3 : 5); }
// tap t of class z (ascending): the filter's row and column, and the output position's step from (iy / 2, ix / 2)
struct ClassTap {
    int r, dy, dx;
};
__device__ __forceinline__ ClassTap class_tap(int z, int t) {
    const int nx = z & 1 ? 2 : 1, ty = t / nx, tx = t - ty * nx;
    const int ky = z & 2 ? 2 * ty : 1, kx = z & 1 ? 2 * tx : 1;
    return {ky * 3 + kx, z & 2 ? 1 - ty : 0, z & 1 ? 1 - tx : 0};
}
__global__ void k_conv32_wt(const float *__restrict__ w, int CO, int CI, float *__restrict__ wt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= CO * CI * 9) return;
    const int row = i / CI, ci = i - row * CI;
    int z = 3;
    while (z > 0 && row < class_base(z, CO)) --z;
    const int k = row - class_base(z, CO), nt = class_taps(z), co = k / nt;
    wt[i] = w[((long)co * CI + ci) * 9 + class_tap(z, k - co * nt).r];
}

// gx[b][ci][iy][ix] = (a[b][ci][iy][ix] > 0) sum over (co, taps) of w g[b][co][oy][ox]
template <int CI, int CO, int SO, int BM, int BN>
__global__ void __launch_bounds__(NT) k_conv32_dx(const float *__restrict__ g, const float *__restrict__ wt,
                                                  const float *__restrict__ mask, int B, float *__restrict__ gx) {
    constexpr int Q = SO * SO, S = 2 * SO, PER = BK * BN / NT, KSTEP = NT / BN;
    static_assert(CO % BK == 0 && CI % BM == 0, "whole slices and row tiles");
    __shared__ __align__(16) Tile<BM, BN> t;
    __shared__ int tap[CO * 4];   // (offset) * 4 + dy * 2 + dx
    const int tid = threadIdx.x, z = 3 - blockIdx.z;   // the four-tap class first: the short ones fill its tail
    const int nt = class_taps(z), K = CO * nt, m0 = blockIdx.y * BM;
    for (int k = tid; k < K; k += NT) {
        const int co = k / nt;
        const ClassTap c = class_tap(z, k - co * nt);
        tap[k] = (co * Q + c.dy * SO + c.dx) * 4 + c.dy * 2 + c.dx;
    }
    wt += (long)class_base(z, CO) * CI + m0;
    const long n0 = (long)blockIdx.x * BN, N = (long)B * Q, n = n0 + tid % BN;
    const int kq = tid / BN;
    const bool in = n < N;
    const int p = (int)(n % Q);
    const float *src = g + (in ? (n / Q) * (long)CO * Q + p : 0);
    const int border = in ? (p / SO == SO - 1) * 2 + (p % SO == SO - 1) : 3;
    constexpr int A4 = BK * BM / 4 / NT;   // 16-byte pieces of the weights per thread
    float4 wa[A4];
    float xb[PER];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < A4; ++i) {
            const int e = tid + i * NT;
            wa[i] = *reinterpret_cast<const float4 *>(wt + (long)(k0 + e / (BM / 4)) * CI + e % (BM / 4) * 4);
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int e = tap[k0 + kq + KSTEP * i];
            xb[i] = in && !(e & border) ? src[e >> 2] : 0.f;
        }
    };
    auto put = [&](int s) {
#pragma unroll
        for (int i = 0; i < A4; ++i) {
            const int e = tid + i * NT;
            *reinterpret_cast<float4 *>(&t.a[s][e / (BM / 4)][e % (BM / 4) * 4]) = wa[i];
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) t.b[s][kq + KSTEP * i][tid % BN] = xb[i];
    };
    constexpr int TM = Tile<BM, BN>::TM, TN = Tile<BM, BN>::TN;
    float acc[TM][TN] = {};
    __syncthreads();
    fetch(0);
    put(0);
    __syncthreads();
    for (int k0 = 0, s = 0; k0 < K; k0 += BK, s ^= 1) {
        if (k0 + BK < K) fetch(k0 + BK);
        multiply(t, s, acc);
        if (k0 + BK < K) put(s ^ 1);
        __syncthreads();
    }
    const int tx = tid & 15, ty = tid >> 4;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
        const long c = n0 + tx * 4 + 16 * (j & ~3) + (j & 3);
        if (c >= N) continue;
        const int q = (int)(c % Q);
        const long o = ((c / Q) * CI + m0 + ty * TM) * (long)(S * S) + (2 * (q / SO) + (z >> 1)) * S + 2 * (q % SO) + (z & 1);
#pragma unroll
        for (int i = 0; i < TM; ++i) gx[o + (long)i * S * S] = mask[o + (long)i * S * S] > 0.f ? acc[i][j] : 0.f;
    }
}

// ----------------------------------------------- gradient into the weights
// part[split][co][ci 9 + r] = sum over the split's positions of g[b][co][p] x[b][ci][..];
// bpart[split][co] = sum over them of g[b][co][p]
template <int CI, int CO, int S>
__global__ void __launch_bounds__(NT) k_conv32_dw(const float *__restrict__ g, const float *__restrict__ x, int B,
                                                  int kper, float *__restrict__ part, float *__restrict__ bpart) {
    constexpr int BM = 64, BN = 64, SO = S / 2, Q = SO * SO, N = CI * 9;
    static_assert(Q % BK == 0 && CO % BM == 0, "a slice stays within an image");
    __shared__ __align__(16) Tile<BM, BN> t;
    const int tid = threadIdx.x, m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const long kb = (long)blockIdx.z * kper, ke = min((long)B * Q, kb + kper);
    // g: rows tid / 4 and + 32, positions 4 (tid % 4) ..; x: position tid % 16, columns tid / 16 + 8 i
    int off[8];   // (offset from the window's centre) * 4 + border bits, or 3 beyond the last column
    const int nq = tid >> 4, kp = tid & 15;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int c = n0 + nq + 8 * i, ci = c / 9, r = c - ci * 9, ky = r / 3, kx = r - ky * 3;
        off[i] = c < N ? (ci * S * S + (ky - 1) * S + (kx - 1)) * 4 + (ky == 0) * 2 + (kx == 0) : 3;
    }
    float4 ga[2];
    float xb[8];
    float bs[2] = {0.f, 0.f};
    auto fetch = [&](long k0) {
        const long b = k0 / Q;
        const int p0 = (int)(k0 - b * Q);
        const float *gs = g + (b * CO + m0 + (tid >> 2)) * Q + p0 + (tid & 3) * 4;
        ga[0] = *reinterpret_cast<const float4 *>(gs);
        ga[1] = *reinterpret_cast<const float4 *>(gs + 32 * Q);
        const int p = p0 + kp, oy = p / SO, ox = p % SO;
        const float *src = x + b * (long)CI * S * S + 2 * oy * S + 2 * ox;
        const int border = (oy == 0) * 2 + (ox == 0);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const bool ok = !(off[i] & border) && n0 + nq + 8 * i < N;
            xb[i] = ok ? src[off[i] >> 2] : 0.f;
        }
    };
    auto put = [&](int s) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float v[4] = {ga[h].x, ga[h].y, ga[h].z, ga[h].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) t.a[s][(tid & 3) * 4 + j][(tid >> 2) + 32 * h] = v[j];
            bs[h] += (v[0] + v[1]) + (v[2] + v[3]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) t.b[s][kp][nq + 8 * i] = xb[i];
    };
    float acc[8][4] = {};
    if (kb < ke) {   // uniform
        fetch(kb);
        put(0);
        __syncthreads();
        int s = 0;
        for (long k0 = kb; k0 < ke; k0 += BK, s ^= 1) {
            if (k0 + BK < ke) fetch(k0 + BK);
            multiply(t, s, acc);
            if (k0 + BK < ke) put(s ^ 1);
            __syncthreads();
        }
    }
    const int tx = tid & 15, ty = tid >> 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = n0 + tx * 4 + j;
        if (c >= N) continue;
#pragma unroll
        for (int i = 0; i < 8; ++i) part[((long)blockIdx.z * CO + m0 + ty * 8 + i) * N + c] = acc[i][j];
    }
    if (blockIdx.x == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v = bs[h];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if ((tid & 3) == 0) bpart[(long)blockIdx.z * CO + m0 + (tid >> 2) + 32 * h] = v;
        }
    }
}

// the first layer's weight gradient: a warp takes 4 filters, its lanes 32
// positions at a time, 9 taps and the bias in registers
__global__ void __launch_bounds__(256) k_conv32_dw_first(const float *__restrict__ g, CnnInput in,
                                                         const float2 *__restrict__ affine, int B, int kper,
                                                         float *__restrict__ part, float *__restrict__ bpart) {
    constexpr int S = 128, SO = 64, CO = 32, Q = SO * SO;
    const int lane = threadIdx.x & 31, c0 = (threadIdx.x >> 5) * 4;
    const long kb = (long)blockIdx.x * kper, ke = min((long)B * Q, kb + kper);
    float acc[4][10] = {};
    for (long k = kb + lane; k < ke; k += 32) {
        const int b = (int)(k / Q), p = (int)(k % Q), oy = p / SO, ox = p % SO;
        const float2 a = affine[b];
        const float *img = in.x + b * in.img_stride + (long)in.oy * in.row_stride + in.ox;
        float gv[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) gv[c] = g[((long)b * CO + c0 + c) * Q + p];
#pragma unroll
        for (int r = 0; r < 9; ++r) {
            const int iy = 2 * oy - 1 + r / 3, ix = 2 * ox - 1 + r % 3;
            const float v = iy >= 0 && ix >= 0 && iy < S && ix < S ? fmaf(img[(long)iy * in.row_stride + ix], a.x, a.y) : 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c][r] = fmaf(gv[c], v, acc[c][r]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c][9] += gv[c];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int r = 0; r < 10; ++r) {
            float v = acc[c][r];
#pragma unroll
            for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) {
                if (r < 9)
                    part[((long)blockIdx.x * CO + c0 + c) * 9 + r] = v;
                else
                    bpart[(long)blockIdx.x * CO + c0 + c] = v;
            }
        }
}

// out[i] = sum over z of part[z][i]: eight interleaved partial sums per output,
// added in order (a fixed order: the same inputs give the same sums on every run)
__global__ void __launch_bounds__(256) k_conv32_sum(const float *__restrict__ part, int splits, int n,
                                                    float *__restrict__ out) {
    __shared__ float sh[8][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (i < n)
        for (int z = w; z < splits; z += 8) s += part[(long)z * n + i];
    sh[w][lane] = s;
    __syncthreads();
    if (w == 0 && i < n) {
        for (int k = 1; k < 8; ++k) s += sh[k][lane];
        out[i] = s;
    }
}

template <int CI, int CO, int S, int BN>
cudaError_t fwd(const float *x, const float *w, const float *bias, int B, float *y, cudaStream_t st) {
    const long N = (long)B * (S / 2) * (S / 2);
    k_conv32_fwd<CI, CO, S, BN><<<dim3((unsigned)((N + BN - 1) / BN), CO / 64), NT, 0, st>>>(x, w, bias, B, y);
    return cudaGetLastError();
}
template <int CI, int CO, int S, int BM, int BN>
cudaError_t dx(const float *g, const float *w, const float *mask, int B, float *wt, float *gx, cudaStream_t st) {
    constexpr int SO = S / 2;
    k_conv32_wt<<<(CO * CI * 9 + 255) / 256, 256, 0, st>>>(w, CO, CI, wt);
    const long N = (long)B * SO * SO;
    k_conv32_dx<CI, CO, SO, BM, BN><<<dim3((unsigned)((N + BN - 1) / BN), CI / BM, 4), NT, 0, st>>>(g, wt, mask, B, gx);
    return cudaGetLastError();
}
cudaError_t sum(const float *part, int splits, int n, float *out, cudaStream_t st) {
    k_conv32_sum<<<(n + 31) / 32, 256, 0, st>>>(part, splits, n, out);
    return cudaGetLastError();
}
// positions per split (whole slices) for about `want` CTAs in all, within the partials' buffer
int split_positions(long K, long tiles, long want, size_t out, size_t room, int unit) {
    long splits = (want + tiles - 1) / tiles;
    if (splits > (long)(room / out)) splits = (long)(room / out);
    const long units = (K + unit - 1) / unit;
    if (splits > units) splits = units;
    if (splits < 1) splits = 1;
    return (int)((units + splits - 1) / splits * unit);
}
template <int CI, int CO, int S>
cudaError_t dw(const float *g, const float *x, int B, float *part, size_t part_floats, float *bpart, size_t bpart_floats,
               float *gw, float *gb, int num_sms, cudaStream_t st) {
    const long K = (long)B * (S / 2) * (S / 2);
    const int N = CI * 9, tn = (N + 63) / 64, tm = CO / 64;
    size_t room = part_floats;   // bpart holds splits x CO: as many splits as both buffers hold
    if (bpart_floats / CO < room / ((size_t)CO * N)) room = bpart_floats / CO * ((size_t)CO * N);
    const int kper = split_positions(K, (long)tn * tm, 4L * num_sms, (size_t)CO * N, room, BK);
    const int splits = (int)((K + kper - 1) / kper);
    k_conv32_dw<CI, CO, S><<<dim3(tn, tm, splits), NT, 0, st>>>(g, x, B, kper, part, bpart);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = sum(part, splits, CO * N, gw, st);
    if (e == cudaSuccess) e = sum(bpart, splits, CO, gb, st);
    return e;
}

}  // namespace

cudaError_t launch_conv32_forward(int layer, const float *x, const CnnInput &in, const float2 *affine, const float *w,
                                  const float *bias, int B, float *y, cudaStream_t st) {
    if (B <= 0) return cudaSuccess;
    switch (layer) {
        case 0: {
            const long n = (long)B * 64 * 64;
            k_conv32_first<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, affine, w, bias, B, y);
            return cudaGetLastError();
        }
        case 1: return fwd<32, 64, 64, 128>(x, w, bias, B, y, st);
        case 2: return fwd<64, 64, 32, 128>(x, w, bias, B, y, st);
        case 3: return fwd<64, 128, 16, 64>(x, w, bias, B, y, st);
        case 4: return fwd<128, 128, 8, 64>(x, w, bias, B, y, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_conv32_dx(int layer, const float *g, const float *w, const float *mask, int B, float *wt, float *gx,
                             cudaStream_t st) {
    if (B <= 0) return cudaSuccess;
    switch (layer) {
        case 1: return dx<32, 64, 64, 32, 128>(g, w, mask, B, wt, gx, st);
        case 2: return dx<64, 64, 32, 64, 128>(g, w, mask, B, wt, gx, st);
        case 3: return dx<64, 128, 16, 64, 64>(g, w, mask, B, wt, gx, st);
        case 4: return dx<128, 128, 8, 64, 64>(g, w, mask, B, wt, gx, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_conv32_dw(int layer, const float *g, const float *x, const CnnInput &in, const float2 *affine, int B,
                             float *part, size_t part_floats, float *bpart, size_t bpart_floats, float *gw, float *gb,
                             int num_sms, cudaStream_t st) {
    if (B <= 0) return cudaSuccess;
    switch (layer) {
        case 0: {
            const int kper = split_positions((long)B * 64 * 64, 1, 4L * num_sms, 32, bpart_floats, 32);
            const int splits = (int)(((long)B * 64 * 64 + kper - 1) / kper);
            k_conv32_dw_first<<<splits, 256, 0, st>>>(g, in, affine, B, kper, part, bpart);
            cudaError_t e = cudaGetLastError();
            if (e == cudaSuccess) e = sum(part, splits, 32 * 9, gw, st);
            if (e == cudaSuccess) e = sum(bpart, splits, 32, gb, st);
            return e;
        }
        case 1: return dw<32, 64, 64>(g, x, B, part, part_floats, bpart, bpart_floats, gw, gb, num_sms, st);
        case 2: return dw<64, 64, 32>(g, x, B, part, part_floats, bpart, bpart_floats, gw, gb, num_sms, st);
        case 3: return dw<64, 128, 16>(g, x, B, part, part_floats, bpart, bpart_floats, gw, gb, num_sms, st);
        case 4: return dw<128, 128, 8>(g, x, B, part, part_floats, bpart, bpart_floats, gw, gb, num_sms, st);
        default: return cudaErrorInvalidValue;
    }
}
