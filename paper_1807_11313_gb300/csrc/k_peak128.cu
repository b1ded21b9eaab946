// Single-surface peak at N = 128: one real correlation surface per pattern, its
// integer argmax (ties: the lowest row-major shift) and the 3-point parabola
// per axis.
//
// Paper: Eqs. 3 and 6 (the surface), peak up-sampling read as the parabola.
//
// One CTA of 256 threads per pattern, two CTAs per SM.  The transform is the
// search kernel's three register rounds (k_search128.cu) on the products of
// the two spectra, read once from global memory in coalesced rows; the surface
// is then left in the shared-memory buffer for the neighbours of its maximum.
// Bound by the spectra's 133 KB per pattern and the latency of its few phases.
// The kernel it replaces transformed a pair of patterns per 1,024-thread CTA
// line by line in shared memory (133 KB, one CTA per SM): 205 us per 2,000
// patterns, now 82; three CTAs per SM (80 registers) measured 115.
#include "common.cuh"
#include "fft128.cuh"
#include "kernels.cuh"

namespace {

using namespace fft128;

constexpr int N = 128, HW = 65, NT = 256;

struct Smem {
    float2 buf[N * N / 2];   // eight regions of 1,024, one per warp
    float2 tw1[128];         // W128^(l k2) at [l][k2]
    float2 tw2[128];         // W128^(g k3) at [k3][g]
    float2 p0[N];            // the packed column X[u][0] + i X[u][64]
    float wmax[NT / 32];
    float top;
    int at;
};

// as in the search: round-1 output (k2 pairs by warp) and a warp's lines
__device__ __forceinline__ int idxA(int l, int k2, int q) { return ((k2 >> 1) << 10) + (l << 7) + ((k2 & 1) << 6) + q; }
__device__ __forceinline__ int idxB(int r, int g) { return (r << 5) + ((((g >> 1) ^ (r & 7)) << 1) | (g & 1)); }
// where surface point (y, x) is left: line y mod 64 = k2 + 16 j, residue x mod 4
__device__ __forceinline__ float surface(const float2 *buf, int y, int x) {
    const int pr = y & 63, k2 = pr & 15, r = 8 * (pr >> 4) + 4 * (k2 & 1) + (x & 3);
    const float2 z = buf[((k2 >> 1) << 10) + idxB(r, x >> 2)];
    return y < 64 ? z.x : z.y;
}
__device__ __forceinline__ float parabola(float cm, float c0, float cp) {
    const float den = cm - 2.f * c0 + cp;
    if (!(den < 0.f)) return 0.f;
    const float d = (cm - cp) / (2.f * den);
    return fminf(0.5f, fmaxf(-0.5f, d));
}

__global__ void __launch_bounds__(NT, 2)
k_peak128(const float2 *__restrict__ St, const int *__restrict__ tidx, const float2 *__restrict__ Sp,
          const int *__restrict__ degen, const int *__restrict__ active, float *__restrict__ peak,
          float *__restrict__ shift, int *__restrict__ argmax) {
    extern __shared__ float4 smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    float2 *buf = sm.buf;
    const int p = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (active && !active[p]) return;
    const int t = tidx ? tidx[p] : p;
    if ((degen && degen[p]) || t < 0) {
        if (tid == 0) {
            peak[p] = 0.f;
            shift[2 * (size_t)p] = 0.f;
            shift[2 * (size_t)p + 1] = 0.f;
        }
        return;
    }
    const float2 *ta = St + (size_t)t * N * HW, *sa = Sp + (size_t)p * N * HW;
    if (tid < 128) {
        const float2 x0 = c_mulcj(__ldg(ta + tid * HW), __ldg(sa + tid * HW));
        const float2 xh = c_mulcj(__ldg(ta + tid * HW + 64), __ldg(sa + tid * HW + 64));
        sm.p0[tid] = make_float2(x0.x - xh.y, x0.y + xh.x);
        sm.tw1[tid] = w128((tid >> 4) * (tid & 15));
    } else {
        const int i = tid - 128;
        sm.tw2[i] = w128((i & 31) * (i >> 5));
    }
    if (tid == 0) sm.at = 0x7fffffff;
    // ---- round 1: stored column q, rows u = l + 8 m for l = l1 and l1 + 4
    const int q = ((warp & 1) << 5) + lane, l1 = warp >> 1;
    float2 a[2][16];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float2 s[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int k = (l1 + 4 * h + 8 * m) * HW + q;
            a[h][m] = __ldg(ta + k);
            s[m] = __ldg(sa + k);
        }
#pragma unroll
        for (int m = 0; m < 16; ++m) a[h][m] = c_mulcj(a[h][m], s[m]);
    }
    __syncthreads();   // the packed column and the tables
    if (q == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int m = 0; m < 16; ++m) a[h][m] = sm.p0[l1 + 4 * h + 8 * m];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        fft_reg_dif<16, +1>(a[h]);
        const int l = l1 + 4 * h;
        const float4 *tw = reinterpret_cast<const float4 *>(sm.tw1 + l * 16);
        StaticFor<0, 8>::run([&](auto kk) {
            constexpr int ka = 2 * decltype(kk)::value, R0 = cx_bitrev(ka, 4), R1 = cx_bitrev(ka + 1, 4);
            const float4 w = tw[ka >> 1];
            buf[idxA(l, ka, q)] = ka ? c_mul(a[h][R0], make_float2(w.x, w.y)) : a[h][R0];
            buf[idxA(l, ka + 1, q)] = c_mul(a[h][R1], make_float2(w.z, w.w));
        });
    }
    __syncthreads();
    // ---- round 2, and the exchange within the warp's region
    const int k2 = 2 * warp + (lane >> 4), g = lane & 15, gb = residue_b(g);
    float2 *own = buf + warp * 1024;
    {
        float2 x[4][8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 *src = buf + idxA(0, k2, col_of(g, k));
#pragma unroll
            for (int l = 0; l < 8; ++l) x[k][l] = src[l * 128];
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k) fft_reg_dif<8, +1>(x[k]);   // x[k][bitrev(j)] = row k2 + 16 j
        const float2 wa1 = sm.tw2[32 + g], wa2 = sm.tw2[64 + g], wa3 = sm.tw2[96 + g];
        const float2 wb1 = sm.tw2[32 + gb], wb2 = sm.tw2[64 + gb], wb3 = sm.tw2[96 + gb];
        const int r0 = (lane >> 4) * 4;
        StaticFor<0, 4>::run([&](auto jj) {
            constexpr int j = decltype(jj)::value, RA = cx_bitrev(j, 3), RB = cx_bitrev(j + 4, 3);
            const float2 ra[4] = {x[0][RA], x[1][RA], x[2][RA], x[3][RA]};
            const float2 rb[4] = {x[0][RB], x[1][RB], x[2][RB], x[3][RB]};
            float2 A[4], B[4];
            merge_rows(ra, rb, g == 0, A, B);
            dft4<+1>(A[0], A[1], A[2], A[3]);
            dft4<+1>(B[0], B[1], B[2], B[3]);
            const int r = 8 * j + r0;
            own[idxB(r, g)] = A[0];
            own[idxB(r + 1, g)] = c_mul(A[1], wa1);
            own[idxB(r + 2, g)] = c_mul(A[2], wa2);
            own[idxB(r + 3, g)] = c_mul(A[3], wa3);
            own[idxB(r, gb)] = B[0];
            own[idxB(r + 1, gb)] = c_mul(B[1], wb1);
            own[idxB(r + 2, gb)] = c_mul(B[2], wb2);
            own[idxB(r + 3, gb)] = c_mul(B[3], wb3);
        });
    }
    __syncwarp();
    // ---- round 3: lane r's line k2 + 16 j (r = 8 j + 4 (k2 & 1) + k3), columns k3 + 4 k4
    float2 z[32];
    float4 *line = reinterpret_cast<float4 *>(own) + (lane << 4);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const float4 v = line[j ^ (lane & 7)];
        z[2 * j] = make_float2(v.x, v.y);
        z[2 * j + 1] = make_float2(v.z, v.w);
    }
    fft_reg_dif<32, +1>(z);   // z[bitrev(k4)] = (row y, row y + 64) at column k3 + 4 k4
    float top = -INFINITY;
    StaticFor<0, 16>::run([&](auto ii) {   // each lane rewrites its own line
        constexpr int i = decltype(ii)::value, R0 = cx_bitrev(2 * i, 5), R1 = cx_bitrev(2 * i + 1, 5);
        line[i ^ (lane & 7)] = make_float4(z[R0].x, z[R0].y, z[R1].x, z[R1].y);
        top = fmaxf(top, fmaxf(fmaxf(z[R0].x, z[R0].y), fmaxf(z[R1].x, z[R1].y)));
    });
    float wtop = top;
#pragma unroll
    for (int o = 16; o; o >>= 1) wtop = fmaxf(wtop, __shfl_xor_sync(0xffffffffu, wtop, o));
    if (lane == 0) sm.wmax[warp] = wtop;
    __syncthreads();
    wtop = sm.wmax[0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) wtop = fmaxf(wtop, sm.wmax[w]);
    if (top == wtop) {   // the lowest row-major index of this thread's points that attain the maximum
        const int y = 2 * warp + ((lane >> 2) & 1) + 16 * (lane >> 3), x0 = lane & 3;
        int best = 0x7fffffff;
        StaticFor<0, 32>::run([&](auto kk) {
            constexpr int k4 = 31 - decltype(kk)::value, R = cx_bitrev(k4, 5);
            if (z[R].y == wtop) best = min(best, (y + 64) * N + x0 + 4 * k4);
            if (z[R].x == wtop) best = min(best, y * N + x0 + 4 * k4);
        });
        atomicMin(&sm.at, best);
    }
    __syncthreads();
    if (tid == 0) {
        const int i0 = sm.at < N * N ? sm.at : 0;   // nothing compares equal on a surface of NaN
        const int y0 = i0 / N, x0 = i0 % N;
        const float c0 = surface(buf, y0, x0);
        const float cxm = surface(buf, y0, (x0 + N - 1) % N), cxp = surface(buf, y0, (x0 + 1) % N);
        const float cym = surface(buf, (y0 + N - 1) % N, x0), cyp = surface(buf, (y0 + 1) % N, x0);
        peak[p] = c0;
        shift[2 * (size_t)p] = (float)(x0 < N / 2 ? x0 : x0 - N) + parabola(cxm, c0, cxp);
        shift[2 * (size_t)p + 1] = (float)(y0 < N / 2 ? y0 : y0 - N) + parabola(cym, c0, cyp);
        if (argmax) argmax[p] = i0;
    }
}

}  // namespace

cudaError_t launch_peak128(const float2 *St, const int *tidx, const float2 *Sp, const int *degen, const int *active,
                           int P, float *peak, float *shift, int *argmax, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_peak128, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (e != cudaSuccess) return e;
    k_peak128<<<P, NT, sizeof(Smem), st>>>(St, tidx, Sp, degen, active, peak, shift, argmax);
    return cudaGetLastError();
}
