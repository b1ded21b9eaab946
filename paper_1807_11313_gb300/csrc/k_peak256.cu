// 256 x 256 cross-correlation of one template and one pattern and its peak: the
// value, the 3-point parabolic position per axis (clamped to +-0.5) and optionally
// the row-major index of the maximum (ties: the lowest).
//
// One surface per cluster of four CTAs, through the passes of passes256.cuh: the
// products conj(S_t) S_p go from memory into the column passes, and the finished
// lines stay in shared memory until the cluster's maximum is known and its four
// neighbours are read from wherever they lie.
//
// What bounds it: latency (five cluster barriers per surface, 528 KB of spectra from
// memory).  1,000 surfaces: 0.45 -> 0.22 ms against two surfaces per complex
// transform, rows first, one cluster of 256-thread CTAs per four SMs and the columns
// around each maximum transformed again.
#include "kernels.cuh"
#include "passes256.cuh"

namespace {

using namespace p256;

struct Smem {
    float2 buf[OWN * N];    // columns: [128][2 OWN] (column, mirror); lines: [OWN][256]
    float2 tw[256];         // W256^(a b) at [a][b]
    float2 p0[N];           // CTA 0: the packed column
    float2 top[NT / 32];    // the warps' maxima: value, index
};

__device__ __forceinline__ void better(float &bv, int &bi, float v, int i) {
    if (v > bv || (v == bv && i < bi)) {
        bv = v;
        bi = i;
    }
}
__device__ __forceinline__ float parabola_c(float cm, float c0, float cp) {
    const float den = cm - 2.f * c0 + cp;
    if (!(den < 0.f)) return 0.f;
    const float d = (cm - cp) / (2.f * den);
    return fminf(0.5f, fmaxf(-0.5f, d));
}

__global__ void __launch_bounds__(NT, 2)
k_peak256(const float2 *__restrict__ St, const int *__restrict__ tidx, const float2 *__restrict__ Sp,
          const int *__restrict__ degen, const int *__restrict__ active, int P, float *__restrict__ peak,
          float *__restrict__ shift, int *__restrict__ argmax) {
    extern __shared__ float4 smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    float2 *buf = sm.buf;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = (int)cluster_rank(), cid = blockIdx.x / NC, ncl = gridDim.x / NC;
    for (int i = tid; i < 256; i += NT) sm.tw[i] = twiddle(i);
    const int lr = tid >> 4, b = tid & 15;
    const int ql = tid & (OWN - 1), a8 = tid / OWN, q = OWN * c + ql;
    const bool packed = q == 0;
    uint32_t base[NC];
#pragma unroll
    for (int r = 0; r < NC; ++r) base[r] = map_to_rank(buf, r);
    __syncthreads();

    for (int p = cid; p < P; p += ncl) {   // every branch below is uniform over the cluster
        if (active && !active[p]) continue;
        const int t = tidx ? tidx[p] : p;
        if ((degen && degen[p]) || t < 0) {
            if (tid == 0 && c == 0) {
                peak[p] = 0.f;
                shift[2 * p] = 0.f;
                shift[2 * p + 1] = 0.f;
            }
            continue;
        }
        const float2 *tp = St + (size_t)t * N * HW, *sp = Sp + (size_t)p * N * HW;
        if (c == 0) {
            static_assert(NT == N, "a thread per row of the packed column");
            const float2 a = c_mulcj(__ldg(tp + tid * HW), __ldg(sp + tid * HW)),
                         h = c_mulcj(__ldg(tp + tid * HW + 128), __ldg(sp + tid * HW + 128));
            sm.p0[tid] = make_float2(a.x - h.y, a.y + h.x);
            __syncthreads();
        }
        // ---- columns
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
            column_store<+1>(x, buf, sm.tw, ql, a8, h);
        }
        __syncthreads();
        columns_to_lines(buf, ql, a8, packed);
        cluster_arrive_shared();
        cluster_wait();   // the columns are complete
        // ---- lines
        float2 z[2][16];
        gather_lines(z, base, OWN * c + lr, b);
        cluster_arrive();   // releases this thread's gathers
        cluster_wait();     // every thread of the cluster has its values: the buffer takes the lines
        float bv = -INFINITY;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float2 *line = buf + (lr + h * (OWN / 2)) * N;
            line_store<+1>(z[h], line, sm.tw, b);
            __syncwarp();
            line_load(z[h], line, b);
            fft_reg_dif<16, +1>(z[h]);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                line[b + 16 * cx_bitrev(k, 4)] = z[h][k];
                bv = fmaxf(bv, fmaxf(z[h][k].x, z[h][k].y));
            }
        }
        // the first of the thread's values that is the maximum, in row-major order
        int bi = 0x7fffffff;
#pragma unroll
        for (int s = 1; s >= 0; --s)
#pragma unroll
            for (int h = 1; h >= 0; --h)
#pragma unroll
                for (int j = 15; j >= 0; --j) {
                    const float2 v = z[h][cx_bitrev(j, 4)];
                    if ((s ? v.y : v.x) == bv) bi = (OWN * c + lr + h * (OWN / 2) + 128 * s) * N + b + 16 * j;
                }
#pragma unroll
        for (int o = 16; o; o >>= 1)
            better(bv, bi, __shfl_xor_sync(0xffffffffu, bv, o), __shfl_xor_sync(0xffffffffu, bi, o));
        if (lane == 0) sm.top[warp] = make_float2(bv, __int_as_float(bi));
        cluster_arrive_shared();
        cluster_wait();   // lines and maxima are in place
        float c0 = 0.f, cxm = 0.f, cxp = 0.f, cym = 0.f, cyp = 0.f;
        if (c == 0 && warp == 0) {
            const float2 v = ld_cluster(map_to_rank(&sm.top[lane & (NT / 32 - 1)], lane / (NT / 32)));
            bv = v.x;
            bi = __float_as_int(v.y);
#pragma unroll
            for (int o = 16; o; o >>= 1)
                better(bv, bi, __shfl_xor_sync(0xffffffffu, bv, o), __shfl_xor_sync(0xffffffffu, bi, o));
            bi = min(bi, N * N - 1);   // no finite value: any place
            const int y0 = bi >> 8, x0 = bi & (N - 1);
            // lanes 0 .. 4: the maximum, left, right, above, below
            const int y = (y0 + (lane == 3 ? N - 1 : lane == 4 ? 1 : 0)) & (N - 1);
            const int x = (x0 + (lane == 1 ? N - 1 : lane == 2 ? 1 : 0)) & (N - 1);
            const float2 w = ld_cluster(map_to_rank(buf + (y & (OWN - 1)) * N + x, (y & 127) / OWN));
            const float mine = y & 128 ? w.y : w.x;
            c0 = __shfl_sync(0xffffffffu, mine, 0);
            cxm = __shfl_sync(0xffffffffu, mine, 1);
            cxp = __shfl_sync(0xffffffffu, mine, 2);
            cym = __shfl_sync(0xffffffffu, mine, 3);
            cyp = __shfl_sync(0xffffffffu, mine, 4);
        }
        cluster_arrive();   // releases CTA 0's reads of the other CTAs' lines and maxima (the results follow it: no store to wait for)
        if (c == 0 && tid == 0) {
            const int y0 = bi >> 8, x0 = bi & (N - 1);
            peak[p] = c0;
            shift[2 * p] = (float)(x0 < N / 2 ? x0 : x0 - N) + parabola_c(cxm, c0, cxp);
            shift[2 * p + 1] = (float)(y0 < N / 2 ? y0 : y0 - N) + parabola_c(cym, c0, cyp);
            if (argmax) argmax[p] = bi;
        }
        __syncwarp();
        cluster_wait();
    }
    cluster_arrive();   // no CTA leaves while another may still read its shared memory
    cluster_wait();
}

}  // namespace

cudaError_t launch_pair_peak_c256(const float2 *St, const int *tidx, const float2 *Sp, const int *degen,
                                  const int *active, int P, float *peak, float *shift, cudaStream_t st,
                                  int *argmax) {
    if (P <= 0) return cudaSuccess;
    static std::atomic<int> resident{0};
    int most = 0;
    const cudaError_t e = resident_clusters(k_peak256, NC, NT, sizeof(Smem), resident, &most);
    if (e != cudaSuccess) return e;
    return launch_clusters(k_peak256, NC, NT, sizeof(Smem), P < most ? P : most, st, St, tidx, Sp, degen, active, P, peak, shift, argmax);
}
