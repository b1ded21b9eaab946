// The 128 x 128 all-pairs search as a device function (see k_search128.cu for
// the design), shared by the search kernel and the multi-map kernel.
#pragma once
#include "common.cuh"
#include "fft128.cuh"

namespace s128 {

constexpr int N = 128;
constexpr int HW = 65;          // stored columns of a half spectrum
constexpr int SPEC = N * HW;    // complex values per half spectrum
constexpr int NT = 512, NG = 256;   // threads per CTA; per group (one template at a time)
constexpr int COL64 = 8192;     // offset of column 64 in the packed layout

// shared layout (float2 units)
constexpr int OFF_SP = 0;                  // pattern, packed layout, 8320
constexpr int OFF_BUF = SPEC;              // per group: staged template / transposes, 2 x 8192
constexpr int OFF_TW1 = OFF_BUF + 2 * 8192;  // W128^(l k2) at [l][k2], l < 8, k2 < 16
constexpr int OFF_TW2 = OFF_TW1 + 128;     // W128^(g k3) at [k3][g], k3 < 4, g < 32
constexpr int OFF_EDGE = OFF_TW2 + 128;    // per group: the next template's columns 0 and 64, 2 x [2][128]
constexpr int OFF_P0 = OFF_EDGE + 512;     // per group: the packed column X[u][0] + i X[u][64], 2 x [128]
constexpr int OFF_RED = OFF_P0 + 256;      // per group: eight warps' maxima, two templates, 2 x 8
constexpr int SMEM_F2 = OFF_RED + 16;
constexpr size_t SMEM_BYTES = sizeof(float2) * SMEM_F2;

// packed position of (row u, stored column q < 64): [u & 7][(u >> 3) / 2][q][(u >> 3) & 1]
__host__ __device__ __forceinline__ int pk(int u, int q) {
    const int l = u & 7, m = u >> 3;
    return (((l * 8 + (m >> 1)) * 64 + q) << 1) + (m & 1);
}

// A group's buffer is eight regions of 1,024, one per warp: round 2's warp w
// takes the round-1 outputs of k2 = 2 w and 2 w + 1, which lie in its region
__device__ __forceinline__ int idxA(int l, int k2, int q) { return ((k2 >> 1) << 10) + (l << 7) + ((k2 & 1) << 6) + q; }
// round-2 output within a warp's region, line r = 8 j + 4 (k2 & 1) + k3 over g:
// 16-byte pairs of g swizzled by r & 7, so that round 3's loads (one line per
// lane) spread over every bank
__device__ __forceinline__ int idxB(int r, int g) { return (r << 5) + ((((g >> 1) ^ (r & 7)) << 1) | (g & 1)); }

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_wait_one() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// one radix-2 decimation-in-frequency stage (sign +) of an R-point register FFT
template <int R, int STAGE>
__device__ __forceinline__ void dif_stage(float2 (&x)[R]) {
    constexpr int span = R >> (STAGE + 1);
    StaticFor<0, R / (2 * span)>::run([&](auto blk) {
        StaticFor<0, span>::run([&](auto k) {
            constexpr int kk = decltype(k)::value;
            constexpr int i0 = decltype(blk)::value * 2 * span + kk;
            constexpr int i1 = i0 + span;
            const float2 a = x[i0], b = x[i1];
            x[i0] = c_add(a, b);
            x[i1] = tw_mul<kk, 2 * span, +1>(c_sub(a, b));
        });
    });
}

// stages 1..3 of a 32-point DIF FFT (stage 0 done by the caller) followed by
// the maximum over the real and imaginary parts of its outputs: the last
// butterfly stage is folded into the maximum, max(a + b, a - b) = a + |b|
// (exact: rounding is monotonic)
__device__ __forceinline__ float fft32_rest_max(float2 (&x)[32]) {
    dif_stage<32, 1>(x);
    dif_stage<32, 2>(x);
    dif_stage<32, 3>(x);
    float m = fmaxf(x[0].x + fabsf(x[1].x), x[0].y + fabsf(x[1].y));
#pragma unroll
    for (int j = 2; j < 32; j += 2) m = fmaxf(m, fmaxf(x[j].x + fabsf(x[j + 1].x), x[j].y + fabsf(x[j + 1].y)));
    return m;
}

// One work item of the search: pattern p against template pairs [pb, pe)
// (templates 2 pb .. min(2 pe, T) - 1, the even ones by group 0, the odd ones
// by group 1).  Runs on the calling CTA's NT threads and SMEM_BYTES of dynamic
// shared memory (named barriers 1 and 2) and folds the best (peak, template)
// of the item into keys[p].  ALL: also write every template's peak to
// peaks_all [P][T].  LIST: the T positions are the pattern's candidate list
// (library indices in any order, < 0: none).
template <bool ALL, bool LIST = false>
__device__ __forceinline__ void search_body(const float2 *__restrict__ Spk, int T, const float2 *__restrict__ Sp,
                                              int p, int pb, int pe, unsigned long long *__restrict__ keys,
                                              float *__restrict__ peaks_all, const int *__restrict__ list = nullptr) {
    static_assert(!(ALL && LIST), "lists keep the best only");
    using namespace fft128;
    extern __shared__ float4 smem_raw[];
    float2 *sm = reinterpret_cast<float2 *>(smem_raw);
    const int grp = threadIdx.x / NG, tid = threadIdx.x % NG, lane = tid & 31, warp = tid >> 5;
    float2 *sp = sm + OFF_SP;
    float2 *buf = sm + OFF_BUF + grp * 8192;
    float2 *edge = sm + OFF_EDGE + grp * 256;
    float2 *p0 = sm + OFF_P0 + grp * 128;
    auto sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(NG) : "memory"); };

    // round 1: lane -> stored column q, warp -> its half and the row residues l1 and l1 + 4 mod 8
    const int q = ((warp & 1) << 5) + lane, l1 = warp >> 1;
    // round 2: (k2, g), columns +-g mod 32
    const int k2 = 2 * warp + (lane >> 4), g = lane & 15, gb = residue_b(g);
    const bool special = g == 0;
    float2 *own = buf + warp * 1024;   // this warp's region

    const int te = min(2 * pe, T);
    auto id = [&](int j) { return LIST ? __ldg(list + j) : j; };
    // the group's next position from j on with a template (te or above: none)
    auto used = [&](int j) {
        if (LIST)
            while (j < te && id(j) < 0) j += 2;
        return j;
    };
    // a template's columns 0..63 fill the group's buffer exactly; each warp copies into its region
    auto stage = [&](int t) {
        const float4 *s = reinterpret_cast<const float4 *>(Spk + (size_t)t * SPEC);
        float4 *d = reinterpret_cast<float4 *>(buf);
#pragma unroll
        for (int k = 0; k < 16; ++k) cp_async16(d + warp * 512 + k * 32 + lane, s + warp * 512 + k * 32 + lane);
        cp_async_commit();
    };
    // columns 0 and 64 at row u = tid < 128, copied by the thread that turns
    // them into p0[u] (so no barrier separates the two)
    auto stage_edge = [&](int t) {
        if (tid < N) {
            const float2 *s = Spk + (size_t)t * SPEC;
            cp_async8(edge + tid, s + pk(tid, 0));
            cp_async8(edge + N + tid, s + COL64 + tid);
        }
        cp_async_commit();
    };
    auto make_p0 = [&]() {
        if (tid < N) {
            const float2 x0 = c_mulcj(edge[tid], sp[pk(tid, 0)]), xh = c_mulcj(edge[N + tid], sp[COL64 + tid]);
            p0[tid] = make_float2(x0.x - xh.y, x0.y + xh.x);
        }
    };

    {   // pattern spectrum (packed into shared memory) and twiddle tables
        const float2 *src = Sp + (size_t)p * SPEC;
        for (int i = threadIdx.x; i < SPEC; i += NT) {
            const int u = i / HW, v = i % HW;
            sp[v < 64 ? pk(u, v) : COL64 + u] = src[i];
        }
        float2 *tw1 = sm + OFF_TW1, *tw2 = sm + OFF_TW2;
        if (threadIdx.x < 128)
            tw1[threadIdx.x] = w128((threadIdx.x >> 4) * (threadIdx.x & 15));   // [l][k2]
        else if (threadIdx.x < 256)
            tw2[threadIdx.x - 128] = w128((threadIdx.x & 31) * ((threadIdx.x - 128) >> 5));   // [k3][g]
    }
    int t = used(2 * pb + grp);
    if (t < te) {
        stage_edge(id(t));
        stage(id(t));
        cp_async_wait_all();
    }
    __syncthreads();   // the pattern and the tables are in place
    if (t < te) make_p0();

    float best_v = -INFINITY;   // this thread's largest value and its template (the lowest among equals)
    int best_t = -1;

    // Per template three barriers of the group: the staged template is complete; it
    // has been read (the register work of round 1 runs before this one); the columns
    // are exchanged.  From there on a warp works in its own region alone.
    for (int it = 0, tn; t < te; t = tn, ++it) {
        tn = used(t + 2);
        cp_async_wait_all();
        sync();   // buf holds template t, p0 its packed column; the previous round 3 is done with buf
        if (ALL && it > 0 && tid == 0) {
            const float *r = reinterpret_cast<const float *>(sm + OFF_RED + grp * 8) + ((it - 1) & 1) * 8;
            float m = r[0];
#pragma unroll
            for (int w = 1; w < 8; ++w) m = fmaxf(m, r[w]);
            peaks_all[(size_t)p * T + t - 2] = m;
        }

        // ---------------- round 1: 16-point column sub-FFTs ----------------
        float2 a[2][16];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 *sp4 = reinterpret_cast<const float4 *>(sp) + (l1 + 4 * h) * 512 + q;
            const float4 *tp4 = reinterpret_cast<const float4 *>(buf) + (l1 + 4 * h) * 512 + q;
#pragma unroll
            for (int mp = 0; mp < 8; ++mp) {
                const float4 s4 = sp4[mp * 64], t4 = tp4[mp * 64];
                a[h][2 * mp] = c_mulcj(make_float2(t4.x, t4.y), make_float2(s4.x, s4.y));
                a[h][2 * mp + 1] = c_mulcj(make_float2(t4.z, t4.w), make_float2(s4.z, s4.w));
            }
        }
        if (q == 0) {   // one lane of four warps
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int m = 0; m < 16; ++m) a[h][m] = p0[l1 + 4 * h + 8 * m];
        }
        fft_reg_dif<16, +1>(a[0]);
        fft_reg_dif<16, +1>(a[1]);
        sync();   // every thread has read the staged template: buf is free
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int l = l1 + 4 * h;
            const float4 *tw = reinterpret_cast<const float4 *>(sm + OFF_TW1 + l * 16);
            StaticFor<0, 8>::run([&](auto kk) {
                constexpr int ka = 2 * decltype(kk)::value, R0 = cx_bitrev(ka, 4), R1 = cx_bitrev(ka + 1, 4);
                const float4 w = tw[ka >> 1];
                buf[idxA(l, ka, q)] = ka ? c_mul(a[h][R0], make_float2(w.x, w.y)) : a[h][R0];
                buf[idxA(l, ka + 1, q)] = c_mul(a[h][R1], make_float2(w.z, w.w));
            });
        }
        sync();

        // ------- round 2: radix 8 over l finishes the columns; rows paired; radix 4 starts the lines -------
        float2 x[4][8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 *src = buf + idxA(0, k2, col_of(g, k));
#pragma unroll
            for (int l = 0; l < 8; ++l) x[k][l] = src[l * 128];
        }
        __syncwarp();   // the warp has read its columns: its region is free
        if (tn < te) stage_edge(id(tn));   // edge was last read for this template's p0
#pragma unroll
        for (int k = 0; k < 4; ++k) fft_reg_dif<8, +1>(x[k]);   // x[k][bitrev(j)] = row k2 + 16 j
        {
            const float2 *tw = sm + OFF_TW2;
            const float2 wa1 = tw[32 + g], wa2 = tw[64 + g], wa3 = tw[96 + g];
            const float2 wb1 = tw[32 + gb], wb2 = tw[64 + gb], wb3 = tw[96 + gb];
            const int r0 = (lane >> 4) * 4;
            StaticFor<0, 4>::run([&](auto jj) {
                constexpr int j = decltype(jj)::value, RA = cx_bitrev(j, 3), RB = cx_bitrev(j + 4, 3);
                const float2 ra[4] = {x[0][RA], x[1][RA], x[2][RA], x[3][RA]};
                const float2 rb[4] = {x[0][RB], x[1][RB], x[2][RB], x[3][RB]};
                float2 A[4], B[4];
                merge_rows(ra, rb, special, A, B);
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

        // ------- round 3: 32-point line FFTs, maximum; the next template streams in meanwhile -------
        float2 z[32];
        {
            const float4 *line = reinterpret_cast<const float4 *>(own) + (lane << 4);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const float4 v = line[j ^ (lane & 7)];
                z[2 * j] = make_float2(v.x, v.y);
                z[2 * j + 1] = make_float2(v.z, v.w);
            }
        }
        __syncwarp();   // every lane holds its line's values: the region is free
        if (tn < te) stage(id(tn));
        dif_stage<32, 0>(z);
        float m = fft32_rest_max(z);
        if (m > best_v || (LIST && m == best_v && id(t) < best_t)) {
            best_v = m;
            best_t = id(t);
        }
        if (ALL) {
#pragma unroll
            for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == 0) reinterpret_cast<float *>(sm + OFF_RED + grp * 8)[(it & 1) * 8 + warp] = m;
        }
        if (tn < te) {   // the next template's edge columns (all but the newest copy group have landed)
            cp_async_wait_one();
            make_p0();
        }
    }
    if (ALL) {
        sync();
        if (tid == 0 && 2 * pb + grp < te) {
            const int it = (t - 2 - (2 * pb + grp)) / 2;
            const float *r = reinterpret_cast<const float *>(sm + OFF_RED + grp * 8) + (it & 1) * 8;
            float m = r[0];
#pragma unroll
            for (int w = 1; w < 8; ++w) m = fmaxf(m, r[w]);
            peaks_all[(size_t)p * T + t - 2] = m;
        }
    }
    unsigned long long key = best_t >= 0 ? pack_key(best_v, best_t) : 0ull;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long k = __shfl_xor_sync(0xffffffffu, key, o);
        key = k > key ? k : key;
    }
    if (lane == 0 && key) atomicMax(keys + p, key);
}

}  // namespace s128
