// All-pairs search body for N = 64 and 96 in three register rounds on units of
// a few warps (the plan of the 128 search, search128.cuh, for smaller sides).
//
// Paper: the correlation surface of Eqs. 3/6 and its maximum (Fig. 1 B-C).
//
// A unit (64 threads at N = 64, 192 at 96) correlates one template at a time:
// the real surface as N / 2 packed complex lines (rows y and y + N / 2), its
// half spectrum as N / 2 columns (columns 0 and N / 2, real after the column
// transform, packed in one), 32 (24) complex values per thread:
//   round 1: thread (q, l): the products conj(S_t) S_p of stored column q at
//            rows l + 8 m, straight from the template's spectrum in L2 and the
//            pattern's in shared memory; N/8-point transforms over m, twiddle;
//   round 2: thread (k2, g): radix 8 over l, the rows k2 + (N/8) j paired into
//            lines, radix N/32 over the lines' columns g + 32 i, twiddle (g and
//            32 - g together: their columns mirror each other);
//   round 3: lane (line, k3): a 32-point transform; the maximum per thread.
// Rounds 2 and 3 exchange within a warp, so a template takes two barriers of its
// unit, and the eight (four) units of an SM run freely against one another: while
// one waits for its template, the others compute.
#pragma once
#include "common.cuh"
#include "fft128.cuh"
#include "generic.cuh"

namespace rnd {

template <int N>
struct Shape {
    static constexpr int HW = N / 2 + 1, C = N / 2;      // stored columns; columns and lines of a surface
    static constexpr int S1 = N / 32, R1 = N / 8;        // radices
    static constexpr int IPT = N == 64 ? 2 : 1;          // round-2 items (k2, g) per thread
    static constexpr int UT = 2 * N / IPT;               // threads of a unit
    static constexpr int F1 = 8 * C / UT;                // round-1 transforms per thread
    static constexpr int LQ = UT / C;                    // round 1: row residues taken side by side
    static constexpr int K2W = 2 * IPT;                  // k2 per warp in round 2
    static constexpr int REG = K2W * 8 * C;              // a warp's region of the unit's buffer
    static constexpr int LINES = 4 * K2W * S1;           // 32-point lines of a warp (32 at N = 64, 24 at 96)
    static constexpr int BUF = C * N, P0 = UT / 32 * 32; // per unit: buffer; packed-column values, 32 per warp
    static constexpr int TW = 8 * R1 + S1 * 32;          // W^(l k2) at [l][k2], W^(g k3) at [k3][g]
};
// shared memory of a group of nt threads: the pattern, the tables, its units
template <int N>
__host__ __device__ constexpr size_t smem_bytes(int nt) {
    using S = Shape<N>;
    return sizeof(float2) * ((size_t)N * S::HW + S::TW + (size_t)(nt / S::UT) * (S::BUF + S::P0));
}

template <int N>
__device__ __forceinline__ float2 wn(int e) {   // e^{+2 pi i e / N}, 0 <= e < N
    const int r = e < N / 2 ? e : e - N / 2;
    const float2 w = make_float2(kTwTable<N>.re[r], kTwTable<N>.im[r]);
    return e < N / 2 ? w : make_float2(-w.x, -w.y);
}

// 3-point inverse transform
__device__ __forceinline__ void dft3(float2 &a, float2 &b, float2 &c) {
    constexpr float h = 0.86602540378443864676f;   // sqrt(3) / 2
    const float2 s = c_add(b, c), d = c_sub(b, c);
    const float2 t = make_float2(fmaf(-0.5f, s.x, a.x), fmaf(-0.5f, s.y, a.y));
    a = c_add(a, s);
    b = make_float2(fmaf(-h, d.y, t.x), fmaf(h, d.x, t.y));
    c = make_float2(fmaf(h, d.y, t.x), fmaf(-h, d.x, t.y));
}
// R1-point inverse transform in registers; output k is left at x[out<R1>(k)]
template <int R>
__host__ __device__ constexpr int out(int k) {
    return R == 8 ? cx_bitrev(k, 3) : k % 3 * 4 + k / 3;   // 12: X[k1 + 3 k2] at 4 k1 + k2
}
template <int R>
__device__ __forceinline__ void dft_r1(float2 (&x)[R]) {
    if constexpr (R == 8) {
        fft_reg_dif<8, +1>(x);
    } else {   // 12 = 3 x 4: n = 4 n1 + n2, k = k1 + 3 k2
        static_assert(R == 12, "radix 8 or 12");
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) dft3(x[n2], x[4 + n2], x[8 + n2]);   // k1 at 4 k1 + n2
        StaticFor<1, 3>::run([&](auto kk) {
            StaticFor<1, 4>::run([&](auto nn) {
                constexpr int k1 = decltype(kk)::value, n2 = decltype(nn)::value;
                x[4 * k1 + n2] = tw_mul<k1 * n2, 12, +1>(x[4 * k1 + n2]);
            });
        });
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) fft128::dft4<+1>(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);
    }
}

// the k-th column of class g: g, 32 - g, 32 + g; g = 0: the packed column, 16, 32
__device__ __forceinline__ int col_of(int g, int k) { return g ? (k == 0 ? g : k == 1 ? 32 - g : 32 + g) : 16 * k; }

// rows ra and rb at the class's S1 columns -> the packed line Z = Ra + i Rb (Z[N - v]
// = conj Ra + i conj Rb) at the columns g + 32 i (A) and 32 - g (16 for g = 0) + 32 i (B)
template <int S1>
__device__ __forceinline__ void merge_rows(const float2 (&ra)[S1], const float2 (&rb)[S1], bool special,
                                           float2 (&A)[S1], float2 (&B)[S1]) {
    auto zv = [&](int k) { return make_float2(ra[k].x - rb[k].y, ra[k].y + rb[k].x); };
    auto zn = [&](int k) { return make_float2(ra[k].x + rb[k].y, rb[k].x - ra[k].y); };
    const float2 P0 = make_float2(ra[0].x, rb[0].x), PH = make_float2(ra[0].y, rb[0].y);   // columns 0 and N / 2
    B[0] = zv(1);
    if constexpr (S1 == 2) {
        A[0] = zv(0), A[1] = zn(1), B[1] = zn(0);
        if (special) A[0] = P0, A[1] = PH, B[1] = zn(1);
    } else {
        A[0] = zv(0), A[1] = zv(2), A[2] = zn(1), B[1] = zn(2), B[2] = zn(0);
        if (special) A[0] = P0, A[2] = zn(2), B[1] = PH, B[2] = zn(1);
    }
}

__device__ __forceinline__ int idxB(int r, int g) { return (r << 5) + ((((g >> 1) ^ (r & 7)) << 1) | (g & 1)); }

// One work item: pattern p against slot pairs [pb, pe) (slots 2 pb .. min(2 pe, n)
// - 1 of the library, or of the pattern's candidate list; entries < 0 are empty),
// the slots dealt to the group's units in turn.  Runs on the group's threads and
// its shared memory (smem_bytes), with named barriers 5 + (unit of the CTA);
// folds the item's best into keys[p].  ALL: also write every slot's peak to
// peaks_all [P][n].
template <int N, bool ALL>
__device__ void search_body(const float2 *__restrict__ St, int T, const float2 *__restrict__ Sp, int p, int pb, int pe,
                            unsigned long long *__restrict__ keys, float *__restrict__ peaks_all,
                            const int *__restrict__ cand, int kc, const gen::Grp &gr) {
    using S = Shape<N>;
    constexpr int HW = S::HW, C = S::C, S1 = S::S1, R1 = S::R1, F1 = S::F1, UT = S::UT, K2W = S::K2W;
    float2 *sp = reinterpret_cast<float2 *>(gr.smem), *tw1 = sp + N * HW, *tw2 = tw1 + 8 * R1;
    const int unit = gr.t / UT, units = gr.n / UT, tid = gr.t - unit * UT, lane = tid & 31, warp = tid >> 5;
    float2 *buf = tw2 + S1 * 32 + unit * (S::BUF + S::P0), *p0 = buf + S::BUF + warp * 32, *own = buf + warp * S::REG;
    const int bar = 5 + (int)threadIdx.x / UT;
    auto sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(UT) : "memory"); };

    const int q = tid % C, lq = tid / C;                        // round 1: column, row residues lq + LQ i
    const int g = lane & 15, gb = g ? 32 - g : 16, kb = lane >> 4;   // round 2: class; k2 = K2W warp + kb + 2 i
    // the warp whose lanes hold column 0 of residues lq0 + LQ i makes that packed column for itself
    const int lq0 = (32 * warp + 31) / C;
    const bool has0 = lq0 * C >= 32 * warp;
    const int u0 = lane < F1 * R1 ? lq0 + S::LQ * (lane / R1) + 8 * (lane % R1) : 0;

    {   // the pattern's spectrum and the tables
        const float2 *src = Sp + (size_t)p * N * HW;
        for (int i = gr.t; i < N * HW; i += gr.n) sp[i] = src[i];
        for (int i = gr.t; i < 8 * R1; i += gr.n) tw1[i] = wn<N>(i / R1 * (i % R1));        // [l][k2]
        for (int i = gr.t; i < S1 * 32; i += gr.n) tw2[i] = wn<N>((i >> 5) * (i & 31));     // [k3][g]
    }
    gr.sync();
    const int n = cand ? kc : T, end = min(2 * pe, n);
    float best_v = -INFINITY;
    int best_t = -1;
    for (int s = 2 * pb + unit; s < end; s += units) {
        const int t = cand ? cand[(size_t)p * kc + s] : s;
        if (t < 0) {   // uniform over the unit
            if (ALL && tid == 0) peaks_all[(size_t)p * n + s] = -INFINITY;
            continue;
        }
        const float2 *tp = St + (size_t)t * N * HW;
        // ---- round 1
        float2 x[F1][R1];
#pragma unroll
        for (int i = 0; i < F1; ++i)
#pragma unroll
            for (int m = 0; m < R1; ++m) x[i][m] = __ldg(tp + (lq + S::LQ * i + 8 * m) * HW + q);
        if (has0) {   // the packed column X[u][0] + i X[u][N / 2] at the warp's rows
            const float2 a = c_mulcj(__ldg(tp + u0 * HW), sp[u0 * HW]);
            const float2 h = c_mulcj(__ldg(tp + u0 * HW + C), sp[u0 * HW + C]);
            p0[lane] = make_float2(a.x - h.y, a.y + h.x);
            __syncwarp();
        }
#pragma unroll
        for (int i = 0; i < F1; ++i) {
#pragma unroll
            for (int m = 0; m < R1; ++m) x[i][m] = c_mulcj(x[i][m], sp[(lq + S::LQ * i + 8 * m) * HW + q]);
            if (q == 0) {
#pragma unroll
                for (int m = 0; m < R1; ++m) x[i][m] = p0[i * R1 + m];
            }
            dft_r1<R1>(x[i]);
        }
        sync();   // the previous template's lines have been read: the buffer is free
#pragma unroll
        for (int i = 0; i < F1; ++i) {
            const int l = lq + S::LQ * i;
            StaticFor<0, R1>::run([&](auto kk) {
                constexpr int k2 = decltype(kk)::value;
                const float2 v = x[i][out<R1>(k2)];
                buf[(k2 / K2W) * S::REG + l * (K2W * C) + (k2 % K2W) * C + q] = k2 ? c_mul(v, tw1[l * R1 + k2]) : v;
            });
        }
        sync();
        // ---- round 2
        float2 y[S::IPT][S1][8];
#pragma unroll
        for (int i = 0; i < S::IPT; ++i)
#pragma unroll
            for (int k = 0; k < S1; ++k) {
                const float2 *src = own + (kb + 2 * i) * C + col_of(g, k);
#pragma unroll
                for (int l = 0; l < 8; ++l) y[i][k][l] = src[l * (K2W * C)];
            }
        __syncwarp();   // the warp has read its columns: its region is free
#pragma unroll
        for (int i = 0; i < S::IPT; ++i) {
#pragma unroll
            for (int k = 0; k < S1; ++k) fft_reg_dif<8, +1>(y[i][k]);   // row k2 + R1 j at bitrev(j)
            StaticFor<0, 4>::run([&](auto jj) {
                constexpr int j = decltype(jj)::value, RA = cx_bitrev(j, 3), RB = cx_bitrev(j + 4, 3);
                float2 ra[S1], rb[S1], A[S1], B[S1];
#pragma unroll
                for (int k = 0; k < S1; ++k) ra[k] = y[i][k][RA], rb[k] = y[i][k][RB];
                merge_rows<S1>(ra, rb, g == 0, A, B);
                if constexpr (S1 == 2) {
                    const float2 a = A[0], b = B[0];
                    A[0] = c_add(a, A[1]), A[1] = c_sub(a, A[1]);
                    B[0] = c_add(b, B[1]), B[1] = c_sub(b, B[1]);
                } else {
                    dft3(A[0], A[1], A[2]);
                    dft3(B[0], B[1], B[2]);
                }
                const int r = (j * K2W + kb + 2 * i) * S1;
                own[idxB(r, g)] = A[0];
                own[idxB(r, gb)] = B[0];
#pragma unroll
                for (int k3 = 1; k3 < S1; ++k3) {
                    own[idxB(r + k3, g)] = c_mul(A[k3], tw2[k3 * 32 + g]);
                    own[idxB(r + k3, gb)] = c_mul(B[k3], tw2[k3 * 32 + gb]);
                }
            });
        }
        __syncwarp();
        // ---- round 3
        float m = -INFINITY;
        if (S::LINES == 32 || lane < S::LINES) {
            float2 z[32];
            const float4 *line = reinterpret_cast<const float4 *>(own) + (lane << 4);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const float4 v = line[j ^ (lane & 7)];
                z[2 * j] = make_float2(v.x, v.y);
                z[2 * j + 1] = make_float2(v.z, v.w);
            }
            fft_reg_dif<32, +1>(z);
#pragma unroll
            for (int j = 0; j < 32; ++j) m = fmaxf(m, fmaxf(z[j].x, z[j].y));
        }
        if (m > best_v || (m == best_v && t < best_t)) {
            best_v = m;
            best_t = t;
        }
        if (ALL) {   // the packed column's buffer carries the warps' maxima
#pragma unroll
            for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == 0) p0[0].x = m;
            sync();
            if (tid == 0) {
                for (int w = 1; w < UT / 32; ++w) m = fmaxf(m, p0[32 * w].x);
                peaks_all[(size_t)p * n + s] = m;
            }
            sync();
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

}  // namespace rnd
