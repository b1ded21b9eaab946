// Zero-shift correlation screen on the 5th-generation tensor cores.
//
// Paper: Eq. 1 (the normalised dot product is the correlation at zero shift)
// and Eq. 3 (the FFT cross-correlation it is a special case of).  Score[p, t]
// = <y_p, y_t>, the inner product of the unit-norm filtered, windowed spatial
// images, is r(0) of the XCF surface; computed here as a GEMM
// S = Yp . Yt^T with BF16 operands and FP32 accumulation, it ranks the
// library cheaply before the FP32 FFT cross-correlation rescores the best k.
//
// k_screen_tc: one CTA (128 threads) computes a 128 (patterns) x 256
// (templates) tile of S, or two CTAs a 256 x 256 tile.  Warp 0 is the loader:
// one thread issues TMA (cp.async.bulk.tensor) copies of 64-wide K-slices of
// both operands into a ring of stages, 128-byte swizzled, each stage completing
// an mbarrier by transaction count.  Warp 1 is the tensor-core issuer: one thread
// waits for a stage, issues four tcgen05.mma (K = 16, BF16 in, FP32 accumulated in
// 256 TMEM columns) and commits them to the stage's "empty" mbarrier, which hands
// the stage back to the loader.  After the last commit all four warps read the
// accumulator with tcgen05.ld (each warp its 32 TMEM lanes = tile rows) and
// write S.  Tiles are ordered in groups of eight pattern tiles, so that the CTAs
// resident at one time share the template tiles they stream.  Every wait is
// bounded: on time-out the kernel records an error flag, waits (bounded) for its
// copies in flight and frees its tensor memory.
//
// What bounds it: shared-memory traffic of the operands with one CTA per tile (per
// K-slice 48 KB in by TMA and 48 KB out to the tensor core, 768 cycles of the 128
// bytes a cycle against 512 of MMA).  A pair holds half of the template slice in
// each CTA (32 KB in and out, 512 cycles): rank 0 issues instructions that read both
// CTAs' shared memory and write both accumulators; rank 1's second warp passes
// "stage loaded" on to it, releasing only shared memory (a full release at each
// stage waits a microsecond: 4.7 ms instead of 1.5).  2,000 patterns x 39,784
// templates at K = 16,384: 1.88 -> 1.65 ms by storing S through shared memory, a row
// at a time, -> 1.50 by pairs (1.74 PFLOP/s, 90 % of the measured BF16 burst);
// 1,000 x 19,944 at K = 65,536: 1.86 -> 1.77 -> 1.65 (5 rounds of tiles for 4.1).
// Template tiles of 224 there: 1.63, but 1.64 against 1.50 for the former: 256.
#include <cuda.h>
#include <cuda_bf16.h>

#include "cluster.cuh"
#include "common.cuh"
#include "kernels.cuh"

namespace {

constexpr int BM = 128, BN = 256, BK = 64, NT = 128, GROUP_M = 8;
constexpr int A_BYTES = BM * BK * 2;              // 16 KB
constexpr unsigned kSpinLimit = 1u << 26;         // bounded waits

// CG CTAs work on one tile: 128 CG patterns x 256 templates
template <int CG>
struct Ring {
    static constexpr int STAGE_BYTES = A_BYTES + BN / CG * BK * 2, STAGES = CG == 1 ? 4 : 6;   // 48 or 32 KB
    static constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 1024 + 256;
};

// shared-memory matrix descriptor of a K-major operand tile written by TMA
// with 128-byte swizzling: start address, leading byte offset 16 (unused for
// this layout), stride byte offset 1024 (between 8-row groups), version 1,
// swizzle mode 2 = 128 B.  Stage bases are 1024-byte aligned, so advancing
// the start by 32 bytes per K = 16 step keeps the swizzle phase.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}

// instruction descriptor of kind::f16: D = F32, A = B = BF16, both K-major,
// N = 256, M = 128 per CTA
template <int CG>
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                            ((uint32_t)(CG * BM >> 4) << 24);

__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity) {
    for (unsigned spin = 0; spin < kSpinLimit; ++spin) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred P;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 P, [%1], %2;\n selp.b32 %0, 1, 0, P;\n}\n"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// 2-D tiled TMA load: box at (x = K element, y = row), completes `bar` by transaction bytes
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// arrives on the barrier (of every CTA of the tile) when all MMAs issued so far have completed
template <int CG>
__device__ __forceinline__ void commit(uint32_t bar) {
    if constexpr (CG == 1)
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar));
    else
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
            "h"((uint16_t)3));
}

template <int CG>
__global__ void __launch_bounds__(NT, 1)
k_screen_tc(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, int P, int T, int K,
            float *__restrict__ S, int *__restrict__ err) {
    using R = Ring<CG>;
    constexpr int STAGES = R::STAGES;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t sbase0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const uint32_t sbase = (sbase0 + 1023u) & ~1023u;            // 1024-aligned stages (swizzle atoms)
    const uint32_t full_bar = sbase + STAGES * R::STAGE_BYTES;    // STAGES mbarriers: stage loaded
    const uint32_t empty_bar = full_bar + 8 * STAGES;             // STAGES mbarriers: stage consumed
    const uint32_t peer_bar = empty_bar + 8 * STAGES;             // rank 0: STAGES mbarriers: the peer's stage loaded
    const uint32_t done_bar = peer_bar + 8 * STAGES;              // accumulator complete
    const uint32_t tmem_slot = done_bar + 8;                      // tcgen05.alloc writes here
    unsigned char *gen_base = smem_raw + (sbase - sbase0);
    unsigned char *gen_bars = gen_base + STAGES * R::STAGE_BYTES;
    volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(gen_bars + 24 * STAGES + 8);
    volatile int *flag = reinterpret_cast<volatile int *>(gen_bars + 24 * STAGES + 16);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = CG == 1 ? 0 : (int)cluster_rank();
    // grouped tile order: GROUP_M / CG pattern tiles per template-tile sweep
    const int num_m = (P + CG * BM - 1) / (CG * BM), num_n = (T + BN - 1) / BN;
    const int id = blockIdx.x / CG, per_group = GROUP_M / CG * num_n;
    const int first_m = (id / per_group) * (GROUP_M / CG);
    const int gsize = min(num_m - first_m, GROUP_M / CG);
    const int m_tile = first_m + (id % per_group) % gsize, n_tile = (id % per_group) / gsize;
    const int p0 = (m_tile * CG + rank) * BM, t0 = n_tile * BN;   // this CTA's rows of A and of S
    const int nk = K / BK;

    if (tid == 0) {
        for (int s = 0; s < 3 * STAGES + 1; ++s) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full_bar + 8 * s));
        asm volatile("fence.mbarrier_init.release.cluster;");
        *flag = 0;
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapB)) : "memory");
    }
    if (warp == 0) {
        if constexpr (CG == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(BN));
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        } else {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(BN));
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if constexpr (CG == 2) {   // both CTAs' barriers are initialised and their tensor memory allocated
        cluster_arrive();
        cluster_wait();
    }
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot_ptr;

    int issued = 0;   // loader: stages issued (for the drain on a time-out)
    if (warp == 0 && lane == 0) {
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % STAGES;
            if (kb >= STAGES && !mbar_wait(empty_bar + 8 * s, (uint32_t)((kb / STAGES - 1) & 1))) {
                *flag = 1;
                break;
            }
            if (*flag) break;
            const uint32_t sa = sbase + s * R::STAGE_BYTES, sb = sa + A_BYTES;
            mbar_expect_tx(full_bar + 8 * s, R::STAGE_BYTES);
            tma_load_2d(sa, &mapA, kb * BK, p0, full_bar + 8 * s);
            tma_load_2d(sb, &mapB, kb * BK, t0 + rank * (BN / CG), full_bar + 8 * s);
            issued = kb + 1;
        }
        // rank 0's commits arrive on this CTA's barriers: they have before it leaves
        if (CG == 2)
            for (int kb = max(0, nk - STAGES); kb < issued && issued == nk; ++kb)
                if (!mbar_wait(empty_bar + 8 * (kb % STAGES), (uint32_t)((kb / STAGES) & 1))) {
                    *flag = 1;
                    break;
                }
    } else if (warp == 1 && lane == 0 && rank == 1) {
        // this half of every stage is there: tell rank 0, whose tensor core instructions read both halves
        const uint32_t remote = map_to_rank(gen_bars + 16 * STAGES, 0);
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % STAGES;
            if (!mbar_wait(full_bar + 8 * s, (uint32_t)((kb / STAGES) & 1)) || *flag) {
                *flag = 1;
                break;
            }
            asm volatile(
                "fence.release.sync_restrict::shared::cta.cluster;\n"
                "mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote + 8 * s)
                : "memory");
        }
    } else if (warp == 1 && lane == 0) {
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % STAGES;
            const uint32_t par = (uint32_t)((kb / STAGES) & 1);
            if (!mbar_wait(full_bar + 8 * s, par) || (CG == 2 && !mbar_wait(peer_bar + 8 * s, par)) || *flag) {
                *flag = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t sa = sbase + s * R::STAGE_BYTES, sb = sa + A_BYTES;
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {
                const uint64_t ad = smem_desc_sw128(sa + kk * 32), bd = smem_desc_sw128(sb + kk * 32);
                const uint32_t acc = (kb > 0 || kk > 0) ? 1u : 0u;
                if constexpr (CG == 1)
                    asm volatile(
                        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                        "l"(ad), "l"(bd), "r"(kIdesc<CG>), "r"(acc));
                else
                    asm volatile(
                        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                        "l"(ad), "l"(bd), "r"(kIdesc<CG>), "r"(acc));
            }
            commit<CG>(empty_bar + 8 * s);
        }
        // the done barrier fires when every MMA issued above has completed
        commit<CG>(done_bar);
    }
    __syncwarp();
    bool ok = mbar_wait(done_bar, 0u);
    if (!ok) *flag = 1;
    __syncthreads();
    const bool good = *flag == 0;
    if (!good && warp == 0 && lane == 0) {
        // drain: every issued stage's copies must land before the shared memory is released
        for (int kb = 0; kb < issued; ++kb) {
            const int s = kb % STAGES;
            if (kb + STAGES >= issued) mbar_wait(full_bar + 8 * s, (uint32_t)((kb / STAGES) & 1));
        }
        atomicExch(err, 1);
    }
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (good) {
        // 32 columns at a time through shared memory (the stages are consumed), so that a
        // warp stores 128 bytes of one row: a lane per row would touch 32 rows per store
        float *sh = reinterpret_cast<float *>(gen_base) + warp * 32 * 33;
#pragma unroll 1
        for (int c0 = 0; c0 < BN; c0 += 32) {
            uint32_t v[32];
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
                "[%32];"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                  "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                  "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),
                  "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),
                  "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                : "r"(taddr));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 32; ++j) sh[lane * 33 + j] = __uint_as_float(v[j]);
            __syncwarp();
            const int t = t0 + c0 + lane, rows = min(32, P - p0 - warp * 32);
            if (t < T) {
                float *dst = S + (size_t)(p0 + warp * 32) * T + t;
#pragma unroll 8
                for (int r = 0; r < rows; ++r) dst[(size_t)r * T] = sh[r * 33 + lane];
            }
            __syncwarp();
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if constexpr (CG == 1) {
        if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN));
    } else {
        cluster_arrive();   // neither CTA frees its memory while the other may still use it
        cluster_wait();
        if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN));
    }
}

// --------------------------------------------------------------------------
// top-k of each row of S (k <= 64) by (score desc, index asc), on
// order-preserving 32-bit keys held in registers, NV per thread (the row is read
// once, with every load in flight).  The k-th largest of the maxima of 64 groups
// of eight threads is a lower bound of the k-th largest key, so only the few keys at
// or above it go on (about 130 of 40,000 at k = 32) and are ranked by counting.
// Rows where more than kTopList keys remain (long runs of equal scores) find the
// k-th largest key by a 4-pass radix select over the row first.
// Bound by reading the row: the earlier kernel (radix select on a copy of the row
// in shared memory, one 256-thread CTA per SM at 39,784 templates) took 946 us
// for 2,000 rows of 39,784, this one 163 us (the scores are 318 MB: 47 us at the
// measured copy rate).
constexpr int TK_THREADS = 512;
constexpr int kTopList = 2048;

template <int NV>
__global__ void __launch_bounds__(TK_THREADS, 1) k_topk_rows(const float *__restrict__ S, int P, int T, int k,
                                                             int *__restrict__ cand, float *__restrict__ score) {
    __shared__ unsigned long long list[kTopList];   // (key, ~index)
    __shared__ uint32_t gmax[64], hist[256], s_tau, s_need;
    __shared__ int s_count, wcount[TK_THREADS / 32];
    const int p = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float *row = S + (size_t)p * T;
    const int kk = min(k, T);
    uint32_t v[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int i = tid + j * TK_THREADS;
        v[j] = i < T ? float_to_ordered(__ldcs(row + i)) : 0u;
    }
    uint32_t m = 0;
#pragma unroll
    for (int j = 0; j < NV; ++j) m = max(m, v[j]);
#pragma unroll
    for (int o = 4; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((lane & 7) == 0) gmax[tid >> 3] = m;
    if (tid == 0) s_count = 0;
    __syncthreads();
    if (tid < 64) {
        const uint32_t g = gmax[tid];
        int r = 0;
        for (int j = 0; j < 64; ++j) r += gmax[j] > g || (gmax[j] == g && j < tid);
        if (r == kk - 1) s_tau = g;
    }
    __syncthreads();
    auto push = [&](int slot, uint32_t key, int i) {
        if (slot < kTopList) list[slot] = ((unsigned long long)key << 32) | (0xffffffffu - (uint32_t)i);
    };
    uint32_t tau = s_tau;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int i = tid + j * TK_THREADS;
        if (i < T && v[j] >= tau) push(atomicAdd(&s_count, 1), v[j], i);
    }
    __syncthreads();
    if (s_count > kTopList) {   // uniform
        __syncthreads();
        if (tid == 0) {
            s_tau = 0;
            s_need = (uint32_t)kk;
            s_count = 0;
        }
        uint32_t mask = 0;
        for (int shift = 24; shift >= 0; shift -= 8) {
            if (tid < 256) hist[tid] = 0;
            __syncthreads();
            const uint32_t pre = s_tau;
            for (int i = tid; i < T; i += TK_THREADS) {
                const uint32_t key = float_to_ordered(row[i]);
                if ((key & mask) == pre) atomicAdd(&hist[(key >> shift) & 255], 1u);
            }
            __syncthreads();
            if (tid == 0) {
                uint32_t need = s_need, d = 255;
                for (;; --d) {   // from the top digit down
                    if (hist[d] >= need || d == 0) break;
                    need -= hist[d];
                }
                s_tau = pre | (d << shift);
                s_need = need;
            }
            mask |= 255u << shift;
            __syncthreads();
        }
        tau = s_tau;   // the kk-th largest key: the keys above it (fewer than kk) ...
        const int need = (int)s_need;
        for (int i = tid; i < T; i += TK_THREADS) {
            const uint32_t key = float_to_ordered(row[i]);
            if (key > tau) push(atomicAdd(&s_count, 1), key, i);
        }
        __syncthreads();
        const int ngt = s_count;
        // ... and the lowest indices equal to it, ranked by warp ballots in index order
        for (int base = 0, taken = 0; base < T && taken < need; base += TK_THREADS) {
            const int i = base + tid;
            const bool eq = i < T && float_to_ordered(row[i]) == tau;
            const unsigned bal = __ballot_sync(0xffffffffu, eq);
            if (lane == 0) wcount[warp] = __popc(bal);
            __syncthreads();
            int before = __popc(bal & ((1u << lane) - 1u)), tot = 0;
            for (int w = 0; w < TK_THREADS / 32; ++w) {
                if (w < warp) before += wcount[w];
                tot += wcount[w];
            }
            if (eq && taken + before < need) push(ngt + taken + before, tau, i);
            taken += tot;   // the same in every thread
            __syncthreads();
        }
        if (tid == 0) s_count = kk;
        __syncthreads();
    }
    const int n = s_count;   // at least kk: the groups at or above tau each hold one
    for (int e = tid; e < n; e += TK_THREADS) {
        const unsigned long long key = list[e];
        int r = 0;
        for (int j = 0; j < n; ++j) r += list[j] > key;
        if (r < kk) {
            cand[(size_t)p * k + r] = (int)(0xffffffffu - (uint32_t)key);
            score[(size_t)p * k + r] = ordered_to_float((uint32_t)(key >> 32));
        }
    }
    if (tid >= kk && tid < k) {
        cand[(size_t)p * k + tid] = -1;
        score[(size_t)p * k + tid] = -INFINITY;
    }
}

__global__ void k_to_bf16(const float *__restrict__ x, size_t n, __nv_bfloat16 *__restrict__ y) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

}  // namespace

namespace {
// cuTensorMapEncodeTiled through the runtime's driver entry point (no link to libcuda)
typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encode_fn() {
    static EncodeTiled fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    }
    return fn;
}
// rows x K BF16 matrix (row-major), boxes of box_rows x 64 (128 bytes, the swizzle span)
bool make_map(CUtensorMap *m, const void *base, int rows, int K, int box_rows) {
    EncodeTiled f = encode_fn();
    if (!f) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return f(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace

cudaError_t launch_screen_tc(const void *A, int P, const void *B, int T, int K, float *S, int *err,
                             cudaStream_t st) {
    if (P <= 0 || T <= 0) return cudaSuccess;
    // TMA: 16-byte aligned bases and row strides; K a multiple of the 64-element slice
    if (K % BK || (reinterpret_cast<uintptr_t>(A) & 15) || (reinterpret_cast<uintptr_t>(B) & 15))
        return cudaErrorInvalidValue;
    // Two CTAs per tile where every CTA has patterns (an even number of 128-pattern
    // tiles), the tiles fill the SMs more than once and K is long.  One CTA against two,
    // K = 4,096, 20,000 templates: 256 patterns 68 -> 66 us, 1,200 (10,000 templates) 94
    // -> 88; but 128 patterns 41 -> 64, 1,400 (11 tiles) 181 -> 194, 256 x 3,000 27 -> 31
    // (the pair starts later).  K = 16,384, 2,000 x 39,784: 1.65 -> 1.50 ms.
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long num_m = (P + BM - 1) / BM, tiles = num_m * ((T + BN - 1) / BN);
    const bool pair = num_m % 2 == 0 && tiles > sms && K >= 4096;
    CUtensorMap ma, mb;
    if (!make_map(&ma, A, P, K, BM) || !make_map(&mb, B, T, K, pair ? BN / 2 : BN)) return cudaErrorInvalidValue;
    if (tiles > 0x7fffffffL) return cudaErrorInvalidValue;
    if (pair) return launch_clusters(k_screen_tc<2>, 2, NT, Ring<2>::SMEM, tiles / 2, st, ma, mb, P, T, K, S, err);
    e = cudaFuncSetAttribute(k_screen_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Ring<1>::SMEM);
    if (e != cudaSuccess) return e;
    k_screen_tc<1><<<(unsigned)tiles, NT, Ring<1>::SMEM, st>>>(ma, mb, P, T, K, S, err);
    return cudaGetLastError();
}

cudaError_t launch_topk_rows(const float *S, int P, int T, int k, int *cand, float *score, cudaStream_t st) {
    if (P <= 0) return cudaSuccess;
    if (k < 1 || k > 64) return cudaErrorInvalidValue;
    const int nv = (T + TK_THREADS - 1) / TK_THREADS;
    // registers for NV keys per thread; the callers admit 51,200 templates
    if (nv <= 4) k_topk_rows<4><<<P, TK_THREADS, 0, st>>>(S, P, T, k, cand, score);
    else if (nv <= 10) k_topk_rows<10><<<P, TK_THREADS, 0, st>>>(S, P, T, k, cand, score);
    else if (nv <= 20) k_topk_rows<20><<<P, TK_THREADS, 0, st>>>(S, P, T, k, cand, score);
    else if (nv <= 40) k_topk_rows<40><<<P, TK_THREADS, 0, st>>>(S, P, T, k, cand, score);
    else if (nv <= 60) k_topk_rows<60><<<P, TK_THREADS, 0, st>>>(S, P, T, k, cand, score);
    else if (nv <= 80) k_topk_rows<80><<<P, TK_THREADS, 0, st>>>(S, P, T, k, cand, score);
    else if (nv <= 100) k_topk_rows<100><<<P, TK_THREADS, 0, st>>>(S, P, T, k, cand, score);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_to_bf16(const float *x, size_t n, void *y, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const size_t blocks = (n + 255) / 256 < 65536 ? (n + 255) / 256 : 65536;
    k_to_bf16<<<(unsigned)blocks, 256, 0, st>>>(x, n, static_cast<__nv_bfloat16 *>(y));
    return cudaGetLastError();
}
