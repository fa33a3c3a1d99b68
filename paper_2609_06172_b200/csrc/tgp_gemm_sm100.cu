// GEMM on the 5th-generation tensor cores (sm_100a): C[M, n] (=|+=) A[M, K] * W[n, K]^T,
// bf16 operands, fp32 accumulation in tensor memory.  tgpk_gemm_tc() and tgpk_gemm_tc_list() choose between
//   tgp_wstream_tc_kernel         one tile of 128 weight rows x up to 128 activation rows per CTA, K in 1, 2 or 4 slices: up to 128
//                                 activation rows, and more of them on few tiles with a long K;
//   tgp_matmul_tc_pair_kernel     tiles of 256 weight rows x up to 256 activation rows on the two SMs of a CTA pair, or shared by two pairs: the rest;
//   tgp_matmul_tc_kernel          one narrow tile per CTA (below): more than 128 activation rows on few tiles, launched alone.
// tgp_matmul_tc_persistent_kernel and the other forms of tgp_matmul_tc_kernel run by request only (tgp_k_gemm_tc_variant): they
// cross-check the others.
//
// tgp_matmul_tc_kernel:
// One CTA computes a 128 x BN tile.  Warp 0 (one elected thread) feeds a shared-memory ring of ST stages with TMA
// (128-byte swizzle, 64 bf16 of K per stage); warp 1 (one elected thread) issues tcgen05.mma (M=128, N=BN, K=16,
// four per stage) into a TMEM accumulator and releases stages with tcgen05.commit; warps 2-5 wait for the
// last commit, read the accumulator with tcgen05.ld (each warp its own 32-lane quarter) and store fp32 rows.
// Out-of-range rows / columns / K are zero-filled by TMA and masked in the epilogue, so any M, n and
// any K % 8 == 0 work.  Every mbarrier wait is bounded in time: a wait that runs out records an error code
// and the CTA drains and returns instead of hanging the GPU.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <algorithm>
#include <cstdint>
#include <cstring>
#include "tgp.h"
#include "tgp_kernels.h"
#include "tgp_sm100.cuh"

namespace {

using namespace tgp_sm100;
constexpr int BK = 64, GROUP_M = 16;

__device__ int g_gemm_tc_error = 0;                    // 0 ok; else (role << 8) | stage of the first wait that ran out

// Optional epilogue: the accumulator is the up projection u of a SwiGLU FFN and the gate projection g of the same
// elements is already in memory (fp32, same geometry as C).  Instead of storing u, the epilogue stores
// a = bf16(g / (1 + exp(-g)) * u) - the arithmetic of the stand-alone SwiGLU kernel, on the very values it would have
// read - so u never goes to memory, g is read once instead of twice and the SwiGLU launch disappears.
struct Epi { const float *gate; __nv_bfloat16 *aout; };

// 32 consecutive elements of one output row, element offset `off` in C's geometry, `cnt` of them inside the matrix
__device__ __forceinline__ void swiglu_store32(const Epi &ep, size_t off, const float *v, uint32_t cnt) {
    const float *g = ep.gate + off;
    __nv_bfloat16 *a = ep.aout + off;
    if (cnt == 32 && (off & 7) == 0 && ((reinterpret_cast<uintptr_t>(ep.gate) | reinterpret_cast<uintptr_t>(ep.aout)) & 15u) == 0) {
#pragma unroll
        for (int j = 0; j < 32; j += 8) {
            const float4 g0 = *reinterpret_cast<const float4 *>(g + j), g1 = *reinterpret_cast<const float4 *>(g + j + 4);
            const float gv[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                __nv_bfloat162 pk = __floats2bfloat162_rn(gv[2 * i] / (1.0f + expf(-gv[2 * i])) * v[j + 2 * i],
                                                          gv[2 * i + 1] / (1.0f + expf(-gv[2 * i + 1])) * v[j + 2 * i + 1]);
                w[i] = *reinterpret_cast<uint32_t *>(&pk);
            }
            *reinterpret_cast<uint4 *>(a + j) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else {
        for (uint32_t j = 0; j < cnt; ++j) a[j] = __float2bfloat16_rn(g[j] / (1.0f + expf(-g[j])) * v[j]);
    }
}

template <int BN, int ST, int KH>
struct Smem {
    static constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, HALF_BYTES = A_BYTES + B_BYTES, STAGE_BYTES = KH * HALF_BYTES;
    static constexpr int BAR_OFF = ST * STAGE_BYTES;
    static constexpr int TOTAL = BAR_OFF + 256 + 1024;        // barriers (2 * ST + 1, TMEM slot, flag) + slack to align the base to 1024 bytes
};

// (ST stages of KH 64-wide K blocks each: with KH = 2 the producer and the MMA thread meet half as often)
// SWAP: the operands trade places - the tile's 128 rows are weight rows (M counts them), its BN columns activation rows
// (n counts them) - and the tile is stored transposed, C[activation row][col0 + weight row].  For products of up to 128
// activation rows a CTA then streams 128 weight rows through its TMA ring instead of BN, which is what such a product
// is bound by.
template <int BN, int ST, int KH, bool SWAP>
__global__ void __launch_bounds__(192) tgp_matmul_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                                                      float *__restrict__ C, uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate, const Epi ep) {
    extern __shared__ uint8_t smem_raw[];
    using S = Smem<BN, ST, KH>;
    constexpr int STAGES = ST;                      // depth of this instantiation's TMA ring
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + S::BAR_OFF);
    uint64_t *empty = full + STAGES;
    uint64_t *acc_full = empty + STAGES;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_full + 1);
    volatile uint32_t *failed = tmem_slot + 1;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Tile order: groups of GROUP_M row tiles are swept across all column tiles before the next group starts, so the
    // CTAs in flight together share a few A panels and a few W panels that fit in L2 (instead of re-streaming A from
    // HBM once per column tile when M is large).
    const uint32_t tiles_m = (M + BM - 1) / BM, tiles_n = (n + BN - 1) / BN;
    const uint32_t group = blockIdx.x / (GROUP_M * tiles_n), first_m = group * GROUP_M;
    const uint32_t rows_in_group = min((uint32_t)GROUP_M, tiles_m - first_m);
    const uint32_t in_group = blockIdx.x - group * GROUP_M * tiles_n;
    const uint32_t m0 = (first_m + in_group % rows_in_group) * BM, n0 = (in_group / rows_in_group) * BN;
    const uint32_t num_k = (K + KH * BK - 1) / (KH * BK);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(acc_full, 1);
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");     // not before the allocation: see tgp_sm100.cuh
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (elect_one()) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            uint32_t armed = 0;
            const uint32_t withhold = blockIdx.x == 0 ? (uint32_t)g_withhold_step : 0xffffffffu;     // test hook: this stage is never loaded
            for (uint32_t kb = 0; kb < num_k; ++kb) {
                const uint32_t s = kb % STAGES, ph = (kb / STAGES) & 1;
                if (kb == withhold) break;
                if (!mbar_wait(&empty[s], ph ^ 1, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (1 << 8) | (int)s); } break; }
                mbar_expect_tx(&full[s], S::STAGE_BYTES);
#pragma unroll
                for (int h = 0; h < KH; ++h) {
                    tma_load_2d(smem + s * S::STAGE_BYTES + h * S::HALF_BYTES, &tmA, (int)((kb * KH + h) * BK), (int)m0, &full[s]);
                    tma_load_2d(smem + s * S::STAGE_BYTES + h * S::HALF_BYTES + S::A_BYTES, &tmB, (int)((kb * KH + h) * BK), (int)n0, &full[s]);
                }
                armed = kb + 1;
            }
            if (*failed) {
                // let the copies this thread started land before the CTA's shared memory is given up
                volatile uint32_t never = 0;
                for (uint32_t kb = armed > STAGES ? armed - STAGES : 0; kb < armed; ++kb) mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1, &never);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            asm volatile("griddepcontrol.wait;" ::: "memory");    // the limit of its waits counts from here
            constexpr uint32_t idesc = umma_idesc(BN);
            bool ok = true;
            for (uint32_t kb = 0; kb < num_k && ok; ++kb) {
                const uint32_t s = kb % STAGES, ph = (kb / STAGES) & 1;
                if (!mbar_wait(&full[s], ph, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (2 << 8) | (int)s); } ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (uint32_t h = 0; h < KH; ++h) {
                    const uint64_t da = umma_desc(smem_u32(smem + s * S::STAGE_BYTES + h * S::HALF_BYTES));
                    const uint64_t db = umma_desc(smem_u32(smem + s * S::STAGE_BYTES + h * S::HALF_BYTES + S::A_BYTES));
#pragma unroll
                    for (uint32_t k = 0; k < BK / 16; ++k) umma(tmem_base, da + 2 * k, db + 2 * k, idesc, (kb | h | k) != 0);   // +32 bytes of K per step
                }
                umma_commit(&empty[s]);
            }
            if (ok) umma_commit(acc_full);
        }
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");        // what C, the gate and a hold is the previous kernel's work
        bool ready = !*failed && mbar_wait(acc_full, 0, failed);
        if (!ready && !*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, 3 << 8); }
        ready = __all_sync(0xffffffffu, ready && !*failed);      // tcgen05.ld is warp-collective: decide per warp
        if (ready) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t quarter = warp & 3;                    // TMEM lanes this warp may read
            const uint32_t row = m0 + quarter * 32 + lane;
            const bool vec = ((ldc | col0) & 3u) == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0;
#pragma unroll 1
            for (uint32_t c = 0; c < BN / 32; ++c) {
                float v[32];
                tmem_ld32(tmem_base + ((quarter * 32) << 16) + c * 32, v);
                if (SWAP) {
                    // a warp's 32 lanes hold 32 consecutive weight rows: for each activation row they write 128 contiguous bytes
                    if (row < M) {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (n0 + c * 32 + j < n) {
                                float *d = C + (size_t)(n0 + c * 32 + j) * ldc + col0 + row;
                                *d = accumulate ? *d + v[j] : v[j];
                            }
                    }
                } else if (row < M) {
                    float *dst = C + (size_t)row * ldc + col0 + n0 + c * 32;
                    const uint32_t col = n0 + c * 32;
                    if (ep.aout) { if (col < n) swiglu_store32(ep, (size_t)row * ldc + col0 + col, v, min(32u, n - col)); }
                    else if (vec && col + 32 <= n) {
#pragma unroll
                        for (int j = 0; j < 32; j += 4) {
                            float4 o = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                            if (accumulate) { const float4 old = *reinterpret_cast<const float4 *>(dst + j); o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w; }
                            *reinterpret_cast<float4 *>(dst + j) = o;
                        }
                    } else {
                        // (a lane's row is a line of its own, and what L1 the ring leaves does not keep them from one element to the next: the old sums are all
                        // requested before the first is stored)
                        if (accumulate) {
                            float old[32];
#pragma unroll
                            for (int j = 0; j < 32; ++j) old[j] = col + j < n ? dst[j] : 0.f;
#pragma unroll
                            for (int j = 0; j < 32; ++j) v[j] = old[j] + v[j];
                        }
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (col + j < n) dst[j] = v[j];
                    }
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)BN) : "memory");
    }
}

// ---- persistent variant for large problems ------------------------------------------------------------------
// One CTA per SM walks 128 x 256 tiles (grouped order as above).  Four TMA stages of 48 KB; the TMEM holds two
// 256-column accumulators, so the MMA warp starts the next tile while the four epilogue warps drain the previous
// one (acc_full / acc_empty barriers per buffer).  Same bounded waits and error word as the kernel above.
constexpr int P_BN = 256, P_STAGES = 4;

__global__ void __launch_bounds__(192, 1) tgp_matmul_tc_persistent_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                                                                    float *__restrict__ C, uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate, const Epi ep) {
    extern __shared__ uint8_t smem_raw[];
    constexpr int A_BYTES = BM * BK * 2, B_BYTES = P_BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + P_STAGES * STAGE_BYTES);
    uint64_t *empty = full + P_STAGES;
    uint64_t *acc_full = empty + P_STAGES;           // [2]
    uint64_t *acc_empty = acc_full + 2;              // [2]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 2);
    volatile uint32_t *failed = tmem_slot + 1;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t num_k = (K + BK - 1) / BK;
    const uint32_t tiles_m = (M + BM - 1) / BM, tiles_n = (n + P_BN - 1) / P_BN, tiles = tiles_m * tiles_n;

    if (threadIdx.x == 0) {
        for (int s = 0; s < P_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 4); }
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    auto tile_origin = [&](uint32_t tile, uint32_t &m0, uint32_t &n0) {
        const uint32_t group = tile / (GROUP_M * tiles_n), first_m = group * GROUP_M;
        const uint32_t rows_in_group = min((uint32_t)GROUP_M, tiles_m - first_m);
        const uint32_t in_group = tile - group * GROUP_M * tiles_n;
        m0 = (first_m + in_group % rows_in_group) * BM;
        n0 = (in_group / rows_in_group) * P_BN;
    };

    if (warp == 0) {
        if (elect_one()) {
            uint32_t it = 0, armed = 0;
            bool ok = true;
            const uint32_t withhold = blockIdx.x == 0 ? (uint32_t)g_withhold_step : 0xffffffffu;     // test hook: this stage is never loaded
            for (uint32_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
                uint32_t m0, n0;
                tile_origin(tile, m0, n0);
                for (uint32_t kb = 0; kb < num_k; ++kb, ++it) {
                    const uint32_t s = it % P_STAGES, ph = (it / P_STAGES) & 1;
                    if (it == withhold) { ok = false; break; }
                    if (!mbar_wait(&empty[s], ph ^ 1, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (1 << 8) | (int)s); } ok = false; break; }
                    mbar_expect_tx(&full[s], STAGE_BYTES);
                    tma_load_2d(smem + s * STAGE_BYTES, &tmA, (int)(kb * BK), (int)m0, &full[s]);
                    tma_load_2d(smem + s * STAGE_BYTES + A_BYTES, &tmB, (int)(kb * BK), (int)n0, &full[s]);
                    armed = it + 1;
                }
            }
            if (*failed) {
                volatile uint32_t never = 0;
                for (uint32_t k = armed > P_STAGES ? armed - P_STAGES : 0; k < armed; ++k) mbar_wait(&full[k % P_STAGES], (k / P_STAGES) & 1, &never);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            constexpr uint32_t idesc = umma_idesc(P_BN);
            uint32_t it = 0, lt = 0;
            bool ok = true;
            for (uint32_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++lt) {
                const uint32_t buf = lt & 1, use = lt >> 1;
                if (!mbar_wait(&acc_empty[buf], (use & 1) ^ 1, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (2 << 8) | 0x80 | (int)buf); } break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tacc = tmem_base + buf * P_BN;
                for (uint32_t kb = 0; kb < num_k; ++kb, ++it) {
                    const uint32_t s = it % P_STAGES, ph = (it / P_STAGES) & 1;
                    if (!mbar_wait(&full[s], ph, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (2 << 8) | (int)s); } ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t da = umma_desc(smem_u32(smem + s * STAGE_BYTES));
                    const uint64_t db = umma_desc(smem_u32(smem + s * STAGE_BYTES + A_BYTES));
#pragma unroll
                    for (uint32_t k = 0; k < BK / 16; ++k) umma(tacc, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
                    umma_commit(&empty[s]);
                }
                if (ok) umma_commit(&acc_full[buf]);
            }
        }
    } else {
        const uint32_t quarter = warp & 3;
        const bool vec = ((ldc | col0) & 3u) == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0;
        uint32_t lt = 0;
        for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++lt) {
            const uint32_t buf = lt & 1, use = lt >> 1;
            bool ready = !*failed && mbar_wait(&acc_full[buf], use & 1, failed);
            if (!ready && !*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, 3 << 8); }
            ready = __all_sync(0xffffffffu, ready && !*failed);
            if (!ready) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint32_t m0, n0;
            tile_origin(tile, m0, n0);
            const uint32_t row = m0 + quarter * 32 + lane;
#pragma unroll 1
            for (uint32_t c = 0; c < P_BN / 32; ++c) {
                float v[32];
                tmem_ld32(tmem_base + ((quarter * 32) << 16) + buf * P_BN + c * 32, v);
                const uint32_t col = n0 + c * 32;
                if (row < M && col < n) {
                    float *dst = C + (size_t)row * ldc + col0 + col;
                    if (ep.aout) swiglu_store32(ep, (size_t)row * ldc + col0 + col, v, min(32u, n - col));
                    else if (vec && col + 32 <= n) {
#pragma unroll
                        for (int j = 0; j < 32; j += 4) {
                            float4 o = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                            if (accumulate) { const float4 old = *reinterpret_cast<const float4 *>(dst + j); o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w; }
                            *reinterpret_cast<float4 *>(dst + j) = o;
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (col + j < n) dst[j] = accumulate ? dst[j] + v[j] : v[j];
                    }
                }
            }
            // this warp has read its quarter of the buffer: hand it back to the MMA warp
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[buf])) : "memory");
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// ---- paired variant: tiles of 256 weight rows x up to 256 activation rows per CTA pair (cta_group::2) ----------------
// What limits the kernel above is what an SM can pull from L2: 48 KB per 64-wide K block of 512 cycles, 96 bytes a clock where a full ring brings in 80.
// Here the two CTAs of a pair sit on the two SMs of a TPC and share one MMA: its 256 rows are WEIGHT rows (128 per CTA), its N columns activation rows, of
// which each CTA loads half - 32 KB per K block at N = 256 for the same arithmetic per SM.  An MMA takes N / 2 cycles (43 at least).  Weights as
// rows means that a warp's 32 TMEM lanes are 32 consecutive columns of C: every store, residual add and gate load of the epilogue is one full line of
// one output row (with activations as rows each lane walked a row of its own: the SwiGLU epilogue of 32768 x 4096 x 4096
// took 1280 us against 970 us of the plain one), and N, a multiple of 16, follows the batch: M = 603 costs 3 x 208 rows and not 3 x 256.
//   Few tiles: what counts is not the tensor pipe but the first load (1.5 us), the K blocks' loads (80 bytes a clock) and the stores (32 bytes a
// clock and SM, 16 for residual adds), so smaller tiles on more SMs are ahead (M=509, n=2048, K=2048: 64 tiles of N=64 11.4 us, 32 of N=128 13.2).
//   Parts.  Up to TGP_GEMM_GROUP_MAX weight blocks that read the same activations are walked as one list of tiles.
//   Pairs are persistent, with two accumulators in TMEM: the epilogue of a tile overlaps the MMAs of the next.
//   A stage holds two 64-wide K blocks (half the barrier hand-overs of one, 4 % faster), p.stages of them.  Only the
// even CTA of a pair (its leader) issues MMAs; the TMA loads of both CTAs count on the leader's `full` barrier; an MMA
// commit arrives on the `empty` / `acc_full` barriers of both; the epilogue warps of both arrive on the leader's `acc_empty`.
// No multicast load anywhere.  Same bounded waits and error word; a cluster barrier before TMEM is freed keeps a CTA from
// leaving while its partner may still touch its memory.
//   The launch is a programmatic dependent one: barriers, TMEM and tensor maps are set up while the previous kernel drains.
constexpr int Q_WARPS = 10, Q_EPI = Q_WARPS - 2;       // TMA, MMA, eight epilogue warps (two per TMEM lane quarter)
constexpr int KH = 2;                                  // 64-wide K blocks per stage

struct ListArgs {
    CUtensorMap x, w[TGP_GEMM_GROUP_MAX];
    float *C[TGP_GEMM_GROUP_MAX];
    uint32_t n[TGP_GEMM_GROUP_MAX], ldc[TGP_GEMM_GROUP_MAX], tiles[TGP_GEMM_GROUP_MAX];      // tiles: of weight rows, per part
    uint32_t count, tiles_n, M, N, tiles_m, K, stages, slices;                              // N: activation rows per tile
    int accumulate;
    Epi ep;                                                                                 // with one part only
};

// 32 activation rows of one column of C, from element offset `at` on, `cnt` of them inside the matrix.  A warp's lanes are neighbouring
// columns: every access is one full line of one row.  The gates are all requested before the first is used; a product
// added to C goes out as one add per element by one thread - the rounded sum of load, add and store, but not waited for.
__device__ __forceinline__ void store32(const ListArgs &p, uint32_t part, size_t at, uint32_t ldc, const float (&v)[32], uint32_t cnt) {
    if (p.ep.aout) {
        const float *g = p.ep.gate + at;
        __nv_bfloat16 *a = p.ep.aout + at;
        float gv[32];
#pragma unroll
        for (uint32_t j = 0; j < 32; ++j) gv[j] = j < cnt ? g[(size_t)j * ldc] : 0.f;
#pragma unroll
        for (uint32_t j = 0; j < 32; ++j)
            if (j < cnt) a[(size_t)j * ldc] = __float2bfloat16_rn(gv[j] / (1.0f + expf(-gv[j])) * v[j]);
        return;
    }
    float *C = p.C[part] + at;
    if (p.accumulate) {
#pragma unroll
        for (uint32_t j = 0; j < 32; ++j) if (j < cnt) atomicAdd(C + (size_t)j * ldc, v[j]);
    } else {
#pragma unroll
        for (uint32_t j = 0; j < 32; ++j) if (j < cnt) C[(size_t)j * ldc] = v[j];
    }
}

// 32 columns of one TMEM lane, summed over four accumulators 128 columns apart: (0 + 1) + (2 + 3)
__device__ __forceinline__ void sum_four(uint32_t at, float (&v)[32]) {
    float w[32], y[32];
    tmem_ld32_pair(at, at + 128, v, w);
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] += w[j];
    tmem_ld32_pair(at + 256, at + 384, w, y);
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] += w[j] + y[j];
}

// SHARED: a tile (of N <= 128) is shared by the two pairs of a cluster, one half of K each, added into four accumulators by turns; the halves meet
// through shared memory, and each pair stores half of the activation rows.
template <bool SHARED>
__global__ void __launch_bounds__(Q_WARPS * 32, 1) tgp_matmul_tc_pair_kernel(const __grid_constant__ ListArgs p) {
    extern __shared__ uint8_t smem_raw[];
    constexpr uint32_t W_BYTES = BM * BK * 2;                     // one K block of this CTA's 128 weight rows
    const uint32_t N = p.N, ST = p.stages;
    const uint32_t X_BYTES = N / 2 * BK * 2, HALF = W_BYTES + X_BYTES, STAGE = KH * HALF;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    // barriers ahead of the ring (the first 1024 bytes): full[8], empty[8], acc_full[2], acc_empty[2], TMEM slot, flag
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);          // used in the leader only
    uint64_t *empty = full + 8;
    uint64_t *acc_full = empty + 8;                               // [2]
    uint64_t *acc_empty = acc_full + 2;                           // [2], used in the leader only: the epilogue warps of both CTAs
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 2);
    volatile uint32_t *failed = tmem_slot + 1;
    uint8_t *ring = smem + 1024;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t SL = SHARED ? 2 : 1;
    const uint32_t cta = cluster_ctarank(), rank = cta & 1, slice = cta >> 1;      // CTA of the cluster, of its pair; its pair
    const uint32_t pair = blockIdx.x / (2 * SL), pairs = gridDim.x / (2 * SL);      // (clusters, where two pairs share a tile)
    const uint32_t stages_k = (p.K + KH * BK - 1) / (KH * BK), half_k = (stages_k + 1) / 2;     // stages of all K and of its first half; a block past K reads zeros
    const uint32_t kb_lo = slice ? half_k : 0, num_k = SL == 1 ? stages_k : slice ? stages_k - half_k : half_k;
    const uint32_t tiles = p.tiles_m * p.tiles_n;
    const uint32_t buf_cols = SHARED ? 128u : N <= 64 ? 64u : N <= 128 ? 128u : 256u;           // TMEM columns of one accumulator
    const uint32_t cols = SHARED ? 4 * buf_cols : 2 * buf_cols;

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < 8; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * Q_EPI); }
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {                                  // the same warp in both CTAs of the pair
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");     // not before the allocation: see tgp_sm100.cuh
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    cluster_sync_all();                               // barriers of all CTAs initialised, TMEM allocated
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    // Tile order: groups of GROUP_M activation tiles are swept across all weight tiles before the next group starts (see the
    // per-tile kernel above).  part: the weight block, w0: first weight row of the tile in it, m0: first activation row
    auto tile_origin = [&](uint32_t tile, uint32_t &part, uint32_t &w0, uint32_t &m0) {
        const uint32_t group = tile / (GROUP_M * p.tiles_n), first_m = group * GROUP_M;
        const uint32_t rows_in_group = min((uint32_t)GROUP_M, p.tiles_m - first_m);
        const uint32_t in_group = tile - group * GROUP_M * p.tiles_n;
        m0 = (first_m + in_group % rows_in_group) * N;
        uint32_t wt = in_group / rows_in_group;
        part = 0;
        while (part + 1 < p.count && wt >= p.tiles[part]) wt -= p.tiles[part++];
        w0 = wt * (2 * BM);
    };

    if (warp == 0) {
        if (elect_one()) {                            // TMA thread of this CTA: its 128 weight rows, its half of the activation rows
            asm volatile("griddepcontrol.wait;" ::: "memory");
            uint32_t it = 0, s = 0, ph = 0;
            const uint32_t withhold = pair == 0 ? (uint32_t)g_withhold_step : 0xffffffffu;     // test hook: both CTAs of the first pair never load this stage
            bool ok = true;
            for (uint32_t tile = pair; tile < tiles && ok; tile += pairs) {
                uint32_t part, w0, m0;
                tile_origin(tile, part, w0, m0);
                const CUtensorMap *mw = &p.w[part];
                for (uint32_t kb = 0; kb < num_k; ++kb, ++it) {
                    if (it == withhold) { ok = false; break; }
                    if (!mbar_wait(&empty[s], ph ^ 1, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (1 << 8) | (int)s); } ok = false; break; }
                    if (rank == 0) mbar_expect_tx(&full[s], 2 * STAGE);
#pragma unroll
                    for (int h = 0; h < KH; ++h) {
                        const int k = (int)(((kb_lo + kb) * KH + h) * BK);
                        tma_load_2d_pair(ring + s * STAGE + h * HALF, mw, k, (int)(w0 + rank * BM), &full[s]);
                        tma_load_2d_pair(ring + s * STAGE + h * HALF + W_BYTES, &p.x, k, (int)(m0 + rank * (N / 2)), &full[s]);
                    }
                    if (++s == ST) { s = 0; ph ^= 1; }
                }
            }
            if (*failed && rank == 0) {               // loads of both CTAs still in flight land on these barriers (bounded wait)
                volatile uint32_t never = 0;
                for (uint32_t q = it > ST ? it - ST : 0; q < it; ++q) mbar_wait(&full[q % ST], (q / ST) & 1, &never);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (rank == 0 && elect_one()) {               // MMA thread of the pair
            asm volatile("griddepcontrol.wait;" ::: "memory");    // the limit of its waits counts from here
            const uint32_t idesc = umma_idesc_pair(N), mask = 3u << (cta & 2);
            uint32_t s = 0, ph = 0, lt = 0;
            bool ok = true;
            for (uint32_t tile = pair; tile < tiles && ok; tile += pairs, ++lt) {
                const uint32_t buf = lt & 1, use = lt >> 1;
                if (!mbar_wait(&acc_empty[buf], (use & 1) ^ 1, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (2 << 8) | 0x80 | (int)buf); } break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tacc = tmem_base + buf * buf_cols;
                for (uint32_t kb = 0; kb < num_k; ++kb) {
                    if (!mbar_wait(&full[s], ph, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (2 << 8) | (int)s); } ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (uint32_t h = 0; h < KH; ++h) {
                        const uint64_t dw = umma_desc(smem_u32(ring + s * STAGE + h * HALF));
                        const uint64_t dx = umma_desc(smem_u32(ring + s * STAGE + h * HALF + W_BYTES));
#pragma unroll
                        for (uint32_t k = 0; k < BK / 16; ++k) {
                            if (SHARED) umma_pair(tacc + k * 128, dw + 2 * k, dx + 2 * k, idesc, (kb | h) != 0);
                            else umma_pair(tacc, dw + 2 * k, dx + 2 * k, idesc, (kb | h | k) != 0);
                        }
                    }
                    umma_commit_pair(&empty[s], mask);
                    if (++s == ST) { s = 0; ph ^= 1; }
                }
                if (ok) umma_commit_pair(&acc_full[buf], mask);
            }
        }
        __syncwarp();
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");        // what C, the gate and a hold is the previous kernel's work
        const uint32_t quarter = warp & 3, half = (warp - 2) >> 2, wrow = rank * BM + quarter * 32 + lane, tm = tmem_base + ((quarter * 32) << 16);
        uint32_t lt = 0, out = 0, rows_out = 0;       // (a tile that two pairs share: weight block, activation rows, element of C)
        size_t at_out = 0;
        for (uint32_t tile = pair; tile < tiles; tile += pairs, ++lt) {
            const uint32_t buf = lt & 1, use = lt >> 1;
            uint32_t part, w0, m0;
            tile_origin(tile, part, w0, m0);
            bool ready = !*failed && mbar_wait(&acc_full[buf], use & 1, failed);
            if (!ready && !*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, 3 << 8); }
            ready = __all_sync(0xffffffffu, ready && !*failed);
            if (!ready) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t row = w0 + wrow, ldc = p.ldc[part], rows = min(N, p.M - m0);      // this lane's column of C; activation rows of the tile
            const bool mine = row < p.n[part];
            if constexpr (SHARED) {                               // the partial sums of the rows that the other pair stores: over the idle ring
                for (uint32_t c = half * 32; c < N / 2; c += 64) {
                    float v[32];
                    sum_four(tm + (slice ^ 1) * (N / 2) + c, v);
                    float *part_s = reinterpret_cast<float *>(ring) + quarter * 32 + lane;
#pragma unroll
                    for (uint32_t j = 0; j < 32; ++j) if (c + j < N / 2) part_s[(c + j) * BM] = v[j];
                }
                out = part; at_out = (size_t)m0 * ldc + row; rows_out = mine ? rows : 0;
                break;                                            // a cluster has one tile
            } else {
#pragma unroll 1
                for (uint32_t c = half * 32; c < N; c += 64) {    // 32 activation rows at a time
                    float v[32];
                    tmem_ld32(tm + buf * buf_cols + c, v);
                    store32(p, part, (size_t)(m0 + c) * ldc + row, ldc, v, mine && c < rows ? rows - c : 0);
                }
            }
            // this warp has read its share of this CTA's half of the buffer: tell the pair's MMA thread
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(&acc_empty[buf], cta & 2);
        }
        if constexpr (SHARED) {
            __syncwarp();
            cluster_sync_all();                       // every partial sum is in its CTA's shared memory
            const uint32_t lo = slice * (N / 2);
            uint32_t bad = 0;
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) bad |= ld_remote_u32(smem_u32((const void *)failed), q);
            for (uint32_t c = half * 32; c < N / 2; c += 64) {
                float v[32], w[32];
#pragma unroll
                for (uint32_t j = 0; j < 32; ++j) w[j] = ld_remote_f32(smem_u32(ring) + ((c + j) * BM + quarter * 32 + lane) * 4, cta ^ 2);
                if (bad) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                sum_four(tm + lo + c, v);
#pragma unroll
                for (uint32_t j = 0; j < 32; ++j) v[j] += w[j];
                const uint32_t ldc = p.ldc[out];
                store32(p, out, at_out + (size_t)(lo + c) * ldc, ldc, v, lo + c < rows_out ? min(rows_out - lo, N / 2) - c : 0);
            }
        }
    }
    if (SHARED && warp < 2) cluster_sync_all();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    cluster_sync_all();                               // neither CTA frees TMEM or leaves while its partner may still touch it
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(cols) : "memory");
    }
}

// ---- up to 128 activation rows, and products of few tiles: one tile of 128 weight rows per CTA ----------------------
// A product of up to 128 activation rows is bound by HBM, one of more rows and few tiles by the length of K.  Every CTA takes 128
// weight rows (the rows of the MMA; N <= 128 activation rows, a multiple of 16, are its columns) and a slice of K.  One CTA
// per MMA and not a pair: there are four times as many tiles to share out, and the tensor pipe (48 cycles an MMA at N = 64, 64 at 128) waits for HBM.
//   K slices: a block of few tiles is split along K over the SL CTAs of a cluster; their partial tiles meet in shared memory
// and are summed pairwise.  The split depends on M, n, K and the number of SMs: a block computes the same bits alone or in a list.
//   Accumulators: consecutive MMAs go to different ones (eight up to 32 activation rows, four up to 64, else two), summed at the end.
// The tensor core adds into fp32 without rounding to nearest, so the error of a sum grows with the number of additions in a
// row, and MMAs into one accumulator or into several take the same time (M=61, n=4096, K=4096: distance from 64 bits 1.0e-6 with
// one, 2.4e-7 with four; n=14336 unsplit 4.4e-6, 1.0e-6).
//   Ring: 200 KB where the launch gives an SM one CTA (M=61, n=14336, K=4096: 24.9 us; 28.4 us with 100 KB), else 100 KB, so that
// an SM holds two (28672 rows: 43.0 us; 50.3 us with 200 KB).
constexpr uint32_t S_RING = 100 * 1024, S_RING_LONE = 200 * 1024, S_STAGES = 12;

// Sum of the SL partial tiles of a cluster ([activation row][128 weight rows] fp32 at `addr` in every CTA), neighbours first: J activation
// rows `stride` bytes apart, four weight rows each.  All loads are under way before the first sum (a load
// from another CTA of the cluster takes about 0.3 us).
template <int SL, int J>
__device__ __forceinline__ void sum_slices(uint32_t addr, uint32_t stride, float4 (&sum)[J]) {
    float4 v[SL][J];
#pragma unroll
    for (uint32_t q = 0; q < SL; ++q)
#pragma unroll
        for (uint32_t j = 0; j < J; ++j) v[q][j] = ld_remote_f32x4(addr + j * stride, q);
#pragma unroll
    for (uint32_t w = 1; w < SL; w *= 2)
#pragma unroll
        for (uint32_t q = 0; q < SL; q += 2 * w)
#pragma unroll
            for (uint32_t j = 0; j < J; ++j) {
                v[q][j].x += v[q + w][j].x; v[q][j].y += v[q + w][j].y; v[q][j].z += v[q + w][j].z; v[q][j].w += v[q + w][j].w;
            }
#pragma unroll
    for (uint32_t j = 0; j < J; ++j) sum[j] = v[0][j];
}

// four consecutive columns of one row of C (element offset `at` in its geometry, `cnt` of them inside the matrix)
__device__ __forceinline__ void store4(float *C, size_t at, const float4 &v, uint32_t cnt, int accumulate, const Epi &ep, bool vec) {
    const float f[4] = {v.x, v.y, v.z, v.w};
    if (ep.aout) {
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i)
            if (i < cnt) { const float g = ep.gate[at + i]; ep.aout[at + i] = __float2bfloat16_rn(g / (1.0f + expf(-g)) * f[i]); }
    } else if (accumulate) {
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) if (i < cnt) atomicAdd(C + at + i, f[i]);
    } else if (vec && cnt == 4) {
        *reinterpret_cast<float4 *>(C + at) = v;
    } else {
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) if (i < cnt) C[at + i] = f[i];
    }
}

__global__ void __launch_bounds__(192, 2) tgp_wstream_tc_kernel(const __grid_constant__ ListArgs p) {
    extern __shared__ uint8_t smem_raw[];
    constexpr uint32_t W_BYTES = BM * BK * 2;
    const uint32_t N = p.N, ST = p.stages, SL = p.slices, STAGE = W_BYTES + N * BK * 2;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    // barriers ahead of the ring (the first 1024 bytes): full[S_STAGES], empty[S_STAGES], acc_full, TMEM slot, flag
    uint64_t *full = reinterpret_cast<uint64_t *>(smem), *empty = full + S_STAGES, *acc_full = empty + S_STAGES;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_full + 1);
    volatile uint32_t *failed = tmem_slot + 1;
    uint8_t *ring = smem + 1024;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t slice = SL > 1 ? cluster_ctarank() : 0, tile = blockIdx.x / SL;
    const uint32_t kblocks = (p.K + BK - 1) / BK, kb_lo = kblocks * slice / SL, num_k = kblocks * (slice + 1) / SL - kb_lo;
    const uint32_t acc_cols = N <= 32 ? 32u : N <= 64 ? 64u : 128u, cols = 256;     // TMEM: up to 256 / acc_cols accumulators
    const uint32_t accs = N > 64 ? 2u : N > 32 || num_k < 2 ? 4u : 8u;
    const uint32_t m0 = tile % p.tiles_m * N, rows = min(N, p.M - m0);              // this tile's activation rows
    uint32_t part = 0, wt = tile / p.tiles_m;
    while (part + 1 < p.count && wt >= p.tiles[part]) wt -= p.tiles[part++];
    const uint32_t w0 = wt * BM;
    const CUtensorMap *mw = &p.w[part];

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < S_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(acc_full, 1);
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&p.x) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(mw) : "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");     // not before the allocation: see tgp_sm100.cuh
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (elect_one()) {
            // The weights of the first ring come into L2 while the previous kernel still runs; loading them here would be wrong where that
            // kernel writes them (M=61: n=4096, K=4096 13.3 -> 12.3 us, the list of 2 x 14336 45.7 -> 43.6, with 16 rows 42.4 -> 40.6; from the
            // end of the norm before).  Requests ahead of the ring further on make it slower.
            for (uint32_t kb = 0; kb < min(num_k, ST); ++kb) tma_prefetch_2d(mw, (int)((kb_lo + kb) * BK), (int)w0);
            asm volatile("griddepcontrol.wait;" ::: "memory");
            uint32_t s = 0, ph = 0, armed = 0;
            const uint32_t withhold = blockIdx.x == 0 ? (uint32_t)g_withhold_step : 0xffffffffu;     // test hook: this stage is never loaded
            for (uint32_t kb = 0; kb < num_k; ++kb) {
                if (kb == withhold) break;
                if (!mbar_wait(&empty[s], ph ^ 1, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (1 << 8) | (int)s); } break; }
                mbar_expect_tx(&full[s], STAGE);
                tma_load_2d(ring + s * STAGE, mw, (int)((kb_lo + kb) * BK), (int)w0, &full[s]);
                tma_load_2d(ring + s * STAGE + W_BYTES, &p.x, (int)((kb_lo + kb) * BK), (int)m0, &full[s]);
                armed = kb + 1;
                if (++s == ST) { s = 0; ph ^= 1; }
            }
            if (*failed) {
                volatile uint32_t never = 0;
                for (uint32_t q = armed > ST ? armed - ST : 0; q < armed; ++q) mbar_wait(&full[q % ST], (q / ST) & 1, &never);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (elect_one()) {
            asm volatile("griddepcontrol.wait;" ::: "memory");    // the limit of its waits counts from here
            const uint32_t idesc = umma_idesc((int)N);
            uint32_t s = 0, ph = 0;
            bool ok = true;
            for (uint32_t kb = 0; kb < num_k; ++kb) {
                if (!mbar_wait(&full[s], ph, failed)) { if (!*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, (2 << 8) | (int)s); } ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t dw = umma_desc(smem_u32(ring + s * STAGE)), dx = umma_desc(smem_u32(ring + s * STAGE + W_BYTES));
#pragma unroll
                for (uint32_t k = 0; k < BK / 16; ++k) umma(tmem_base + ((4 * kb + k) & (accs - 1)) * acc_cols, dw + 2 * k, dx + 2 * k, idesc, 4 * kb + k >= accs);
                umma_commit(&empty[s]);
                if (++s == ST) { s = 0; ph ^= 1; }
            }
            if (ok) umma_commit(acc_full);
        }
        __syncwarp();
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");        // what C holds is the previous kernel's work
        bool ready = !*failed && mbar_wait(acc_full, 0, failed);
        if (!ready && !*failed) { *failed = 1; atomicCAS(&g_gemm_tc_error, 0, 3 << 8); }
        ready = __all_sync(0xffffffffu, ready && !*failed);
        if (ready) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t quarter = warp & 3, wrow = quarter * 32 + lane, row = w0 + wrow, ldc = p.ldc[part];
            const bool mine = row < p.n[part];
#pragma unroll 1
            for (uint32_t c = 0; c < N; c += 32) {
                const uint32_t at_t = tmem_base + ((quarter * 32) << 16) + c;  // (N = 16, 48, ...: the columns past N are not used)
                float v[32], w[32], y[32];
                tmem_ld32(at_t, v);
                tmem_ld32(at_t + acc_cols, w);
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] += w[j];
                for (uint32_t i = 2; i < accs; i += 2) {
                    tmem_ld32(at_t + i * acc_cols, w);
                    tmem_ld32(at_t + (i + 1) * acc_cols, y);
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] += w[j] + y[j];
                }
                if (SL > 1) {                                      // this slice's partial over the idle ring
                    float *part_s = reinterpret_cast<float *>(ring) + wrow;
#pragma unroll
                    for (uint32_t j = 0; j < 32; ++j) if (c + j < N) part_s[(c + j) * BM] = v[j];
                    continue;
                }
                const size_t at = (size_t)(m0 + c) * ldc + row;
                store32(p, part, at, ldc, v, mine && c < rows ? rows - c : 0);
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    if (SL > 1) {
        cluster_sync_all();                           // every slice's partial tile is in its CTA's shared memory
        if (warp >= 2) {
            uint32_t bad = 0;
            for (uint32_t q = 0; q < SL; ++q) bad |= ld_remote_u32(smem_u32((const void *)failed), q);
            const uint32_t row = w0 + 4 * lane, n = p.n[part], ldc = p.ldc[part], ew = warp - 2, j_hi = N * (slice + 1) / SL;
            const uint32_t cnt = bad || row >= n ? 0u : min(4u, n - row), base = smem_u32(ring) + lane * 16;
            const bool vec = (ldc & 3u) == 0 && (reinterpret_cast<uintptr_t>(p.C[part]) & 15u) == 0;
            for (uint32_t j0 = N * slice / SL + ew; j0 < j_hi; j0 += 8) {
                float4 sum[2];                                     // rows j0 and j0 + 4 (past this slice's share: read, not stored)
                const uint32_t at = base + j0 * (BM * 4);
                if (SL == 2) sum_slices<2, 2>(at, 4 * BM * 4, sum);
                else sum_slices<4, 2>(at, 4 * BM * 4, sum);
#pragma unroll
                for (uint32_t j = 0; j < 2; ++j) {
                    const uint32_t m = j0 + 4 * j;
                    if (m < rows && m < j_hi) store4(p.C[part], (size_t)(m0 + m) * ldc + row, sum[j], cnt, p.accumulate, p.ep, vec);
                }
            }
        }
        __syncwarp();
        cluster_sync_all();                           // no CTA leaves while another may still read its partial tile
    } else {
        __syncthreads();
    }
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(cols) : "memory");
    }
}

// 2-D bf16 row-major [rows, K] map with a [box_rows, 64] box, 128-byte swizzle, zero fill outside.
bool make_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t K, uint32_t box_rows) {
    static_assert(BK == 64, "the shared tensor-map helper encodes 64-element boxes");
    return tensor_map_bf16_2d(map, base, rows, K, K * 2, box_rows);
}

}  // namespace

extern thread_local uint64_t tgpk_launches;

template <int BN, int ST, int KH, bool SWAP = false>
static bool launch_tile(const CUtensorMap &ma, const CUtensorMap &mb, float *C, uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate, cudaStream_t st, const Epi ep = Epi{nullptr, nullptr}) {
    if (!tgpk_allow_smem<tgp_matmul_tc_kernel<BN, ST, KH, SWAP>>(Smem<BN, ST, KH>::TOTAL)) return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(((M + BM - 1) / BM) * ((n + BN - 1) / BN)); cfg.blockDim = dim3(192); cfg.dynamicSmemBytes = Smem<BN, ST, KH>::TOTAL; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, tgp_matmul_tc_kernel<BN, ST, KH, SWAP>, ma, mb, C, M, n, K, ldc, col0, accumulate, ep) == cudaSuccess;
}

static int g_tc_variant = 0;     // 0 by size (see the top of this file), 1 force the 128x128 per-tile kernel, 2 the persistent 128x256 kernel, 3 the paired
                                 // kernel with its largest tiles, 4 the per-tile kernel with the weights as the 128-row operand (M <= 128 only; else as 0)

bool tgpk_gemm_tc_forced() { return g_tc_variant != 0; }

static uint32_t tc_sms() { return (uint32_t)tgpk_sms(); }

// Does the paired kernel share the tiles of a block between two pairs?  Blocks of more than 128 activation rows and K >= 8192, more tiles than the one-tile-per-CTA
// kernel holds in one wave of slices and at most a cluster's tile each in one wave.  The sums are those of half of K in four accumulators each, as near 64 bits as
// that kernel's four slices with two (M=509, n=2048, K=8192: 29.2 us in slices, 23.9 shared; M=150, n=4096, K=14336: 44.8, 41.8; but n=2048, K=8192
// 16.8, 18.3).  With a shorter K sharing gains 5 % at best over smaller tiles.  The choice depends on M, n, K and the number of SMs (the bits may differ between
// devices of different sizes), not on a list.
//   One wave: a cluster of four lies in one GPC, of which two to four SMs stay over, so that 148 SMs hold 33 clusters and not 37, fewer where GPCs are cut
// differently; counted on are seven eighths, 32 (K=8192, M=236 in slices and shared: 32 tiles 29.0 / 25.5 us, 34 tiles 29.4 / 40.5; M=364, 27 tiles in rows
// of 128, which is one wave, 23, in rows of 96, which would be one of 37, 32).
static uint32_t shared_at_once() { return tc_sms() * 7 / 32; }

static bool shared_tiles(uint32_t M, uint32_t n, uint32_t K) {
    const uint64_t rows = (M + BM - 1) / BM;
    return M > BM && K >= 8192 && rows * ((n + BM - 1) / BM) * 4 > tc_sms() && rows * ((n + 2 * BM - 1) / (2 * BM)) <= shared_at_once();
}

// K slices of a block in the one-tile-per-CTA kernel, 0: the paired kernel serves it.  No list counts here either.  Measured (us; M=61):
//   n=4096, K=4096        22.4 unsplit, 15.3 in two slices, 11.9 in four, 12.4 in eight
//   n=2048, K=8192        41.6, 24.7, 15.4, 21.1 (few clusters of eight fit the GPU at a time: no eight anywhere)
//   n=8192, K=8192        42.4, 28.1, 26.4 (256 CTAs, two per SM)
//   n=8192 twice, K=2048  14.4, 16.5, 22.2; n=32000, K=4096: 46.2, 51.3, 62.3
static uint32_t cta_slices(uint32_t M, uint32_t n, uint32_t K) {
    const uint64_t tiles = (uint64_t)((n + BM - 1) / BM) * ((M + BM - 1) / BM), sms = tc_sms();
    if (M > BM) return tiles * 4 <= 2 * sms && K >= 8192 && !shared_tiles(M, n, K) ? 4 : 0;
    if (tiles * 4 <= (K >= 8192 ? 2 * sms : sms) && K >= 1024) return 4;
    return tiles * 2 <= sms && K >= 1024 ? 2 : 1;
}

// Estimated cycles of the paired kernel for `wt` tiles of 256 weight rows at M activation rows in tiles of N, with room for `at_once` tiles.  A 64-wide block of K
// of a pair takes 2 N cycles of the tensor pipe (172 at least) and (16384 + 64 N) bytes per SM, which arrive at 80 a clock (what a full ring
// asks for in the 1.4 us a load takes); the first stage arrives after 3000 cycles, and a tile's epilogue, under the MMAs of the next one, takes 1600 cycles and
// writes 512 N bytes per SM at 32 a clock (residual adds leave at 16, which is not counted).  The 1600 count for every tile, not only behind the last: 66 forms
// of M=212 - 2000, K=64 - 2048 take 1.001 of the time of their best tiles so, 1.05 otherwise, by K=64 most (M=288, n=14464 in tiles of 144 rows 9.8 us, of 32 14.1).
// Where K is no multiple of 64 the 128 bytes that a box takes of a row lie in two lines, and arrive at 70 a clock (M=501, n=11469+352+1013, K=5832 in tiles
// of 256 rows 95 us, of 128, which 80 a clock would make the faster ones, 103; over 80 such forms 1.002 of the best, 1.007 otherwise).
static uint64_t pair_cost(uint32_t M, uint32_t wt, uint32_t K, uint32_t N, uint32_t at_once) {
    const uint64_t tiles = (uint64_t)((M + N - 1) / N) * wt, rounds = (tiles + at_once - 1) / at_once;
    const uint64_t mma = (uint64_t)((K + BK - 1) / BK) * std::max<uint64_t>(std::max(2 * N, 172u), (16384 + 64 * N) / (K % BK ? 70 : 80)), epi = 16 * N + 1600;
    return 3000 + mma + (rounds - 1) * std::max(mma, epi) + epi;
}

// Activation rows per tile: what the estimate above says is fastest (us with the norm before; estimates rank the choices as the clock does: M=509, n=2048, K=2048
// N=128 13.9, 96 12.8, 64 12.1; M=603, n=4096 and 1024 twice, K=4096 N=208 30.3, 160 38.1, 112 34.0; M=1024, n=2048, K=2048 N=256 21.1, 176 17.3, 128 14.4).
static uint32_t pair_rows(uint32_t M, uint32_t wt, uint32_t K, uint32_t at_once, uint32_t most) {
    const uint32_t t0 = (M + most - 1) / most, unit = most == 256 ? 16 : 32;            // (shared: each pair stores half of them)
    uint32_t best = 0;
    uint64_t cost = 0;
    for (uint32_t t = t0; t <= (g_tc_variant == 3 ? t0 : t0 + 8); ++t) {                 // (forced: the largest tiles)
        const uint32_t N = std::max(32u, ((M + t - 1) / t + unit - 1) / unit * unit);
        const uint64_t c = pair_cost(M, wt, K, N, at_once);
        if (!best || c * 25 < cost * 24) { best = N; cost = c; }                          // (of equals the largest: less traffic, and less power)
    }
    return best;
}

constexpr uint32_t Q_RING = 227u * 1024u - 2048u;

template <bool SHARED>
static int launch_pair(ListArgs &p, cudaStream_t st) {
    if (!tgpk_allow_smem<tgp_matmul_tc_pair_kernel<SHARED>>(Q_RING + 2048)) return TGP_E_CUDA;
    const uint32_t stage = KH * (BM * BK * 2 + p.N / 2 * BK * 2);
    p.stages = std::min(8u, Q_RING / stage);
    const uint32_t tiles = p.tiles_m * p.tiles_n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SHARED ? 4 * tiles : 2 * std::min(tiles, tc_sms() / 2));
    cfg.blockDim = dim3(Q_WARPS * 32);
    cfg.dynamicSmemBytes = 2048 + p.stages * stage;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = SHARED ? 4 : 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, tgp_matmul_tc_pair_kernel<SHARED>, p) == cudaSuccess ? TGP_OK : TGP_E_CUDA;
}

static int launch_stream(ListArgs &p, cudaStream_t st) {
    if (!tgpk_allow_smem<tgp_wstream_tc_kernel>(S_RING_LONE + 2048)) return TGP_E_CUDA;
    const uint32_t stage = BM * BK * 2 + p.N * BK * 2, ctas = p.tiles_m * p.tiles_n * p.slices;
    p.stages = std::min(S_STAGES, (ctas <= tc_sms() ? S_RING_LONE : S_RING) / stage);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(192);
    cfg.dynamicSmemBytes = 2048 + std::max(p.stages * stage, p.slices > 1 ? p.N * (uint32_t)BM * 4u : 0u);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = p.slices; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.slices > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, tgp_wstream_tc_kernel, p) == cudaSuccess ? TGP_OK : TGP_E_CUDA;
}

// Blocks of one class may share a launch: kernel, slices of K and accumulators are the same.
uint32_t tgpk_gemm_tc_class(uint32_t M, uint32_t n, uint32_t K) { return cta_slices(M, n, K) + 1 + (shared_tiles(M, n, K) ? 8 : 0); }

// Blocks of equal tgpk_gemm_tc_class() over the same activations, in one launch.
int tgpk_gemm_tc_list(const void *A, uint32_t count, const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t M, uint32_t K,
                      int accumulate, cudaStream_t st, const float *gate, void *aout) {
    if (!count || count > TGP_GEMM_GROUP_MAX || !M || !K || K % 8) return TGP_E_INVAL;
    ListArgs p;
    memset(&p, 0, sizeof(p));
    p.ep = Epi{aout ? gate : nullptr, gate ? (__nv_bfloat16 *)aout : nullptr};
    if (p.ep.aout && (accumulate || count != 1)) return TGP_E_INVAL;
    const bool stream = g_tc_variant != 3 && cta_slices(M, n[0], K) != 0;
    const uint32_t rows_w = stream ? BM : 2 * BM;
    uintptr_t bits = reinterpret_cast<uintptr_t>(A);
    for (uint32_t s = 0; s < count; ++s) {
        bits |= reinterpret_cast<uintptr_t>(W[s]);
        p.C[s] = C[s]; p.n[s] = n[s]; p.ldc[s] = ldc[s]; p.tiles[s] = (n[s] + rows_w - 1) / rows_w;
        p.tiles_n += p.tiles[s];
    }
    if (bits & 15u) return TGP_E_INVAL;                                                                  // TMA needs 16-byte aligned bases
    p.count = count; p.M = M; p.K = K; p.accumulate = accumulate;
    if (stream) {
        p.slices = cta_slices(M, n[0], K);
        const uint32_t t = (M + BM - 1) / BM;
        p.N = ((M + t - 1) / t + 15) / 16 * 16;
    } else {
        p.slices = g_tc_variant != 3 && shared_tiles(M, n[0], K) ? 2 : 1;
        p.N = p.slices == 2 ? pair_rows(M, p.tiles_n, K / 2, shared_at_once(), 128) : pair_rows(M, p.tiles_n, K, tc_sms() / 2, 256);
    }
    p.tiles_m = (M + p.N - 1) / p.N;
    if (!make_map(&p.x, A, M, K, stream ? p.N : p.N / 2)) return TGP_E_CUDA;
    for (uint32_t s = 0; s < count; ++s) if (!make_map(&p.w[s], W[s], n[s], K, BM)) return TGP_E_CUDA;
    const int rc = stream ? launch_stream(p, st) : p.slices == 2 ? launch_pair<true>(p, st) : launch_pair<false>(p, st);
    if (rc) return rc;
    tgpk_launches += 1;
    tgpk_last_gemm_kernel = stream ? "tgp_wstream_tc_kernel" : "tgp_matmul_tc_pair_kernel";
    return TGP_OK;
}

// Weight rows per tile if the one-tile-per-CTA kernel serves a block of more than 128 activation rows that is launched alone, else 0: where its narrow
// tiles are one wave.  Without a cluster's barriers it is level with the pairs or ahead of them for a short K or four tiles of rows and more, up to a
// tenth behind for a longer K (us with the norm before: M=1024, n=512, K=512 7.1 against 8.3 in pairs, K=2048 10.5 / 11.8; M=509, n=512, K=512
// 6.5 / 6.5; M=256, n=1024, K=2048 9.4 / 8.9).  Stages of two blocks of K for 32 weight rows (M=129, n=512, K=4096: three blocks 14.9, one 14.3, two 12.5).
// Both kernels add K in one order into one accumulator: the bits are those of the pairs, which a list takes.
static uint32_t lone_tile(uint32_t M, uint32_t n, uint32_t K) {
    if (M <= BM || n > 2048 || (n > 1024 && K < 4096) || cta_slices(M, n, K) || shared_tiles(M, n, K)) return 0;
    const uint32_t bn = n > 1024 && (M + BM - 1) / BM * ((n + 31) / 32) > tc_sms() ? 64 : 32;
    return (M + BM - 1) / BM * ((n + bn - 1) / bn) <= tc_sms() ? bn : 0;
}

int tgpk_gemm_tc(const void *A, const void *W, float *C, uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate, cudaStream_t st,
                 const float *gate, void *aout) {
    constexpr int BN = 128;
    const Epi ep{aout ? gate : nullptr, gate ? (__nv_bfloat16 *)aout : nullptr};
    if (ep.aout && accumulate) return TGP_E_INVAL;
    if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(W)) & 15u) return TGP_E_INVAL;     // TMA needs 16-byte aligned bases
    if (K % 8) return TGP_E_INVAL;                                                                       // and 16-byte row strides
    if (const uint32_t bn = g_tc_variant == 0 && !ep.aout ? lone_tile(M, n, K) : 0) {
        CUtensorMap ma, mb;
        if (!make_map(&ma, A, M, K, BM) || !make_map(&mb, W, n, K, bn)) return TGP_E_CUDA;
        if (!(bn == 32 ? launch_tile<32, 5, 2>(ma, mb, C, M, n, K, ldc, col0, accumulate, st) : launch_tile<64, 8, 1>(ma, mb, C, M, n, K, ldc, col0, accumulate, st))) return TGP_E_CUDA;
        if (cudaGetLastError() != cudaSuccess) return TGP_E_CUDA;
        tgpk_launches += 1;
        tgpk_last_gemm_kernel = "tgp_matmul_tc_kernel";
        return TGP_OK;
    }
    if (g_tc_variant == 0 || g_tc_variant == 3 || (g_tc_variant == 4 && (ep.aout || M > 128))) {
        float *Cb = C + col0;
        return tgpk_gemm_tc_list(A, 1, &W, &Cb, &n, &ldc, M, K, accumulate, st, gate ? gate + col0 : nullptr, aout ? (__nv_bfloat16 *)aout + col0 : nullptr);
    }
    // the kernels of one CTA per tile, by request only (they cross-check the paired one)
    const uint32_t sms = tc_sms();
    if (g_tc_variant == 4) {                                     // the weights as the 128-row operand, M <= 128
        CUtensorMap mw, mx;
        const uint32_t bx = M <= 32 ? 32 : M <= 64 ? 64 : 128;
        if (!make_map(&mw, W, n, K, BM) || !make_map(&mx, A, M, K, bx)) return TGP_E_CUDA;
        const bool ok = bx == 32 ? launch_tile<32, 3, 3, true>(mw, mx, C, n, M, K, ldc, col0, accumulate, st)
                      : bx == 64 ? launch_tile<64, 3, 3, true>(mw, mx, C, n, M, K, ldc, col0, accumulate, st)
                                 : launch_tile<128, 2, 3, true>(mw, mx, C, n, M, K, ldc, col0, accumulate, st);
        if (!ok || cudaGetLastError() != cudaSuccess) return TGP_E_CUDA;
        tgpk_launches += 1;
        tgpk_last_gemm_kernel = "tgp_matmul_tc_kernel (weights as the 128-row operand)";
        return TGP_OK;
    }
    const bool persistent = g_tc_variant == 2;
    CUtensorMap ma, mb;
    if (!make_map(&ma, A, M, K, BM) || !make_map(&mb, W, n, K, persistent ? P_BN : BN)) return TGP_E_CUDA;
    if (persistent) {
        const uint32_t tiles_p = ((M + BM - 1) / BM) * ((n + P_BN - 1) / P_BN);
        constexpr int SMEM = P_STAGES * (BM * BK * 2 + P_BN * BK * 2) + 128 + 1024;
        if (!tgpk_allow_smem<tgp_matmul_tc_persistent_kernel>(SMEM)) return TGP_E_CUDA;
        tgp_matmul_tc_persistent_kernel<<<tiles_p < sms ? tiles_p : sms, 192, SMEM, st>>>(ma, mb, C, M, n, K, ldc, col0, accumulate, ep);
    } else {
        // fewer tiles than SMs: one CTA per SM, so the ring may take all of shared memory (a 3-stage ring leaves a lone
        // CTA waiting on L2 latency); otherwise two CTAs per SM with three stages each
        const bool lone = ((M + BM - 1) / BM) * ((n + 127) / 128) <= sms;
        if (!(lone ? launch_tile<128, 2, 3>(ma, mb, C, M, n, K, ldc, col0, accumulate, st, ep) : launch_tile<128, 3, 1>(ma, mb, C, M, n, K, ldc, col0, accumulate, st, ep))) return TGP_E_CUDA;
    }
    if (cudaGetLastError() != cudaSuccess) return TGP_E_CUDA;
    tgpk_launches += 1;
    tgpk_last_gemm_kernel = persistent ? "tgp_matmul_tc_persistent_kernel" : "tgp_matmul_tc_kernel";
    return TGP_OK;
}

extern "C" int tgp_k_gemm_tc_variant(int v) {
    if (v < 0 || v > 4) return TGP_E_INVAL;
    g_tc_variant = v;
    return TGP_OK;
}

int tgpk_gemm_wait_test(unsigned long long limit_ns, int withhold_step) {
    if (cudaMemcpyToSymbol(g_wait_limit_ns, &limit_ns, sizeof(limit_ns)) != cudaSuccess) return TGP_E_CUDA;
    return cudaMemcpyToSymbol(g_withhold_step, &withhold_step, sizeof(withhold_step)) == cudaSuccess ? TGP_OK : TGP_E_CUDA;
}

int tgpk_gemm_status_clear() { const int z = 0; return cudaMemcpyToSymbol(g_gemm_tc_error, &z, sizeof(z)) == cudaSuccess ? TGP_OK : TGP_E_CUDA; }

extern "C" int tgp_k_gemm_status(int *error_code) {
    if (!error_code) return TGP_E_INVAL;
    if (cudaMemcpyFromSymbol(error_code, g_gemm_tc_error, sizeof(int)) != cudaSuccess) return TGP_E_CUDA;
    return TGP_OK;
}
