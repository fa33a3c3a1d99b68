// Hand-written sm_100a kernels of the forward pass and their C entry points.
// Precision contract: bf16 weights / KV / GEMM inputs, fp32 accumulation and residual stream.
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cfloat>
#include <cstdint>
#include <type_traits>
#include <algorithm>
#include <atomic>
#include "tgp.h"
#include "tgp_kernels.h"

thread_local uint64_t tgpk_launches = 0;     // kernels launched by this thread (reported in the step statistics)
// true while the caller vouches that this thread's launches are all that is enqueued on their streams (tgp_step does; direct
// callers say so through tgp_k_gemm_chain): consecutive weight products over the same activations may then read them early
thread_local bool tgpk_chain_ok = false;
namespace { struct ProductChain { const void *A; cudaStream_t st; uint64_t launches_before; }; thread_local ProductChain g_chain = {nullptr, nullptr, 0}; }
thread_local const char *tgpk_last_gemm_kernel = "";   // name of the kernel the last weight-block product of this thread launched
#define LAUNCH_CHECK(n) do { cudaError_t e_ = cudaGetLastError(); if (e_ != cudaSuccess) return TGP_E_CUDA; tgpk_launches += (n); } while (0)

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ void unpack8(const uint4 &v, float *f) {
    const __nv_bfloat162 *p = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) { float2 t = __bfloat1622float2(p[i]); f[2 * i] = t.x; f[2 * i + 1] = t.y; }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Activations are produced by the grid under which this one may already have been launched (programmatic dependent
// launch), so they are read with an ordinary load after griddepcontrol.wait - never through the read-only path
// (ld.global.nc, what __ldg and const __restrict__ pointers compile to), whose cached lines may predate the wait and
// were seen to serve the previous layer's values.  The activation pointers of these kernels are therefore not
// __restrict__, and the load is a plain one (an asm volatile load costs the M <= 2 kernel a tenth of its speed, an
// L2-only load a third).
__device__ __forceinline__ uint4 ld_act(const uint4 *p) { return *p; }

// Programmatic dependent launch for the small kernels of a decode step: the grid lets its successor be scheduled at
// once and then waits for its predecessor to complete and flush, before it reads anything - the dependency is the full
// one, but the successor's launch latency (a microsecond or two, as long as these kernels run) overlaps this grid's
// execution.  Every thread of every kernel launched through launch_pdl() executes this first.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

int tgpk_sms() {
    static std::atomic<int> known[TGP_DEVICES];
    const int dev = tgpk_device();
    int sms = dev < 0 ? 0 : known[dev].load(std::memory_order_relaxed);
    if (!sms) {
        int d = 0;
        if (cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d) != cudaSuccess || sms < 1) return 148;
        if (dev >= 0) known[dev].store(sms, std::memory_order_relaxed);
    }
    return sms;
}
static int device_sms() { return tgpk_sms(); }

static int g_small_pdl = 1;      // small kernels are launched as programmatic dependents of their predecessor (0: plain launches)
thread_local bool tgpk_whole_edge = false;     // this thread's next launches wait for their predecessors as a whole, however the switches stand
static int small_overlap() { return g_small_pdl && !tgpk_whole_edge ? 1 : 0; }

template <typename... KArgs, typename... Args>
static void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = small_overlap();
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// ---- embedding gather ------------------------------------------------------------------------
// A token id outside [0, V) would index past the table (which may be mapped host memory): such a row is written as
// zeros and the first offending (row, id) is recorded in g_embed_error for tgp_k_embed_status().
__device__ unsigned long long g_embed_error = 0;      // 0, or 1 << 63 | row << 32 | (uint32_t)id of the first bad token

__global__ void tgp_embed_kernel(const bf16 *__restrict__ table, const int32_t *tok, float *x, uint32_t d, uint32_t V) {
    pdl_enter();
    const uint32_t m = blockIdx.x;
    const int32_t id = tok[m];
    float4 *out = reinterpret_cast<float4 *>(x + (size_t)m * d);
    if (id < 0 || (uint32_t)id >= V) {
        for (uint32_t i = threadIdx.x; i < d / 4; i += blockDim.x) out[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (threadIdx.x == 0) atomicCAS(&g_embed_error, 0ull, (1ull << 63) | ((unsigned long long)m << 32) | (uint32_t)id);
        return;
    }
    const uint4 *row = reinterpret_cast<const uint4 *>(table + (size_t)id * d);
    for (uint32_t i = threadIdx.x; i < d / 8; i += blockDim.x) {
        float f[8];
        unpack8(row[i], f);
        out[2 * i] = make_float4(f[0], f[1], f[2], f[3]);
        out[2 * i + 1] = make_float4(f[4], f[5], f[6], f[7]);
    }
}

// ---- RMSNorm -> bf16 -------------------------------------------------------------------------
// One step of a thread's sum of squares, written with explicit roundings so that the fused form below (a consumer that
// normalises its activations itself) reproduces the kernel's statistics bit for bit.
__device__ __forceinline__ float sumsq4(float ss, const float4 &v) {
    return __fadd_rn(ss, __fmaf_rn(v.w, v.w, __fmaf_rn(v.z, v.z, __fmaf_rn(v.y, v.y, __fmul_rn(v.x, v.x)))));
}

// One CTA of 256 threads per row.  NV > 0: the row has at most NV x 1024 elements, which stay in registers between the two passes, and
// every load, the gains' too, is under way before the first is used: a decode step's norms are two latencies long (8 rows of
// 4096: 5.4 -> 3.5 us from the end of the kernel before).  NV == 0: longer rows, read twice, and gains or
// outputs that are not 8-byte aligned.  The sum of squares is the same
// for every NV: thread t adds elements 4 t, 4 (t + 256), ... in that order.
template <int NV>
__global__ void __launch_bounds__(256) tgp_rmsnorm_kernel(const float *x, uint32_t ldx, const bf16 *__restrict__ g, bf16 *h, uint32_t d, float eps) {
    pdl_enter();
    __shared__ float red[8];
    const float4 *row = reinterpret_cast<const float4 *>(x + (size_t)blockIdx.x * ldx);
    const uint2 *gg = reinterpret_cast<const uint2 *>(g);
    uint2 *out = reinterpret_cast<uint2 *>(h + (size_t)blockIdx.x * d);
    const uint32_t n4 = d / 4;
    float4 v[NV ? NV : 1];
    uint2 gv[NV ? NV : 1];
    float ss = 0.f;
    if constexpr (NV > 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) { const uint32_t k = threadIdx.x + 256 * i; if (k < n4) v[i] = row[k]; }
#pragma unroll
        for (int i = 0; i < NV; ++i) { const uint32_t k = threadIdx.x + 256 * i; if (k < n4) gv[i] = gg[k]; }
#pragma unroll
        for (int i = 0; i < NV; ++i) if (threadIdx.x + 256 * i < n4) ss = sumsq4(ss, v[i]);
    } else {
        for (uint32_t i = threadIdx.x; i < n4; i += 256) ss = sumsq4(ss, row[i]);
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    // every warp adds the eight partial sums itself, in the one order
    const float t = warp_sum((threadIdx.x & 31) < 8 ? red[threadIdx.x & 31] : 0.f);
    const float r = 1.0f / sqrtf(t / (float)d + eps);
    auto scaled = [&](const float4 &w, const uint2 &gw) {
        const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gw.x)), g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gw.y));
        const __nv_bfloat162 lo = __floats2bfloat162_rn(w.x * r * g0.x, w.y * r * g0.y), hi = __floats2bfloat162_rn(w.z * r * g1.x, w.w * r * g1.y);
        return make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
    };
    if constexpr (NV > 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) { const uint32_t k = threadIdx.x + 256 * i; if (k < n4) out[k] = scaled(v[i], gv[i]); }
    } else {
        const __nv_bfloat162 *g2 = reinterpret_cast<const __nv_bfloat162 *>(g);
        __nv_bfloat162 *o2 = reinterpret_cast<__nv_bfloat162 *>(h + (size_t)blockIdx.x * d);
        for (uint32_t i = threadIdx.x; i < n4; i += 256) {
            const uint2 w = scaled(row[i], make_uint2(*reinterpret_cast<const uint32_t *>(&g2[2 * i]), *reinterpret_cast<const uint32_t *>(&g2[2 * i + 1])));
            o2[2 * i] = *reinterpret_cast<const __nv_bfloat162 *>(&w.x);
            o2[2 * i + 1] = *reinterpret_cast<const __nv_bfloat162 *>(&w.y);
        }
    }
}

// ---- GEMV / skinny GEMM (M <= 8 activation rows): pure weight streaming --------------------------------
// Persistent warps: the grid fills every SM once; each warp walks row groups of R output rows with a
// grid stride and keeps R x U independent 16-byte loads in flight per lane (U chunks of 256 K-elements).
// No block barrier and no shared memory, so no SM idles while another warp reduces; the summation order
// is fixed (lane-strided partials, butterfly), hence results are deterministic run to run.
template <int MT, int R, int U>
__global__ void __launch_bounds__(256) tgp_wstream_kernel(const bf16 *A, const bf16 *__restrict__ W, float *__restrict__ C,
                                                   uint32_t Mrows, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarp = (gridDim.x * blockDim.x) >> 5;
    // Programmatic dependent launch: the weights are not produced by the previous kernel in the stream, so this grid
    // may start streaming them while that kernel drains.  Everything it does produce (the activations A, the output C)
    // is touched only after griddepcontrol.wait, which returns once the previous grid has completed and flushed.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool synced = false;
    for (uint32_t row0 = gwarp * R; row0 < n; row0 += nwarp * R) {
        float acc[R][MT];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int m = 0; m < MT; ++m) acc[r][m] = 0.f;
        const bf16 *wrow[R];
#pragma unroll
        for (int r = 0; r < R; ++r) wrow[r] = W + (size_t)min(row0 + r, n - 1) * K;   // tail rows re-read the last row, never stored
        for (uint32_t k0 = lane * 8; k0 < K; k0 += 256 * U) {
            uint4 wv[U][R];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int r = 0; r < R; ++r)
                    wv[u][r] = (k0 + 256 * u < K) ? __ldcs(reinterpret_cast<const uint4 *>(wrow[r] + k0 + 256 * u)) : make_uint4(0, 0, 0, 0);
            if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t k = k0 + 256 * u;
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    float xf[8];
                    unpack8((k < K && m < (int)Mrows) ? ld_act(reinterpret_cast<const uint4 *>(A + (size_t)m * K + k)) : make_uint4(0, 0, 0, 0), xf);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        float wf[8];
                        unpack8(wv[u][r], wf);
#pragma unroll
                        for (int i = 0; i < 8; ++i) acc[r][m] = fmaf(wf[i], xf[i], acc[r][m]);
                    }
                }
            }
        }
        if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }      // K == 0 never happens; belt and braces
        // a product added to the residual stream goes out as a reduction (one add per element, by one thread: the same
        // rounded sum as load, add, store, and deterministic) that nothing waits for: the launch ends a memory round trip sooner
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const float s = warp_sum(acc[r][m]);
                if ((int)lane == r * MT + m && row0 + r < n && m < (int)Mrows) {
                    if (accumulate) atomicAdd(&C[(size_t)m * ldc + col0 + row0 + r], s);
                    else C[(size_t)m * ldc + col0 + row0 + r] = s;
                }
            }
    }
}

// Several products that read the same activations (the q, k and v projections of a layer) in one launch: the output
// rows of the parts are walked as one list, one warp per row, with exactly the arithmetic of tgp_wstream_kernel<MT, 1, U>, so
// the result is bit-identical to separate launches; what is saved is two launch floors of about a microsecond each.
// (groups[s]: CTAs' worth of rows in part s, for the kernels that walk row groups instead of rows)
struct GemvParts { const bf16 *W[TGP_GEMM_GROUP_MAX]; float *C[TGP_GEMM_GROUP_MAX]; uint32_t n[TGP_GEMM_GROUP_MAX], ldc[TGP_GEMM_GROUP_MAX], groups[TGP_GEMM_GROUP_MAX], count; };

// Where the activations of a product come from.  mode 0: bf16 rows A[m, K].  mode 1: the RMSNorm of the fp32 rows x[m, :K]
// (row stride ldx) with gain g - the warp computes the row statistics itself, exactly as tgp_rmsnorm_kernel's 256 threads
// do (lane l plays threads l, 32 + l, ... of that kernel), and rounds each normalised value to bf16 as that kernel
// stores it.  mode 2: SwiGLU of the fp32 rows g32, u32 [m, K], rounded to bf16 as tgp_swiglu_kernel stores it.  The fused
// modes give bit for bit what the separate kernels followed by mode 0 give; they save a launch and a round trip for
// the decode steps of small models, where every warp recomputing a row of a few hundred elements costs nothing.
struct ASrc { int mode; const float *x; uint32_t ldx; const bf16 *gain; float eps; const float *g32, *u32; };

__device__ __forceinline__ float rms_scale_as_kernel(const float *xrow, uint32_t d, float eps, uint32_t lane) {
    const float4 *row = reinterpret_cast<const float4 *>(xrow);
    float red[8];
#pragma unroll
    for (uint32_t w = 0; w < 8; ++w) {
        float ss = 0.f;
        for (uint32_t i = 32 * w + lane; i < d / 4; i += 256) ss = sumsq4(ss, row[i]);
        red[w] = warp_sum(ss);
    }
    float t = 0.f;
#pragma unroll
    for (uint32_t w = 0; w < 8; ++w) if (lane == w) t = red[w];
    t = warp_sum(t);
    return 1.0f / sqrtf(t / (float)d + eps);
}

__device__ __forceinline__ void act8(const ASrc &s, uint32_t m, uint32_t K, uint32_t k, float r, float *xf) {
    if (s.mode == 1) {
        const float4 *xr = reinterpret_cast<const float4 *>(s.x + (size_t)m * s.ldx + k);
        const float4 v0 = xr[0], v1 = xr[1];
        float g[8];
        unpack8(*reinterpret_cast<const uint4 *>(s.gain + k), g);
        const float v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) xf[i] = __bfloat162float(__float2bfloat16_rn(v[i] * r * g[i]));
        return;
    }
    const float4 *gr = reinterpret_cast<const float4 *>(s.g32 + (size_t)m * K + k), *ur = reinterpret_cast<const float4 *>(s.u32 + (size_t)m * K + k);
    const float4 g0 = gr[0], g1 = gr[1], u0 = ur[0], u1 = ur[1];
    const float gv[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w}, uv[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) xf[i] = __bfloat162float(__float2bfloat16_rn(gv[i] / (1.0f + expf(-gv[i])) * uv[i]));
}

// FUSED: src.mode is 1 or 2.  The plain form has its own instance: with the choice of source between them the activation loads of a
// row's U chunks waited for one another (M=1, three blocks of 3072 rows in all, K=2048: 6.0 us, 2.9 us without).
template <int MT, int U, bool FUSED>
__global__ void __launch_bounds__(256) tgp_wstream_group_kernel(const bf16 *A, const GemvParts p, uint32_t Mrows, uint32_t n_total, uint32_t K, int accumulate, const ASrc src) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarp = (gridDim.x * blockDim.x) >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool synced = false;
    float rs[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) rs[m] = 0.f;
    for (uint32_t row = gwarp; row < n_total; row += nwarp) {
        const bf16 *W = p.W[0];
        float *C = p.C[0];
        uint32_t ldc = p.ldc[0], r = row, start = p.n[0];
#pragma unroll
        for (int s = 1; s < (int)TGP_GEMM_GROUP_MAX; ++s)
            if (s < (int)p.count) {
                if (row >= start) { W = p.W[s]; C = p.C[s]; ldc = p.ldc[s]; r = row - start; }
                start += p.n[s];
            }
        const bf16 *wrow = W + (size_t)r * K;
        float acc[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) acc[m] = 0.f;
        for (uint32_t k0 = lane * 8; k0 < K; k0 += 256 * U) {
            uint4 wv[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                wv[u] = (k0 + 256 * u < K) ? __ldcs(reinterpret_cast<const uint4 *>(wrow + k0 + 256 * u)) : make_uint4(0, 0, 0, 0);
            if (!synced) {
                asm volatile("griddepcontrol.wait;" ::: "memory");
                synced = true;
                if (FUSED && src.mode == 1) {
#pragma unroll
                    for (int m = 0; m < MT; ++m) if (m < (int)Mrows) rs[m] = rms_scale_as_kernel(src.x + (size_t)m * src.ldx, K, src.eps, lane);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t k = k0 + 256 * u;
                float wf[8];
                unpack8(wv[u], wf);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    float xf[8];
                    if constexpr (!FUSED) unpack8((k < K && m < (int)Mrows) ? ld_act(reinterpret_cast<const uint4 *>(A + (size_t)m * K + k)) : make_uint4(0, 0, 0, 0), xf);
                    else if (k < K && m < (int)Mrows) act8(src, m, K, k, rs[m], xf);
                    else {
#pragma unroll
                        for (int i = 0; i < 8; ++i) xf[i] = 0.f;
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[m] = fmaf(wf[i], xf[i], acc[m]);
                }
            }
        }
        if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const float s = warp_sum(acc[m]);
            if ((int)lane == m && m < (int)Mrows) {
                if (accumulate) atomicAdd(&C[(size_t)m * ldc + r], s);
                else C[(size_t)m * ldc + r] = s;
            }
        }
    }
}

// Gate, up and SwiGLU of one or two rows in one launch, for the decode steps of a planned run: a warp takes a row of gate and the same row of up (blocks of a
// matrix are walked as one list), so that the two sums meet in its registers and only a = bf16(silu(gate) * up) is stored.  HBM bounds it as it bounds the
// products; what goes is the launch of tgp_swiglu_kernel and the ramp between the matrices.  A row's sums are those of
// tgp_wstream_kernel and the expression is that of tgp_swiglu_kernel: the same bits.
// (Whole captured runs of 48 steps, before and after: 4 layers of 2048 x 512 4.77 -> 4.44 ms, 4096 x 1024 8.27 -> 7.67, 8192 x 2048 18.28 -> 18.14, 5632 x 2048
// 15.73 -> 15.34; two rows, 8192 x 2048 20.40 -> 20.18, 2 layers of 14336 x 4096 33.95 -> 33.40, 8960 x 1536 14.30 -> 13.78.)
struct GluParts { const bf16 *gate[TGP_GEMM_GROUP_MAX / 2], *up[TGP_GEMM_GROUP_MAX / 2]; uint32_t n[TGP_GEMM_GROUP_MAX / 2], count; };

template <int MT, int U>
__global__ void __launch_bounds__(256) tgp_wstream_glu_kernel(const bf16 *A, const GluParts p, bf16 *out, uint32_t Mrows, uint32_t F, uint32_t K) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarp = (gridDim.x * blockDim.x) >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool synced = false;
    for (uint32_t row = gwarp; row < F; row += nwarp) {
        const bf16 *w[2] = {p.gate[0], p.up[0]};
        uint32_t r = row, start = p.n[0];
#pragma unroll
        for (int s = 1; s < (int)TGP_GEMM_GROUP_MAX / 2; ++s)
            if (s < (int)p.count) {
                if (row >= start) { w[0] = p.gate[s]; w[1] = p.up[s]; r = row - start; }
                start += p.n[s];
            }
        w[0] += (size_t)r * K;
        w[1] += (size_t)r * K;
        float acc[2][MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) acc[0][m] = acc[1][m] = 0.f;
        for (uint32_t k0 = lane * 8; k0 < K; k0 += 256 * U) {
            uint4 wv[U][2];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int i = 0; i < 2; ++i) wv[u][i] = (k0 + 256 * u < K) ? __ldcs(reinterpret_cast<const uint4 *>(w[i] + k0 + 256 * u)) : make_uint4(0, 0, 0, 0);
            if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t k = k0 + 256 * u;
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    float xf[8];
                    unpack8((k < K && m < (int)Mrows) ? ld_act(reinterpret_cast<const uint4 *>(A + (size_t)m * K + k)) : make_uint4(0, 0, 0, 0), xf);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        float wf[8];
                        unpack8(wv[u][i], wf);
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[i][m] = fmaf(wf[j], xf[j], acc[i][m]);
                    }
                }
            }
        }
        if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }       // a lane without columns
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const float g = warp_sum(acc[0][m]), u = warp_sum(acc[1][m]);
            if ((int)lane == m && m < (int)Mrows) out[(size_t)m * F + row] = __float2bfloat16_rn(g / (1.0f + expf(-g)) * u);
        }
    }
    if (!synced) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Same product for blocks with few rows (n below two waves of warps): one CTA of 8 warps owns RB rows and its warps
// split K in interleaved chunks of 256 elements, so n / RB CTAs spread over the SMs almost evenly where n warps of whole
// rows leave a quarter of them with half the work.  The 8 partial sums of a row meet in shared memory and are added in
// warp order: deterministic.  Same dependent-launch protocol.
template <int MT, int RB, int U>
__global__ void __launch_bounds__(256) tgp_wstream_splitk_kernel(const bf16 *A, const bf16 *__restrict__ W, float *__restrict__ C,
                                                          uint32_t Mrows, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate) {
    __shared__ float part[8][RB * MT];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool synced = false;
    for (uint32_t row0 = blockIdx.x * RB; row0 < n; row0 += gridDim.x * RB) {
        float acc[RB][MT];
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
            for (int m = 0; m < MT; ++m) acc[r][m] = 0.f;
        const bf16 *wrow[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) wrow[r] = W + (size_t)min(row0 + r, n - 1) * K;
        const bool mine = threadIdx.x < RB * MT && row0 + threadIdx.x / MT < n && threadIdx.x % MT < Mrows;
        for (uint32_t k0 = warp * 256 + lane * 8; k0 < K; k0 += 2048 * U) {
            uint4 wv[U][RB];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int r = 0; r < RB; ++r)
                    wv[u][r] = (k0 + 2048 * u < K) ? __ldcs(reinterpret_cast<const uint4 *>(wrow[r] + k0 + 2048 * u)) : make_uint4(0, 0, 0, 0);
            if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t k = k0 + 2048 * u;
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    float xf[8];
                    unpack8((k < K && m < (int)Mrows) ? ld_act(reinterpret_cast<const uint4 *>(A + (size_t)m * K + k)) : make_uint4(0, 0, 0, 0), xf);
#pragma unroll
                    for (int r = 0; r < RB; ++r) {
                        float wf[8];
                        unpack8(wv[u][r], wf);
#pragma unroll
                        for (int i = 0; i < 8; ++i) acc[r][m] = fmaf(wf[i], xf[i], acc[r][m]);
                    }
                }
            }
        }
        if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }     // a warp whose K slice is empty
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const float sacc = warp_sum(acc[r][m]);
                if (lane == 0) part[warp][r * MT + m] = sacc;
            }
        __syncthreads();
        if (mine) {
            float t = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) t += part[w][threadIdx.x];
            float *cptr = C + (size_t)(threadIdx.x % MT) * ldc + col0 + row0 + threadIdx.x / MT;
            if (accumulate) atomicAdd(cptr, t);                 // one add per element by one thread, not waited for
            else *cptr = t;
        }
        __syncthreads();
    }
}

// ---- skinny GEMM for 3 <= M <= 16 activation rows: weight streaming through mma.sync ---------------------------
// out^T[16 rows of W, 8 activation rows] += W[16 x 16] * x^T[16 x 8] per instruction.  Each lane loads 16 contiguous
// bytes (8 values of K) of W rows g and g+8 and of activation row g straight from global memory; the 8 values feed two
// instructions.  Which physical k lands in which logical k-slot of the instruction does not matter for a dot product
// as long as both operands use the same assignment, and they do (same lane, same byte offsets), so no shuffle or
// shared-memory staging is needed and every weight byte is loaded exactly once.  Persistent warps, 16 rows each,
// NB groups of 8 activation rows re-use the weight registers.  Same dependent-launch protocol as tgp_wstream_kernel.
__device__ __forceinline__ void mma_bf16_16816(float *d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

template <int NB, int U>
__global__ void __launch_bounds__(256) tgp_wstream_mma_kernel(const bf16 *A, const bf16 *__restrict__ W, float *__restrict__ C,
                                                       uint32_t Mrows, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate) {
    const uint32_t lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarp = (gridDim.x * blockDim.x) >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool synced = false;
    for (uint32_t row0 = gwarp * 16; row0 < n; row0 += nwarp * 16) {
        const bf16 *wlo = W + (size_t)min(row0 + g, n - 1) * K + c * 8;        // tail rows re-read the last row, never stored
        const bf16 *whi = W + (size_t)min(row0 + g + 8, n - 1) * K + c * 8;
        float acc[NB][4];
#pragma unroll
        for (int b = 0; b < NB; ++b) { acc[b][0] = acc[b][1] = acc[b][2] = acc[b][3] = 0.f; }
        for (uint32_t k0 = 0; k0 < K; k0 += 32 * U) {
            uint4 lo[U], hi[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool in = k0 + 32 * u < K;
                lo[u] = in ? __ldcs(reinterpret_cast<const uint4 *>(wlo + k0 + 32 * u)) : make_uint4(0, 0, 0, 0);
                hi[u] = in ? __ldcs(reinterpret_cast<const uint4 *>(whi + k0 + 32 * u)) : make_uint4(0, 0, 0, 0);
            }
            if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t k = k0 + 32 * u;
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const uint32_t m = b * 8 + g;
                    const uint4 xv = (k < K && m < Mrows) ? ld_act(reinterpret_cast<const uint4 *>(A + (size_t)m * K + k + c * 8)) : make_uint4(0, 0, 0, 0);
                    mma_bf16_16816(acc[b], lo[u].x, hi[u].x, lo[u].y, hi[u].y, xv.x, xv.y);
                    mma_bf16_16816(acc[b], lo[u].z, hi[u].z, lo[u].w, hi[u].w, xv.z, xv.w);
                }
            }
        }
        if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t m = b * 8 + 2 * c + (i & 1), row = row0 + g + 8 * (i >> 1);
                if (m < Mrows && row < n) {
                    float *p = C + (size_t)m * ldc + col0 + row;
                    if (accumulate) atomicAdd(p, acc[b][i]);      // one add per element by one thread, not waited for
                    else *p = acc[b][i];
                }
            }
    }
}

// ---- generic tiled GEMM on CUDA cores (any M, n; K % 8 == 0): 64x64 tile, 4x4 per thread ---------
__global__ void __launch_bounds__(256) tgp_matmul_simt_kernel(const bf16 *A, const bf16 *__restrict__ W, float *__restrict__ C,
                                                        uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate) {
    __shared__ float As[32][64 + 4];
    __shared__ float Ws[32][64 + 4];
    const uint32_t m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const uint32_t tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[4][4] = {};
    const uint32_t lr = threadIdx.x >> 2, lk = (threadIdx.x & 3) * 8;     // 64 rows x 4 vectors of 8
    for (uint32_t k0 = 0; k0 < K; k0 += 32) {
        float fa[8], fw[8];
        uint4 va = make_uint4(0, 0, 0, 0), vw = va;
        if (m0 + lr < M && k0 + lk < K) va = *reinterpret_cast<const uint4 *>(A + (size_t)(m0 + lr) * K + k0 + lk);
        if (n0 + lr < n && k0 + lk < K) vw = *reinterpret_cast<const uint4 *>(W + (size_t)(n0 + lr) * K + k0 + lk);
        unpack8(va, fa); unpack8(vw, fw);
#pragma unroll
        for (int i = 0; i < 8; ++i) { As[lk + i][lr] = fa[i]; Ws[lk + i][lr] = fw[i]; }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 32; ++kk) {
            float a[4], w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { a[i] = As[kk][ty * 4 + i]; w[i] = Ws[kk][tx * 4 + i]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], w[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t m = m0 + ty * 4 + i, c = n0 + tx * 4 + j;
            if (m < M && c < n) { float *p = C + (size_t)m * ldc + col0 + c; *p = accumulate ? *p + acc[i][j] : acc[i][j]; }
        }
}

// ---- RoPE + bf16 rounding + KV append -----------------------------------------------------------
// A dimension and its partner half a head away, rotated, with explicit roundings: the decode attention that rotates for itself gives the same bits.
__device__ __forceinline__ float rope_lo(float x0, float x1, float c, float s) { return __fmaf_rn(x0, c, -__fmul_rn(x1, s)); }
__device__ __forceinline__ float rope_hi(float x0, float x1, float c, float s) { return __fmaf_rn(x1, c, __fmul_rn(x0, s)); }

struct RopeArgs {
    const float *q32, *k32, *v32; bf16 *qb; const float *cos_t, *sin_t;
    uint32_t Hq, Hkv, Dh, TK, q_len, pos0;
    TgpTilePtrs tiles;
};

__global__ void tgp_rope_kv_kernel(RopeArgs a) {
    pdl_enter();
    const uint32_t m = blockIdx.x, b = m / a.q_len, pos = a.pos0 + m % a.q_len;
    const uint32_t half = a.Dh / 2, qd = a.Hq * a.Dh, kd = a.Hkv * a.Dh;
    const float *cs = a.cos_t + (size_t)pos * half, *sn = a.sin_t + (size_t)pos * half;
    const uint32_t j = pos / a.TK, slot = pos % a.TK;
    for (uint32_t idx = threadIdx.x; idx < (a.Hq + 2 * a.Hkv) * half; idx += blockDim.x) {
        const uint32_t h = idx / half, i = idx % half;
        if (h < a.Hq) {
            const float *s = a.q32 + (size_t)m * qd + h * a.Dh;
            float x0 = s[i], x1 = s[i + half], c = cs[i], sv = sn[i];
            bf16 *o = a.qb + (size_t)m * qd + h * a.Dh;
            o[i] = __float2bfloat16_rn(rope_lo(x0, x1, c, sv));
            o[i + half] = __float2bfloat16_rn(rope_hi(x0, x1, c, sv));
        } else if (h < a.Hq + a.Hkv) {
            const uint32_t hk = h - a.Hq;
            const float *s = a.k32 + (size_t)m * kd + hk * a.Dh;
            float x0 = s[i], x1 = s[i + half], c = cs[i], sv = sn[i];
            bf16 *o = reinterpret_cast<bf16 *>(a.tiles.k[j]) + ((size_t)(b * a.Hkv + hk) * a.TK + slot) * a.Dh;
            o[i] = __float2bfloat16_rn(rope_lo(x0, x1, c, sv));
            o[i + half] = __float2bfloat16_rn(rope_hi(x0, x1, c, sv));
        } else {
            const uint32_t hk = h - a.Hq - a.Hkv;
            const float *s = a.v32 + (size_t)m * kd + hk * a.Dh;
            bf16 *o = reinterpret_cast<bf16 *>(a.tiles.v[j]) + ((size_t)(b * a.Hkv + hk) * a.TK + slot) * a.Dh;
            o[i] = __float2bfloat16_rn(s[i]);
            o[i + half] = __float2bfloat16_rn(s[i + half]);
        }
    }
}

// The same for heads of 64 or 128 dimensions and 16-byte aligned buffers: a thread takes four neighbouring dimensions and their
// partners half a head away - two 16-byte loads, two 8-byte stores - and a position's heads are spread over gridDim.y CTAs,
// so that a decode step of a few sequences is one item per thread (8 positions of 48 heads x 128: 11 us with one CTA of twelve
// dependent rounds per position, 2.5 us now; 32768 positions of them: 381 us, 5.8 TB/s at 208 us now).
template <int DH>
__global__ void __launch_bounds__(256) tgp_rope_kv_vec_kernel(RopeArgs a) {
    pdl_enter();
    constexpr uint32_t HALF = DH / 2, V = HALF / 4;              // items per head
    const uint32_t m = blockIdx.x, b = m / a.q_len, pos = a.pos0 + m - b * a.q_len;
    const uint32_t qd = a.Hq * DH, kd = a.Hkv * DH, j = pos / a.TK, slot = pos - j * a.TK;
    for (uint32_t idx = blockIdx.y * blockDim.x + threadIdx.x; idx < (a.Hq + 2 * a.Hkv) * V; idx += gridDim.y * blockDim.x) {
        const uint32_t h = idx / V, i = idx % V * 4;
        const bool rot = h < a.Hq + a.Hkv;
        const uint32_t hk = h < a.Hq ? h : rot ? h - a.Hq : h - a.Hq - a.Hkv;
        const float *s = h < a.Hq ? a.q32 + (size_t)m * qd : (rot ? a.k32 : a.v32) + (size_t)m * kd;
        s += hk * DH + i;
        float4 x0 = *reinterpret_cast<const float4 *>(s), x1 = *reinterpret_cast<const float4 *>(s + HALF);
        if (rot) {
            const float4 c = *reinterpret_cast<const float4 *>(a.cos_t + (size_t)pos * HALF + i), sv = *reinterpret_cast<const float4 *>(a.sin_t + (size_t)pos * HALF + i);
            const float4 y0 = x0, y1 = x1;
            x0 = make_float4(rope_lo(y0.x, y1.x, c.x, sv.x), rope_lo(y0.y, y1.y, c.y, sv.y), rope_lo(y0.z, y1.z, c.z, sv.z), rope_lo(y0.w, y1.w, c.w, sv.w));
            x1 = make_float4(rope_hi(y0.x, y1.x, c.x, sv.x), rope_hi(y0.y, y1.y, c.y, sv.y), rope_hi(y0.z, y1.z, c.z, sv.z), rope_hi(y0.w, y1.w, c.w, sv.w));
        }
        bf16 *o = h < a.Hq ? a.qb + (size_t)m * qd + hk * DH
                           : reinterpret_cast<bf16 *>(rot ? a.tiles.k[j] : a.tiles.v[j]) + ((size_t)(b * a.Hkv + hk) * a.TK + slot) * DH;
        const __nv_bfloat162 p[4] = {__floats2bfloat162_rn(x0.x, x0.y), __floats2bfloat162_rn(x0.z, x0.w), __floats2bfloat162_rn(x1.x, x1.y), __floats2bfloat162_rn(x1.z, x1.w)};
        *reinterpret_cast<uint2 *>(o + i) = make_uint2(*reinterpret_cast<const uint32_t *>(&p[0]), *reinterpret_cast<const uint32_t *>(&p[1]));
        *reinterpret_cast<uint2 *>(o + i + HALF) = make_uint2(*reinterpret_cast<const uint32_t *>(&p[2]), *reinterpret_cast<const uint32_t *>(&p[3]));
    }
}

// ---- attention -------------------------------------------------------------------------------------
struct AttnArgs {
    const bf16 *qb; bf16 *ob; float *scratch;
    uint32_t Hq, Hkv, Dh, TK, q_len, pos0, n_tiles;
    float scale;
    TgpTilePtrs tiles;
    uint32_t n_parts;                 // partials per head the merge kernel reads; 0: one per KV tile with valid keys
    TgpRopeIn rope;                   // of the instances that rotate for themselves: the new position's projections and the tables
};

// One warp per query row, 32 keys per pass: lane = key for the scores, lane = output dims for P.V.
template <int DH>
__global__ void __launch_bounds__(128) tgp_attn_rows_kernel(AttnArgs a) {
    __shared__ float qs[4][DH];
    const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t p = blockIdx.x * 4 + w, hq = blockIdx.y, b = blockIdx.z;
    const bool live = p < a.q_len;
    const uint32_t m = b * a.q_len + (live ? p : 0), hk = hq / (a.Hq / a.Hkv);
    const bf16 *q = a.qb + (size_t)m * a.Hq * DH + hq * DH;
    for (int i = lane; i < DH; i += 32) qs[w][i] = __bfloat162float(q[i]);
    __syncwarp();
    if (!live) return;
    const uint32_t nkeys = a.pos0 + p + 1;
    constexpr int DPL = DH / 32;
    float o[DPL];
#pragma unroll
    for (int i = 0; i < DPL; ++i) o[i] = 0.f;
    float mx = -FLT_MAX, l = 0.f;                           // finite: first keys of score -inf weigh nothing
    for (uint32_t j0 = 0; j0 < nkeys; j0 += 32) {
        const uint32_t j = j0 + lane;
        float s = -INFINITY;
        if (j < nkeys) {
            const uint4 *kr = reinterpret_cast<const uint4 *>(reinterpret_cast<const bf16 *>(a.tiles.k[j / a.TK]) + ((size_t)(b * a.Hkv + hk) * a.TK + j % a.TK) * DH);
            float acc = 0.f;
#pragma unroll
            for (int v = 0; v < DH / 8; ++v) {
                float f[8];
                unpack8(kr[v], f);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc = fmaf(qs[w][v * 8 + i], f[i], acc);
            }
            s = acc * a.scale;
        }
        const float mnew = fmaxf(mx, warp_max(s));
        const float alpha = expf(mx - mnew);
        const float pj = (j < nkeys) ? expf(s - mnew) : 0.f;
        l = l * alpha + warp_sum(pj);
#pragma unroll
        for (int i = 0; i < DPL; ++i) o[i] *= alpha;
        const uint32_t cnt = min(32u, nkeys - j0);
        for (uint32_t t = 0; t < cnt; ++t) {
            const float pt = __shfl_sync(0xffffffffu, pj, t);
            const uint32_t jj = j0 + t;
            const bf16 *vr = reinterpret_cast<const bf16 *>(a.tiles.v[jj / a.TK]) + ((size_t)(b * a.Hkv + hk) * a.TK + jj % a.TK) * DH;
#pragma unroll
            for (int i = 0; i < DPL; ++i) o[i] = fmaf(pt, __bfloat162float(vr[lane + 32 * i]), o[i]);
        }
        mx = mnew;
    }
    bf16 *out = a.ob + (size_t)m * a.Hq * DH + hq * DH;
#pragma unroll
    for (int i = 0; i < DPL; ++i) out[lane + 32 * i] = __float2bfloat16_rn(o[i] / l);
}

// Decode (one query per sequence): grid (tile, kv head, batch).  The block has G x SPLIT warps: SPLIT warps share
// one query head of the group and take the tile's keys in strided 32-key passes (lane = key for the scores, lane =
// output dims for P.V, fully unrolled so a pass's V loads are in flight together); their partial (max, sum, o[Dh])
// meet in shared memory and one unnormalised partial per (query head, tile) goes to scratch.
template <int DH>
__global__ void tgp_attn_decode_partial_kernel(AttnArgs a, uint32_t SPLIT) {
    pdl_enter();
    extern __shared__ float dsm[];
    const uint32_t G = a.Hq / a.Hkv;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t g = warp / SPLIT, sp = warp % SPLIT;
    const uint32_t tile = blockIdx.x, hk = blockIdx.y, b = blockIdx.z;
    const uint32_t hq = hk * G + g;
    const uint32_t kvlen = a.pos0 + 1;
    const uint32_t nk = min(a.TK, kvlen - tile * a.TK);
    float *qs = dsm + g * DH;                               // [G][DH] query rows as fp32
    float *parts = dsm + G * DH;                            // [G][SPLIT][DH + 2]
    if (sp == 0) {
        const bf16 *q = a.qb + (size_t)b * a.Hq * DH + hq * DH;
        for (int i = lane; i < DH; i += 32) qs[i] = __bfloat162float(q[i]);
    }
    __syncthreads();
    constexpr int DPL = DH / 32;
    float o[DPL];
#pragma unroll
    for (int i = 0; i < DPL; ++i) o[i] = 0.f;
    float mx = -FLT_MAX, l = 0.f;                           // finite: first keys of score -inf weigh nothing
    const bf16 *kt = reinterpret_cast<const bf16 *>(a.tiles.k[tile]) + (size_t)(b * a.Hkv + hk) * a.TK * DH;
    const bf16 *vt = reinterpret_cast<const bf16 *>(a.tiles.v[tile]) + (size_t)(b * a.Hkv + hk) * a.TK * DH;
    for (uint32_t j0 = sp * 32; j0 < nk; j0 += SPLIT * 32) {
        const uint32_t j = j0 + lane;
        float s = -INFINITY;
        if (j < nk) {
            const uint4 *kr = reinterpret_cast<const uint4 *>(kt + (size_t)j * DH);
            float acc = 0.f;
#pragma unroll
            for (int v = 0; v < DH / 8; ++v) {
                float f[8];
                unpack8(kr[v], f);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc = fmaf(qs[v * 8 + i], f[i], acc);
            }
            s = acc * a.scale;
        }
        const float mnew = fmaxf(mx, warp_max(s));
        const float alpha = expf(mx - mnew);
        const float pj = (j < nk) ? expf(s - mnew) : 0.f;
        l = l * alpha + warp_sum(pj);
#pragma unroll
        for (int i = 0; i < DPL; ++i) o[i] *= alpha;
        const uint32_t cnt = min(32u, nk - j0);
#pragma unroll
        for (uint32_t t = 0; t < 32; ++t) {                 // rows past the end re-read the last valid row with weight 0
            const float pt = __shfl_sync(0xffffffffu, pj, t);
            const bf16 *vr = vt + (size_t)(j0 + min(t, cnt - 1)) * DH;
#pragma unroll
            for (int i = 0; i < DPL; ++i) o[i] = fmaf(pt, __bfloat162float(vr[lane + 32 * i]), o[i]);
        }
        mx = mnew;
    }
    float *mine = parts + (size_t)(g * SPLIT + sp) * (DH + 2);
    if (lane == 0) { mine[0] = mx; mine[1] = l; }
#pragma unroll
    for (int i = 0; i < DPL; ++i) mine[2 + lane + 32 * i] = o[i];
    __syncthreads();
    if (sp == 0) {                                          // fixed-order merge of the SPLIT partials of this head
        const float *p0 = parts + (size_t)g * SPLIT * (DH + 2);
        float m = -INFINITY;
        for (uint32_t k = 0; k < SPLIT; ++k) m = fmaxf(m, p0[k * (DH + 2)]);
        float lsum = 0.f, acc[DPL];
#pragma unroll
        for (int i = 0; i < DPL; ++i) acc[i] = 0.f;
        for (uint32_t k = 0; k < SPLIT; ++k) {
            const float w = expf(p0[k * (DH + 2)] - m);     // a warp that saw no key has the lowest finite max and sums of 0
            lsum += w * p0[k * (DH + 2) + 1];
#pragma unroll
            for (int i = 0; i < DPL; ++i) acc[i] += w * p0[k * (DH + 2) + 2 + lane + 32 * i];
        }
        float *part = a.scratch + ((size_t)(b * a.Hq + hq) * a.n_tiles + tile) * (DH + 2);
        if (lane == 0) { part[0] = m; part[1] = lsum; }
#pragma unroll
        for (int i = 0; i < DPL; ++i) part[2 + lane + 32 * i] = acc[i];
    }
}

// Merge the per-tile partials of one (batch, query head): grid (Hq, B), DH threads.
// Decode attention over one KV tile for all G query heads of a KV head at once (G = Hq / Hkv in {1, 2, 4, 8}): the tile's
// K and V rows are read once, not once per query head.  One CTA per (tile, KV head, sequence); warp w walks the keys
// w*32, (w + SPLIT)*32, ... of the tile in chunks of 32: lane = key for the scores (the lane reads its whole K row with
// 16-byte loads, all in flight at once, and dots it with the G queries held in shared memory), then lane = DH/32
// consecutive output dimensions for P V (each V row is one coalesced warp load; the G weights of a key come by
// shuffle).  Per-warp online softmax; the SPLIT partials of a head are merged in warp order; output as in the
// per-head kernel: (max, sum, unnormalised o[DH]) per (sequence, head, tile) for tgp_attn_decode_merge_kernel.
template <int DH, int G>
__global__ void __launch_bounds__(256, 2) tgp_attn_decode_group_kernel(AttnArgs a, uint32_t SPLIT) {
    pdl_enter();
    extern __shared__ float dsm[];
    constexpr int DPL = DH / 32;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tile = blockIdx.x, hk = blockIdx.y, b = blockIdx.z;
    const uint32_t kvlen = a.pos0 + 1;
    const uint32_t nk = min(a.TK, kvlen - tile * a.TK);
    float *qs = dsm;                                        // [G][DH] query rows as fp32
    float *parts = dsm + G * DH;                            // [G][SPLIT][DH + 2]
    {
        const bf16 *q = a.qb + ((size_t)b * a.Hq + hk * G) * DH;          // the G heads of this group are contiguous
        for (uint32_t i = threadIdx.x; i < G * DH; i += blockDim.x) qs[i] = __bfloat162float(q[i]);
    }
    __syncthreads();
    float o[G][DPL], mx[G], l[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        mx[g] = -FLT_MAX; l[g] = 0.f;                      // finite: first keys of score -inf weigh nothing
#pragma unroll
        for (int i = 0; i < DPL; ++i) o[g][i] = 0.f;
    }
    const bf16 *kt = reinterpret_cast<const bf16 *>(a.tiles.k[tile]) + (size_t)(b * a.Hkv + hk) * a.TK * DH;
    const bf16 *vt = reinterpret_cast<const bf16 *>(a.tiles.v[tile]) + (size_t)(b * a.Hkv + hk) * a.TK * DH;
    for (uint32_t j0 = warp * 32; j0 < nk; j0 += SPLIT * 32) {
        const uint32_t j = j0 + lane, cnt = min(32u, nk - j0);
        const bool valid = j < nk;
        // the first 16 value rows are requested before the scores are computed: they depend on nothing computed here, and
        // the chunk is one serial chain per warp (key rows, scores, softmax, value rows), so every load moved off it counts
        typedef typename std::conditional<DPL == 4, uint2, uint32_t>::type vraw_t;
        constexpr uint32_t PRE = (G * DPL >= 32) ? 4 : 16;          // eight heads of 128 dimensions leave few registers for it
        vraw_t vpre[PRE];
#pragma unroll
        for (uint32_t t = 0; t < PRE; ++t)
            vpre[t] = *reinterpret_cast<const vraw_t *>(vt + (size_t)(j0 + min(t, cnt - 1)) * DH + lane * DPL);
        // ---- scores: this lane's key against the G queries ----
        float acc[G];
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] = 0.f;
        {
            const uint4 *kr = reinterpret_cast<const uint4 *>(kt + (size_t)min(j, nk - 1) * DH);
            uint4 kv[4], nx[4];                                      // 64 bytes of the row at a time, the next 64 already requested
#pragma unroll
            for (int v = 0; v < 4; ++v) kv[v] = kr[v];
#pragma unroll 1
            for (int v0 = 0; v0 < DH / 8; v0 += 4) {
                if (v0 + 4 < DH / 8) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) nx[v] = kr[v0 + 4 + v];
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    float f[8];
                    unpack8(kv[v], f);
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const float4 q0 = *reinterpret_cast<const float4 *>(qs + g * DH + (v0 + v) * 8), q1 = *reinterpret_cast<const float4 *>(qs + g * DH + (v0 + v) * 8 + 4);
                        acc[g] = fmaf(q0.x, f[0], acc[g]); acc[g] = fmaf(q0.y, f[1], acc[g]); acc[g] = fmaf(q0.z, f[2], acc[g]); acc[g] = fmaf(q0.w, f[3], acc[g]);
                        acc[g] = fmaf(q1.x, f[4], acc[g]); acc[g] = fmaf(q1.y, f[5], acc[g]); acc[g] = fmaf(q1.z, f[6], acc[g]); acc[g] = fmaf(q1.w, f[7], acc[g]);
                    }
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) kv[v] = nx[v];
            }
        }
        float p[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float sc = valid ? acc[g] * a.scale : -INFINITY;
            const float mnew = fmaxf(mx[g], warp_max(sc));
            const float alpha = expf(mx[g] - mnew);
            p[g] = valid ? expf(sc - mnew) : 0.f;
            l[g] = l[g] * alpha + warp_sum(p[g]);
#pragma unroll
            for (int i = 0; i < DPL; ++i) o[g][i] *= alpha;
            mx[g] = mnew;
        }
        // ---- P V: this lane's DPL output dimensions; rows past the end re-read the last valid row with weight 0 ----
        vraw_t vlate[16];
#pragma unroll
        for (uint32_t t = 0; t < 16; ++t)
            vlate[t] = *reinterpret_cast<const vraw_t *>(vt + (size_t)(j0 + min(t + PRE, cnt - 1)) * DH + lane * DPL);
#pragma unroll
        for (uint32_t t = 0; t < 32; ++t) {
            if constexpr (PRE < 16) {                                // fewer than 16 rows were requested early: a third batch
                if (t == PRE + 16) {
#pragma unroll
                    for (uint32_t u = 0; u + PRE < 16; ++u)
                        vlate[u] = *reinterpret_cast<const vraw_t *>(vt + (size_t)(j0 + min(u + PRE + 16, cnt - 1)) * DH + lane * DPL);
                }
            }
            const vraw_t raw = t < PRE ? vpre[t % PRE] : vlate[(t - PRE) % 16];
            float f[DPL];
            if constexpr (DPL == 4) {
                const __nv_bfloat162 a0 = *reinterpret_cast<const __nv_bfloat162 *>(&raw.x), a1 = *reinterpret_cast<const __nv_bfloat162 *>(&raw.y);
                f[0] = __low2float(a0); f[1] = __high2float(a0); f[2] = __low2float(a1); f[3] = __high2float(a1);
            } else {
                const __nv_bfloat162 a0 = *reinterpret_cast<const __nv_bfloat162 *>(&raw);
                f[0] = __low2float(a0); f[1 % DPL] = __high2float(a0);
            }
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const float pt = __shfl_sync(0xffffffffu, p[g], t);
#pragma unroll
                for (int i = 0; i < DPL; ++i) o[g][i] = fmaf(pt, f[i], o[g][i]);
            }
        }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
        float *mine = parts + (size_t)(g * SPLIT + warp) * (DH + 2);
        if (lane == 0) { mine[0] = mx[g]; mine[1] = l[g]; }
#pragma unroll
        for (int i = 0; i < DPL; ++i) mine[2 + lane * DPL + i] = o[g][i];
    }
    __syncthreads();
    for (uint32_t g = warp; g < G; g += SPLIT) {            // fixed-order merge of the SPLIT partials of head g
        const float *p0 = parts + (size_t)g * SPLIT * (DH + 2);
        float m = -INFINITY;
        for (uint32_t k = 0; k < SPLIT; ++k) m = fmaxf(m, p0[k * (DH + 2)]);
        float lsum = 0.f, accm[DPL];
#pragma unroll
        for (int i = 0; i < DPL; ++i) accm[i] = 0.f;
        for (uint32_t k = 0; k < SPLIT; ++k) {
            const float w = expf(p0[k * (DH + 2)] - m);     // a warp that saw no key has the lowest finite max and sums of 0
            lsum += w * p0[k * (DH + 2) + 1];
#pragma unroll
            for (int i = 0; i < DPL; ++i) accm[i] += w * p0[k * (DH + 2) + 2 + lane * DPL + i];
        }
        float *part = a.scratch + ((size_t)(b * a.Hq + hk * G + g) * a.n_tiles + tile) * (DH + 2);
        if (lane == 0) { part[0] = m; part[1] = lsum; }
#pragma unroll
        for (int i = 0; i < DPL; ++i) part[2 + lane * DPL + i] = accm[i];
    }
}

// One warp holds 32 partials' maxima and sums in its lanes at a time, so the loads of a round are independent of one another, and the
// outputs of four partials are under way at once: two latencies for up to 32 partials instead of two per partial.
template <int DH>
__global__ void __launch_bounds__(DH) tgp_attn_decode_merge_kernel(AttnArgs a) {
    pdl_enter();
    const uint32_t hq = blockIdx.x, b = blockIdx.y, i = threadIdx.x, lane = threadIdx.x & 31;
    const uint32_t nt = a.n_parts ? a.n_parts : (a.pos0 + 1 + a.TK - 1) / a.TK;
    const float *part = a.scratch + (size_t)(b * a.Hq + hq) * a.n_tiles * (DH + 2);
    float m0 = lane < nt ? part[lane * (DH + 2)] : -INFINITY, mx = m0;
    const float l0 = lane < nt ? part[lane * (DH + 2) + 1] : 0.f;
    for (uint32_t t = lane + 32; t < nt; t += 32) mx = fmaxf(mx, part[t * (DH + 2)]);
    mx = warp_max(mx);
    float l = 0.f, o = 0.f, w = 0.f, lw = 0.f;
    for (uint32_t t0 = 0; t0 < nt; t0 += 4) {
        float v[4];
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) v[q] = t0 + q < nt ? part[(t0 + q) * (DH + 2) + 2 + i] : 0.f;
        if ((t0 & 31) == 0) {                                  // the weights of the next 32 partials, one per lane
            const uint32_t t = t0 + lane;
            const float mt = t0 == 0 ? m0 : t < nt ? part[t * (DH + 2)] : -INFINITY;
            lw = t0 == 0 ? l0 : t < nt ? part[t * (DH + 2) + 1] : 0.f;
            w = t < nt ? expf(mt - mx) : 0.f;
        }
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (t0 + q < nt) {
                const float wt = __shfl_sync(0xffffffffu, w, (t0 + q) & 31), lt = __shfl_sync(0xffffffffu, lw, (t0 + q) & 31);
                l += wt * lt;
                o += wt * v[q];
            }
    }
    a.ob[(size_t)b * a.Hq * DH + hq * DH + i] = __float2bfloat16_rn(o / l);
}

// ---- decode attention on the tensor cores (mma.sync), K and V staged through shared memory ---------------------------------
// The group kernel above is a latency chain: a warp's 32-key chunk is loads, 4*G*Dh FMAs per lane and shuffles, one after
// the other, and a B200 needs ~35 KB in flight per SM to keep HBM busy.  Here the G query heads of a KV head are the rows
// of a 16-row MMA tile (rows >= G are zero), a warp works on chunks of 16 keys, and the K and V rows of the next chunks are
// already on their way: every warp owns DEC_STAGES private stages that it fills with cp.async (16 bytes per lane and
// instruction, rows past the sequence zero-filled) - no block-wide barrier in the key loop.  Per chunk:
//   S[16 x 16 keys] = Q K^T      2 x Dh/16 MMAs (m16n8k16, bf16 -> fp32), K fragments by ldmatrix from the swizzled stage;
//   online softmax per row       (the running maximum moves rarely: O is rescaled only when a row's maximum grew);
//   O[16 x Dh] += P V            Dh/8 MMAs, P straight from the S accumulators as the A fragment, V fragments by
//                                ldmatrix.trans (V rows are keys: the transposed load makes keys the contraction index).
// P is rounded to bf16 for the second product, as in the prefill kernels; in short contexts (SPLIT_P) it counts with all of its 24 bits:
// as three bf16 parts, each what the rounding of those before it left over.  The second part takes the rows 8 - 15 that the
// tile has to spare, the third a product of its own.  Both are summed apart from the first and dropped where that sum is not
// finite: an infinity in V makes their products NaN (0 x inf), and the first part alone says what the row becomes.
// A CTA of four warps owns a contiguous range of
// chunks of one (sequence, KV head); its warps take every fourth chunk and merge their four partials through shared memory.  The CTAs of
// one (sequence, KV head) are a cluster where they are few and merge theirs through distributed shared memory (one sequence of 32 heads over
// 8 x 64, 400 keys: 4.6 -> 3.4 us); else each writes one (max, sum, unnormalised O) per query head to the scratch array
// that tgp_attn_decode_merge_kernel reads.
// Stage layout: row = key, 2*DH bytes, 16-byte chunk j of row r at chunk position j ^ (r & 7): conflict-free for the
// ldmatrix reads (eight rows, same j) and for the cp.async writes.
constexpr int DEC_STAGES = 3, DEC_WARPS = 4, DEC_KEYS = 16, DEC_CLUSTER = 8;

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float fast_ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

// (CLUSTER is an instance of its own: what only clusters need makes the others 5 - 14 % slower.  The second bound is the number of CTAs that
// shared memory leaves room for: told so, the compiler keeps its loads apart with 177 - 179 registers at DH = 128; left to itself it takes 141 to 165,
// by what the instance holds besides, and is up to 20 % slower: 8 heads over one, 9000 keys of one sequence 19.1 -> 15.0 us with the norm before, in clusters 3 - 6 %.  All bits of P
// take 151 registers at DH = 64, and the few CTAs they are for fit an SM in threes.)
// ROPE: the kernel does what tgp_rope_kv_vec_kernel does, too, with its bits: every CTA rotates its queries in registers, and the warp whose chunk holds the new
// position rotates its key, puts key and value into the stage behind the copies, and writes both to the tiles.  One launch and its hand-over less per layer
// of a decode step (one sequence, 16 layers of 32 heads over 8 x 64, a run of 192 steps: 41.2 -> 40.5 ms).
template <int DH, int G, bool SPLIT_P, bool CLUSTER, bool ROPE>
__global__ void __launch_bounds__(DEC_WARPS * 32, DH == 128 ? 2 : SPLIT_P ? 3 : 4) tgp_attn_decode_mma_kernel(AttnArgs a, uint32_t chunks_per_cta) {
    pdl_enter();
    extern __shared__ __align__(128) uint8_t dec_sm[];
    constexpr uint32_t ROW = DH * 2, CPR = ROW / 16;                  // bytes and 16-byte chunks per key row
    constexpr uint32_t KV_BYTES = DEC_KEYS * ROW, STAGE = 2 * KV_BYTES;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
    const uint32_t part = blockIdx.x, hk = blockIdx.y, b = blockIdx.z;
    const uint32_t kvlen = a.pos0 + 1, nchunks = (kvlen + DEC_KEYS - 1) / DEC_KEYS;
    const uint32_t q_lo = part * chunks_per_cta, q_hi = min(nchunks, q_lo + chunks_per_cta);
    uint8_t *mine = dec_sm + (size_t)warp * DEC_STAGES * STAGE;
    const uint32_t mine_u = (uint32_t)__cvta_generic_to_shared(mine);
    const float sl2 = a.scale * 1.4426950408889634f;                  // scores are kept in units of log2

    // Q fragments of this group: rows 0..G-1 real, the rest zero; held in registers for the whole kernel
    uint32_t qf[DH / 16][2];
    constexpr uint32_t HALF = DH / 2;
    auto bits2 = [](float lo, float hi) { const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi); return *reinterpret_cast<const uint32_t *>(&p); };
    uint32_t new_k[2] = {0u, 0u}, new_v[2] = {0u, 0u};                // ROPE: dimensions 2 lane and half a head on of the new key and value
    const uint32_t in_tiles = ROPE ? kvlen - 1 : kvlen;               // keys that the tiles hold
    if constexpr (ROPE) {
        const float *cs = a.rope.cos_t + (size_t)a.pos0 * HALF, *sn = a.rope.sin_t + (size_t)a.pos0 * HALF;
        const float *q = a.rope.q32 + ((size_t)b * a.Hq + hk * G + (r < G ? r : 0)) * DH;
#pragma unroll
        for (int ks = 0; ks < DH / 32; ++ks)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint32_t i = ks * 16 + 2 * c + 8 * e;
                const float2 x0 = *reinterpret_cast<const float2 *>(q + i), x1 = *reinterpret_cast<const float2 *>(q + HALF + i);
                const float2 co = *reinterpret_cast<const float2 *>(cs + i), si = *reinterpret_cast<const float2 *>(sn + i);
                qf[ks][e] = r < G ? bits2(rope_lo(x0.x, x1.x, co.x, si.x), rope_lo(x0.y, x1.y, co.y, si.y)) : 0u;
                qf[ks + DH / 32][e] = r < G ? bits2(rope_hi(x0.x, x1.x, co.x, si.x), rope_hi(x0.y, x1.y, co.y, si.y)) : 0u;
            }
        if (q_hi == nchunks && (nchunks - 1 - q_lo) % DEC_WARPS == warp && 2 * lane < HALF) {      // this warp has the chunk of the new position
            const size_t row = ((size_t)b * a.Hkv + hk) * DH;
            const uint32_t i = 2 * lane, tile = a.pos0 / a.TK;
            const float2 x0 = *reinterpret_cast<const float2 *>(a.rope.k32 + row + i), x1 = *reinterpret_cast<const float2 *>(a.rope.k32 + row + HALF + i);
            const float2 v0 = *reinterpret_cast<const float2 *>(a.rope.v32 + row + i), v1 = *reinterpret_cast<const float2 *>(a.rope.v32 + row + HALF + i);
            const float2 co = *reinterpret_cast<const float2 *>(cs + i), si = *reinterpret_cast<const float2 *>(sn + i);
            new_k[0] = bits2(rope_lo(x0.x, x1.x, co.x, si.x), rope_lo(x0.y, x1.y, co.y, si.y));
            new_k[1] = bits2(rope_hi(x0.x, x1.x, co.x, si.x), rope_hi(x0.y, x1.y, co.y, si.y));
            new_v[0] = bits2(v0.x, v0.y);
            new_v[1] = bits2(v1.x, v1.y);
            const size_t at = (((size_t)b * a.Hkv + hk) * a.TK + (a.pos0 - tile * a.TK)) * DH + i;
            bf16 *kt = reinterpret_cast<bf16 *>(a.tiles.k[tile]) + at, *vt = reinterpret_cast<bf16 *>(a.tiles.v[tile]) + at;
            *reinterpret_cast<uint32_t *>(kt) = new_k[0]; *reinterpret_cast<uint32_t *>(kt + HALF) = new_k[1];
            *reinterpret_cast<uint32_t *>(vt) = new_v[0]; *reinterpret_cast<uint32_t *>(vt + HALF) = new_v[1];
        }
    } else {
        const bf16 *q = a.qb + ((size_t)b * a.Hq + hk * G) * DH + (size_t)r * DH;
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) {
            qf[ks][0] = r < G ? *reinterpret_cast<const uint32_t *>(q + ks * 16 + 2 * c) : 0u;
            qf[ks][1] = r < G ? *reinterpret_cast<const uint32_t *>(q + ks * 16 + 2 * c + 8) : 0u;
        }
    }
    // chunk q: its KV tile and offset; lane l copies 16-byte pieces idx = i * 32 + l of the chunk's K and V rows
    auto issue = [&](uint32_t q, uint32_t stage) {
        const uint32_t key0 = q * DEC_KEYS, tile = key0 / a.TK, off = key0 - tile * a.TK;
        const uint8_t *kg = reinterpret_cast<const uint8_t *>(a.tiles.k[tile]) + ((size_t)(b * a.Hkv + hk) * a.TK + off) * ROW;
        const uint8_t *vg = reinterpret_cast<const uint8_t *>(a.tiles.v[tile]) + ((size_t)(b * a.Hkv + hk) * a.TK + off) * ROW;
        const uint32_t base = mine_u + stage * STAGE;
#pragma unroll
        for (uint32_t i = 0; i < DEC_KEYS * CPR / 32; ++i) {
            const uint32_t idx = i * 32 + lane, row = idx / CPR, j = idx % CPR;
            const uint32_t dst = row * ROW + ((j ^ (row & 7)) << 4);
            const uint32_t nbytes = key0 + row < in_tiles ? 16u : 0u;  // rows past the sequence are written as zeros, not read
            cp_async16(base + dst, kg + (size_t)row * ROW + j * 16, nbytes);
            cp_async16(base + KV_BYTES + dst, vg + (size_t)row * ROW + j * 16, nbytes);
        }
    };
    // this warp's chunks: q_lo + warp, q_lo + warp + 4, ...
    uint32_t issued = 0, total = 0;
    for (uint32_t q = q_lo + warp; q < q_hi; q += DEC_WARPS) ++total;
#pragma unroll
    for (int s = 0; s < DEC_STAGES - 1; ++s) {
        if (issued < total) { issue(q_lo + warp + issued * DEC_WARPS, issued % DEC_STAGES); ++issued; }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    float o[DH / 8][4], o3[SPLIT_P ? DH / 8 : 1][4];                  // o: the first part of P in elements 0 and 1, the second in 2 and 3; o3: the third
#pragma unroll
    for (int j = 0; j < DH / 8; ++j) {
        o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
        if constexpr (SPLIT_P) o3[j][0] = o3[j][1] = o3[j][2] = o3[j][3] = 0.f;
    }
    // The maximum starts at the least number, not at -inf: keys of score -inf weigh nothing then (ex2(-inf - it) = 0) wherever a warp's chunks
    // begin, while from -inf the first of them would be ex2(-inf + inf) = NaN, and which keys those are depends on the number of parts
    float m_run = -FLT_MAX, l_run = 0.f;                              // of row r (replicated over the four lanes of the row)
    for (uint32_t it = 0; it < total; ++it) {
        if (issued < total) { issue(q_lo + warp + issued * DEC_WARPS, issued % DEC_STAGES); ++issued; }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group %0;" ::"n"(DEC_STAGES - 1) : "memory");
        __syncwarp();
        const uint32_t q = q_lo + warp + it * DEC_WARPS, key0 = q * DEC_KEYS;
        const uint32_t kb = mine_u + (it % DEC_STAGES) * STAGE, vb = kb + KV_BYTES;
        if (ROPE && q + 1 == nchunks) {                               // the new position's row, over the zeros that the copy has put there
            const uint32_t row = a.pos0 - key0;
            if (2 * lane < HALF)
#pragma unroll
                for (uint32_t e = 0; e < 2; ++e) {
                    const uint32_t i = 2 * lane + e * HALF, at = row * ROW + ((i / 8 ^ (row & 7)) << 4) + i % 8 * 2;
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(kb + at), "r"(new_k[e]) : "memory");
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(vb + at), "r"(new_v[e]) : "memory");
                }
            __syncwarp();
        }
        // ---- S = Q K^T: two n-tiles of 8 keys ----
        float sacc[2][4];
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            sacc[nt][0] = sacc[nt][1] = sacc[nt][2] = sacc[nt][3] = 0.f;
#pragma unroll
            for (int kp = 0; kp < DH / 32; ++kp) {
                const uint32_t row = nt * 8 + (lane & 7), j = kp * 4 + (lane >> 3);
                uint32_t b0, b1, b2, b3;
                ldsm_x4(kb + row * ROW + ((j ^ (row & 7)) << 4), b0, b1, b2, b3);
                mma_bf16(sacc[nt], qf[2 * kp][0], 0u, qf[2 * kp][1], 0u, b0, b1);
                mma_bf16(sacc[nt], qf[2 * kp + 1][0], 0u, qf[2 * kp + 1][1], 0u, b2, b3);
            }
        }
        // ---- online softmax of row r over the chunk's 16 keys (this lane: keys 2c, 2c+1, 8+2c, 9+2c) ----
        float sv[4] = {sacc[0][0] * sl2, sacc[0][1] * sl2, sacc[1][0] * sl2, sacc[1][1] * sl2};
        if (key0 + DEC_KEYS > kvlen) {
            const uint32_t kk[4] = {2 * c, 2 * c + 1, 8 + 2 * c, 9 + 2 * c};
#pragma unroll
            for (int i = 0; i < 4; ++i) if (key0 + kk[i] >= kvlen) sv[i] = -INFINITY;
        }
        float mx = fmaxf(fmaxf(sv[0], sv[1]), fmaxf(sv[2], sv[3]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run, mx);
        if (__any_sync(0xffffffffu, m_new > m_run)) {
            const float alpha = fast_ex2(m_run - m_new);              // first chunk: on zeros
            l_run *= alpha;
#pragma unroll
            for (int j = 0; j < DH / 8; ++j) {
                o[j][0] *= alpha; o[j][1] *= alpha;
                if constexpr (SPLIT_P) { o[j][2] *= alpha; o[j][3] *= alpha; o3[j][0] *= alpha; o3[j][1] *= alpha; }
            }
            m_run = m_new;
        }
        float p[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i] = fast_ex2(sv[i] - m_run);
        float ls = (p[0] + p[1]) + (p[2] + p[3]);
        ls += __shfl_xor_sync(0xffffffffu, ls, 1);
        ls += __shfl_xor_sync(0xffffffffu, ls, 2);
        l_run += ls;
        // rounds p to bf16 and leaves the remainder in it
        auto take_part = [&](uint32_t &lo, uint32_t &hi) {
            const __nv_bfloat162 a01 = __floats2bfloat162_rn(p[0], p[1]), a23 = __floats2bfloat162_rn(p[2], p[3]);
            p[0] -= __low2float(a01); p[1] -= __high2float(a01); p[2] -= __low2float(a23); p[3] -= __high2float(a23);
            lo = *reinterpret_cast<const uint32_t *>(&a01); hi = *reinterpret_cast<const uint32_t *>(&a23);
        };
        uint32_t pa0, pa2, pb0 = 0, pb2 = 0, pc0 = 0, pc2 = 0;
        take_part(pa0, pa2);
        if constexpr (SPLIT_P) { take_part(pb0, pb2); take_part(pc0, pc2); }
        // ---- O += P V: Dh/8 n-tiles, two per ldmatrix ----
#pragma unroll
        for (int jp = 0; jp < DH / 16; ++jp) {
            const uint32_t row = ((lane >> 3) & 1) * 8 + (lane & 7), j = 2 * jp + (lane >> 4);
            uint32_t v0, v1, v2, v3;
            ldsm_x4_t(vb + row * ROW + ((j ^ (row & 7)) << 4), v0, v1, v2, v3);
            mma_bf16(o[2 * jp], pa0, pb0, pa2, pb2, v0, v1);
            mma_bf16(o[2 * jp + 1], pa0, pb0, pa2, pb2, v2, v3);
            if constexpr (SPLIT_P) { mma_bf16(o3[2 * jp], pc0, 0u, pc2, 0u, v0, v1); mma_bf16(o3[2 * jp + 1], pc0, 0u, pc2, 0u, v2, v3); }
        }
        __syncwarp();                                                 // the stage may be refilled two iterations from now
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if constexpr (SPLIT_P) {
#pragma unroll
        for (int j = 0; j < DH / 8; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float rest = o[j][2 + i] + o3[j][i];
                if (fabsf(rest) < INFINITY) o[j][i] += rest;
            }
    }
    // ---- merge the four warps' partials (rows < G), write one partial per head for this CTA ----
    // (each warp's partial goes to the start of its own stages, which it no longer needs: [G][DH + 2] floats)
    __syncwarp();
    constexpr size_t WSTRIDE = (size_t)DEC_STAGES * STAGE / sizeof(float);
    float *wp = reinterpret_cast<float *>(dec_sm);
    if (r < G) {
        float *dst = wp + (size_t)warp * WSTRIDE + (size_t)r * (DH + 2);
        // (NaN scores: the sum is NaN and makes the row NaN with any weight; a row of nothing but -inf: 0 / 0)
        if (c == 0) { dst[0] = m_run; dst[1] = l_run; }
#pragma unroll
        for (int j = 0; j < DH / 8; ++j) { dst[2 + j * 8 + 2 * c] = o[j][0]; dst[2 + j * 8 + 2 * c + 1] = o[j][1]; }
    }
    __syncthreads();
    constexpr uint32_t CLUSTER_AT = 16 * DH;                              // floats: behind the partial of warp 0, in stages nobody reads any more
    static_assert(CLUSTER_AT >= G * (DH + 2) && CLUSTER_AT + G * (DH + 2) <= WSTRIDE, "the CTA's partial lies in warp 0's stages");
    for (uint32_t e = threadIdx.x; e < G * DH; e += blockDim.x) {
        const uint32_t g = e / DH, d = e % DH;
        float M = -FLT_MAX;
#pragma unroll
        for (int w = 0; w < DEC_WARPS; ++w) M = fmaxf(M, wp[(size_t)w * WSTRIDE + (size_t)g * (DH + 2)]);
        float l = 0.f, acc = 0.f;
#pragma unroll
        for (int w = 0; w < DEC_WARPS; ++w) {
            const float *src = wp + (size_t)w * WSTRIDE + (size_t)g * (DH + 2);
            const float wgt = fast_ex2(src[0] - M);                        // (a warp without a chunk: any weight of zeros)
            l += wgt * src[1];
            acc += wgt * src[2 + d];
        }
        if (!CLUSTER && a.n_parts == 1) {                                  // the CTA saw the whole context: this is the result
            a.ob[((size_t)b * a.Hq + hk * G + g) * DH + d] = __float2bfloat16_rn(acc / l);
            continue;
        }
        if constexpr (CLUSTER) {
            float *cp = wp + CLUSTER_AT + (size_t)g * (DH + 2);
            if (d == 0) { cp[0] = M; cp[1] = l; }
            cp[2 + d] = acc;
            continue;
        }
        float *out = a.scratch + ((size_t)(b * a.Hq + hk * G + g) * a.n_tiles + part) * (DH + 2);
        if (d == 0) { out[0] = M * 0.6931471805599453f; out[1] = l; }      // the merge kernel works in natural-log units
        out[2 + d] = acc;
    }
    if constexpr (!CLUSTER) return;
    // The CTAs of a cluster are the parts of one sequence and KV head: every CTA takes a share of the outputs and reads all partials of it.
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const uint32_t cp_u = (uint32_t)__cvta_generic_to_shared(wp + CLUSTER_AT), rank = part, ctas = gridDim.x;
    auto remote = [&](uint32_t part_at, uint32_t offset) {
        uint32_t at;
        float v;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(cp_u + offset * 4), "r"(part_at));
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
        return v;
    };
    for (uint32_t e = G * DH * rank / ctas + threadIdx.x; e < G * DH * (rank + 1) / ctas; e += blockDim.x) {
        const uint32_t g = e / DH, d = e % DH;
        float m[DEC_CLUSTER], l[DEC_CLUSTER], o_p[DEC_CLUSTER], M = -FLT_MAX;
#pragma unroll
        for (uint32_t q = 0; q < DEC_CLUSTER; ++q)
            if (q < ctas) { m[q] = remote(q, g * (DH + 2)); l[q] = remote(q, g * (DH + 2) + 1); o_p[q] = remote(q, g * (DH + 2) + 2 + d); }
#pragma unroll
        for (uint32_t q = 0; q < DEC_CLUSTER; ++q) if (q < ctas) M = fmaxf(M, m[q]);
        float lsum = 0.f, acc = 0.f;
#pragma unroll
        for (uint32_t q = 0; q < DEC_CLUSTER; ++q)
            if (q < ctas) { const float w = fast_ex2(m[q] - M); lsum += w * l[q]; acc += w * o_p[q]; }
        a.ob[((size_t)b * a.Hq + hk * G + g) * DH + d] = __float2bfloat16_rn(acc / lsum);
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");        // no CTA leaves while another may still read its partial
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---- SwiGLU -----------------------------------------------------------------------------------------
__global__ void tgp_swiglu_kernel(const float4 *g, const float4 *u, __nv_bfloat162 *out, uint64_t n4) {
    pdl_enter();
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n4; i += (uint64_t)gridDim.x * blockDim.x) {
        float4 a = g[i], b = u[i];
        float r0 = a.x / (1.0f + expf(-a.x)) * b.x, r1 = a.y / (1.0f + expf(-a.y)) * b.y;
        float r2 = a.z / (1.0f + expf(-a.z)) * b.z, r3 = a.w / (1.0f + expf(-a.w)) * b.w;
        out[2 * i] = __floats2bfloat162_rn(r0, r1);
        out[2 * i + 1] = __floats2bfloat162_rn(r2, r3);
    }
}

// ---- argmax, lowest index on ties -----------------------------------------------------------------
// A row is shared by the CTAs of a cluster (up to 8 for long rows): each scans a contiguous part with four independent 16-byte loads per
// thread under way, and the parts' winners meet in the first CTA's shared memory (8 rows of 32000: 9.5 us with one CTA of 1024
// threads and one dependent element per thread and round, 3.4 us now, from the end of the kernel before).
__global__ void __launch_bounds__(256) tgp_argmax_kernel(const float *logits, int32_t *out, int32_t *out2, uint32_t V, int vec) {
    pdl_enter();
    __shared__ float bv[8], cv[8];
    __shared__ uint32_t bi[8], ci[8];
    uint32_t rank, parts;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(parts));
    // (the wait stands before the first access to the first CTA's memory: only then is that CTA known to run, however short this part is)
    if (parts > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float *row = logits + (size_t)(blockIdx.x / parts) * V;
    const uint32_t per = ((V + parts - 1) / parts + 3) / 4 * 4, lo = min(V, rank * per), hi = min(V, lo + per);
    // the index starts at 0, not at a sentinel: a row of NaNs (no comparison holds) must still give a legal token id
    float best = -INFINITY; uint32_t idx = 0u;
    auto merge = [](float &v, uint32_t &i, float ov, uint32_t oi) { if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; } };
    if (vec) {
        for (uint32_t j0 = lo + threadIdx.x * 4; j0 < hi; j0 += 4096) {
            float4 v[4];
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) v[q] = j0 + 1024 * q < hi ? *reinterpret_cast<const float4 *>(row + j0 + 1024 * q) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                const uint32_t j = j0 + 1024 * q;
                if (v[q].x > best) { best = v[q].x; idx = j; }          // a thread's indices ascend: the first of equals stays
                if (v[q].y > best) { best = v[q].y; idx = j + 1; }
                if (v[q].z > best) { best = v[q].z; idx = j + 2; }
                if (v[q].w > best) { best = v[q].w; idx = j + 3; }
            }
        }
    } else {
        for (uint32_t j = lo + threadIdx.x; j < hi; j += 256) { const float v = row[j]; if (v > best) { best = v; idx = j; } }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) merge(best, idx, __shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, idx, o));
    if (lane == 0) { bv[warp] = best; bi[warp] = idx; }
    __syncthreads();
    if (warp == 0) {
        best = lane < 8 ? bv[lane] : -INFINITY;
        idx = lane < 8 ? bi[lane] : 0u;
#pragma unroll
        for (int o = 4; o; o >>= 1) merge(best, idx, __shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, idx, o));
    }
    if (parts == 1) {
        if (threadIdx.x == 0) { out[blockIdx.x] = (int32_t)idx; if (out2) out2[blockIdx.x] = (int32_t)idx; }
        return;
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (threadIdx.x == 0) {                                    // to slot `rank` of the cluster's first CTA
        uint32_t rv, ri;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(rv) : "r"((uint32_t)__cvta_generic_to_shared(&cv[rank])));
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(ri) : "r"((uint32_t)__cvta_generic_to_shared(&ci[rank])));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(rv), "f"(best) : "memory");
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(ri), "r"(idx) : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (rank == 0 && warp == 0) {
        best = lane < parts ? cv[lane] : -INFINITY;
        idx = lane < parts ? ci[lane] : 0u;
#pragma unroll
        for (int o = 4; o; o >>= 1) merge(best, idx, __shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, idx, o));
        if (lane == 0) { out[blockIdx.x / parts] = (int32_t)idx; if (out2) out2[blockIdx.x / parts] = (int32_t)idx; }
    }
}

// ---- MoE: router, top-2, gates (one warp per token) ------------------------------------------------------
// logits[e] = sum_k h[m,k] * Wr[e,k] + bias[e] in fp32; the two largest (ties: lower expert id); gates = softmax
// over those two logits.
template <int E>
__device__ __forceinline__ void route_pick(const float (&acc)[E], uint32_t topk, int &i0, int &i1, float &g0, float &g1) {
    i0 = 0;                                            // strict > while visiting ascending ids keeps the lower id on ties
#pragma unroll
    for (int e = 1; e < E; ++e) if (acc[e] > acc[i0]) i0 = e;
    i1 = -1; g0 = 1.0f; g1 = 0.0f;
    if (E == 1 || topk == 1) return;
    i1 = i0 == 0 ? 1 : 0;
#pragma unroll
    for (int e = 0; e < E; ++e) if (e != i0 && acc[e] > acc[i1]) i1 = e;
    const float e1 = expf(acc[i1] - acc[i0]);
    g0 = 1.0f / (1.0f + e1);
    g1 = e1 / (1.0f + e1);
}

template <int E>
__global__ void __launch_bounds__(256) tgp_router_kernel(const bf16 *h, const bf16 *__restrict__ Wr, const float *__restrict__ bias,
                                                     int32_t *idx, float *gate, uint32_t M, uint32_t d, uint32_t topk) {
    pdl_enter();
    const uint32_t m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (m >= M) return;
    float acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    for (uint32_t k = lane * 8; k < d; k += 256) {
        float xf[8];
        unpack8(ld_act(reinterpret_cast<const uint4 *>(h + (size_t)m * d + k)), xf);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            float wf[8];
            unpack8(__ldg(reinterpret_cast<const uint4 *>(Wr + (size_t)e * d + k)), wf);
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[e] = fmaf(xf[i], wf[i], acc[e]);
        }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = warp_sum(acc[e]) + bias[e];
    if (lane == 0) {
        int i0, i1; float g0, g1;
        route_pick<E>(acc, topk, i0, i1, g0, g1);
        idx[2 * m] = i0; idx[2 * m + 1] = i1;
        gate[2 * m] = g0; gate[2 * m + 1] = g1;
    }
}

// Up to ROUTE_SMALL tokens: router and token lists in one launch of a cluster, with the arithmetic of tgp_router_kernel.  It is a chain of
// latencies, so the tokens are spread over up to eight CTAs and a warp computes one logit at a time, up to eight loads of each operand under way; the weights of
// its first one, which no kernel writes, are requested before the previous kernel has finished (8 experts, d=1024, 16 tokens: a warp per token and
// all its experts, eight tokens per CTA 6.3 us, 3.7 us now; 8 experts, d=4096, 32 tokens 15.9, 7.2).  The picks meet in the first CTA, whose warps
// list the tokens of the experts in ascending order.  pos[2 m + s]: the place of
// token m in the list of its s-th expert.  counts_host (may be NULL): mapped host memory that receives the counts too.
constexpr uint32_t ROUTE_SMALL = 64, ROUTE_WARPS = 16;

template <int E>
__global__ void __launch_bounds__(ROUTE_WARPS * 32) tgp_route_small_kernel(const bf16 *h, const bf16 *__restrict__ Wr, const float *__restrict__ bias, int32_t *idx, float *gate, int32_t *rows,
                                                             float *gates, int32_t *counts, int32_t *pos, int32_t *counts_host, uint32_t M, uint32_t stride, uint32_t d, uint32_t topk) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ __align__(8) int32_t si[2 * ROUTE_SMALL];     // the first CTA's: the picks of all tokens
    __shared__ __align__(8) float sg[2 * ROUTE_SMALL];
    __shared__ float logit[ROUTE_SMALL / 8][E];              // of this CTA's tokens
    constexpr int U = 8;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t rank, parts;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(parts));
    if (parts > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    const uint32_t per = (M + parts - 1) / parts, m0 = rank * per, mine = m0 < M ? min(per, M - m0) : 0u;       // this CTA's tokens
    uint4 w[U];
    auto load_w = [&](uint32_t e, uint32_t k0) {
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = k0 + 256 * u < d ? __ldg(reinterpret_cast<const uint4 *>(Wr + (size_t)e * d + k0 + 256 * u)) : make_uint4(0, 0, 0, 0);
    };
    load_w(warp % E, lane * 8);
    const float b0 = bias[warp % E];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (uint32_t q = warp; q < mine * E; q += ROUTE_WARPS) {        // logit q % E of token m0 + q / E
        const uint32_t e = q % E;
        const bf16 *x = h + (size_t)(m0 + q / E) * d;
        float acc = 0.f;
        for (uint32_t k0 = lane * 8; k0 < d; k0 += 256 * U) {
            uint4 xv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) xv[u] = k0 + 256 * u < d ? ld_act(reinterpret_cast<const uint4 *>(x + k0 + 256 * u)) : make_uint4(0, 0, 0, 0);
            if (q != warp || k0 != lane * 8) load_w(e, k0);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float xf[8], wf[8];
                unpack8(xv[u], xf);
                unpack8(w[u], wf);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc = fmaf(xf[i], wf[i], acc);
            }
        }
        acc = warp_sum(acc) + (q == warp ? b0 : bias[e]);
        if (lane == 0) logit[q / E][e] = acc;
    }
    __syncthreads();
    int i0 = 0, i1 = -1; float g0 = 0.f, g1 = 0.f;
    if (threadIdx.x < mine) {
        float acc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = logit[threadIdx.x][e];
        route_pick<E>(acc, topk, i0, i1, g0, g1);
    }
    __syncwarp();
    if (parts > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");         // (the first CTA is known to run)
    if (threadIdx.x < mine) {
        const uint32_t m = m0 + threadIdx.x;
        idx[2 * m] = i0; idx[2 * m + 1] = i1;
        gate[2 * m] = g0; gate[2 * m + 1] = g1;
        uint32_t ri, rg;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(ri) : "r"((uint32_t)__cvta_generic_to_shared(&si[2 * m])));
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(rg) : "r"((uint32_t)__cvta_generic_to_shared(&sg[2 * m])));
        asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(ri), "r"(i0), "r"(i1) : "memory");
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(rg), "f"(g0), "f"(g1) : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (rank) return;
    for (uint32_t e = warp; e < (uint32_t)E; e += ROUTE_WARPS) {
        uint32_t base = 0;
        for (uint32_t m0 = 0; m0 < M; m0 += 32) {
            const uint32_t t = m0 + lane;
            int slot = -1;
            if (t < M) slot = si[2 * t] == (int)e ? 0 : topk > 1 && si[2 * t + 1] == (int)e ? 1 : -1;
            const uint32_t bal = __ballot_sync(0xffffffffu, slot >= 0), at = base + __popc(bal & ((1u << lane) - 1));
            if (slot >= 0) { rows[(size_t)e * stride + at] = (int32_t)t; gates[(size_t)e * stride + at] = sg[2 * t + slot]; pos[2 * t + slot] = (int32_t)at; }
            base += __popc(bal);
        }
        if (lane == 0) { counts[e] = (int32_t)base; if (counts_host) *(volatile int32_t *)(counts_host + e) = (int32_t)base; }
    }
}

// Tokens of expert e in ascending token order: rows[e*stride + pos] = m, gates[e*stride + pos] = that token's gate for e.
// One block per expert walks the tokens in chunks; positions come from a block-wide exclusive scan, so the
// grouping is deterministic.  topk = number of routed slots per token (1 or 2).
__global__ void __launch_bounds__(1024) tgp_route_fill_kernel(const int32_t *__restrict__ idx, const float *__restrict__ gate, int32_t *__restrict__ rows,
                                                          float *__restrict__ gates, int32_t *__restrict__ counts, uint32_t M, uint32_t stride, uint32_t topk) {
    __shared__ uint32_t warp_tot[32];
    __shared__ uint32_t base;
    const uint32_t e = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    for (uint32_t m0 = 0; m0 < M; m0 += blockDim.x) {
        const uint32_t m = m0 + threadIdx.x;
        int slot = -1;
        if (m < M) {
            if (idx[2 * m] == (int)e) slot = 0;
            else if (topk > 1 && idx[2 * m + 1] == (int)e) slot = 1;
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, slot >= 0);
        const uint32_t before = __popc(bal & ((1u << lane) - 1));
        if (lane == 0) warp_tot[warp] = __popc(bal);
        __syncthreads();
        uint32_t woff = 0;
        for (uint32_t w = 0; w < warp; ++w) woff += warp_tot[w];
        const uint32_t b0 = base;
        if (slot >= 0) { rows[(size_t)e * stride + b0 + woff + before] = (int32_t)m; gates[(size_t)e * stride + b0 + woff + before] = gate[2 * m + slot]; }
        __syncthreads();
        if (threadIdx.x == 0) { uint32_t t = 0; for (uint32_t w = 0; w < (blockDim.x >> 5); ++w) t += warp_tot[w]; base = b0 + t; }
        __syncthreads();
    }
    if (threadIdx.x == 0) counts[e] = (int32_t)base;
}

__global__ void tgp_gather_rows_kernel(const bf16 *__restrict__ src, const int32_t *__restrict__ rows, bf16 *__restrict__ dst, uint32_t d) {
    const uint4 *s = reinterpret_cast<const uint4 *>(src + (size_t)rows[blockIdx.x] * d);
    uint4 *o = reinterpret_cast<uint4 *>(dst + (size_t)blockIdx.x * d);
    for (uint32_t i = threadIdx.x; i < d / 8; i += blockDim.x) o[i] = s[i];
}

// x[rows[i], :] += gates[i] * y[i, :]   (each token appears at most once per expert: no write conflicts)
__global__ void tgp_scatter_add_kernel(float *__restrict__ x, const float *__restrict__ y, const int32_t *__restrict__ rows, const float *__restrict__ gates, uint32_t d) {
    const float g = gates[blockIdx.x];
    float4 *o = reinterpret_cast<float4 *>(x + (size_t)rows[blockIdx.x] * d);
    const float4 *s = reinterpret_cast<const float4 *>(y + (size_t)blockIdx.x * d);
    for (uint32_t i = threadIdx.x; i < d / 4; i += blockDim.x) {
        float4 a = o[i];
        const float4 b = s[i];
        a.x += g * b.x; a.y += g * b.y; a.z += g * b.z; a.w += g * b.w;
        o[i] = a;
    }
}

// ============================ launchers (internal) ===================================================
int tgpk_router(const void *h, const void *Wr, const float *bias, int32_t *idx, float *gate, int32_t *rows, float *gates, int32_t *counts, int32_t *pos,
                int32_t *counts_host, uint32_t M, uint32_t stride, uint32_t d, uint32_t E, uint32_t topk, cudaStream_t st) {
    if (!M) return TGP_OK;
    if (d % 8 || topk < 1 || topk > 2) return TGP_E_INVAL;
    const bool small = M <= ROUTE_SMALL;
    if (counts_host && !small) return TGP_E_INVAL;
    const uint32_t blocks = (M + 7) / 8;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(M <= 2 ? M : M <= 4 ? 4 : 8); cfg.blockDim = dim3(ROUTE_WARPS * 32); cfg.stream = st;        // one cluster
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = small_overlap();
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cfg.gridDim.x; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
#define TGP_ROUTE(E_) do { \
        if (small) cudaLaunchKernelEx(&cfg, tgp_route_small_kernel<E_>, (const bf16 *)h, (const bf16 *)Wr, bias, idx, gate, rows, gates, counts, pos, counts_host, M, stride, d, topk); \
        else launch_pdl(tgp_router_kernel<E_>, dim3(blocks), dim3(256), 0, st, (const bf16 *)h, (const bf16 *)Wr, bias, idx, gate, M, d, topk); } while (0)
    switch (E) {
    case 1: TGP_ROUTE(1); break;
    case 2: TGP_ROUTE(2); break;
    case 4: TGP_ROUTE(4); break;
    case 8: TGP_ROUTE(8); break;
    case 16: TGP_ROUTE(16); break;
    default: return TGP_E_INVAL;
    }
#undef TGP_ROUTE
    if (!small) tgp_route_fill_kernel<<<E, 1024, 0, st>>>(idx, gate, rows, gates, counts, M, stride, topk);
    LAUNCH_CHECK(small ? 1 : 2);
    return TGP_OK;
}

int tgpk_gather_rows(const void *src, const int32_t *rows, void *dst, uint32_t m, uint32_t d, cudaStream_t st) {
    if (!m) return TGP_OK;
    tgp_gather_rows_kernel<<<m, 128, 0, st>>>((const bf16 *)src, rows, (bf16 *)dst, d);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

int tgpk_scatter_add(float *x, const float *y, const int32_t *rows, const float *gates, uint32_t m, uint32_t d, cudaStream_t st) {
    if (!m) return TGP_OK;
    tgp_scatter_add_kernel<<<m, 256, 0, st>>>(x, y, rows, gates, d);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

int tgpk_embed(const void *table, const int32_t *tok, float *x, uint32_t M, uint32_t d, uint32_t V, cudaStream_t st) {
    if (!M) return TGP_OK;
    if (d % 8 || !V) return TGP_E_INVAL;
    launch_pdl(tgp_embed_kernel, dim3(M), dim3(128), 0, st, (const bf16 *)table, tok, x, d, V);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

int tgpk_rmsnorm(const float *x, uint32_t ldx, const void *g, void *h, uint32_t M, uint32_t d, float eps, cudaStream_t st) {
    if (!M) return TGP_OK;
    if (d % 4 || ldx % 4) return TGP_E_INVAL;
#define TGP_RMSNORM(NV_) launch_pdl(tgp_rmsnorm_kernel<NV_>, dim3(M), dim3(256), 0, st, x, ldx, (const bf16 *)g, (bf16 *)h, d, eps)
    // (many long rows: read twice by more CTAs per SM - 8192 rows of 8192: 63.0 us, 65.5 us from registers)
    if (((reinterpret_cast<uintptr_t>(g) | reinterpret_cast<uintptr_t>(h)) & 7u) || (d > 4096 && M > 1024)) TGP_RMSNORM(0);
    else if (d <= 1024) TGP_RMSNORM(1); else if (d <= 2048) TGP_RMSNORM(2); else if (d <= 4096) TGP_RMSNORM(4); else if (d <= 8192) TGP_RMSNORM(8); else TGP_RMSNORM(0);
#undef TGP_RMSNORM
    LAUNCH_CHECK(1);
    return TGP_OK;
}

static int g_skinny_impl = 0;    // 0: tensor-core skinny kernels for 3 <= M <= 16; 1: CUDA-core GEMV (an on-device cross-check)
static int g_gemm_impl = 0;      // 0: tensor cores for M > 16; 1: CUDA-core tiles (kept as an on-device cross-check)
static int g_gemv_splitk = 1;    // small-n blocks at M <= 2: CTA per RB rows with K split over its warps (0: one warp per row)
static int g_gemm_group = 1;     // products over the same activations: one launch where the parts allow it (0: always one launch each)
bool tgpk_gemm_grouping() { return g_gemm_group != 0; }
static int g_gemv_balance = 1;   // grouped skinny launches: rows per group chosen so that every persistent CTA gets the same number of groups
static int g_gemv_pdl = 1;       // consecutive weight-streaming launches may overlap (programmatic dependent launch)
bool tgpk_launch_overlap() { return g_gemv_pdl != 0 && !tgpk_whole_edge; }

// Launches a kernel that streams weights through registers.  Its loads under way take up L1, 64 KB of them and more per SM, and a kernel without a
// preference of its own runs on the split of L1 and shared memory that the SM has: next to nothing is left of L1 behind an attention or tcgen05
// kernel that overlaps it (n=32000, K=4096 at 3 rows behind the products of a prefill: 68 us, 42 with half of it kept for
// L1; a decode step of 8 users at d=4096 249 us, 233; a quarter or all of it for L1 is the same).
template <auto KERNEL, typename... Args>
static void launch_weights(const cudaLaunchConfig_t &cfg, Args... args) {
    static std::atomic<uint64_t> hinted{0};                  // a bit per device: the attribute is a device's own
    int dev = 0;
    const uint64_t bit = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 ? 1ull << dev : 0;
    if (bit & ~hinted.load(std::memory_order_relaxed)) {
        if (cudaFuncSetAttribute(KERNEL, cudaFuncAttributePreferredSharedMemoryCarveout, 50) != cudaSuccess) cudaGetLastError();        // only a hint: it fails no product
        hinted.fetch_or(bit, std::memory_order_relaxed);
    }
    cudaLaunchKernelEx(&cfg, KERNEL, args...);
}

// CTAs of tgp_wstream_kernel that the GPU holds at a time.
template <int MT, int R, int U>
static uint32_t gemv_slots() {
    static int blocks_per_sm = 0;
    if (!blocks_per_sm && (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, tgp_wstream_kernel<MT, R, U>, 256, 0) != cudaSuccess || blocks_per_sm < 1)) blocks_per_sm = 1;
    return (uint32_t)(device_sms() * blocks_per_sm);
}

template <int MT, int R, int U>
static void launch_gemv(const bf16 *A, const bf16 *W, float *C, uint32_t Mrows, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int acc, cudaStream_t st) {
    const uint32_t need = (n + R * 8 - 1) / (R * 8), full = gemv_slots<MT, R, U>();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(need < full ? need : full);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    launch_weights<tgp_wstream_kernel<MT, R, U>>(cfg, A, W, C, Mrows, n, K, ldc, col0, acc);
    tgpk_last_gemm_kernel = "tgp_wstream_kernel";
}

// Same product for blocks of a short K with two to eight 16-row groups per SM: one CTA owns 16 rows of W and its NW warps split K
// (interleaved chunks of 32*U), so n/16 CTAs of NW warps fill the machine where n/16 warps would not.  The partial
// tiles meet in shared memory and are summed in warp order: deterministic.
// (Blocks of fewer rows or a longer K take tgp_wstream_mma_group_kernel.)
template <int NB, int U, int NW>
__global__ void __launch_bounds__(NW * 32) tgp_wstream_mma_splitk_kernel(const bf16 *A, const bf16 *__restrict__ W, float *__restrict__ C,
                                                              uint32_t Mrows, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate) {
    __shared__ float part[NW][NB * 4][32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, c = lane & 3;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool synced = false;
    for (uint32_t row0 = blockIdx.x * 16; row0 < n; row0 += gridDim.x * 16) {
        const uint32_t rlast = min(row0 + 16, n) - 1;
        const bf16 *wlo = W + (size_t)min(row0 + g, rlast) * K + c * 8;
        const bf16 *whi = W + (size_t)min(row0 + g + 8, rlast) * K + c * 8;
        float acc[2][NB][4];                               // a load step's two MMAs have sums of their own: half as many additions in a row
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[0][b][i] = acc[1][b][i] = 0.f;
        for (uint32_t k0 = warp * 32 * U; k0 < K; k0 += NW * 32 * U) {
            uint4 lo[U], hi[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool in = k0 + 32 * u < K;
                lo[u] = in ? __ldcs(reinterpret_cast<const uint4 *>(wlo + k0 + 32 * u)) : make_uint4(0, 0, 0, 0);
                hi[u] = in ? __ldcs(reinterpret_cast<const uint4 *>(whi + k0 + 32 * u)) : make_uint4(0, 0, 0, 0);
            }
            if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t k = k0 + 32 * u;
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const uint32_t m = b * 8 + g;
                    const uint4 xv = (k < K && m < Mrows) ? ld_act(reinterpret_cast<const uint4 *>(A + (size_t)m * K + k + c * 8)) : make_uint4(0, 0, 0, 0);
                    mma_bf16_16816(acc[0][b], lo[u].x, hi[u].x, lo[u].y, hi[u].y, xv.x, xv.y);
                    mma_bf16_16816(acc[1][b], lo[u].z, hi[u].z, lo[u].w, hi[u].w, xv.z, xv.w);
                }
            }
        }
        if (!synced) { asm volatile("griddepcontrol.wait;" ::: "memory"); synced = true; }
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int i = 0; i < 4; ++i) part[warp][b * 4 + i][lane] = acc[0][b][i] + acc[1][b][i];
        __syncthreads();
        for (uint32_t v = threadIdx.x; v < NB * 4 * 32; v += NW * 32) {
            const uint32_t slot = v >> 5, ln = v & 31, b = slot >> 2, i = slot & 3;
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) sum += part[w][slot][ln];
            const uint32_t m = b * 8 + 2 * (ln & 3) + (i & 1), row = row0 + (ln >> 2) + 8 * (i >> 1);
            if (m < Mrows && row < n) {
                float *p = C + (size_t)m * ldc + col0 + row;
                if (accumulate) atomicAdd(p, sum);               // one add per element by one thread, not waited for
                else *p = sum;
            }
        }
        __syncthreads();
    }
}

// The product for 3 - 16 activation rows on blocks of few rows or of a long K (pick_skinny), one block or a list of blocks that read the same
// activations (the pieces of one matrix; the q, k and v projections): one persistent CTA per SM walks the row groups
// as one list, RG consecutive groups at a time, whose MMAs share each activation fragment - every CTA reads its K
// slices of all activation rows from L2, so at 16 rows per CTA that traffic equals the weights'; RG row groups divide
// it by RG.  K is split over the CTA's NW warps in interleaved chunks of 32*U columns and the partial tiles are summed
// in warp order.  A group's arithmetic (which warp adds which k, in which order) depends on the width of these chunks, NW and K alone -
// not on RG, the rows per group or the list: a block gives the same bits alone or in any list.
// CS: load steps per chunk, U unless a warp's U steps under way are to cover several of its chunks.
template <int NB, int U, int NW, int RG, int CS = U>
__global__ void __launch_bounds__(NW * 32) tgp_wstream_mma_group_kernel(const bf16 *A, const GemvParts p, uint32_t Mrows, uint32_t groups_total,
                                                              uint32_t K, int accumulate, uint32_t rpc, int acts_early) {
    constexpr int G = RG, SK = U / (2 * G);              // a register set holds SK load steps of G groups: two sets are as many loads as U steps of one group
    static_assert(U % (2 * G) == 0 && SK >= 1, "row groups per CTA must divide half the load steps");
    static_assert(U % CS == 0 && CS % SK == 0, "a register set lies in one chunk");
    // the warps' partial tiles: static where they fit the 48 KB a kernel may declare, else the launch's dynamic shared memory
    constexpr bool PART_DYNAMIC = NW * G * NB * 4 * 32 * 4 > 48 * 1024;
    __shared__ float part_static[PART_DYNAMIC ? 1 : NW * G * NB * 4 * 32];
    extern __shared__ float part_dynamic[];
    auto part = [&](uint32_t w, uint32_t slot, uint32_t ln) -> float & {
        const uint32_t at = (w * (G * NB * 4) + slot) * 32 + ln;
        if constexpr (PART_DYNAMIC) return part_dynamic[at]; else return part_static[at];
    };
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, c = lane & 3;
    uint32_t grp0 = blockIdx.x * G;
    if (grp0 >= groups_total) return;
    const bf16 *wlo[G], *whi[G];
    uint4 lo[2][G][SK], hi[2][G][SK];                     // two register sets of SK load steps of every group
    // the activation fragments of a set are loaded with its weights (they come from L2 more often than from L1 -
    // a long K does not fit there - and would otherwise be waited for inside the MMA sequence)
    uint4 xs[2][SK][NB];
    float acc[G][NB][4];
    // which block a group belongs to: looked up here for the weights and again after the K loop for the output, so
    // that the output's pointer and stride do not occupy registers while the loads are in flight
    auto locate = [&](uint32_t first) {
#pragma unroll
        for (int r = 0; r < G; ++r) {
            const uint32_t grp = min(first + r, groups_total - 1);         // a group past the end re-reads the last one, never stored
            const bf16 *W = p.W[0];
            uint32_t n = p.n[0], local = grp;
            {
                uint32_t start = p.groups[0];
#pragma unroll
                for (int s = 1; s < (int)TGP_GEMM_GROUP_MAX; ++s)
                    if (s < (int)p.count) {
                        if (grp >= start) { W = p.W[s]; n = p.n[s]; local = grp - start; }
                        start += p.groups[s];
                    }
            }
            // rpc <= 16 rows per group, chosen by the launcher so that the persistent CTAs all get the same number of
            // groups; the tile's rows beyond rpc re-read the group's last row and are not stored (a row's sum does not
            // depend on its place in the tile)
            const uint32_t rlast = min(local * rpc + rpc, n) - 1;
            wlo[r] = W + (size_t)min(local * rpc + g, rlast) * K + c * 8;
            whi[r] = W + (size_t)min(local * rpc + g + 8, rlast) * K + c * 8;
        }
    };
    auto issue = [&](auto set, uint32_t kb) {              // SK load steps of every group, from column kb on, into one register set
        constexpr int S = decltype(set)::value;
#pragma unroll
        for (int u = 0; u < SK; ++u) {
            const uint32_t k = kb + 32 * u;
#pragma unroll
            for (int r = 0; r < G; ++r) {
                lo[S][r][u] = k < K ? __ldcs(reinterpret_cast<const uint4 *>(wlo[r] + k)) : make_uint4(0, 0, 0, 0);
                hi[S][r][u] = k < K ? __ldcs(reinterpret_cast<const uint4 *>(whi[r] + k)) : make_uint4(0, 0, 0, 0);
            }
        }
    };
    auto issue_act = [&](auto set, uint32_t kb) {          // the activation fragments that go with a set; only after griddepcontrol.wait
        constexpr int S = decltype(set)::value;
#pragma unroll
        for (int u = 0; u < SK; ++u) {
            const uint32_t k = kb + 32 * u;
#pragma unroll
            for (int b = 0; b < NB; ++b)
                xs[S][u][b] = (k < K && b * 8 + g < Mrows) ? ld_act(reinterpret_cast<const uint4 *>(A + (size_t)(b * 8 + g) * K + k + c * 8)) : make_uint4(0, 0, 0, 0);
        }
    };
    auto consume = [&](auto set) {
        constexpr int S = decltype(set)::value;
#pragma unroll
        for (int u = 0; u < SK; ++u) {
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const uint4 xv = xs[S][u][b];
#pragma unroll
                for (int r = 0; r < G; ++r) {
                    mma_bf16_16816(acc[r][b], lo[S][r][u].x, hi[S][r][u].x, lo[S][r][u].y, hi[S][r][u].y, xv.x, xv.y);
                    mma_bf16_16816(acc[r][b], lo[S][r][u].z, hi[S][r][u].z, lo[S][r][u].w, hi[S][r][u].w, xv.z, xv.w);
                }
            }
        }
    };
    auto clear = [&]() {
#pragma unroll
        for (int r = 0; r < G; ++r)
#pragma unroll
            for (int b = 0; b < NB; ++b) { acc[r][b][0] = acc[r][b][1] = acc[r][b][2] = acc[r][b][3] = 0.f; }
    };
    const std::integral_constant<int, 0> set0;
    const std::integral_constant<int, 1> set1;
    // One stream of loads over all the groups this CTA takes.  A warp's chunk of 32 * U columns is G pairs of load steps;
    // the two register sets alternate, a set is loaded again as soon as its MMAs are issued, so a warp always has one
    // or two sets in flight - also across the end of a group: the next group's first pair is on its way while the CTA
    // meets in shared memory to sum and store the group it has finished, and the memory pipe never drains.  Per group
    // the k order of a warp's additions is that of its chunks, ascending: the bits do not depend on the pairing.  A warp
    // whose first chunk lies beyond K runs one pair of zeros (the sums do not change).
    uint32_t grp = grp0, k0 = warp * 32 * CS, pr = 0;       // the pair that is loaded next: group, first chunk, pair within its chunks
    constexpr uint32_t SET1 = CS == SK ? NW * 32 * CS : 32 * SK;       // from a pair's first set to its second
    auto column = [&]() -> uint32_t {                       // first column of that pair
        if constexpr (CS == U) return k0 + pr * 64 * SK;
        else return k0 + 2 * pr * SK / CS * (NW * 32 * CS) + 2 * pr * SK % CS * 32;
    };
    auto advance = [&]() -> bool {                         // moves on by one pair; true: the pair just passed ended its group
        if (++pr == (uint32_t)G) { pr = 0; k0 += NW * 32 * U; }
        if (CS == U ? k0 < K : column() < K) return false;
        grp += gridDim.x * G;
        k0 = warp * 32 * CS;
        pr = 0;
        if (grp < groups_total) locate(grp);
        return true;
    };
    locate(grp);
    const uint32_t kb_first = column();
    issue(set0, kb_first);
    issue(set1, kb_first + SET1);
    bool cur_last = advance();
    // Weights are never written by a kernel, so they are requested before the previous launch of the stream has finished.
    // The activations are read after it has - unless the launcher knows that they are older than that launch (it read the
    // same activations): then they are requested with the weights.  The next launch is released only here, after the wait:
    // when it starts, everything before this launch is complete, which is what lets it read its activations early in turn.
    if (acts_early) { issue_act(set0, kb_first); issue_act(set1, kb_first + SET1); }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!acts_early) { issue_act(set0, kb_first); issue_act(set1, kb_first + SET1); }
    clear();
    for (;;) {
        const bool have_next = grp < groups_total;
        const uint32_t kb_next = column();
        consume(set0);
        if (have_next) { issue(set0, kb_next); issue_act(set0, kb_next); }
        consume(set1);
        if (have_next) { issue(set1, kb_next + SET1); issue_act(set1, kb_next + SET1); }
        const bool next_last = have_next ? advance() : false;
        if (!cur_last) { cur_last = next_last; continue; }
        cur_last = next_last;
        // this warp has finished the group(s) at grp0
#pragma unroll
        for (int r = 0; r < G; ++r)
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int i = 0; i < 4; ++i) part(warp, (r * NB + b) * 4 + i, lane) = acc[r][b][i];
        __syncthreads();
        for (uint32_t v = threadIdx.x; v < G * NB * 4 * 32; v += NW * 32) {
            const uint32_t slot = v >> 5, ln = v & 31, r = slot / (NB * 4), b = (slot >> 2) % NB, i = slot & 3;
            const uint32_t gi = grp0 + r;
            if (gi >= groups_total) continue;
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) sum += part(w, slot, ln);
            float *C = p.C[0];
            uint32_t ldc = p.ldc[0], n = p.n[0], row0 = gi * rpc;
            {
                uint32_t start = p.groups[0];
#pragma unroll
                for (int s = 1; s < (int)TGP_GEMM_GROUP_MAX; ++s)
                    if (s < (int)p.count) {
                        if (gi >= start) { C = p.C[s]; ldc = p.ldc[s]; n = p.n[s]; row0 = (gi - start) * rpc; }
                        start += p.groups[s];
                    }
            }
            const uint32_t m = b * 8 + 2 * (ln & 3) + (i & 1), row = row0 + (ln >> 2) + 8 * (i >> 1);
            if (m < Mrows && row < min(row0 + rpc, n)) {
                float *out = C + (size_t)m * ldc + row;
                if (accumulate) atomicAdd(out, sum);             // one add per element by one thread, not waited for
                else *out = sum;
            }
        }
        grp0 += gridDim.x * G;
        if (grp0 >= groups_total) break;
        __syncthreads();
        clear();
    }
}

// Which skinny kernel serves a block of n rows at M activation rows: NB groups of 8 activation rows (M <= 16), U load steps in
// flight, and for blocks too small to give every SM eight 16-row warps the split-K kernel with NW warps per CTA over
// 16 rows.  The choice depends on the block alone, so a block computes the same bits alone or as part of a group.
struct SkinnyPick { int nb, u, nw; bool split, persistent; };

// 9 - 16 activation rows on a block of at least this many weight rows (64 tiles of 128): the tcgen05 kernel is ahead of the
// mma.sync ones (M=16, from the end of the norm before: two blocks of 28672 rows, K=8192 144 us against 160; two of 8192 rows, K=2048 14.8 / 15.8;
// n=32000, K=4096 43.2 / 48.3; below, n=4096, K=4096 about 11 against 9.7).  From 17 rows on it is ahead on blocks of any size (M=32:
// n=6144 in three blocks, K=4096 14.7 us against 18.4 us; n=4096, K=14336 24 us against 35 us).
constexpr uint32_t TILES_WIN_ROWS = 8065;

// a product that the tcgen05 kernels serve (tgpk_gemm_tc)
static bool takes_tiles(uint32_t M, uint32_t n, uint32_t K) {
    if (g_gemm_impl || K % 8) return false;
    if (M > 16) return true;
    // (K not a multiple of 32: the CUDA cores' sums are closer to 64 bits, 6.9e-8 against 1.24e-7 at n=12000, K=1000)
    if (M < 9 || n < TILES_WIN_ROWS || K % 32 || g_skinny_impl || tgpk_gemm_tc_forced()) return false;
    // A short K on fewer tiles than SMs is over before the ring is under way (M=9, K=1024: n=8192 4.6 us in tgp_wstream_mma_splitk_kernel against
    // 7.0, n=12288 5.5 against 8.1; K=1536, n=16384 12.8 against 10.7; n=32000, K=1024 17.1 against 9.4).  From K=1536 on lists
    // decide: two blocks of 8192 rows as above, though one alone takes 9.9 - 11.0 us against 11.2 at K=2048, and one of 12288 rows (96
    // tiles) 10.9 - 11.9 against 14.3.
    return K >= 1536 || (n + 127) / 128 > (uint32_t)device_sms();
}

static SkinnyPick pick_skinny(uint32_t M, uint32_t n, uint32_t K) {
    const uint32_t sms = (uint32_t)device_sms(), groups16 = (n + 15) / 16;
    SkinnyPick k;
    k.nb = M <= 8 ? 1 : 2;
    k.split = n < 16u * 8u * sms;                         // too few 16-row groups to give every SM eight warps
    // One persistent CTA per SM walks the row groups of the block, or of a list of such blocks (tgp_wstream_mma_group_kernel).
    // It is bound by HBM: its loads never drain between row groups (n=14336, K=4096: 18.5 us = 6.36 TB/s at M=8;
    // one CTA per row group took 22.7 us.  n=32000, K=4096, M=8: 40.1 us against 55.3 us of one warp per 16
    // rows).  Its warps share K in chunks of 4096 columns (2048 above 8 rows), so a short K leaves most of them without work: with two or more
    // row groups per SM it is taken from K=3072 on at M <= 8 (K=2048: ahead from five row groups per SM on - n=32000: 23.1 us
    // against 29.5 us, n=6144: 6.3 us against 5.6 us) and from K=4096 on at M <= 16 (K=2048, M=16, n=12288: 15.1 us against 11.5 us).
    // One choice per class of M for all of them, so that the pieces of a matrix share a launch whatever the rows of its
    // last piece:
    //   M <= 8   16 warps, 8 load steps per warp and chunk
    //   M <= 16  16 warps, 4 load steps: a chunk of 2048 columns, so that a K of 1024 still occupies half of the warps, and registers for the
    //            activation fragments of both sets (M=16, from the end of the norm before: n=1024, K=1024 8.5 us with 8 warps of 16 steps,
    //            2.0 us; n=2048, K=2048 9.9 / 3.8; n=2048, K=8192 20.5 / 10.1; n=4096, K=14336 31.4 / 26.8.  Twice as many CTAs
    //            of 8 warps are no faster: 2.1, 3.8.  Half the additions in a row, too: 1.4e-7 from 64 bits at K=2048, 4.8e-7 before)
    const bool few = k.split && groups16 < 2u * sms;
    const bool deep = k.nb == 1 ? K >= 3072 || (K >= 2048 && groups16 >= 5u * sms) : K >= 4096;
    k.persistent = few || deep;
    if (k.persistent) k.split = true;
    if (k.persistent) {
        k.nw = 16;
        k.u = k.nb == 1 ? 8 : 4;
    } else {
        k.nw = 8;
        k.u = 4;
    }
    return k;
}

template <int NB, int U>
static void launch_skinny(const bf16 *A, GemvParts p, const SkinnyPick &k, uint32_t Mrows, uint32_t K, int acc, cudaStream_t st) {
    static int blocks_per_sm = 0, blocks_per_sm_split = 0;
    constexpr bool STREAMS = U <= 4;                         // the load depths of the kernels that are not persistent
    if constexpr (STREAMS) {
        if (!blocks_per_sm && (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, tgp_wstream_mma_kernel<NB, U>, 256, 0) != cudaSuccess || blocks_per_sm < 1)) blocks_per_sm = 1;
        if (!blocks_per_sm_split && (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm_split, tgp_wstream_mma_splitk_kernel<NB, U, 8>, 256, 0) != cudaSuccess || blocks_per_sm_split < 1))
            blocks_per_sm_split = 1;
    }
    const uint32_t sms = (uint32_t)device_sms();
    constexpr uint32_t tile = 16;                           // rows of an MMA
    uint32_t need = 0, rpc = tile;
    if (k.split) for (uint32_t s = 0; s < p.count; ++s) { p.groups[s] = (p.n[s] + tile - 1) / tile; need += p.groups[s]; }
    else need = (p.n[0] + 16 * 8 - 1) / (16 * 8);           // whole blocks of many rows are launched alone
    const bool persistent = k.persistent;                   // one block or several: the kernel that walks a list of row groups
    // (one CTA per SM of the persistent kernels: up to 8 activation rows they take the whole register file, above three quarters of it)
    const uint32_t full = persistent ? sms : sms * (uint32_t)(k.split ? blocks_per_sm_split : blocks_per_sm);
    uint32_t per_cta = 1;
    if (persistent) {
        // The grid is one persistent CTA per SM, each walking its share of the row groups, G groups at a time whose MMAs share
        // each activation fragment (every CTA reads its K slices of all activation rows per round, so at one group per round
        // that traffic equals the weights').  Rows per group r <= the tile's rows: fewer rows make more groups, so that a
        // block of few rows reaches every SM and no CTA waits for the others' last round (4096 rows: 256 groups of 16 leave
        // 40 SMs one round short, 293 of 14 do not) - but the rows a tile lacks still occupy its load slots (their lanes
        // re-read the group's last row; fewer than 9 rows per group measured no faster for blocks of few rows).  G and r are the
        // pair with the least estimated time of the busiest CTA: rounds x (G x (r + tile rows) / 2 + 4 NB), in rows read; of equal
        // estimates above 8 activation rows the one of fewer groups and more rows (5120 rows, K=4096 as three rounds of 12 rows 13.2 us at M=9,
        // 14.3 at M=16, as two of 2 x 9 rows 14.3 and 15.5, from the end of the norm before).
        const uint32_t gmax = 2;
        uint32_t best = 0xffffffffu, best_r = tile;
        for (uint32_t G = gmax; G >= 1; G >>= 1)
            for (uint32_t r = g_gemv_balance ? tile / 2 + 1 : tile; r <= tile; ++r) {
                uint32_t groups = 0;
                for (uint32_t s = 0; s < p.count; ++s) groups += (p.n[s] + r - 1) / r;
                const uint32_t ctas = (groups + G - 1) / G, rounds = (ctas + full - 1) / full;
                const uint32_t cost = rounds * (G * (r + tile) + 8 * NB);           // twice the estimate
                if (cost < best || (cost == best && NB == 2)) { best = cost; best_r = r; per_cta = G; }
            }
        rpc = best_r;
        need = 0;
        for (uint32_t s = 0; s < p.count; ++s) { p.groups[s] = (p.n[s] + rpc - 1) / rpc; need += p.groups[s]; }
        need = (need + per_cta - 1) / per_cta;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(need < full ? need : full);
    cfg.blockDim = dim3(k.split ? k.nw * 32 : 256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    uint32_t total = 0;
    for (uint32_t s = 0; k.split && s < p.count; ++s) total += p.groups[s];
    // the previous launch of this thread was a product of this family over the same activations on the same stream, and the
    // caller vouches that nothing else was enqueued there in between: the activations are older than that launch
    const int early = persistent && tgpk_chain_ok && g_gemv_pdl && g_chain.A == (const void *)A && g_chain.st == st && g_chain.launches_before + 1 == tgpk_launches;
    if (persistent) { g_chain.A = A; g_chain.st = st; g_chain.launches_before = tgpk_launches; }
    else g_chain.A = nullptr;
    tgpk_last_gemm_kernel = !k.split ? "tgp_wstream_mma_kernel" : persistent ? "tgp_wstream_mma_group_kernel" : "tgp_wstream_mma_splitk_kernel";
    if (persistent) {
        if constexpr (NB == 2 || U == 8) {                  // (their partial tiles, 32 KB at most, are static)
            if (per_cta == 2) launch_weights<tgp_wstream_mma_group_kernel<NB, U, 16, 2>>(cfg, A, p, Mrows, total, K, acc, rpc, early);
            else launch_weights<tgp_wstream_mma_group_kernel<NB, U, 16, 1>>(cfg, A, p, Mrows, total, K, acc, rpc, early);
        }
    } else if constexpr (STREAMS) {
        if (!k.split) launch_weights<tgp_wstream_mma_kernel<NB, U>>(cfg, A, p.W[0], p.C[0], Mrows, p.n[0], K, p.ldc[0], 0u, acc);
        else launch_weights<tgp_wstream_mma_splitk_kernel<NB, U, 8>>(cfg, A, p.W[0], p.C[0], Mrows, p.n[0], K, p.ldc[0], 0u, acc);
    }
}

static void launch_skinny_pick(const bf16 *A, const GemvParts &p, const SkinnyPick &k, uint32_t Mrows, uint32_t K, int acc, cudaStream_t st) {
    if (k.nb == 1) { if (k.u == 8) launch_skinny<1, 8>(A, p, k, Mrows, K, acc, st); else launch_skinny<1, 4>(A, p, k, Mrows, K, acc, st); }
    else launch_skinny<2, 4>(A, p, k, Mrows, K, acc, st);
}

template <int MT, int RB, int U>
static void launch_gemv_splitk(const bf16 *A, const bf16 *W, float *C, uint32_t Mrows, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int acc, cudaStream_t st) {
    static int blocks_per_sm = 0;
    if (!blocks_per_sm) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, tgp_wstream_splitk_kernel<MT, RB, U>, 256, 0) != cudaSuccess || blocks_per_sm < 1) blocks_per_sm = 1;
    }
    uint32_t need = (n + RB - 1) / RB, full = (uint32_t)(device_sms() * blocks_per_sm);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(need < full ? need : full);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    launch_weights<tgp_wstream_splitk_kernel<MT, RB, U>>(cfg, A, W, C, Mrows, n, K, ldc, col0, acc);
    tgpk_last_gemm_kernel = "tgp_wstream_splitk_kernel";
}

// From this many rows on a block of one or two activation rows gives every SM two rows for each of its warps.
constexpr uint32_t GEMV_MANY_ROWS = 2 * 148 * 16;

// One activation row on a block of many rows whose K is two to four times the 2048 columns of eight load steps: a row per warp with all eight under
// way is ahead of two rows with four each (n=14336, K=4096 18.3 us against 19.7, n=32000, K=8192 76 / 81; with K=1024 25 / 16, K=28672 78 / 72).
static bool one_row_deep(uint32_t M, uint32_t K) { return M == 1 && K % 2048 == 0 && K >= 4096 && K <= 8192; }

// ... alone, where its last wave of CTAs of eight rows is no emptier than that of CTAs of sixteen (three and four CTAs per SM: n=8192, K=6144 is 2.3 waves of
// eight and 0.9 of sixteen rows, 19.1 us and 17.8; n=10240, K=4096 2.9 and 1.1, 15.0 and 17.3); in a list the waves of all blocks are one ramp.
static bool one_row_fuller(uint32_t n) {
    auto fill = [n](uint32_t wave) { return (float)n / (float)((n + wave - 1) / wave * wave); };
    return fill(8 * gemv_slots<1, 1, 8>()) >= fill(16 * gemv_slots<1, 2, 4>());
}

// Two activation rows on a block of many rows: listed (a row per warp, eight load steps under way) where the block alone leaves the last wave of its CTAs - three of
// sixteen rows per SM - more than a quarter empty (us in one list / one behind the other: 2 x 4736, K=2048 11.4 / 11.9; 2 x 7168 14.4 / 17.9, 2 x 8192 17.0 / 19.8;
// K=8192, 3 x 8192 75 / 90; but 2 x 6144, three quarters to all of one wave, 13.3 / 12.6, K=8192 40.1 / 39.0).  K is a multiple of the 2048 columns of the eight load steps, which it
// otherwise leaves partly empty (2 x 8192: K=2560 26.6 / 24.7, 3072 27.1 / 26.2, 5120 even).  Beyond two waves the ramps count for less (2 x 14336 even, 2 x 20480
// 36.2 / 33.2); of the second wave's blocks those of up to 8704 rows are listed (54.8 / 63.4 at K=8192; 9216 and 10240 rows would gain 14 - 20 and 4 - 10 %, 12288 nothing).
static bool two_rows_listed(uint32_t M, uint32_t n, uint32_t K) {
    const uint32_t wave = 3 * 16 * (uint32_t)device_sms();
    return M == 2 && K % 2048 == 0 && n <= 8704 && (n > wave || 4 * n <= 3 * wave);
}

// rows per warp: fewer when the block has few rows, so that every SM still gets warps
template <int MT>
static void launch_gemv_rows(const bf16 *A, const bf16 *W, float *C, uint32_t Mrows, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int acc, cudaStream_t st) {
    if constexpr (MT <= 2) {
        if (n >= GEMV_MANY_ROWS && !(one_row_deep(MT, K) && one_row_fuller(n))) return launch_gemv<MT, 2, 4>(A, W, C, Mrows, n, K, ldc, col0, acc, st);
        if (n < GEMV_MANY_ROWS && g_gemv_splitk && K >= 8192) {                    // at least four 256-element chunks per warp and row
            if (n <= 1024) return launch_gemv_splitk<MT, 1, 4>(A, W, C, Mrows, n, K, ldc, col0, acc, st);
            return launch_gemv_splitk<MT, 2, 4>(A, W, C, Mrows, n, K, ldc, col0, acc, st);
        }
        return launch_gemv<MT, 1, 8>(A, W, C, Mrows, n, K, ldc, col0, acc, st);
    } else {
        if (n >= GEMV_MANY_ROWS) return launch_gemv<MT, 2, 2>(A, W, C, Mrows, n, K, ldc, col0, acc, st);
        return launch_gemv<MT, 1, 4>(A, W, C, Mrows, n, K, ldc, col0, acc, st);
    }
}

template <int MT, bool FUSED>
static void launch_gemv_group(const bf16 *A, const GemvParts &p, uint32_t Mrows, uint32_t n_total, uint32_t K, int acc, cudaStream_t st, const ASrc &src = ASrc{}) {
    static int blocks_per_sm = 0;
    if (!blocks_per_sm) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, tgp_wstream_group_kernel<MT, 8, FUSED>, 256, 0) != cudaSuccess || blocks_per_sm < 1) blocks_per_sm = 1;
    }
    uint32_t need = (n_total + 7) / 8, full = (uint32_t)(device_sms() * blocks_per_sm);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(need < full ? need : full);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    launch_weights<tgp_wstream_group_kernel<MT, 8, FUSED>>(cfg, A, p, Mrows, n_total, K, acc, src);
    tgpk_last_gemm_kernel = "tgp_wstream_group_kernel";
}

// ---- all experts of a layer in one launch ------------------------------------------------------------------------------------
// A decode step of a mixture routes a few tokens to each of several experts.  One launch per expert and matrix, sized by counts that
// the host has to wait for, left the GPU idle most of the time (16 users, 8 experts of 3 x 3584 x 1024: 190 us per layer, of which
// the weights in use take 18 us); here one launch covers the gate and up projections with SwiGLU of every expert that has
// tokens, a second one the down projections, and a third adds a token's two results to its residual row.  The counts
// are read on the device: work items are (expert, up to 8 NB of its tokens, 16 rows of gate and of up, or two groups of `rpc`
// rows of down), and the CTAs walk the list of those that exist.
//   The arithmetic of an item is that of tgp_wstream_mma_group_kernel<NB, EXP_U, NW, RG>: which warp adds which k in which order
// depends on K alone, so the bits are those of the expert's own products (tgpk_gemm_rows).
//   Experts of one or two tokens have no items: their rows follow, a warp each, on the CUDA cores, whose sums are closer to 64 bits
// (K=1024: 7.1e-8 against 1.3e-7 through mma.sync, K=14336: 9.3e-8 against 8.7e-7), as in the products of one and two rows.
struct ExpertParts {
    const bf16 *w[2][TGP_MOE_EXPERTS][TGP_MOE_BLOCKS];       // GLU: gate and up; else [0]: down; in blocks of `per` rows
    const bf16 *A;                                           // GLU: [M, K], rows picked by `rows`; else one row per routed slot
    const int32_t *rows, *counts;                            // token lists, `stride` apart
    void *out;                                               // GLU: bf16 [slots, n]; else fp32 [slots, n]
    uint32_t n, K, per, E, stride, rpc;
};

// 16 warps of four load steps, or up to K=2047 twice as many CTAs of eight: a chunk of 1024 columns, so that the K of a small expert
// keeps every warp at work.  Either way an SM has 64 KB of loads under way, as many as HBM needs.  More warps mean fewer
// additions in a row per warp: a warp adds K / (16 NW) MMAs, no more than in the products of 3 - 16 rows above.
constexpr int EXP_U = 4;
static int expert_warps(uint32_t K) { return K >= 2048 ? 16 : 8; }

// From this K on the products of one or two tokens of an expert have the sums of tgp_wstream_splitk_kernel, below it those of tgp_wstream_kernel.
constexpr uint32_t EXP_SPLIT_K = 8192;

// The rows of the `ns` experts listed in `small` (at most two tokens each), one warp per row (GLU: per row of gate and of up), eight 16-byte
// loads of weights under way.
template <bool GLU>
__device__ __forceinline__ void expert_rows_fma(const ExpertParts &p, const uint32_t *small, uint32_t ns, const uint32_t *s_slot, const uint32_t *s_cnt, uint32_t warp0, uint32_t warps) {
    constexpr int R = GLU ? 2 : 1, U = 8 / R;
    const uint32_t lane = threadIdx.x & 31, K = p.K, parts = K >= EXP_SPLIT_K ? 8 : 1;
    for (uint32_t i = warp0; i < ns * p.n; i += warps) {
        const uint32_t e = small[i / p.n], row = i % p.n, cnt = s_cnt[e];
        const bf16 *w[R], *x[2];
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = p.w[r][e][row / p.per] + (size_t)(row % p.per) * K;
#pragma unroll
        for (uint32_t m = 0; m < 2; ++m) x[m] = p.A + (size_t)(GLU ? (uint32_t)p.rows[(size_t)e * p.stride + min(m, cnt - 1)] : s_slot[e] + min(m, cnt - 1)) * K;
        float sum[R][2];
        for (uint32_t v = 0; v < parts; ++v) {              // (the eight warps of the split-K kernel, one after the other)
            float acc[R][2];
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r][0] = acc[r][1] = 0.f;
            for (uint32_t k0 = v * 256 + lane * 8; k0 < K; k0 += parts * 256 * U) {
                uint4 wv[U][R];
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const uint32_t k = k0 + parts * 256 * u;
                        wv[u][r] = k < K ? __ldcs(reinterpret_cast<const uint4 *>(w[r] + k)) : make_uint4(0, 0, 0, 0);
                    }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t k = k0 + parts * 256 * u;
#pragma unroll
                    for (uint32_t m = 0; m < 2; ++m) {
                        float xf[8];
                        unpack8(k < K && m < cnt ? ld_act(reinterpret_cast<const uint4 *>(x[m] + k)) : make_uint4(0, 0, 0, 0), xf);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            float wf[8];
                            unpack8(wv[u][r], wf);
#pragma unroll
                            for (int j = 0; j < 8; ++j) acc[r][m] = fmaf(wf[j], xf[j], acc[r][m]);
                        }
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int m = 0; m < 2; ++m) { const float t = warp_sum(acc[r][m]); sum[r][m] = v ? sum[r][m] + t : t; }
        }
        if (lane < cnt) {
            const size_t at = (size_t)(s_slot[e] + lane) * p.n + row;
            const float a = lane ? sum[0][1] : sum[0][0];
            if constexpr (GLU) { const float up = lane ? sum[1][1] : sum[1][0]; reinterpret_cast<bf16 *>(p.out)[at] = __float2bfloat16_rn(a / (1.0f + expf(-a)) * up); }
            else reinterpret_cast<float *>(p.out)[at] = a;
        }
    }
}

template <int NB, int NW, bool GLU>
__global__ void __launch_bounds__(NW * 32, 16 / NW) tgp_expert_mma_kernel(const ExpertParts p) {
    constexpr int U = EXP_U, G = 2, SK = U / (2 * G), T = NB * 8;       // T: tokens per item
    __shared__ float part[NW][G * NB * 4][32];
    __shared__ uint32_t s_first[TGP_MOE_EXPERTS + 1], s_slot[TGP_MOE_EXPERTS], s_cnt[TGP_MOE_EXPERTS], s_small[TGP_MOE_EXPERTS], s_ns;
    pdl_enter();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, c = lane & 3, K = p.K;
    const uint32_t span = GLU ? p.rpc : 2 * p.rpc, groups = (p.n + span - 1) / span;     // items per expert and token chunk
    if (threadIdx.x == 0) {
        uint32_t items = 0, slot = 0, ns = 0;
        for (uint32_t e = 0; e < p.E; ++e) {
            const uint32_t cnt = (uint32_t)p.counts[e];
            s_first[e] = items; s_slot[e] = slot; s_cnt[e] = cnt;
            if (cnt > 2) items += (cnt + T - 1) / T * groups;
            else if (cnt) s_small[ns++] = e;
            slot += cnt;
        }
        s_first[p.E] = items;
        s_ns = ns;
    }
    __syncthreads();
    const uint32_t total = s_first[p.E];
    // (the last CTAs, which have the fewest items, begin with the rows of the small experts)
    auto small = [&]() { expert_rows_fma<GLU>(p, s_small, s_ns, s_slot, s_cnt, (gridDim.x - 1 - blockIdx.x) * NW + warp, gridDim.x * NW); };
    if (blockIdx.x >= total) { small(); return; }
    const bf16 *wlo[G], *whi[G], *arow[NB];                  // of the item that is being loaded
    uint4 lo[2][G][SK], hi[2][G][SK], xs[2][SK][NB];
    float acc[G][NB][4];
    auto find = [&](uint32_t item, uint32_t &e, uint32_t &chunk, uint32_t &row0) {
        e = 0;
        while (item >= s_first[e + 1]) ++e;
        const uint32_t local = item - s_first[e];
        chunk = local / groups;
        row0 = local % groups * span;
    };
    auto locate = [&](uint32_t item) {
        uint32_t e, chunk, row0;
        find(item, e, chunk, row0);
#pragma unroll
        for (int r = 0; r < G; ++r) {
            const uint32_t first = GLU ? row0 : min(row0 + r * p.rpc, p.n - 1), last = min(first + p.rpc, p.n) - 1;
            const uint32_t a = min(first + g, last), b = min(first + g + 8, last);       // rows a group lacks re-read its last one
            const bf16 *const *blocks = p.w[GLU ? r : 0][e];
            wlo[r] = blocks[a / p.per] + (size_t)(a % p.per) * K + c * 8;
            whi[r] = blocks[b / p.per] + (size_t)(b % p.per) * K + c * 8;
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const uint32_t i = chunk * T + b * 8 + g;
            arow[b] = i >= s_cnt[e] ? nullptr : p.A + (size_t)(GLU ? (uint32_t)p.rows[(size_t)e * p.stride + i] : s_slot[e] + i) * K + c * 8;
        }
    };
    auto issue = [&](auto set, uint32_t kb) {
        constexpr int S = decltype(set)::value;
#pragma unroll
        for (int s = 0; s < SK; ++s) {
            const uint32_t k = kb + 32 * s;
#pragma unroll
            for (int r = 0; r < G; ++r) {
                lo[S][r][s] = k < K ? __ldcs(reinterpret_cast<const uint4 *>(wlo[r] + k)) : make_uint4(0, 0, 0, 0);
                hi[S][r][s] = k < K ? __ldcs(reinterpret_cast<const uint4 *>(whi[r] + k)) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int b = 0; b < NB; ++b) xs[S][s][b] = k < K && arow[b] ? ld_act(reinterpret_cast<const uint4 *>(arow[b] + k)) : make_uint4(0, 0, 0, 0);
        }
    };
    auto consume = [&](auto set) {
        constexpr int S = decltype(set)::value;
#pragma unroll
        for (int s = 0; s < SK; ++s)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const uint4 xv = xs[S][s][b];
#pragma unroll
                for (int r = 0; r < G; ++r) {
                    mma_bf16_16816(acc[r][b], lo[S][r][s].x, hi[S][r][s].x, lo[S][r][s].y, hi[S][r][s].y, xv.x, xv.y);
                    mma_bf16_16816(acc[r][b], lo[S][r][s].z, hi[S][r][s].z, lo[S][r][s].w, hi[S][r][s].w, xv.z, xv.w);
                }
            }
    };
    auto clear = [&]() {
#pragma unroll
        for (int r = 0; r < G; ++r)
#pragma unroll
            for (int b = 0; b < NB; ++b) { acc[r][b][0] = acc[r][b][1] = acc[r][b][2] = acc[r][b][3] = 0.f; }
    };
    const std::integral_constant<int, 0> set0;
    const std::integral_constant<int, 1> set1;
    // one stream of loads over all items of this CTA, two register sets, as in tgp_wstream_mma_group_kernel
    uint32_t cur = blockIdx.x, item = cur, k0 = warp * 32 * U, pr = 0;
    auto advance = [&]() -> bool {
        if (++pr == (uint32_t)G) { pr = 0; k0 += NW * 32 * U; }
        if (k0 < K) return false;
        item += gridDim.x;
        k0 = warp * 32 * U;
        pr = 0;
        if (item < total) locate(item);
        return true;
    };
    locate(item);
    issue(set0, k0);
    issue(set1, k0 + 32 * SK);
    bool cur_last = advance();
    clear();
    for (;;) {
        const bool have_next = item < total;
        const uint32_t kb = k0 + pr * 64 * SK;
        consume(set0);
        if (have_next) issue(set0, kb);
        consume(set1);
        if (have_next) issue(set1, kb + 32 * SK);
        const bool next_last = have_next ? advance() : false;
        const bool ended = cur_last;
        cur_last = next_last;
        if (!ended) continue;
#pragma unroll
        for (int r = 0; r < G; ++r)
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int i = 0; i < 4; ++i) part[warp][(r * NB + b) * 4 + i][lane] = acc[r][b][i];
        __syncthreads();
        uint32_t e, chunk, row0;
        find(cur, e, chunk, row0);
        for (uint32_t v = threadIdx.x; v < (GLU ? 1 : G) * NB * 4 * 32; v += NW * 32) {
            const uint32_t slot = v >> 5, ln = v & 31, r = slot / (NB * 4), b = (slot >> 2) % NB, i = slot & 3;
            float sum = 0.f, up = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) sum += part[w][slot][ln];
            if constexpr (GLU) {
#pragma unroll
                for (int w = 0; w < NW; ++w) up += part[w][NB * 4 + slot][ln];
            }
            const uint32_t first = row0 + r * p.rpc, row = first + (ln >> 2) + 8 * (i >> 1), t = chunk * T + b * 8 + 2 * (ln & 3) + (i & 1);
            if (t < s_cnt[e] && row < min(first + p.rpc, p.n)) {
                const size_t at = (size_t)(s_slot[e] + t) * p.n + row;
                if constexpr (GLU) reinterpret_cast<bf16 *>(p.out)[at] = __float2bfloat16_rn(sum / (1.0f + expf(-sum)) * up);
                else reinterpret_cast<float *>(p.out)[at] = sum;
            }
        }
        cur += gridDim.x;
        if (cur >= total) break;
        __syncthreads();
        clear();
    }
    small();
}

// x[m, :] += gate * y[slot of m in its expert, :], experts in ascending order: the sums of tgp_scatter_add_kernel expert by expert.
__global__ void __launch_bounds__(256) tgp_expert_combine_kernel(float *x, const float *y, const int32_t *idx, const float *gate, const int32_t *pos, const int32_t *counts, uint32_t d) {
    pdl_enter();
    const uint32_t m = blockIdx.x;
    int e[2] = {idx[2 * m], idx[2 * m + 1]}, s[2] = {0, 1};
    if (e[1] >= 0 && e[1] < e[0]) { s[0] = 1; s[1] = 0; }
    const float4 *src[2] = {nullptr, nullptr};
    float g[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int ex = e[s[i]];
        if (ex < 0) continue;
        uint32_t slot = (uint32_t)pos[2 * m + s[i]];
        for (int q = 0; q < ex; ++q) slot += (uint32_t)counts[q];
        src[i] = reinterpret_cast<const float4 *>(y + (size_t)slot * d);
        g[i] = gate[2 * m + s[i]];
    }
    float4 *o = reinterpret_cast<float4 *>(x + (size_t)m * d);
    for (uint32_t i = blockIdx.y * 256 + threadIdx.x; i < d / 4; i += gridDim.y * 256) {
        float4 a = o[i];
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (src[q]) {
                const float4 b = src[q][i];
                a.x += g[q] * b.x; a.y += g[q] * b.y; a.z += g[q] * b.z; a.w += g[q] * b.w;
            }
        o[i] = a;
    }
}

// Whether the products of a step's experts take tgpk_gemm_rows() and may run all in one launch: the step has 3 to 32 tokens.
bool tgpk_expert_rows(uint32_t M, uint32_t K) { return M >= 3 && M <= 32 && K % 32 == 0 && g_skinny_impl == 0 && g_gemm_impl == 0; }

// EXP_U load steps per chunk everywhere; 16 warps on up to 8 activation rows have registers for twice as many steps under way, from one
// chunk of two row groups or two chunks of one.
template <int NB, int NW, int RG>
static void launch_expert_rows(cudaLaunchConfig_t &cfg, const bf16 *A, const GemvParts &p, uint32_t me, uint32_t groups, uint32_t K, uint32_t rpc) {
    auto launch = [&](auto steps) {
        constexpr int U = decltype(steps)::value;
        constexpr size_t smem = (size_t)NW * RG * NB * 4 * 32 * 4;
        if constexpr (smem > 48 * 1024) {
            tgpk_allow_smem<tgp_wstream_mma_group_kernel<NB, U, NW, RG, EXP_U>>(smem);
            cfg.dynamicSmemBytes = smem;
        }
        launch_weights<tgp_wstream_mma_group_kernel<NB, U, NW, RG, EXP_U>>(cfg, A, p, me, groups, K, 0, rpc, 0);
    };
    if constexpr (NB == 1 && NW == 16)
        if (RG == 2 || K > NW * 32 * EXP_U) return launch(std::integral_constant<int, 2 * EXP_U>());
    launch(std::integral_constant<int, EXP_U>());
}

// Blocks over the same `me` activation rows (at most 32) with the arithmetic of the expert kernels, in one launch: the row groups and rows per
// group of launch_skinny(), which the bits do not depend on.  One or two rows: the CUDA cores' products, one launch per block from EXP_SPLIT_K on.
int tgpk_gemm_rows(const void *A, uint32_t count, const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t me, uint32_t K, cudaStream_t st) {
    if (!count || count > TGP_GEMM_GROUP_MAX || K % 32 || me > 32) return TGP_E_INVAL;
    if (!me) return TGP_OK;
    const bf16 *a = (const bf16 *)A;
    if (me <= 2 && K >= EXP_SPLIT_K) {
        for (uint32_t s = 0; s < count; ++s) {
            if (n[s] <= 1024) { if (me == 1) launch_gemv_splitk<1, 1, 4>(a, (const bf16 *)W[s], C[s], me, n[s], K, ldc[s], 0, 0, st); else launch_gemv_splitk<2, 1, 4>(a, (const bf16 *)W[s], C[s], me, n[s], K, ldc[s], 0, 0, st); }
            else { if (me == 1) launch_gemv_splitk<1, 2, 4>(a, (const bf16 *)W[s], C[s], me, n[s], K, ldc[s], 0, 0, st); else launch_gemv_splitk<2, 2, 4>(a, (const bf16 *)W[s], C[s], me, n[s], K, ldc[s], 0, 0, st); }
        }
        LAUNCH_CHECK(count);
        return TGP_OK;
    }
    GemvParts p;
    memset(&p, 0, sizeof(p));
    uint32_t total = 0;
    for (uint32_t s = 0; s < count; ++s) { p.W[s] = (const bf16 *)W[s]; p.C[s] = C[s]; p.n[s] = n[s]; p.ldc[s] = ldc[s]; total += n[s]; }
    p.count = count;
    if (me <= 2) {
        if (count == 1) { if (me == 1) launch_gemv_rows<1>(a, p.W[0], p.C[0], me, n[0], K, ldc[0], 0, 0, st); else launch_gemv_rows<2>(a, p.W[0], p.C[0], me, n[0], K, ldc[0], 0, 0, st); }
        else if (me == 1) launch_gemv_group<1, false>(a, p, me, total, K, 0, st);
        else launch_gemv_group<2, false>(a, p, me, total, K, 0, st);
        LAUNCH_CHECK(1);
        return TGP_OK;
    }
    const uint32_t nb = me <= 8 ? 1 : me <= 16 ? 2 : 4, nw = (uint32_t)expert_warps(K), full = 16 / nw * (uint32_t)device_sms();
    uint32_t best = 0xffffffffu, rpc = 16, RG = 1, groups = 0;
    for (uint32_t G = 2; G >= 1; --G)
        for (uint32_t r = 9; r <= 16; ++r) {
            uint32_t g = 0;
            for (uint32_t s = 0; s < count; ++s) g += (n[s] + r - 1) / r;
            const uint32_t rounds = ((g + G - 1) / G + full - 1) / full, cost = rounds * (G * (r + 16) + 8 * nb);
            if (cost < best) { best = cost; rpc = r; RG = G; groups = g; }
        }
    for (uint32_t s = 0; s < count; ++s) p.groups[s] = (n[s] + rpc - 1) / rpc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min((groups + RG - 1) / RG, full)); cfg.blockDim = dim3(nw * 32); cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
#define TGP_EXPERT_ROWS(NB_) do { \
        if (nw == 8) { if (RG == 2) launch_expert_rows<NB_, 8, 2>(cfg, a, p, me, groups, K, rpc); else launch_expert_rows<NB_, 8, 1>(cfg, a, p, me, groups, K, rpc); } \
        else { if (RG == 2) launch_expert_rows<NB_, 16, 2>(cfg, a, p, me, groups, K, rpc); else launch_expert_rows<NB_, 16, 1>(cfg, a, p, me, groups, K, rpc); } } while (0)
    if (nb == 1) TGP_EXPERT_ROWS(1); else if (nb == 2) TGP_EXPERT_ROWS(2); else TGP_EXPERT_ROWS(4);
#undef TGP_EXPERT_ROWS
    tgpk_last_gemm_kernel = "tgp_wstream_mma_group_kernel";
    LAUNCH_CHECK(1);
    return TGP_OK;
}

template <bool GLU>
static void launch_experts(const ExpertParts &p, uint32_t T, cudaStream_t st) {
    const uint32_t warps = (uint32_t)expert_warps(p.K);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16 / warps * (uint32_t)device_sms()); cfg.blockDim = dim3(32 * warps); cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = small_overlap();
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (warps == 8) { if (T == 8) launch_weights<tgp_expert_mma_kernel<1, 8, GLU>>(cfg, p); else launch_weights<tgp_expert_mma_kernel<2, 8, GLU>>(cfg, p); }
    else { if (T == 8) launch_weights<tgp_expert_mma_kernel<1, 16, GLU>>(cfg, p); else launch_weights<tgp_expert_mma_kernel<2, 16, GLU>>(cfg, p); }
}

int tgpk_experts(const TgpExperts &x, cudaStream_t st) {
    if (x.E > TGP_MOE_EXPERTS || !tgpk_expert_rows(x.M, x.d) || x.F % 32) return TGP_E_INVAL;
    const uint32_t sms = (uint32_t)device_sms(), T = x.M <= 8 ? 8 : 16;
    ExpertParts p;
    memset(&p, 0, sizeof(p));
    p.rows = x.rows; p.counts = x.counts; p.E = x.E; p.stride = x.stride;
    for (uint32_t e = 0; e < x.E; ++e)
        for (uint32_t b = 0; b < TGP_MOE_BLOCKS; ++b) { p.w[0][e][b] = (const bf16 *)x.w[0][e][b]; p.w[1][e][b] = (const bf16 *)x.w[1][e][b]; }
    p.A = (const bf16 *)x.h; p.out = x.a; p.n = x.F; p.K = x.d; p.per = x.per_f; p.rpc = 16;
    launch_experts<true>(p, T, st);
    for (uint32_t e = 0; e < x.E; ++e)
        for (uint32_t b = 0; b < TGP_MOE_BLOCKS; ++b) { p.w[0][e][b] = (const bf16 *)x.w[2][e][b]; p.w[1][e][b] = nullptr; }
    p.A = (const bf16 *)x.a; p.out = x.y; p.n = x.d; p.K = x.F; p.per = x.per_d;
    // rows per group: the fewest rounds of the busiest CTA, weighted with its loads (rows a group lacks still take load slots), if three
    // quarters of the experts that could have tokens do
    const uint32_t slots = 16 / (uint32_t)expert_warps(x.F) * sms, busy = std::max(1u, std::min(x.E, x.M * x.topk) * 3 / 4);
    uint64_t best = ~0ull;
    for (uint32_t r = 16; r >= 5; --r) {
        const uint64_t items = (uint64_t)busy * ((x.d + 2 * r - 1) / (2 * r)), cost = (items + slots - 1) / slots * (r + 16 + 4);
        if (cost < best) { best = cost; p.rpc = r; }
    }
    launch_experts<false>(p, T, st);
    launch_pdl(tgp_expert_combine_kernel, dim3(x.M, x.d > 2048 ? 2 : 1), dim3(256), 0, st, x.x, (const float *)x.y, x.idx, x.gate, x.pos, x.counts, x.d);
    tgpk_last_gemm_kernel = "tgp_expert_mma_kernel";
    LAUNCH_CHECK(3);
    return TGP_OK;
}

// Which neighbours of a list may share a launch: those with the same non-zero key.  A key names the kernel a block takes on its own
// (M <= 2: tgp_wstream_kernel<MT, 1, 8>, or a kernel with its sums; 3 <= M <= 32: one instance of the persistent list kernel, or the tcgen05 kernel and
// split of K); blocks that gain nothing from a list, and the shapes served by other kernels, have key 0 and are launched alone.
uint32_t tgpk_gemm_group_key(uint32_t M, uint32_t n, uint32_t K) {
    if (!g_gemm_group || !M || !n || !K || K % 8) return 0;
    // Blocks of many rows at M <= 2 run one behind the other at little cost, but a list of them has one ramp instead of several (one row,
    // with the norm before: 2 x 14336, K=4096 41.0 -> 37.0 us).
    if (M <= 2 && n >= GEMV_MANY_ROWS) return one_row_deep(M, K) || two_rows_listed(M, n, K) ? 0x100u | M : 0;
    if (M <= 2) return !(g_gemv_splitk && K >= 8192) ? M : 0;
    if (M > 32) return 0;
    if (takes_tiles(M, n, K)) return tgpk_gemm_tc_forced() ? 0 : 0x2000000u | tgpk_gemm_tc_class(M, n, K);
    if (M > 16 || K % 32 || g_skinny_impl) return 0;
    const SkinnyPick k = pick_skinny(M, n, K);
    return k.persistent ? (0x1100000u | (uint32_t)k.nb | (uint32_t)k.u << 4 | (uint32_t)k.nw << 8) : 0;
}

// Blocks of one key below 0x2000000 over the same activations, in one launch.
static int gemm_list(const bf16 *A, uint32_t count, const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t M, uint32_t K, int accumulate, cudaStream_t st) {
    GemvParts p;
    memset(&p, 0, sizeof(p));
    uint32_t total = 0;
    for (uint32_t s = 0; s < count; ++s) { p.W[s] = (const bf16 *)W[s]; p.C[s] = C[s]; p.n[s] = n[s]; p.ldc[s] = ldc[s]; total += n[s]; }
    p.count = count;
    if (M == 1) launch_gemv_group<1, false>(A, p, M, total, K, accumulate, st);
    else if (M == 2) launch_gemv_group<2, false>(A, p, M, total, K, accumulate, st);
    else launch_skinny_pick(A, p, pick_skinny(M, n[0], K), M, K, accumulate, st);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

int tgpk_gemm_group(const void *A, uint32_t count, const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t M, uint32_t K,
                    int accumulate, cudaStream_t st) {
    if (!count || !M) return TGP_OK;
    // Neighbours with one key share a launch, the others are launched alone (q of a large model takes the tcgen05 kernel at 16 rows, its k and v
    // the list kernel: each in a launch of its own 62 us at d=8192, 1024 rows of k and of v, 37 with k and v in one).  From 33 rows on the key is that of the tcgen05 kernels.
    auto key_of = [&](uint32_t s) -> uint32_t {
        if (M <= 32) return tgpk_gemm_group_key(M, n[s], K);
        return g_gemm_group && n[s] && takes_tiles(M, n[s], K) && !tgpk_gemm_tc_forced() ? 0x2000000u | tgpk_gemm_tc_class(M, n[s], K) : 0u;
    };
    for (uint32_t s = 0; s < count;) {
        const uint32_t key = key_of(s);
        uint32_t e = s + 1;
        while (key && e < count && e - s < TGP_GEMM_GROUP_MAX && key_of(e) == key) ++e;
        int rc;
        if (e - s == 1) rc = tgpk_gemm(A, W[s], C[s], M, n[s], K, ldc[s], 0, accumulate, st);
        else if (key >= 0x2000000u) rc = tgpk_gemm_tc_list(A, e - s, W + s, C + s, n + s, ldc + s, M, K, accumulate, st);
        else rc = gemm_list((const bf16 *)A, e - s, W + s, C + s, n + s, ldc + s, M, K, accumulate, st);
        if (rc) return rc;
        s = e;
    }
    return TGP_OK;
}

// Products of M <= 2 activation rows whose activations are computed on the fly (see ASrc): the RMSNorm of x, or SwiGLU of
// (g32, u32).  Every block must carry the M <= 2 group key (tgpk_gemm_group_key(M, n, K) == M); K % 8 == 0.
int tgpk_gemm_group_fused(int mode, const float *x, uint32_t ldx, const void *gain, float eps, const float *g32, const float *u32, uint32_t count,
                          const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t M, uint32_t K, int accumulate, cudaStream_t st) {
    if (!count || count > TGP_GEMM_GROUP_MAX || !M || M > 2 || K % 8 || (mode != 1 && mode != 2)) return TGP_E_INVAL;
    for (uint32_t s = 0; s < count; ++s) if (tgpk_gemm_group_key(M, n[s], K) != M) return TGP_E_INVAL;
    GemvParts p;
    memset(&p, 0, sizeof(p));
    uint32_t total = 0;
    for (uint32_t s = 0; s < count; ++s) { p.W[s] = (const bf16 *)W[s]; p.C[s] = C[s]; p.n[s] = n[s]; p.ldc[s] = ldc[s]; total += n[s]; }
    p.count = count;
    const ASrc src{mode, x, ldx, (const bf16 *)gain, eps, g32, u32};
    if (M == 1) launch_gemv_group<1, true>(nullptr, p, M, total, K, accumulate, st, src);
    else launch_gemv_group<2, true>(nullptr, p, M, total, K, accumulate, st, src);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

template <int MT, int U>
static void launch_glu(const bf16 *A, const GluParts &p, bf16 *out, uint32_t Mrows, uint32_t F, uint32_t K, cudaStream_t st) {
    static int blocks_per_sm = 0;
    if (!blocks_per_sm && (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, tgp_wstream_glu_kernel<MT, U>, 256, 0) != cudaSuccess || blocks_per_sm < 1)) blocks_per_sm = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min((F + 7) / 8, (uint32_t)(device_sms() * blocks_per_sm)));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tgpk_launch_overlap() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    launch_weights<tgp_wstream_glu_kernel<MT, U>>(cfg, A, p, out, Mrows, F, K);
    tgpk_last_gemm_kernel = "tgp_wstream_glu_kernel";
}

// Would each of a matrix's blocks, alone or in a list, have the sums of tgp_wstream_kernel?
bool tgpk_glu_rows_ok(uint32_t M, uint32_t n, uint32_t K) {
    return g_gemm_group && M && M <= 2 && n && K && K % 8 == 0 && (n >= GEMV_MANY_ROWS || !(g_gemv_splitk && K >= 8192));
}

// a = bf16(silu(A gate^T) * (A up^T)) for M <= 2 rows, gate and up in `count` blocks of n[s] rows each, every one of them with tgpk_glu_rows_ok().
int tgpk_glu_rows(const void *A, uint32_t count, const void *const *gate, const void *const *up, const uint32_t *n, void *out, uint32_t M, uint32_t K, cudaStream_t st) {
    if (!count || count > TGP_GEMM_GROUP_MAX / 2) return TGP_E_INVAL;
    GluParts p;
    memset(&p, 0, sizeof(p));
    uint32_t F = 0;
    for (uint32_t s = 0; s < count; ++s) {
        if (!tgpk_glu_rows_ok(M, n[s], K)) return TGP_E_INVAL;
        p.gate[s] = (const bf16 *)gate[s]; p.up[s] = (const bf16 *)up[s]; p.n[s] = n[s]; F += n[s];
    }
    p.count = count;
    // One row from K = 4096 on: all sixteen loads of 2048 columns under way (a run of 48 steps, 2 layers of 14336 x 4096 30.69 ms against 30.81 with eight;
    // 4 x 4096 x 1024 7.67 with eight, 7.92 with sixteen).
    if (M == 1 && K >= 4096) launch_glu<1, 8>((const bf16 *)A, p, (bf16 *)out, M, F, K, st);
    else if (M == 1) launch_glu<1, 4>((const bf16 *)A, p, (bf16 *)out, M, F, K, st);
    else launch_glu<2, 4>((const bf16 *)A, p, (bf16 *)out, M, F, K, st);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

int tgpk_gemm(const void *A, const void *W, float *C, uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate, cudaStream_t st) {
    if (!M || !n) return TGP_OK;
    if (K % 8 || !K) return TGP_E_INVAL;
    const bf16 *a = (const bf16 *)A, *w = (const bf16 *)W;
    if (takes_tiles(M, n, K)) return tgpk_gemm_tc(A, W, C, M, n, K, ldc, col0, accumulate, st);
    if (M >= 3 && M <= 16 && K % 32 == 0 && g_skinny_impl == 0) {
        GemvParts p;
        memset(&p, 0, sizeof(p));
        p.W[0] = w; p.C[0] = C + col0; p.n[0] = n; p.ldc[0] = ldc; p.count = 1;
        launch_skinny_pick(a, p, pick_skinny(M, n, K), M, K, accumulate, st);
    } else if (M <= 16) {
        for (uint32_t m0 = 0; m0 < M; m0 += 8) {
            uint32_t mr = M - m0 < 8 ? M - m0 : 8;
            const bf16 *am = a + (size_t)m0 * K;
            float *cm = C + (size_t)m0 * ldc;
            if (mr == 1) launch_gemv_rows<1>(am, w, cm, mr, n, K, ldc, col0, accumulate, st);
            else if (mr == 2) launch_gemv_rows<2>(am, w, cm, mr, n, K, ldc, col0, accumulate, st);
            else if (mr <= 4) launch_gemv_rows<4>(am, w, cm, mr, n, K, ldc, col0, accumulate, st);
            else launch_gemv_rows<8>(am, w, cm, mr, n, K, ldc, col0, accumulate, st);
            if (m0) tgpk_launches += 1;
        }
    } else {
        dim3 grid((n + 63) / 64, (M + 63) / 64);
        tgp_matmul_simt_kernel<<<grid, 256, 0, st>>>(a, w, C, M, n, K, ldc, col0, accumulate);
        tgpk_last_gemm_kernel = "tgp_matmul_simt_kernel";
    }
    LAUNCH_CHECK(1);
    return TGP_OK;
}

bool tgpk_swiglu_fusable(uint32_t M) { return M > 128 && g_gemm_impl == 0; }

int tgpk_rope_kv(const float *q32, const float *k32, const float *v32, void *qb, const TgpTilePtrs &tiles, const float *cos_t, const float *sin_t,
                 const tgp_model_cfg *c, uint32_t B, uint32_t q_len, uint32_t pos0, cudaStream_t st) {
    if (!B || !q_len) return TGP_OK;
    RopeArgs a{q32, k32, v32, (bf16 *)qb, cos_t, sin_t, c->Hq, c->Hkv, c->Dh, c->TK, q_len, pos0, tiles};
    uintptr_t bits = reinterpret_cast<uintptr_t>(q32) | reinterpret_cast<uintptr_t>(k32) | reinterpret_cast<uintptr_t>(v32) | reinterpret_cast<uintptr_t>(cos_t) |
                     reinterpret_cast<uintptr_t>(sin_t) | reinterpret_cast<uintptr_t>(qb);
    for (uint32_t j = pos0 / c->TK; j <= (pos0 + q_len - 1) / c->TK && j < TGP_MAX_TILES; ++j) bits |= reinterpret_cast<uintptr_t>(tiles.k[j]) | reinterpret_cast<uintptr_t>(tiles.v[j]);
    const uint32_t items = (c->Hq + 2 * c->Hkv) * (c->Dh / 8);
    // CTAs per position: one item per thread while the positions alone do not fill the GPU (four CTAs of 256 threads per SM)
    const uint32_t split = std::max(1u, std::min((items + 255) / 256, 4u * (uint32_t)device_sms() / (B * q_len)));
    if (c->Dh == 64 && (bits & 15u) == 0) launch_pdl(tgp_rope_kv_vec_kernel<64>, dim3(B * q_len, split), dim3(256), 0, st, a);
    else if (c->Dh == 128 && (bits & 15u) == 0) launch_pdl(tgp_rope_kv_vec_kernel<128>, dim3(B * q_len, split), dim3(256), 0, st, a);
    else launch_pdl(tgp_rope_kv_kernel, dim3(B * q_len), dim3(256), 0, st, a);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

static int g_attn_decode_grouped = 1;   // decode: one pass over a KV tile serves all query heads of the group (0: one pass per head)
static int g_attn_decode_impl = 0;      // decode: 0 and 2 the tensor-core kernel wherever its geometry allows, 1 the CUDA-core per-tile kernels only
static int g_attn_impl = 0;      // q_len >= 16: 0 by problem size, 3 tcgen05 kernel, 2 mma.sync flash kernel, 1 warp-per-row CUDA-core kernel

// Does the tensor-core decode kernel serve a step?  Whole 16-key chunks inside a tile, 16-byte aligned rows, 1, 2, 4 or 8 query heads per KV head.  It is ahead at any
// length (us with the merge, against the per-tile kernels: 40 keys of 4 heads 1.8 / 4.3, which is one CTA per head and no merge; one sequence
// of 32 over 8 heads x 64, 130 keys 4.2 / 5.8, 700 keys 4.9 / 6.6; 1500 keys of 8 heads over 1 x 128: 6.7 / 13.3)
static bool decode_mma(const void *qb, const TgpTilePtrs &tiles, const tgp_model_cfg *c, uint32_t q_len, uint32_t pos0, const float *scratch) {
    const uint32_t G = c->Hq / c->Hkv, nt = (pos0 + 1 + c->TK - 1) / c->TK;
    if (q_len != 1 || !scratch || !g_attn_decode_grouped || (G != 1 && G != 2 && G != 4 && G != 8) || c->Hq % c->Hkv || g_attn_decode_impl == 1 || c->TK % DEC_KEYS) return false;
    bool aligned = (reinterpret_cast<uintptr_t>(qb) & 3u) == 0;
    for (uint32_t t = 0; t < nt && aligned; ++t) aligned = ((reinterpret_cast<uintptr_t>(tiles.k[t]) | reinterpret_cast<uintptr_t>(tiles.v[t])) & 15u) == 0;
    return aligned;
}

// (rope: the projections of a decode step's new position, not yet rotated; qb is then written only where the two ops are launched apart)
int tgpk_attn(const void *qb, const TgpTilePtrs &tiles, uint32_t n_tiles, void *ob, const tgp_model_cfg *c, uint32_t B, uint32_t q_len, uint32_t pos0,
              float *scratch, cudaStream_t st, const TgpRopeIn *rope) {
    if (!B || !q_len) return TGP_OK;
    if (c->Dh != 64 && c->Dh != 128) return TGP_E_INVAL;
    AttnArgs a{(const bf16 *)qb, (bf16 *)ob, scratch, c->Hq, c->Hkv, c->Dh, c->TK, q_len, pos0, n_tiles, 1.0f / sqrtf((float)c->Dh), tiles, 0, {}};
    bool rotates = false;
    if (rope) {
        const uintptr_t bits = reinterpret_cast<uintptr_t>(rope->q32) | reinterpret_cast<uintptr_t>(rope->k32) | reinterpret_cast<uintptr_t>(rope->v32) |
                               reinterpret_cast<uintptr_t>(rope->cos_t) | reinterpret_cast<uintptr_t>(rope->sin_t);
        const uint32_t G = c->Hkv ? c->Hq / c->Hkv : 0;
        rotates = decode_mma(qb, tiles, c, q_len, pos0, scratch) && (bits & 15u) == 0 && G * c->Hkv == c->Hq;
        if (rotates) a.rope = *rope;
        else if (int rc = tgpk_rope_kv(rope->q32, rope->k32, rope->v32, const_cast<void *>(qb), tiles, rope->cos_t, rope->sin_t, c, B, q_len, pos0, st)) return rc;
    }
    if (q_len == 1 && scratch) {
        const uint32_t nt = (pos0 + 1 + c->TK - 1) / c->TK, G = c->Hq / c->Hkv;
        if (G > 32) return TGP_E_TOO_LARGE;
        uint32_t split = (c->TK + 31) / 32;
        if (split > 32 / G) split = 32 / G;
        if (split < 1) split = 1;
        dim3 grid(nt, c->Hkv, B);
        const bool grouped = g_attn_decode_grouped && (G == 1 || G == 2 || G == 4 || G == 8) && c->Hq % c->Hkv == 0;
        const uint32_t nchunks = (pos0 + 1 + DEC_KEYS - 1) / DEC_KEYS;
        if (decode_mma(qb, tiles, c, q_len, pos0, scratch)) {
            const int sms = device_sms();
            const uint32_t units = B * c->Hkv, per_sm = c->Dh == 64 ? 4 : 2;             // CTAs that fit an SM (96 / 48 KB of shared memory each)
            uint32_t parts = (uint32_t)sms * per_sm / units;                              // CTAs per (sequence, KV head): one wave at most
            const uint32_t slots = (uint32_t)sms * per_sm;
            parts = std::max(1u, std::min(parts, (nchunks + DEC_WARPS - 1) / DEC_WARPS));
            // A short context stays in one CTA, whose chain of a few chunks per warp is over sooner than a cluster has met, the longer a chain the
            // more CTAs there are (one part against four, us with the norm before: 32 heads over 8 x 64, one sequence, 100 keys 4.7 / 5.3, 200 keys
            // 5.8 / 5.3; 16 sequences, 200 keys 5.3 / 6.8, 400 keys 6.8 / 7.4 but 14.5 / 13.0 with a product on either side; x 128 against two, 400 keys 9.4 / 10.4).
            const bool one = nchunks <= std::max(12u, 8 + (units * c->Dh + 511) / 512);
            // Up to DEC_CLUSTER parts can be a cluster, which merges them itself; more parts meet in the scratch array and a second kernel.
            // Eight CTAs need one GPC to hold them: a context takes eight only while its clusters leave half of the GPU free, and beyond 1024 keys only if they are few
            // (eight parts against all, us: 32 heads over 8 x 64, B=1, 700 keys 3.7 / 5.2, 2112 keys 5.3 / 8.8, 4000 6.8 / 6.9, 9000 11.8 / 10.6; x 128, 2112 keys
            // 7.1 / 9.5, 4000 9.5 / 8.3; a step of two layers, B=4, 16000 keys 356 / 321; 32 units x 128, 700 keys with a product on either side:
            // 17.7 in eight parts, 14.5 in four).
            const bool eight = (nchunks <= 64 && 16 * units <= slots) || (units <= 16 && (nchunks <= 192 || n_tiles <= DEC_CLUSTER));
            // Up to four parts are one if seven eighths of the GPU hold all clusters: in the rest there is room for CTAs, but not for clusters, and the last of
            // them run alone (a layer of d=512, 24 sequences of 8 heads x 64, 6000 keys, three parts each for 592 places: 94.5 us in clusters, 80.5 through the scratch array).
            // (the scratch array holds a partial per KV tile: where that is four or fewer, a cluster of four is at least as many)
            const bool clustered = eight || ((nchunks <= 64 || parts <= 4 || n_tiles <= 4) && 8 * units * std::min(parts, 4u) <= 7 * slots);
            parts = one ? 1u : std::min(parts, eight ? (uint32_t)DEC_CLUSTER : clustered ? 4u : n_tiles);
            const uint32_t per_cta = (nchunks + parts - 1) / parts;
            parts = (nchunks + per_cta - 1) / per_cta;                                    // no CTA without a chunk
            const bool cluster = clustered && parts > 1, merge = !clustered && parts > 1;
            a.n_parts = parts;
            // below 256 chunks in all the kernel is bound by latency and takes no longer with all of P (1183 shapes of 1 - 4000 keys: 3.4 us
            // on average, 3.4 with two parts, 7.8 on the CUDA cores; results that are not the rounded exact value: 1 in 7750, 1 in 720, 1 in 7500)
            const bool split_p = nchunks * B * c->Hkv < 256;
            const size_t smem = (size_t)DEC_WARPS * DEC_STAGES * 2 * DEC_KEYS * c->Dh * 2;        // 96 KB at Dh = 128, 48 KB at 64
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(parts, c->Hkv, B); cfg.blockDim = dim3(DEC_WARPS * 32); cfg.dynamicSmemBytes = smem; cfg.stream = st;
            cudaLaunchAttribute attr[2];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = small_overlap();
            attr[1].id = cudaLaunchAttributeClusterDimension;
            attr[1].val.clusterDim.x = parts; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = cluster ? 2 : 1;
#define TGP_DECODE_MMA_R(DH_, G_, SP_, CL_, RO_) do { \
                if (!tgpk_allow_smem<tgp_attn_decode_mma_kernel<DH_, G_, SP_, CL_, RO_>>(smem)) return TGP_E_CUDA; \
                cudaLaunchKernelEx(&cfg, tgp_attn_decode_mma_kernel<DH_, G_, SP_, CL_, RO_>, a, per_cta); } while (0)
#define TGP_DECODE_MMA_P(DH_, G_, SP_, CL_) do { if (rotates) TGP_DECODE_MMA_R(DH_, G_, SP_, CL_, true); else TGP_DECODE_MMA_R(DH_, G_, SP_, CL_, false); } while (0)
#define TGP_DECODE_MMA(DH_, G_) do { if (cluster) { if (split_p) TGP_DECODE_MMA_P(DH_, G_, true, true); else TGP_DECODE_MMA_P(DH_, G_, false, true); } \
                else { if (split_p) TGP_DECODE_MMA_P(DH_, G_, true, false); else TGP_DECODE_MMA_P(DH_, G_, false, false); } } while (0)
#define TGP_DECODE_MMA_G(DH_) do { if (G == 1) TGP_DECODE_MMA(DH_, 1); else if (G == 2) TGP_DECODE_MMA(DH_, 2); else if (G == 4) TGP_DECODE_MMA(DH_, 4); else TGP_DECODE_MMA(DH_, 8); } while (0)
            if (c->Dh == 64) { TGP_DECODE_MMA_G(64); if (merge) launch_pdl(tgp_attn_decode_merge_kernel<64>, dim3(c->Hq, B), dim3(64), 0, st, a); }
            else { TGP_DECODE_MMA_G(128); if (merge) launch_pdl(tgp_attn_decode_merge_kernel<128>, dim3(c->Hq, B), dim3(128), 0, st, a); }
#undef TGP_DECODE_MMA_G
#undef TGP_DECODE_MMA
#undef TGP_DECODE_MMA_P
#undef TGP_DECODE_MMA_R
            LAUNCH_CHECK(merge ? 2 : 1);
            return TGP_OK;
        }
        if (grouped) {                                      // K and V read once for the whole group of query heads
            split = (c->TK + 31) / 32;
            if (split > 8) split = 8;
        }
        const size_t sm = (size_t)(G * c->Dh + G * split * (c->Dh + 2)) * sizeof(float);
#define TGP_DECODE_GROUP(DH_) do { \
            if (G == 1) launch_pdl(tgp_attn_decode_group_kernel<DH_, 1>, grid, dim3(32 * split), sm, st, a, split); \
            else if (G == 2) launch_pdl(tgp_attn_decode_group_kernel<DH_, 2>, grid, dim3(32 * split), sm, st, a, split); \
            else if (G == 4) launch_pdl(tgp_attn_decode_group_kernel<DH_, 4>, grid, dim3(32 * split), sm, st, a, split); \
            else launch_pdl(tgp_attn_decode_group_kernel<DH_, 8>, grid, dim3(32 * split), sm, st, a, split); } while (0)
        if (c->Dh == 64) {
            if (grouped) TGP_DECODE_GROUP(64); else launch_pdl(tgp_attn_decode_partial_kernel<64>, grid, dim3(32 * G * split), sm, st, a, split);
            launch_pdl(tgp_attn_decode_merge_kernel<64>, dim3(c->Hq, B), dim3(64), 0, st, a);
        } else {
            if (grouped) TGP_DECODE_GROUP(128); else launch_pdl(tgp_attn_decode_partial_kernel<128>, grid, dim3(32 * G * split), sm, st, a, split);
            launch_pdl(tgp_attn_decode_merge_kernel<128>, dim3(c->Hq, B), dim3(128), 0, st, a);
        }
#undef TGP_DECODE_GROUP
        tgpk_launches += 1;
    } else if (q_len >= 16 && (g_attn_impl == 0 || g_attn_impl == 2 || g_attn_impl == 3)) {
        // the tcgen05 kernel works on 128 queries per CTA (it hands geometries it cannot map with TMA to the mma.sync
        // kernel itself); below that the mma.sync kernel's 64-query CTAs waste less
        if (g_attn_impl == 3 || (g_attn_impl == 0 && q_len >= 128)) return tgpk_attn_prefill_tc5(qb, tiles, ob, c, B, q_len, pos0, st);
        return tgpk_attn_prefill_tc(qb, tiles, ob, c, B, q_len, pos0, st);
    } else {
        dim3 grid((q_len + 3) / 4, c->Hq, B);
        if (c->Dh == 64) tgp_attn_rows_kernel<64><<<grid, 128, 0, st>>>(a);
        else tgp_attn_rows_kernel<128><<<grid, 128, 0, st>>>(a);
    }
    LAUNCH_CHECK(1);
    return TGP_OK;
}

int tgpk_swiglu(const float *g, const float *u, void *ab, uint64_t n, cudaStream_t st) {
    if (!n) return TGP_OK;
    if (n % 4) return TGP_E_INVAL;
    uint64_t n4 = n / 4;
    uint32_t blocks = (uint32_t)((n4 + 255) / 256 < 148 * 16 ? (n4 + 255) / 256 : 148 * 16);
    launch_pdl(tgp_swiglu_kernel, dim3(blocks), dim3(256), 0, st, (const float4 *)g, (const float4 *)u, (__nv_bfloat162 *)ab, n4);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

int tgpk_argmax(const float *logits, int32_t *out, int32_t *out2, uint32_t B, uint32_t V, cudaStream_t st) {
    if (!B) return TGP_OK;
    // Rows of up to 8192 logits are two rounds of one CTA, faster than a cluster at any B (8192 x 1: 2.0 us, 2.3 in eight parts).  Longer ones
    // have eight parts, fewer where the CTAs are one and a half waves and more and a part would be short: the clusters' launches add up (us in
    // 1 / 2 / 4 / 8 parts: 32000 x 8 3.8 / 3.3 / 2.8 / 2.5, x 61 4.0 / 3.5 / 3.7 / 3.8, x 1024 24 / 25 / 26 / 34; 16384 x 256 4.2 / 4.7 / 5.6 / 8.5;
    // 128256 x 96 10.9 / 9.4 / 8.0 / 6.5)
    uint32_t parts = V > 8192 ? 8 : 1;
    while (parts > 1 && 2ull * B * parts > 3ull * (uint32_t)device_sms() && V / parts < 12288) parts /= 2;
    const int vec = V % 4 == 0 && (reinterpret_cast<uintptr_t>(logits) & 15u) == 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(B * parts); cfg.blockDim = dim3(256); cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = small_overlap();
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = parts; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, tgp_argmax_kernel, logits, out, out2, V, vec);
    LAUNCH_CHECK(1);
    return TGP_OK;
}

// ============================ C entry points ===========================================================
// The tiles of a call whose kernels access tiles first <= i < end <= n: those may not be NULL.
static int fill_tiles(TgpTilePtrs &t, void *const *k, void *const *v, uint32_t n, uint32_t first, uint32_t end) {
    if (n > TGP_MAX_TILES) return TGP_E_TOO_LARGE;
    if (!k || !v) return TGP_E_INVAL;
    for (uint32_t i = 0; i < n; ++i) {
        t.k[i] = k[i]; t.v[i] = v[i];
        if (i >= first && i < end && (!k[i] || !v[i])) return TGP_E_INVAL;
    }
    return TGP_OK;
}

extern "C" {

int tgp_k_embed(const void *table, const int32_t *tok_dev, float *x_dev, uint32_t M, uint32_t d, uint32_t V, void *stream) {
    if (!table || !tok_dev || !x_dev) return TGP_E_INVAL;
    return tgpk_embed(table, tok_dev, x_dev, M, d, V, (cudaStream_t)stream);
}

int tgp_k_embed_status(int *bad, uint32_t *row, int32_t *token) {
    if (!bad) return TGP_E_INVAL;
    unsigned long long w = 0;
    if (cudaMemcpyFromSymbol(&w, g_embed_error, sizeof(w)) != cudaSuccess) return TGP_E_CUDA;
    *bad = (w >> 63) ? 1 : 0;
    if (row) *row = (uint32_t)((w >> 32) & 0x7fffffffu);
    if (token) *token = (int32_t)(uint32_t)w;
    return TGP_OK;
}

int tgp_k_wait_test(uint64_t limit_ns, int withhold_step) {
    if (cudaDeviceSynchronize() != cudaSuccess) return TGP_E_CUDA;
    if (!limit_ns) { limit_ns = 2000000000ull; withhold_step = -1; }
    if (limit_ns < 100000ull || withhold_step < -1) return TGP_E_INVAL;
    int rc = tgpk_gemm_wait_test(limit_ns, withhold_step);
    return rc ? rc : tgpk_attn_wait_test(limit_ns, withhold_step);
}

int tgp_k_status_clear(void) {
    if (cudaDeviceSynchronize() != cudaSuccess) return TGP_E_CUDA;
    const unsigned long long z = 0;
    if (cudaMemcpyToSymbol(g_embed_error, &z, sizeof(z)) != cudaSuccess) return TGP_E_CUDA;
    int rc = tgpk_gemm_status_clear();
    return rc ? rc : tgpk_attn_status_clear();
}

int tgp_k_rmsnorm(const float *x_dev, uint32_t ldx, const void *g_dev, void *h_dev, uint32_t M, uint32_t d, float eps, void *stream) {
    if (!x_dev || !g_dev || !h_dev) return TGP_E_INVAL;
    return tgpk_rmsnorm(x_dev, ldx, g_dev, h_dev, M, d, eps, (cudaStream_t)stream);
}

int tgp_k_skinny_select(int impl) {
    if (impl != 0 && impl != 1) return TGP_E_INVAL;
    g_skinny_impl = impl;
    return TGP_OK;
}

int tgp_k_gemm_group(const void *A_dev, uint32_t count, const void *const *W_dev, float *const *C_dev, const uint32_t *n, const uint32_t *ldc,
                     uint32_t M, uint32_t K, int accumulate, void *stream) {
    if (!A_dev || !W_dev || !C_dev || !n || !ldc || !count || count > TGP_GEMM_GROUP_MAX || !K || K % 8) return TGP_E_INVAL;
    for (uint32_t s = 0; s < count; ++s) if (!W_dev[s] || !C_dev[s] || n[s] > ldc[s]) return TGP_E_INVAL;
    return tgpk_gemm_group(A_dev, count, W_dev, C_dev, n, ldc, M, K, accumulate, (cudaStream_t)stream);
}

int tgp_k_gemm_group_key(uint32_t M, uint32_t n, uint32_t K, uint32_t *key) {
    if (!key) return TGP_E_INVAL;
    *key = tgpk_gemm_group_key(M, n, K);
    return TGP_OK;
}

int tgp_k_gemm_last_kernel(char *name, uint32_t capacity) {
    if (!name || !capacity) return TGP_E_INVAL;
    const char *k = tgpk_last_gemm_kernel;
    uint32_t i = 0;
    for (; k[i] && i + 1 < capacity; ++i) name[i] = k[i];
    name[i] = 0;
    return TGP_OK;
}

int tgp_k_gemm_group_select(int enable) {
    g_gemm_group = enable ? 1 : 0;
    return TGP_OK;
}

int tgp_k_gemm_chain(int enable) {
    tgpk_chain_ok = enable != 0;
    g_chain.A = nullptr;
    return TGP_OK;
}

int tgp_k_gemv_overlap(int enable) {
    g_gemv_pdl = enable ? 1 : 0;
    g_small_pdl = enable ? 1 : 0;
    return TGP_OK;
}

int tgp_k_attn_decode_select(int impl) {
    if (impl < 0 || impl > 2) return TGP_E_INVAL;
    g_attn_decode_impl = impl;
    return TGP_OK;
}

int tgp_k_attn_select(int impl) {
    if (impl < 0 || impl > 3) return TGP_E_INVAL;
    g_attn_impl = impl;
    return TGP_OK;
}

int tgp_k_gemm_select(int impl) {
    if (impl != 0 && impl != 1) return TGP_E_INVAL;
    g_gemm_impl = impl;
    return TGP_OK;
}

int tgp_k_gemm(const void *A_dev, const void *W_dev, float *C_dev, uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate, void *stream) {
    if (!A_dev || !W_dev || !C_dev || col0 + (uint64_t)n > ldc) return TGP_E_INVAL;
    return tgpk_gemm(A_dev, W_dev, C_dev, M, n, K, ldc, col0, accumulate, (cudaStream_t)stream);
}

int tgp_k_rope_kv(const float *q32, const float *k32, const float *v32, void *qb, void *const *k_tiles, void *const *v_tiles, uint32_t n_tiles,
                  const float *cos_dev, const float *sin_dev, const tgp_model_cfg *cfg, uint32_t B, uint32_t q_len, uint32_t pos0, void *stream) {
    if (!q32 || !k32 || !v32 || !qb || !cfg || !cos_dev || !sin_dev) return TGP_E_INVAL;
    if ((uint64_t)pos0 + q_len > cfg->max_len || (uint64_t)n_tiles * cfg->TK < (uint64_t)pos0 + q_len || cfg->Dh % 2) return TGP_E_INVAL;
    TgpTilePtrs t;
    int rc = fill_tiles(t, k_tiles, v_tiles, n_tiles, cfg->TK ? pos0 / cfg->TK : 0, B && q_len ? (pos0 + q_len - 1) / cfg->TK + 1 : 0);
    if (rc) return rc;
    return tgpk_rope_kv(q32, k32, v32, qb, t, cos_dev, sin_dev, cfg, B, q_len, pos0, (cudaStream_t)stream);
}

int tgp_k_attn(const void *qb, void *const *k_tiles, void *const *v_tiles, uint32_t n_tiles, void *ob, const tgp_model_cfg *cfg, uint32_t B, uint32_t q_len,
               uint32_t pos0, float *scratch_dev, void *stream) {
    if (!qb || !ob || !cfg || !cfg->Hkv || cfg->Hq % cfg->Hkv) return TGP_E_INVAL;
    if ((uint64_t)n_tiles * cfg->TK < (uint64_t)pos0 + q_len) return TGP_E_INVAL;
    TgpTilePtrs t;
    int rc = fill_tiles(t, k_tiles, v_tiles, n_tiles, 0, B && q_len ? (pos0 + q_len - 1) / cfg->TK + 1 : 0);
    if (rc) return rc;
    return tgpk_attn(qb, t, n_tiles, ob, cfg, B, q_len, pos0, scratch_dev, (cudaStream_t)stream);
}

// ---- decode attention for callers that cannot allocate ------------------------------------------------
// The per-tile partials live in a fixed array inside the library image instead of caller memory.  In host
// code the array's name is only a handle; its device address is looked up once per device.
static __device__ __align__(256) float g_static_attn_scratch[TGP_STATIC_SCRATCH_BYTES / sizeof(float)];
static float *g_static_attn_scratch_addr[TGP_STATIC_MAX_DEVICES] = {};

int tgp_k_attn_decode_static(const void *qb, void *const *k_tiles, void *const *v_tiles, uint32_t n_tiles, void *ob,
                             const tgp_model_cfg *cfg, uint32_t B, uint32_t pos0, void *stream) {
    if (!qb || !ob || !cfg || !cfg->Hkv || cfg->Hq % cfg->Hkv || !cfg->TK || !B) return TGP_E_INVAL;
    if ((uint64_t)n_tiles * cfg->TK < (uint64_t)pos0 + 1) return TGP_E_INVAL;
    const uint64_t need = (uint64_t)B * cfg->Hq * n_tiles * (cfg->Dh + 2) * sizeof(float);
    if (need > TGP_STATIC_SCRATCH_BYTES) return TGP_E_TOO_LARGE;
    TgpTilePtrs t;
    int rc = fill_tiles(t, k_tiles, v_tiles, n_tiles, 0, pos0 / cfg->TK + 1);
    if (rc) return rc;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return TGP_E_CUDA;
    if (dev < 0 || dev >= TGP_STATIC_MAX_DEVICES) return TGP_E_TOO_LARGE;
    if (!g_static_attn_scratch_addr[dev]) {                       // first call on this device, with it current
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_attn_scratch) != cudaSuccess || !p) return TGP_E_CUDA;
        g_static_attn_scratch_addr[dev] = (float *)p;
    }
    return tgpk_attn(qb, t, n_tiles, ob, cfg, B, 1, pos0, g_static_attn_scratch_addr[dev], (cudaStream_t)stream);
}

int tgp_k_attn_scratch_bytes(const tgp_model_cfg *cfg, uint64_t *bytes) {
    if (!cfg || !bytes || !cfg->TK) return TGP_E_INVAL;
    uint64_t nt = (cfg->max_len + cfg->TK - 1) / cfg->TK;
    *bytes = (uint64_t)cfg->B * cfg->Hq * nt * (cfg->Dh + 2) * sizeof(float);
    return TGP_OK;
}

int tgp_k_swiglu(const float *g32, const float *u32, void *ab, uint64_t n_elems, void *stream) {
    if (!g32 || !u32 || !ab) return TGP_E_INVAL;
    return tgpk_swiglu(g32, u32, ab, n_elems, (cudaStream_t)stream);
}

int tgp_k_argmax(const float *logits, int32_t *out, uint32_t B, uint32_t V, void *stream) {
    if (!logits || !out || !V) return TGP_E_INVAL;
    return tgpk_argmax(logits, out, nullptr, B, V, (cudaStream_t)stream);
}

}  // extern "C"
