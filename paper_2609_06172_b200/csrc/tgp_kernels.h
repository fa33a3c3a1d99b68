// Internal launch interface between the step engine and the kernels.
#pragma once
#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>
#include "tgp.h"

#define TGP_MAX_TILES 64      // KV tiles per layer a kernel can address (pointer table passed by value)

// Function attributes and the number of SMs are a device's own, and a process may use several: what is kept of them is kept by device.
#define TGP_DEVICES 64        // of these; further ones ask every time
inline int tgpk_device() { int dev = 0; return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < TGP_DEVICES ? dev : -1; }
int tgpk_sms();               // SMs of the current device

// Dynamic shared memory above 48 KB for a kernel on the current device; `shared_first` also asks for the split of L1 and shared memory that leaves it all to the latter (a hint).
template <auto KERNEL>
inline bool tgpk_allow_smem(size_t bytes, bool shared_first = false) {
    static std::atomic<uint64_t> allowed{0};                  // a bit per device
    const int dev = tgpk_device();
    const uint64_t bit = dev < 0 ? 0 : 1ull << dev;
    if (bit & allowed.load(std::memory_order_relaxed)) return true;
    if (cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return false;
    if (shared_first && cudaFuncSetAttribute(KERNEL, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess) cudaGetLastError();
    allowed.fetch_or(bit, std::memory_order_relaxed);
    return true;
}

struct TgpTilePtrs { void *k[TGP_MAX_TILES]; void *v[TGP_MAX_TILES]; };

// rows of token ids outside [0, V) are written as zeros and recorded (tgp_k_embed_status)
int tgpk_embed(const void *table, const int32_t *tok, float *x, uint32_t M, uint32_t d, uint32_t V, cudaStream_t st);
int tgpk_rmsnorm(const float *x, uint32_t ldx, const void *g, void *h, uint32_t M, uint32_t d, float eps, cudaStream_t st);
int tgpk_gemm(const void *A, const void *W, float *C, uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate, cudaStream_t st);
// products over the same activations A [M, K]: C[s][m, j] (=|+=) sum_k A[m, k] * W[s][j, k].  Neighbours with the same non-zero
// tgpk_gemm_group_key() are served by one launch (up to TGP_GEMM_GROUP_MAX of them), anything else by one launch per part;
// the bits are the same either way
uint32_t tgpk_gemm_group_key(uint32_t M, uint32_t n, uint32_t K);
int tgpk_gemm_group(const void *A, uint32_t count, const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t M, uint32_t K,
                    int accumulate, cudaStream_t st);
// tcgen05 path (tgp_gemm_sm100.cu): any M, n; K % 8 == 0; A and W 16-byte aligned
// gate / aout (both or neither): the accumulator is the up projection of a SwiGLU FFN; instead of storing it to C the epilogue
// stores aout[m, col0 + j] = bf16(silu(gate[m, col0 + j]) * acc) (gate fp32 and aout bf16 in C's geometry); not with accumulate
int tgpk_gemm_tc(const void *A, const void *W, float *C, uint32_t M, uint32_t n, uint32_t K, uint32_t ldc, uint32_t col0, int accumulate, cudaStream_t st,
                 const float *gate = nullptr, void *aout = nullptr);
// blocks over the same activations in one launch of a tcgen05 kernel (gate / aout with one block only); all of them must
// have the same tgpk_gemm_tc_class() (kernel and split of K, never 0), then each computes the bits it computes alone
uint32_t tgpk_gemm_tc_class(uint32_t M, uint32_t n, uint32_t K);
int tgpk_gemm_tc_list(const void *A, uint32_t count, const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t M, uint32_t K,
                      int accumulate, cudaStream_t st, const float *gate = nullptr, void *aout = nullptr);
// a kernel other than the automatic choice is selected (tgp_k_gemm_tc_variant)
bool tgpk_gemm_tc_forced();
// programmatic dependent launches are switched on (tgp_k_gemv_overlap)
extern thread_local bool tgpk_whole_edge;      // (and this thread has not set them aside for its next launches)
bool tgpk_launch_overlap();
// true if a product of M activation rows takes the tensor-core GEMM, whose epilogue can apply SwiGLU (M > 128, tensor cores selected)
bool tgpk_swiglu_fusable(uint32_t M);
int tgpk_rope_kv(const float *q32, const float *k32, const float *v32, void *qb, const TgpTilePtrs &tiles, const float *cos_t, const float *sin_t,
                 const tgp_model_cfg *c, uint32_t B, uint32_t q_len, uint32_t pos0, cudaStream_t st);
// what a decode step's attention needs to rotate for itself: the fp32 projections of its new position and the tables
struct TgpRopeIn { const float *q32, *k32, *v32, *cos_t, *sin_t; };
int tgpk_attn(const void *qb, const TgpTilePtrs &tiles, uint32_t n_tiles, void *ob, const tgp_model_cfg *c, uint32_t B, uint32_t q_len, uint32_t pos0,
              float *scratch, cudaStream_t st, const TgpRopeIn *rope = nullptr);
// tcgen05 causal attention for q_len > 1 (tgp_attn_sm100.cu); Dh 64 or 128
int tgpk_attn_prefill_tc5(const void *qb, const TgpTilePtrs &tiles, void *ob, const tgp_model_cfg *c, uint32_t B, uint32_t q_len, uint32_t pos0, cudaStream_t st);
// mma.sync flash-style causal attention for q_len > 1 (tgp_attn_prefill.cu); Dh 64 or 128
int tgpk_attn_prefill_tc(const void *qb, const TgpTilePtrs &tiles, void *ob, const tgp_model_cfg *c, uint32_t B, uint32_t q_len, uint32_t pos0, cudaStream_t st);
int tgpk_swiglu(const float *g, const float *u, void *ab, uint64_t n, cudaStream_t st);
// MoE: router logits + top-k (1 or 2) + gates, then per-expert token lists rows[e*stride + i], gates[e*stride + i], counts[e].  Up to 64
// tokens: one launch, which also writes pos[2 m + s] (place of token m in the list of its s-th expert) and, if given, the
// counts to mapped host memory
int tgpk_router(const void *h, const void *Wr, const float *bias, int32_t *idx, float *gate, int32_t *rows, float *gates, int32_t *counts, int32_t *pos,
                int32_t *counts_host, uint32_t M, uint32_t stride, uint32_t d, uint32_t E, uint32_t topk, cudaStream_t st);
// all experts of a layer for a step of 3 to 32 tokens, from the router's lists on the device: a = SwiGLU of the gate and up
// projections of the routed rows of h (one row per slot), y = their down projections, x += gate * y.  w[0..2]: gate, up, down of
// each expert in blocks of per_f (gate, up) or per_d (down) rows.  Bit-identical to the experts one by one (tgpk_gemm_rows)
#define TGP_MOE_EXPERTS 16
#define TGP_MOE_BLOCKS 4
struct TgpExperts {
    const void *w[3][TGP_MOE_EXPERTS][TGP_MOE_BLOCKS], *h;
    void *a; float *y, *x;
    const int32_t *rows, *counts, *idx, *pos; const float *gate;
    uint32_t E, topk, M, d, F, per_f, per_d, stride;
};
int tgpk_experts(const TgpExperts &x, cudaStream_t st);
bool tgpk_expert_rows(uint32_t M, uint32_t K);
int tgpk_gemm_rows(const void *A, uint32_t count, const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t me, uint32_t K, cudaStream_t st);
// products over the same activations may share a launch (tgp_k_gemm_group_select)
bool tgpk_gemm_grouping();
// gate, up and SwiGLU of at most two rows in one launch, blocks of gate and of up with the same rows (bit-identical to the separate launches)
bool tgpk_glu_rows_ok(uint32_t M, uint32_t n, uint32_t K);
int tgpk_glu_rows(const void *A, uint32_t count, const void *const *gate, const void *const *up, const uint32_t *n, void *out, uint32_t M, uint32_t K, cudaStream_t st);
int tgpk_gather_rows(const void *src, const int32_t *rows, void *dst, uint32_t m, uint32_t d, cudaStream_t st);
int tgpk_scatter_add(float *x, const float *y, const int32_t *rows, const float *gates, uint32_t m, uint32_t d, cudaStream_t st);
// the result also goes to out2 if that is not NULL
int tgpk_argmax(const float *logits, int32_t *out, int32_t *out2, uint32_t B, uint32_t V, cudaStream_t st);
// cos/sin tables [max_len, Dh/2] fp32 (angle = pos * base^(-2i/Dh), evaluated in double) written to device memory
int tgp_rope_tables_upload(uint32_t Dh, uint32_t max_len, float base, float *cos_dev, float *sin_dev);
// reset of the tensor-core kernels' error words (tgp_gemm_sm100.cu, tgp_attn_sm100.cu)
int tgpk_gemm_status_clear();
int tgpk_attn_status_clear();
// name of the kernel the last tgpk_gemm / tgpk_gemm_group / tgpk_gemm_tc call of this thread launched
extern thread_local const char *tgpk_last_gemm_kernel;
// set while the caller vouches that this thread's kernel launches are all that is enqueued on their streams (see tgp_k_gemm_chain)
extern thread_local bool tgpk_chain_ok;
// test hooks of the tensor-core kernels' bounded waits (see tgp_k_wait_test)
int tgpk_gemm_wait_test(unsigned long long limit_ns, int withhold_step);
int tgpk_attn_wait_test(unsigned long long limit_ns, int withhold_step);
// products of M <= 2 rows with the activations computed on the fly: mode 1 the RMSNorm of x (row stride ldx, gain, eps),
// mode 2 SwiGLU of (g32, u32); bit-identical to the separate kernels followed by tgpk_gemm_group()
int tgpk_gemm_group_fused(int mode, const float *x, uint32_t ldx, const void *gain, float eps, const float *g32, const float *u32, uint32_t count,
                          const void *const *W, float *const *C, const uint32_t *n, const uint32_t *ldc, uint32_t M, uint32_t K, int accumulate, cudaStream_t st);
