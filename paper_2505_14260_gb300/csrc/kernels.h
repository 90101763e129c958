// Host-side launchers of the MSD kernels. Every launcher enqueues on `s` and
// returns without synchronising.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

#include "common.cuh"

namespace msd {

// ---- elementwise / row kernels (kernels_rows.cu) ---------------------------

// x[r] = float(src[r] >= 0 ? E[src[r]] : vis[-1 - src[r]]), xn[r] = its RMSNorm
// with gain g, split (lo plane at xn + lo)
template <typename T>
void launch_embed_norm(const T *E, const T *vis, const int *src, const T *g, int R, int H, float eps, float *x, T *xn,
                       long lo, int V, int *status, cudaStream_t s);

// out[r] = x[r] / sqrt(mean(x[r]^2) + eps) * g, split (lo plane at out + lo)
template <typename T>
void launch_rmsnorm(const float *x, const T *g, int R, int H, float eps, T *out, long lo,
                    cudaStream_t s);

// act[r][j] = silu(g) * u with g = gu[r][j], u = gu[r][F + j] (fp32 contexts)
void launch_swiglu(const float *gu, int R, int F, float *act, cudaStream_t s);

// RoPE (rotate-half, table of (cos, sin) per position and pair) on q and k of
// qkv [R][3H]; q -> q_out [R][H]; k, v -> kdst/vdst at slot rows[r].dst of
// request rows[r].req: [B][nh][slots][hd]; all outputs split (lo planes at +lo).
template <typename T>
void launch_rope_kv(const float *qkv, const RowDesc *rows, int R, int nh, int hd,
                    const float2 *rope_tab, int max_pos, T *q_out, T *kdst,
                    T *vdst, int slots, long lo, int *status, cudaStream_t s);

// Row r attends to cache[req][h][0 .. plen) and to the tree slots j of
// request req with bit j of mask[r] set.
template <typename T>
struct AttnArgs {
    const T *q;                 // [R][nh*hd]
    const RowDesc *rows;
    int R;
    const T *cache_k, *cache_v; // [B][nh][cache_slots][hd]
    int cache_slots;
    const T *tree_k, *tree_v;   // [B][nh][tree_slots][hd] (nullable)
    int tree_slots;
    const uint64_t *mask;       // [R][mask_words] (nullable = no tree part)
    int mask_words;
    int nh, hd;
    float scale;
    T *out;                     // [R][nh*hd]
    // row tiles of a packed prefill chunk (first row, rows <= 64 of one request),
    // longest prefix first; null: blocks of rows_per_req rows of one request
    const int2 *tiles;
    int n_tiles;
    bool cache_fresh;           // the kernel launched just before may have written cache_k/v
    long lo;                    // split bf16: lo planes of q, K/V and out sit lo elements on (0: none)
};
// fp32 contexts (CUDA cores); rows come in blocks of rows_per_req rows of one
// request. Returns false if the shape is unsupported or the launch failed.
// attention_setup sets the kernels' shared-memory limits on the current device,
// once before its first launch.
bool attention_setup();
bool launch_attention(const AttnArgs<float> &a, int rows_per_req, int num_sms, cudaStream_t s);

// Scratch of the chunked top-k: per-chunk records and per-row tickets
// (tickets must start at zero; the kernel leaves them at zero).
struct TopkScratch {
    float *ws;
    int *counters;
};
size_t topk_scratch_floats(int max_rows, int V);

// out[r] = argmax_j logits[r][j] (ties: lower j)
void launch_argmax(const float *logits, int R, int V, int *out, cudaStream_t s);

// Top-k of each row (ties: lower id) and their log-softmax values (logp
// nullable). k <= 16.
void launch_topk_logp(const float *logits, int R, int V, int k, int *ids, float *logp,
                      const TopkScratch &sc, cudaStream_t s);
// Whether the top-k kernel takes vocabulary V with k <= 16 (ceil(V / 4096) * k
// candidates <= 256 in its row merge).
bool topk_supported(int V, int k);

// Sets the device status word (first code wins), in stream order.
void launch_flag(int *status, int code, cudaStream_t s);

// ---- GEMM ------------------------------------------------------------------

// Y[m][o] (=|+=) sum_k X[m][k] * W[o][k], with W given as up to three row
// segments stacked along o (e.g. wq;wk;wv).
struct GemmW {
    const void *w[3];
    int rows[3];
    int nseg;
    const void *packed;   // the same weights pre-packed by gemm_pack (bf16), or null
};
enum { EPI_STORE = 0, EPI_ADD = 1, EPI_SWIGLU = 2, EPI_ROPE_KV = 3 };

// fp32 contexts (CUDA cores); gemm_simt_setup as attention_setup
bool gemm_simt_setup();
void launch_gemm_simt(const float *X, int ldx, int M, int K, const GemmW &W, int O, float *Y, int ldy, int epi,
                      int num_sms, cudaStream_t s);

}  // namespace msd
