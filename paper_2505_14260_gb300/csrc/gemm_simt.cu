// CUDA-core GEMM for the fp32 model dtype: Y[m][o] (=|+=) sum_k X[m][k] W[o][k].
//
// What bounds it: the weights' bytes at decode row counts (a 1024 x 2816 fp32
// matrix is 11.5 MB: 1.7 us of HBM), fp32 FMAs at prefill row counts. Both
// operands are K-contiguous, so shared memory holds plain [row][64 k] tiles,
// filled by cp.async (16 bytes where rows are 16-byte aligned, 4 otherwise)
// three or four stages ahead, and a thread reads four consecutive k of a row
// at once: packed fp32 FMAs (f32x2) keep the even-k and the odd-k sums of each
// output in one 64-bit register, added at the end. Rows are padded to 68
// floats, so the 8 rows a warp reads together sit in different banks.
// Tiles of 32 outputs x 8 token rows to 128 x 128, always 256 threads: the
// smaller the tile, the more warps share it by taking different k of a stage
// (their sums meet in shared memory). K may be split over the CTAs of a cluster
// (at most 8), whose partial tiles are summed through distributed shared memory
// in rank order. Every order is fixed by the
// launch's shape, so results are reproducible and an output depends only on
// its own row of X.
#include <cooperative_groups.h>

#include <algorithm>
#include <iterator>

#include "kernels.h"

namespace msd {

namespace {

namespace cg = cooperative_groups;

constexpr int SG_BK = 64;                 // k per stage
constexpr int SG_LD = SG_BK + 4;          // padded row (floats): 17 16-byte chunks
constexpr int SG_THREADS = 256;

__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b,
                                                   unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ float pair_sum(unsigned long long v) {
    return __uint_as_float((unsigned)v) + __uint_as_float((unsigned)(v >> 32));
}

// n source bytes copied (0: zero fill) to a 16-byte / 4-byte shared location
__device__ __forceinline__ void cp16(uint32_t dst, const float *src, int n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp4(uint32_t dst, const float *src, int n) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// BO x BM outputs per CTA; a thread holds TO x TM of them; KS groups of warps
// take different k of every stage.
template <int BO_, int BM_, int TO_, int TM_, int STAGES_>
struct Tile {
    static constexpr int BO = BO_, BM = BM_, TO = TO_, TM = TM_, STAGES = STAGES_;
    static constexpr int GROUP = (BO / TO) * (BM / TM);
    static constexpr int KS = SG_THREADS / GROUP;
    static constexpr int STAGE = (BO + BM) * SG_LD;                        // floats
    static constexpr int SMEM = STAGES * STAGE * 4;
    static_assert(GROUP % 32 == 0 && (SG_BK / 4) % KS == 0, "whole warps, whole 4-k chunks");
    static_assert(KS * BO * BM <= STAGES * STAGE, "the k groups' partial tiles reuse the ring");
};

struct SgArgs {
    const float *X;
    int ldx, M, K;
    const float *w0, *w1, *w2;      // row segments of W, stacked
    int e0, e1;                     // end rows of the first two
    int O;
    float *Y;
    int ldy, epi, splits;
};

template <class TL, bool VEC>
__global__ void __launch_bounds__(SG_THREADS) gemm_simt_kernel(const SgArgs a) {
    extern __shared__ __align__(16) float sm[];
    wait_prior();
    allow_dependents();
    const int tid = threadIdx.x;
    const int o0 = blockIdx.x * TL::BO, m0 = blockIdx.y * TL::BM, split = blockIdx.z;
    const int nb = (a.K + SG_BK - 1) / SG_BK;                     // k blocks
    const int b0 = (int)((long long)split * nb / a.splits), b1 = (int)((long long)(split + 1) * nb / a.splits);

    // the rows this thread copies: 16 threads per row of a stage
    constexpr int RO = TL::BO / 16, RM = (TL::BM + 15) / 16;    // (8- and 24-row tiles: half of the last pass is idle)
    const int crow = tid >> 4, cq = (tid & 15) * 4;
    const float *src[RO + RM];
#pragma unroll
    for (int i = 0; i < RO; ++i) {
        const int o = o0 + crow + 16 * i;
        src[i] = o >= a.O ? nullptr
                          : (o < a.e0 ? a.w0 + (size_t)o * a.K
                                      : (o < a.e1 ? a.w1 + (size_t)(o - a.e0) * a.K
                                                  : a.w2 + (size_t)(o - a.e1) * a.K));
    }
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        const int m = m0 + crow + 16 * i;
        src[RO + i] = m < a.M && crow + 16 * i < TL::BM ? a.X + (size_t)m * a.ldx : nullptr;
    }
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(sm) + (uint32_t)(crow * SG_LD + cq) * 4u;
    auto load = [&](int blk, int st) {
        const int k = blk * SG_BK + cq;
#pragma unroll
        for (int i = 0; i < RO + RM; ++i) {
            if (TL::BM % 16 && i == RO + RM - 1 && crow + 16 * (RM - 1) >= TL::BM) break;
            const uint32_t d = s0 + (uint32_t)(st * TL::STAGE + 16 * i * SG_LD) * 4u;
            const float *p = src[i];
            if constexpr (VEC) {                  // K % 4 == 0: whole chunks
                const bool in = p && k < a.K;
                cp16(d, in ? p + k : a.X, in ? 16 : 0);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool in = p && k + e < a.K;
                    cp4(d + 4 * e, in ? p + k + e : a.X, in ? 4 : 0);
                }
            }
        }
    };

    // thread of a group: lanes run 8 outputs (lane bits 0, 2, 3) x 4 tokens (bits 1, 4),
    // warps tile the rest. Lanes i and i ^ 2 then read the same W, lanes i and i ^ 1 the
    // same X, so that a 16-byte load serves more lanes at a time (24 x 32000 x 1024: 72.8
    // us with bits 0-2 and 3-4, 66.9; 24 x 5632 x 1024: 23.6 and 22.0)
    const int grp = tid / TL::GROUP, t = tid % TL::GROUP, w = t >> 5, lane = t & 31;
    constexpr int WO = TL::BO / (8 * TL::TO);     // warps along the outputs
    const int to = (w % WO) * 8 + ((lane & 1) | (lane >> 1 & 6)), tm = (w / WO) * 4 + ((lane >> 1 & 1) | (lane >> 3 & 2));
    constexpr int SO = TL::BO / TL::TO, SM_ = TL::BM / TL::TM;   // strides between a thread's outputs / tokens
    unsigned long long acc[TL::TO][TL::TM] = {};

    const int n = b1 - b0;
#pragma unroll
    for (int s = 0; s < TL::STAGES - 1; ++s) {
        if (s < n) load(b0 + s, s);
        cp_commit();
    }
    for (int i = 0; i < n; ++i) {
        cp_wait<TL::STAGES - 2>();
        __syncthreads();
        if (i + TL::STAGES - 1 < n) load(b0 + i + TL::STAGES - 1, (i + TL::STAGES - 1) % TL::STAGES);
        cp_commit();
        const float *ws = sm + (i % TL::STAGES) * TL::STAGE, *xs = ws + TL::BO * SG_LD;
        constexpr int CH = SG_BK / 4 / TL::KS;    // 4-k chunks of this group
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int q = (grp * CH + c) * 4;
            ulonglong2 wv[TL::TO], xv[TL::TM];
#pragma unroll
            for (int u = 0; u < TL::TO; ++u)
                wv[u] = *reinterpret_cast<const ulonglong2 *>(ws + (to + u * SO) * SG_LD + q);
#pragma unroll
            for (int u = 0; u < TL::TM; ++u)
                xv[u] = *reinterpret_cast<const ulonglong2 *>(xs + (tm + u * SM_) * SG_LD + q);
#pragma unroll
            for (int u = 0; u < TL::TO; ++u)
#pragma unroll
                for (int v = 0; v < TL::TM; ++v)
                    acc[u][v] = fma2(wv[u].y, xv[v].y, fma2(wv[u].x, xv[v].x, acc[u][v]));
        }
    }
    cp_wait<0>();
    __syncthreads();

    // the groups' sums as [KS][BM][BO] in the idle ring, then added in group order
#pragma unroll
    for (int u = 0; u < TL::TO; ++u)
#pragma unroll
        for (int v = 0; v < TL::TM; ++v)
            sm[(grp * TL::BM + tm + v * SM_) * TL::BO + to + u * SO] = pair_sum(acc[u][v]);
    __syncthreads();
    constexpr int TILE = TL::BO * TL::BM;
    auto put = [&](int e, float v) {
        const int m = m0 + e / TL::BO, o = o0 + e % TL::BO;
        if (m >= a.M || o >= a.O) return;
        float *y = a.Y + (size_t)m * a.ldy + o;
        *y = a.epi == EPI_ADD ? *y + v : v;
    };
    for (int e = tid; e < TILE; e += SG_THREADS) {
        float v = sm[e];
#pragma unroll
        for (int g = 1; g < TL::KS; ++g) v += sm[g * TILE + e];
        if (a.splits == 1) put(e, v);
        else sm[e] = v;                           // (each thread rewrites only places it alone reads)
    }
    if (a.splits == 1) return;
    // K split over the cluster: rank r adds its share of the tile over all ranks
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int S = a.splits, r = (int)cl.block_rank();
    const int lo = r * (TILE / 32) / S * 32, hi = (r + 1) * (TILE / 32) / S * 32;
    for (int e = lo + tid; e < hi; e += SG_THREADS) {
        float p[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < S) p[q] = cl.map_shared_rank(sm, q)[e];
        float v = p[0];
#pragma unroll
        for (int q = 1; q < 8; ++q)
            if (q < S) v += p[q];
        put(e, v);
    }
    cl.sync();                                    // partials stay readable until all ranks are done
}

template <class TL, bool VEC>
void launch_tile(SgArgs a, int S, cudaStream_t s) {
    const int to = (a.O + TL::BO - 1) / TL::BO, tm = (a.M + TL::BM - 1) / TL::BM;
    a.splits = S;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)to, (unsigned)tm, (unsigned)S);
    lc.blockDim = dim3(SG_THREADS);
    lc.dynamicSmemBytes = TL::SMEM;
    lc.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = (unsigned)S;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = programmatic(s) ? 2 : 1;
    cudaLaunchKernelEx(&lc, gemm_simt_kernel<TL, VEC>, (const SgArgs)a);
    note_launch();
}

template <class TL>
bool set_tile() {
    return cudaFuncSetAttribute(gemm_simt_kernel<TL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TL::SMEM) ==
               cudaSuccess &&
           cudaFuncSetAttribute(gemm_simt_kernel<TL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TL::SMEM) ==
               cudaSuccess;
}

// The tiles, with the time of one k block of a tile, its start and end, and what a
// K split's exchange adds (ns, when every SM holds as many as fit).
struct TileRow {
    int BO, BM;
    double block_ns, tile_ns, split_ns;
    void (*launch[2])(SgArgs, int, cudaStream_t);     // [16-byte aligned rows]
    bool (*setup)();
};
template <class TL>
constexpr TileRow tile_row(double block_ns, double tile_ns, double split_ns) {
    return {TL::BO, TL::BM, block_ns, tile_ns, split_ns, {launch_tile<TL, false>, launch_tile<TL, true>}, set_tile<TL>};
}
const TileRow TILES[] = {
    tile_row<Tile<32, 8, 4, 2, 4>>(200, 200, 1500),
    tile_row<Tile<32, 16, 4, 4, 4>>(300, 200, 1500),
    tile_row<Tile<32, 24, 4, 3, 4>>(430, 200, 1500),
    tile_row<Tile<32, 32, 4, 4, 4>>(595, 200, 1500),
    tile_row<Tile<128, 64, 8, 8, 3>>(3450, 800, 10000),
    tile_row<Tile<128, 128, 8, 8, 3>>(6150, 800, 10000),
};

}  // namespace

bool gemm_simt_setup() {
    for (const TileRow &t : TILES)
        if (!t.setup()) return false;
    return true;
}

void launch_gemm_simt(const float *X, int ldx, int M, int K, const GemmW &W, int O, float *Y, int ldy, int epi,
                      int num_sms, cudaStream_t s) {
    if (M <= 0 || O <= 0) return;
    SgArgs a;
    a.X = X; a.ldx = ldx; a.M = M; a.K = K;
    const float *w[3];
    for (int i = 0; i < 3; ++i) w[i] = static_cast<const float *>(W.w[i < W.nseg ? i : 0]);
    a.w0 = w[0]; a.w1 = w[1]; a.w2 = w[2];
    a.e0 = W.nseg > 1 ? W.rows[0] : O;
    a.e1 = W.nseg > 2 ? W.rows[0] + W.rows[1] : O;
    a.O = O; a.Y = Y; a.ldy = ldy; a.epi = epi; a.splits = 1;
    uintptr_t bits = reinterpret_cast<uintptr_t>(X);
    for (int i = 0; i < W.nseg; ++i) bits |= reinterpret_cast<uintptr_t>(w[i]);
    const bool vec = (bits & 15) == 0 && K % 4 == 0 && ldx % 4 == 0;
    // The tile and the K splits whose rounds over the SMs take least. Small tiles leave
    // the least of the chip idle, large ones make the most of a shared-memory load (us, in
    // 32 x 24, 32 x 32, 128 x 64 and 128 x 128 tiles: 24 x 32000 x 1024 50, 67, -, -; 100 x
    // 5632 x 1024 43, 49, 56, 99; 341 x 5632 x 1024 120, 121, 110, 99; 341 x 1024 x 2816
    // 74, 78, 146, 262, and 69 in two splits of 32 x 24). One small tile on a SM hides
    // less of its latency. Over 30 shapes the choice is within 1% of the best on average,
    // 14% at most; splits of three ran up to half a round longer than of two or four.
    const int nb = (K + SG_BK - 1) / SG_BK;
    const TileRow *best = nullptr;
    int S = 1;
    double best_ns = 0;
    for (const TileRow &t : TILES) {
        if (t.BM < 24 && M > 4 * t.BM) continue;
        const long row_tiles = (M + t.BM - 1) / t.BM, tiles = (O + t.BO - 1) / t.BO * row_tiles;
        // (the grid's y; rows past the last, largest tile's 65535 are refused by the launch)
        if (row_tiles > 65535 && &t != &TILES[std::size(TILES) - 1]) continue;
        for (int sp = 1; sp <= 8 && (sp == 1 || sp <= nb / 2); sp *= 2) {
            const long rounds = (tiles * sp + num_sms - 1) / num_sms;
            double ns = rounds * (t.block_ns * ((nb + sp - 1) / sp) + t.tile_ns);
            if (rounds == 1 && t.BM < 64) ns *= 1.25;
            if (sp > 1) ns += rounds * t.split_ns;
            if (!best || ns < best_ns) {
                best = &t;
                best_ns = ns;
                S = sp;
            }
        }
    }
    best->launch[vec](a, S, s);
}

}  // namespace msd
