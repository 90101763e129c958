// Tree-masked attention on CUDA cores (the fp32 path; bf16 contexts run
// attn_tc.cu for every pass). Visible keys of a row: the cache prefix
// [0, plen) of its request, then the tree slots whose bit is set in its mask
// (Sec. 3.2: a candidate sees its prefix only).
//
// What bounds it: latency and fp32 FMAs. A CTA takes a tile of rows of one
// request and one head (16 rows where a block of rows is that small, as in
// decode; 64 otherwise) and walks its keys in tiles of 64, copied by cp.async
// into a two-stage ring: scores S = Q K^T as register tiles (packed fp32 FMAs
// over even and odd elements), an online softmax over the tile in shared
// memory, O += P V in registers. A key that a row does not see takes no part in
// that row's sums: its weight is -0, and in a tile whose V holds a NaN or an
// infinity (of another row, or of an earlier tree in a slot not written yet) it is
// skipped. When the (row tile, head) CTAs leave SMs idle the keys are cut into
// splits of whole tiles, one cluster per (row tile, head), combined through
// distributed shared memory in split order; the last split takes the tree keys.
// Rows are padded to HD + 4 floats, so the rows a warp reads together sit in
// different banks.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "kernels.h"

namespace msd {

namespace {

namespace cg = cooperative_groups;

constexpr int AS_THREADS = 256;
constexpr int AS_KT = 64;               // keys per tile
constexpr int AS_PLD = AS_KT + 4;       // padded score row
constexpr int AS_MAX_SPLITS = 8;
constexpr float HIDDEN = -0.f;          // weight of a key that the row does not see (of one that it sees: +0 or more)

struct AsArgs {
    AttnArgs<float> a;
    int rows_per_req, tiles_per_req, nsplit;
    float scale_log2;
};

__device__ __forceinline__ unsigned long long as_fma2(unsigned long long a, unsigned long long b,
                                                      unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long as_pack(float x, float y) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ float as_lo(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float as_hi(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }

__device__ __forceinline__ float as_exp2(float x) {      // 2^-inf = 0
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int HD, int QR>
struct AsLay {
    static constexpr int LD = HD + 4;
    static constexpr int Q = 0;                                 // [QR][LD]
    static constexpr int KV = Q + QR * LD;                      // 2 stages of K [64][LD], V [64][LD]
    static constexpr int P = KV + 4 * AS_KT * LD;               // [QR][AS_PLD]
    static constexpr int ST = P + QR * AS_PLD;                  // per row: scale, max, sum
    static constexpr int FLOATS = ST + 3 * QR;
    static constexpr int SMEM = FLOATS * 4;
};

template <int HD, int QR>
__global__ void __launch_bounds__(AS_THREADS) attn_simt_kernel(const AsArgs p) {
    using L = AsLay<HD, QR>;
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_live, s_least;         // longest and shortest prefix of the rows
    wait_prior();
    allow_dependents();
    const AttnArgs<float> &a = p.a;
    const int tid = threadIdx.x;
    const int h = blockIdx.x, split = blockIdx.z;
    int r0, nrows;
    if (a.tiles) {
        const int2 t = a.tiles[blockIdx.y];
        r0 = t.x;
        nrows = t.y;
    } else {
        const int blk = blockIdx.y / p.tiles_per_req;
        r0 = blk * p.rows_per_req + (blockIdx.y - blk * p.tiles_per_req) * QR;
        nrows = min(r0 + QR, (blk + 1) * p.rows_per_req) - r0;
    }
    const int H = a.nh * HD;
    const int req = a.rows[r0].req;

    // query rows (zero past the tile's end), the rows' prefix lengths
    if (tid == 0) {
        s_live = 0;
        s_least = 0x7fffffff;
    }
    __syncthreads();
    float *sQ = sm + L::Q, *sP = sm + L::P, *s_scale = sm + L::ST, *s_m = s_scale + QR, *s_l = s_m + QR;
    for (int e = tid; e < QR * (HD / 4); e += AS_THREADS) {
        const int r = e / (HD / 4), c = (e - r * (HD / 4)) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < nrows) v = *reinterpret_cast<const float4 *>(a.q + (size_t)(r0 + r) * H + h * HD + c);
        *reinterpret_cast<float4 *>(sQ + r * L::LD + c) = v;
    }
    if (tid < nrows) {
        const int plen = a.rows[r0 + tid].plen;
        atomicMax(&s_live, plen);
        atomicMin(&s_least, plen);
    }
    if (tid < QR) {
        s_m[tid] = -INFINITY;
        s_l[tid] = 0.f;
    }
    __syncthreads();
    const int live = min(s_live, a.cache_slots), least = s_least;
    const int per = ((live + AS_KT - 1) / AS_KT + p.nsplit - 1) / p.nsplit * AS_KT;
    const int k_lo = split * per, k_hi = min(k_lo + per, live);
    const int nc = k_hi > k_lo ? (k_hi - k_lo + AS_KT - 1) / AS_KT : 0;
    const int ntree = a.mask && split == p.nsplit - 1 ? (a.tree_slots + AS_KT - 1) / AS_KT : 0;
    const int nt = nc + ntree;
    const size_t cbase = (size_t)(req * a.nh + h) * a.cache_slots * HD;
    const size_t tbase = (size_t)(req * a.nh + h) * a.tree_slots * HD;

    auto load = [&](int i) {
        const bool cache = i < nc;
        const int key0 = cache ? k_lo + i * AS_KT : (i - nc) * AS_KT;
        const int lim = cache ? k_hi : a.tree_slots;
        const float *K = cache ? a.cache_k + cbase : a.tree_k + tbase;
        const float *V = cache ? a.cache_v + cbase : a.tree_v + tbase;
        float *dk = sm + L::KV + (i & 1) * 2 * AS_KT * L::LD;
#pragma unroll
        for (int e = tid; e < AS_KT * (HD / 4); e += AS_THREADS) {
            const int r = e / (HD / 4), c = (e - r * (HD / 4)) * 4;
            const bool in = key0 + r < lim;
            const size_t off = in ? (size_t)(key0 + r) * HD + c : 0;
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(dk + r * L::LD + c);
            const int n = in ? 16 : 0;                         // keys past the end: zeros
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(K + off), "r"(n) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + AS_KT * L::LD * 4),
                         "l"(V + off), "r"(n)
                         : "memory");
        }
    };

    // score tile: lanes run 8 keys (lane bits 0, 2, 3) x 4 rows (bits 1, 4), warps 2 (keys)
    // x 4 (rows): neighbouring lanes share every address of one operand, so that a
    // 16-byte load serves more lanes at a time (24 rows over 341 keys, 16 heads: 14.9 us
    // with bits 0-2 and 3-4, 12.2)
    constexpr int SR = QR / 16, SKEYS = 4;                      // rows and keys per thread
    const int warp = tid >> 5, lane = tid & 31;
    const int sk = (warp & 1) * 8 + ((lane & 1) | (lane >> 1 & 6));                     // + 16 * i
    const int sr = (warp >> 1) * 4 + ((lane >> 1 & 1) | (lane >> 3 & 2));
    // softmax: GT neighbouring threads per row
    constexpr int GT = AS_THREADS / QR, KPT = AS_KT / GT;
    const int xr = tid / GT, xk = tid % GT;
    const int xplen = xr < nrows ? min(a.rows[r0 + xr].plen, k_hi) : 0;
    const uint64_t *xmask = a.mask && xr < nrows ? a.mask + (size_t)(r0 + xr) * a.mask_words : nullptr;
    // output tile: DT threads along the head dim, 4 dims each; rows orow + OG * i (16
    // threads a row: two rows side by side in neighbouring lanes)
    constexpr int DT = HD / 4, OG = AS_THREADS / DT, OR = QR / OG > 0 ? QR / OG : 1;
    const int od = (DT == 16 ? lane >> 1 : tid % DT) * 4, orow = DT == 16 ? warp * 2 + (lane & 1) : tid / DT;
    unsigned long long o01[OR] = {}, o23[OR] = {};

    if (nt > 0) load(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int i = 0; i < nt; ++i) {
        if (i + 1 < nt) load(i + 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const float *sK = sm + L::KV + (i & 1) * 2 * AS_KT * L::LD, *sV = sK + AS_KT * L::LD;
        {
            unsigned long long s[SR][SKEYS] = {};
#pragma unroll 8
            for (int c = 0; c < HD; c += 4) {
                ulonglong2 kv[SKEYS], qv[SR];
#pragma unroll
                for (int u = 0; u < SKEYS; ++u)
                    kv[u] = *reinterpret_cast<const ulonglong2 *>(sK + (sk + 16 * u) * L::LD + c);
#pragma unroll
                for (int u = 0; u < SR; ++u)
                    qv[u] = *reinterpret_cast<const ulonglong2 *>(sQ + (sr + 16 * u) * L::LD + c);
#pragma unroll
                for (int u = 0; u < SR; ++u)
#pragma unroll
                    for (int v = 0; v < SKEYS; ++v)
                        s[u][v] = as_fma2(qv[u].y, kv[v].y, as_fma2(qv[u].x, kv[v].x, s[u][v]));
            }
#pragma unroll
            for (int u = 0; u < SR; ++u)
#pragma unroll
                for (int v = 0; v < SKEYS; ++v)
                    sP[(sr + 16 * u) * AS_PLD + sk + 16 * v] = as_lo(s[u][v]) + as_hi(s[u][v]);
        }
        __syncthreads();
        bool odd = false;                       // a value of V that is not finite, in a tile with hidden keys
        {
            const bool tree = i >= nc;
            auto below = [](int n) { return n >= AS_KT ? ~0ull : n <= 0 ? 0ull : (1ull << n) - 1ull; };
            const int key0 = tree ? (i - nc) * AS_KT : k_lo + i * AS_KT;
            // the tile's keys that the row sees, and those that were copied but it does
            // not (the rest of the stage is zeros)
            const uint64_t held = xr < nrows ? below((tree ? a.tree_slots : k_hi) - key0) : 0ull;
            uint64_t vis = !tree ? below(xplen - key0) : (xmask && i - nc < a.mask_words ? xmask[i - nc] & held : 0ull);
            uint64_t hid = held & ~vis;
            vis >>= xk;
            hid >>= xk;
            float v[KPT], mx = -INFINITY;
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                v[j] = (vis >> (GT * j)) & 1ull ? sP[xr * AS_PLD + xk + GT * j] * p.scale_log2 : -INFINITY;
                mx = fmaxf(mx, v[j]);
            }
#pragma unroll
            for (int o = GT / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const float m0 = s_m[xr], mn = fmaxf(m0, mx);
            const float use = mn == -INFINITY ? 0.f : mn;
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                const float e = as_exp2(v[j] - use);
                sum += e;
                sP[xr * AS_PLD + xk + GT * j] = (hid >> (GT * j)) & 1ull ? HIDDEN : e;
            }
#pragma unroll
            for (int o = GT / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            __syncwarp();                       // every lane of the row has read s_m
            if (xk == 0) {
                const float f = as_exp2(m0 - use);             // (first visible keys: 2^-inf = 0)
                s_scale[xr] = f;
                s_m[xr] = mn;
                s_l[xr] = s_l[xr] * f + sum;
            }
        }
        if (i >= nc || min(k_lo + (i + 1) * AS_KT, k_hi) > least) {
            unsigned top = 0u;
#pragma unroll
            for (int e = tid; e < AS_KT * (HD / 4); e += AS_THREADS) {
                const int r = e / (HD / 4), c = (e - r * (HD / 4)) * 4;
                const uint4 w = *reinterpret_cast<const uint4 *>(sV + r * L::LD + c);
                top = max(max(max(top, w.x << 1), max(w.y << 1, w.z << 1)), w.w << 1);
            }
            odd = top >= 0xff000000u;
        }
        const bool skip = __syncthreads_or(odd);
        // O += P V; a hidden key adds -0 * V, nothing, or is skipped where that may be NaN
        auto pv = [&](auto skips) {
#pragma unroll 4
            for (int k = 0; k < AS_KT; k += 4) {
                ulonglong2 vv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) vv[j] = *reinterpret_cast<const ulonglong2 *>(sV + (k + j) * L::LD + od);
#pragma unroll
                for (int u = 0; u < OR; ++u) {
                    const float4 pr = *reinterpret_cast<const float4 *>(sP + (orow + OG * u) * AS_PLD + k);
                    const float pk[4] = {pr.x, pr.y, pr.z, pr.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (decltype(skips)::value && __float_as_uint(pk[j]) == 0x80000000u) continue;
                        const unsigned long long pp = as_pack(pk[j], pk[j]);
                        o01[u] = as_fma2(pp, vv[j].x, o01[u]);
                        o23[u] = as_fma2(pp, vv[j].y, o23[u]);
                    }
                }
            }
        };
        if (orow < QR) {
#pragma unroll
            for (int u = 0; u < OR; ++u) {
                const float f = s_scale[orow + OG * u];
                const unsigned long long ff = as_pack(f, f);
                o01[u] = as_fma2(o01[u], ff, 0ull);
                o23[u] = as_fma2(o23[u], ff, 0ull);
            }
            if (skip) pv(std::true_type());
            else pv(std::false_type());
        }
        __syncthreads();                        // the stage and the scores may be overwritten
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    if (p.nsplit == 1) {
        if (orow < QR)
#pragma unroll
            for (int u = 0; u < OR; ++u) {
                const int r = orow + OG * u;
                if (r >= nrows) continue;
                const float l = s_l[r], inv = l > 0.f ? 1.f / l : 0.f;
                *reinterpret_cast<float4 *>(a.out + (size_t)(r0 + r) * H + h * HD + od) =
                    make_float4(as_lo(o01[u]) * inv, as_hi(o01[u]) * inv, as_lo(o23[u]) * inv, as_hi(o23[u]) * inv);
            }
        return;
    }
    // partial O (unnormalised) over the query rows' place; combined in split order
    __syncthreads();
    if (orow < QR)
#pragma unroll
        for (int u = 0; u < OR; ++u)
            *reinterpret_cast<float4 *>(sQ + (orow + OG * u) * L::LD + od) =
                make_float4(as_lo(o01[u]), as_hi(o01[u]), as_lo(o23[u]), as_hi(o23[u]));
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int S = p.nsplit, rank = (int)cl.block_rank();
    const int n4 = nrows * DT, lo = rank * n4 / S, hi = (rank + 1) * n4 / S;
    for (int e = lo + tid; e < hi; e += AS_THREADS) {
        const int r = e / DT, d = (e - r * DT) * 4;
        float m[AS_MAX_SPLITS], l[AS_MAX_SPLITS];
        float4 v[AS_MAX_SPLITS];
#pragma unroll
        for (int q = 0; q < AS_MAX_SPLITS; ++q)
            if (q < S) {
                m[q] = cl.map_shared_rank(s_m, q)[r];
                l[q] = cl.map_shared_rank(s_l, q)[r];
                v[q] = *reinterpret_cast<const float4 *>(cl.map_shared_rank(sQ, q) + r * L::LD + d);
            }
        float mx = -INFINITY;
#pragma unroll
        for (int q = 0; q < AS_MAX_SPLITS; ++q)
            if (q < S) mx = fmaxf(mx, m[q]);
        const float use = mx == -INFINITY ? 0.f : mx;
        float den = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < AS_MAX_SPLITS; ++q)
            if (q < S) {
                const float f = as_exp2(m[q] - use);
                den += f * l[q];
                o.x += f * v[q].x; o.y += f * v[q].y; o.z += f * v[q].z; o.w += f * v[q].w;
            }
        const float inv = den > 0.f ? 1.f / den : 0.f;
        *reinterpret_cast<float4 *>(a.out + (size_t)(r0 + r) * H + h * HD + d) =
            make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv);
    }
    cl.sync();                                  // partials stay readable until all ranks are done
}

template <int HD, int QR>
cudaError_t launch_as(AsArgs p, int num_sms, cudaStream_t s) {
    const AttnArgs<float> &a = p.a;
    p.tiles_per_req = (p.rows_per_req + QR - 1) / QR;
    const int row_tiles = a.tiles ? a.n_tiles : a.R / p.rows_per_req * p.tiles_per_req;
    // splits while they fit one wave of CTAs, two key tiles of the cache each: a
    // function of the launch's shape
    const long base = (long)row_tiles * a.nh;
    p.nsplit = (int)std::max<long>(
        1, std::min<long>(std::min<long>(AS_MAX_SPLITS, (a.cache_slots + 2 * AS_KT - 1) / (2 * AS_KT)), num_sms / base));
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)a.nh, (unsigned)row_tiles, (unsigned)p.nsplit);
    lc.blockDim = dim3(AS_THREADS);
    lc.dynamicSmemBytes = AsLay<HD, QR>::SMEM;
    lc.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = (unsigned)p.nsplit;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = programmatic(s) ? 2 : 1;
    return cudaLaunchKernelEx(&lc, attn_simt_kernel<HD, QR>, (const AsArgs)p);
}

template <int HD, int QR>
bool set_as() {
    return cudaFuncSetAttribute(attn_simt_kernel<HD, QR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                AsLay<HD, QR>::SMEM) == cudaSuccess;
}

}  // namespace

bool attention_setup() { return set_as<64, 16>() && set_as<64, 64>() && set_as<128, 16>() && set_as<128, 64>(); }

bool launch_attention(const AttnArgs<float> &a, int rows_per_req, int num_sms, cudaStream_t s) {
    if (a.R <= 0) return true;
    if (rows_per_req < 1 || (!a.tiles && a.R % rows_per_req) || (a.hd != 64 && a.hd != 128)) return false;
    AsArgs p;
    p.a = a;
    p.rows_per_req = rows_per_req;
    p.tiles_per_req = p.nsplit = 1;
    p.scale_log2 = a.scale * 1.4426950408889634f;
    const int qr = !a.tiles && rows_per_req <= 32 ? 16 : 64;
    const long row_tiles = a.tiles ? a.n_tiles : (long)(a.R / rows_per_req) * ((rows_per_req + qr - 1) / qr);
    if (row_tiles > 65535) return false;        // the grid's y
    cudaError_t e;
    if (qr == 16)
        e = a.hd == 128 ? launch_as<128, 16>(p, num_sms, s) : launch_as<64, 16>(p, num_sms, s);
    else
        e = a.hd == 128 ? launch_as<128, 64>(p, num_sms, s) : launch_as<64, 64>(p, num_sms, s);
    note_launch();
    return e == cudaSuccess;
}

}  // namespace msd
