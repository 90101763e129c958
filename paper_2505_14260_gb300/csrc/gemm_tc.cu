// bf16 GEMMs on the sm_103a tensor cores.
//
// Operands are swapped: a 128-row weight tile is the MMA's A operand (M = 128,
// or 256 over a CTA pair) and the token rows are its B operand (N = 16 .. 256), so
// the accumulator D^T[128 weight rows][N tokens] sits in TMEM, one weight row per
// TMEM lane. Two kernels share the building blocks below:
//   gemm_cluster_kernel  up to 128 token rows: weight streaming from HBM, K split
//                        over a cluster, fused epilogues
//   gemm_persist_kernel  more token rows: tensor-bound, two-SM tiles
// Both take the context's packed weights, or the caller's row-major weight
// (msd_linear, msd_linear_noalloc) through a tensor map whose 128-byte swizzle
// leaves the same blocks in shared memory, so nothing is re-laid first.
// Every mbarrier wait is bounded (2 s of %globaltimer); on timeout the CTA
// sets the device status word and winds down.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstdio>
#include <algorithm>
#include <cstring>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "gemm_tc.h"
#include "msd.h"

namespace msd {

namespace {

constexpr int BM = 128;          // weight rows per tile (MMA M)
constexpr int BK = 64;           // K per stage: one 128-byte swizzle row of bf16
constexpr uint32_t A_BYTES = BM * BK * 2;          // 16 KB
constexpr unsigned long long TIMEOUT_NS = 2000000000ull;
constexpr size_t WS_BYTES = 64ull << 20;
constexpr int N_COUNTERS = 16384;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Launch stamps (profiling): [0] the earliest CTA entry, [1] the earliest
// return from griddepcontrol.wait (the previous kernel's results are visible),
// [2] the latest CTA exit, in %globaltimer nanoseconds.
__device__ __forceinline__ void stamp_min(unsigned long long *st, int i) {
    if (st) atomicMin(st + i, gtimer());
}
__device__ __forceinline__ void stamp_max(unsigned long long *st, int i) {
    if (st) atomicMax(st + i, gtimer());
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.b32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase with the given parity to complete: gives up when
// another thread of the CTA has set *abort_flag, or after limit_ns, when it
// sets *abort_flag and records ST_TIMEOUT in the status word.
__device__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status,
                          unsigned long long limit_ns = TIMEOUT_NS) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = gtimer();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (gtimer() - t0 > limit_ns) {
            *abort_flag = 1;
            set_status(status, ST_TIMEOUT);
            return false;
        }
    }
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row
// core-matrix groups 1024 bytes apart, sm100 descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) |
           ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor, kind::f16: fp32 accumulate, bf16 A and B, both
// K-major, N = BN, M = 128 (256 for a two-SM tile).
__device__ __forceinline__ uint32_t instr_desc(int BN, int M = BM) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

// Warp-wide forms. The TMA and MMA issue loops run in whole warps: tensor
// instructions take their descriptors, addresses and barriers from uniform
// registers, which a warp in step computes on the uniform datapath, while a loop
// in one diverged lane moves every operand over on its own (about 0.4 us of
// issue a 64-wide K stage, more than the MMAs of a 256 x 176 tile take). Only the
// lane that elect_one() names (`on`) issues.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t on;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.b32 %0, 1, 0, p;\n}" : "=r"(on));
    return on;
}

__device__ __forceinline__ void w_expect_tx(uint32_t on, uint32_t bar, uint32_t bytes) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n"
        "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}" ::"r"(bar),
        "r"(bytes), "r"(on)
        : "memory");
}

// Two-SM tiles (tcgen05 cta_group::2; CTAs 2j and 2j+1 of a cluster are a
// pair). The even CTA issues M = 256 MMAs: each CTA's own 128 weight rows are A,
// at the same shared-memory offset in both; each CTA holds BN/2 token columns
// of B (the even CTA the first half); each CTA's TMEM receives its own 128 rows
// x BN. Both CTAs' copies complete on the even CTA's stage barrier.
// 2-D tensor copy into this CTA's shared memory completing on an mbarrier of
// either CTA of the pair (a shared::cluster address).
__device__ __forceinline__ void w_tma_load_2d_pair(uint32_t on, uint32_t dst, const CUtensorMap *map, int x, int y,
                                                   uint32_t cluster_bar) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.b32 q, %5, 0;\n"
        "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2"
        " [%0], [%1, {%2, %3}], [%4];\n}" ::"r"(dst),
        "l"(map), "r"(x), "r"(y), "r"(cluster_bar), "r"(on)
        : "memory");
}

__device__ __forceinline__ void w_mma_bf16_pair(uint32_t on, uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                                uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p, q;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(on));
}

__device__ __forceinline__ void w_tma_load_2d(uint32_t on, uint32_t dst, const CUtensorMap *map, int x, int y,
                                              uint32_t bar) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.b32 q, %5, 0;\n"
        "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];\n}" ::"r"(dst),
        "l"(map), "r"(x), "r"(y), "r"(bar), "r"(on)
        : "memory");
}

// Contiguous global -> shared copy completing on an mbarrier (16-byte aligned).
__device__ __forceinline__ void w_bulk_load(uint32_t on, uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.b32 q, %4, 0;\n"
        "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n}" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar), "r"(on)
        : "memory");
}

__device__ __forceinline__ void w_mma_bf16(uint32_t on, uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                           uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p, q;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(on));
}

__device__ __forceinline__ void w_mma_commit(uint32_t on, uint32_t bar) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(bar), "r"(on)
        : "memory");
}

// Arrives, once the pair's MMAs issued so far complete, on the mbarrier at the
// same offset in each CTA of cta_mask (cluster ranks).
__device__ __forceinline__ void w_mma_commit_pair(uint32_t on, uint32_t bar, uint16_t cta_mask) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}" ::
            "r"(bar),
        "h"(cta_mask), "r"(on)
        : "memory");
}

// Arrive (release, cluster scope) on an mbarrier of another CTA of the cluster.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.b32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait on a barrier another CTA of the cluster arrives on.
__device__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status) {
    if (mbar_try_cluster(bar, parity)) return true;
    const unsigned long long t0 = gtimer();
    while (true) {
        if (mbar_try_cluster(bar, parity)) return true;
        if (*abort_flag) return false;
        if (gtimer() - t0 > TIMEOUT_NS) {
            *abort_flag = 1;
            set_status(status, ST_TIMEOUT);
            return false;
        }
    }
}

// The bounded waits for a whole warp (every lane waits; the answer is uniform).
__device__ __forceinline__ bool w_mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status) {
    if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status));
}
__device__ __forceinline__ bool w_mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                                    int *status) {
    if (__all_sync(0xffffffffu, mbar_try_cluster(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait_cluster(bar, parity, abort_flag, status));
}

// TMEM loads of this warp's 32 lanes, 16 or 32 columns, each waited for in
// the same asm statement: the compiler sees the registers defined only once
// the data has landed, so no use can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}

// gw (16 or 32: tiles are multiples of 16 columns) columns into r[0 .. gw)
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t *r, int gw) {
    if (gw > 16) tmem_ld32(taddr, r);
    else tmem_ld16(taddr, r);
}

// Two accumulators' columns with one round trip (a load and a wait each: the 7B verify
// call 877 us against 867).
__device__ __forceinline__ void tmem_ld16_two(uint32_t ta, uint32_t *a, uint32_t tb, uint32_t *b) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,"
        "%31}, [%33];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(a[0]), "=&r"(a[1]), "=&r"(a[2]), "=&r"(a[3]), "=&r"(a[4]), "=&r"(a[5]), "=&r"(a[6]),
          "=&r"(a[7]), "=&r"(a[8]), "=&r"(a[9]), "=&r"(a[10]), "=&r"(a[11]), "=&r"(a[12]), "=&r"(a[13]),
          "=&r"(a[14]), "=&r"(a[15]),
          "=&r"(b[0]), "=&r"(b[1]), "=&r"(b[2]), "=&r"(b[3]), "=&r"(b[4]), "=&r"(b[5]), "=&r"(b[6]),
          "=&r"(b[7]), "=&r"(b[8]), "=&r"(b[9]), "=&r"(b[10]), "=&r"(b[11]), "=&r"(b[12]), "=&r"(b[13]),
          "=&r"(b[14]), "=&r"(b[15])
        : "r"(ta), "r"(tb)
        : "memory");
}

__device__ __forceinline__ void tmem_ld32_two(uint32_t ta, uint32_t *a, uint32_t tb, uint32_t *b) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
        "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%64];\n"
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,"
        "%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%65];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(a[0]), "=&r"(a[1]), "=&r"(a[2]), "=&r"(a[3]), "=&r"(a[4]), "=&r"(a[5]), "=&r"(a[6]),
          "=&r"(a[7]), "=&r"(a[8]), "=&r"(a[9]), "=&r"(a[10]), "=&r"(a[11]), "=&r"(a[12]), "=&r"(a[13]),
          "=&r"(a[14]), "=&r"(a[15]), "=&r"(a[16]), "=&r"(a[17]), "=&r"(a[18]), "=&r"(a[19]), "=&r"(a[20]),
          "=&r"(a[21]), "=&r"(a[22]), "=&r"(a[23]), "=&r"(a[24]), "=&r"(a[25]), "=&r"(a[26]), "=&r"(a[27]),
          "=&r"(a[28]), "=&r"(a[29]), "=&r"(a[30]), "=&r"(a[31]),
          "=&r"(b[0]), "=&r"(b[1]), "=&r"(b[2]), "=&r"(b[3]), "=&r"(b[4]), "=&r"(b[5]), "=&r"(b[6]),
          "=&r"(b[7]), "=&r"(b[8]), "=&r"(b[9]), "=&r"(b[10]), "=&r"(b[11]), "=&r"(b[12]), "=&r"(b[13]),
          "=&r"(b[14]), "=&r"(b[15]), "=&r"(b[16]), "=&r"(b[17]), "=&r"(b[18]), "=&r"(b[19]), "=&r"(b[20]),
          "=&r"(b[21]), "=&r"(b[22]), "=&r"(b[23]), "=&r"(b[24]), "=&r"(b[25]), "=&r"(b[26]), "=&r"(b[27]),
          "=&r"(b[28]), "=&r"(b[29]), "=&r"(b[30]), "=&r"(b[31])
        : "r"(ta), "r"(tb)
        : "memory");
}

// gw columns of n accumulators, acc_stride apart, added in order into r[0 .. gw).
__device__ __forceinline__ void tmem_sum_cols(uint32_t taddr, int acc_stride, int n, uint32_t *r, int gw) {
    if (n == 1) {
        tmem_ld_cols(taddr, r, gw);
        return;
    }
    uint32_t e[32];
    if (gw > 16) tmem_ld32_two(taddr, r, taddr + acc_stride, e);
    else tmem_ld16_two(taddr, r, taddr + acc_stride, e);
    for (int q = 2;; ++q) {
#pragma unroll
        for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(e[j]));
        if (q >= n) return;
        tmem_ld_cols(taddr + q * acc_stride, e, gw);
    }
}

// ---------------------------------------------------------------------------
// Persistent two-SM variant (the context GEMM for many token rows).
//
// CTAs 2j and 2j+1 are a cluster that runs 256 x BN tiles with
// tcgen05.mma.cta_group::2: each CTA holds 128 weight rows and half of the
// token columns, so an SM reads half the token bytes per flop of a single-SM
// 128 x BN tile (whose two token planes, 2 x BN x 128 bytes a stage, bounded the
// kernel through L2: 66% of the burst rate in issued flops at 640 rows).
// The work is the list of (tile, K-block) units, tile-major; pair c of G takes
// units [c*U/G, (c+1)*U/G) of the cut tiles, then whole tiles, so every pair
// streams through one continuously running TMA -> MMA pipeline, across tile
// boundaries. Roles (192 threads): warp 0 issues TMA, warp 1 allocates TMEM and, in
// the even CTA, issues the MMAs (whole warps, one elected lane), warps 2-5 drain the
// accumulators. The accumulators come in groups: the K-blocks of an item (a tile, a
// chunk or a piece of one) take turns over those of a group, and where a pair has
// several items they take turns over two groups, so that the epilogue of one overlaps
// the MMAs of the next. A tile whose K range is cut between pairs ("pieces") is
// fixed up through the workspace, each CTA its own 128 rows: each piece is
// written to its CTA's slot (a CTA has at most two cut tiles, its first and its
// last), and the CTA that takes the tile's last ticket sums the pieces in pair
// order (deterministic) and applies the epilogue. No CTA waits on another pair.
// ---------------------------------------------------------------------------
constexpr int P_THREADS = 192;
constexpr int P_MAX_STAGES = 12;
constexpr int P_MAX_ACC = 2;        // groups of accumulators
constexpr int P_MAX_PIECES = 128;   // pieces of one cut tile (CTAs sharing it)

struct PkParams {
    int n_seg;
    int seg_tiles[3];
    int seg_rows[3];
    int seg_out[3];
    int M, kblocks, BN, n_tiles_n, stages, acc_stride, tmem_cols, grid;   // grid: CTA pairs
    int tiles;              // 128-row weight tiles
    long long units;        // stream-K units: T_sk tiles x K-blocks
    int T_sk, dp_rounds;    // stream-K tiles; rounds of whole tiles after them
    int T_all;              // all 256-row tiles x token tiles
    int kb_chunk;           // K-blocks of a whole tile accumulated before they are added to Y
    int n_acc;              // groups of accumulators (<= P_MAX_ACC)
    int n_rot;              // accumulators of a group, summed by the epilogue
    float *Y;
    int ldy, epi;
    float *ws;
    int *counters;
    int *status;
    bf16 *act;              // EPI_SWIGLU (glu-packed gate/up): act [M][F] split bf16
    int F;
    uint32_t stg_off;       // EPI_SWIGLU: byte offset of the 16 KB staging tile
    int has_lo;             // X is a split pair: its lo plane comes through the second map
    long lo;                // lo-plane offset of act (elements)
    unsigned long long *stamp;   // launch stamps (entry, wait, exit ns) or null
};

// silu(g) * u, the SwiGLU product of the fused epilogues.
__device__ __forceinline__ float swiglu_fused(float g, float u) {
    return __fdividef(g, 1.f + __expf(-g)) * u;
}

// CTA pair owning unit u under the balanced partition u0(c) = floor(c * U / G).
__device__ __forceinline__ int owner_cta(long long u, long long U, int G) {
    return (int)(((u + 1) * (long long)G - 1) / U);
}

// The work items of one CTA pair, in order: its share of the stream-K tiles
// [0, T_sk) (a contiguous range of (tile, K-block) units, cut at tile
// boundaries), then its whole tiles T_sk + cta + j*G, each in chunks of K.
struct ItemIter {
    long long u, u1;
    int KB, T_sk, G, cta, dp_j, dp_rounds, T_all, chunk, dp_kb;
    __device__ bool next(int &t, int &kb_b, int &kb_e) {
        if (u < u1) {
            t = (int)(u / KB);
            kb_b = (int)(u - (long long)t * KB);
            kb_e = (int)min((long long)KB, kb_b + (u1 - u));
            u += kb_e - kb_b;
            return true;
        }
        if (dp_j < dp_rounds && T_sk + cta + dp_j * G < T_all) {
            t = T_sk + cta + dp_j * G;
            kb_b = dp_kb;
            kb_e = min(KB, dp_kb + chunk);
            dp_kb = kb_e;
            if (kb_e == KB) {
                dp_kb = 0;
                ++dp_j;
            }
            return true;
        }
        return false;
    }
};

// all threads of both CTAs of the pair
__device__ __forceinline__ void c_cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t c_cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t c_mapa(uint32_t local, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}

// RAW: mw maps the caller's row-major weight (128-byte swizzle), read only after
// the wait on the previous kernel; otherwise the packed blocks.
template <bool RAW>
__global__ void __launch_bounds__(P_THREADS, 1)
    gemm_persist_kernel(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mxl,
                        const __grid_constant__ CUtensorMap mw, const PkParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * P_MAX_STAGES + 2 * P_MAX_ACC + 1];
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    __shared__ int s_reduce;
    __shared__ int s_slot[P_MAX_PIECES];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = (int)(blockIdx.x & 1u);          // cluster rank: the even CTA leads
    const int cta = (int)(blockIdx.x >> 1);           // the pair
    const long long U = p.units;                      // stream-K units
    const long long u0 = (long long)cta * U / p.grid, u1 = (long long)(cta + 1) * U / p.grid;
    const int KB = p.kblocks, stages = p.stages, BN = p.BN;
    const bool has_lo = p.has_lo != 0;
    const uint32_t b_bytes = (uint32_t)(BN / 2) * BK * 2;     // one plane of this CTA's token columns
    const uint32_t bs_bytes = has_lo ? 2 * b_bytes : b_bytes;  // hi, then lo
    const uint32_t stage_tx = 2u * (A_BYTES + bs_bytes);       // both CTAs' copies
    const ItemIter items0{u0, u1, KB, p.T_sk, p.grid, cta, 0, p.dp_rounds, p.T_all, p.kb_chunk, 0};

    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_base = sbase, b_base = sbase + stages * A_BYTES;
    const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[P_MAX_STAGES]);
    const uint32_t accf0 = smem_u32(&bars[2 * P_MAX_STAGES]);
    const uint32_t acce0 = smem_u32(&bars[2 * P_MAX_STAGES + P_MAX_ACC]);
    const uint32_t drain = smem_u32(&bars[2 * P_MAX_STAGES + 2 * P_MAX_ACC]);

    if (threadIdx.x == 0) {
        stamp_min(p.stamp, 0);
        for (int s = 0; s < stages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int a = 0; a < p.n_acc; ++a) {
            mbar_init(accf0 + 8 * a, 1);
            mbar_init(acce0 + 8 * a, 8);        // the epilogue warps of both CTAs
        }
        mbar_init(drain, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {        // both CTAs allocate together (the same columns in each)
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    c_cluster_sync();       // both CTAs' barriers are initialised before either signals the other's

    // (tile) -> this CTA's weight tile, its segment and rows; token rows
    auto tile_geom = [&](int t, int &wt, int &seg, int &row0, int &n0) {
        const int pt = t / p.n_tiles_n, nt = t - pt * p.n_tiles_n;
        wt = 2 * pt + half;             // (== tiles: the odd CTA past an odd tile count; no rows)
        int w = wt;
        seg = 0;
        while (seg < p.n_seg - 1 && w >= p.seg_tiles[seg]) {
            w -= p.seg_tiles[seg];
            ++seg;
        }
        row0 = w * BM;
        n0 = nt * BN;
    };

    if (warp == 0) {
        const uint32_t on = elect_one();
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&mx) : "memory");
            if (has_lo) asm volatile("prefetch.tensormap [%0];" ::"l"(&mxl) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(&mw) : "memory");
        }
        __syncwarp();
        const uint32_t sig0 = c_mapa(full0, 0);         // copies complete on the even CTA's barriers
        const uint32_t on_expect = half == 0 ? on : 0u;
        // the weight block of (weight tile, kb): x, y in the weight map (rows past
        // the last weight tile read as zeros)
        auto load_w = [&](int wt, int kb, int st) {
            w_expect_tx(on_expect, full0 + 8 * st, stage_tx);
            const int x = RAW ? kb * BK : 0, y = RAW ? wt * BM : (wt * KB + kb) * BM;
            w_tma_load_2d_pair(on, a_base + st * A_BYTES, &mw, x, y, sig0 + 8 * st);
        };
        // Packed weights never depend on the previous kernel: the first stages'
        // weight blocks are requested before waiting for it.
        int n_pre = 0;
        if constexpr (!RAW) {
            ItemIter it = items0;
            int t, kb_b, kb_e;
            while (n_pre < stages && it.next(t, kb_b, kb_e)) {
                const int wt = 2 * (t / p.n_tiles_n) + half;
                for (int kb = kb_b; kb < kb_e && n_pre < stages; ++kb, ++n_pre) load_w(wt, kb, n_pre);
            }
        }
        pdl_wait();
        if (lane == 0) stamp_min(p.stamp, 1);
        pdl_trigger();
        ItemIter it = items0;
        int t, kb_b, kb_e, s = 0, i = 0;
        uint32_t ph = 0;
        bool stop = false;
        while (!stop && it.next(t, kb_b, kb_e)) {
            const int pt = t / p.n_tiles_n, wt = 2 * pt + half;
            const int ny = (t - pt * p.n_tiles_n) * BN + half * (BN / 2);
            for (int kb = kb_b; kb < kb_e; ++kb, ++i) {
                if (i >= n_pre) {
                    if (!w_mbar_wait(empty0 + 8 * s, ph ^ 1u, &abort_flag, p.status)) {
                        stop = true;
                        break;
                    }
                    load_w(wt, kb, s);
                }
                w_tma_load_2d_pair(on, b_base + s * bs_bytes, &mx, kb * BK, ny, sig0 + 8 * s);
                if (has_lo)
                    w_tma_load_2d_pair(on, b_base + s * bs_bytes + b_bytes, &mxl, kb * BK, ny, sig0 + 8 * s);
                if (++s == stages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        if (abort_flag && half == 0) {      // (its barriers count both CTAs' copies)
            volatile int never = 0;
            for (int j = (i > stages ? i - stages : 0); j < i; ++j)
                mbar_wait(full0 + 8 * (j % stages), (uint32_t)(j / stages) & 1u, &never, p.status);
        }
        __syncwarp();
    } else if (warp == 1) {
        pdl_wait();
        if (half == 0) {                    // the even CTA issues for both
            const uint32_t on = elect_one();
            const uint32_t idesc = instr_desc(BN, 2 * BM);
            ItemIter it = items0;
            int t, kb_b, kb_e, s = 0;
            uint32_t ph = 0;
            bool stop = false;
            int a = 0;                      // the item's accumulator and its phase
            uint32_t aph = 0;
            for (; !stop && it.next(t, kb_b, kb_e); a = a + 1 == p.n_acc ? (aph ^= 1u, 0) : a + 1) {
                if (!w_mbar_wait_cluster(acce0 + 8 * a, aph ^ 1u, &abort_flag, p.status)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc0 = tmem + a * p.n_rot * p.acc_stride;
                for (int j = kb_b, rot = 0; j < kb_e; ++j) {
                    const uint32_t acc = acc0 + rot * p.acc_stride;
                    const uint32_t more = j - kb_b >= p.n_rot;      // its first block starts an accumulator
                    if (++rot == p.n_rot) rot = 0;
                    if (!w_mbar_wait_cluster(full0 + 8 * s, ph, &abort_flag, p.status)) {
                        stop = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t ad = smem_desc(a_base + s * A_BYTES);
                    const uint64_t bd = smem_desc(b_base + s * bs_bytes);
                    const uint64_t bl = smem_desc(b_base + s * bs_bytes + b_bytes);
                    if (has_lo) {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            w_mma_bf16_pair(on, acc, ad + 2 * kk, bd + 2 * kk, idesc, kk ? 1u : more);
                            w_mma_bf16_pair(on, acc, ad + 2 * kk, bl + 2 * kk, idesc, 1u);
                        }
                    } else {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk)
                            w_mma_bf16_pair(on, acc, ad + 2 * kk, bd + 2 * kk, idesc, kk ? 1u : more);
                    }
                    w_mma_commit_pair(on, empty0 + 8 * s, (uint16_t)3);
                    if (++s == stages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                w_mma_commit_pair(on, accf0 + 8 * a, (uint16_t)3);
            }
            // every MMA issued above completes before either CTA frees its TMEM
            w_mma_commit_pair(on, drain, (uint16_t)3);
            __syncwarp();
        }
        volatile int never = 0;
        mbar_wait_cluster(drain, 0, &never, p.status);
        __syncwarp();
    } else {
        // epilogue warps: TMEM lane quarter (warp % 4)
        pdl_wait();
        const int q = warp & 3;
        const int row = q * 32 + lane;
        const int et = threadIdx.x - 64;     // 0..127
        ItemIter it = items0;
        int t, kb_b, kb_e;
        int a = 0;
        uint32_t aph = 0;
        for (int item = 0; it.next(t, kb_b, kb_e); ++item, a = a + 1 == p.n_acc ? (aph ^= 1u, 0) : a + 1) {
            int wt, seg, row0, n0;
            tile_geom(t, wt, seg, row0, n0);
            const int o_local = row0 + row;
            const bool row_in = wt < p.tiles && o_local < p.seg_rows[seg];
            const int o = p.seg_out[seg] + o_local;
            const bool whole = t >= p.T_sk || (kb_b == 0 && kb_e == KB);
            const uint32_t taddr = tmem + a * p.n_rot * p.acc_stride + ((uint32_t)(q * 32) << 16);
            const int n_sub = min(p.n_rot, kb_e - kb_b);
            // a CTA cuts at most two stream-K tiles: its first item and its last
            const int slot = 2 * (2 * cta + (item == 0 ? 0 : 1)) + half;
            float *part = p.ws + (size_t)slot * BN * BM;
            // (a whole tile's later chunks add to what this thread stored for the first)
            const bool add = p.epi == EPI_ADD || (whole && kb_b > 0);
            const bool glu = p.epi == EPI_SWIGLU;
            float *stg = reinterpret_cast<float *>(smem_raw + p.stg_off);   // [32 columns][128 rows]
            // residual rows of 32 columns, requested one group ahead (the first
            // group's before the accumulator is waited for)
            auto residual = [&](int g0, float *yin) {
                const float *yb = p.Y + (size_t)(n0 + g0) * p.ldy + o;
                const int lim = min(min(32, BN - g0), p.M - (n0 + g0));
#pragma unroll
                for (int j = 0; j < 32; ++j) yin[j] = add && whole && row_in && j < lim ? yb[(size_t)j * p.ldy] : 0.f;
            };
            float ynext[32];
            residual(0, ynext);
            bool landed = mbar_wait_cluster(accf0 + 8 * a, aph, &abort_flag, p.status) && !abort_flag;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const bool ok = landed && wt < p.tiles, row_ok = landed && row_in;
            for (int g0 = 0; g0 < BN; g0 += 32) {
                // up to 32 accumulator columns with one TMEM round trip
                const int gw = min(32, BN - g0);
                float yin[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) yin[j] = ynext[j];
                if (g0 + 32 < BN) residual(g0 + 32, ynext);
                uint32_t r[32];
                tmem_sum_cols(taddr + g0, p.acc_stride, n_sub, r, gw);     // the item's accumulators
                if (whole && glu) {
                    // gate row i and up row 64 + i of the tile sit in different
                    // warps: exchange through shared memory, then thread (i, h)
                    // writes act[m][64 t + i] for the columns of half h
                    asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 32; ++j) stg[j * BM + row] = __uint_as_float(r[j]);
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                    const int i = et & 63, h = et >> 6;
                    const int jo = (row0 >> 1) + i;
                    if (ok && jo < p.F) {
#pragma unroll 4
                        for (int c = 16 * h; c < 16 * h + 16; ++c) {
                            const int m = n0 + g0 + c;
                            if (c < gw && m < p.M)
                                Split<bf16>::store(p.act + (size_t)m * p.F + jo, p.lo,
                                                   swiglu_fused(stg[c * BM + i], stg[c * BM + 64 + i]));
                        }
                    }
                } else if (!whole) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < gw) part[(size_t)(g0 + j) * BM + row] = __uint_as_float(r[j]);
                } else if (row_ok) {
                    float *yb = p.Y + (size_t)(n0 + g0) * p.ldy + o;
                    const int mlim = p.M - (n0 + g0);
                    if (add) {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (j < gw && j < mlim) yb[(size_t)j * p.ldy] = yin[j] + __uint_as_float(r[j]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (j < gw && j < mlim) yb[(size_t)j * p.ldy] = __uint_as_float(r[j]);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(c_mapa(acce0 + 8 * a, 0));
            if (whole) continue;
            // ticket for the cut tile; the last piece reduces all pieces in CTA order
            __threadfence();
            asm volatile("bar.sync 1, 128;" ::: "memory");
            const int c_first = owner_cta((long long)t * KB, U, p.grid);
            const int c_last = owner_cta((long long)(t + 1) * KB - 1, U, p.grid);
            const int np = c_last - c_first + 1;
            if (et == 0) {
                const int prev = atomicAdd(&p.counters[2 * t + half], 1);
                s_reduce = prev == np - 1;
            }
            if (et < np && et < P_MAX_PIECES) {
                const int cc = c_first + et;
                const long long cu0 = (long long)cc * U / p.grid;
                s_slot[et] = 2 * (2 * cc + (cu0 >= (long long)t * KB ? 0 : 1)) + half;
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (!s_reduce) continue;
            if (np > P_MAX_PIECES) {
                set_status(p.status, ST_RANGE);
                continue;
            }
            __threadfence();
            // flat float4 view of the [BN][128] pieces; 16 float4 loads of two pieces
            // (a cut tile mostly has two or three) in flight per thread
            constexpr int GR = 8, PI = 2;
            const int n4 = BN * BM / 4;
            const size_t piece4 = (size_t)BN * BM / 4;
            const float4 *ws4 = reinterpret_cast<const float4 *>(p.ws);
            for (int base4 = et; base4 < n4; base4 += GR * 128) {
                float4 acc[GR];
#pragma unroll
                for (int g = 0; g < GR; ++g) acc[g] = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int i0 = 0; i0 < np; i0 += PI) {
                    float4 v[PI][GR];
#pragma unroll
                    for (int pi = 0; pi < PI; ++pi) {
                        const bool have = i0 + pi < np;
                        const float4 *src = ws4 + (size_t)s_slot[have ? i0 + pi : 0] * piece4;
#pragma unroll
                        for (int g = 0; g < GR; ++g) {
                            const int e4 = base4 + g * 128;
                            v[pi][g] = (have && e4 < n4) ? __ldcg(src + e4)
                                                         : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    }
#pragma unroll
                    for (int pi = 0; pi < PI; ++pi)
#pragma unroll
                        for (int g = 0; g < GR; ++g) {
                            acc[g].x += v[pi][g].x; acc[g].y += v[pi][g].y;
                            acc[g].z += v[pi][g].z; acc[g].w += v[pi][g].w;
                        }
                }
                // (the residual's loads of all groups before any store)
                float4 yin[GR];
                if (p.epi == EPI_ADD) {
#pragma unroll
                    for (int g = 0; g < GR; ++g) {
                        const int e4 = base4 + g * 128, col = (e4 * 4) / BM, r4 = (e4 * 4) - col * BM;
                        const float *y = p.Y + (size_t)(n0 + col) * p.ldy + p.seg_out[seg] + row0 + r4;
                        yin[g] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (e4 < n4 && n0 + col < p.M && ok && row0 + r4 + 4 <= p.seg_rows[seg] &&
                            ((reinterpret_cast<uintptr_t>(y) & 15u) == 0))
                            yin[g] = *reinterpret_cast<const float4 *>(y);
                    }
                }
#pragma unroll
                for (int g = 0; g < GR; ++g) {
                    const int e4 = base4 + g * 128;
                    if (p.epi == EPI_SWIGLU) {
                        // lane l < 16 holds gate rows 4l..4l+3 of a column, lane
                        // l + 16 the matching up rows (e4 % 32 is the lane; the
                        // branch conditions below are uniform over the warp)
                        float4 up;
                        up.x = __shfl_xor_sync(0xffffffffu, acc[g].x, 16);
                        up.y = __shfl_xor_sync(0xffffffffu, acc[g].y, 16);
                        up.z = __shfl_xor_sync(0xffffffffu, acc[g].z, 16);
                        up.w = __shfl_xor_sync(0xffffffffu, acc[g].w, 16);
                        if (e4 >= n4) continue;
                        const int col = (e4 * 4) / BM, r4 = (e4 * 4) - col * BM;
                        const int m = n0 + col;
                        const int jo = (row0 >> 1) + r4;
                        if (m >= p.M || !ok || r4 >= 64 || jo >= p.F) continue;
                        bf16 *dst = p.act + (size_t)m * p.F + jo;     // F % 4 == 0: 8-byte aligned
                        Split<bf16>::store4(dst, p.lo,
                                            make_float4(swiglu_fused(acc[g].x, up.x), swiglu_fused(acc[g].y, up.y),
                                                        swiglu_fused(acc[g].z, up.z), swiglu_fused(acc[g].w, up.w)));
                        continue;
                    }
                    if (e4 >= n4) continue;
                    const int col = (e4 * 4) / BM, r4 = (e4 * 4) - col * BM;
                    const int m = n0 + col;
                    if (m >= p.M || !ok) continue;
                    float *y = p.Y + (size_t)m * p.ldy + p.seg_out[seg] + row0 + r4;
                    if (row0 + r4 + 4 <= p.seg_rows[seg] &&
                        ((reinterpret_cast<uintptr_t>(y) & 15u) == 0)) {      // one 16-byte access
                        float4 out = acc[g];
                        if (p.epi == EPI_ADD) {
                            out.x += yin[g].x; out.y += yin[g].y; out.z += yin[g].z; out.w += yin[g].w;
                        }
                        *reinterpret_cast<float4 *>(y) = out;
                    } else {
                        const float vv[4] = {acc[g].x, acc[g].y, acc[g].z, acc[g].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (row0 + r4 + e < p.seg_rows[seg]) {
                                if (p.epi == EPI_ADD) y[e] = y[e] + vv[e];
                                else y[e] = vv[e];
                            }
                    }
                }
            }
            if (et == 0) p.counters[2 * t + half] = 0;
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) stamp_max(p.stamp, 2);
    // neither CTA leaves, or frees its tensor memory, while the other may still
    // signal its barriers or read its own accumulators
    c_cluster_sync();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(p.tmem_cols)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// Split-K with a cluster reduction (decode shapes, M <= 128 token rows).
//
// One CTA per (weight tile, token tile, K-split); the s K-splits of a tile are
// one thread-block cluster. Each CTA streams its K range (pre-packed weight
// blocks by cp.async.bulk before the previous kernel ends, token blocks by
// TMA), accumulates in TMEM, and, with s > 1, leaves its fp32 partial in its
// own shared memory; after a cluster barrier each CTA sums one slice of the
// tile over all s partials through distributed shared memory, in rank order
// (deterministic), and writes it. At most two CTAs share an SM, so every
// launch of the decode step is a single wave.
// ---------------------------------------------------------------------------
// Eight warps: past the last MMA a CTA runs a chain of tensor-memory reads, shared
// memory, special functions and stores, which four warps left idle for most of it
// (per launch in a replayed 7B step, four warps and then eight: gate/up 35.4 and
// 34.1 us, q/k/v 20.9 and 20.1, down 19.1 and 18.0, O 11.8 and 11.1).
constexpr int C_THREADS = 256;
constexpr int C_STAGES = 4;

struct CkParams {
    int n_seg;
    int seg_tiles[3];
    int seg_rows[3];
    int seg_out[3];
    int M, kblocks, BN, n_tiles_n, splits, tmem_cols;
    int stages;             // ring depth (<= C_STAGES)
    int n_acc, acc_stride;  // accumulators that take turns over the K-blocks (summed in the epilogue)
    int has_lo;             // X is a split pair: its lo plane comes through the second map
    const bf16 *wpacked;
    float *Y;
    int ldy, epi;
    int *status;
    GemmFused fx;           // EPI_SWIGLU / EPI_ROPE_KV operands
    GemmNorm nout, nin;     // folded RMSNorm: producer / consumer side (ss null: off)
    unsigned long long *stamp;   // launch stamps (entry, wait, exit ns) or null
};

// Where a CTA finds the S partials of the token columns it owns, [c_lo,
// c_hi) = [rank * BN / S, (rank + 1) * BN / S): its own partial ([BN][128]
// fp32, all columns) and, for S > 1, the other ranks' slices of its columns,
// pushed into its receive buffer by bulk copies (slot q < rank ? q : q - 1,
// `span` columns each).
struct PartSrc {
    const float *own, *recv;
    int rank, S, c_lo, c_hi, span;
    // shared-window address of a float4 (read with ld.shared)
    __device__ __forceinline__ uint32_t at(int q, int col, int row) const {
        const float *b = q == rank ? own + col * BM : recv + ((q < rank ? q : q - 1) * span + (col - c_lo)) * BM;
        return (uint32_t)__cvta_generic_to_shared(b + row);
    }
};

__device__ __forceinline__ float4 lds4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ float lds1(const float *p) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)));
    return v;
}

// Sums, in rank order, of the S partials' float4 at K (column, row) places
// (all in this CTA's shared memory); every load is issued before the first sum.
template <int K>
__device__ __forceinline__ void c_part_sums(const PartSrc &ps, const int (&col)[K], const int (&row)[K],
                                            const bool (&use)[K], float4 (&out)[K]) {
    if (ps.S == 1) {                 // one partial: plain loads (no unrolled rank loop)
#pragma unroll
        for (int k = 0; k < K; ++k) out[k] = use[k] ? lds4(ps.at(0, col[k], row[k])) : make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    float4 v[K][8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if (q >= ps.S) break;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (use[k]) v[k][q] = lds4(ps.at(q, col[k], row[k]));
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < ps.S && use[k]) {
                a.x += v[k][q].x; a.y += v[k][q].y; a.z += v[k][q].z; a.w += v[k][q].w;
            }
        out[k] = a;
    }
}

// The fused epilogues read the tile's S partials ([BN][128] fp32 in each
// cluster CTA's shared memory at part_s) and take this CTA's rank share of the
// BN * 16 groups of four rows of one token; the partials are summed in rank
// order, as in the plain reduction. Each thread handles two groups per pass,
// with every load of both issued before either is used, so that a pass costs
// about one round trip to distributed shared memory and one to global memory.

// SwiGLU (glu-packed tile: rows 0-63 gate, 64-127 up):
// act[m][64 t + i] = bf16(silu(g) * u), scaled first by the folded-norm 1/rms.
__device__ __forceinline__ void c_epi_swiglu(const CkParams &p, const PartSrc &ps, bool ok, int wt, int n0,
                                             const float *rinv) {
    // the parameters the loop uses, read once before its stores
    bf16 *const act = p.fx.act;
    const int F = p.fx.F, M = p.M;
    const long lo = p.fx.lo;
    const int n = (ps.c_hi - ps.c_lo) * 16;         // groups of this CTA's columns
    auto emit = [&](float4 a, float4 b, int c, int j) {
        const int m = n0 + c;
        if (!ok || m >= M || j >= F) return;          // F % 4 == 0: whole groups
        if (rinv) {
            const float sc = lds1(rinv + c);
            a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc;
            b.x *= sc; b.y *= sc; b.z *= sc; b.w *= sc;
        }
        const float o0 = __fdividef(a.x, 1.f + __expf(-a.x)) * b.x;
        const float o1 = __fdividef(a.y, 1.f + __expf(-a.y)) * b.y;
        const float o2 = __fdividef(a.z, 1.f + __expf(-a.z)) * b.z;
        const float o3 = __fdividef(a.w, 1.f + __expf(-a.w)) * b.w;
        Split<bf16>::store4(act + (size_t)m * F + j, lo, make_float4(o0, o1, o2, o3));
    };
    for (int e = threadIdx.x; e < n; e += C_THREADS) {
        const int c = ps.c_lo + (e >> 4), r = (e & 15) << 2;
        const int col[2] = {c, c}, row[2] = {r, r + 64};
        const bool use[2] = {true, true};
        float4 v[2];
        c_part_sums<2>(ps, col, row, use, v);
        emit(v[0], v[1], c, wt * 64 + r);
    }
}

// Global operands of the first EPI_PRE groups (RoPE) or columns (norm) of a
// thread are requested before the split-K exchange, so that their round trip
// overlaps it; later ones (large column shares only) are loaded in the loop.
constexpr int EPI_PRE = 2;

struct RopePre {
    RowDesc d[EPI_PRE];
    float4 c01[EPI_PRE], c23[EPI_PRE];
};

// RoPE + K/V placement (tile of wq;wk;wv rows, hd | 128): rotate-half pairs
// (i, i + hd/2) of one head; q rotated into q_out [M][H], k rotated and v into
// kdst / vdst [B][nh][slots][hd] at the row's slot. Row descriptors come from
// shared memory (loaded while the MMAs ran).
struct RopeGeom {
    int hd, lh, half, lhd, n;
    __device__ __forceinline__ RopeGeom(int hd_, const PartSrc &ps)
        : hd(hd_), lh(hd_ == 128 ? 6 : 5), half(1 << lh), lhd(lh + 1), n((ps.c_hi - ps.c_lo) * 16) {}
    // group e of this CTA's columns: token column and first row of the pair
    __device__ __forceinline__ void at(const PartSrc &ps, int e, int &c, int &r) const {
        c = ps.c_lo + (e >> 4);
        const int p4 = (e & 15) << 2;
        r = ((p4 >> lh) << lhd) | (p4 & (half - 1));
    }
};

// the rotation-table entries (cos, sin of 4 consecutive frequencies) of one group
__device__ __forceinline__ void c_rope_tab(const CkParams &p, const RopeGeom &g, int pos, int row0, int r,
                                           float4 &c01, float4 &c23) {
    if (pos < 0 || pos >= p.fx.max_pos) {
        set_status(p.status, ST_RANGE);
        pos = 0;
    }
    const int i = (row0 + r) & (g.hd - 1);
    const float4 *cs = reinterpret_cast<const float4 *>(p.fx.rope_tab + (size_t)pos * g.half + i);
    c01 = cs[0];
    c23 = cs[1];
}

__device__ __forceinline__ void c_rope_pre(const CkParams &p, const PartSrc &ps, bool ok, int seg, int row0,
                                           int n0, int rows_here, const RowDesc *srow, RopePre &pre) {
    const RopeGeom g(p.fx.hd, ps);
#pragma unroll
    for (int k = 0; k < EPI_PRE; ++k) {
        const int e = threadIdx.x + k * C_THREADS;
        if (e >= g.n) break;
        int c, r;
        g.at(ps, e, c, r);
        pre.d[k] = srow[c];
        if (ok && seg < 2 && n0 + c < p.M && r < rows_here)
            c_rope_tab(p, g, pre.d[k].pos, row0, r, pre.c01[k], pre.c23[k]);
    }
}

__device__ __forceinline__ void c_epi_rope(const CkParams &p, const PartSrc &ps, bool ok, int seg, int row0,
                                           int n0, int rows_here, const float *rinv, const RowDesc *srow,
                                           const RopePre &pre) {
    const RopeGeom g(p.fx.hd, ps);
    const int slots = p.fx.slots, nh = p.fx.nh, M = p.M, hd = g.hd, half = g.half;
    bf16 *const qo = p.fx.q_out, *const kvd = seg == 1 ? p.fx.kdst : p.fx.vdst;
    const long lo = p.fx.lo;
    int *const status = p.status;
    for (int k = 0;; ++k) {
        const int e = threadIdx.x + k * C_THREADS;
        if (e >= g.n) break;
        int c, r;
        g.at(ps, e, c, r);
        const int m = n0 + c;
        if (!ok || m >= M || r >= rows_here) continue;
        RowDesc d;
        float4 c01, c23;
        if (k < EPI_PRE) {
#pragma unroll
            for (int j = 0; j < EPI_PRE; ++j)       // static indices only
                if (j == k) { d = pre.d[j]; c01 = pre.c01[j]; c23 = pre.c23[j]; }
        } else {
            d = srow[c];
            if (seg < 2) c_rope_tab(p, g, d.pos, row0, r, c01, c23);
        }
        const int col[2] = {c, c}, row[2] = {r, r + half};
        const bool use[2] = {true, true};
        float4 v[2];
        c_part_sums<2>(ps, col, row, use, v);
        float4 a = v[0], b = v[1];
        if (rinv) {
            const float sc = lds1(rinv + c);
            a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc;
            b.x *= sc; b.y *= sc; b.z *= sc; b.w *= sc;
        }
        const int o = row0 + r, h = o >> g.lhd, i = o & (hd - 1);
        if (seg < 2) {
            const float x0 = a.x, x1 = a.y, x2 = a.z, x3 = a.w;
            a.x = x0 * c01.x - b.x * c01.y; b.x = b.x * c01.x + x0 * c01.y;
            a.y = x1 * c01.z - b.y * c01.w; b.y = b.y * c01.z + x1 * c01.w;
            a.z = x2 * c23.x - b.z * c23.y; b.z = b.z * c23.x + x2 * c23.y;
            a.w = x3 * c23.z - b.w * c23.w; b.w = b.w * c23.z + x3 * c23.w;
        }
        bf16 *dst;
        if (seg == 0) {
            dst = qo + (size_t)m * (nh * hd) + o;
        } else {
            if (d.dst >= slots) set_status(status, ST_RANGE);
            if (d.dst < 0 || d.dst >= slots) continue;
            dst = kvd + ((size_t)(d.req * nh + h) * slots + d.dst) * hd + i;
        }
        Split<bf16>::store4(dst, lo, a);
        Split<bf16>::store4(dst + half, lo, b);
    }
}

// Residual rows of the first EPI_PRE columns of a warp (folded-norm producer
// with accumulation), requested before the exchange.
__device__ __forceinline__ void c_norm_pre(const CkParams &p, const PartSrc &ps, bool ok, int o_base,
                                           int rows_here, int n0, float4 (&yv)[EPI_PRE]) {
    const int warp = threadIdx.x >> 5, r4 = (threadIdx.x & 31) * 4;
    if (p.epi != EPI_ADD || r4 + 4 > rows_here) return;
#pragma unroll
    for (int k = 0; k < EPI_PRE; ++k) {
        const int c = ps.c_lo + warp + k * (C_THREADS / 32);
        if (ok && c < ps.c_hi && n0 + c < p.M)
            yv[k] = *reinterpret_cast<const float4 *>(p.Y + (size_t)(n0 + c) * p.ldy + o_base + r4);
    }
}

// Producer side of a folded RMSNorm: this CTA's token columns, one warp per
// column (lane = 4 consecutive weight rows): the S partials summed in rank
// order, the residual added, then Y (fp32), xg = bf16(y * g) and the column's
// sum of squares over the tile's rows (a warp reduction in a fixed order) into
// ss[m][tile].
__device__ __forceinline__ void c_reduce_norm(const CkParams &p, const PartSrc &ps, bool ok, int tile, int o_base,
                                              int rows_here, int n0, const float4 (&yv)[EPI_PRE]) {
    constexpr int NW = C_THREADS / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool add = p.epi == EPI_ADD;
    const int r4 = lane * 4;
    const bool full = r4 + 4 <= rows_here;
    float g4[4] = {0.f, 0.f, 0.f, 0.f};
    if (full) {
        const uint2 gw = *reinterpret_cast<const uint2 *>(p.nout.g + o_base + r4);
        const __nv_bfloat162 g01 = *reinterpret_cast<const __nv_bfloat162 *>(&gw.x);
        const __nv_bfloat162 g23 = *reinterpret_cast<const __nv_bfloat162 *>(&gw.y);
        g4[0] = __low2float(g01); g4[1] = __high2float(g01);
        g4[2] = __low2float(g23); g4[3] = __high2float(g23);
    }
    float *const Y = p.Y;
    bf16 *const XG = p.nout.xg;
    const int ldy = p.ldy, M = p.M;
    const long xlo = p.nout.lo;
    float *const ssd = p.nout.ss;
    const int ssld = p.nout.ld;
    const bf16 *const gn = p.nout.g;
    for (int k = 0;; ++k) {
        const int c = ps.c_lo + warp + k * NW;
        if (c >= ps.c_hi) break;                         // warp-uniform
        const int col[1] = {c}, row[1] = {r4};
        const bool use[1] = {true};
        float4 v[1];
        c_part_sums<1>(ps, col, row, use, v);
        float a[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
        const int m = n0 + c;
        const bool live = ok && m < M;                   // warp-uniform
        float ss = 0.f;
        if (live) {
            float *y = Y + (size_t)m * ldy + o_base + r4;
            bf16 *xg = XG + (size_t)m * ldy + o_base + r4;
            if (full) {
                if (add) {
                    float4 yi;
                    if (k < EPI_PRE) {
#pragma unroll
                        for (int j = 0; j < EPI_PRE; ++j)
                            if (j == k) yi = yv[j];
                    } else {
                        yi = *reinterpret_cast<const float4 *>(y);
                    }
                    a[0] += yi.x; a[1] += yi.y; a[2] += yi.z; a[3] += yi.w;
                }
                *reinterpret_cast<float4 *>(y) = make_float4(a[0], a[1], a[2], a[3]);
                Split<bf16>::store4(xg, xlo, make_float4(a[0] * g4[0], a[1] * g4[1], a[2] * g4[2], a[3] * g4[3]));
                ss = a[0] * a[0] + a[1] * a[1] + a[2] * a[2] + a[3] * a[3];
            } else {
                const bf16 *g = gn + o_base + r4;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (r4 + e < rows_here) {
                        const float ye = add ? y[e] + a[e] : a[e];
                        y[e] = ye;
                        Split<bf16>::store(xg + e, xlo, ye * __bfloat162float(g[e]));
                        ss += ye * ye;
                    }
            }
        }
        ss = warp_sum(ss);
        if (live && lane == 0) ssd[(size_t)m * ssld + tile] = ss;
    }
}

// RAW: mw maps the caller's row-major weight, read only after the wait on the
// previous kernel (which may have written it); otherwise the packed blocks.
template <bool PAIR, bool RAW>
__global__ void __launch_bounds__(C_THREADS, 2)
    gemm_cluster_kernel(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mxl,
                        const __grid_constant__ CUtensorMap mw, const CkParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * C_STAGES + 3];
    __shared__ uint32_t tmem_base;
    __shared__ volatile int abort_flag;
    __shared__ float s_rinv[128];     // folded RMSNorm (consumer): 1/rms of each token column
    __shared__ RowDesc s_rows[128];   // EPI_ROPE_KV: the token columns' row descriptors

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int wt = blockIdx.x, seg = 0;
    while (seg < p.n_seg - 1 && wt >= p.seg_tiles[seg]) {
        wt -= p.seg_tiles[seg];
        ++seg;
    }
    const int row0 = wt * BM;
    const int n0 = blockIdx.y * p.BN;
    const int split = blockIdx.z, S = p.splits;
    const int KB = p.kblocks;
    const int kb0 = (int)((long long)split * KB / S), kb1 = (int)((long long)(split + 1) * KB / S);
    const int nk = kb1 - kb0;
    const int BN = p.BN;
    const int stages = p.stages;
    const bool has_lo = p.has_lo != 0;
    // Two-SM mode (one K split only): CTAs 2j and 2j+1 run one M = 256 tile;
    // each holds its own weight rows and half of the token columns.
    constexpr bool pair = PAIR;
    const uint32_t half = pair ? (blockIdx.x & 1u) : 0u;       // 1: the odd CTA of a pair
    const int BNs = pair ? BN / 2 : BN;                        // token columns in this CTA's stages
    const uint32_t b_bytes = (uint32_t)BNs * BK * 2;         // one plane of a token stage
    const uint32_t bs_bytes = has_lo ? 2 * b_bytes : b_bytes; // hi, then lo
    const size_t blk_elems = A_BYTES / 2;
    const bf16 *wblk = p.wpacked + ((size_t)blockIdx.x * KB + kb0) * blk_elems;

    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_base = sbase, b_base = sbase + stages * A_BYTES;
    const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[C_STAGES]);
    const uint32_t done = smem_u32(&bars[2 * C_STAGES]);
    const uint32_t recv_bar = smem_u32(&bars[2 * C_STAGES + 1]);   // the other ranks' slices have landed
    const uint32_t pexit = smem_u32(&bars[2 * C_STAGES + 2]);      // (pair) the other CTA is done with its TMEM

    // Warp 0's elected lane sets the barriers up and, where the copies complete on
    // this CTA's own barriers, requests the first weight blocks at once (packed
    // weights depend on no earlier kernel): not after the tensor-memory allocation,
    // which waits while CTAs of the previous kernel still hold theirs.
    uint32_t on = 0;
    const int n_pre = RAW ? 0 : min(stages, nk);
    const uint32_t stage_tx = (pair ? 2u : 1u) * (A_BYTES + bs_bytes);
    if (warp == 0) {
        on = elect_one();
        if (on) {
            stamp_min(p.stamp, 0);
            for (int s = 0; s < stages; ++s) {
                mbar_init(full0 + 8 * s, 1);
                mbar_init(empty0 + 8 * s, 1);
            }
            mbar_init(done, 1);
            mbar_init(recv_bar, 1);
            mbar_init(pexit, 1);
            abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        if constexpr (!pair)
            for (int j = 0; j < n_pre; ++j) {
                w_expect_tx(on, full0 + 8 * j, stage_tx);
                w_bulk_load(on, a_base + j * A_BYTES, wblk + (size_t)j * blk_elems, A_BYTES, full0 + 8 * j);
            }
    }
    if (warp == 1) {
        if constexpr (pair) {   // both CTAs of the pair allocate together (the same columns in each)
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tmem_base)),
                         "r"(p.tmem_cols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tmem_base)),
                         "r"(p.tmem_cols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const uint32_t my_rank = pair ? c_cluster_rank() : 0u;
    const uint32_t lead_rank = my_rank & ~1u;                 // (pair) the even CTA
    const uint16_t pair_mask = (uint16_t)(3u << lead_rank);
    // where this CTA's copies complete: its own barriers, or (pair) the even CTA's
    const uint32_t sig0 = pair ? c_mapa(full0, lead_rank) : full0;
    // (pair) both CTAs' barriers are initialised before either signals the other's
    if constexpr (pair) c_cluster_sync();

    if (warp == 0) {
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&mx) : "memory");
            if (has_lo) asm volatile("prefetch.tensormap [%0];" ::"l"(&mxl) : "memory");
            if (pair || RAW) asm volatile("prefetch.tensormap [%0];" ::"l"(&mw) : "memory");
        }
        __syncwarp();
        const uint32_t on_expect = !pair || half == 0 ? on : 0u;
        // the weight block of pipeline step i: a bulk copy, or (pair) a tensor
        // copy of its 128 rows that completes on the even CTA's barrier
        auto load_w = [&](int i, int st) {
            w_expect_tx(on_expect, full0 + 8 * st, stage_tx);
            if constexpr (pair)
                w_tma_load_2d_pair(on, a_base + st * A_BYTES, &mw, 0, ((int)blockIdx.x * KB + kb0 + i) * BM,
                                   sig0 + 8 * st);
            else if constexpr (RAW)
                w_tma_load_2d(on, a_base + st * A_BYTES, &mw, (kb0 + i) * BK, row0, full0 + 8 * st);
            else
                w_bulk_load(on, a_base + st * A_BYTES, wblk + (size_t)i * blk_elems, A_BYTES, full0 + 8 * st);
        };
        // (pair) the first weight blocks, then the wait on the previous kernel
        if constexpr (pair)
            for (int j = 0; j < n_pre; ++j) load_w(j, j);
        pdl_wait();
        if (lane == 0) stamp_min(p.stamp, 1);
        pdl_trigger();
        const int ny = pair ? n0 + (int)half * BNs : n0;
        int s = 0;
        uint32_t ph = 0;
        int i = 0;
        for (; i < nk; ++i) {
            if (i >= n_pre) {
                if (!w_mbar_wait(empty0 + 8 * s, ph ^ 1u, &abort_flag, p.status)) break;
                load_w(i, s);
            }
            if constexpr (pair) {
                w_tma_load_2d_pair(on, b_base + s * bs_bytes, &mx, (kb0 + i) * BK, ny, sig0 + 8 * s);
                if (has_lo)
                    w_tma_load_2d_pair(on, b_base + s * bs_bytes + b_bytes, &mxl, (kb0 + i) * BK, ny, sig0 + 8 * s);
            } else {
                w_tma_load_2d(on, b_base + s * bs_bytes, &mx, (kb0 + i) * BK, ny, full0 + 8 * s);
                if (has_lo)
                    w_tma_load_2d(on, b_base + s * bs_bytes + b_bytes, &mxl, (kb0 + i) * BK, ny, full0 + 8 * s);
            }
            if (++s == stages) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (abort_flag && (!pair || half == 0)) {   // (pair: the even CTA's barriers count both CTAs' copies)
            volatile int never = 0;
            for (int j = (i > stages ? i - stages : 0); j < i; ++j)
                mbar_wait(full0 + 8 * (j % stages), (uint32_t)(j / stages) & 1u, &never, p.status);
        }
        __syncwarp();
    } else if (warp == 1) {
        pdl_wait();
        if (!pair || half == 0) {      // (pair: the even CTA issues for both)
            const uint32_t on = elect_one();
            const uint32_t idesc = instr_desc(BN, pair ? 2 * BM : BM);
            int s = 0, a = 0;
            uint32_t ph = 0;
            for (int i = 0; i < nk; ++i) {
                if (pair ? !w_mbar_wait_cluster(full0 + 8 * s, ph, &abort_flag, p.status)
                         : !w_mbar_wait(full0 + 8 * s, ph, &abort_flag, p.status))
                    break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t ad = smem_desc(a_base + s * A_BYTES);
                const uint64_t bd = smem_desc(b_base + s * bs_bytes);
                const uint64_t bl = smem_desc(b_base + s * bs_bytes + b_bytes);
                const uint32_t more = i >= p.n_acc, acc = tmem + a * p.acc_stride;
                if (++a == p.n_acc) a = 0;
                if (has_lo) {
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) {
                        if constexpr (pair) {
                            w_mma_bf16_pair(on, acc, ad + 2 * kk, bd + 2 * kk, idesc, kk ? 1u : more);
                            w_mma_bf16_pair(on, acc, ad + 2 * kk, bl + 2 * kk, idesc, 1u);
                        } else {
                            w_mma_bf16(on, acc, ad + 2 * kk, bd + 2 * kk, idesc, kk ? 1u : more);
                            w_mma_bf16(on, acc, ad + 2 * kk, bl + 2 * kk, idesc, 1u);
                        }
                    }
                } else {
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) {
                        if constexpr (pair) w_mma_bf16_pair(on, acc, ad + 2 * kk, bd + 2 * kk, idesc, kk ? 1u : more);
                        else w_mma_bf16(on, acc, ad + 2 * kk, bd + 2 * kk, idesc, kk ? 1u : more);
                    }
                }
                if constexpr (pair) w_mma_commit_pair(on, empty0 + 8 * s, pair_mask);
                else w_mma_commit(on, empty0 + 8 * s);
                if (++s == stages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if constexpr (pair) w_mma_commit_pair(on, done, pair_mask);
            else w_mma_commit(on, done);
            volatile int never = 0;     // (no MMA outlives the CTA's TMEM)
            mbar_wait(done, 0, &never, p.status);
        }
        __syncwarp();
    } else {
        pdl_wait();
        // idle during the main loop: the row scales of a folded RMSNorm
        if (p.nin.ss)
            for (int t = threadIdx.x - 64; t < p.BN; t += C_THREADS - 64) {
                const int m = n0 + t;
                float sum = 0.f;
                if (m < p.M)
                    for (int j = 0; j < p.nin.parts; ++j) sum += p.nin.ss[(size_t)m * p.nin.ld + j];
                s_rinv[t] = rsqrtf(sum / (float)p.nin.H + p.nin.eps);
            }
        if (p.epi == EPI_ROPE_KV)
            for (int t = threadIdx.x - 64; t < p.BN; t += C_THREADS - 64) {
                const int m = n0 + t;
                s_rows[t] = m < p.M ? p.fx.rows[m] : RowDesc{0, 0, 0, -1};
            }
    }

    // ---- epilogue: all warps, TMEM lane quarter = warp mod 4; warps 0-3 and
    // 4-7 take the tile's groups of 32 columns in turn ------------------------
    const bool ok = mbar_wait(done, 0, &abort_flag, p.status) && !abort_flag;
    // K split over the cluster: this CTA's MMAs are done, so its ring may now
    // receive the other ranks' slices. It arrives on the cluster barrier here
    // and waits on it only after storing its own partial, which hides the
    // barrier's round trip behind that store.
    if (S > 1) {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    pdl_wait();                       // (every thread) before reading Y, rows or the table
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int row = (warp & 3) * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const int g_first = (warp >> 2) * 32, g_step = C_THREADS / 4;
    const bool add = p.epi == EPI_ADD;
    const int rows_here = p.seg_rows[seg] - row0;           // valid weight rows in this tile
    const int o_base = p.seg_out[seg] + row0;
    const bool paired = p.epi >= EPI_SWIGLU;
    const bool norm_out = p.nout.ss != nullptr;
    // columns [g0, g0 + gw) of the tile, the accumulators that took a K-block added in order
    const int n_acc = min(p.n_acc, nk);
    auto acc_cols = [&](int g0, uint32_t *r, int gw) { tmem_sum_cols(taddr + g0, p.acc_stride, n_acc, r, gw); };
    if (S == 1 && !paired && !norm_out) {
        for (int g0 = g_first; g0 < BN; g0 += g_step) {
            const int gw = min(32, BN - g0);
            uint32_t r[32];
            acc_cols(g0, r, gw);
            if (ok && row < rows_here) {
                float *yb = p.Y + (size_t)(n0 + g0) * p.ldy + o_base + row;
                const int mlim = p.M - (n0 + g0);
                if (add) {
                    float yin[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        yin[j] = (j < gw && j < mlim) ? yb[(size_t)j * p.ldy] : 0.f;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < gw && j < mlim) yb[(size_t)j * p.ldy] = yin[j] + __uint_as_float(r[j]);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < gw && j < mlim) yb[(size_t)j * p.ldy] = __uint_as_float(r[j]);
                }
            }
        }
    } else {
        // partial [BN][128] fp32 in this CTA's (now idle) stage memory
        float *part = reinterpret_cast<float *>(smem_raw + (sbase - smem_u32(smem_raw)));
        for (int g0 = g_first; g0 < BN; g0 += g_step) {
            const int gw = min(32, BN - g0);
            uint32_t r[32];
            acc_cols(g0, r, gw);
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (j < gw) part[(g0 + j) * BM + row] = __uint_as_float(r[j]);
        }
        // Split-K reduction, push style: after a cluster barrier (every rank's
        // MMAs are done, so every rank's stage memory is free), each rank sends
        // every other rank the slice of its partial that holds that rank's
        // columns, by bulk copies into the receiver's buffer that complete on the
        // receiver's mbarrier; each rank then reduces its own columns from its
        // own shared memory, in rank order.
        const uint32_t rank = S > 1 ? c_cluster_rank() : 0u;
        const int span = (BN + S - 1) / S;
        PartSrc ps;
        ps.own = part;
        ps.recv = part + BN * BM;
        ps.rank = (int)rank;
        ps.S = S;
        ps.c_lo = (int)rank * BN / S;
        ps.c_hi = ((int)rank + 1) * BN / S;
        ps.span = span;
        bool okr = ok;
        __syncthreads();                 // the staged row descriptors and the partial, for every warp
        RopePre rpre;
        float4 yv[EPI_PRE];
        // the global operands of the first groups are requested after the
        // cluster barrier, so that they arrive while the slices are exchanged
        auto pre_loads = [&]() {
            if (paired && p.epi == EPI_ROPE_KV) c_rope_pre(p, ps, ok, seg, row0, n0, rows_here, s_rows, rpre);
            if (norm_out) c_norm_pre(p, ps, ok, o_base, rows_here, n0, yv);
        };
        if (S > 1) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");    // part, for the bulk copies
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
            if (warp == 0) {
                if (lane == 0) mbar_expect_tx(recv_bar, (uint32_t)((S - 1) * (ps.c_hi - ps.c_lo) * BM * 4));
                const int t_lo = lane * BN / S, t_hi = (lane + 1) * BN / S;
                if (lane < S && lane != (int)rank && t_hi > t_lo) {      // lane t: rank t's slice
                    const int slot = (int)rank < lane ? (int)rank : (int)rank - 1;
                    const uint32_t src = smem_u32(part + t_lo * BM);
                    const uint32_t dst = c_mapa(smem_u32(ps.recv + slot * span * BM), (uint32_t)lane);
                    asm volatile(
                        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            dst),
                        "r"(src), "r"((uint32_t)((t_hi - t_lo) * BM * 4)), "r"(c_mapa(recv_bar, (uint32_t)lane))
                        : "memory");
                }
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
            pre_loads();
            okr = mbar_wait(recv_bar, 0, &abort_flag, p.status) && ok;
        } else {
            pre_loads();
        }
        if (p.epi == EPI_SWIGLU)
            c_epi_swiglu(p, ps, okr, wt, n0, p.nin.ss ? s_rinv : nullptr);
        else if (paired)
            c_epi_rope(p, ps, okr, seg, row0, n0, rows_here, p.nin.ss ? s_rinv : nullptr, s_rows, rpre);
        else if (norm_out)
            c_reduce_norm(p, ps, okr, wt, o_base, rows_here, n0, yv);
        else {
            // plain reduction of this CTA's columns, float4 = 4 consecutive weight rows of one token
            const int n = (ps.c_hi - ps.c_lo) * (BM / 4);
            for (int e = threadIdx.x; e < n; e += C_THREADS) {
                const int col[1] = {ps.c_lo + e / (BM / 4)}, row[1] = {(e % (BM / 4)) * 4};
                const bool use[1] = {true};
                float4 v[1];
                c_part_sums<1>(ps, col, row, use, v);
                const int m = n0 + col[0], r4 = row[0];
                if (!okr || m >= p.M) continue;
                float4 acc = v[0];
                float *y = p.Y + (size_t)m * p.ldy + o_base + r4;
                if (r4 + 4 <= rows_here && ((reinterpret_cast<uintptr_t>(y) & 15u) == 0)) {
                    if (add) {
                        const float4 yi = *reinterpret_cast<const float4 *>(y);
                        acc.x += yi.x; acc.y += yi.y; acc.z += yi.z; acc.w += yi.w;
                    }
                    *reinterpret_cast<float4 *>(y) = acc;
                } else {
                    const float vv[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (r4 + q < rows_here) {
                            if (add) y[q] = y[q] + vv[q];
                            else y[q] = vv[q];
                        }
                }
            }
        }
        // this CTA's outgoing copies have read its partial before it exits
        if (S > 1 && warp == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) stamp_max(p.stamp, 2);
    if constexpr (pair) {
        // the pair frees its tensor memory together, once both CTAs have read
        // theirs (and, for the odd CTA, once the even one has seen every copy land)
        if (warp == 1) {
            if (lane == 0) {
                mbar_arrive_remote(c_mapa(pexit, my_rank ^ 1u));
                volatile int never = 0;
                mbar_wait_cluster(pexit, 0, &never, p.status);
            }
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                         "r"(p.tmem_cols)
                         : "memory");
        }
    } else if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(p.tmem_cols)
                     : "memory");
    }
}

// One 16 KB packed block per CTA: rows row0..row0+127 of the block's segment,
// columns kb*64 .. kb*64+63, written in the swizzled shared-memory order.
__global__ void pack_kernel(GemmW W, int K, int KB, uint8_t *dst) {
    const long long blk = blockIdx.x;
    const int wt = (int)(blk / KB), kb = (int)(blk - (long long)wt * KB);
    int seg = 0, w = wt;
    while (seg < W.nseg - 1 && w >= (W.rows[seg] + BM - 1) / BM) {
        w -= (W.rows[seg] + BM - 1) / BM;
        ++seg;
    }
    const bf16 *src = static_cast<const bf16 *>(W.w[seg]);
    const int rows = W.rows[seg], row0 = w * BM;
    uint8_t *out = dst + blk * (long long)A_BYTES;
    for (int q = threadIdx.x; q < BM * 8; q += blockDim.x) {
        const int r = q >> 3, c = q & 7;
        const int row = row0 + r, k = kb * BK + c * 8;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (row < rows && k + 8 <= K) v = *reinterpret_cast<const uint4 *>(src + (size_t)row * K + k);
        *reinterpret_cast<uint4 *>(out + r * 128 + ((c ^ (r & 7)) << 4)) = v;
    }
}

// Glu-packed gate/up: block (t, kb) takes gate rows 64t.. into its rows 0..63
// and up rows 64t.. into rows 64..127 (rows past F are 0).
__global__ void pack_glu_kernel(const bf16 *gate, const bf16 *up, int F, int K, int KB, uint8_t *dst) {
    const long long blk = blockIdx.x;
    const int t = (int)(blk / KB), kb = (int)(blk - (long long)t * KB);
    uint8_t *out = dst + blk * (long long)A_BYTES;
    for (int q = threadIdx.x; q < BM * 8; q += blockDim.x) {
        const int r = q >> 3, c = q & 7;
        const int frow = t * 64 + (r & 63), k = kb * BK + c * 8;
        const bf16 *src = r < 64 ? gate : up;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (frow < F && k + 8 <= K) v = *reinterpret_cast<const uint4 *>(src + (size_t)frow * K + k);
        *reinterpret_cast<uint4 *>(out + r * 128 + ((c ^ (r & 7)) << 4)) = v;
    }
}

// Records a host-detected problem in the device status word, in stream order.
__global__ void flag_kernel(int *status, int code) { set_status(status, code); }

struct MapKey {
    const void *ptr;
    long rows, cols, ld, box_rows;
    bool operator==(const MapKey &o) const {
        return ptr == o.ptr && rows == o.rows && cols == o.cols && ld == o.ld &&
               box_rows == o.box_rows;
    }
};
struct MapKeyHash {
    size_t operator()(const MapKey &k) const {
        size_t h = std::hash<const void *>()(k.ptr);
        h ^= std::hash<long>()(k.rows * 1315423911L + k.cols * 2654435761L + k.ld * 97 + k.box_rows);
        return h;
    }
};

}  // namespace

constexpr int MAX_STAMPS = 2048;   // GEMM launches per stamping window
constexpr int MAX_XSTAMPS = 512;   // other stamped launches (attention) per window, slots after the GEMMs'
constexpr int ALL_STAMPS = MAX_STAMPS + MAX_XSTAMPS;

// Sums of the closed stamping windows (device memory).
struct StampAcc {
    unsigned long long span_ns;   // sum over launches of exit - entry
    unsigned long long crit_ns;   // sum over launches of exit - wait
    unsigned long long launches, windows;
    double bytes, wbytes;         // algorithmic bytes of those launches
    double flops, mma_flops;      // 2 M O K of those launches; as issued (x2 for split operands)
    double pre_bytes;             // weight bytes requested before the wait on the previous kernel
};

__global__ void stamp_init_kernel(unsigned long long *st, int n, StampAcc *acc, unsigned long long *slot_acc) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        st[3 * i] = ~0ull;
        st[3 * i + 1] = ~0ull;
        st[3 * i + 2] = 0ull;
        slot_acc[3 * i] = slot_acc[3 * i + 1] = slot_acc[3 * i + 2] = 0ull;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *acc = StampAcc{0, 0, 0, 0, 0.0, 0.0, 0.0, 0.0, 0.0};
}

// A stamp's spans: exit - max(wait, entry) and exit - entry (0, 0 if unused).
__device__ __forceinline__ bool stamp_spans(const unsigned long long *st, unsigned long long &crit,
                                            unsigned long long &span) {
    const unsigned long long e0 = st[0], w0 = st[1], e1 = st[2];
    if (e0 == ~0ull || e1 < e0) return false;
    span = e1 - e0;
    crit = e1 - (w0 <= e1 ? (w0 > e0 ? w0 : e0) : e0);
    return true;
}

// Closes a window of n GEMM launches and xn other launches: adds the GEMMs'
// spans to acc, every launch's spans to its slot's sums in slot_acc, and
// clears the slots for the next window (one block; runs after the window's
// launches).
__global__ void stamp_collect_kernel(unsigned long long *st, int n, int xn, double bytes, double wbytes, double flops,
                                     double mma_flops, double pre_bytes, StampAcc *acc, unsigned long long *slot_acc) {
    __shared__ unsigned long long s_span, s_crit, s_cnt;
    if (threadIdx.x == 0) s_span = s_crit = s_cnt = 0;
    __syncthreads();
    unsigned long long span = 0, crit = 0, cnt = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        unsigned long long c1, s1;
        if (stamp_spans(st + 3 * i, c1, s1)) {
            span += s1;
            crit += c1;
            ++cnt;
            slot_acc[3 * i] += c1;
            slot_acc[3 * i + 1] += s1;
            slot_acc[3 * i + 2] += 1;
        }
        st[3 * i] = ~0ull;
        st[3 * i + 1] = ~0ull;
        st[3 * i + 2] = 0ull;
    }
    for (int j = threadIdx.x; j < xn; j += blockDim.x) {
        const int i = MAX_STAMPS + j;
        unsigned long long c1, s1;
        if (stamp_spans(st + 3 * i, c1, s1)) {
            slot_acc[3 * i] += c1;
            slot_acc[3 * i + 1] += s1;
            slot_acc[3 * i + 2] += 1;
        }
        st[3 * i] = ~0ull;
        st[3 * i + 1] = ~0ull;
        st[3 * i + 2] = 0ull;
    }
    atomicAdd(&s_span, span);
    atomicAdd(&s_crit, crit);
    atomicAdd(&s_cnt, cnt);
    __syncthreads();
    if (threadIdx.x == 0) {
        acc->span_ns += s_span;
        acc->crit_ns += s_crit;
        acc->launches += s_cnt;
        acc->windows += 1;
        acc->bytes += bytes;
        acc->wbytes += wbytes;
        acc->flops += flops;
        acc->mma_flops += mma_flops;
        acc->pre_bytes += pre_bytes;
    }
}

struct GemmPlan {
    float *ws = nullptr;        // stream-K pieces and their tickets
    int *counters = nullptr;
    size_t ws_bytes = WS_BYTES;
    int n_counters = N_COUNTERS;
    bool clear_counters = false;    // tickets are cleared before each launch that uses them
    int num_sms = 148;
    PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    std::unordered_map<MapKey, CUtensorMap, MapKeyHash> maps;
    bool smem_set = false;
    bool cluster_attr_set = false;
    bool profile = false;
    std::vector<cudaEvent_t> ev;
    size_t ev_used = 0;
    double prof_bytes = 0.0, prof_wbytes = 0.0, prof_flops = 0.0, prof_mma = 0.0, prof_pre = 0.0;
    // launch stamps: one slot of 3 per launch of a stamping window
    bool stamp_mode = false, stamp_active = false;
    int stamp_next = 0, xstamp_next = 0, cur_slot = -1;
    double stamp_bytes = 0.0, stamp_wbytes = 0.0, stamp_flops = 0.0, stamp_mma = 0.0, stamp_pre = 0.0;
    unsigned long long *stamps = nullptr;
    StampAcc *stamp_acc = nullptr;
    // per slot: sums of exit - wait, exit - entry and the stamped launches
    // ([ALL_STAMPS][3]); what each slot of the last closed window held
    unsigned long long *slot_acc = nullptr;
    std::vector<GemmSlot> slot_info = std::vector<GemmSlot>(ALL_STAMPS);
    int slot_n = 0, xslot_n = 0;
};

bool gemm_plan_create(GemmPlan **out, int, int, int, int) {
    GemmPlan *p = new GemmPlan();
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&p->num_sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
        delete p;
        return false;
    }
    p->encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    if (cudaMalloc(&p->ws, WS_BYTES) != cudaSuccess ||
        cudaMalloc(&p->counters, sizeof(int) * N_COUNTERS) != cudaSuccess ||
        cudaMalloc(&p->stamps, sizeof(unsigned long long) * 3 * ALL_STAMPS) != cudaSuccess ||
        cudaMalloc(&p->slot_acc, sizeof(unsigned long long) * 3 * ALL_STAMPS) != cudaSuccess ||
        cudaMalloc(&p->stamp_acc, sizeof(StampAcc)) != cudaSuccess) {
        gemm_plan_destroy(p);
        return false;
    }
    cudaMemset(p->counters, 0, sizeof(int) * N_COUNTERS);
    *out = p;
    return true;
}

void gemm_plan_destroy(GemmPlan *p) {
    if (!p) return;
    if (p->ws) cudaFree(p->ws);
    if (p->counters) cudaFree(p->counters);
    if (p->stamps) cudaFree(p->stamps);
    if (p->stamp_acc) cudaFree(p->stamp_acc);
    if (p->slot_acc) cudaFree(p->slot_acc);
    for (cudaEvent_t e : p->ev) cudaEventDestroy(e);
    delete p;
}

bool gemm_profile_enable(GemmPlan *p, int mode) {
    p->profile = mode == 1;
    p->stamp_mode = mode == 2;
    p->stamp_active = false;
    p->ev_used = 0;
    p->prof_bytes = p->prof_wbytes = p->prof_flops = p->prof_mma = p->prof_pre = 0.0;
    if (p->stamp_mode) {
        stamp_init_kernel<<<8, 256>>>(p->stamps, ALL_STAMPS, p->stamp_acc, p->slot_acc);
        if (cudaDeviceSynchronize() != cudaSuccess) return false;
    }
    return true;
}

bool gemm_profile_on(const GemmPlan *p) { return p->profile; }
bool gemm_stamp_on(const GemmPlan *p) { return p->stamp_mode; }

void gemm_stamp_begin(GemmPlan *p) {
    if (!p->stamp_mode) return;
    p->stamp_active = true;
    p->stamp_next = 0;
    p->xstamp_next = 0;
    p->cur_slot = -1;
    p->stamp_bytes = p->stamp_wbytes = p->stamp_flops = p->stamp_mma = p->stamp_pre = 0.0;
}

void gemm_stamp_end(GemmPlan *p, cudaStream_t s) {
    if (!p->stamp_active) return;
    p->stamp_active = false;
    p->slot_n = p->stamp_next;
    p->xslot_n = p->xstamp_next;
    stamp_collect_kernel<<<1, 256, 0, s>>>(p->stamps, p->stamp_next, p->xstamp_next, p->stamp_bytes, p->stamp_wbytes,
                                           p->stamp_flops, p->stamp_mma, p->stamp_pre, p->stamp_acc, p->slot_acc);
    note_launch();
}

// The stamp slot of the next launch (null outside a window or when full).
static unsigned long long *stamp_slot(GemmPlan *p) {
    if (!p->stamp_active || p->stamp_next >= MAX_STAMPS) return nullptr;
    p->cur_slot = p->stamp_next;
    return p->stamps + 3 * (p->stamp_next++);
}

unsigned long long *gemm_stamp_external(GemmPlan *p, int kind, int rows, int outputs, int inner) {
    if (!p || !p->stamp_active || p->xstamp_next >= MAX_XSTAMPS) return nullptr;
    const int i = MAX_STAMPS + p->xstamp_next++;
    p->slot_info[i] = GemmSlot{kind, rows, outputs, inner, 0, 0.0, 0.0, 0.0};
    return p->stamps + 3 * i;
}

int gemm_profile_slots(GemmPlan *p, GemmSlot *out, int max) {
    if (!p->stamp_mode) return 0;
    std::vector<unsigned long long> acc(3 * (size_t)ALL_STAMPS);
    cudaDeviceSynchronize();
    if (cudaMemcpy(acc.data(), p->slot_acc, acc.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost) !=
        cudaSuccess)
        return -1;
    cudaMemset(p->slot_acc, 0, acc.size() * sizeof(unsigned long long));
    int n = 0;
    auto put = [&](int i) {
        if (n >= max) return;
        GemmSlot g = p->slot_info[i];
        g.launches = (long)acc[3 * i + 2];
        g.critical_ms = acc[3 * i] * 1e-6;
        g.ms = acc[3 * i + 1] * 1e-6;
        out[n++] = g;
    };
    for (int i = 0; i < p->slot_n; ++i) put(i);
    for (int j = 0; j < p->xslot_n; ++j) put(MAX_STAMPS + j);
    return n;
}

// Algorithmic bytes and flops of a launch of M token rows x O outputs x K for
// the open profile (events or stamps); nb = 2 for split token operands (two
// MMAs per tile); pre = weight bytes its CTAs request before they wait for
// the previous kernel.
static void account(GemmPlan *p, double weight_bytes, double total_bytes, int M, int O, int K, int nb,
                    double pre) {
    const double fl = 2.0 * M * O * K;
    if (p->cur_slot >= 0) {          // the launch that just took a stamp slot
        p->slot_info[p->cur_slot] = GemmSlot{0, M, O, K, 0, total_bytes, 0.0, 0.0};
        p->cur_slot = -1;
    }
    if (p->profile) {
        p->prof_wbytes += weight_bytes;
        p->prof_bytes += total_bytes;
        p->prof_flops += fl;
        p->prof_mma += fl * nb;
        p->prof_pre += pre;
    }
    if (p->stamp_active) {
        p->stamp_wbytes += weight_bytes;
        p->stamp_bytes += total_bytes;
        p->stamp_flops += fl;
        p->stamp_mma += fl * nb;
        p->stamp_pre += pre;
    }
}

GemmProfile gemm_profile_read(GemmPlan *p) {
    GemmProfile r{};
    if (p->stamp_mode) {
        StampAcc a{};
        cudaDeviceSynchronize();
        cudaMemcpy(&a, p->stamp_acc, sizeof a, cudaMemcpyDeviceToHost);
        cudaMemset(p->stamp_acc, 0, sizeof a);
        r.launches = (long)a.launches;
        r.ms = a.span_ns * 1e-6;
        r.critical_ms = a.crit_ns * 1e-6;
        r.windows = (long)a.windows;
        r.bytes = a.bytes;
        r.weight_bytes = a.wbytes;
        r.flops = a.flops;
        r.mma_flops = a.mma_flops;
        r.prefetch_bytes = a.pre_bytes;
        return r;
    }
    r.bytes = p->prof_bytes;
    r.weight_bytes = p->prof_wbytes;
    r.flops = p->prof_flops;
    r.mma_flops = p->prof_mma;
    r.prefetch_bytes = p->prof_pre;
    for (size_t i = 0; i + 1 < p->ev_used; i += 2) {
        float ms = 0.f;
        cudaEventSynchronize(p->ev[i + 1]);
        if (cudaEventElapsedTime(&ms, p->ev[i], p->ev[i + 1]) == cudaSuccess) r.ms += ms;
        r.launches += 1;
    }
    p->ev_used = 0;
    p->prof_bytes = p->prof_wbytes = p->prof_flops = p->prof_mma = p->prof_pre = 0.0;
    return r;
}

// Tensor map over rows of `cols` bf16, boxes of 64 columns x box_rows rows in the
// 128-byte swizzle (columns and rows past the end read as zeros).
static bool make_map(GemmPlan *p, const void *ptr, long rows, long cols, long ld, long box_rows, CUtensorMap *m) {
    memset(m, 0, sizeof *m);
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    const CUresult r = p->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box,
                                 estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        fprintf(stderr, "msd: cuTensorMapEncodeTiled failed (%d) rows=%ld cols=%ld ld=%ld\n", (int)r, rows, cols, ld);
    return r == CUDA_SUCCESS;
}

// The map of a context buffer, cached.
static const CUtensorMap *get_map(GemmPlan *p, const void *ptr, long rows, long cols, long ld, long box_rows) {
    MapKey key{ptr, rows, cols, ld, box_rows};
    auto it = p->maps.find(key);
    if (it != p->maps.end()) return &it->second;
    CUtensorMap m;
    if (!make_map(p, ptr, rows, cols, ld, box_rows, &m)) return nullptr;
    return &p->maps.emplace(key, m).first->second;
}

// Tensor map over a packed weight buffer as rows of 64 bf16 (blocks of 128 rows
// are the 16 KB pipeline blocks, already in shared-memory order: no swizzle).
static const CUtensorMap *get_wmap(GemmPlan *p, const void *packed, long rows) {
    MapKey key{packed, rows, BK, -1, BM};
    auto it = p->maps.find(key);
    if (it != p->maps.end()) return &it->second;
    CUtensorMap m;
    memset(&m, 0, sizeof m);
    cuuint64_t dims[2] = {(cuuint64_t)BK, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)BK * 2};
    cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)BM};
    cuuint32_t estr[2] = {1, 1};
    if (p->encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(packed), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
        fprintf(stderr, "msd: cuTensorMapEncodeTiled failed for packed weights (%ld rows)\n", rows);
        return nullptr;
    }
    return &p->maps.emplace(key, m).first->second;
}

size_t gemm_pack_bytes(const GemmW &W, int K) {
    long long tiles = 0;
    for (int i = 0; i < W.nseg; ++i) tiles += (W.rows[i] + BM - 1) / BM;
    return (size_t)tiles * ((K + BK - 1) / BK) * A_BYTES;
}

void gemm_pack(const GemmW &W, int K, void *dst, cudaStream_t s) {
    const long long blocks = (long long)(gemm_pack_bytes(W, K) / A_BYTES);
    if (blocks <= 0) return;
    pack_kernel<<<(unsigned)blocks, 256, 0, s>>>(W, K, (K + BK - 1) / BK, static_cast<uint8_t *>(dst));
    note_launch();
}

size_t gemm_pack_glu_bytes(int F, int K) {
    return (size_t)((F + 63) / 64) * ((K + BK - 1) / BK) * A_BYTES;
}

void gemm_pack_glu(const void *gate, const void *up, int F, int K, void *dst, cudaStream_t s) {
    const long long blocks = (long long)(gemm_pack_glu_bytes(F, K) / A_BYTES);
    if (blocks <= 0) return;
    pack_glu_kernel<<<(unsigned)blocks, 256, 0, s>>>(static_cast<const bf16 *>(gate),
                                                      static_cast<const bf16 *>(up), F, K,
                                                      (K + BK - 1) / BK, static_cast<uint8_t *>(dst));
    note_launch();
}

constexpr size_t HALF_SM = 104u * 1024u, FULL_SM = 200u * 1024u;     // ring bytes of two CTAs / one CTA per SM

// How the cluster split-K kernel runs: S K-splits per tile (a cluster), chosen
// so that tiles * S fills the CTAs the SMs hold at once, S <= 8 and >= 2
// K-blocks each. Two CTAs share an SM when three stages fit in half of its
// shared memory (token tiles of up to 64 split rows), otherwise one with up to
// four stages; the split count keeps every split's partial slices within the
// stage memory they reuse.
struct ClusterShape {
    int S, stages, n_acc, acc_stride, tmem_cols, chain;     // chain: K-blocks that one accumulator takes, at most
    bool pair;
    size_t smem;
};

static ClusterShape cluster_shape(int tiles, int BN, int kblocks, int nb, bool packed, int num_sms) {
    size_t stage = A_BYTES + (size_t)nb * BN * BK * 2;
    int per_sm = 3 * stage <= HALF_SM ? 2 : 1;
    // one-plane products over more than 64 rows that leave half of the CTAs unused: one
    // per SM, whose stage memory holds the partials of up to eight splits
    if (nb == 1 && BN > 64 && 2 * tiles <= num_sms) per_sm = 1;
    int stages = (int)((per_sm == 2 ? HALF_SM : FULL_SM) / stage);
    stages = std::max(2, std::min(stages, C_STAGES));
    int S = (per_sm * num_sms) / tiles;
    S = std::max(1, std::min(S, 8));
    // Clusters stay within a GPC, so fewer CTAs run at once the larger they are, and
    // a launch past that runs a second wave. Two CTAs per SM on 152 SMs: 32 clusters
    // of 8, 40 of 6, 56 of 5 and 96 of 3 ran as one, 40 of 7 and 48 of 6 did not
    // (60 x 5120 x 13824: 43.6 us in sevens, 29.6 in sixes; 60 x 6144 x 4096: 22.9
    // in sixes, 14.8 in fives).
    auto one_wave = [&](int c) {
        const int slots = c >= 6 ? 256 : (c >= 4 ? 280 : (c == 3 ? 288 : 304));
        return (long)tiles * c * 304 <= (long)slots * per_sm * num_sms;
    };
    while (S > 1 && !one_wave(S)) --S;
    // The accumulators truncate: the K-blocks take turns over two of them, in one-plane
    // products (msd_linear) over as many as the CTA's TMEM columns hold, and there K is
    // split further where that leaves chains past 16 blocks (17 x 4096 x 11008: 1.1e-6
    // relative in chains of 22, below 0.8e-6 in chains of 3), as far as the partial slices
    // have room: past 64 rows with a CTA on every half SM that is two splits of two
    // accumulators (128 x 11008 x 20000: chains of 43, 2.9e-6)
    int acc_stride = 32;
    while (acc_stride < BN) acc_stride <<= 1;
    const int all_acc = 512 / per_sm / acc_stride;
    const int n_acc = nb == 1 ? all_acc : std::min(kblocks <= 8 ? 4 : 2, all_acc);
    if (nb == 1) S = std::max(S, std::min(8, (kblocks + 16 * n_acc - 1) / (16 * n_acc)));
    // a short K runs in one CTA: four blocks take 3.5 us, 4.6 split and exchanged
    // (16 x 256 x 256), eight 4.5 against 4.7; one-plane products split past n_acc blocks
    if (kblocks <= 8) {
        S = nb == 1 ? (kblocks + n_acc - 1) / n_acc : 1;
        if (!one_wave(S)) S = 1;
    }
    while (S > 1 && kblocks / S < 2) --S;
    // own partial [BN][128] fp32 plus the other ranks' slices of this rank's columns
    while (S > 1 && (size_t)BN * BM * 4 + (size_t)(S - 1) * ((BN + S - 1) / S) * BM * 4 > stages * stage) --S;
    // Two-SM tiles for unsplit launches whose token stage is as large as the
    // weight block (split token rows, 32 or more): each CTA of a pair holds
    // half the token columns, so the ring gets a fourth stage.
    const bool pair = S == 1 && nb == 2 && BN >= 32 && tiles % 2 == 0 && per_sm == 2 && packed;
    if (pair) {
        stage = A_BYTES + (size_t)nb * (BN / 2) * BK * 2;
        stages = std::max(2, std::min((int)(HALF_SM / stage), C_STAGES));
    }
    const int tmem_cols = tmem_columns(n_acc * acc_stride);
    const size_t smem = std::max<size_t>(1024 + (size_t)stages * stage, tmem_smem_floor(tmem_cols));
    const int chain = ((kblocks + S - 1) / S + n_acc - 1) / n_acc;
    return ClusterShape{S, stages, n_acc, acc_stride, tmem_cols, chain, pair, smem};
}

static bool gemm_cluster(GemmPlan *p, const bf16 *X, const bf16 *X_lo, int ldx, int M, int K, const GemmW &W,
                         int tiles, int BN, int kblocks, float *Y, int ldy, int epi, int *status,
                         cudaStream_t s, int O, const GemmFused *fx = nullptr,
                         const GemmNorm *nout = nullptr, const GemmNorm *nin = nullptr) {
    CkParams ck;
    memset(&ck, 0, sizeof ck);
    if (fx) ck.fx = *fx;
    if (nout) ck.nout = *nout;
    if (nin) ck.nin = *nin;
    ck.n_seg = W.nseg;
    int out_off = 0;
    for (int i = 0; i < W.nseg; ++i) {
        ck.seg_rows[i] = W.rows[i];
        ck.seg_tiles[i] = (W.rows[i] + BM - 1) / BM;
        ck.seg_out[i] = out_off;
        out_off += W.rows[i];
    }
    const int nb = X_lo ? 2 : 1;
    const ClusterShape g = cluster_shape(tiles, BN, kblocks, nb, W.packed != nullptr, p->num_sms);
    const int S = g.S, stages = g.stages, BNs = g.pair ? BN / 2 : BN;
    const bool pair = g.pair;
    ck.M = M;
    ck.kblocks = kblocks;
    ck.BN = BN;
    ck.n_tiles_n = 1;
    ck.splits = S;
    ck.stages = stages;
    ck.has_lo = X_lo ? 1 : 0;
    ck.n_acc = g.n_acc;
    ck.acc_stride = g.acc_stride;
    ck.tmem_cols = g.tmem_cols;
    ck.wpacked = static_cast<const bf16 *>(W.packed);
    ck.Y = Y;
    ck.ldy = ldy;
    ck.epi = epi;
    ck.status = status;
    // a caller's row-major weight and rows: maps of this call alone
    const bool raw = !W.packed;
    CUtensorMap rawx, raww;
    const CUtensorMap *mx = raw ? (make_map(p, X, M, K, ldx, BNs, &rawx) ? &rawx : nullptr)
                                : get_map(p, X, M, K, ldx, BNs);
    ck.stamp = stamp_slot(p);
    const CUtensorMap *mxl = X_lo ? get_map(p, X_lo, M, K, ldx, BNs) : mx;
    const CUtensorMap *mw = raw    ? (make_map(p, W.w[0], O, K, K, BM, &raww) ? &raww : nullptr)
                            : pair ? get_wmap(p, W.packed, (long)tiles * kblocks * BM)
                                   : mx;
    if (!mx || !mxl || !mw) {
        flag_kernel<<<1, 1, 0, s>>>(status, ST_RANGE);
        return false;
    }
    if (!p->cluster_attr_set) {
        auto set = [](const void *f) {
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(1024 + FULL_SM));
        };
        set((const void *)gemm_cluster_kernel<false, false>);
        set((const void *)gemm_cluster_kernel<true, false>);
        set((const void *)gemm_cluster_kernel<false, true>);
        p->cluster_attr_set = true;
    }
    const bool prof = p->profile;
    if (prof) {
        while (p->ev.size() < p->ev_used + 2) {
            cudaEvent_t e;
            cudaEventCreate(&e);
            p->ev.push_back(e);
        }
        cudaEventRecord(p->ev[p->ev_used], s);
    }
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof lc);
    lc.gridDim = dim3((unsigned)tiles, 1, (unsigned)S);
    lc.blockDim = dim3(C_THREADS);
    lc.dynamicSmemBytes = g.smem;
    lc.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = pair ? 2u : 1u;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = (unsigned)S;
    lc.attrs = at;
    lc.numAttrs = 2;
    const auto kernel = raw ? gemm_cluster_kernel<false, true>
                            : (pair ? gemm_cluster_kernel<true, false> : gemm_cluster_kernel<false, false>);
    const bool launched = cudaLaunchKernelEx(&lc, kernel, *mx, *mxl, *mw, ck) == cudaSuccess;
    if (!launched) {
        cudaGetLastError();
        flag_kernel<<<1, 1, 0, s>>>(status, ST_RANGE);
        fprintf(stderr, "msd: cluster GEMM launch failed (M=%d K=%d O=%d S=%d)\n", M, K, O, S);
    }
    note_launch();
    if (prof) {
        cudaEventRecord(p->ev[p->ev_used + 1], s);
        p->ev_used += 2;
    }
    const double wb = (double)O * K * 2.0;
    double yb = (double)M * O * 4.0 * (epi == EPI_ADD ? 2 : 1);
    if (epi == EPI_SWIGLU) yb = (double)M * fx->F * 2.0 * nb;
    if (epi == EPI_ROPE_KV) yb = (double)M * O * 2.0 * nb;
    double pre = 0.0;      // the blocks each split requests before its wait (padded rows included)
    for (int z = 0; z < S; ++z)
        pre += (double)tiles * std::min(stages, (int)((long long)(z + 1) * kblocks / S - (long long)z * kblocks / S)) *
               A_BYTES;
    if (raw) pre = 0.0;
    account(p, wb, wb + (double)M * K * 2.0 * nb + yb, M, O, K, nb, std::min(pre, wb));
    return launched;
}

// The persistent stream-K GEMM (many token rows). fx: EPI_SWIGLU writes
// act = silu(g) * u from glu-packed gate/up weights instead of Y.
static bool gemm_persist(GemmPlan *p, const bf16 *X, const bf16 *X_lo, int ldx, int M, int K, const GemmW &W,
                         int O, float *Y, int ldy, int epi, const GemmFused *fx, int *status, cudaStream_t s);

bool gemm_bf16_fused(GemmPlan *p, const bf16 *X, const bf16 *X_lo, int ldx, int M, int K, const GemmW &W,
                     int O, const GemmFused &fx, int *status, cudaStream_t s, const GemmNorm *norm_in) {
    if (M <= 0 || !W.packed || W.nseg < 1) return false;
    if (fx.epi == EPI_SWIGLU && (W.nseg != 1 || W.rows[0] != glu_rows(fx.F) || fx.F % 4)) return false;
    if (M > 128) {
        // many token rows: the persistent GEMM with SwiGLU fused into its
        // epilogue (RoPE/KV stays a separate kernel there: fused, its
        // per-column gathers outlasted the main loop, measured slower)
        if (fx.epi != EPI_SWIGLU || norm_in || !fx.act) return false;
        gemm_persist(p, X, X_lo, ldx, M, K, W, O, nullptr, 0, EPI_SWIGLU, &fx, status, s);   // (or flags the status)
        return true;
    }
    if (fx.epi == EPI_ROPE_KV &&
        (W.nseg != 3 || (fx.hd != 64 && fx.hd != 128) || fx.nh * fx.hd != W.rows[0] ||
         W.rows[1] != W.rows[0] || W.rows[2] != W.rows[0]))
        return false;
    if (fx.epi != EPI_SWIGLU && fx.epi != EPI_ROPE_KV) return false;
    int tiles = 0;
    for (int i = 0; i < W.nseg; ++i) tiles += (W.rows[i] + BM - 1) / BM;
    const int BN = ((M + 15) / 16) * 16;
    if (norm_in && (!norm_in->ss || norm_in->parts <= 0 || norm_in->parts > norm_in->ld || BN > 128))
        return false;
    gemm_cluster(p, X, X_lo, ldx, M, K, W, tiles, BN, (K + BK - 1) / BK, nullptr, 0, fx.epi, status, s, O, &fx,
                 nullptr, norm_in);
    return true;
}

bool gemm_bf16(GemmPlan *p, const bf16 *X, const bf16 *X_lo, int ldx, int M, int K, const GemmW &W, int O,
               float *Y, int ldy, int epi, int *status, cudaStream_t s, const GemmNorm *norm_out) {
    if (M <= 0 || O <= 0) return true;
    if (norm_out && (M > 128 || !W.packed || W.nseg != 1 || !norm_out->ss || !norm_out->xg || !norm_out->g ||
                     (O + BM - 1) / BM > norm_out->ld || O % 4 || ldy % 4))
        return false;
    if (!W.packed && W.nseg != 1) return false;
    if (M <= 128) {
        int tiles = 0;
        for (int i = 0; i < W.nseg; ++i) tiles += (W.rows[i] + BM - 1) / BM;
        gemm_cluster(p, X, X_lo, ldx, M, K, W, tiles, ((M + 15) / 16) * 16, (K + BK - 1) / BK, Y, ldy, epi,
                     status, s, O, nullptr, norm_out);
        return true;
    }
    gemm_persist(p, X, X_lo, ldx, M, K, W, O, Y, ldy, epi, nullptr, status, s);
    return true;
}

// How the persistent GEMM cuts its work: token tiles of BN columns, G CTA
// pairs, T_sk of the T_all tiles stream-K, the others whole in chunks of
// kb_chunk K-blocks.
struct PersistShape {
    int BN, nt, G, T_all, T_sk, dp_rounds, kb_chunk, n_acc, n_rot;
    int stages, acc_stride, tmem_cols;
    int chain;                          // K-blocks that one accumulator takes, at most
    uint32_t stage_bytes, stg_off;      // a ring stage; where the SwiGLU staging tile starts
    size_t smem;
};
constexpr uint32_t P_BUDGET = 220u * 1024u;     // ring and staging bytes of a CTA
constexpr int P_STAGES = 6;
constexpr int P_CHAIN = 32, P_CHUNK_CHAIN = 24;

// Clocks, measured at 333 to 1024 rows and K = 4096, 11008. A K-block of a 256 x
// BN tile takes 2.08 nb BN (4% above the MMAs' own time: 0.35 us at 160 columns
// and two planes, 0.48 us at 224), and not less than 420 + 0.8 nb BN (0.26 to
// 0.32 us at 96 to 112, by the clock the power limit leaves). For each count of token tiles that keeps BN <= 256: whole tiles
// alone take ceil(T / G) rounds; with the remainder cut stream-K the units are
// even, but the pieces' round trip through the workspace then costs 330 BN
// where every tile is cut (O at 640 rows, 224 columns: 68 us against 40 in whole
// tiles), about 180 BN where whole tiles follow to hide part of it.
// The accumulators truncate, so the error grows with the chain of K-blocks that one
// takes (one-plane products of 4096 terms: 2.2e-6 relative in chains of 32 to 40
// blocks, 4.4e-6 in one of 64). The K-blocks of an item take turns over as many
// accumulators as there is room for: 512 TMEM columns where a pair has one item,
// half of them where its next item runs beside the epilogue. One-plane products
// (msd_linear), which have no other error, are also cut into narrower tiles while
// one round holds them: a K-block of 32 columns takes no longer than one of 96, and
// 16 accumulators fit (1245 x 3664 x 129: 27.3 us and 9.0e-7 with tiles of 64 columns
// or more, 23.2 us and 1.3e-7; 1000 x 512 x 1024: 15.0 to 12.9 us). Where a pair has
// several whole tiles, chunks of K are added to Y one after another, with at most 24
// blocks in every accumulator; a lone tile takes up to 32. Tiles whose pieces would put
// more than 32 into one stay whole (500 x 11008 x 14336 in pieces of 82 blocks: 3.0e-6
// and 158 us, 1.4e-6 and 186 us whole; 576 x 11008 x 9728, 86: 3.7e-6 and 113 us,
// 1.4e-6 and 126 us; the pieces in chunks added to the workspace: 209 and 144 us).
static PersistShape persist_shape(int tiles, int M, int K, int nb, bool glu, int pairs, size_t ws_bytes,
                                  int n_counters) {
    const int kblocks = (K + BK - 1) / BK, wt = (tiles + 1) / 2;
    PersistShape best{};
    double best_cost = 1e300;
    for (int nt = (M + 255) / 256, n = 0; n < 6 || (nb == 1 && (long long)wt * nt <= pairs); ++nt, ++n) {
        const int BN = ((M + nt - 1) / nt + 15) / 16 * 16;
        if (n > 0 && BN < (nb == 1 ? 32 : 64)) break;
        const long long T = (long long)wt * nt;
        const double tk = std::max(2.08 * nb * BN, 420.0 + 0.8 * nb * BN);
        // at least 4 K-blocks a pair
        const long long G = std::max<long long>(1, std::min<long long>(pairs, T * kblocks / 4));
        int stride = 32;
        while (stride < BN) stride <<= 1;
        const int most = nb == 1 ? 16 : 4;
        const bool chunked = nb == 1 && !glu;
        const bool lone = T <= G && (!chunked || (kblocks + P_CHAIN - 1) / P_CHAIN <= 512 / stride);    // one item a pair
        const int n_acc = lone ? 1 : 2, n_rot = std::min(512 / n_acc / stride, most);
        const int n_ch = chunked && !lone ? (kblocks + P_CHUNK_CHAIN * n_rot - 1) / (P_CHUNK_CHAIN * n_rot) : 1;
        const int chunk = (kblocks + n_ch - 1) / n_ch;
        PersistShape g{BN, nt, (int)G, (int)T, 0, (int)((T + G - 1) / G), chunk, n_acc, n_rot};
        g.chain = (chunk + n_rot - 1) / n_rot;
        double cost = g.dp_rounds * tk * kblocks;
        int rounds = (int)(T / G), T_sk = (int)(T - rounds * G);
        if (T_sk > 0) {
            const bool few = rounds > 0 && G > 8LL * T_sk;
            // a few short-K tiles join a round of whole tiles: every tile in two
            // or three pieces, fixed up at the end of the launch
            if (few && kblocks <= 64 && !glu) {
                --rounds;
                T_sk += (int)G;
            }
            const double sk = T * tk * kblocks / G + (rounds == 0 ? 330.0 : 180.0) * BN;
            const int sk_acc = chunked && rounds == 0 ? 1 : 2, sk_rot = std::min(512 / sk_acc / stride, most);
            const long long piece = std::min<long long>(kblocks, (T_sk * (long long)kblocks + G - 1) / G);
            const int sk_chain = (int)((piece + sk_rot - 1) / sk_rot);
            // (every pair holds a unit, and the pieces and tickets have their place)
            if (sk < cost && (long long)T_sk * kblocks >= G && 16ull * G * BN * BM <= ws_bytes &&
                2LL * T_sk <= n_counters && (!chunked || sk_chain <= P_CHAIN)) {
                g.T_sk = T_sk;
                g.dp_rounds = rounds;
                g.n_acc = sk_acc;
                g.n_rot = sk_rot;
                g.chain = std::max(sk_chain, rounds > 0 ? (chunk + sk_rot - 1) / sk_rot : 0);
                cost = sk;
            }
        }
        if (cost < best_cost) {
            best_cost = cost;
            best = g;
        }
    }
    // the fused SwiGLU epilogue takes 16 KB of staging from the ring's budget
    const uint32_t stg_bytes = glu ? 32u * BM * 4u : 0u;
    best.stage_bytes = A_BYTES + (uint32_t)nb * (best.BN / 2) * BK * 2;
    best.stages = std::max(2, std::min((int)((P_BUDGET - stg_bytes) / best.stage_bytes), P_STAGES));
    best.stg_off = (uint32_t)(1024 + (size_t)best.stages * best.stage_bytes);
    best.acc_stride = 32;
    while (best.acc_stride < best.BN) best.acc_stride <<= 1;
    best.tmem_cols = tmem_columns(best.n_acc * best.n_rot * best.acc_stride);
    best.smem = std::max<size_t>(best.stg_off + stg_bytes, tmem_smem_floor(best.tmem_cols));
    return best;
}

static bool gemm_persist(GemmPlan *p, const bf16 *X, const bf16 *X_lo, int ldx, int M, int K, const GemmW &W,
                         int O, float *Y, int ldy, int epi, const GemmFused *fx, int *status, cudaStream_t s) {
    const bool glu = fx && fx->epi == EPI_SWIGLU;
    PkParams pk;
    memset(&pk, 0, sizeof pk);
    pk.n_seg = W.nseg;
    int tiles = 0, out_off = 0;
    for (int i = 0; i < W.nseg; ++i) {
        pk.seg_rows[i] = W.rows[i];
        pk.seg_tiles[i] = (W.rows[i] + BM - 1) / BM;
        pk.seg_out[i] = out_off;
        out_off += W.rows[i];
        tiles += pk.seg_tiles[i];
    }
    const int nb = X_lo ? 2 : 1;
    const PersistShape g = persist_shape(tiles, M, K, nb, glu, p->num_sms / 2, p->ws_bytes, p->n_counters);
    const int BN = g.BN, nt = g.nt, kblocks = (K + BK - 1) / BK, G = g.G;
    const int stages = g.stages;
    const long long units = (long long)g.T_sk * kblocks;
    const long long all_units = (long long)g.T_all * kblocks;
    pk.M = M;
    pk.kblocks = kblocks;
    pk.BN = BN;
    pk.n_tiles_n = nt;
    pk.stages = stages;
    pk.acc_stride = g.acc_stride;
    pk.n_acc = g.n_acc;
    pk.n_rot = g.n_rot;
    pk.tmem_cols = g.tmem_cols;
    pk.grid = G;
    pk.tiles = tiles;
    pk.units = units;
    pk.T_sk = g.T_sk;
    pk.dp_rounds = g.dp_rounds;
    pk.T_all = g.T_all;
    pk.kb_chunk = g.kb_chunk;
    pk.Y = Y;
    pk.ldy = ldy;
    pk.epi = epi;
    pk.ws = p->ws;
    pk.counters = p->counters;
    pk.status = status;
    pk.has_lo = X_lo ? 1 : 0;
    if (glu) {
        pk.epi = EPI_SWIGLU;
        pk.act = fx->act;
        pk.F = fx->F;
        pk.lo = fx->lo;
        pk.stg_off = g.stg_off;
    }
    const bool raw = !W.packed;
    CUtensorMap rawx, raww;
    const CUtensorMap *mx = raw ? (make_map(p, X, M, K, ldx, BN / 2, &rawx) ? &rawx : nullptr)
                                : get_map(p, X, M, K, ldx, BN / 2);
    const CUtensorMap *mxl = X_lo ? get_map(p, X_lo, M, K, ldx, BN / 2) : mx;
    const CUtensorMap *mw = raw ? (make_map(p, W.w[0], O, K, K, BM, &raww) ? &raww : nullptr)
                                : get_wmap(p, W.packed, (long)tiles * kblocks * BM);
    if (!mx || !mxl || !mw) {
        flag_kernel<<<1, 1, 0, s>>>(status, ST_RANGE);
        return false;
    }
    pk.stamp = stamp_slot(p);
    if (!p->smem_set) {
        cudaFuncSetAttribute(gemm_persist_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(P_BUDGET + 1024));
        cudaFuncSetAttribute(gemm_persist_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(P_BUDGET + 1024));
        p->smem_set = true;
    }
    if (p->clear_counters && g.T_sk > 0 &&
        cudaMemsetAsync(p->counters, 0, sizeof(int) * 2 * g.T_sk, s) != cudaSuccess)
        return false;
    const bool prof = p->profile;
    if (prof) {
        while (p->ev.size() < p->ev_used + 2) {
            cudaEvent_t e;
            cudaEventCreate(&e);
            p->ev.push_back(e);
        }
        cudaEventRecord(p->ev[p->ev_used], s);
    }
    // Programmatic dependent launch: the kernel may start while the previous
    // kernel on the stream finishes; it waits (griddepcontrol.wait) before
    // touching anything but weights.
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof lc);
    lc.gridDim = dim3((unsigned)(2 * G));
    lc.blockDim = dim3(P_THREADS);
    lc.dynamicSmemBytes = g.smem;
    lc.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 2;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 2;
    const auto kernel = raw ? gemm_persist_kernel<true> : gemm_persist_kernel<false>;
    const bool launched = cudaLaunchKernelEx(&lc, kernel, *mx, *mxl, *mw, pk) == cudaSuccess;
    if (!launched) {
        cudaGetLastError();
        flag_kernel<<<1, 1, 0, s>>>(status, ST_RANGE);
        fprintf(stderr, "msd: persistent GEMM launch failed (M=%d K=%d O=%d)\n", M, K, O);
    }
    note_launch();
    if (prof) {
        cudaEventRecord(p->ev[p->ev_used + 1], s);
        p->ev_used += 2;
    }
    const double wb = (double)O * K * 2.0;
    account(p, wb, wb + (double)M * K * 2.0 * nb +
                       (glu ? (double)M * fx->F * 2.0 * nb : (double)M * O * 4.0 * (epi == EPI_ADD ? 2 : 1)),
            M, O, K, nb, raw ? 0.0 : std::min(wb, 2.0 * G * std::min<long long>(stages, all_units / G) * A_BYTES));
    return launched;
}

}  // namespace msd

// ---------------------------------------------------------------------------
// Allocation-free GEMM entry point (msd_linear_noalloc in include/msd.h).
//
// Some callers cannot call cudaMalloc: a host program whose device memory is
// entirely owned by its own pool allocator, code that runs where an allocation
// would synchronise the device or is not permitted, or a plug-in that is handed
// buffers but no allocator. For them the split-K scratch of the tensor-core
// GEMM lives in one file-scope device array, loaded with the library and held
// by every GPU that loads it until the process exits.
//
// Layout of the array: a status word (padded to 256 bytes), NOALLOC_COUNTERS
// int tile tickets, then the fp32 pieces of stream-K tiles (NOALLOC_PARTIAL_BYTES).
// In host code the array's name is only a host-side stand-in; the device address
// comes from cudaGetSymbolAddress, taken once per device (with that device
// current) on the first call made on it. Every call shares the array and it
// keeps the last call's contents: the tickets are cleared on the caller's
// stream before each launch that uses them, and calls that overlap on the GPU
// race on the array. A product of up to 128 rows splits K over a cluster and
// needs none of it; with more rows, a shape whose pieces would not fit runs in
// whole tiles.
// The status word that kernels set is a word of this library's own host memory,
// page-locked on the first call and written by the GPU in place, so that a call
// reads it after a stream synchronisation alone (a copy back to pageable memory
// took most of a small call: 66 us for 17 x 4096 x 11008 before, with the rows'
// kernel at 30); where it cannot be mapped, the array's word is copied back.
// ---------------------------------------------------------------------------
namespace msd {
namespace {
constexpr size_t NOALLOC_STATUS_BYTES = 256;
constexpr int NOALLOC_COUNTERS = 4096;
constexpr size_t NOALLOC_PARTIAL_BYTES = 16ull << 20;
constexpr size_t NOALLOC_BYTES = NOALLOC_STATUS_BYTES + NOALLOC_COUNTERS * sizeof(int) + NOALLOC_PARTIAL_BYTES;
constexpr int NOALLOC_MAX_DEVICES = 64;
// 65535 token tiles of 256 rows: with up to 2^15 pairs of weight tiles (8 million
// outputs) the launch's tile counts stay within an int.
constexpr long NOALLOC_MAX_ROWS = 65535L * 256;
}  // namespace

static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

namespace {
struct NoAllocDevice {
    bool ready = false;
    unsigned char *scratch = nullptr;   // device address of g_noalloc_scratch
    GemmPlan *plan = nullptr;           // maps nothing and owns nothing: scratch is the array's
    int *status = nullptr;              // device address of the status word
    volatile int *host = nullptr;       // the same word in host memory (null: copied back)
    int status_copy = 0;
};
std::mutex g_noalloc_mu;
NoAllocDevice g_noalloc_dev[NOALLOC_MAX_DEVICES];
alignas(4096) unsigned char g_noalloc_host[NOALLOC_MAX_DEVICES * 64];   // one cache line per device

// One-time set-up of the current device (caller holds g_noalloc_mu).
bool noalloc_setup(int dev) {
    NoAllocDevice &d = g_noalloc_dev[dev];
    if (d.ready) return true;
    void *ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return false;
    if (!d.plan) d.plan = new GemmPlan();
    GemmPlan *p = d.plan;
    if (cudaDeviceGetAttribute(&p->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
        return false;
    p->encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    d.scratch = static_cast<unsigned char *>(ptr);
    p->counters = reinterpret_cast<int *>(d.scratch + NOALLOC_STATUS_BYTES);
    p->ws = reinterpret_cast<float *>(d.scratch + NOALLOC_STATUS_BYTES + NOALLOC_COUNTERS * sizeof(int));
    p->ws_bytes = NOALLOC_PARTIAL_BYTES;
    p->n_counters = NOALLOC_COUNTERS;
    p->clear_counters = true;
    d.status = reinterpret_cast<int *>(d.scratch);
    void *mapped = nullptr;
    const cudaError_t e = cudaHostRegister(g_noalloc_host, sizeof g_noalloc_host,
                                           cudaHostRegisterMapped | cudaHostRegisterPortable);
    if ((e == cudaSuccess || e == cudaErrorHostMemoryAlreadyRegistered) &&
        cudaHostGetDevicePointer(&mapped, g_noalloc_host, 0) == cudaSuccess && mapped) {
        d.status = reinterpret_cast<int *>(static_cast<unsigned char *>(mapped) + 64 * dev);
        d.host = reinterpret_cast<volatile int *>(g_noalloc_host + 64 * dev);
    }
    cudaGetLastError();
    d.ready = true;
    return true;
}

// Waits for the work queued before on `s`, then takes (and clears) the status word.
cudaError_t noalloc_take_status(NoAllocDevice &d, cudaStream_t s, int *code) {
    if (!d.host) {
        cudaError_t e = cudaMemcpyAsync(&d.status_copy, d.status, sizeof(int), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        *code = e == cudaSuccess ? d.status_copy : 0;
        return e == cudaSuccess && *code ? cudaMemsetAsync(d.status, 0, sizeof(int), s) : e;
    }
    const cudaError_t e = cudaStreamSynchronize(s);
    *code = e == cudaSuccess ? *d.host : 0;
    if (*code) *d.host = 0;
    return e;
}
}  // namespace

// Device address of the no-alloc status word on the current device (set-up
// included); null if the set-up failed.
int *noalloc_status_word() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return nullptr;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!noalloc_setup(dev)) return nullptr;
    return g_noalloc_dev[dev].status;
}

// Test hook of the bounded waits: one CTA waits on an mbarrier that nothing
// arrives at, through the same bounded wait as the GEMM kernels, gives up
// after limit_ns and records ST_TIMEOUT in *status. No copy or MMA is in
// flight while it waits.
__global__ void wait_probe_kernel(int *status, unsigned long long limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ volatile int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_wait(smem_u32(&bar), 0, &abort_flag, status, limit_ns);
    }
}

bool launch_wait_probe(int *status, long long limit_ns, cudaStream_t s) {
    wait_probe_kernel<<<1, 32, 0, s>>>(status, (unsigned long long)limit_ns);
    note_launch();
    return cudaGetLastError() == cudaSuccess;
}

}  // namespace msd

extern "C" msd_status msd_linear_noalloc(const void *x, int32_t ldx, int32_t m, int32_t k,
                                         const void *w, int32_t o, float *y, int32_t ldy,
                                         int32_t accumulate, void *stream) {
    using namespace msd;
    constexpr msd_status OK = MSD_OK, INVALID = MSD_ERR_INVALID, CAPACITY = MSD_ERR_CAPACITY,
                         CUDA_ERR = MSD_ERR_CUDA;
    if (!x || !w || !y || m <= 0 || k <= 0 || o <= 0 || ldx < k || ldy < o) return INVALID;
    if (ldx % 8 || k % 8) return INVALID;
    if ((long)m > NOALLOC_MAX_ROWS) return CAPACITY;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return CUDA_ERR;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!noalloc_setup(dev)) return CUDA_ERR;
    NoAllocDevice &d = g_noalloc_dev[dev];
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // The status word left by earlier launches on this device (a bounded wait
    // that ran out), once the work queued before on `stream` has finished; a set
    // word is cleared and reported once.
    int code = 0;
    if (noalloc_take_status(d, s, &code) != cudaSuccess) return CUDA_ERR;
    if (code != 0) return MSD_ERR_DEVICE;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(w)) & 15) return INVALID;
    const GemmW W{{w, nullptr, nullptr}, {o, 0, 0}, 1, nullptr};
    const bf16 *X = static_cast<const bf16 *>(x);
    const int epi = accumulate ? EPI_ADD : EPI_STORE;
    const bool ok = m <= 128 ? gemm_cluster(d.plan, X, nullptr, ldx, m, k, W, (o + BM - 1) / BM, (m + 15) / 16 * 16,
                                            (k + BK - 1) / BK, y, ldy, epi, d.status, s, o)
                             : gemm_persist(d.plan, X, nullptr, ldx, m, k, W, o, y, ldy, epi, nullptr, d.status, s);
    return ok && cudaGetLastError() == cudaSuccess ? OK : CUDA_ERR;
}

extern "C" msd_status msd_test_gemm_shape(int32_t m, int32_t k, int32_t o, int32_t planes, int32_t glu, int32_t sms,
                                          msd_gemm_shape *out) {
    using namespace msd;
    if (m <= 0 || k <= 0 || o <= 0 || (planes != 1 && planes != 2) || (glu && planes == 1) || sms < 2 || !out)
        return MSD_ERR_INVALID;
    const int kblocks = (k + BK - 1) / BK, tiles = (o + BM - 1) / BM;
    if (m <= 128) {
        const ClusterShape g = cluster_shape(tiles, (m + 15) / 16 * 16, kblocks, planes, planes == 2, sms);
        *out = msd_gemm_shape{tiles * g.S, g.pair ? 2 : g.S, (int32_t)g.smem, g.tmem_cols, g.chain, 1, 0};
    } else {
        const PersistShape g = persist_shape(tiles, m, k, planes, glu != 0, sms / 2, WS_BYTES, N_COUNTERS);
        const int chunks = (kblocks + g.kb_chunk - 1) / g.kb_chunk;
        *out = msd_gemm_shape{2 * g.G, 2, (int32_t)g.smem, g.tmem_cols, g.chain, g.dp_rounds > 0 ? chunks : 0, g.T_sk};
    }
    return MSD_OK;
}
