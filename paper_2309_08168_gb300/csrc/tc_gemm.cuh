// tc_gemm.cuh - the prompt-encoding GEMM on the 5th-generation tensor cores
// (tcgen05, sm_103a), with the fused epilogues of the prefill:
//     D[feature][token] = W[feature][K] * (X_hi + X_lo)[token][K]^T.
//
// The prefill (Sec. 3.1: the prompt is encoded before Algorithms 1 / 2 start
// decoding) runs every prompt row through the full model at once, so its
// projections are dense GEMMs over 17 .. 2048 token rows: bound by HBM (the
// weights) below ~140 rows, by the tensor cores above.
//
// Weights are the M side and tokens the N side: M is always full (a pair of
// CTAs holds 256 weight rows) and N can be any multiple of 32 up to 256, so a
// ragged token count is padded to 32 rows per tile instead of a full tile, and
// the epilogue's lanes are consecutive features (coalesced rows).  Two CTAs of
// a cluster work on one tile (tcgen05 cta_group::2): each stages its own 128
// weight rows and half of the token rows, so a k block of 64 costs 16 KB +
// nt * 128 bytes of shared-memory traffic per CTA for 2 * 128 * nt * 64
// multiply-adds (hi and lo), 25 % less L2 -> SM traffic than a CTA alone with a
// 128 x 256 tile.  Per CTA:
//   warp 16            : TMA producer, a ring of S stages (as many as fit);
//                        the copies of both CTAs complete on the even CTA's
//                        barrier;
//   warp 17            : (even CTA) MMA issuer: tcgen05.mma kind::f16 (bf16 x
//                        bf16 -> fp32), M = 256, N = nt, K = 16, eight per k
//                        block (four k steps x hi and lo), into one of two
//                        TMEM accumulators of up to 256 columns;
//   warps 0-15         : epilogue of a finished accumulator while the next one
//                        fills.  Warp w reads TMEM lanes 32 (w mod 4) .. +31 and
//                        the columns of quarter w / 4, 16 at a time.
// The grid is persistent, one CTA pair per two SMs.  Work = tiles (256 features
// x nt tokens; token tiles fastest, so pairs that share weights run together)
// x k blocks of 64.  A remainder that would leave a wave of tiles part empty
// is split over all pairs by k block instead (TcSched below).
//
// Operands are K-major with the canonical 128-byte-swizzle layout that TMA
// writes: row r of a tile at r * 128 bytes, 8-row groups 1024 bytes apart
// (the descriptor's stride byte offset), each k step of 16 moves the start
// address by 32 bytes inside the swizzle row.
//
// Precision: as in the decode forwards, the fp32 activations enter as bf16
// hi = rn(x) and lo = rn(x - hi); W * hi + W * lo accumulate in the same fp32
// TMEM accumulator (~16 mantissa bits of x).
//
// Every wait is bounded (~2 s): on a timeout the thread records the error
// code and stops waiting; the CTAs then give copies and MMAs in flight time to
// finish, free their TMEM and return.
#pragma once

#include "ssd_internal.cuh"

namespace ssd {
namespace tc {

constexpr int kBK = 64;            // k per stage: 128 bytes of bf16 = one swizzle row
constexpr int kFeat = 256;         // weight rows per tile (two CTAs x 128 TMEM lanes)
constexpr int kMaxTok = 256;       // token columns per tile (TMEM columns of one accumulator)
constexpr int kEpiWarps = 16;
constexpr int kThreads = (kEpiWarps + 2) * 32;
constexpr int kATile = 128 * kBK * 2;         // 16 KB: this CTA's weight rows of a k block
constexpr int kRingBytes = 224 * 1024;
constexpr int kMaxStages = 11;                // 20 KB stages at 32 tokens
constexpr size_t kSmemBytes = 1024 + (size_t)kRingBytes;
constexpr int kTmemCols = 512;                // two accumulators of 256 columns
constexpr unsigned long long kWaitNs = 2000000000ull;
constexpr int kErrTimeout = 1;
constexpr int kMinSplit = 8;                  // k blocks a pair gets at least when tiles are split

// epilogues of the prefill GEMMs
enum TcEpi { TC_RESID = 1, TC_SWIGLU = 2, TC_QKV = 3 };

// How tiles are spread over the pairs: the first n_split tiles by k block over
// split_pairs pairs, in contiguous ranges (a tile cut by a range end is summed
// by the pair holding its first k blocks, in range order; the others leave
// their partial sums in the workspace), the others whole, pair by pair.
struct TcSched {
    int n_tiles, n_split, split_pairs, pairs, n_tt;
};

struct TcArgs {
    // TMA maps.  Weights: RESID {K, N}, box {64, 128}; SWIGLU gate and up in one
    // map {K, 16, 2, N / 16}, box {64, 16, 2, 4} (the lower matrix in memory
    // first: swapped = 1 if that is up), or [1] != nullptr: gate, up {K, N}, box
    // {64, 16} each; QKV wq, wk, wv as {K, 16, 2, hd / 32, heads}, box = 128 rows, or
    // (ROWS16) {K, N}, box {64, 16}.
    // Tokens: planes as {K, rows, 2}, box {64, nt / 2, 2}.
    const void* tm_w[3];
    const void* tm_x;
    int rows;              // valid token rows
    int nt;                // token rows per tile: a multiple of 32, at most 256
    int n_kb;              // ceil(K / 64)
    int stages;            // ring depth
    int N;                 // output features (SWIGLU: ffn)
    int swapped;           // SWIGLU: lanes 0-15 hold up, 16-31 gate
    TcSched sched;
    float* ws;             // [pairs][2][256][128] fp32 partial sums
    unsigned* flags;       // [pairs][2][16] epoch of the partial sums a warp left
    unsigned epoch;        // of this launch, never 0 or an earlier one
    float* out;            // RESID: residual h [rows][N] (+= D)
    bf16* act_hi;          // SWIGLU: planes [rows][ffn] of silu(gate) * up
    bf16* act_lo;
    // QKV: q (fp32, rotated) [rows][H*hd]; K / V cache of the layer
    // [Hkv][max_seq][hd] fp16; RoPE table [max_seq][hd/2] (cos, sin)
    int n_heads, n_kv_heads, head_dim, max_seq, pos0;
    float* q;
    f16* k_cache;
    f16* v_cache;
    const float2* rope;
    int* err;
};

// One pair's work, segment by segment: k blocks [kb0, kb1) of a tile.
struct TcWork {
    long long U;
    int cur, end, next_tile;
    int tile, kb0, kb1;
    int contributors;  // > 0: this segment ends the pair's range inside the tile; that many pairs follow
    bool partial;      // the segment starts inside the tile: its sums go to the workspace
};
// The i-th tile of the split ones: all feature tiles of a token tile, then the
// next token tile's.  The ranges of two token tiles then start at (about) the
// same k block of the same feature tile, so that the pairs reading a weight tile
// do so at the same time and HBM delivers it once.  With token tiles fastest
// they are out of step: the down projection of the 7B widths over 511 rows read
// 319 MB for 112 MB of operands, 71.7 us; now 61.4-63.5.  70B widths, 300 rows,
// down: 205 -> 172; 1023 rows, output projection: 153.6 -> 147.5.
__host__ __device__ __forceinline__ int tc_split_tile(const TcSched& s, int i) {
    const int q = s.n_split / s.n_tt, r = s.n_split - q * s.n_tt;  // r token tiles have q + 1 feature tiles, the others q
    const int j = i - r * (q + 1);
    return j < 0 ? i % (q + 1) * s.n_tt + i / (q + 1) : j % q * s.n_tt + r + j / q;
}
__host__ __device__ __forceinline__ void tc_work_init(TcWork& w, const TcSched& s, int n_kb, int pair) {
    w.U = (long long)s.n_split * n_kb;
    w.cur = w.end = 0;
    if (pair < s.split_pairs) {
        w.cur = (int)(pair * w.U / s.split_pairs);
        w.end = (int)((pair + 1) * w.U / s.split_pairs);
    }
    w.next_tile = s.n_split + pair;
}
__host__ __device__ __forceinline__ bool tc_work_next(TcWork& w, const TcSched& s, int n_kb, int pair) {
    w.contributors = 0;
    w.partial = false;
    if (w.cur < w.end) {
        const int i = w.cur / n_kb;
        w.tile = tc_split_tile(s, i);
        w.kb0 = w.cur - i * n_kb;
        w.kb1 = w.kb0 + w.end - w.cur < n_kb ? w.kb0 + w.end - w.cur : n_kb;
        w.cur += w.kb1 - w.kb0;
        w.partial = w.kb0 > 0;
        if (!w.partial && w.kb1 < n_kb) {
            const long long last = (long long)(i + 1) * n_kb - 1;  // the pair holding the tile's last k block
            w.contributors = (int)(((last + 1) * s.split_pairs + w.U - 1) / w.U - 1) - pair;
        }
        return true;
    }
    if (w.next_tile >= s.n_tiles) return false;
    w.tile = w.next_tile;
    w.kb0 = 0;
    w.kb1 = n_kb;
    w.next_tile += s.pairs;
    return true;
}

// ---------------------------------------------------------------------------
// PTX wrappers (tcgen05, TMA, mbarrier, cluster)
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long gtime() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of the same shared-memory object in the cluster's CTA `rank`
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mb_init(uint64_t* b, unsigned n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mb_arrive_tx(uint64_t* b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
// arrival on a barrier of either CTA of the pair (cluster address)
__device__ __forceinline__ void mb_arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ bool mb_try(uint64_t* b, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait; false (error recorded) after kWaitNs or once another thread
// of the grid recorded an error and 20 us have passed
__device__ __forceinline__ bool mb_wait(uint64_t* b, unsigned parity, int* err) {
    if (mb_try(b, parity)) return true;
    const unsigned long long t0 = gtime();
    while (!mb_try(b, parity)) {
        const unsigned long long dt = gtime() - t0;
        if (dt > 20000ull && *(volatile int*)err) return false;
        if (dt > kWaitNs) {
            atomicCAS(err, 0, kErrTimeout);
            return false;
        }
    }
    return true;
}
// tiled TMA loads into this CTA's shared memory, completing on a barrier of
// either CTA of the pair (cluster address); x (the k coordinate) is always a
// multiple of 64 elements
__device__ __forceinline__ void tma2d(void* dst, const void* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma3d(void* dst, const void* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma4d_pair(void* dst, const void* map, int x, int group, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(x), "r"(0), "r"(group), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma5d_head(void* dst, const void* map, int x, int head, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %3, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(x), "r"(0), "r"(head), "r"(bar)
        : "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart; the start address may sit 32 / 64 / 96 bytes into a
// swizzle row (k steps of 16 bf16)
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
    d |= (uint64_t)1 << 16;                           // leading byte offset (unused with this swizzle)
    d |= (uint64_t)(1024 >> 4) << 32;                 // stride byte offset
    d |= (uint64_t)1 << 46;                           // descriptor version
    d |= (uint64_t)2 << 61;                           // 128-byte swizzle
    return d;
}
// instruction descriptor: kind::f16, A = B = bf16, D = fp32, both K-major,
// M = 256 over the pair, N = nt
__device__ __forceinline__ uint32_t tc_idesc(int nt) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(nt >> 3) << 17) | ((uint32_t)(kFeat >> 4) << 24);
}
__device__ __forceinline__ void mma_pair(uint32_t tmem_d, uint64_t ad, uint64_t bd, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(tmem_d), "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate)
        : "memory");
}
// the barrier at this offset in both CTAs completes once every tcgen05 op this
// thread issued so far is done
__device__ __forceinline__ void mma_commit(uint64_t* b) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(smem_u32(b)), "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void store_hilo(bf16* hi, bf16* lo, float x) {
    const bf16 h = __float2bfloat16_rn(x);
    *hi = h;
    *lo = __float2bfloat16_rn(x - __bfloat162float(h));
}

// The lanes of a warp hold features in two groups of 16: lane l < 16 one
// member of a pair, lane l + 16 the other (gate / up, or the two halves of a
// rotation).  Exchanges the columns of a chunk so that every lane has both
// members for half of the tokens: on return lane l < 16 holds (a, b) of the
// even columns, lane l + 16 of the odd columns, a = the lower lanes' feature.
__device__ __forceinline__ void pair_up(const float (&v)[16], int upper, float (&a)[8], float (&b)[8]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float recv = __shfl_xor_sync(0xffffffffu, upper ? v[2 * j] : v[2 * j + 1], 16);
        a[j] = upper ? recv : v[2 * j];
        b[j] = upper ? v[2 * j + 1] : recv;
    }
}

// ---------------------------------------------------------------------------
// the kernel: grid = 2 * pairs, clusters of 2
// ---------------------------------------------------------------------------
// ROWS16 (QKV): the weights in eight boxes of 16 rows per k block instead of one of 128
template <int EPI, bool ROWS16>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1) tc_gemm_kernel(const TcArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ __align__(8) uint64_t full[kMaxStages];   // (even CTA) both CTAs' copies of a stage have landed
    __shared__ __align__(8) uint64_t empty[kMaxStages];  // the pair's MMAs have read the stage
    __shared__ __align__(8) uint64_t acc_full[2];        // accumulator complete
    __shared__ __align__(8) uint64_t acc_empty[2];       // (even CTA) read by the epilogue warps of both CTAs
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    // the highest ranges start first: a pair only waits for partial sums of pairs
    // with higher numbers, whose blocks come first in dispatch order (which CUDA does
    // not promise: the wait is bounded)
    const int pair = a.sched.pairs - 1 - (int)(blockIdx.x >> 1);
    const int S = a.stages, stage_bytes = kATile + a.nt * 128;
    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < S; ++s) {
            mb_init(full + s, 1);
            mb_init(empty + s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mb_init(acc_full + b, 1);
            mb_init(acc_empty + b, 2 * kEpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kEpiWarps) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    pdl_launch_dependents();
    fence_before();
    __syncthreads();
    cluster_sync();
    fence_after();
    const uint32_t tmem = s_tmem;

    bool ok = true;
    TcWork w;
    tc_work_init(w, a.sched, a.n_kb, pair);
    if (warp == kEpiWarps) {
        // producer: weights, and activations that the previous kernel wrote.
        // The weights of the first S k blocks are requested before that kernel
        // has finished.
        const uint32_t full0 = map_rank(smem_u32(full), 0);
        int s = 0;
        unsigned ph = 1;  // parity of the next "empty" completion to wait for (the ring starts empty)
        bool waited = false;
        while (ok && tc_work_next(w, a.sched, a.n_kb, pair)) {
            const int ft = w.tile / a.sched.n_tt, tt = w.tile - ft * a.sched.n_tt;
            const int tok0 = tt * a.nt + (int)rank * (a.nt >> 1);
            const int box = 2 * ft + (int)rank;  // this CTA's 128 TMEM lanes
            const void* map = a.tm_w[0];
            int row0 = box * 128;
            if (EPI == TC_QKV) {  // [Wq; Wk; Wv] in 128-row boxes of whole heads (past the end: zeros)
                const int qd = a.n_heads * a.head_dim, kvd = a.n_kv_heads * a.head_dim;
                if (row0 >= qd + kvd) { map = a.tm_w[2]; row0 -= qd + kvd; }
                else if (row0 >= qd) { map = a.tm_w[1]; row0 -= qd; }
                row0 /= a.head_dim;
            }
            auto weights = [&](int kb, int st_i) {  // (one lane) k block kb into stage st_i
                unsigned char* st = smem + st_i * stage_bytes;
                const uint32_t bar = full0 + 8u * (uint32_t)st_i;
                if (rank == 0) mb_arrive_tx(full + st_i, 2u * (unsigned)stage_bytes);
                if (EPI == TC_QKV) {
                    if (!ROWS16) {
                        tma5d_head(st, map, kb * kBK, row0, bar);
                    } else {  // the same rows, 16 at a time: heads row0 .., a half's 16, their partners, ...
                        const int per = a.head_dim >> 4;
#pragma unroll
                        for (int p = 0; p < 8; ++p) {
                            const int j = p % per;
                            tma2d(st + p * 2048, map, kb * kBK,
                                  (row0 + p / per) * a.head_dim + (j & 1) * (a.head_dim >> 1) + (j >> 1) * 16, bar);
                        }
                    }
                } else if (EPI == TC_SWIGLU) {
                    if (a.tm_w[1] == nullptr) {
                        tma4d_pair(st, map, kb * kBK, box * 4, bar);
                    } else {
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            tma2d(st + g * 4096, map, kb * kBK, box * 64 + g * 16, bar);
                            tma2d(st + g * 4096 + 2048, a.tm_w[1], kb * kBK, box * 64 + g * 16, bar);
                        }
                    }
                } else {
                    tma2d(st, map, kb * kBK, row0, bar);
                }
            };
            int n_pre = 0;
            if (!waited) {  // (the ring is empty)
                n_pre = min(S, w.kb1 - w.kb0);
                for (int i = 0; i < n_pre; ++i) {
                    if (elect_one()) weights(w.kb0 + i, i);
                    __syncwarp();
                }
                pdl_wait();
                asm volatile("fence.proxy.async.global;" ::: "memory");
                waited = true;
            }
            for (int kb = w.kb0; kb < w.kb1; ++kb) {
                const bool pre = kb - w.kb0 < n_pre;
                if (!pre) ok = __all_sync(0xffffffffu, mb_wait(empty + s, ph, a.err));
                if (!ok) break;
                if (elect_one()) {
                    if (!pre) weights(kb, s);
                    tma3d(smem + s * stage_bytes + kATile, a.tm_x, kb * kBK, tok0, 0, full0 + 8u * (uint32_t)s);
                }
                __syncwarp();
                if (++s == S) { s = 0; ph ^= 1u; }
            }
        }
        // the commits that release the last stages also arrive here: do not
        // leave before them
        for (int i = 0; i < S && ok; ++i) {
            ok = __all_sync(0xffffffffu, mb_wait(empty + s, ph, a.err));
            if (++s == S) { s = 0; ph ^= 1u; }
        }
    } else if (warp == kEpiWarps + 1 && rank == 0) {
        // MMA issuer of the pair
        const uint32_t idesc = tc_idesc(a.nt);
        const uint64_t desc0 = sdesc(smem_u32(smem));
        int s = 0, b = 0;
        unsigned ph = 0, aph = 3u;  // aph bit b: parity of the next release of accumulator b (both start free)
        while (ok && tc_work_next(w, a.sched, a.n_kb, pair)) {
            ok = __all_sync(0xffffffffu, mb_wait(acc_empty + b, (aph >> b) & 1u, a.err));
            if (!ok) break;
            aph ^= 1u << b;
            fence_after();
            const uint32_t d = tmem + (uint32_t)(b * kMaxTok);
            for (int kb = w.kb0; kb < w.kb1; ++kb) {
                ok = __all_sync(0xffffffffu, mb_wait(full + s, ph, a.err));
                if (!ok) break;
                fence_after();
                if (elect_one()) {
                    const uint64_t ad = desc0 + (uint64_t)((uint32_t)(s * stage_bytes) >> 4);
                    const uint64_t xh = ad + (kATile >> 4), xl = xh + (uint64_t)(a.nt * 4);
#pragma unroll
                    for (int kk = 0; kk < kBK / 16; ++kk) {  // 16 k = 32 bytes
                        mma_pair(d, ad + 2 * kk, xh + 2 * kk, idesc, (kb != w.kb0 || kk) ? 1u : 0u);
                        mma_pair(d, ad + 2 * kk, xl + 2 * kk, idesc, 1u);
                    }
                    mma_commit(empty + s);  // the stage is free once these MMAs have read it
                }
                __syncwarp();
                if (++s == S) { s = 0; ph ^= 1u; }
            }
            if (ok && elect_one()) mma_commit(acc_full + b);
            __syncwarp();
            b ^= 1;
        }
    } else if (warp < kEpiWarps) {
        const int q4 = warp & 3, quarter = warp >> 2, upper = lane >> 4;
        pdl_wait();  // h, the workspace and the outputs may still be in use
        const int hc = a.nt >> 2;  // columns of this warp: quarter * hc .. + hc (a multiple of 8)
        const uint32_t empty0[2] = {map_rank(smem_u32(acc_empty), 0), map_rank(smem_u32(acc_empty + 1), 0)};
        int b = 0;
        unsigned fph = 0;  // bit b: parity of the next completion of accumulator b
        while (ok && tc_work_next(w, a.sched, a.n_kb, pair)) {
            const int ft = w.tile / a.sched.n_tt, tt = w.tile - ft * a.sched.n_tt;
            const int box = 2 * ft + (int)rank;
            const int tok0 = tt * a.nt + quarter * hc;
            const int n_col = min(hc, a.rows - tok0);  // valid columns of this warp (may be <= 0)
            // (by the warp: a lane alone must not leave its tcgen05.ld, votes and shuffles)
            ok = __all_sync(0xffffffffu, mb_wait(acc_full + b, (fph >> b) & 1u, a.err));
            fph ^= 1u << b;
            if (!ok) break;
            fence_after();
            const uint32_t tl = tmem + (uint32_t)(b * kMaxTok + quarter * hc) + ((uint32_t)(q4 * 32) << 16);
            // partial sums [pair][cta][column][lane], 128 bytes per warp and column
            auto slot = [&](int p) {
                return a.ws + (((size_t)p * 2 + rank) * kMaxTok + quarter * hc) * 128 + q4 * 32 + lane;
            };
            if (w.partial) {
                float* o = slot(pair);
                for (int c0 = 0; c0 < n_col; c0 += 16) {
                    float v[16];
                    tmem_ld16(tl + c0, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (c0 + i < n_col) __stcg(o + (size_t)(c0 + i) * 128, v[i]);
                }
                __threadfence();
                __syncwarp();
                if (lane == 0)
                    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.flags + (pair * 2 + rank) * kEpiWarps + warp),
                                 "r"(a.epoch)
                                 : "memory");
            } else {
                for (int c = 1; c <= w.contributors && ok; ++c) {  // (bounded) until their partial sums are there
                    const unsigned* f = a.flags + ((pair + c) * 2 + rank) * kEpiWarps + warp;
                    const unsigned long long t0 = gtime();
                    for (;;) {
                        unsigned x;
                        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(f) : "memory");
                        if (x == a.epoch) break;
                        const unsigned long long dt = gtime() - t0;
                        if ((dt > 20000ull && *(volatile int*)a.err) || dt > kWaitNs) {
                            atomicCAS(a.err, 0, kErrTimeout);
                            ok = false;
                            break;
                        }
                    }
                }
                ok = __all_sync(0xffffffffu, ok);
                // feature / rotation pair of this lane
                const int hd = a.head_dim, half_d = hd >> 1;
                const int ii = EPI == TC_QKV ? (q4 % (hd / 32)) * 16 + (lane & 15) : 0;
                const int n = EPI == TC_SWIGLU ? box * 64 + q4 * 16 + (lane & 15) : box * 128 + q4 * 32 + lane;
                for (int c0 = 0; c0 < n_col && ok; c0 += 16) {
                    const int tok = tok0 + c0;  // token row of v[0]
                    // what the epilogue reads from memory is requested before the
                    // accumulator and the partial sums are
                    float h[EPI == TC_RESID ? 16 : 1];
                    float2 cs[EPI == TC_QKV ? 8 : 1];
                    if (EPI == TC_RESID) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            h[i] = c0 + i < n_col && n < a.N ? __ldcg(a.out + (size_t)(tok + i) * a.N + n) : 0.f;
                    }
                    if (EPI == TC_QKV) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            cs[j] = c0 + 2 * j + upper < n_col
                                        ? __ldg(a.rope + (size_t)(a.pos0 + tok + 2 * j + upper) * half_d + ii)
                                        : make_float2(0.f, 0.f);
                    }
                    float ps[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) ps[i] = 0.f;
                    for (int c = 1; c <= w.contributors; c += 2) {  // two ranges in flight, added in order
                        const bool two = c < w.contributors;
                        const float* p = slot(pair + c) + (size_t)c0 * 128;
                        const float* p2 = slot(pair + (two ? c + 1 : c)) + (size_t)c0 * 128;
                        float x[16], y[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            x[i] = c0 + i < n_col ? __ldcg(p + i * 128) : 0.f;
                            y[i] = c0 + i < n_col && two ? __ldcg(p2 + i * 128) : 0.f;
                        }
#pragma unroll
                        for (int i = 0; i < 16; ++i) ps[i] = (ps[i] + x[i]) + y[i];
                    }
                    float v[16];
                    tmem_ld16(tl + c0, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] += ps[i];
                    if (EPI == TC_RESID) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (c0 + i < n_col && n < a.N) a.out[(size_t)(tok + i) * a.N + n] = h[i] + v[i];
                    } else if (EPI == TC_SWIGLU) {
                        float g[8], u[8];
                        pair_up(v, upper, g, u);
                        if (n < a.N) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const int c = 2 * j + upper;
                                if (c0 + c >= n_col) continue;
                                const float gt = a.swapped ? u[j] : g[j], up = a.swapped ? g[j] : u[j];
                                const float x = gt / (1.f + expf(-gt)) * up;
                                const size_t at = (size_t)(tok + c) * a.N + n;
                                store_hilo(a.act_hi + at, a.act_lo + at, x);
                            }
                        }
                    } else {  // TC_QKV: this CTA's box is whole heads of q, k or v
                        const int qd = a.n_heads * hd, kvd = a.n_kv_heads * hd;
                        const int f0 = box * 128;
                        const int kind = f0 < qd ? 0 : (f0 < qd + kvd ? 1 : 2);
                        const int head = (f0 - (kind == 0 ? 0 : (kind == 1 ? qd : qd + kvd))) / hd + q4 / (hd / 32);
                        if (f0 >= qd + 2 * kvd) continue;  // (uniform: past the last box)
                        if (kind == 2) {
                            f16* o = a.v_cache + ((size_t)head * a.max_seq + a.pos0 + tok) * hd + ii + upper * half_d;
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                if (c0 + i < n_col) o[(size_t)i * hd] = __float2half_rn(v[i]);
                        } else {
                            float x1[8], x2[8];
                            pair_up(v, upper, x1, x2);
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const int c = 2 * j + upper;
                                if (c0 + c >= n_col) continue;
                                const float y1 = x1[j] * cs[j].x - x2[j] * cs[j].y;
                                const float y2 = x2[j] * cs[j].x + x1[j] * cs[j].y;
                                if (kind == 0) {
                                    float* q = a.q + (size_t)(tok + c) * qd + head * hd;
                                    q[ii] = y1;
                                    q[ii + half_d] = y2;
                                } else {
                                    f16* k = a.k_cache + ((size_t)head * a.max_seq + a.pos0 + tok + c) * hd;
                                    k[ii] = __float2half_rn(y1);
                                    k[ii + half_d] = __float2half_rn(y2);
                                }
                            }
                        }
                    }
                }
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mb_arrive_cluster(empty0[b]);  // this warp is done with the accumulator
            b ^= 1;
        }
    }
    if (!ok) s_fail = 1;
    __syncwarp();
    __syncthreads();
    if (s_fail && threadIdx.x == 0) {
        // a wait gave up: let copies and MMAs in flight finish before shared
        // memory and TMEM are released
        const unsigned long long t0 = gtime();
        while (gtime() - t0 < 2000000ull) __nanosleep(1000);
    }
    fence_before();
    __syncthreads();
    cluster_sync();  // the other CTA's MMAs, arrivals and commits are done with this CTA
    if (warp == kEpiWarps) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// Tile shape and schedule of a GEMM over `rows` tokens and n_ft feature tiles
// of K inputs: token tiles of equal size (a multiple of 32) and either whole
// tiles only, pair by pair, or the tiles that do not fill a wave of pairs split
// by k block over all of them (with less than half a wave left, one more wave
// is split with it, so that a tile is cut in two or three rather than many), in
// pieces of at least kMinSplit k blocks.  The choice with the least estimated
// time, from times measured on GB300: every choice of the 7B, 13B and 70B
// projections for 64 .. 2047 rows, 1100 points (us):
//   a k block of a tile   0.059 + 0.00229 nt, at least 0.24 (issue bound);
//   the rest, mostly the last tile's epilogue: whole tiles 8.4 nt / 256; split
//   tiles, the partial sums' way through L2 included, 17 nt / 256 + 6.5, or
//   12 nt / 256 + 7 if whole tiles follow;
//   split tiles walk K at offsets of their own: token planes of more than ~73
//   MB do not stay in L2 and both operands come from HBM (6.8 TB/s).
// Over those shapes the choice is 0.8 % slower than the best measured one on
// average (19.69 ms of 19.45 in the sum).
inline void tc_plan(TcArgs& a, int n_ft, int pairs, int K) {
    const int least = (a.rows + kMaxTok - 1) / kMaxTok;
    double best = 1e30;
    for (int n_tt = least; n_tt <= 4 * least; ++n_tt) {
        const int nt = ((a.rows + n_tt - 1) / n_tt + 31) / 32 * 32;
        if ((a.rows + nt - 1) / nt != n_tt) continue;
        const int tiles = n_ft * n_tt, waves = tiles / pairs, rest = tiles % pairs;
        const double t_kb = 0.059 + 0.00229 * nt > 0.24 ? 0.059 + 0.00229 * nt : 0.24;
        for (int split = 0; split < 2; ++split) {
            int n_split = 0, p = 1;
            double us = (double)(waves + (rest ? 1 : 0)) * a.n_kb * t_kb + 8.4 * nt / 256;
            if (split) {
                if (rest == 0) continue;
                n_split = waves > 0 && 2 * rest < pairs ? rest + pairs : rest;
                const long long q = (long long)n_split * a.n_kb / kMinSplit;
                p = q < pairs ? (int)q : pairs;
                // too short for every pair: only useful if there is no whole wave
                if (p < pairs && (waves > 0 || p <= rest)) continue;
                double part = (double)n_split * a.n_kb / p * t_kb;
                if (4e0 * a.rows * K > 73e6) {
                    const double hbm = n_split * (512.0 * K + 4.0 * nt * K) / 6.8e6;
                    if (hbm > part) part = hbm;
                }
                const int whole = (tiles - n_split) / pairs;
                us = part + whole * a.n_kb * t_kb + (whole ? 12.0 * nt / 256 + 7 : 17.0 * nt / 256 + 6.5);
            }
            if (us < best) {
                best = us;
                a.nt = nt;
                a.sched = {tiles, n_split, p, pairs, n_tt};
                if (tiles - n_split < pairs) a.sched.pairs = p > tiles - n_split ? p : tiles - n_split;
            }
        }
    }
    const int stage = kATile + a.nt * 128;
    a.stages = kRingBytes / stage < kMaxStages ? kRingBytes / stage : kMaxStages;
}

template <int EPI, bool ROWS16 = false>
inline int tc_configure() {
    return (int)cudaFuncSetAttribute(tc_gemm_kernel<EPI, ROWS16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemBytes);
}

// launch that may start while the previous kernel of the stream ends
template <typename... P, typename... A>
inline int launch_pdl(void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, k, args...);
}

template <int EPI, bool ROWS16 = false>
inline int tc_launch(const TcArgs& a, cudaStream_t s) {
    return launch_pdl(tc_gemm_kernel<EPI, ROWS16>, dim3(2 * a.sched.pairs), kThreads, kSmemBytes, s, a);
}

}  // namespace tc
}  // namespace ssd
