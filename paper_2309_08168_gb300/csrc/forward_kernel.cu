// forward_kernel.cu - one decoder forward (draft step, verification, prefill
// chunk) as a single persistent, cooperative kernel.
//
// Batch-1 decoding streams every weight byte once per forward and is bound by
// HBM (Sec. 3.1).  At LLaMA-2 7B scale a projection takes 5-30 us at full
// bandwidth, so per-kernel ramp-up and drain would cost a large fraction of
// the step.  Instead one CTA per SM walks the forward's op list
//     embed -> [QKV -> attention -> O] -> [gate/up -> down] -> ... -> lm_head
// (sublayers in the skip set z are simply absent from the draft's list,
// Sec. 3.2 / 3.3) with a grid barrier between dependent ops.  The CTA's roles
// (consumer warps, TMA producer, MMA issuer) walk the list on their own: once
// the consumers have arrived at a barrier the producer requests the weights of
// the CTA's first units of the next projection (they do not depend on the
// previous op), so the barrier's latency overlaps HBM streaming, and it is told
// by thread 0, not by a CTA barrier, that the inputs may be requested.  Every wait is bounded: a barrier that does
// not complete within ~2 s records an error code and the CTAs return.
//
// Projections (all of them: q/k/v + RoPE + KV write, output and down with the
// residual add, gate/up with SwiGLU, lm_head) run on the 5th-generation
// tensor cores: work unit = 128-row tile x 128-wide k chunk (32 KB of
// weights), each CTA owns an equal contiguous range of units in tile-major
// order, streamed by TMA (128-byte swizzle) through a 5-stage ring; an
// elected lane of the MMA warp issues tcgen05.mma kind::f16 per unit (M = 128 weight
// rows, N = the activation rows as bf16 hi + lo planes, ~16 mantissa bits of
// the fp32 activations) into a TMEM accumulator and releases the stage with
// tcgen05.commit; the consumer warps read a finished tile segment from TMEM
// (tcgen05.ld) while the next segment accumulates in the other accumulator.
// A tile split over several CTAs is summed in segment order by the CTA
// holding its first chunks; the others store their partials tagged with the
// op (three input rows' sums and the tag in one 128-bit word), so they neither
// fence nor signal, and the finaliser polls the words themselves.  That exchange
// is what an op's end waits for (weights of the next op in flight slow every L2
// round trip to ~1.5 us), so it takes as few words and round trips as it can:
// with a word per sum a 13-row verification of 4 layers at 13B widths took 640 us,
// with a word per three rows 597 us.
// RMSNorm is folded in: the producer of the residual stream writes the planes
// of h * g_next and per-128-column sums of h^2, the consumer scales row m by
// rsqrt(mean(h^2) + eps) in its epilogue (W (h g r) = r W (h g)).
//
// Attention: items = (KV head, group of 16 query vectors, absolute
// 128-position segment); the partial softmax of a row over a segment depends
// only on the row and the segment.  After a grid barrier every CTA combines a share
// of the (KV head, query vector) outputs over their segments in segment
// order.
//
// Coherence: L1 is not coherent across SMs within one launch, so every load of
// data another CTA wrote during this launch goes through L2 (cp.async.cg,
// ld.global.cg); stores are write-through.
//
// Batch invariance (greedy self-speculative output must equal autoregressive
// output bit for bit, Sec. 1 / App. G.2): row m's result depends only on row
// m - the MMA's output columns are independent (an input row is one column of
// D whatever N is), unit partitions and combine orders depend on the shapes
// and the grid only, epilogues are per row, attention segments are absolute
// positions.
#include "ssd_internal.cuh"

namespace ssd {
namespace {

constexpr unsigned long long kBarrierTimeoutNs = 2000000000ull;
// A wait reads the shared error flag only after this long (20 us): until
// then each poll is a single load.
constexpr unsigned long long kErrPollAfterNs = 20000ull;
// 8 consumer warps (epilogues, attention, embedding) + 1 producer warp (TMA)
// + 1 MMA warp (tcgen05.mma issue, TMEM allocation)
constexpr int kConsumers = 256;
constexpr int kFwdThreads = kConsumers + 64;

// barrier among the consumer warps only (the producer and MMA warps go on)
__device__ __forceinline__ void consumer_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// the same; true in every consumer thread if any of them passed true
__device__ __forceinline__ bool consumer_or(bool x) {
    unsigned r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, 256, p;\n selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"((unsigned)x)
        : "memory");
    return r != 0;
}


__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid-wide barrier for a cooperative launch (all CTAs co-resident), in two
// halves so that a CTA can do work that publishes nothing between them.  The
// counter only grows during a launch; `target` = gridDim.x * (barrier index).
// grid_arrive (one thread, after a CTA barrier that orders the CTA's stores
// before it): the release of the arrival publishes those stores and needs no
// reply.  grid_wait (the same thread): acquire - later loads, ordered after it
// by a CTA barrier, see the others' stores.  Returns false (and records
// SSD_DEV_ERR_TIMEOUT) if the others do not arrive within limit_ns, or if
// another CTA already gave up.
__device__ __forceinline__ void grid_arrive(unsigned* bar) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}
// Each poll is one L2 round trip: the error flag (another CTA gave up) is
// read only once the wait has lasted kErrPollAfterNs, so that a second load
// does not double the poll period of ordinary waits.
__device__ bool grid_wait(unsigned* bar, unsigned target, int* err, unsigned long long limit_ns) {
    const unsigned long long t0 = globaltimer();
    while (ld_acquire(bar) < target) {
        const unsigned long long dt = globaltimer() - t0;
        if (dt > kErrPollAfterNs) {
            if (*(volatile int*)err) return false;
            if (dt > limit_ns) {
                atomicCAS(err, 0, kDevErrTimeout);
                return false;
            }
        }
    }
    return true;
}

// Split-K partials: up to three input rows' sums of a tile row and the tag of
// the op that wrote them (forward sequence number << 10 | op index) in one
// 128-bit word, written and read as single 128-bit accesses.
struct PartWord {
    unsigned long long lo, hi;  // rows 0, 1; row 2, tag
};
__device__ __forceinline__ unsigned tag_of(const PartWord& w) { return (unsigned)(w.hi >> 32); }
__device__ __forceinline__ float value_of(const PartWord& w, int j) {
    return __uint_as_float((unsigned)(j == 0 ? w.lo : j == 1 ? w.lo >> 32 : w.hi));
}
__device__ __forceinline__ void st_relaxed(PartWord* p, unsigned tag, float v0, float v1, float v2) {
    const unsigned long long lo = (unsigned long long)__float_as_uint(v1) << 32 | __float_as_uint(v0);
    const unsigned long long hi = (unsigned long long)tag << 32 | __float_as_uint(v2);
    asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}\n" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}
__device__ __forceinline__ PartWord ld_relaxed(const PartWord* p) {
    PartWord w;
    asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}\n"
                 : "=l"(w.lo), "=l"(w.hi)
                 : "l"(p)
                 : "memory");
    return w;
}
__device__ __forceinline__ int unit_owner(long long u, long long U, long long G) {
    return (int)(((u + 1) * G + U - 1) / U - 1);
}

// An op's units are split over the first min(U, grid) CTAs, so every CTA that
// takes part owns at least one unit and the owners of consecutive units are
// consecutive CTAs (the segment arithmetic of the projection op relies on it).
// Keeping tiles of two or three chunks whole (units one after the other instead of a
// split-K exchange) is no gain: forwards of 1 / 5 / 16 rows take 188.5 / 209.0 / 253.2 us
// so at d 384 (8 layers) and 165.4 / 189.6 / 247.7 split, 86.1 / 96.4 / 127.7 against
// 85.8 / 95.8 / 129.0 at d 256.
__device__ __forceinline__ long long op_ctas(long long U) { return U < gridDim.x ? U : (long long)gridDim.x; }

__device__ __forceinline__ void my_units(long long U, int* u_begin, int* n_my) {
    const long long G = op_ctas(U), b = blockIdx.x;
    if (b >= G) { *u_begin = 0; *n_my = 0; return; }
    *u_begin = (int)(b * U / G);
    *n_my = (int)((b + 1) * U / G) - *u_begin;
}

__device__ __forceinline__ bool is_gemm(int type) { return type >= OP_QKV && type <= OP_LOGITS && type != OP_ATTN; }

__device__ __forceinline__ int epi_of(int type) {
    return type == OP_QKV ? EPI_QKV : type == OP_RESID ? EPI_RESID : type == OP_SWIGLU ? EPI_SWIGLU : EPI_LOGITS;
}

// ---------------------------------------------------------------------------
// TMA + mbarrier helpers
// ---------------------------------------------------------------------------
constexpr unsigned long long kWaitTimeoutNs = 2000000000ull;

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// adds expected bytes without arriving (the weights of a unit, requested early)
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// plain arrival (a consumer warp releasing a stage)
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// arrives (count 1) and adds expected bytes (the activations of the unit)
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait: false after kWaitTimeoutNs (timeout recorded), or once it has
// waited kErrPollAfterNs while another thread has already recorded an error
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, int* err) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    while (!mbar_try_wait(bar, parity)) {
        const unsigned long long dt = globaltimer() - t0;
        if (dt > kErrPollAfterNs && *(volatile int*)err) return false;
        if (dt > kWaitTimeoutNs) {
            atomicCAS(err, 0, kDevErrTimeout);
            return false;
        }
    }
    return true;
}
// 2D tiled TMA load of one box into shared memory, completing on `bar`.  x is
// the innermost (k) coordinate; every x used here is a multiple of 64
// elements (128 bytes), so the 16-byte rule for x * element size holds.
__device__ __forceinline__ void tma_load_2d(void* dst, const void* tmap, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"(tmap), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const void* tmap, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// brings a tensor map descriptor (global memory) into the descriptor cache
__device__ __forceinline__ void prefetch_tmap(const void* tmap) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory");
}

// fp16 tensor-core MMA (attention: K / V are fp16) and 8x8 matrix loads
__device__ __forceinline__ void mma_f16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                              uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}

// ---------------------------------------------------------------------------
// projection op: TMA ring -> tcgen05.mma -> TMEM -> epilogue
// ---------------------------------------------------------------------------
// Work unit = a 128-row tile x 128-wide k chunk of a weight matrix (32 KB).
// Stage layout (1 KB aligned; TMA writes the 128-byte swizzle, which is the
// canonical K-major operand layout of tcgen05.mma: row r of a 64-wide k box
// at r * 128 bytes, 8-row groups 1024 bytes apart):
//   weights : k box kb (k0 + 64 kb ..) of the tile's 128 rows at kb * 16 KB
//             (SwiGLU tiles: rows 0-63 gate, 64-127 up, of features 64 t ..)
//   inputs  : k box kb at 32 KB + kb * XKB; rows p = plane * R + row (the R
//             hi rows, then the R lo rows); rows 2R .. NP-1 are not written and
//             only feed accumulator columns that nobody reads
// One thread of the MMA warp issues, per unit, eight tcgen05.mma kind::f16
// (bf16 x bf16 -> fp32; M = 128 weight rows, N = NP input rows, K = 16) into
// one of two TMEM accumulators (one per tile segment, so the consumers read a
// finished segment while the next one accumulates) and releases the stage
// with tcgen05.commit.  The consumer warps only run the segment epilogue.
//
// attention: 64-position chunks per segment (one ring stage each).  Segments
// are absolute, so a row's softmax partials do not depend on M; two chunks
// per segment balance ~150 CTAs well at LLaMA-2 KV-head counts and contexts
// and keep the final combine short.
constexpr int kAttnSegChunks = 2;

// Attention unit in a stage: K rows of the 64-position chunk at 0 (dims 0-63,
// then 64-127 at 8 KB), V rows at 16 KB; position t, 16-byte chunk c of a
// 64-dim box at box + t * 128 + ((c ^ (t & 7)) << 4).
// After the ring: the consumers' scratch - the finished segment of a
// projection, or (same bytes: one op at a time) q / scores of attention.
// index of the input-plane tensor map of R rows
__host__ __device__ constexpr int plane_cls(int R) {
    return R == 1 ? 0 : (R == 4 ? 1 : (R == 8 ? 2 : (R == 12 ? 3 : 4)));
}

template <int R>
struct GemmSmem {
    static constexpr int NP = R <= 8 ? 16 : 32;     // MMA N: input rows (hi + lo), padded
    static constexpr int WB = kFTile * kFKC * 2;    // 32 KB of weights per unit
    static constexpr int XKB = NP * 128;            // input bytes per 64-wide k box
    static constexpr int STAGE = WB + 2 * XKB;
    static constexpr int S = 5;                     // ring depth (160 KB of weights in flight)
    static constexpr int VG = 16;  // attention: query vectors per item (one MMA M / N tile)
    static constexpr int YS = S * STAGE;            // [128][16] floats: the finished segment
    // attention scratch: q hi / lo (fp16, rows padded by 16 bytes), scores
    // (fp32), P hi / lo (fp16, padded rows)
    static constexpr int QST = 128 + 8, PST = kAttnSegChunks * kAttnChunk + 8;  // halves per row
    static constexpr int ATT = S * STAGE;
    static constexpr int ATT_SC = ATT + 2 * VG * QST * 2;
    static constexpr int ATT_P = ATT_SC + 2 * (kConsumers / 32) * VG * 4;  // per-warp maxima and sums
    static constexpr int SCRATCH_GEMM = kFTile * 16 * 4;
    static constexpr int SCRATCH_ATT = ATT_P + 2 * VG * PST * 2 - ATT;
    static constexpr size_t BYTES =
        1024 + (size_t)S * STAGE + (SCRATCH_GEMM > SCRATCH_ATT ? SCRATCH_GEMM : SCRATCH_ATT);
    static_assert(STAGE >= 2 * kAttnChunk * 128 * 2, "a stage holds the K and V rows of one 64-position chunk");
    static_assert(BYTES + 4096 <= 232448, "dynamic + static shared memory within the per-CTA limit");
};

// ---------------------------------------------------------------------------
// tcgen05 helpers
// ---------------------------------------------------------------------------
constexpr int kTmemCols = 64;  // two accumulators of up to 32 fp32 columns

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart; the start address may sit 32 / 64 / 96 bytes into a
// swizzle row (k steps of 16 bf16)
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
    d |= (uint64_t)1 << 16;                           // leading byte offset (unused with this swizzle)
    d |= (uint64_t)(1024 >> 4) << 32;                 // stride byte offset
    d |= (uint64_t)1 << 46;                           // descriptor version
    d |= (uint64_t)2 << 61;                           // 128-byte swizzle
    return d;
}
// instruction descriptor: kind::f16, A = B = bf16, D = fp32, both K-major,
// M = 128, N = np
__host__ __device__ constexpr uint32_t umma_idesc(int np) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(np >> 3) << 17) | ((uint32_t)(kFTile >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(tmem_d), "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}
// the mbarrier completes once every tcgen05 op this thread issued so far is done
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// NP consecutive fp32 columns of this thread's TMEM lane
template <int NP>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[NP]);
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, float (&v)[16]) {
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
template <>
__device__ __forceinline__ void tmem_ld<32>(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

template <>
__device__ __forceinline__ void tmem_ld<24>(uint32_t taddr, float (&v)[24]) {
    uint32_t r[24];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
                   "=r"(r[23])
                 : "r"(taddr + 16u));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 24; ++i) v[i] = __uint_as_float(r[i]);
}

// Weight rows of tile t: one 128-row box (matrix s0 from row r0), or for
// SwiGLU two 64-row boxes (the gate and the up rows of features 64 t ..).
// The q / k / v widths are whole tiles, so a q / k tile is 128 / head_dim
// whole heads in natural order and holds every RoPE pair (j, j + hd / 2).
struct TileSrc {
    int s0, r0, s1, r1;  // s1 < 0: one box
};
__device__ __forceinline__ TileSrc tile_src(const GemmArgs& a, int epi, int tile) {
    if (epi == EPI_SWIGLU) return {0, tile * 64, 1, tile * 64};
    if (epi == EPI_QKV) {
        const int qt = a.n_heads * a.head_dim / kFTile, kt = a.n_kv_heads * a.head_dim / kFTile;
        if (tile < qt) return {0, tile * kFTile, -1, 0};
        if (tile < qt + kt) return {1, (tile - qt) * kFTile, -1, 0};
        return {2, (tile - qt - kt) * kFTile, -1, 0};
    }
    return {0, tile * kFTile, -1, 0};
}

// weights of unit u into a stage (one lane): expect_tx without arriving.
// Always a full 128 x 128 tile of bytes (rows / columns out of range are
// delivered as zeros and counted).  Every x used here is a multiple of 64
// elements (128 bytes), so the 16-byte rule for x * element size holds.
template <int R>
__device__ __forceinline__ void tma_weights(const GemmArgs& a, int epi, int u, unsigned char* st, uint64_t* bar) {
    const int tile = u / a.n_chunks, k0 = (u - tile * a.n_chunks) * kFKC;
    const TileSrc ts = tile_src(a, epi, tile);
    mbar_expect_tx(bar, (unsigned)GemmSmem<R>::WB);
#pragma unroll
    for (int kb = 0; kb < 2; ++kb) {
        tma_load_2d(st + kb * 16384, a.tm_w[ts.s0], k0 + kb * 64, ts.r0, bar);
        if (ts.s1 >= 0) tma_load_2d(st + kb * 16384 + 8192, a.tm_w[ts.s1], k0 + kb * 64, ts.r1, bar);
    }
}

// input planes of unit u into a stage (one lane): arrive + expect_tx
template <int R>
__device__ __forceinline__ void tma_inputs(const GemmArgs& a, int u, unsigned char* st, uint64_t* bar) {
    using L = GemmSmem<R>;
    const int k0 = (u % a.n_chunks) * kFKC;
    const int cls = plane_cls(R);
    mbar_arrive_expect_tx(bar, 2u * 2u * (unsigned)R * 128u);
#pragma unroll
    for (int kb = 0; kb < 2; ++kb) tma_load_3d(st + L::WB + kb * L::XKB, a.tm_x[cls], k0 + kb * 64, 0, 0, bar);
}

// Pipeline state, carried across ops; every thread keeps its own copy and
// flips the bits of the waits it takes part in (or, for ring positions whose
// waits another role took, the same bits arithmetically).
//   pphase bit s : parity of the next "empty" completion of stage s (producer)
//   cphase bit s : parity of the next "full" completion of stage s (MMA thread
//                  in projections, consumers in attention)
//   afull bit b  : parity of the next completion of accumulator b (consumers)
//   aempty bit b : parity of the next release of accumulator b (MMA thread)
//   ab           : accumulator of the next tile segment
//   rb           : ring stage of the op's first unit (the ring runs on from op
//                  to op, so a stage is reused in the order it was released)
struct Pipe {
    uint64_t* full;     // [stages] TMA completion (count 1: the producer's arrive)
    uint64_t* empty;    // [stages] stage released (count 1: tcgen05.commit, or consumer thread 0)
    uint64_t* acc_full;   // [2] accumulator complete (tcgen05.commit)
    uint64_t* acc_empty;  // [2] accumulator read by the consumers (count 8: one arrival per consumer warp)
    uint32_t tmem;      // TMEM base address (two accumulators of kTmemCols / 2 columns)
    unsigned pphase;
    unsigned cphase;
    unsigned afull;
    unsigned aempty;
    int ab;
    int rb;
};

// ring stage of the op's unit i
template <int S>
__device__ __forceinline__ int ring_stage(const Pipe& pp, int i) {
    return (pp.rb + i) % S;
}
// the op's n ring positions are used up
template <int S>
__device__ __forceinline__ void ring_advance(Pipe& pp, int n) {
    pp.rb = (pp.rb + n) % S;
}
// flips the full-barrier parity bits of the op's n ring positions, whose waits
// another role took
template <int S>
__device__ __forceinline__ void advance_full(Pipe& pp, int n) {
#pragma unroll
    for (int k = 0; k < S; ++k)
        if (((n / S) + (k < n % S ? 1 : 0)) & 1) pp.cphase ^= 1u << ring_stage<S>(pp, k);
}

// A projection op in a CTA has three roles:
//   producer (warp 8, one elected lane) streams this CTA's units through the ring;
//   MMA issuer (warp 9, one elected lane) runs tcgen05.mma per unit into the
//     accumulator of the unit's tile segment;
//   consumers (warps 0-7), per finished segment: TMEM -> hi + lo summed ->
//     split-K exchange -> epilogue (contributors and residual finalisers
//     per warp from registers, the other finalisers through shared memory).
// Each returns false if a wait timed out (error recorded).  ut: nullptr, or
// [64][4] timestamps of this CTA's first units (producer issue, MMAs issued, 0,
// segment flush done); ct: nullptr, or this CTA's op stamps (FwdParams::trace) -
// profiling aids.

// Producer warp, once the consumers have left the previous op: the weights of
// the first S units, which depend on nothing, while the grid gathers; then the
// inputs, once `go` says that the grid barrier has passed.
template <int R>
__device__ bool gemm_produce(const GemmArgs& a, int epi, unsigned char* smem, Pipe& pp, uint64_t* go, unsigned go_parity,
                             int* err, unsigned long long* ut) {
    using L = GemmSmem<R>;
    constexpr int S = L::S;
    int u_begin, n_my;
    my_units(a.n_units, &u_begin, &n_my);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (n_my > 0 && elect_one()) prefetch_tmap(a.tm_x[plane_cls(R)]);
    __syncwarp();
    const int n_pre = min(S, n_my);
    for (int i = 0; i < n_pre; ++i) {
        const int s = ring_stage<S>(pp, i);
        if (!__all_sync(0xffffffffu, mbar_wait(pp.empty + s, (pp.pphase >> s) & 1u, err))) return false;
        pp.pphase ^= 1u << s;
        if (elect_one()) tma_weights<R>(a, epi, u_begin + i, smem + s * L::STAGE, pp.full + s);
        __syncwarp();
    }
    if (!__all_sync(0xffffffffu, mbar_wait(go, go_parity, err))) return false;
    if (ut) ut[2] = globaltimer();
    asm volatile("fence.proxy.async.global;" ::: "memory");  // inputs written by the previous op
    for (int i = 0; i < n_my; ++i) {
        const int s = ring_stage<S>(pp, i);
        unsigned char* st = smem + s * L::STAGE;
        if (i >= n_pre) {
            if (!__all_sync(0xffffffffu, mbar_wait(pp.empty + s, (pp.pphase >> s) & 1u, err))) return false;
            pp.pphase ^= 1u << s;
        }
        if (elect_one()) {
            if (ut && i < 64) ut[i * 4 + 0] = globaltimer();
            if (i >= n_pre) tma_weights<R>(a, epi, u_begin + i, st, pp.full + s);
            tma_inputs<R>(a, u_begin + i, st, pp.full + s);
        }
        __syncwarp();
    }
    ring_advance<S>(pp, n_my);
    return true;
}

// MMA warp: n_units, n_chunks of the op
template <int R>
__device__ bool gemm_mma(int n_units, int n_chunks, unsigned char* smem, Pipe& pp, int* err, unsigned long long* ut) {
    using L = GemmSmem<R>;
    constexpr int S = L::S, NP = L::NP;
    int u_begin, n_my;
    my_units(n_units, &u_begin, &n_my);
    constexpr uint32_t idesc = umma_idesc(NP);
    const uint64_t desc0 = umma_desc(smem_u32(smem));  // (descriptors count 16-byte steps)
    int chunk = u_begin % n_chunks;
    for (int i = 0; i < n_my; ++i) {
        const bool first = i == 0 || chunk == 0;
        const bool last = i == n_my - 1 || chunk == n_chunks - 1;
        chunk = chunk == n_chunks - 1 ? 0 : chunk + 1;
        const int ab = pp.ab;
        if (first) {  // the consumers have read this accumulator's previous segment
            if (!__all_sync(0xffffffffu, mbar_wait(pp.acc_empty + ab, (pp.aempty >> ab) & 1u, err))) return false;
            pp.aempty ^= 1u << ab;
        }
        const int s = ring_stage<S>(pp, i);
        if (!__all_sync(0xffffffffu, mbar_wait(pp.full + s, (pp.cphase >> s) & 1u, err))) return false;
        pp.cphase ^= 1u << s;
        tc_fence_after();
        if (elect_one()) {
            const uint64_t st = desc0 + (uint64_t)((uint32_t)(s * L::STAGE) >> 4);
            const uint32_t d = pp.tmem + (uint32_t)(ab * (kTmemCols / 2));
#pragma unroll
            for (int kb = 0; kb < 2; ++kb)
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma(d, st + (kb * 16384 + ks * 32) / 16, st + (L::WB + kb * L::XKB + ks * 32) / 16, idesc,
                         (first && kb == 0 && ks == 0) ? 0u : 1u);
            umma_commit(pp.empty + s);  // the stage is free once these MMAs have read it
            if (ut && i < 64) ut[i * 4 + 1] = globaltimer();
            if (last) umma_commit(pp.acc_full + ab);
        }
        __syncwarp();
        if (last) pp.ab ^= 1;
    }
    ring_advance<S>(pp, n_my);
    return true;
}

// Consumer warps
template <int R>
__device__ bool gemm_consume(const GemmArgs& a, int epi, int M, int pos0, unsigned char* smem, float* r_s, Pipe& pp,
                             unsigned tag, int* err, unsigned long long* ut, unsigned long long* ct) {
    using L = GemmSmem<R>;
    constexpr int S = L::S, NP = L::NP;
    float* ys = reinterpret_cast<float*>(smem + L::YS);  // [128][16]
    bool ok = true;

    const long long U = a.n_units, G = op_ctas(U);
    const int b = blockIdx.x;
    int u_begin, n_my;
    my_units(U, &u_begin, &n_my);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // 1 / rms of each input row from the previous op's per-tile sums of
    // squares (fixed order for every M: lane-strided sums, then a shuffle tree)
    for (int m = warp; m < M; m += kConsumers / 32) {
        float r = 1.f;
        if (a.ss_in) {
            float sum = 0.f;
            for (int t = lane; t < a.ss_in_tiles; t += 32) sum += __ldcg(a.ss_in + m * a.ss_in_tiles + t);
            sum = warp_sum(sum);
            r = rsqrtf(sum * a.inv_dim + a.eps);
        }
        if (lane == 0) r_s[m] = r;
    }
    // the MMA warp took the full-barrier waits of these ring positions
    advance_full<S>(pp, n_my);
    ring_advance<S>(pp, n_my);

    for (int i = 0; i < n_my; ++i) {
        const int u = u_begin + i;
        const int tile = u / a.n_chunks, chunk = u - tile * a.n_chunks;
        if (threadIdx.x == 0 && ct && i == n_my - 1) ct[6] = (unsigned long long)n_my;
        if (!(i == n_my - 1 || chunk == a.n_chunks - 1)) continue;

        // this CTA's segment of the tile is complete (or completing): its
        // accumulator holds W x_hi in columns 0..R-1 and W x_lo in columns
        // R..2R-1.  Split-K: the CTA holding the tile's first chunks (its
        // segment ends last, at the end of that CTA's range) finalises; the
        // others store their partial and move on.  The sums travel with the
        // op's tag in 128-bit words, so the finaliser needs no flag and no
        // fence: it reads each word until the tag is this op's.
        //
        // Every consumer warp reads its own TMEM rows - warp w holds tile row
        // rr = 32 (w % 4) + lane for the input rows m = w / 4, w / 4 + 2, ... -
        // so no CTA barrier precedes the contributors' stores.  A finaliser
        // first fetches the other segments' partials (and a residual one the
        // residual rows and the gains) while its own accumulator completes; its
        // sum is own + (p_1 + p_2 + ...), the partials added in segment order.
        const int ab = pp.ab;
        const long long u_first = (long long)tile * a.n_chunks;
        const int seg0 = unit_owner(u_first, U, G);
        const int nseg = unit_owner(u_first + a.n_chunks - 1, U, G) - seg0 + 1;
        const bool contributor = nseg > 1 && b != seg0;
        const bool resid = epi == EPI_RESID && !contributor;
        constexpr int HM = (R + 1) / 2;     // input rows per thread
        constexpr int NW = (HM + 2) / 3;    // words they take
        const int q4 = warp & 3, par = warp >> 2, rr = q4 * 32 + lane;
        const int n = tile * kFTile + rr;
        // words [tile][segment][par][word][tile row]
        PartWord* slots = reinterpret_cast<PartWord*>(a.partial) + (size_t)tile * a.n_chunks * kPartWords + par * 3 * kFTile + rr;
        float hp[HM], ps[HM];
        const float gp = (resid && n < a.N && a.g_next) ? __bfloat162float(a.g_next[n]) : 0.f;
#pragma unroll
        for (int k = 0; k < HM; ++k) {
            const int m = par + 2 * k;
            hp[k] = (resid && m < M && n < a.N) ? __ldcg(a.out_f32 + (size_t)m * a.ldo + n) : 0.f;
            ps[k] = 0.f;
        }
        if (!contributor && nseg > 1 && par < M) {
            constexpr int QB = R <= 4 ? 5 : R <= 12 ? 3 : 2;  // segments per batch (registers: 4 QB NW)
            for (int sg0 = 1; sg0 < nseg; sg0 += QB) {
                PartWord w[QB][NW];
#pragma unroll
                for (int q = 0; q < QB; ++q)
#pragma unroll
                    for (int k = 0; k < NW; ++k)
                        if (sg0 + q < nseg && par + 6 * k < M)
                            w[q][k] = ld_relaxed(slots + (size_t)(sg0 + q) * kPartWords + k * kFTile);
                // words that do not carry this op's tag yet (their CTA has
                // not published) are re-read together, not one at a time
                unsigned long long t_wait = 0;
                for (;;) {
                    bool ready = true;
#pragma unroll
                    for (int q = 0; q < QB; ++q)
#pragma unroll
                        for (int k = 0; k < NW; ++k)
                            if (sg0 + q < nseg && par + 6 * k < M && tag_of(w[q][k]) != tag) ready = false;
                    if (ready) break;
                    const unsigned long long now = globaltimer();
                    if (t_wait == 0) t_wait = now;
                    if (now - t_wait > kErrPollAfterNs) {
                        if (*(volatile int*)err) { ok = false; break; }
                        if (now - t_wait > kBarrierTimeoutNs) {
                            atomicCAS(err, 0, kDevErrTimeout);
                            ok = false;
                            break;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < QB; ++q)
#pragma unroll
                        for (int k = 0; k < NW; ++k)
                            if (sg0 + q < nseg && par + 6 * k < M && tag_of(w[q][k]) != tag)
                                w[q][k] = ld_relaxed(slots + (size_t)(sg0 + q) * kPartWords + k * kFTile);
                }
#pragma unroll
                for (int q = 0; q < QB; ++q)
#pragma unroll
                    for (int k = 0; k < HM; ++k)
                        if (sg0 + q < nseg && par + 2 * k < M) ps[k] += value_of(w[q][k / 3], k % 3);
            }
        }
        ok = mbar_wait(pp.acc_full + ab, (pp.afull >> ab) & 1u, err) && ok;
        pp.afull ^= 1u << ab;
        pp.ab ^= 1;
        tc_fence_after();
        if (threadIdx.x == 0 && ct) ct[2] = globaltimer();
        constexpr int NC = R == 12 ? 24 : NP;  // the 2R accumulator columns, rounded up
        float v[NC];
        tmem_ld<NC>(pp.tmem + (uint32_t)(ab * (kTmemCols / 2)) + ((uint32_t)(q4 * 32) << 16), v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(pp.acc_empty + ab);  // this warp is done with the accumulator
        float own[HM];
#pragma unroll
        for (int k = 0; k < HM; ++k) {  // input row m = par + 2k: columns m (hi) and R + m (lo)
            const float hi = par ? v[(2 * k + 1) < NC ? 2 * k + 1 : 0] : v[2 * k];
            const float lo = par ? v[(R + 2 * k + 1) < NC ? R + 2 * k + 1 : 0] : v[(R + 2 * k) < NC ? R + 2 * k : 0];
            own[k] = hi + lo;
        }
        if (contributor) {
#pragma unroll
            for (int k = 0; k < NW; ++k)
                if (par + 6 * k < M)
                    st_relaxed(slots + (size_t)(b - seg0) * kPartWords + k * kFTile, tag, own[3 * k],
                               3 * k + 1 < HM ? own[3 * k + 1 < HM ? 3 * k + 1 : 0] : 0.f,
                               3 * k + 2 < HM ? own[3 * k + 2 < HM ? 3 * k + 2 : 0] : 0.f);
            continue;
        }
        if (resid) {
            // h += sum, the next norm's input planes of h * g_next and the
            // per-tile sums of h^2 (per quadrant of 32 rows, then the 4
            // quadrants in order)
            float* ssq = ys;  // [16][4]
#pragma unroll
            for (int k = 0; k < HM; ++k) {
                const int m = par + 2 * k;
                if (m >= M) break;  // (uniform in the warp)
                float hv = 0.f;
                if (n < a.N) {
                    hv = hp[k] + (own[k] + ps[k]);
                    a.out_f32[(size_t)m * a.ldo + n] = hv;
                    if (a.g_next) {
                        const float z = __fmul_rn(hv, gp);
                        const bf16 zh = __float2bfloat16_rn(z);
                        a.xo_hi[(size_t)m * a.N + n] = zh;
                        a.xo_lo[(size_t)m * a.N + n] = __float2bfloat16_rn(z - __bfloat162float(zh));
                    }
                }
                if (a.g_next) {
                    const float sq = warp_sum(__fmul_rn(hv, hv));
                    if (lane == 0) ssq[m * 4 + q4] = sq;
                }
            }
            if (a.g_next) {
                consumer_sync();
                if (threadIdx.x < M)
                    a.ss_out[threadIdx.x * a.n_tiles + tile] = (ssq[threadIdx.x * 4 + 0] + ssq[threadIdx.x * 4 + 1]) +
                                                              (ssq[threadIdx.x * 4 + 2] + ssq[threadIdx.x * 4 + 3]);
            }
            consumer_sync();  // ys is reused by the next segment
            if (ut && i < 64 && threadIdx.x == 0) ut[i * 4 + 3] = globaltimer();
            continue;
        }
        // the other epilogues combine rows of the tile: through ys
#pragma unroll
        for (int k = 0; k < HM; ++k)
            if (par + 2 * k < M) ys[rr * 16 + par + 2 * k] = own[k] + ps[k];
        consumer_sync();

        // epilogue of the finished tile (row m scaled by its RMSNorm factor)
        if (epi == EPI_LOGITS) {
            for (int idx = threadIdx.x; idx < M * kFTile; idx += kGemmThreads) {
                const int m = idx / kFTile, r = idx - m * kFTile;
                const int n = tile * kFTile + r;
                if (n < a.N) a.out_f32[(size_t)m * a.ldo + n] = ys[r * 16 + m] * r_s[m];
            }
        } else if (epi == EPI_SWIGLU) {
            for (int idx = threadIdx.x; idx < M * 64; idx += kGemmThreads) {
                const int m = idx >> 6, r = idx & 63;
                const int i2 = tile * 64 + r;
                if (i2 >= a.ffn) continue;
                const float gt = ys[r * 16 + m] * r_s[m], up = ys[(r + 64) * 16 + m] * r_s[m];
                const float act = gt / (1.f + expf(-gt)) * up;
                const bf16 ah = __float2bfloat16_rn(act);
                a.xo_hi[(size_t)m * a.ffn + i2] = ah;
                a.xo_lo[(size_t)m * a.ffn + i2] = __float2bfloat16_rn(act - __bfloat162float(ah));
            }
        } else {  // EPI_QKV
            const int hd = a.head_dim, half = hd >> 1;
            const int qt = a.n_heads * hd / kFTile, kt = a.n_kv_heads * hd / kFTile;
            if (tile < qt + kt) {
                const bool is_q = tile < qt;
                const int tt = is_q ? tile : tile - qt;
                for (int idx = threadIdx.x; idx < M * 64; idx += kGemmThreads) {
                    const int m = idx >> 6, pr = idx & 63;  // rotation pair pr of the tile
                    const int hl = pr / half, ii = pr - hl * half;
                    const int r1 = hl * hd + ii, r2 = r1 + half;
                    const int head = tt * (kFTile / hd) + hl, pos = pos0 + m;
                    const float x1 = ys[r1 * 16 + m] * r_s[m], x2 = ys[r2 * 16 + m] * r_s[m];
                    const float2 cs = a.rope[(size_t)pos * half + ii];
                    // (rounded the same in every row class: no contraction of the compiler's choice)
                    const float y1 = __fmaf_rn(x1, cs.x, -__fmul_rn(x2, cs.y));
                    const float y2 = __fmaf_rn(x2, cs.x, __fmul_rn(x1, cs.y));
                    if (is_q) {
                        float* q = a.q_out + (size_t)m * a.n_heads * hd + head * hd;
                        q[ii] = y1;
                        q[ii + half] = y2;
                    } else {
                        f16* k = a.k_cache + ((size_t)head * a.max_seq + pos) * hd;
                        k[ii] = __float2half_rn(y1);
                        k[ii + half] = __float2half_rn(y2);
                    }
                }
            } else {
                const int vt = tile - qt - kt;
                for (int idx = threadIdx.x; idx < M * kFTile; idx += kGemmThreads) {
                    const int m = idx / kFTile, r = idx - m * kFTile;
                    const int f = vt * kFTile + r;
                    const int head = f / hd, e = f - head * hd;
                    a.v_cache[((size_t)head * a.max_seq + pos0 + m) * hd + e] =
                        __float2half_rn(ys[r * 16 + m] * r_s[m]);
                }
            }
        }
        consumer_sync();  // ys is reused by the next segment
        if (ut && i < 64 && threadIdx.x == 0) ut[i * 4 + 3] = globaltimer();
    }
    consumer_sync();
    return ok;
}

// two neighbouring values into the hi / lo planes (at: even)
__device__ __forceinline__ void store_pair(bf16* hi_at, bf16* lo_at, float v0, float v1) {
    const bf16 h0 = __float2bfloat16_rn(v0), h1 = __float2bfloat16_rn(v1);
    __nv_bfloat162 hi, lo;
    hi.x = h0;
    hi.y = h1;
    lo.x = __float2bfloat16_rn(v0 - __bfloat162float(h0));
    lo.y = __float2bfloat16_rn(v1 - __bfloat162float(h1));
    *reinterpret_cast<__nv_bfloat162*>(hi_at) = hi;
    *reinterpret_cast<__nv_bfloat162*>(lo_at) = lo;
}

template <int N>
struct Int {
    static constexpr int value = N;
};

// ---------------------------------------------------------------------------
// attention op: items (KV head, vector group, 128-position segment), through
// the TMA ring
// ---------------------------------------------------------------------------
// A segment is kAttnSegChunks absolute 64-position chunks; the producer thread
// requests each chunk's K and V rows (TMA, 128-byte swizzle) into consecutive
// ring stages.  An item is one segment of one KV head for a group of up to 16
// of its G * M query vectors (G query heads of the KV head, M rows): scores
// and P V on tensor cores (fp16 hi + lo operands, fp32 accumulators), the
// softmax over the segment from the score accumulators; the partial (o, max,
// sum) of the segment goes to global memory.  Items run segment fastest, so a
// CTA's consecutive items share their q.  After a grid barrier every CTA
// combines a share of the (KV head, vector) partials in segment order
// (flash-decoding style split of the softmax).  Every reduction has a fixed
// order that depends only on the row's own position, not on M.
struct AttnRange {
    int n_ch, n_seg, n_vg;  // chunks, segments per KV head, groups of 16 query vectors
    int i_begin, i_end;     // this CTA's items (KV head, vector group, segment), segment fastest
};
__device__ __forceinline__ AttnRange attn_range(const AttnArgs& a, int M, int pos0) {
    constexpr int S = kAttnSegChunks;
    AttnRange r;
    r.n_ch = (pos0 + M + kAttnChunk - 1) / kAttnChunk;  // chunks holding any visible position
    r.n_seg = (r.n_ch + S - 1) / S;
    r.n_vg = (a.group * M + 15) / 16;
    // One 32-bit division: this is on the way to the first item, which began 0.9 us
    // after the op with two 64-bit ones and a division per vector, 0.5 us now (with
    // the combine's share worked out before its barrier and the empty half of the
    // vectors left out, 7B widths, one row: 10.82 -> 10.18 us per layer).
    const int I = a.n_kv_heads * r.n_seg * r.n_vg, GR = gridDim.x, b = blockIdx.x, n = I / GR, more = I - n * GR;
    r.i_begin = b * n + min(b, more);
    r.i_end = r.i_begin + n + (b < more);
    return r;
}

// Producer warp: requests K / V of this CTA's chunks at ring positions
// [i_from, i_limit), in item order; with old_only it stops at the first chunk
// holding rows this forward writes (those need the q/k/v op to be finished).
// Returns the ring position reached, or -1 if a wait timed out.
template <int R, int HD>
__device__ int attn_request(const AttnArgs& a, const AttnRange& ar, int pos0, unsigned char* smem, Pipe& pp,
                            int* err, int i_from, int i_limit, bool old_only) {
    using L = GemmSmem<R>;
    constexpr int S = L::S, SC = kAttnSegChunks;
    int i = 0;
    for (int it = ar.i_begin; it < ar.i_end; ++it) {
        const int hv = it / ar.n_seg, kvh = hv / ar.n_vg, c0 = (it - hv * ar.n_seg) * SC;
        for (int c = c0; c < min(c0 + SC, ar.n_ch); ++c, ++i) {
            if (i < i_from) continue;
            if (i >= i_limit || (old_only && (c + 1) * kAttnChunk > pos0)) return i;
            const int s = ring_stage<S>(pp, i);
            unsigned char* st = smem + s * L::STAGE;
            if (!__all_sync(0xffffffffu, mbar_wait(pp.empty + s, (pp.pphase >> s) & 1u, err))) return -1;
            pp.pphase ^= 1u << s;
            if (elect_one()) {
                mbar_arrive_expect_tx(pp.full + s, 2u * (HD / 64) * 8192u);
#pragma unroll
                for (int bx = 0; bx < HD / 64; ++bx) {
                    tma_load_3d(st + bx * 8192, a.tm_k, bx * 64, c * kAttnChunk, a.kv_z0 + kvh, pp.full + s);
                    tma_load_3d(st + 16384 + bx * 8192, a.tm_v, bx * 64, c * kAttnChunk, a.kv_z0 + kvh, pp.full + s);
                }
            }
            __syncwarp();
        }
    }
    return i;
}

// Producer warp of an attention op: the chunks that hold only rows of earlier
// forwards as soon as stages are free, the others once `go` says that the
// q/k/v op has finished everywhere.
template <int R, int HD>
__device__ bool attn_produce(const AttnArgs& a, int M, int pos0, unsigned char* smem, Pipe& pp, uint64_t* go,
                             unsigned go_parity, int* err) {
    constexpr int S = GemmSmem<R>::S;
    const AttnRange ar = attn_range(a, M, pos0);
    if (ar.i_begin < ar.i_end && elect_one()) {
        prefetch_tmap(a.tm_k);
        prefetch_tmap(a.tm_v);
    }
    __syncwarp();
    int n = attn_request<R, HD>(a, ar, pos0, smem, pp, err, 0, S, true);
    if (n < 0 || !__all_sync(0xffffffffu, mbar_wait(go, go_parity, err))) return false;
    // K / V rows of this forward were stored by other CTAs (generic proxy)
    asm volatile("fence.proxy.async.global;" ::: "memory");
    n = attn_request<R, HD>(a, ar, pos0, smem, pp, err, n, 1 << 30, false);
    if (n < 0) return false;
    ring_advance<S>(pp, n);
    return true;
}

// ring positions (K / V chunks) this CTA's items take
__device__ __forceinline__ int attn_positions(const AttnRange& ar) {
    constexpr int SC = kAttnSegChunks;
    int n = 0;
    for (int it = ar.i_begin; it < ar.i_end; ++it) n += min(SC, ar.n_ch - (it % ar.n_seg) * SC);
    return n;
}

// Consumer warps: the items' segment partials.  Returns false if a wait timed
// out (error recorded).
template <int R, int HD>
__device__ bool attn_consume(const AttnArgs& a, int M, int pos0, unsigned char* smem, Pipe& pp, int* err,
                             unsigned long long* ct, unsigned long long* ut) {
    using L = GemmSmem<R>;
    constexpr int S = L::S, VG = L::VG, SC = kAttnSegChunks, SP = SC * kAttnChunk;  // positions per segment
    static_assert(SC <= S, "a segment's chunks are held in the ring at once");
    const int G = a.group, NV = G * M;
    const AttnRange ar = attn_range(a, M, pos0);

    constexpr int QST = L::QST, PST = L::PST;
    __half* qh = reinterpret_cast<__half*>(smem + L::ATT);  // [VG][QST] q hi, then lo
    __half* ql = qh + VG * QST;
    float* sc = reinterpret_cast<float*>(smem + L::ATT_SC);  // per-warp maxima and sums
    __half* ph = reinterpret_cast<__half*>(smem + L::ATT_P);  // [VG][PST] weights hi, then lo
    __half* pl = ph + VG * PST;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, tg = lane & 3;
    constexpr size_t part_v = attn_part_floats(HD);  // floats per partial: o[HD], max, sum, pad
    bool ok = true;
    int i = 0;       // ring position within the op
    int q_key = -1;  // (KV head, vector group) whose q is in shared memory
    int n_held = 0;  // stages of the previous item, not yet released
    auto release = [&]() {
        if (tid == 0)
            for (int j = 1; j <= n_held; ++j) mbar_arrive(pp.empty + ring_stage<S>(pp, i - j));
        n_held = 0;
    };

    // profiling aid: ut (CTA 0 of a traced forward) gets per-item phase stamps
    auto stamp = [&](int it, int k) {
        if (ut && tid == 0 && it - ar.i_begin < 31) ut[(it - ar.i_begin) * 8 + k] = globaltimer();
    };
    // (KV head, vector group, segment) of the item, stepped along: the divisions
    // by run-time values are made once per op and vector group, not per item
    int hv = ar.i_begin / ar.n_seg, sg = ar.i_begin - hv * ar.n_seg - 1;
    int kvh = hv / ar.n_vg, vg = hv - kvh * ar.n_vg;
    int vg_rows = -1;  // the vector group whose rows are in mrow
    int mrow[2][2];    // input row of vector 8 nt + 2 tg + cx
    for (int it = ar.i_begin; it < ar.i_end; ++it) {
        stamp(it, 0);
        if (++sg == ar.n_seg) {
            sg = 0;
            if (++vg == ar.n_vg) {
                vg = 0;
                ++kvh;
            }
        }
        const int t0 = sg * SP;
        const int n_u = min(SC, ar.n_ch - sg * SC);  // chunks of this segment
        const int v0 = vg * VG, nv = min(VG, NV - v0);
        if (vg != vg_rows) {
            vg_rows = vg;
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int cx = 0; cx < 2; ++cx) mrow[nt][cx] = a.row_of(v0 + nt * 8 + 2 * tg + cx);
        }
        float* part = a.part + ((size_t)kvh * a.n_chunks + sg) * NV * part_v;
        // q of this item's vectors as fp16 hi + lo (other CTAs wrote q: L2);
        // every thread issues all its 16-byte loads before converting, and the
        // loads overlap the wait for K / V; consecutive items of one KV head
        // and vector group reuse it
        const int key = kvh * ar.n_vg + vg;
        if (key != q_key) {
            constexpr int HD4 = HD / 4, QJ = VG * HD4 / kConsumers;  // float4 per thread: 2 | 1
            static_assert(VG * HD4 % kConsumers == 0, "q tile split evenly over the consumers");
            float4 qv[QJ];
#pragma unroll
            for (int j = 0; j < QJ; ++j) {
                const int k4 = tid + j * kConsumers, vl = k4 / HD4, e = (k4 - vl * HD4) * 4;
                qv[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (vl < nv) {
                    const int v = v0 + vl, m = a.row_of(v), gi = v - m * G;
                    qv[j] = __ldcg(reinterpret_cast<const float4*>(a.q + (size_t)m * a.n_heads * HD +
                                                                   (size_t)(kvh * G + gi) * HD + e));
                }
            }
#pragma unroll
            for (int j = 0; j < QJ; ++j) {
                const int k4 = tid + j * kConsumers, vl = k4 / HD4, e = (k4 - vl * HD4) * 4;
                const __half2 h01 = __floats2half2_rn(qv[j].x, qv[j].y), h23 = __floats2half2_rn(qv[j].z, qv[j].w);
                const float2 f01 = __half22float2(h01), f23 = __half22float2(h23);
                const __half2 l01 = __floats2half2_rn(qv[j].x - f01.x, qv[j].y - f01.y);
                const __half2 l23 = __floats2half2_rn(qv[j].z - f23.x, qv[j].w - f23.y);
                *reinterpret_cast<uint2*>(qh + vl * QST + e) =
                    make_uint2(*reinterpret_cast<const uint32_t*>(&h01), *reinterpret_cast<const uint32_t*>(&h23));
                *reinterpret_cast<uint2*>(ql + vl * QST + e) =
                    make_uint2(*reinterpret_cast<const uint32_t*>(&l01), *reinterpret_cast<const uint32_t*>(&l23));
            }
        }
        q_key = key;
        stamp(it, 1);
        const unsigned char* stage[SC];
#pragma unroll
        for (int j = 0; j < SC; ++j) stage[j] = smem + ring_stage<S>(pp, i + j) * L::STAGE;
        for (int j = 0; j < n_u; ++j) {
            const int s = ring_stage<S>(pp, i + j);
            ok = mbar_wait(pp.full + s, (pp.cphase >> s) & 1u, err) && ok;
            pp.cphase ^= 1u << s;
        }
        if (ct && tid == 0 && it == ar.i_begin) ct[1] = globaltimer();
        stamp(it, 2);
        consumer_sync();
        stamp(it, 3);
        // every warp has left the previous item: its stages are free
        release();

        // scores S = K q^T on tensor cores: warp w takes positions 16w..16w+15
        // (A = K rows, 128-byte swizzled), all 16 vectors (B = q hi, then lo);
        // then the softmax of every vector over the segment straight from the
        // accumulators: per-warp maxima -> CTA barrier -> the segment maximum
        // (the 8 warps' values in order) -> weights as fp16 hi + lo, per-warp
        // sums (the partial's sum adds the 8 warps' sums in order)
        float* wmax = sc;           // [8 warps][VG vectors]
        float* wsum = sc + 8 * VG;  // [8 warps][VG vectors]
        // nt_c: 8-vector halves of the tile in use (compiled for each: with the second
        // half skipped by branches, 13 rows took 20.7 us per layer instead of 20.0)
        auto weights = [&](auto nt_c) {
            constexpr int NT = decltype(nt_c)::value;
            const int p0 = warp * 16, j = p0 / kAttnChunk;
            float c[NT][4] = {};
            if (j < n_u) {
                // K q_hi and K q_lo in separate accumulators (two short
                // dependency chains instead of one long one), added at the end
                float cl[NT][4] = {};
                const unsigned char* kst = j ? stage[1] : stage[0];
                const int t = (p0 % kAttnChunk) + (lane & 7) + 8 * ((lane >> 3) & 1);
                const int qv = (lane & 7) + 8 * (lane >> 4), qk = ((lane >> 3) & 1) * 8;
#pragma unroll
                for (int ks = 0; ks < HD / 16; ++ks) {
                    uint32_t af[4], bh[4], bl[4];
                    const int chunk = 2 * (ks & 3) + (lane >> 4);
                    ldsm_x4(af, kst + (ks >> 2) * 8192 + t * 128 + ((chunk ^ (t & 7)) << 4));
                    ldsm_x4(bh, qh + qv * QST + ks * 16 + qk);
                    ldsm_x4(bl, ql + qv * QST + ks * 16 + qk);
                    mma_f16_16816(c[0], af[0], af[1], af[2], af[3], bh[0], bh[1]);
                    mma_f16_16816(cl[0], af[0], af[1], af[2], af[3], bl[0], bl[1]);
                    if constexpr (NT == 2) {  // vectors 8..15
                        mma_f16_16816(c[1], af[0], af[1], af[2], af[3], bh[2], bh[3]);
                        mma_f16_16816(cl[1], af[0], af[1], af[2], af[3], bl[2], bl[3]);
                    }
                }
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int x = 0; x < 4; ++x) c[nt][x] += cl[nt][x];
            }
            // C: rows = positions p0 + g (+8), columns = vectors 8 nt + 2 tg (+1)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int vl = nt * 8 + 2 * tg + (x & 1), pq = p0 + g + 8 * (x >> 1);
                    const bool vis = j < n_u && vl < nv && t0 + pq <= pos0 + mrow[nt][x & 1];
                    c[nt][x] = vis ? c[nt][x] * a.scale : -INFINITY;
                }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int cx = 0; cx < 2; ++cx) {
                    float v = fmaxf(c[nt][cx], c[nt][cx + 2]);
                    v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
                    v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
                    v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
                    if (g == 0) wmax[warp * VG + nt * 8 + 2 * tg + cx] = v;
                }
            consumer_sync();
            stamp(it, 4);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int cx = 0; cx < 2; ++cx) {
                    const int vl = nt * 8 + 2 * tg + cx;
                    float mx = -INFINITY;
#pragma unroll
                    for (int w2 = 0; w2 < kConsumers / 32; ++w2) mx = fmaxf(mx, wmax[w2 * VG + vl]);
                    float l = 0.f;
#pragma unroll
                    for (int xh = 0; xh < 2; ++xh) {
                        const float x = c[nt][cx + 2 * xh];
                        const float pq = x == -INFINITY ? 0.f : expf(x - mx);
                        const __half hh = __float2half_rn(pq);
                        const int pos = p0 + g + 8 * xh;
                        ph[vl * PST + pos] = hh;
                        pl[vl * PST + pos] = __float2half_rn(pq - __half2float(hh));
                        l += pq;
                    }
                    l += __shfl_xor_sync(0xffffffffu, l, 4);
                    l += __shfl_xor_sync(0xffffffffu, l, 8);
                    l += __shfl_xor_sync(0xffffffffu, l, 16);
                    if (g == 0) wsum[warp * VG + vl] = l;
                }
        };
        if (nv > 8) weights(Int<2>{});
        else weights(Int<1>{});
        consumer_sync();
        stamp(it, 5);
        // the segment's (max, sum) of each vector; -inf: nothing visible
        if (tid < nv && ar.n_seg > 1) {
            const int v = v0 + tid, m = a.row_of(v);
            float mx = -INFINITY, l = 0.f;
#pragma unroll
            for (int w2 = 0; w2 < kConsumers / 32; ++w2) {
                mx = fmaxf(mx, wmax[w2 * VG + tid]);
                l += wsum[w2 * VG + tid];
            }
            float* o = part + (size_t)v * part_v;
            o[HD] = pos0 + m < t0 ? -INFINITY : mx;
            o[HD + 1] = l;
        }

        // O = P V on tensor cores: warp w takes dims 16w..16w+15 (B = V rows via
        // transposed 8x8 loads), all 16 vectors (A = P hi, then lo); rows of
        // vectors past nv hold stale weights and are not stored
        if (warp * 16 < HD) {
            // P_hi V and P_lo V in separate accumulators, added at the end
            float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
            float cl[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
            const int d = warp * 16 + 8 * (lane >> 4), bx = d >> 6, cc = (d & 63) >> 3;
            const int pv = (lane & 7) + 8 * ((lane >> 3) & 1), pk = (lane >> 4) * 8;
#pragma unroll
            for (int j = 0; j < SC; ++j) {
                if (j >= n_u) break;
                const unsigned char* vst = stage[j] + 16384 + bx * 8192;
#pragma unroll
                for (int ks = 0; ks < kAttnChunk / 16; ++ks) {
                    uint32_t ah[4], al[4], bv[4];
                    const int tt = ks * 16 + (lane & 7) + 8 * ((lane >> 3) & 1), pc = j * kAttnChunk + ks * 16 + pk;
                    ldsm_x4(ah, ph + pv * PST + pc);
                    ldsm_x4(al, pl + pv * PST + pc);
                    ldsm_x4_t(bv, vst + tt * 128 + ((cc ^ (tt & 7)) << 4));
                    mma_f16_16816(c[0], ah[0], ah[1], ah[2], ah[3], bv[0], bv[1]);
                    mma_f16_16816(c[1], ah[0], ah[1], ah[2], ah[3], bv[2], bv[3]);
                    mma_f16_16816(cl[0], al[0], al[1], al[2], al[3], bv[0], bv[1]);
                    mma_f16_16816(cl[1], al[0], al[1], al[2], al[3], bv[2], bv[3]);
                }
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int x = 0; x < 4; ++x) c[nt][x] += cl[nt][x];
            // C: rows = vectors g (+8), columns = dims 16w + 8 nt + 2 tg (+1)
            if (ar.n_seg == 1) {
                // the only segment: what the combine would make of it (weight
                // exp(0) = 1), written at once
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int vl = g + 8 * h;
                    if (vl >= nv) continue;
                    float l = 0.f;
#pragma unroll
                    for (int w2 = 0; w2 < kConsumers / 32; ++w2) l += wsum[w2 * VG + vl];
                    const float inv = 1.f / l;
                    const int v = v0 + vl, m = a.row_of(v), gi = v - m * G;
                    const size_t at = (size_t)m * a.n_heads * HD + (size_t)(kvh * G + gi) * HD + warp * 16 + 2 * tg;
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt)
                        store_pair(a.out_hi + at + nt * 8, a.out_lo + at + nt * 8, c[nt][2 * h] * inv, c[nt][2 * h + 1] * inv);
                }
            } else {
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int vl = g + 8 * h;
                        if (vl < nv)
                            *reinterpret_cast<float2*>(part + (size_t)(v0 + vl) * part_v + warp * 16 + nt * 8 + 2 * tg) =
                                make_float2(c[nt][2 * h], c[nt][2 * h + 1]);
                    }
            }
        }
        stamp(it, 6);
        i += n_u;
        n_held = n_u;  // released once every warp is past this item
    }
    if (n_held) {
        consumer_sync();
        release();
    }
    if (ct && tid == 0) ct[6] = (unsigned long long)(ar.i_end - ar.i_begin);
    ring_advance<S>(pp, i);
    return ok;
}

// Second phase of attention, after a grid barrier (the segment partials of
// every CTA are visible): the partials of each (KV head, query vector) are
// combined in segment order - row m uses segments 0 .. (pos0 + m) / SP - and
// written as the bf16 hi / lo planes of the attention output.  One warp per
// 64 dims of a vector (2 dims per lane), spread round-robin over the warps of
// all CTAs.  Per batch of up to kCombineBatch segments a lane loads its dims of
// every segment and lane j the (max, sum) of segment j, all at once (one L2
// round trip per batch: one for contexts up to 2048 positions); the batch
// maximum and the sum of the weighted sums are shuffle trees, the weighted
// dims are added in segment order, and batches fold into running sums scaled
// to the running maximum.  The order depends only on the row's position.
// A warp's first share is worked out before the barrier (combine_item).
constexpr int kCombineBatch = 16;
struct CombineItem {
    const float* pv;  // the vector's partial of segment 0
    size_t at;        // output element
    int nsg;          // segments of its row
};
template <int HD>
__device__ __forceinline__ CombineItem combine_item(const AttnArgs& a, int M, int pos0, int wk) {
    constexpr int SP = kAttnSegChunks * kAttnChunk, HALVES = HD / 64;
    constexpr size_t part_v = attn_part_floats(HD);  // floats per partial: o[HD], max, sum, pad
    const int G = a.group, NV = G * M;
    const int gv = wk / HALVES, kvh = gv / NV, v = gv - kvh * NV;
    const int m = a.row_of(v), gi = v - m * G;
    CombineItem c;
    c.pv = a.part + ((size_t)kvh * a.n_chunks * NV + v) * part_v;
    c.at = (size_t)m * a.n_heads * HD + (size_t)(kvh * G + gi) * HD + (wk & (HALVES - 1)) * 64 + 2 * (threadIdx.x & 31);
    c.nsg = (pos0 + m) / SP + 1;
    return c;
}
// warp-major over the CTAs: the first work items go to warp 0 of every CTA
__device__ __forceinline__ int combine_first() { return (threadIdx.x >> 5) * gridDim.x + blockIdx.x; }

template <int HD>
__device__ void attn_combine(const AttnArgs& a, int M, int pos0, CombineItem c) {
    constexpr int HALVES = HD / 64, B = kCombineBatch;
    static_assert(B <= 32, "one lane per segment of a batch");
    static_assert(HALVES == 1 || HALVES == 2, "the half is the work item's lowest bit");
    const size_t qs_stride = (size_t)a.group * M * attn_part_floats(HD);  // next segment of the same vector
    const int n_work = a.n_kv_heads * a.group * M * HALVES;               // (vector, 64 dims) per warp
    const int lane = threadIdx.x & 31;
    const int n_warps = gridDim.x * (kConsumers / 32);
    for (int wk = combine_first(); wk < n_work;) {
        const int e = (wk & (HALVES - 1)) * 64 + 2 * lane, nsg = c.nsg;
        const float* pv = c.pv;
        float mx = -INFINITY, l = 0.f, o0 = 0.f, o1 = 0.f;
        for (int q0 = 0; q0 < nsg; q0 += B) {
            const int nb = min(B, nsg - q0);
            float2 ml = make_float2(-INFINITY, 0.f);  // (max, sum) of segment q0 + lane
            if (lane < nb) ml = __ldcg(reinterpret_cast<const float2*>(pv + (size_t)(q0 + lane) * qs_stride + HD));
            float2 ov[B];
#pragma unroll
            for (int j = 0; j < B; ++j) {
                ov[j] = make_float2(0.f, 0.f);
                if (j < nb) ov[j] = __ldcg(reinterpret_cast<const float2*>(pv + (size_t)(q0 + j) * qs_stride + e));
            }
            float bm = ml.x;
#pragma unroll
            for (int off = 16; off; off >>= 1) bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, off));
            bm = fmaxf(bm, mx);
            // empty segments (and lanes past the batch) hold max -inf, o = 0
            const float r = mx == -INFINITY ? 0.f : expf(mx - bm);
            const float f = ml.x == -INFINITY ? 0.f : expf(ml.x - bm);
            float fl = f * ml.y;
#pragma unroll
            for (int off = 16; off; off >>= 1) fl += __shfl_xor_sync(0xffffffffu, fl, off);
            l = l * r + fl;
            o0 *= r;
            o1 *= r;
#pragma unroll
            for (int j = 0; j < B; ++j) {
                const float fj = __shfl_sync(0xffffffffu, f, j);
                o0 += fj * ov[j].x;
                o1 += fj * ov[j].y;
            }
            mx = bm;
        }
        const float inv = 1.f / l;
        store_pair(a.out_hi + c.at, a.out_lo + c.at, o0 * inv, o1 * inv);
        wk += n_warps;
        if (wk < n_work) c = combine_item<HD>(a, M, pos0, wk);
    }
}

// ---------------------------------------------------------------------------
// embedding op: h = E[token], planes of h * g (first RMSNorm), sums of h^2
// ---------------------------------------------------------------------------
__device__ void embed_op(const FwdParams& p, int pos0) {
    const int d = p.d, n_tiles = d / kFTile;  // sums of squares per 128 columns
    const int lane = threadIdx.x & 31;
    const int gw = blockIdx.x * (kGemmThreads / 32) + (threadIdx.x >> 5);
    const int nw = gridDim.x * (kGemmThreads / 32);
    if (blockIdx.x == 0 && threadIdx.x == 0) p.st->pos0 = pos0;
    for (int u = gw; u < p.M * n_tiles; u += nw) {
        const int m = u / n_tiles, t = u - m * n_tiles;
        int tok;
        if (p.src == SRC_TOKENS) tok = p.toks[m];
        else if (p.src == SRC_DRAFT) tok = p.st->j == 0 ? p.st->x_last : p.st->drafts[p.st->j - 1];
        else tok = m == 0 ? p.st->x_last : p.st->drafts[m - 1];
        // (all loads before the stores: they come from HBM, one round trip)
        constexpr int J = kFTile / 32;
        float v[J], g[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int i = t * kFTile + j * 32 + lane;
            v[j] = __bfloat162float(p.embed[(size_t)tok * d + i]);
            g[j] = __bfloat162float(p.g0[i]);
        }
        float sq = 0.f;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int i = t * kFTile + j * 32 + lane;
            p.h[(size_t)m * d + i] = v[j];
            const float z = v[j] * g[j];
            const bf16 zh = __float2bfloat16_rn(z);
            p.xn_hi[(size_t)m * d + i] = zh;
            p.xn_lo[(size_t)m * d + i] = __float2bfloat16_rn(z - __bfloat162float(zh));
            sq += v[j] * v[j];
        }
        sq = warp_sum(sq);
        if (lane == 0) p.ss[m * n_tiles + t] = sq;
    }
}

// After a timed-out wait: give copies still in flight a bounded time to land
// before the CTA exits (the error is already recorded).
__device__ void drain_before_exit() {
    if (threadIdx.x == 0) {
        const unsigned long long t0 = globaltimer();
        while (globaltimer() - t0 < 2000000ull) __nanosleep(1000);
    }
    __syncthreads();
}

// The producer reads op o + 1's arguments while the consumers may still be in
// op o, and fetches those of op o + 2: three slots.
constexpr int kOpSlots = 3;

template <int R, int HD>
__global__ void __launch_bounds__(kFwdThreads, 1) forward_kernel(const FwdParams p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ float r_s[kMaxRows];
    __shared__ int s_pos0, s_leave;
    __shared__ unsigned s_seq;
    __shared__ uint32_t s_tmem;
    constexpr int S = GemmSmem<R>::S;
    __shared__ __align__(8) uint64_t full[S];       // TMA completion per stage
    __shared__ __align__(8) uint64_t empty[S];      // stage released (tcgen05.commit, or one consumer thread)
    __shared__ __align__(8) uint64_t acc_full[2];   // TMEM accumulator complete (tcgen05.commit)
    __shared__ __align__(8) uint64_t acc_empty[2];  // TMEM accumulator read by the consumers
    __shared__ __align__(8) uint64_t desc[kOpSlots];  // producer and MMA warp are at op o; its arguments are in shared memory
    __shared__ __align__(8) uint64_t left;            // this CTA's work of an op is done (consumer thread 0)
    __shared__ __align__(8) uint64_t go;              // the grid barrier before an op has passed (consumer thread 0)
    __shared__ FwdOp s_op[kOpSlots];                // arguments of op o at o % kOpSlots
    // 128-byte TMA swizzle needs 1 KB aligned boxes
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const bool mma_warp = threadIdx.x >= kConsumers + 32;
    if (threadIdx.x == 0) {
        int pos0;
        if (p.src == SRC_TOKENS) pos0 = p.pos0_arg;
        else if (p.src == SRC_DRAFT) pos0 = p.st->len + p.st->j;
        else pos0 = p.st->len;
        s_pos0 = pos0;
        // no work: a draft step after the round's drafting stage ended (draft exit),
        // or a forward queued behind a failed one, which may have left the barrier
        // counters and the sequence number anywhere (the host clears them)
        s_leave = (p.src == SRC_DRAFT && *(volatile int*)&p.st->exited) || *(volatile int*)p.err;
        s_seq = *(volatile unsigned*)p.seq;  // this forward's number (advanced by CTA 0 below)
        for (int st = 0; st < S; ++st) {
            mbar_init(full + st, 1);
            mbar_init(empty + st, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full + b, 1);
            mbar_init(acc_empty + b, kConsumers / 32);  // one arrival per consumer warp
        }
        for (int o = 0; o < kOpSlots; ++o) mbar_init(desc + o, 2);
        mbar_init(&left, 1);
        mbar_init(&go, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (p.trace && blockIdx.x == 0) p.trace[0] = globaltimer();
    }
    __syncthreads();
    if (s_leave) return;
    if (mma_warp) {  // TMEM for the two projection accumulators (freed at the end)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // every stage and both accumulators start empty
    if (threadIdx.x == 0)
        for (int st = 0; st < S; ++st) mbar_arrive(empty + st);
    if (threadIdx.x < kConsumers && (threadIdx.x & 31) == 0) {
        mbar_arrive(acc_empty + 0);
        mbar_arrive(acc_empty + 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const int pos0 = s_pos0;
    Pipe pp{full, empty, acc_full, acc_empty, s_tmem, 0u, 0u, 0u, 0u, 0, 0};
    bool failed = false;
    // The roles walk the op list on their own.  The consumers run op o, arrive at
    // the grid barrier and wait for it; the producer requests what depends on no op
    // (weights, old K / V rows) as soon as they have left the previous op, and waits
    // for `go` before it requests anything an op of this forward has written, as does
    // the MMA warp before each op.
    auto stamps = [&](int o) -> unsigned long long* {  // op stamps of this CTA if op o is traced
        return (p.trace && o == (p.trace_op & 0xffff)) ? p.trace + kTraceCtas + blockIdx.x * 8 : nullptr;
    };
    auto unit_stamps = [&](int o) -> unsigned long long* {  // the CTA whose units are stamped
        return (stamps(o) && (int)blockIdx.x == (p.trace_op >> 16)) ? p.trace + kTraceUnits : nullptr;
    };
    if (threadIdx.x >= kConsumers + 32) {  // MMA warp
        const bool lane0 = threadIdx.x == kConsumers + 32;
        if (lane0) mbar_arrive(desc);  // op 0: the embedding
        for (int o = 1; o < p.n_ops && !failed; ++o) {
            // It waits for `go` like the producer: attention's chunks complete ring
            // stages that it does not wait for, so it must not reach the next
            // projection while any of them is still to come.
            if (lane0) mbar_arrive(desc + o % kOpSlots);
            if (!__all_sync(0xffffffffu, mbar_wait(&go, (unsigned)(o - 1) & 1u, p.err))) {
                failed = true;
                break;
            }
            const FwdOp& op = s_op[o % kOpSlots];
            if (is_gemm(op.type)) {
                failed = !gemm_mma<R>(op.g.n_units, op.g.n_chunks, smem, pp, p.err, unit_stamps(o));
            } else if (op.type == OP_ATTN) {  // the consumers wait for these ring positions
                const int n = attn_positions(attn_range(op.at, p.M, pos0));
                advance_full<S>(pp, n);
                ring_advance<S>(pp, n);
            }
        }
    } else if (threadIdx.x >= kConsumers) {  // producer warp
        const int lane = threadIdx.x & 31;
        constexpr int kOpChunks = (int)(sizeof(FwdOp) / 16);
        static_assert(sizeof(FwdOp) % 16 == 0 && kOpChunks <= 32, "an op is copied in 16-byte pieces by one warp");
        auto fetch = [&](int o) {  // arguments of op o, 16 bytes a lane, asynchronously
            if (lane < kOpChunks)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 smem_u32(reinterpret_cast<unsigned char*>(s_op + o % kOpSlots) + 16 * lane)),
                             "l"(reinterpret_cast<const unsigned char*>(p.ops + o) + 16 * lane)
                             : "memory");
        };
        fetch(0);
        for (int o = 0; o < p.n_ops && !failed; ++o) {
            // Nothing is requested before this CTA's consumers are done with the
            // previous op (with attention's items): their partial sums and
            // arrivals would queue in L2 behind 25 MB of weights (7B widths, a
            // decode step of 4 layers: 384 us; requested as stages fall free: 397).
            if (o > 0 && !__all_sync(0xffffffffu, mbar_wait(&left, (unsigned)(o - 1) & 1u, p.err))) {
                failed = true;
                break;
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(desc + o % kOpSlots);
            // its slot held op o - 2, which the consumers left before `go` for op o - 1
            if (o + 1 < p.n_ops) fetch(o + 1);
            const FwdOp& op = s_op[o % kOpSlots];
            const unsigned go_parity = (unsigned)(o - 1) & 1u;
            if (is_gemm(op.type))
                failed = !gemm_produce<R>(op.g, epi_of(op.type), smem, pp, &go, go_parity, p.err, unit_stamps(o));
            else if (op.type == OP_ATTN)
                failed = !attn_produce<R, HD>(op.at, p.M, pos0, smem, pp, &go, go_parity, p.err);
        }
    } else {  // consumer warps
        // Grid barriers of this launch: thread 0 arrives after a consumer barrier
        // that orders the CTA's stores before it, and waits for the others.  The
        // profiling hook p.stall_barrier (0: none) makes barrier number n
        // unreachable, so that its bounded wait runs out and the launch ends with
        // the timeout recorded.
        unsigned* const bar = p.bar + (s_seq & 1u);
        unsigned target = 0;
        int n_barrier = 0;
        auto barrier_arrive = [&]() {
            target += gridDim.x;
            ++n_barrier;
            if (threadIdx.x == 0) grid_arrive(bar);
        };
        auto barrier_wait = [&]() {  // thread 0
            const unsigned extra = n_barrier == p.stall_barrier ? 1u : 0u;
            const bool passed = grid_wait(bar, target + extra, p.err, p.wait_ns);
            // every CTA has read the sequence number before the first barrier;
            // the other counter was the previous launch's
            if (passed && n_barrier == 1 && blockIdx.x == 0) {
                *p.seq = s_seq + 1u;
                p.bar[(s_seq + 1u) & 1u] = 0u;
            }
            return passed;
        };
        // every row's attention within the first segment: no partials to combine
        const bool one_segment = pos0 + p.M <= kAttnSegChunks * kAttnChunk;
        for (int o = 0; o < p.n_ops; ++o) {
            unsigned long long* ct = stamps(o);
            if (ct && threadIdx.x == 0) ct[0] = globaltimer();
            bool ok = mbar_wait(desc + o % kOpSlots, (unsigned)(o / kOpSlots) & 1u, p.err);
            if (consumer_or(!ok)) {
                failed = true;
                break;
            }
            const FwdOp& op = s_op[o % kOpSlots];
            const int type = op.type;
            if (is_gemm(type)) {
                ok = gemm_consume<R>(op.g, epi_of(type), p.M, pos0, smem, r_s, pp, (s_seq << 10) | (unsigned)o, p.err,
                                     unit_stamps(o), ct);
            } else if (type == OP_EMBED) {
                embed_op(p, pos0);
            } else {
                // attention: segment partials; a grid barrier; then every CTA
                // combines a share of the partials (tiny model at contexts up to
                // 128, one segment: 6.8 us per layer with both, 4.8 without)
                ok = attn_consume<R, HD>(op.at, p.M, pos0, smem, pp, p.err, ct, unit_stamps(o));
                if (!one_segment) {
                    if (consumer_or(!ok)) {
                        failed = true;
                        break;
                    }
                    if (ct && threadIdx.x == 0) ct[2] = globaltimer();
                    barrier_arrive();
                    const CombineItem first = combine_item<HD>(op.at, p.M, pos0, combine_first());
                    if (threadIdx.x == 0) {
                        mbar_arrive(&left);
                        ok = barrier_wait();
                        if (ct) ct[7] = globaltimer();
                    }
                    if (consumer_or(!ok)) {
                        failed = true;
                        break;
                    }
                    attn_combine<HD>(op.at, p.M, pos0, first);
                }
            }
            if (ct && threadIdx.x == 0) ct[3] = globaltimer();
            // the end of op o in this CTA (its stores ordered before thread 0's
            // arrival); the last op needs no grid barrier
            if (consumer_or(!ok)) {
                failed = true;
                break;
            }
            if (ct && threadIdx.x == 0) ct[4] = globaltimer();
            if (o + 1 < p.n_ops) {
                barrier_arrive();
                if (threadIdx.x == 0) {
                    if (type != OP_ATTN || one_segment) mbar_arrive(&left);
                    ok = barrier_wait();
                    // producer and MMA warp have left op o, i.e. seen `go` for
                    // it: no completion of `go` is ever two ahead of a waiter
                    ok = ok && mbar_wait(desc + (o + 1) % kOpSlots, (unsigned)((o + 1) / kOpSlots) & 1u, p.err);
                    if (ok) mbar_arrive(&go);
                    if (ct && is_gemm(type)) ct[7] = globaltimer();
                }
                if (consumer_or(!ok)) {
                    failed = true;
                    break;
                }
            }
            if (ct && threadIdx.x == 0) ct[5] = globaltimer();
            if (p.trace && blockIdx.x == 0 && threadIdx.x == 0) p.trace[o + 1] = globaltimer();
        }
    }
    __syncwarp();
    failed = __syncthreads_or(failed);
    // After a failed wait, copies and MMAs still in flight get a bounded time
    // to land; otherwise every MMA this CTA issued has completed (the
    // consumers waited for each accumulator).  Then TMEM is freed.
    if (failed) drain_before_exit();
    tc_fence_before();
    __syncthreads();
    if (mma_warp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(kTmemCols)
                     : "memory");
    }
}

template <int R, int HD>
int launch_fwd(const FwdParams& p, int grid, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(kFwdThreads, 1, 1);
    cfg.dynamicSmemBytes = GemmSmem<R>::BYTES;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, forward_kernel<R, HD>, p);
}

template <int R, int HD>
int configure_fwd() {
    return (int)cudaFuncSetAttribute(forward_kernel<R, HD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)GemmSmem<R>::BYTES);
}

}  // namespace

int forward_configure() {
    int e = 0;
    e = e ? e : configure_fwd<1, 64>();
    e = e ? e : configure_fwd<4, 64>();
    e = e ? e : configure_fwd<8, 64>();
    e = e ? e : configure_fwd<12, 64>();
    e = e ? e : configure_fwd<16, 64>();
    e = e ? e : configure_fwd<1, 128>();
    e = e ? e : configure_fwd<4, 128>();
    e = e ? e : configure_fwd<8, 128>();
    e = e ? e : configure_fwd<12, 128>();
    e = e ? e : configure_fwd<16, 128>();
    return e;
}

template <int HD>
int launch_hd(const FwdParams& p, int grid, cudaStream_t s) {
    switch (fwd_plane_rows(p.M)) {
        case 1: return launch_fwd<1, HD>(p, grid, s);
        case 4: return launch_fwd<4, HD>(p, grid, s);
        case 8: return launch_fwd<8, HD>(p, grid, s);
        case 12: return launch_fwd<12, HD>(p, grid, s);
        default: return launch_fwd<16, HD>(p, grid, s);
    }
}

int launch_forward(const FwdParams& p, int head_dim, int grid, cudaStream_t s) {
    if (head_dim == 128) return launch_hd<128>(p, grid, s);
    if (head_dim == 64) return launch_hd<64>(p, grid, s);
    return (int)cudaErrorInvalidValue;
}

}  // namespace ssd
