// prefill.cu - prompt encoding on the tensor cores (Sec. 3.1: the prompt is
// run through the full model once, filling the KV cache, before the
// decoding rounds of Algorithms 1 / 2 start).
//
// The decode forwards are HBM-bound skinny GEMMs (M <= 16 rows); a prompt of
// hundreds of rows is compute-bound, so it gets its own kernels, layer by
// layer over a chunk of up to `rows` prompt positions:
//   embed      h[r] = E[token r]
//   norm       x = RMSNorm(h) * g as bf16 hi / lo planes (fp32 statistics)
//   QKV GEMM   tcgen05 (tc_gemm.cuh), epilogue: RoPE, q (fp32) and the fp16
//              K / V cache rows of the chunk's positions
//   attention  causal flash attention of the chunk's rows over the cache
//              [0, position] (tcgen05, fp16, online softmax), output as bf16
//              hi / lo planes
//   O GEMM     tcgen05, epilogue: h += D
//   norm, gate/up GEMM (epilogue: SwiGLU as bf16 hi / lo planes), down GEMM
//              (epilogue: h += D)
// Numerics follow the decode forwards (bf16 weights, fp32 residual stream,
// activations as bf16 hi + lo, fp16 KV, fp32 softmax), in another summation
// order.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cmath>
#include <string>
#include <vector>

#include "ssd_internal.cuh"
#include "tc_gemm.cuh"

namespace ssd {
namespace {

constexpr int kNormThreads = 256;

__global__ void __launch_bounds__(kNormThreads) pf_embed_kernel(const bf16* __restrict__ embed,
                                                                 const int* __restrict__ toks, int d,
                                                                 float* __restrict__ h) {
    pdl_launch_dependents();
    pdl_wait();
    const int r = blockIdx.x;
    const bf16* e = embed + (size_t)toks[r] * d;
    for (int i = threadIdx.x; i < d; i += kNormThreads) h[(size_t)r * d + i] = __bfloat162float(e[i]);
}

// x = h / sqrt(mean(h^2) + eps) * g, written as bf16 hi = rn(x), lo = rn(x - hi).
// One CTA per row, four features a thread and step (d is a multiple of 128); the
// row stays in registers between the sum and the scaling up to d = 8192.  Bound
// by L2 (h was just written there): 511 rows of d 4096, 5.6 us; one
// feature a thread and two passes over h took 7.5.
// (h through __ldcg: the kernel that writes it may still run when this one starts,
// so its loads must not be taken for loads of constants.  Four CTAs an SM: at 66
// registers, three, 7.2 us.)
__global__ void __launch_bounds__(kNormThreads, 4) pf_norm_kernel(const float* h, const bf16* __restrict__ g, int d,
                                                               float eps, bf16* __restrict__ x_hi,
                                                               bf16* __restrict__ x_lo) {
    constexpr int KEEP = 8;
    __shared__ float s_part[kNormThreads / 32];
    pdl_launch_dependents();
    pdl_wait();
    const size_t r0 = (size_t)blockIdx.x * d;
    const float4* hr = reinterpret_cast<const float4*>(h + r0);
    const int n4 = d >> 2;
    float4 v[KEEP];
#pragma unroll
    for (int k = 0; k < KEEP; ++k) {
        const int i = threadIdx.x + k * kNormThreads;
        v[k] = i < n4 ? __ldcg(hr + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float ss = 0.f;
#pragma unroll
    for (int k = 0; k < KEEP; ++k) ss += (v[k].x * v[k].x + v[k].y * v[k].y) + (v[k].z * v[k].z + v[k].w * v[k].w);
    for (int i = threadIdx.x + KEEP * kNormThreads; i < n4; i += kNormThreads) {
        const float4 x = __ldcg(hr + i);
        ss += (x.x * x.x + x.y * x.y) + (x.z * x.z + x.w * x.w);
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < kNormThreads / 32; ++w) tot += s_part[w];
    const float rinv = rsqrtf(tot / (float)d + eps);
    auto store = [&](int i, const float4& x) {
        const uint2 gw = __ldg(reinterpret_cast<const uint2*>(g) + i);
        const float f[4] = {x.x * rinv * bf16_lo(gw.x), x.y * rinv * bf16_hi(gw.x), x.z * rinv * bf16_lo(gw.y),
                            x.w * rinv * bf16_hi(gw.y)};
        uint32_t hi[2], lo[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const __nv_bfloat162 hv = __floats2bfloat162_rn(f[2 * p], f[2 * p + 1]);
            const float2 hf = __bfloat1622float2(hv);
            const __nv_bfloat162 lv = __floats2bfloat162_rn(f[2 * p] - hf.x, f[2 * p + 1] - hf.y);
            hi[p] = *reinterpret_cast<const uint32_t*>(&hv);
            lo[p] = *reinterpret_cast<const uint32_t*>(&lv);
        }
        *reinterpret_cast<uint2*>(x_hi + r0 + 4 * (size_t)i) = make_uint2(hi[0], hi[1]);
        *reinterpret_cast<uint2*>(x_lo + r0 + 4 * (size_t)i) = make_uint2(lo[0], lo[1]);
    };
#pragma unroll
    for (int k = 0; k < KEEP; ++k) {
        const int i = threadIdx.x + k * kNormThreads;
        if (i < n4) store(i, v[k]);
    }
    for (int i = threadIdx.x + KEEP * kNormThreads; i < n4; i += kNormThreads) store(i, __ldcg(hr + i));
}

// ---------------------------------------------------------------------------
// causal attention of the chunk's rows (flash attention on tcgen05)
// ---------------------------------------------------------------------------
// CTA = 128 query rows of one query head (the TMEM lanes), key blocks of 64
// positions from the fp16 cache by TMA.  Rows r < n_rows sit at positions pos0 +
// r and see keys [0, pos0 + r].
//   warp 4      : TMA producer, kAttStages blocks of K and V;
//   warp 5      : MMA issuer: S_j = q K_j^T (q as fp16 hi + lo in shared memory,
//                 16 MMAs 128 x 64 x 16) one block ahead of O += P_j V_j (P as
//                 fp16 hi + lo in TMEM, where it replaces S_j; V as it lies in
//                 the cache, i.e. MN-major);
//   warps 0-3   : softmax, one row per thread: S_j from TMEM, P_j back to it, the
//                 running sum; at the end O / sum as bf16 hi / lo planes.
// O is rescaled only when a row's maximum has grown by more than kAttSlack
// (in log2) over the one its weights are relative to, so the weights stay below
// 2^8 and the accumulator is rarely touched between blocks (the running softmax of
// Milakov and Gimelshein, 2018; small rescales left out as in FlashAttention-4).
// Bound by the softmax's issue slots (a thread per row, ~12 instructions a key).
// The m16n8k16 kernel this replaces took 183 us a layer at 70B widths (1023 rows)
// and 45 us at 7B widths (511 rows); this one 66 and 20 us.
constexpr int kAttQ = 128, kAttKB = 64, kAttStages = 4, kAttThreads = 192;
constexpr float kAttSlack = 8.f;
template <int HD>
struct AttSmem {
    static constexpr int BOXES = HD / 64;               // 64-dim boxes of a row
    static constexpr int QB = kAttQ * 128;              // bytes of one box of q (hi or lo)
    static constexpr int KB = kAttKB * 128;             // bytes of one box of K or V
    static constexpr int STAGE = 2 * BOXES * KB;        // K boxes, then V boxes
    static constexpr int Q = 2 * BOXES * QB;            // hi boxes, then lo boxes
    static constexpr size_t BYTES = 1024 + (size_t)Q + (size_t)kAttStages * STAGE;
};
constexpr int kAttTmem = 256;  // O: 0 .. HD, S / P of even blocks at 128, of odd ones at 192

__device__ __forceinline__ void att_tma3d(void* dst, const void* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}
// kind::f16, A = B = fp16, D = fp32, M = 128, N = n; B K-major or (V) MN-major
__device__ __forceinline__ constexpr uint32_t att_idesc(int n, bool b_mn) {
    return (1u << 4) | (b_mn ? 1u << 16 : 0u) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void att_mma_ss(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(d), "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void att_mma_ts(uint32_t d, uint32_t a, uint64_t bd, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
        ::"r"(d), "r"(a), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void att_commit(uint64_t* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(b))
                 : "memory");
}
__device__ __forceinline__ void att_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
#define SSD_R8(r, o) "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]), "=r"(r[o + 7])
#define SSD_I8(r, o) "r"(r[o]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]), "r"(r[o + 6]), "r"(r[o + 7])
// 32 columns of this thread's TMEM lane
__device__ __forceinline__ void att_ld32(uint32_t t, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : SSD_R8(r, 0), SSD_R8(r, 8), SSD_R8(r, 16), SSD_R8(r, 24)
        : "r"(t));
}
__device__ __forceinline__ void att_st32(uint32_t t, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31};"
        ::SSD_I8(r, 0), SSD_I8(r, 8), SSD_I8(r, 16), SSD_I8(r, 24), "r"(t)
        : "memory");
}
#undef SSD_R8
#undef SSD_I8
__device__ __forceinline__ void att_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void att_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_h2(float a, float b) {
    const __half2 v = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}
// hi = rn(a, b), lo = rn((a, b) - hi), packed
__device__ __forceinline__ void split_h2(float a, float b, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = pack_h2(a - f.x, b - f.y);
}

struct AttArgs {
    const float* q;     // [n_rows][H*hd] fp32, rotated
    const void* tm_k;   // K / V cache as {hd, max_seq, L * Hkv} fp16, box {64, 64, 1}, 128-byte swizzle
    const void* tm_v;
    int kv_z0;          // z of this layer's KV head 0
    int n_rows, pos0, n_heads, n_kv_heads;
    float scale2;       // log2(e) / sqrt(hd)
    bf16* out_hi;       // [n_rows][H*hd]
    bf16* out_lo;
    int* err;
};

// grid: heads x query tiles, the longest key ranges (last tiles) first
template <int HD>
__global__ void __launch_bounds__(kAttThreads, 1) pf_attn_kernel(const AttArgs a) {
    using L = AttSmem<HD>;
    constexpr int BOXES = L::BOXES;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ __align__(8) uint64_t kv_full[kAttStages], kv_empty[kAttStages];
    __shared__ __align__(8) uint64_t q_ready, s_full[2], p_ready[2], pv_done[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int head = blockIdx.x, kvh = (int)(((long long)head * a.n_kv_heads) / a.n_heads);
    const int qr0 = (int)(gridDim.y - 1 - blockIdx.y) * kAttQ;
    const int qd = a.n_heads * HD;
    const int n_kb = (a.pos0 + min(a.n_rows, qr0 + kAttQ) - 1) / kAttKB + 1;
    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < kAttStages; ++s) {
            tc::mb_init(kv_full + s, 1);
            tc::mb_init(kv_empty + s, 1);
        }
        tc::mb_init(&q_ready, 4);
        for (int b = 0; b < 2; ++b) {
            tc::mb_init(s_full + b, 1);
            tc::mb_init(p_ready + b, 4);  // one arrival per softmax warp
            tc::mb_init(pv_done + b, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kAttTmem)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_launch_dependents();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = s_tmem;
    unsigned char* kv = smem + L::Q;
    pdl_wait();  // q, K and V come from the previous kernel
    bool ok = true;

    if (warp == 4) {
        asm volatile("fence.proxy.async.global;" ::: "memory");  // K / V rows the previous kernel wrote
        for (int j = 0; j < n_kb && ok; ++j) {
            const int s = j % kAttStages;
            ok = __all_sync(0xffffffffu, tc::mb_wait(kv_empty + s, (j / kAttStages + 1) & 1u, a.err));
            if (!ok) break;
            if (elect_one()) {
                unsigned char* st = kv + s * L::STAGE;
                tc::mb_arrive_tx(kv_full + s, (unsigned)L::STAGE);
#pragma unroll
                for (int b = 0; b < BOXES; ++b) {
                    att_tma3d(st + b * L::KB, a.tm_k, b * 64, j * kAttKB, a.kv_z0 + kvh, kv_full + s);
                    att_tma3d(st + (BOXES + b) * L::KB, a.tm_v, b * 64, j * kAttKB, a.kv_z0 + kvh, kv_full + s);
                }
            }
            __syncwarp();
        }
    } else if (warp == 5) {
        const uint64_t q0 = tc::sdesc(smem_u32(smem)), kv0 = tc::sdesc(smem_u32(kv));
        auto wait = [&](uint64_t* b, int phase) {
            ok = ok && __all_sync(0xffffffffu, tc::mb_wait(b, (unsigned)phase & 1u, a.err));
            return ok;
        };
        // S_j; the block's K has landed and P_{j-2}, which held these columns, is used up
        auto scores = [&](int j) {
            if (!wait(kv_full + j % kAttStages, j / kAttStages)) return;
            if (j >= 2 && !wait(pv_done + (j & 1), (j - 2) >> 1)) return;
            tc::fence_after();
            if (elect_one()) {
                const uint64_t k0 = kv0 + (uint64_t)((j % kAttStages) * (L::STAGE >> 4));
                const uint32_t d = tmem + 128u + 64u * (uint32_t)(j & 1);
#pragma unroll
                for (int h = 0; h < 2; ++h)  // hi, lo
#pragma unroll
                    for (int b = 0; b < BOXES; ++b)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            att_mma_ss(d, q0 + (uint64_t)(((h * BOXES + b) * L::QB + ks * 32) >> 4),
                                       k0 + (uint64_t)((b * L::KB + ks * 32) >> 4), att_idesc(64, false),
                                       (h | b | ks) ? 1u : 0u);
                att_commit(s_full + (j & 1));
            }
            __syncwarp();
        };
        wait(&q_ready, 0);
        if (ok) scores(0);
        for (int j = 0; j < n_kb && ok; ++j) {
            if (j + 1 < n_kb) scores(j + 1);
            if (!ok || !wait(p_ready + (j & 1), j >> 1)) break;
            tc::fence_after();
            if (elect_one()) {
                // V: 64 dims (MN) x 16 keys (K) per MMA; 8 keys are 1024 bytes apart
                const uint64_t v0 = kv0 + (uint64_t)(((j % kAttStages) * L::STAGE + BOXES * L::KB) >> 4);
                const uint64_t mn = (uint64_t)((1024 >> 4) - 1) << 16;  // leading byte offset 1024 too
                const uint32_t p = tmem + 128u + 64u * (uint32_t)(j & 1);
#pragma unroll
                for (int b = 0; b < BOXES; ++b)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            att_mma_ts(tmem + 64u * b, p + 32u * h + 8u * ks, v0 + mn + (uint64_t)((b * L::KB + ks * 2048) >> 4),
                                       att_idesc(64, true), (j | ks | h) ? 1u : 0u);
                att_commit(kv_empty + j % kAttStages);
                att_commit(pv_done + (j & 1));
            }
            __syncwarp();
        }
    } else {
        // q of the tile as fp16 hi + lo, scaled to log2 units: a warp takes 32
        // rows, a row at a time (K-major, 128-byte swizzle: row r of a 64-dim
        // box at r * 128, 16-byte chunk c at (c ^ (r & 7)) * 16)
        constexpr int LPR = HD / 4, RPI = 32 / LPR;  // lanes per row, rows per step
        for (int i0 = 0; i0 < 32; i0 += 8 * RPI) {
            float4 x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = warp * 32 + i0 + i * RPI + lane / LPR, e = (lane % LPR) * 4;
                x[i] = qr0 + r < a.n_rows
                           ? __ldcg(reinterpret_cast<const float4*>(a.q + (size_t)(qr0 + r) * qd + head * HD + e))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = warp * 32 + i0 + i * RPI + lane / LPR, e = (lane % LPR) * 4;
                uint2 hi, lo;
                split_h2(x[i].x * a.scale2, x[i].y * a.scale2, hi.x, lo.x);
                split_h2(x[i].z * a.scale2, x[i].w * a.scale2, hi.y, lo.y);
                unsigned char* at = smem + (e >> 6) * L::QB + r * 128 + ((((e & 63) >> 3) ^ (r & 7)) << 4) + (e & 7) * 2;
                *reinterpret_cast<uint2*>(at) = hi;
                *reinterpret_cast<uint2*>(at + BOXES * L::QB) = lo;
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) att_arrive(&q_ready);

        const int row = qr0 + warp * 32 + lane, pos = a.pos0 + row;  // this thread's query row
        const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16);
        float mx = 0.f, l = 0.f;  // reference maximum of the weights, their sum
        for (int j = 0; j < n_kb && ok; ++j) {
            const uint32_t ts = tl + 128u + 64u * (uint32_t)(j & 1);
            ok = __all_sync(0xffffffffu, tc::mb_wait(s_full + (j & 1), (unsigned)(j >> 1) & 1u, a.err));
            if (!ok) break;
            tc::fence_after();
            uint32_t u0[32], u1[32];
            att_ld32(ts, u0);
            att_ld32(ts + 32, u1);
            att_wait_ld();
            const int last = pos - j * kAttKB;  // the row sees keys 0 .. last of the block
            if ((j + 1) * kAttKB - 1 > a.pos0 + qr0) {  // (uniform) some row of the tile does not see all
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (i > last) u0[i] = __float_as_uint(-INFINITY);
                    if (i + 32 > last) u1[i] = __float_as_uint(-INFINITY);
                }
            }
            float bm4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};  // (short dependency chains)
#pragma unroll
            for (int i = 0; i < 32; ++i)
                bm4[i & 3] = fmaxf(bm4[i & 3], fmaxf(__uint_as_float(u0[i]), __uint_as_float(u1[i])));
            const float bm = fmaxf(fmaxf(bm4[0], bm4[1]), fmaxf(bm4[2], bm4[3]));
            if (j == 0) {
                mx = bm;
            } else if (__any_sync(0xffffffffu, bm > mx + kAttSlack)) {
                // O and the sum move to the new maximum (all rows of the warp)
                ok = __all_sync(0xffffffffu, tc::mb_wait(pv_done + ((j - 1) & 1), (unsigned)((j - 1) >> 1) & 1u, a.err));
                if (!ok) break;
                tc::fence_after();
                const float nm = fmaxf(mx, bm), f = nm == -INFINITY ? 1.f : exp2f(mx - nm);
                for (int c = 0; c < HD; c += 32) {
                    uint32_t o[32];
                    att_ld32(tl + c, o);
                    att_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                    att_st32(tl + c, o);
                }
                l *= f;
                mx = nm;
            }
            // (a row whose scores so far are all -inf, against infinite keys: weights 0)
            const float ref = mx == -INFINITY ? 0.f : mx;
            uint32_t hi[32], lo[32];
            float l4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float p0 = exp2f(__uint_as_float(u0[2 * i]) - ref), p1 = exp2f(__uint_as_float(u0[2 * i + 1]) - ref);
                const float p2 = exp2f(__uint_as_float(u1[2 * i]) - ref), p3 = exp2f(__uint_as_float(u1[2 * i + 1]) - ref);
                l4[i & 3] += (p0 + p1) + (p2 + p3);
                split_h2(p0, p1, hi[i], lo[i]);
                split_h2(p2, p3, hi[i + 16], lo[i + 16]);
            }
            l += (l4[0] + l4[1]) + (l4[2] + l4[3]);
            att_st32(ts, hi);
            att_st32(ts + 32, lo);
            att_wait_st();
            tc::fence_before();
            __syncwarp();
            if (lane == 0) att_arrive(p_ready + (j & 1));
        }
        if (ok) ok = __all_sync(0xffffffffu, tc::mb_wait(pv_done + ((n_kb - 1) & 1), (unsigned)((n_kb - 1) >> 1) & 1u, a.err));
        if (ok) {
            tc::fence_after();
            const float inv = l > 0.f ? 1.f / l : 0.f;
            for (int c = 0; c < HD; c += 32) {
                uint32_t o[32];
                att_ld32(tl + c, o);
                att_wait_ld();
                if (row < a.n_rows) {
                    const size_t at = (size_t)row * qd + head * HD + c;
#pragma unroll
                    for (int i = 0; i < 32; i += 8) {
                        __align__(16) bf16 h8[8], l8[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const float v = __uint_as_float(o[i + k]) * inv;
                            h8[k] = __float2bfloat16_rn(v);
                            l8[k] = __float2bfloat16_rn(v - __bfloat162float(h8[k]));
                        }
                        *reinterpret_cast<uint4*>(a.out_hi + at + i) = *reinterpret_cast<const uint4*>(h8);
                        *reinterpret_cast<uint4*>(a.out_lo + at + i) = *reinterpret_cast<const uint4*>(l8);
                    }
                }
            }
        }
    }
    if (!ok) s_fail = 1;
    tc::fence_before();
    __syncwarp();
    __syncthreads();
    if (s_fail && threadIdx.x == 0) {  // let copies and MMAs in flight finish
        const unsigned long long t0 = tc::gtime();
        while (tc::gtime() - t0 < 2000000ull) __nanosleep(1000);
    }
    __syncthreads();
    if (warp == 4) {
        tc::fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kAttTmem) : "memory");
    }
}

template <int HD>
int launch_attn(const AttArgs& a, cudaStream_t s) {
    return tc::launch_pdl(pf_attn_kernel<HD>, dim3(a.n_heads, (a.n_rows + kAttQ - 1) / kAttQ), kAttThreads,
                          AttSmem<HD>::BYTES, s, a);
}

}  // namespace

int prefill_configure() {
    int e = (int)cudaFuncSetAttribute(pf_attn_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)AttSmem<128>::BYTES);
    if (!e)
        e = (int)cudaFuncSetAttribute(pf_attn_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)AttSmem<64>::BYTES);
    if (!e) e = tc::tc_configure<tc::TC_QKV>();
    if (!e) e = tc::tc_configure<tc::TC_QKV, true>();
    if (!e) e = tc::tc_configure<tc::TC_RESID>();
    if (!e) e = tc::tc_configure<tc::TC_SWIGLU>();
    return e;
}

size_t prefill_ws_floats(int pairs) { return (size_t)pairs * 2 * tc::kMaxTok * 128; }
size_t prefill_flag_words(int pairs) { return (size_t)pairs * 2 * tc::kEpiWarps; }

// One chunk of prompt rows at positions pos0 .. pos0 + n - 1 through every
// layer (launches only).  toks: device token ids of the chunk.  Every kernel is
// a programmatic dependent launch: its set-up (and a GEMM's first weights)
// overlap the previous kernel's end, and it waits for that kernel's results
// before it reads or writes anything else.
int prefill_chunk(PrefillPlan& P, const int* toks, int n, int pos0, cudaStream_t s) {
    const int d = P.d, qd = P.n_heads * P.head_dim, kvd = P.n_kv_heads * P.head_dim;
    // the arguments every GEMM shares: n_out outputs in n_ft tiles of 256 weight rows, K inputs
    auto gemm = [&](const void* const* tm_x, int n_out, int n_ft, int K) {
        tc::TcArgs a{};
        a.rows = n;
        a.N = n_out;
        a.n_kb = (K + tc::kBK - 1) / tc::kBK;
        tc::tc_plan(a, n_ft, P.pairs, K);
        a.tm_x = tm_x[a.nt / 32 - 1];
        a.ws = P.ws;
        a.flags = P.flags;
        if (++P.epoch == 0) ++P.epoch;
        a.epoch = P.epoch;
        a.err = P.err;
        return a;
    };
    int e = tc::launch_pdl(pf_embed_kernel, dim3(n), kNormThreads, 0, s, P.embed, toks, d, P.h);
    for (int l = 0; l < P.n_layers && !e; ++l) {
        const PrefillLayer& L = P.layers[l];
        e = tc::launch_pdl(pf_norm_kernel, dim3(n), kNormThreads, 0, s, (const float*)P.h, L.attn_norm, d, P.eps, P.x_hi, P.x_lo);
        if (e) break;
        tc::TcArgs a = gemm(P.tm_x, qd + 2 * kvd, (qd + 2 * kvd + tc::kFeat - 1) / tc::kFeat, d);
        a.tm_w[0] = L.tm_w[0];
        a.tm_w[1] = L.tm_w[1];
        a.tm_w[2] = L.tm_w[2];
        a.n_heads = P.n_heads;
        a.n_kv_heads = P.n_kv_heads;
        a.head_dim = P.head_dim;
        a.max_seq = P.max_seq;
        a.pos0 = pos0;
        a.q = P.q;
        a.k_cache = L.k_cache;
        a.v_cache = L.v_cache;
        a.rope = P.rope;
        e = L.qkv_rows16 ? tc::tc_launch<tc::TC_QKV, true>(a, s) : tc::tc_launch<tc::TC_QKV>(a, s);
        if (e) break;
        AttArgs t{};
        t.q = P.q;
        t.tm_k = P.tm_k;
        t.tm_v = P.tm_v;
        t.kv_z0 = l * P.n_kv_heads;
        t.n_rows = n;
        t.pos0 = pos0;
        t.n_heads = P.n_heads;
        t.n_kv_heads = P.n_kv_heads;
        t.scale2 = (float)(1.4426950408889634 / std::sqrt((double)P.head_dim));
        t.out_hi = P.at_hi;
        t.out_lo = P.at_lo;
        t.err = P.err;
        e = P.head_dim == 128 ? launch_attn<128>(t, s) : launch_attn<64>(t, s);
        if (e) break;
        tc::TcArgs o = gemm(P.tm_at, d, (d + tc::kFeat - 1) / tc::kFeat, qd);
        o.tm_w[0] = L.tm_w[3];
        o.out = P.h;
        e = tc::tc_launch<tc::TC_RESID>(o, s);
        if (e) break;
        e = tc::launch_pdl(pf_norm_kernel, dim3(n), kNormThreads, 0, s, (const float*)P.h, L.mlp_norm, d, P.eps, P.x_hi, P.x_lo);
        if (e) break;
        tc::TcArgs gu = gemm(P.tm_x, P.ffn, (P.ffn + 127) / 128, d);  // 128 features: gate and up rows
        gu.tm_w[0] = L.tm_w[4];
        gu.tm_w[1] = L.tm_w[5];
        gu.swapped = L.swapped;
        gu.act_hi = P.ac_hi;
        gu.act_lo = P.ac_lo;
        e = tc::tc_launch<tc::TC_SWIGLU>(gu, s);
        if (e) break;
        tc::TcArgs dn = gemm(P.tm_ac, d, (d + tc::kFeat - 1) / tc::kFeat, P.ffn);
        dn.tm_w[0] = L.tm_w[6];
        dn.out = P.h;
        e = tc::tc_launch<tc::TC_RESID>(dn, s);
    }
    return e;
}

}  // namespace ssd
