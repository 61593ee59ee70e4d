// gemm.cu - the stand-alone skinny projection GEMM of ssd_linear_noalloc:
// Y[M x N] = X[M x K] * W^T with W bf16 [N][K], fp32 X and Y, M <= 16.
//
// Bound by HBM: every weight is read once.  The weights are the large operand,
// so the kernel is "swap-AB": 16 weight rows form the M side of an m16n8k16
// tensor-core MMA and the <= 16 activation rows form its N side.  (mma.sync: a
// block of 64 k needs 8 to 16 of them per 2 KB of weights, a few percent of the
// tensor pipe, and its operands come from registers.)
//
// CTA = 8 warps x 16 weight rows = 128 rows, over a range of K.  A warp loads
// its weights from global memory into MMA fragments directly, 16 bytes a
// thread, two or four 64-wide k blocks ahead of the MMAs: thread (g, t) reads 8
// consecutive bf16 of rows g and g + 8, which the A and B fragments both interpret
// as the same logical k slots, so the product is unchanged, and a quad reads whole
// 128-byte lines.  The activations pass through shared memory as bf16 pairs, up
// to 1024 k at a time.
//
// Few row tiles: K is split over a cluster of 2, 4 or 8 CTAs, which add their
// sums through distributed shared memory in rank order: no scratch in global
// memory, no counters, one launch.  The split depends on (N, K) and the SM
// count only and MMA columns are independent, so the result for activation row
// m depends on row m alone.
//
// Precision: the fp32 activation rows are split into bf16 hi = rn(x) and
// lo = rn(x - hi) and both are multiplied (the MMA's N side holds the hi rows
// then the lo rows), so the product sees ~16 mantissa bits of x; the weights
// are exact bf16; accumulation is fp32.
#include <mutex>
#include <string>

#include "ssd.h"
#include "ssd_internal.cuh"

namespace ssd {
namespace {

constexpr int kLinThreads = 256;
constexpr int kLinRows = 128;    // weight rows per CTA
constexpr int kLinChunk = 1024;  // k staged in shared memory at a time
constexpr int kLinFold = 4;      // 64-wide k blocks per fp32 fold
constexpr int kPrefetchK = 256;  // k of each row brought into L2 ahead
constexpr int kRedPitch = kLinRows + 4;

struct LinearArgs {
    const bf16* w;
    const float* x;
    float* y;
    int N, K, M;
    int kc;  // k per CTA of the cluster, a multiple of 64

#ifdef SSD_CHECKED  // what the kernel's accesses have to satisfy
    __host__ __device__ bool weights_in(const bf16* p, size_t elems) const {
        return ((uintptr_t)p & 15u) == 0 && p >= w && p + elems <= w + (size_t)N * K;
    }
    __host__ __device__ bool inputs_in(const float* p, size_t elems) const {
        return ((uintptr_t)p & 15u) == 0 && p >= x && p + elems <= x + (size_t)M * K;
    }
    __host__ __device__ bool output_in(const float* p) const { return p >= y && p < y + (size_t)M * N; }
#endif
};
#ifdef SSD_CHECKED
__device__ int g_linear_err;  // code of the first failed check
#endif

__device__ __forceinline__ float ld_cluster(uint32_t saddr, unsigned rank) {
    uint32_t r;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(r) : "memory");
    return v;
}
// 16 weight bytes, read once: not kept in L1.  Not the non-coherent path (.nc): the
// weights may come from the kernel before, which can still run when this one starts
// (calls back to back over 12 matrices, 16 x 4096 x 4096 12.0 us, 11.5 with .nc; 4 x 4096
// x 32000 50.0 / 49.9, 8 x 8192 x 8192 26.5 / 26.5; .cg 12.2 / 52.9 / 28.8, .cs 12.0 / 49.7 /
// 26.6).
// volatile, like the MMAs, so that the loads stay as far ahead of them as they are
// written
__device__ __forceinline__ uint4 ld_weights(const LinearArgs& a, const bf16* p) {
    uint4 v = make_uint4(0, 0, 0, 0);
    SSD_GUARD(&g_linear_err, a.weights_in(p, 8), 101)
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ void lin_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// P = 8 or 16 activation rows; the MMA's N side holds P rows of x_hi, then P of
// x_lo.  4 CTAs an SM with 2 blocks a warp ahead where registers allow it (P = 8;
// N 22016, K 4096, cold: 45 us against 61 with 2 CTAs and 4 blocks), else 2 CTAs with
// 4 blocks (P = 16; N = K = 4096, cold, before the L2 prefetch: 18.0 us against 20.1).
// Where the grid fills every SM so, 128 KB of weights are in flight per SM; with few
// row tiles less: 256 CTAs for N = 4096 leave 48 of 152 SMs with one.
template <int P>
struct LinShape {
    static constexpr int CTAS = P == 8 ? 4 : 2, DEPTH = P == 8 ? 2 : 4;
};
template <int P>
__global__ void __launch_bounds__(kLinThreads, LinShape<P>::CTAS) linear_kernel(const LinearArgs a) {
    constexpr int NT = P / 4;  // n8 tiles: hi, then lo
    constexpr int D = LinShape<P>::DEPTH;
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_launch_dependents();
    unsigned rank, n_ranks;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n_ranks));
    const int tile = blockIdx.x / n_ranks;
    const int k0 = (int)rank * a.kc, k1 = min(a.K, k0 + a.kc);
    const int nb = k1 > k0 ? (k1 - k0 + 63) / 64 : 0;
    const int pitch = min(a.kc, kLinChunk) * 2 + 64;  // bytes; pitch % 128 == 64: conflict-free LDS.128
    float* red = reinterpret_cast<float*>(smem);       // [P][kRedPitch]
    unsigned char* xs = smem + P * kRedPitch * 4;      // [2P][pitch] hi rows, then lo rows
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    // rows past N read row N - 1 again; their sums are not stored
    const int r0 = tile * kLinRows + warp * 16 + g;
    const bf16* w0 = a.w + (size_t)min(r0, a.N - 1) * a.K + t * 8;
    const bf16* w1 = a.w + (size_t)min(r0 + 8, a.N - 1) * a.K + t * 8;
    uint4 wr[D][4];
    // K is a multiple of 16: a thread's 8 values are all inside or all outside
    auto load = [&](uint4 (&d)[4], int b) {
        const int k = k0 + b * 64;
        const uint4 z = make_uint4(0, 0, 0, 0);
        const bool in0 = k + t * 8 < k1, in1 = k + 32 + t * 8 < k1;
        d[0] = in0 ? ld_weights(a, w0 + k) : z;
        d[1] = in0 ? ld_weights(a, w1 + k) : z;
        d[2] = in1 ? ld_weights(a, w0 + k + 32) : z;
        d[3] = in1 ? ld_weights(a, w1 + k + 32) : z;
    };
    // The weights on their way into L2 while the previous kernel ends (a prefetch
    // returns nothing, so it may run ahead of a kernel that writes them).  Calls
    // back to back, 0 / 256 / 512 k ahead (loads through .nc): 16 x 4096 x 4096 12.3 / 11.2 / 10.7 us,
    // 4 x 4096 x 32000 51.3 / 48.5 / 49.8, 8 x 8192 x 8192 28.2 / 25.8 / 27.0.
    if (threadIdx.x < kLinRows && k1 > k0) {
        const bf16* row = a.w + (size_t)min(tile * kLinRows + (int)threadIdx.x, a.N - 1) * a.K + k0;
        const unsigned bytes = (unsigned)min(k1 - k0, kPrefetchK) * 2u;  // (K is a multiple of 16: 32-byte steps)
        SSD_GUARD(&g_linear_err, a.weights_in(row, bytes / 2), 102)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row), "r"(bytes) : "memory");
    }
    pdl_wait();  // weights and activations may come from the previous kernel
#pragma unroll
    for (int d = 0; d < D; ++d) load(wr[d], d);

    // the MMAs' running sums, folded into fp32 sums of hi + lo every
    // kLinFold k blocks (256 k): the tensor cores' own accumulation rounds less
    // well over long chains (K 4096 in chains of 2048 k: error 3.2e-6, of 256 k 2.5e-6)
    float acc[NT][4], sum[NT / 2][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
#pragma unroll
    for (int nt = 0; nt < NT / 2; ++nt) sum[nt][0] = sum[nt][1] = sum[nt][2] = sum[nt][3] = 0.f;
    for (int c0 = 0; c0 < nb; c0 += kLinChunk / 64) {
        const int cb = min(kLinChunk / 64, nb - c0);  // k blocks of this chunk
        if (c0) __syncthreads();
        for (int i = threadIdx.x; i < P * cb * 8; i += kLinThreads) {
            const int n = i / (cb * 8), cc = i - n * (cb * 8), k = k0 + c0 * 64 + cc * 8;
            uint4 hi = make_uint4(0, 0, 0, 0), lo = make_uint4(0, 0, 0, 0);
            if (n < a.M && k < k1) {
                const float4* src = reinterpret_cast<const float4*>(a.x + (size_t)n * a.K + k);
                SSD_GUARD(&g_linear_err, a.inputs_in(reinterpret_cast<const float*>(src), 8), 103)
                split8(__ldcg(src), __ldcg(src + 1), hi, lo);
            }
            SSD_GUARD(&g_linear_err, n < P && cc * 16 + 16 <= pitch, 104) {
                *reinterpret_cast<uint4*>(xs + n * pitch + cc * 16) = hi;
                *reinterpret_cast<uint4*>(xs + (P + n) * pitch + cc * 16) = lo;
            }
        }
        __syncthreads();
        for (int b = 0; b < cb; b += kLinFold) {
#pragma unroll
            for (int d = 0; d < kLinFold; ++d) {
                if (b + d < cb) {
                    const unsigned char* xb = xs + g * pitch + (b + d) * 128 + t * 16;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint4 wa = wr[d % D][2 * h], wb = wr[d % D][2 * h + 1];
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            const uint4 xv = *reinterpret_cast<const uint4*>(xb + nt * 8 * pitch + h * 64);
                            mma_bf16_16816(acc[nt], wa.x, wb.x, wa.y, wb.y, xv.x, xv.y);
                            mma_bf16_16816(acc[nt], wa.z, wb.z, wa.w, wb.w, xv.z, xv.w);
                        }
                    }
                    load(wr[d % D], c0 + b + d + D);
                }
            }
#pragma unroll
            for (int nt = 0; nt < NT / 2; ++nt)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    sum[nt][x] += acc[nt][x] + acc[nt + NT / 2][x];
                    acc[nt][x] = acc[nt + NT / 2][x] = 0.f;
                }
        }
    }
    // this CTA's sums, then the ranks' sums in order
#pragma unroll
    for (int nt = 0; nt < NT / 2; ++nt)
#pragma unroll
        for (int x = 0; x < 4; ++x)
            red[(nt * 8 + 2 * t + (x & 1)) * kRedPitch + warp * 16 + g + 8 * (x >> 1)] = sum[nt][x];
    if (n_ranks > 1) lin_cluster_sync();
    else __syncthreads();
    const int rows = kLinRows / (int)n_ranks, row0 = (int)rank * rows;  // (a power of two of ranks)
    for (int i = threadIdx.x; i < a.M * rows; i += kLinThreads) {
        const int m = i / rows, r = row0 + i - m * rows, n = tile * kLinRows + r;
        if (n >= a.N) continue;
        float s;
        if (n_ranks == 1) {
            s = red[m * kRedPitch + r];
        } else {
            float v[8];
#pragma unroll
            for (unsigned q = 0; q < 8; ++q) v[q] = q < n_ranks ? ld_cluster(smem_u32(red + m * kRedPitch + r), q) : 0.f;
            s = v[0];
#pragma unroll
            for (unsigned q = 1; q < 8; ++q)
                if (q < n_ranks) s += v[q];
        }
        SSD_GUARD(&g_linear_err, a.output_in(a.y + (size_t)m * a.N + n), 105)
        a.y[(size_t)m * a.N + n] = s;
    }
    if (n_ranks > 1) lin_cluster_sync();  // the other ranks have read this CTA's sums
}

size_t linear_smem_bytes(int kc, int P) {
    const int k = kc < kLinChunk ? kc : kLinChunk;
    return (size_t)P * kRedPitch * 4 + (size_t)2 * P * (k * 2 + 64);
}

template <int P>
int launch_linear(const LinearArgs& a, int ranks, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((a.N + kLinRows - 1) / kLinRows * ranks), 1, 1);
    cfg.blockDim = dim3(kLinThreads, 1, 1);
    cfg.dynamicSmemBytes = linear_smem_bytes(a.kc, P);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)ranks;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return (int)cudaLaunchKernelEx(&cfg, linear_kernel<P>, a);
}

// Per device, once: kernel attributes and the SM count.
struct LinearDevice {
    bool ready = false;
    int n_sms = 0;
};
constexpr int kLinMaxDevices = 64;
LinearDevice g_lin_dev[kLinMaxDevices];
std::mutex g_lin_mu;

int linear_setup(int dev, int* n_sms) {
    std::lock_guard<std::mutex> lock(g_lin_mu);
    LinearDevice& d = g_lin_dev[dev];
    if (!d.ready) {
        cudaError_t e = cudaFuncSetAttribute(linear_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)linear_smem_bytes(kLinChunk, 8));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(linear_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)linear_smem_bytes(kLinChunk, 16));
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&d.n_sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess)
            return set_last_error(SSD_ERR_CUDA, (std::string("ssd_linear_noalloc set-up: ") +
                                                 cudaGetErrorString(e)).c_str());
        d.ready = true;
    }
    *n_sms = d.n_sms;
    return SSD_OK;
}

}  // namespace
}  // namespace ssd

// ---------------------------------------------------------------------------
// ssd_linear_noalloc: the projection GEMM alone, for callers that cannot
// allocate device memory at the point where they need a projection: a serving
// process that reserves every byte of HBM at start-up and treats any later
// allocation as a failure, a plug-in whose host framework owns all device
// allocations, or a latency-critical loop that must not call cudaMalloc /
// cudaFree because those calls can synchronise the whole device.
// ---------------------------------------------------------------------------
extern "C" int ssd_linear_noalloc(const void* w, const float* x, float* y, int N, int K, int M,
                                  void* cuda_stream) {
    using namespace ssd;
    if (!w || !x || !y) return set_last_error(SSD_ERR_INVALID_ARG, "ssd_linear_noalloc: NULL pointer");
    if (((uintptr_t)w & 15u) || ((uintptr_t)x & 15u))
        return set_last_error(SSD_ERR_INVALID_ARG, "ssd_linear_noalloc: w and x must be 16-byte aligned");
    if (M < 1 || M > kMaxRows || N < 1 || K < 16 || K % 16)
        return set_last_error(SSD_ERR_INVALID_ARG,
                              "ssd_linear_noalloc: need 1 <= M <= 16, N >= 1, K a positive multiple of 16");
    // the sizes the call takes (ssd.h)
    const size_t tiles64 = ((size_t)N + 63) / 64, need = K > 512 ? (size_t)((K + 511) / 512) * M * 64 * tiles64 : 0;
    if (tiles64 > 4096 || need > (size_t(1) << 20))
        return set_last_error(SSD_ERR_CAPACITY,
                              ("ssd_linear_noalloc: sizes beyond the call's limits (kept from the time it had scratch "
                               "memory): " + std::to_string(tiles64) + " of 4096 tiles of 64 rows, " +
                               std::to_string(need) + " of 1048576 partial sums")
                                  .c_str());
    int dev = 0, n_sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kLinMaxDevices)
        return set_last_error(SSD_ERR_CUDA, "ssd_linear_noalloc: no usable current device");
    const int rc = linear_setup(dev, &n_sms);
    if (rc) return rc;
    // K split over a cluster until there are two CTAs per SM, at least 128 k each
    const int tiles = (N + kLinRows - 1) / kLinRows;
    int ranks = 1;
    while (ranks < 8 && tiles * ranks < 2 * n_sms && K / (2 * ranks) >= 128) ranks *= 2;
    LinearArgs a{};
    a.w = (const bf16*)w;
    a.x = x;
    a.y = y;
    a.N = N;
    a.K = K;
    a.M = M;
    a.kc = ((K + ranks - 1) / ranks + 63) / 64 * 64;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    e = (cudaError_t)(M > 8 ? launch_linear<16>(a, ranks, s) : launch_linear<8>(a, ranks, s));
    if (e != cudaSuccess)
        return set_last_error(SSD_ERR_CUDA, (std::string("ssd_linear_noalloc: ") + cudaGetErrorString(e)).c_str());
#ifdef SSD_CHECKED
    // read the flag back (which makes the call synchronous), clear it for the next call, report it
    int derr = 0, *flag = nullptr;
    e = cudaGetSymbolAddress((void**)&flag, g_linear_err);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&derr, flag, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && derr) e = cudaMemsetAsync(flag, 0, sizeof(int), s);
    if (e != cudaSuccess)
        return set_last_error(SSD_ERR_CUDA, (std::string("ssd_linear_noalloc: ") + cudaGetErrorString(e)).c_str());
    if (derr)
        return set_last_error(SSD_ERR_CUDA,
                              ("ssd_linear_noalloc: device check failed with code " + std::to_string(derr)).c_str());
#endif
    return SSD_OK;
}
