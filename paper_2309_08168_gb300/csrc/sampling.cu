// sampling.cu - the token choice and acceptance kernels that follow a
// forward in self-speculative decoding:
//   greedy draft      x_{j+1} = argmax p(x | z*, ...)              (Algorithm 2)
//   greedy accept     longest prefix d_j == argmax p_{j-1}; the first
//                     mismatch is corrected, or a bonus token added (Alg. 2)
//   sampling draft    d_j ~ q_j = nucleus(softmax(logits / T))        (Alg. 4)
//   sampling accept   accept d_j iff r < min(1, p_{j-1}(d_j) / q_j(d_j)); the
//                     first rejected one is resampled from
//                     norm(max(0, p_{j-1} - q_j)); bonus ~ p_K      (Alg. 4)
// followed by the KV rollback len <- len + 1 + n (a length pointer: later
// writes overwrite the rejected positions).
//
// Random numbers: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), key =
// 64-bit seed, counter = (position, purpose, 0, 0), purpose 0 = draft sample,
// 1 = acceptance uniform, 2 = resample / bonus; u = ((w0 >> 8) + 0.5) * 2^-24,
// a uniform on (0, 1) that is exact in fp32.
//
// Every reduction has a fixed shape (thread-contiguous segments, warp
// shuffle trees, then one warp over the warp totals), so all results are
// run-to-run deterministic.
#include "ssd_internal.cuh"

namespace ssd {
namespace {

constexpr int kRowThreads = 1024;
constexpr int kSegMax = 32;  // row elements per thread (vocab <= 32768)

// Rows in shared memory: element i at row_at(i).  Thread t owns the contiguous
// segment [t * seg, t * seg + seg), so without the padding the lanes of a warp
// would meet in one bank (seg = 32: every access 32 cycles).
__device__ __forceinline__ int row_at(int i) { return i + (i >> 5); }
size_t row_bytes(int V) { return ((size_t)V + V / 32 + 1) * sizeof(float); }

// ---------------------------------------------------------------------------
// Philox4x32-10
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t philox_w0(unsigned long long seed, uint32_t pos, uint32_t purpose) {
    uint32_t c0 = pos, c1 = purpose, c2 = 0u, c3 = 0u;
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
        const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c0;
}

__device__ __forceinline__ float uniform01(unsigned long long seed, int pos, int purpose) {
    return ((float)(philox_w0(seed, (uint32_t)pos, (uint32_t)purpose) >> 8) + 0.5f) *
           (1.0f / 16777216.0f);
}

// ---------------------------------------------------------------------------
// block reductions (blockDim = 1024, fixed order)
// ---------------------------------------------------------------------------
__device__ float block_sum(float v, float* red) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    v = warp_sum(v);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        float r = warp_sum(red[lane]);
        if (lane == 0) red[32] = r;
    }
    __syncthreads();
    float r = red[32];
    __syncthreads();
    return r;
}

__device__ float block_max(float v, float* red) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    v = warp_max(v);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        float r = warp_max(red[lane]);
        if (lane == 0) red[32] = r;
    }
    __syncthreads();
    float r = red[32];
    __syncthreads();
    return r;
}

// argmax with the lowest index among equal maxima (NaN never wins)
__device__ __forceinline__ void better(float& v, int& i, float v2, int i2) {
    if (v2 > v || (v2 == v && i2 < i)) { v = v2; i = i2; }
}

__device__ int block_argmax(const float* x, int V, float* redf, int* redi) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float bv = -INFINITY;
    int bi = 0x7fffffff;
    for (int i = threadIdx.x; i < V; i += kRowThreads) better(bv, bi, x[i], i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float v2 = __shfl_xor_sync(0xffffffffu, bv, o);
        int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
        better(bv, bi, v2, i2);
    }
    if (lane == 0) { redf[warp] = bv; redi[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
        bv = redf[lane];
        bi = redi[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            float v2 = __shfl_xor_sync(0xffffffffu, bv, o);
            int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
            better(bv, bi, v2, i2);
        }
        if (lane == 0) redi[32] = bi;
    }
    __syncthreads();
    int r = redi[32];
    __syncthreads();
    return (r < 0 || r >= V) ? 0 : r;
}

// ---------------------------------------------------------------------------
// sampling distribution of one row: softmax(logits / T) restricted to the
// nucleus {x : pi(x) >= tau*}, tau* = the largest value whose upper set holds
// >= top_p of the mass, renormalised.  s: shared row; thread t owns the
// contiguous segment [t*seg, t*seg + seg) and keeps exp(x - max) in registers;
// the search runs on these values (tau* and the mass scaled by their sum z), so
// that a kept value is divided once.  tau* is found exactly by bisection over the
// fp32 bit patterns (non-negative floats order like their bits), from below
// (1 - top_p) z / 2V, where at most half of 1 - top_p is cut off.  The row is a
// CTA's, so a pass over it costs its instructions (two per element): one
// threshold at a time, until the bracket is 2^20 patterns wide (1/8 octave, 7
// passes at top_p 0.95).  The values inside it, 2-3 % of a flat row, are then
// listed in the row's shared memory, and the other 20 bits take 10 passes of
// three thresholds over the list, by one warp if it is short (with 32 warps
// such a pass is 960 shuffles, 0.8 us; with one 0.2 us).
// (Vocabulary 32000, top-p 0.95, the whole sampling draft kernel: 302 us with 15
// thresholds a pass and the row in shared memory without padding, 48.7 with 30
// one-threshold passes over registers, 44.9 with the list, all warps and two
// divisions, 33.1 now; a row of the acceptance kernel 58.8, 53.7, 41.1.)
// ---------------------------------------------------------------------------
constexpr uint32_t kBracket = 1u << 20;
constexpr int kShortList = 1024;

__device__ void nucleus_row(const float* logits, int V, float inv_t, float top_p, float* s,
                            float* red) {
    const int seg = (V + kRowThreads - 1) / kRowThreads;
    const int beg = min(V, threadIdx.x * seg), n = min(V, beg + seg) - beg;
    for (int i = threadIdx.x; i < V; i += kRowThreads) s[row_at(i)] = logits[i] * inv_t;
    __syncthreads();
    float r[kSegMax];
    float mx = -INFINITY;
#pragma unroll
    for (int k = 0; k < kSegMax; ++k) {
        r[k] = k < n ? s[row_at(beg + k)] : -INFINITY;
        mx = fmaxf(mx, r[k]);
    }
    mx = block_max(mx, red);
    float z = 0.f;
#pragma unroll
    for (int k = 0; k < kSegMax; ++k) {
        r[k] = k < n ? expf(r[k] - mx) : 0.f;
        z += r[k];
    }
    z = block_sum(z, red);
    if (top_p < 1.f) {
        __shared__ float wsum[2][3][32];
        __shared__ int first[33];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        // invariant: f(lo) >= top_p z > f(hi), f(t) = sum of the values >= t; f(hi) = above
        // (the largest value is exp(0) = 1; the first lo only where rounding is far below 1 - top_p)
        const float target = top_p * z;
        uint32_t lo = top_p < 0.999f ? __float_as_uint((1.f - top_p) * z / (2.f * V)) : 0u;
        uint32_t hi = __float_as_uint(1.f) + 1u;
        if (!(z >= 1.f)) lo = 0u;  // NaN
        float above = 0.f;
        int it = 0;  // (two buffers: a warp is at most one pass ahead of another's reads)
        for (; hi - lo > kBracket; ++it) {
            const uint32_t mid = lo + ((hi - lo) >> 1);
            const float t = __uint_as_float(mid);
            float part = 0.f;
#pragma unroll
            for (int k = 0; k < kSegMax; ++k)
                if (r[k] >= t) part += r[k];
            part = warp_sum(part);
            if (lane == 0) wsum[it & 1][0][warp] = part;
            __syncthreads();
            const float tot = warp_sum(wsum[it & 1][0][lane]);
            if (tot >= target) lo = mid;
            else { hi = mid; above = tot; }
        }
        if (hi - lo > 1u) {  // (uniform)
            // (zeros, the padding of the last segments among them, are never listed: at most V values)
            const float from = __uint_as_float(max(lo, 1u)), to = __uint_as_float(hi);
            int mine = 0;
#pragma unroll
            for (int k = 0; k < kSegMax; ++k) mine += r[k] >= from && r[k] < to;
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) first[warp] = incl;
            __syncthreads();
            if (warp == 0) {
                const int c = first[lane];
                int in2 = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, in2, o);
                    if (lane >= o) in2 += y;
                }
                first[lane] = in2 - c;
                if (lane == 31) first[32] = in2;
            }
            __syncthreads();
            int at = first[warp] + incl - mine;
#pragma unroll
            for (int k = 0; k < kSegMax; ++k)
                if (r[k] >= from && r[k] < to) s[at++] = r[k];
            __syncthreads();
            const int n_list = first[32];
            const bool one = n_list <= kShortList;
            const int i0 = one ? lane : threadIdx.x, step = one ? 32 : kRowThreads;
            for (; hi - lo > 1u && !(one && warp); ++it) {
                uint32_t m[3];
                float part[3] = {0.f, 0.f, 0.f};
#pragma unroll
                for (int j = 0; j < 3; ++j) m[j] = lo + max(1u, (uint32_t)(j + 1) * (hi - lo) >> 2);
#pragma unroll 4
                for (int i = i0; i < n_list; i += step) {
                    const float v = s[i];
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        if (v >= __uint_as_float(m[j])) part[j] += v;
                }
#pragma unroll
                for (int j = 0; j < 3; ++j) part[j] = warp_sum(part[j]);
                if (!one) {
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        if (lane == 0) wsum[it & 1][j][warp] = part[j];
                    __syncthreads();
#pragma unroll
                    for (int j = 0; j < 3; ++j) part[j] = warp_sum(wsum[it & 1][j][lane]);
                }
                if (above + part[2] >= target) lo = m[2];
                else if (above + part[1] >= target) { lo = m[1]; hi = m[2]; }
                else if (above + part[0] >= target) { lo = m[0]; hi = m[1]; }
                else hi = m[0];
            }
            if (threadIdx.x == 0) first[0] = (int)lo;
            __syncthreads();  // (also: the list has been read)
            lo = (uint32_t)first[0];
        }
        // kept mass (deterministic recount) and renormalisation (a NaN row keeps nothing)
        const float tau = z >= 1.f ? __uint_as_float(lo) : z;
        float kept = 0.f;
#pragma unroll
        for (int k = 0; k < kSegMax; ++k)
            if (r[k] >= tau) kept += r[k];
        kept = block_sum(kept, red);
#pragma unroll
        for (int k = 0; k < kSegMax; ++k) r[k] = r[k] >= tau ? r[k] / kept : 0.f;
    } else {
#pragma unroll
        for (int k = 0; k < kSegMax; ++k) r[k] = r[k] / z;
    }
#pragma unroll
    for (int k = 0; k < kSegMax; ++k)
        if (k < n) s[row_at(beg + k)] = r[k];
    __syncthreads();
}

// Inverse-CDF draw over the shared row s: the first x (ascending) with
// cumsum(x) > u * total.  Thread t owns the contiguous segment of the row and
// the interval [E_t, E_{t+1}) of the cumulative mass, E the exclusive scan of
// the segment sums (E_1024 = total), so exactly one segment holds the target;
// its thread walks it.  A target at or beyond the total (rounding as u -> 1)
// takes the last token with positive mass.
__device__ int sample_row(const float* s, int V, float u, float* red, int* redi) {
    __shared__ float ex[kRowThreads];
    const int seg = (V + kRowThreads - 1) / kRowThreads;
    const int beg = min(V, threadIdx.x * seg), end = min(V, beg + seg);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float mine = 0.f;
    int last_pos = -1;
    for (int i = beg; i < end; ++i) {
        const float v = s[row_at(i)];
        mine += v;
        if (v > 0.f) last_pos = i;
    }
    float incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        float y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) red[warp] = incl;
    int lp = last_pos;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lp = max(lp, __shfl_xor_sync(0xffffffffu, lp, o));
    if (lane == 0) redi[warp] = lp;
    __syncthreads();
    if (warp == 0) {
        const float wt = red[lane];
        float wi = wt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            float y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        red[lane] = wi - wt;
        if (lane == 31) red[32] = wi;
        int l2 = redi[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l2 = max(l2, __shfl_xor_sync(0xffffffffu, l2, o));
        if (lane == 0) { redi[32] = l2; redi[33] = -1; }
    }
    __syncthreads();
    const float e_mine = red[warp] + (incl - mine);
    ex[threadIdx.x] = e_mine;
    __syncthreads();
    const float total = red[32];
    const float e_next = threadIdx.x + 1 < kRowThreads ? ex[threadIdx.x + 1] : total;
    const float target = u * total;
    if (e_mine <= target && target < e_next) {
        float cum = e_mine;
        int pick = last_pos;
        for (int i = beg; i < end; ++i) {
            const float v = s[row_at(i)];
            cum += v;
            if (cum > target && v > 0.f) { pick = i; break; }
        }
        redi[33] = pick;
    }
    __syncthreads();
    const int r = redi[33] >= 0 ? redi[33] : redi[32];
    __syncthreads();
    return r < 0 ? 0 : r;
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
// greedy drafting: d_{j+1} = argmax of the draft logits.  With the draft
// exit on, the draft's confidence max softmax = 1 / sum_x exp(l_x - l_max)
// below gamma ends the round's drafting (Sec. 3.4; the draft is kept); a
// drafting stage that has ended adds nothing.
__global__ void __launch_bounds__(kRowThreads) greedy_draft_kernel(const float* __restrict__ logits,
                                                                   int V, DecodeState* st) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ float redf[33];
    __shared__ int redi[34];
    if (st->exited) return;
    int best = block_argmax(logits, V, redf, redi);
    bool stop = false;
    if (st->exit_on) {
        const float lmax = logits[best];
        float s = 0.f;
        for (int i = threadIdx.x; i < V; i += kRowThreads) s += expf(logits[i] - lmax);
        s = block_sum(s, redf);
        stop = 1.f / s < st->gamma;
    }
    if (threadIdx.x == 0) {
        st->drafts[st->j] = best;
        st->j = st->j + 1;
        if (stop) st->exited = 1;
    }
}

// emission + rollback shared by both acceptance kernels (one thread)
__device__ void emit_round(DecodeState* st, int n, int y, int Kd, int* out_tokens) {
    const int e = st->emitted;
    for (int i = 0; i < n; ++i) out_tokens[e + i] = st->drafts[i];
    out_tokens[e + n] = y;
    st->emitted = e + n + 1;
    st->len = st->len + n + 1;
    st->x_last = y;
    st->rounds += 1;
    st->drafted += Kd;
    st->accepted += n;
    st->hist[n] += 1;
    st->j = 0;
    // adaptive draft exit: Eqs. 2-4 after a verification that had drafts
    if (st->exit_on && Kd > 0) {
        const float ar_e = (float)n / (float)Kd;
        const float b1 = st->exit_updates == 0 ? 0.f : st->beta1;
        st->ar_smooth = b1 * st->ar_smooth + (1.f - b1) * ar_e;
        const float gt = st->ar_smooth <= st->alpha ? st->gamma + st->eps : st->gamma - st->eps;
        st->gamma = st->beta2 * st->gamma + (1.f - st->beta2) * gt;
        st->exit_updates += 1;
    }
    st->exited = 0;
}

// greedy verification: one CTA per row computes argmax p_m; the last CTA
// accepts the longest matching prefix and emits (Algorithm 2)
__global__ void __launch_bounds__(kRowThreads) greedy_accept_kernel(
    const float* __restrict__ logits, int V, int M, DecodeState* st, int* out_tokens,
    unsigned* counter, int* argbuf) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ float redf[33];
    __shared__ int redi[34];
    __shared__ int s_last;
    const int m = blockIdx.x;
    int best = block_argmax(logits + (size_t)m * V, V, redf, redi);
    if (threadIdx.x == 0) {
        argbuf[m] = best;
        __threadfence();
        unsigned prev = atomicAdd(counter, 1u);
        s_last = prev == (unsigned)(M - 1);
    }
    __syncthreads();
    if (!s_last || threadIdx.x != 0) return;
    __threadfence();
    int n = 0;
    while (n < M - 1 && st->drafts[n] == __ldcg(&argbuf[n])) ++n;
    const int y = __ldcg(&argbuf[n]);
    emit_round(st, n, y, M - 1, out_tokens);
    *counter = 0u;
}

// sampling drafting: q_{j+1} row kept for the acceptance test, d ~ q
__global__ void __launch_bounds__(kRowThreads) sample_draft_kernel(const float* __restrict__ logits,
                                                                   int V, DecodeState* st,
                                                                   float* q_rows) {
    extern __shared__ float s[];
    pdl_launch_dependents();
    pdl_wait();
    __shared__ float red[33];
    __shared__ int redi[34];
    if (st->exited) return;  // the round's drafting stage has ended
    const int j = st->j;
    nucleus_row(logits, V, st->inv_temperature, st->top_p, s, red);
    float* q = q_rows + (size_t)j * V;
    float qmax = 0.f;
    for (int i = threadIdx.x; i < V; i += kRowThreads) {
        const float v = s[row_at(i)];
        q[i] = v;
        qmax = fmaxf(qmax, v);
    }
    const bool stop = st->exit_on && block_max(qmax, red) < st->gamma;  // confidence = max q (Sec. 3.4)
    const float u = uniform01(st->seed, st->len + j + 1, 0);
    int d = sample_row(s, V, u, red, redi);
    if (threadIdx.x == 0) {
        st->drafts[j] = d;
        st->j = j + 1;
        if (stop) st->exited = 1;
    }
}

// Algorithm 4's verification for one round, executed by one 1024-thread CTA
// over target rows p (Kd+1 rows) and draft rows q (Kd rows).  Returns n via
// *n_out and the correction / bonus token.
__device__ int spec_accept_core(const float* p, const float* q, const int* drafts, int Kd, int V,
                                unsigned long long seed, int len, float* s, float* red,
                                int* redi, int* n_out) {
    __shared__ int s_rej;
    if (threadIdx.x < 32) {  // lane j tests draft j (Kd <= 15), all loads at once
        const int j = threadIdx.x;
        bool reject = false;
        if (j < Kd) {
            const int x = drafts[j];
            const float pj = __ldcg(p + (size_t)j * V + x);
            const float qj = __ldcg(q + (size_t)j * V + x);
            const float r = uniform01(seed, len + j + 1, 1);
            // r < min(1, pj / qj)  <=>  r * qj < pj  (qj > 0)
            reject = qj > 0.f && !(r * qj < pj);
        }
        const unsigned rejected = __ballot_sync(0xffffffffu, reject);
        // index of the first rejected draft (0-based), Kd = none
        if (j == 0) s_rej = rejected ? __ffs(rejected) - 1 : Kd;
    }
    __syncthreads();
    const int rej = s_rej;
    const int seg = (V + kRowThreads - 1) / kRowThreads;
    const int beg = min(V, threadIdx.x * seg), end = min(V, beg + seg);
    int y;
    if (rej < Kd) {
        const float* pj = p + (size_t)rej * V;
        const float* qj = q + (size_t)rej * V;
        for (int i = threadIdx.x; i < V; i += kRowThreads) {
            const float dlt = __ldcg(pj + i) - __ldcg(qj + i);
            s[row_at(i)] = dlt > 0.f ? dlt : 0.f;
        }
        __syncthreads();
        float tot = 0.f;
        for (int i = beg; i < end; ++i) tot += s[row_at(i)];
        tot = block_sum(tot, red);
        if (!(tot > 1e-30f)) {
            for (int i = threadIdx.x; i < V; i += kRowThreads) s[row_at(i)] = __ldcg(pj + i);
        }
        __syncthreads();
        y = sample_row(s, V, uniform01(seed, len + rej + 1, 2), red, redi);
    } else {
        const float* pk = p + (size_t)Kd * V;
        for (int i = threadIdx.x; i < V; i += kRowThreads) s[row_at(i)] = __ldcg(pk + i);
        __syncthreads();
        y = sample_row(s, V, uniform01(seed, len + Kd + 1, 2), red, redi);
    }
    *n_out = rej;
    return y;
}

__global__ void __launch_bounds__(kRowThreads) sample_accept_kernel(
    const float* __restrict__ logits, int V, int M, DecodeState* st, float* p_rows,
    const float* q_rows, int* out_tokens, unsigned* counter) {
    extern __shared__ float s[];
    pdl_launch_dependents();
    pdl_wait();
    __shared__ float red[33];
    __shared__ int redi[34];
    __shared__ int s_last;
    const int m = blockIdx.x;
    nucleus_row(logits + (size_t)m * V, V, st->inv_temperature, st->top_p, s, red);
    float* pr = p_rows + (size_t)m * V;
    for (int i = threadIdx.x; i < V; i += kRowThreads) pr[i] = s[row_at(i)];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned prev = atomicAdd(counter, 1u);
        s_last = prev == (unsigned)(M - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    int n;
    const int y = spec_accept_core(p_rows, q_rows, st->drafts, M - 1, V, st->seed, st->len, s, red,
                                   redi, &n);
    if (threadIdx.x == 0) {
        emit_round(st, n, y, M - 1, out_tokens);
        *counter = 0u;
    }
}

__global__ void __launch_bounds__(kRowThreads) spec_accept_batch_kernel(
    const float* p, const float* q, int V, int Kd, const int* drafts,
    const unsigned long long* seeds, int pos0, int* out) {
    extern __shared__ float s[];
    __shared__ float red[33];
    __shared__ int redi[34];
    const int t = blockIdx.x;
    int n;
    const int y = spec_accept_core(p, q, drafts + (size_t)t * Kd, Kd, V, seeds[t], pos0, s, red,
                                   redi, &n);
    if (threadIdx.x == 0) {
        out[2 * t] = n;
        out[2 * t + 1] = y;
    }
}

template <typename Kern, typename... Args>
int launch_pdl(Kern k, dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace

int sampling_configure() {
    // load every kernel of this file now, outside any stream capture
    cudaFuncAttributes fa;
    cudaError_t e0 = cudaFuncGetAttributes(&fa, greedy_draft_kernel);
    if (e0 == cudaSuccess) e0 = cudaFuncGetAttributes(&fa, greedy_accept_kernel);
    if (e0 != cudaSuccess) return (int)e0;
    const int big = 160 * 1024;
    cudaError_t e = cudaFuncSetAttribute(sample_draft_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(sample_accept_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(spec_accept_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    return (int)e;
}

int launch_greedy_draft(const float* logits, int V, DecodeState* st, cudaStream_t s) {
    return launch_pdl(greedy_draft_kernel, dim3(1), dim3(kRowThreads), 0, s, logits, V, st);
}

int launch_greedy_accept(const float* logits, int V, int M, DecodeState* st, int* out_tokens,
                         unsigned* counter, int* argmax_buf, cudaStream_t s) {
    return launch_pdl(greedy_accept_kernel, dim3(M), dim3(kRowThreads), 0, s, logits, V, M, st,
                      out_tokens, counter, argmax_buf);
}

int launch_sample_draft(const float* logits, int V, DecodeState* st, float* q_rows, cudaStream_t s) {
    return launch_pdl(sample_draft_kernel, dim3(1), dim3(kRowThreads), row_bytes(V), s, logits, V,
                      st, q_rows);
}

int launch_sample_accept(const float* logits, int V, int M, DecodeState* st, float* p_rows,
                         const float* q_rows, int* out_tokens, unsigned* counter, cudaStream_t s) {
    return launch_pdl(sample_accept_kernel, dim3(M), dim3(kRowThreads), row_bytes(V), s, logits, V,
                      M, st, p_rows, q_rows, out_tokens, counter);
}

int launch_spec_accept_batch(const float* p_rows, const float* q_rows, int V, int Kd,
                             const int* drafts, const unsigned long long* seeds, int trials,
                             int pos0, int* out, cudaStream_t s) {
    spec_accept_batch_kernel<<<trials, kRowThreads, row_bytes(V), s>>>(p_rows, q_rows, V, Kd, drafts,
                                                                        seeds, pos0, out);
    return (int)cudaGetLastError();
}

}  // namespace ssd
