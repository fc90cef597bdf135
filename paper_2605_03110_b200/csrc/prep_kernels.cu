// HBM-bound helper kernels of the selection path: fused row-norm + representative
// gather (with validation of the inherited list), and the prefix-sum compaction that
// turns gamma into sorted index lists.
#include <new>

#include "gram_tc_dev.cuh"

namespace ada {

// ---------------------------------------------------------------------------
// Row normalisation fused with the representative gather (Section 2.1;
// Algorithm 1 lines 1-2).  One warp per row, 128-bit loads.  inv_norm[t] =
// 1/||x_t|| in fp32 (0 for a zero row).  The rows of the inherited list are
// copied, raw, to Xrep[position] together with their inverse norm.
// ---------------------------------------------------------------------------
template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ float sumsq(const uint4& v) {
        const float a = __uint_as_float(v.x), b = __uint_as_float(v.y), c = __uint_as_float(v.z),
                    e = __uint_as_float(v.w);
        return a * a + b * b + c * c + e * e;
    }
    static __device__ __forceinline__ uint4 scale(const uint4& v, float f) {
        uint4 o;
        o.x = __float_as_uint(__uint_as_float(v.x) * f);
        o.y = __float_as_uint(__uint_as_float(v.y) * f);
        o.z = __float_as_uint(__uint_as_float(v.z) * f);
        o.w = __float_as_uint(__uint_as_float(v.w) * f);
        return o;
    }
};
template <>
struct Vec16<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ float2 up(unsigned w) {
        // a bf16 is the upper half of an fp32
        return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
    static __device__ __forceinline__ float sumsq(const uint4& v) {
        const float2 a = up(v.x), b = up(v.y), c = up(v.z), e = up(v.w);
        return (a.x * a.x + a.y * a.y) + (b.x * b.x + b.y * b.y) + (c.x * c.x + c.y * c.y) +
               (e.x * e.x + e.y * e.y);
    }
    static __device__ __forceinline__ unsigned scale2(unsigned w, float f) {
        const float2 a = up(w);
        const __nv_bfloat162 r = __floats2bfloat162_rn(a.x * f, a.y * f);
        return *reinterpret_cast<const unsigned*>(&r);
    }
    static __device__ __forceinline__ uint4 scale(const uint4& v, float f) {
        return make_uint4(scale2(v.x, f), scale2(v.y, f), scale2(v.z, f), scale2(v.w, f));
    }
};

// Warps [0, ceil(n_rows / NORM_ROWS)) normalise NORM_ROWS rows each: inv_norm[row] (and Xhat).  The warps
// after them serve the inherited list (Algorithm 1 "Require" and line 2): warp (b, i) with i < count
// validates entry i (in range, strictly above entry i-1), records role[token] = i+1, copies the raw
// row to Xrep[b, i] and stores its inverse norm.  Both kinds read X directly, so there is
// no dependency between them and no separate scatter pass.
constexpr int NORM_ROWS = 2;

template <typename T>
__global__ void __launch_bounds__(256)
k_norm_gather(const T* __restrict__ X, int64_t n_rows, int Tseq, int d, int64_t ldx, int64_t xb,
              float* __restrict__ inv_norm, T* __restrict__ Xhat,
              const int32_t* __restrict__ rep_in, const int32_t* __restrict__ rep_in_cnt,
              int32_t* __restrict__ role, int32_t* __restrict__ r_eff, T* __restrict__ Xrep,
              float* __restrict__ inv_rep, unsigned* __restrict__ status) {
    grid_dep_wait();
    grid_dep_launch_next();
    const int lane = threadIdx.x & 31;
    int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t n_norm_warps = (n_rows + NORM_ROWS - 1) / NORM_ROWS;
    if (inv_norm == nullptr && Xhat == nullptr) w += n_norm_warps;   // gather-only launch: list warps only
    constexpr int N = Vec16<T>::N;
    const int nvec = d / N;  // d*es is a multiple of 16 bytes
    if (w < n_norm_warps) {
        // row (b, t) of X starts at b * xb + t * ldx (xb = Tseq * ldx for stacked sequences,
        // the head width for heads interleaved inside one row)
        const uint4* src[NORM_ROWS];
        float ss[NORM_ROWS];
#pragma unroll
        for (int u = 0; u < NORM_ROWS; ++u) {
            const unsigned row = (unsigned)min(w * NORM_ROWS + u, n_rows - 1);
            src[u] = reinterpret_cast<const uint4*>(X + (int64_t)(row / (unsigned)Tseq) * xb + (int64_t)(row % (unsigned)Tseq) * ldx);
            ss[u] = 0.f;
        }
        for (int v = lane; v < nvec; v += 128) {
            uint4 x[NORM_ROWS][4];
#pragma unroll
            for (int u = 0; u < NORM_ROWS; ++u)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    x[u][q] = v + 32 * q < nvec ? __ldg(src[u] + v + 32 * q) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < NORM_ROWS; ++u)
                ss[u] += (Vec16<T>::sumsq(x[u][0]) + Vec16<T>::sumsq(x[u][1])) + (Vec16<T>::sumsq(x[u][2]) + Vec16<T>::sumsq(x[u][3]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int u = 0; u < NORM_ROWS; ++u) ss[u] += __shfl_xor_sync(0xffffffffu, ss[u], o);
#pragma unroll
        for (int u = 0; u < NORM_ROWS; ++u) {
            const int64_t row = w * NORM_ROWS + u;
            if (row >= n_rows) break;
            float inv = 0.f;
            if (!(ss[u] <= 3.0e38f)) {  // NaN or overflow to Inf
                if (lane == 0) atomicOr(status, ST_NONFINITE);
            } else if (ss[u] > 0.f) {
                inv = 1.0f / sqrtf(ss[u]);
            } else if (lane == 0) {
                atomicAdd(status + 1, 1u);
            }
            if (inv_norm != nullptr && lane == 0) inv_norm[row] = inv;
            if (Xhat != nullptr) {
                uint4* dst = reinterpret_cast<uint4*>(Xhat + row * (int64_t)d);
                for (int v = lane; v < nvec; v += 32) dst[v] = Vec16<T>::scale(__ldg(src[u] + v), inv);
            }
        }
        return;
    }
    w -= n_norm_warps;
    if (rep_in == nullptr || w >= n_rows) return;
    const int b = (int)(w / Tseq), i = (int)(w % Tseq);
    int cnt = rep_in_cnt[b];
    if (cnt < 0 || cnt > Tseq) {
        if (i == 0 && lane == 0) atomicOr(status, ST_BAD_COUNT);
        cnt = cnt < 0 ? 0 : Tseq;
    }
    if (i == 0 && lane == 0 && r_eff != nullptr) r_eff[b] = cnt;
    if (i >= cnt) return;
    const int32_t* list = rep_in + (int64_t)b * Tseq;
    const int32_t idx = list[i];
    bool ok = idx >= 0 && idx < Tseq;
    if (ok && i > 0) ok = list[i - 1] < idx;
    if (!ok) {
        if (lane == 0) atomicOr(status, ST_BAD_INDEX);
        return;
    }
    const int64_t prow = (int64_t)b * Tseq + i;
    const uint4* src = reinterpret_cast<const uint4*>(X + (int64_t)b * xb + (int64_t)idx * ldx);
    uint4* dst = reinterpret_cast<uint4*>(Xrep + prow * (int64_t)d);
    float ss = 0.f;
    int v = lane;
    for (; v + 224 < nvec; v += 256) {          // eight loads in flight per lane
        uint4 x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = __ldg(src + v + 32 * q);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            ss += Vec16<T>::sumsq(x[q]);
            dst[v + 32 * q] = x[q];
        }
    }
    for (; v < nvec; v += 32) {
        const uint4 x = __ldg(src + v);
        ss += Vec16<T>::sumsq(x);
        dst[v] = x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) {
        inv_rep[prow] = (ss <= 3.0e38f && ss > 0.f) ? 1.0f / sqrtf(ss) : 0.f;
        if (role != nullptr) role[(int64_t)b * Tseq + idx] = i + 1;
    }
}

constexpr int NORM_U = 4;   // rows per lane group of the short-row kernel

// The same work for short rows (at most 16 vectors, e.g. one attention head), where a warp
// per row would leave most lanes idle behind a single load.  Warps [0, n_norm_warps) take
// rpw rows each, the warps after them rpw consecutive positions of one sequence's list.
template <typename T>
__global__ void __launch_bounds__(256)
k_norm_gather_short(const T* __restrict__ X, int64_t n_rows, int Tseq, int d, int64_t ldx, int64_t xb,
                    int rpw, int64_t n_norm_warps, float* __restrict__ inv_norm, T* __restrict__ Xhat,
                    const int32_t* __restrict__ rep_in, const int32_t* __restrict__ rep_in_cnt,
                    int32_t* __restrict__ role, int32_t* __restrict__ r_eff, T* __restrict__ Xrep,
                    float* __restrict__ inv_rep, unsigned* __restrict__ status) {
    grid_dep_wait();
    grid_dep_launch_next();
    const int lane = threadIdx.x & 31;
    int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (inv_norm == nullptr && Xhat == nullptr) w += n_norm_warps;   // gather-only launch: list warps only
    constexpr int N = Vec16<T>::N;
    const int nvec = d / N;  // d*es is a multiple of 16 bytes
    if (w < n_norm_warps) {
        // Short rows (at most 16 vectors, e.g. one attention head): a group of G lanes owns a
        // row, the warp's 32/G groups take NORM_U rows each, and every lane has NORM_U loads in
        // flight; a warp per row would leave most lanes idle behind one load.  Rows are taken
        // in memory order: head-fastest when the heads of a token lie side by side.
        const int R = rpw / NORM_U, G = 32 / R, sub = lane / G, gl = lane % G;
        // (row counts fit 31 bits; 32-bit division is several times cheaper than 64-bit)
        const unsigned nseq = (unsigned)n_rows / (unsigned)Tseq;
        uint4 x[NORM_U];
        int64_t orow[NORM_U];
#pragma unroll
        for (int u = 0; u < NORM_U; ++u) {
            const int64_t r = w * rpw + u * R + sub;
            x[u] = make_uint4(0u, 0u, 0u, 0u);
            orow[u] = -1;
            if (r < n_rows) {
                const unsigned r32 = (unsigned)r;
                const int64_t b = xb < ldx ? r32 % nseq : r32 / (unsigned)Tseq,
                              t = xb < ldx ? r32 / nseq : r32 % (unsigned)Tseq;
                orow[u] = b * Tseq + t;
                if (gl < nvec) x[u] = __ldg(reinterpret_cast<const uint4*>(X + b * xb + t * ldx) + gl);
            }
        }
#pragma unroll
        for (int u = 0; u < NORM_U; ++u) {
            float ss = Vec16<T>::sumsq(x[u]);
            for (int o = G >> 1; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (orow[u] < 0) continue;
            float inv = 0.f;
            if (!(ss <= 3.0e38f)) {
                if (gl == 0) atomicOr(status, ST_NONFINITE);
            } else if (ss > 0.f) {
                inv = 1.0f / sqrtf(ss);
            } else if (gl == 0) {
                atomicAdd(status + 1, 1u);
            }
            if (inv_norm != nullptr && gl == 0) inv_norm[orow[u]] = inv;
            if (Xhat != nullptr && gl < nvec)
                reinterpret_cast<uint4*>(Xhat + orow[u] * (int64_t)d)[gl] = Vec16<T>::scale(x[u], inv);
        }
        return;
    }
    w -= n_norm_warps;
    if (rep_in == nullptr) return;
    {
        // short rows: a lane group per list entry, NORM_U entries per group, as above; a warp
        // covers rpw consecutive positions of one sequence's list
        const int R = rpw / NORM_U, G = 32 / R, sub = lane / G, gl = lane % G;
        const unsigned wps = (unsigned)(Tseq + rpw - 1) / (unsigned)rpw;   // warps per sequence
        if (w >= (int64_t)wps * ((unsigned)n_rows / (unsigned)Tseq)) return;
        const int b = (int)((unsigned)w / wps);
        const int i0 = (int)((unsigned)w % wps) * rpw;
        int cnt = rep_in_cnt[b];
        if (cnt < 0 || cnt > Tseq) {
            if (i0 == 0 && lane == 0) atomicOr(status, ST_BAD_COUNT);
            cnt = cnt < 0 ? 0 : Tseq;
        }
        if (i0 == 0 && lane == 0 && r_eff != nullptr) r_eff[b] = cnt;
        if (i0 >= cnt) return;
        const int32_t* list = rep_in + (int64_t)b * Tseq;
        int32_t idx[NORM_U], prev[NORM_U];
#pragma unroll
        for (int u = 0; u < NORM_U; ++u) {
            const int i = i0 + u * R + sub;
            idx[u] = i < cnt ? list[i] : -1;
            prev[u] = (i < cnt && i > 0) ? list[i - 1] : -1;
        }
        uint4 x[NORM_U];
        bool ok[NORM_U];
#pragma unroll
        for (int u = 0; u < NORM_U; ++u) {
            const int i = i0 + u * R + sub;
            ok[u] = i < cnt && idx[u] >= 0 && idx[u] < Tseq && prev[u] < idx[u];
            if (i < cnt && !ok[u] && gl == 0) atomicOr(status, ST_BAD_INDEX);
            x[u] = make_uint4(0u, 0u, 0u, 0u);
            if (ok[u] && gl < nvec)
                x[u] = __ldg(reinterpret_cast<const uint4*>(X + (int64_t)b * xb + (int64_t)idx[u] * ldx) + gl);
        }
#pragma unroll
        for (int u = 0; u < NORM_U; ++u) {
            const int i = i0 + u * R + sub;
            float ss = Vec16<T>::sumsq(x[u]);
            for (int o = G >> 1; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (!ok[u]) continue;
            const int64_t prow = (int64_t)b * Tseq + i;
            if (gl < nvec) reinterpret_cast<uint4*>(Xrep + prow * (int64_t)d)[gl] = x[u];
            if (gl == 0) {
                inv_rep[prow] = (ss <= 3.0e38f && ss > 0.f) ? 1.0f / sqrtf(ss) : 0.f;
                if (role != nullptr) role[(int64_t)b * Tseq + idx[u]] = i + 1;
            }
        }
        return;
    }
}

cudaError_t launch_norm_gather(ada_ctx* ctx, const void* X, int B, int T, int d, int64_t ldx,
                               int64_t xb, ada_dtype dt, float* inv_norm, void* Xhat, const int32_t* rep_in,
                               const int32_t* rep_in_cnt, int32_t* role, int32_t* r_eff, void* Xrep,
                               float* inv_rep, cudaStream_t s) {
    const int64_t n_rows = (int64_t)B * T;
    const int warps = 8;
    const bool gather_only = inv_norm == nullptr && Xhat == nullptr;
    // rows per norm warp: lane groups of the next power of two at or above the row's vector count
    const int nvec = d / (dt == ADA_F32 ? 4 : 8);
    int G = 32;
    if (nvec <= 16) for (G = 1; G < nvec; G <<= 1) {}
    const int rpw = G == 32 ? 1 : (32 / G) * NORM_U;
    const int64_t n_norm_warps = rpw == 1 ? (n_rows + NORM_ROWS - 1) / NORM_ROWS : (n_rows + rpw - 1) / rpw;
    // list warps: one per list position, or one per rpw positions of a sequence (short rows)
    const int64_t n_list_warps = rpw == 1 ? n_rows : (int64_t)B * ((T + rpw - 1) / rpw);
    const int64_t n_warps = gather_only ? n_list_warps
                                        : (rep_in != nullptr ? n_norm_warps + n_list_warps : n_norm_warps);
    const unsigned grid = (unsigned)((n_warps + warps - 1) / warps);
    prof_begin(ctx, K_NORM_GATHER, s);
    if (rpw > 1) {
        if (dt == ADA_F32) {
            launch_k(ctx, k_norm_gather_short<float>, dim3(grid), dim3(warps * 32), 0, s,
                (const float*)X, n_rows, T, d, ldx, xb, rpw, n_norm_warps, inv_norm, (float*)Xhat, rep_in,
                rep_in_cnt, role, r_eff, (float*)Xrep, inv_rep, ctx->status);
        } else {
            launch_k(ctx, k_norm_gather_short<__nv_bfloat16>, dim3(grid), dim3(warps * 32), 0, s,
                (const __nv_bfloat16*)X, n_rows, T, d, ldx, xb, rpw, n_norm_warps, inv_norm,
                (__nv_bfloat16*)Xhat, rep_in, rep_in_cnt, role, r_eff, (__nv_bfloat16*)Xrep, inv_rep,
                ctx->status);
        }
    } else if (dt == ADA_F32) {
        launch_k(ctx, k_norm_gather<float>, dim3(grid), dim3(warps * 32), 0, s,
            (const float*)X, n_rows, T, d, ldx, xb, inv_norm, (float*)Xhat, rep_in, rep_in_cnt, role,
            r_eff, (float*)Xrep, inv_rep, ctx->status);
    } else {
        launch_k(ctx, k_norm_gather<__nv_bfloat16>, dim3(grid), dim3(warps * 32), 0, s,
            (const __nv_bfloat16*)X, n_rows, T, d, ldx, xb, inv_norm, (__nv_bfloat16*)Xhat, rep_in,
            rep_in_cnt, role, r_eff, (__nv_bfloat16*)Xrep, inv_rep, ctx->status);
    }
    prof_end(ctx, s);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Preparation of an fp32 call as a launch of its own, for the one-CTA tensor-core kernel (the
// pair kernel does the same work inside its launch): bf16 planes and inverse norms of the rows of
// X and of the inherited list.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_split_bf16(const SplitJob job, unsigned* __restrict__ status) {
    grid_dep_wait();
    const int warps = blockDim.x >> 5;
    tc::split_rows(job, (threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x, (int)gridDim.x * warps, threadIdx.x & 31,
                   status);
}

cudaError_t launch_split(ada_ctx* ctx, const SplitJob& job, cudaStream_t s) {
    const int64_t rows = (int64_t)job.B * job.T;
    const int64_t want = (rows + 7) / 8;
    prof_begin(ctx, K_SPLIT, s);
    launch_k(ctx, k_split_bf16, dim3((unsigned)(want < 8 * ctx->sm_count ? want : 8 * ctx->sm_count)), dim3(256), 0, s,
             job, ctx->status);
    prof_end(ctx, s);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Compaction (Definition 1's threshold; Algorithm 1 lines 5, 9, 10-11 and the lists of
// Eq. 6).  One cluster of up to eight 1024-thread blocks per sequence; a block owns V x 1024
// consecutive tokens of every round of (blocks x V x 1024), one token per thread and slice, so
// all loads are coalesced and the whole sequence is in flight at once.  Ballots give a warp's
// three counts, one warp per block scans them, the block totals go to the other blocks through
// distributed shared memory, and after ONE cluster barrier every thread knows its places in the
// ascending lists.  Every thread clears the scratch it read, so the workspace is all-zero again
// when the kernel ends and no memset is needed between calls.
//
// Bound by latency: a chain of dependent round trips on O(T) integers.  The blocks used to
// exchange their totals through global memory (publish, poll, and a fence and a counter to know
// when the words may be cleared); the outputs' first touch also misses the TLB when a chain of
// layers keeps its lists apart, hence the prefetches before the wait.
// ---------------------------------------------------------------------------
constexpr int COMPACT_CTAS = 8;      // largest portable cluster
constexpr unsigned COUNT_BITS = 21;  // three counts share a 64-bit word
constexpr unsigned long long COUNT_MASK = (1ull << COUNT_BITS) - 1;

struct CompactArgs {
    unsigned* g_tok;             // gamma (full) / gamma_cross by token, bit patterns
    unsigned* g_rep;             // gamma_rep by position (cascade) or NULL
    unsigned* g_rep_tok;         // the same by token, or NULL: read by position, behind the role map
    int32_t* role;               // 0 / position+1 (cascade) or NULL
    unsigned* dep_ctr;           // dependency counters of the Gram launch (cleared here)
    unsigned* status;
    int T;
    int prefetch;                // outputs are device memory
    float thr;
    int32_t *keep_idx, *keep_cnt, *add_idx, *add_cnt, *rem_idx, *rem_cnt;
    float *gamma_a, *gamma_b;    // full: gamma | cascade: gamma_rep, gamma_cross (optional)
    const float* row_scale;      // cascade: 1/||x_t|| still to be applied to g_tok, or NULL
    // adaptive threshold (Section 8.1): thresholds come from tu.tau_state
    const int32_t* r_in;         // [B] inherited counts (Eq. 6 denominator)
    TauUpdate tu;
};

__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// BY_TOK: gamma_rep comes by token.  (A parameter of the template: asked in the kernel it cost the steps without
// it 0.9 us, 2048 x 384 17.4 -> 18.4.)
template <int V, bool BY_TOK>
__global__ void __launch_bounds__(1024) k_compact(const CompactArgs a) {
    __shared__ unsigned long long s_off[V * 32];               // counts, then exclusive offsets, by slice and warp
    __shared__ unsigned long long s_total[2][COMPACT_CTAS];    // block totals of the cluster, by round parity
    const int b = blockIdx.y, rank = blockIdx.x, nblk = gridDim.x;   // the cluster is the x extent of the grid
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t o = (int64_t)b * a.T;
    const bool cascade = a.role != nullptr;
    if (a.prefetch) {
        const int t = rank * V * 1024 + V * (int)threadIdx.x;
        if ((threadIdx.x & 31) == 0 && t < a.T) {              // one touch per 128 V bytes of each output
            prefetch_l2(a.keep_idx + o + t);
            if (cascade) { prefetch_l2(a.add_idx + o + t); prefetch_l2(a.rem_idx + o + t); }
            if (a.gamma_a != nullptr) prefetch_l2(a.gamma_a + o + t);
            if (a.gamma_b != nullptr) prefetch_l2(a.gamma_b + o + t);
        }
        if (threadIdx.x == 1) {
            prefetch_l2(a.keep_cnt + b);
            if (cascade) { prefetch_l2(a.add_cnt + b); prefetch_l2(a.rem_cnt + b); }
        }
    }
    // every block of the cluster has started before any writes into another's shared memory
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    grid_dep_wait();
    grid_dep_launch_next();
    const unsigned faulted = a.status[0];
    float thr = a.thr;
    if (a.tu.tau_state != nullptr) {
        const double tau = a.tu.tau_state[b];
        thr = tau_threshold(tau);
        if (rank == 0 && threadIdx.x == 0 && !(tau > 0.0 && tau < 1.0)) atomicOr(a.status, ST_BAD_TAU);
    }
    unsigned long long carry = 0;                              // counts of the rounds before this one
    int par = 0;
    for (int t0 = 0; t0 < a.T; t0 += nblk * V * 1024, par ^= 1) {
        const int tb = t0 + rank * V * 1024 + (int)threadIdx.x;
        // independent loads first, the position-indexed gather second
        int pos[V];
        unsigned gt[V], gp[V];
        float rs[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int t = tb + v * 1024;
            const bool in = t < a.T;
            pos[v] = (cascade && in) ? a.role[o + t] : 0;
            gt[v] = in ? a.g_tok[o + t] : 0u;
            rs[v] = (in && a.row_scale != nullptr) ? a.row_scale[o + t] : 1.0f;
            if (BY_TOK) gp[v] = in ? a.g_rep_tok[o + t] : 0u;
        }
        if (!BY_TOK) {
#pragma unroll
            for (int v = 0; v < V; ++v) gp[v] = pos[v] > 0 ? a.g_rep[o + pos[v] - 1] : 0u;
        }
        unsigned bk[V], ba[V], br[V];                          // ballots: kept, added, removed
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int t = tb + v * 1024;
            bool keep = false, add = false, rem = false;
            if (t < a.T) {
                float ga = 0.f, gb = 0.f;
                if (pos[v] > 0) {                 // inherited representative: line 5
                    ga = __uint_as_float(gp[v]);
                    keep = ga < thr;
                    rem = !keep;
                    a.g_rep[o + pos[v] - 1] = 0u;
                    if (BY_TOK) a.g_rep_tok[o + t] = 0u;
                    a.role[o + t] = 0;
                } else {                          // Definition 1 / line 9
                    // (an untouched entry is a maximum over nothing: 0 whatever the row's norm)
                    gb = gt[v] != 0u ? __uint_as_float(gt[v]) * rs[v] : 0.f;
                    keep = gb < thr;
                    add = cascade && keep;
                }
                a.g_tok[o + t] = 0u;
                if (cascade) {
                    if (a.gamma_a != nullptr) a.gamma_a[o + t] = ga;
                    if (a.gamma_b != nullptr) a.gamma_b[o + t] = gb;
                    if (faulted != 0u) {              // a rejected list leaves positions without a token
                        a.g_rep[o + t] = 0u;
                        if (BY_TOK) a.g_rep_tok[o + t] = 0u;
                    }
                } else if (a.gamma_a != nullptr) {
                    a.gamma_a[o + t] = gb;
                }
            }
            bk[v] = __ballot_sync(0xffffffffu, keep);
            ba[v] = __ballot_sync(0xffffffffu, add);
            br[v] = __ballot_sync(0xffffffffu, rem);
            if (lane == 0)
                s_off[v * 32 + warp] = (unsigned long long)__popc(bk[v]) |
                                       ((unsigned long long)__popc(ba[v]) << COUNT_BITS) |
                                       ((unsigned long long)__popc(br[v]) << (2 * COUNT_BITS));
        }
        __syncthreads();
        if (warp == 0) {                          // lane l scans entries l V .. l V + V - 1 (token order)
            unsigned long long c[V], mine = 0;
#pragma unroll
            for (int v = 0; v < V; ++v) { c[v] = s_off[lane * V + v]; mine += c[v]; }
            unsigned long long incl = mine;
#pragma unroll
            for (int q = 1; q < 32; q <<= 1) {
                const unsigned long long n = __shfl_up_sync(0xffffffffu, incl, q);
                if (lane >= q) incl += n;
            }
            const unsigned long long total = __shfl_sync(0xffffffffu, incl, 31);
            unsigned long long off = incl - mine;
#pragma unroll
            for (int v = 0; v < V; ++v) { s_off[lane * V + v] = off; off += c[v]; }
            if (lane < nblk) {                    // this block's total, to every block of the cluster
                unsigned dst;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                             : "=r"(dst)
                             : "r"((unsigned)__cvta_generic_to_shared(&s_total[par][rank])), "r"(lane));
                asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(dst), "l"(total) : "memory");
            }
        }
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        unsigned long long base = carry;
        for (int j = 0; j < nblk; ++j) {
            const unsigned long long n = s_total[par][j];
            carry += n;
            if (j < rank) base += n;
        }
        const unsigned below = (1u << lane) - 1u;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int t = tb + v * 1024;
            const unsigned long long off = base + s_off[v * 32 + warp];
            if ((bk[v] >> lane) & 1u) a.keep_idx[o + (int)(off & COUNT_MASK) + __popc(bk[v] & below)] = t;
            if ((ba[v] >> lane) & 1u) a.add_idx[o + (int)((off >> COUNT_BITS) & COUNT_MASK) + __popc(ba[v] & below)] = t;
            if ((br[v] >> lane) & 1u) a.rem_idx[o + (int)(off >> (2 * COUNT_BITS)) + __popc(br[v] & below)] = t;
        }
        if (t0 + nblk * V * 1024 < a.T) __syncthreads();       // s_off is reused
    }
    if (rank == 0 && threadIdx.x == 0) {
        a.keep_cnt[b] = (int)(carry & COUNT_MASK);
        if (cascade) {
            const int n_add = (int)((carry >> COUNT_BITS) & COUNT_MASK), n_rem = (int)(carry >> (2 * COUNT_BITS));
            a.add_cnt[b] = n_add;
            a.rem_cnt[b] = n_rem;
            if (a.tu.tau_state != nullptr) {
                // Eq. (6), then the threshold of the next layer: one rounded fp64 operation at a
                // time (no fused multiply-add), so that the state is reproducible bit for bit
                const int r_in = a.r_in[b];
                const bool defined = r_in > 0;
                const double rho = defined ? __ddiv_rn((double)(n_add + n_rem), (double)r_in) : 0.0;
                if (a.tu.turnover != nullptr)
                    a.tu.turnover[b] = defined ? (float)rho : __int_as_float(0x7fc00000);
                if (a.tu.update) {
                    // (every block of the cluster has read the old value: they are past the barrier)
                    double t = a.tu.tau_state[b];
                    if (defined) t = __dadd_rn(t, __dmul_rn(a.tu.gain, __dsub_rn(a.tu.target, rho)));
                    if (t < a.tu.tau_min) t = a.tu.tau_min;
                    if (t > a.tu.tau_max) t = a.tu.tau_max;
                    a.tu.tau_state[b] = t;
                }
            }
        }
        if (b == 0) {
            a.dep_ctr[0] = 0u;
            a.dep_ctr[1] = 0u;   // norm warps' counter of the Gram launch
            a.dep_ctr[3] = 0u;   // in-launch gather counter
        }
    }
}

// Nearest-representative map (Section 2.3): turns the packed keys of the argmax Gram launch
// into token indices.  A representative is its own nearest representative; a token whose
// correlations are all zero gets the first representative (lowest index among equals); an
// empty set gives -1.  Clears the keys and the role map it reads.
__global__ void __launch_bounds__(256)
k_nearest_finish(unsigned long long* __restrict__ near_key, int32_t* __restrict__ role,
                 const int32_t* __restrict__ r_eff, const float* __restrict__ inv_norm,
                 const int32_t* __restrict__ rep_idx, int T, int32_t* __restrict__ nearest_idx,
                 float* __restrict__ nearest_gamma, unsigned* __restrict__ dep_ctr) {
    grid_dep_wait();
    grid_dep_launch_next();
    const int b = blockIdx.y, t = blockIdx.x * blockDim.x + threadIdx.x;
    if (b == 0 && blockIdx.x == 0 && threadIdx.x < 4) dep_ctr[threadIdx.x] = 0u;   // counters of the Gram launch
    if (t >= T) return;
    const int64_t o = (int64_t)b * T;
    const unsigned long long key = near_key[o + t];
    const int p = role[o + t];
    const float inv = inv_norm[o + t];
    near_key[o + t] = 0ull;
    role[o + t] = 0;
    int idx;
    float g;
    if (p > 0) {
        idx = t;
        g = inv > 0.f ? 1.f : 0.f;
    } else if (r_eff[b] <= 0) {
        idx = -1;
        g = 0.f;
    } else {
        // (the key's value still lacks the row's own factor, GramProblem::defer_row; where that is 0 -- a
        // zero row, or one so small that its squares vanish -- the row correlates with nothing)
        g = __uint_as_float((unsigned)(key >> 32)) * inv;
        const bool some = g > 0.f;
        idx = rep_idx[o + (some ? 0xFFFFFFFFu - (unsigned)(key & 0xFFFFFFFFull) : 0u)];
        if (!some) g = 0.f;
    }
    nearest_idx[o + t] = idx;
    if (nearest_gamma != nullptr) nearest_gamma[o + t] = g;
}

cudaError_t launch_nearest_finish(ada_ctx* ctx, int B, int T, const int32_t* rep_idx,
                                  int32_t* nearest_idx, float* nearest_gamma, cudaStream_t s) {
    prof_begin(ctx, K_NEAREST_FINISH, s);
    launch_k(ctx, k_nearest_finish, dim3((T + 255) / 256, B), dim3(256), 0, s, ctx->near_key, ctx->role, ctx->r_eff,
                                                               ctx->inv_norm, rep_idx, T, nearest_idx,
                                                               nearest_gamma, ctx->tile_ctr);
    prof_end(ctx, s);
    return cudaGetLastError();
}

static cudaError_t launch_compact(ada_ctx* ctx, int kid, const CompactArgs& a, int B, cudaStream_t s) {
    // as few tokens per thread as the cluster allows; longer sequences than 4 x 8 x 1024 take rounds
    const int slices = (a.T + 1023) / 1024;
    const int V = slices <= COMPACT_CTAS ? 1 : (slices <= 2 * COMPACT_CTAS ? 2 : 4);
    const int nblk = slices < COMPACT_CTAS ? slices : COMPACT_CTAS;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(nblk, B);
    cfg.blockDim = dim3(1024);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nblk; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->dep_launch ? 2 : 1;
    prof_begin(ctx, kid, s);
    const bool by_tok = a.g_rep_tok != nullptr;
    void (*const kernel)(CompactArgs) = V == 1 ? (by_tok ? k_compact<1, true> : k_compact<1, false>)
                                      : V == 2 ? (by_tok ? k_compact<2, true> : k_compact<2, false>)
                                               : (by_tok ? k_compact<4, true> : k_compact<4, false>);
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
    if (e != cudaSuccess) cudaGetLastError();   // returned; the next launcher that asks must not find it again
    prof_end(ctx, s);
    return e;
}

cudaError_t launch_compact_full(ada_ctx* ctx, int B, int T, float thr, int32_t* rep_idx,
                                int32_t* rep_cnt, float* gamma, cudaStream_t s) {
    CompactArgs a;
    a.g_tok = ctx->g_tok; a.g_rep = nullptr; a.g_rep_tok = nullptr; a.role = nullptr;
    a.dep_ctr = ctx->tile_ctr; a.status = ctx->status;
    a.T = T; a.thr = thr; a.prefetch = ctx->host_out ? 0 : 1;
    a.keep_idx = rep_idx; a.keep_cnt = rep_cnt;
    a.add_idx = nullptr; a.add_cnt = nullptr; a.rem_idx = nullptr; a.rem_cnt = nullptr;
    a.gamma_a = gamma; a.gamma_b = nullptr; a.row_scale = nullptr;
    a.r_in = nullptr;
    memset(&a.tu, 0, sizeof(a.tu));
    return launch_compact(ctx, K_COMPACT_FULL, a, B, s);
}

cudaError_t launch_compact_cascade(ada_ctx* ctx, int B, int T, float thr, int32_t* rep_out,
                                   int32_t* rep_out_cnt, int32_t* add_idx, int32_t* add_cnt,
                                   int32_t* rem_idx, int32_t* rem_cnt, float* gamma_rep,
                                   float* gamma_cross, const TauUpdate& tu, bool row_scale, bool by_tok,
                                   cudaStream_t s) {
    CompactArgs a;
    a.g_tok = ctx->g_tok; a.g_rep = ctx->g_rep; a.g_rep_tok = by_tok ? ctx->g_rep_tok : nullptr; a.role = ctx->role;
    a.dep_ctr = ctx->tile_ctr; a.status = ctx->status;
    a.T = T; a.thr = thr; a.prefetch = ctx->host_out ? 0 : 1;
    a.keep_idx = rep_out; a.keep_cnt = rep_out_cnt;
    a.add_idx = add_idx; a.add_cnt = add_cnt; a.rem_idx = rem_idx; a.rem_cnt = rem_cnt;
    a.gamma_a = gamma_rep; a.gamma_b = gamma_cross;
    a.row_scale = row_scale ? ctx->inv_norm : nullptr;
    a.r_in = ctx->r_eff;
    a.tu = tu;
    return launch_compact(ctx, K_COMPACT_CASCADE, a, B, s);
}

void* new_map_cache() { return new (std::nothrow) tc::MapCache; }
void delete_map_cache(void* c) { delete static_cast<tc::MapCache*>(c); }

}  // namespace ada
