// C ABI of libada.so: argument checks, workspace, kernel sequencing.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <atomic>
#include <new>

#include "common.cuh"

using namespace ada;

namespace {

const char* const kKernelNames[K_COUNT] = {
    "norm_gather",     "gram_ffma_tri",    "gram_ffma_cross",
    "gram_tc_tri",     "gram_tc_cross",    "gram_tc_cascade", "split_bf16x3",  "compact_full",
    "compact_cascade", "nearest_finish",  "step_short",
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

ada_status check_common(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d, int64_t ldx,
                        ada_dtype dt) {
    if (ctx == nullptr || X == nullptr) return ADA_ERR_INVALID_ARG;
    if (B < 1 || T < 1 || d < 1 || ldx < d) return ADA_ERR_INVALID_ARG;
    if (dt != ADA_F32 && dt != ADA_BF16) return ADA_ERR_INVALID_ARG;
    if (dt != ctx->dt) return ADA_ERR_UNSUPPORTED;
    if (B > ctx->maxB || T > ctx->maxT || d > ctx->maxd) return ADA_ERR_WORKSPACE;
    const int64_t es = dt == ADA_F32 ? 4 : 2;
    if (!aligned16(X) || (ldx * es) % 16 != 0 || (d * es) % 16 != 0) return ADA_ERR_UNSUPPORTED;
    return ADA_OK;
}

inline bool tau_ok(double tau) { return tau > 0.0 && tau < 1.0; }  // also rejects NaN

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        cudaGetDevice(&prev);
        if (prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

bool use_tc(const ada_ctx* ctx, ada_dtype dt) {
    if (dt != ADA_BF16) return false;
    if (ctx->engine == ADA_ENGINE_FFMA) return false;
    return gram_tc_available();
}

// fp32 storage on the bf16 tensor cores through the three-term split
bool use_split(const ada_ctx* ctx, ada_dtype dt) {
    return dt == ADA_F32 && ctx->engine != ADA_ENGINE_FFMA && ctx->splitX != nullptr &&
           gram_tc_available();
}

// the pair-CTA form of the tensor-core kernel, or the one-CTA form?  full: full selection, else a cross-Gram
bool use_pair(const ada_ctx* ctx, int64_t B, int64_t T, int64_t d, ada_dtype dt, bool full) {
    if (ctx->engine == ADA_ENGINE_TCGEN05_PAIR) return true;
    if (ctx->engine != ADA_ENGINE_AUTO) return false;
    // Measured against the one-CTA kernel, whose narrow tiles occupy every SM where the pair kernel
    // has to split its few tiles along K: with the split the pair kernel is faster from 512 tokens
    // on (T = 1024, d = 4096: full selection 27.4 -> 24.0 us, step 34.8 -> 28.2; fp32, T = 700,
    // d = 1600: 55.8 -> 23.7, step 67.8 -> 30.3), where the contraction is too long to be split only from a few
    // thousand rows on (T = 700, d = 5120, when that was not split: 31.0 against 34.7 us).
    if (dt == ADA_F32) return d >= 256 && (d <= MAX_SPLIT_D_F32 || B * T >= 4096);
    if (d >= 2048) return B * T >= (d <= MAX_SPLIT_D ? 512 : 4096);
    // Shorter contractions: a step saves the launch that gathers and normalises (8 x 2048 x 768: 37 -> 29 us
    // per step; at d = 512 between 0.95 and 1.1 times as fast), a full selection is as fast at
    // d = 1024, gains above (T = 4096, d = 1536: 32.3 -> 30.0 us) and loses below (T = 4096, d = 768: 23.2
    // -> 24.8 us).
    return full ? d > 1024 && B * T >= 1024 : d >= 512;
}

// plane width of an fp32 row of d elements: whole 64-element K blocks
inline int64_t plane_len(int64_t d) { return (d + 63) / 64 * 64; }


#define CU(x)                                  \
    do {                                       \
        cudaError_t e__ = (x);                 \
        if (e__ != cudaSuccess) {              \
            cudaGetLastError(); /* reported by the status; the next launcher that asks must not find it */ \
            return ADA_ERR_CUDA;               \
        }                                      \
    } while (0)

}  // namespace

namespace ada {

// Which launches have to be cooperative: see launch_policy.h
namespace {
constexpr int kMaxSole = 64;
SoleStream g_sole[kMaxSole];
std::atomic<int> g_mps[kMaxSole];        // 0: not asked yet, 1: no, 2: yes (or unknown)

bool under_mps(int device) {
    int v = g_mps[device].load(std::memory_order_relaxed);
    if (v == 0) {
        int on = 0;
        if (cudaDeviceGetAttribute(&on, cudaDevAttrMpsEnabled, device) != cudaSuccess) { cudaGetLastError(); on = 1; }
        v = on != 0 ? 2 : 1;
        g_mps[device].store(v, std::memory_order_relaxed);
    }
    return v == 2;
}
}  // namespace

bool coop_begin(ada_ctx* ctx, cudaStream_t s) {
    if (!ctx->cooperative) return false;
    if (ctx->device < 0 || ctx->device >= kMaxSole) return true;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) { cudaGetLastError(); return true; }
    if (cap != cudaStreamCaptureStatusNone) return true;
    if (cudaStreamGetId(s, &id) != cudaSuccess) { cudaGetLastError(); return true; }
    return under_mps(ctx->device) || !g_sole[ctx->device].begin(id);
}

void coop_end(ada_ctx* ctx, bool coop) {
    if (!coop && ctx->cooperative) g_sole[ctx->device].end();
}

unsigned long long sole_mark(int device) {
    return device < 0 || device >= kMaxSole ? 0 : g_sole[device].mark();
}

void sole_idle(int device, bool all, cudaStream_t s, unsigned long long mark) {
    if (device < 0 || device >= kMaxSole) return;
    unsigned long long id = 0;
    if (!all && cudaStreamGetId(s, &id) != cudaSuccess) { cudaGetLastError(); return; }
    g_sole[device].idle(all, id, mark);
}

bool sole_holds(int device, cudaStream_t s) {
    unsigned long long id = 0;
    if (device < 0 || device >= kMaxSole) return false;
    if (cudaStreamGetId(s, &id) != cudaSuccess) { cudaGetLastError(); return false; }
    return g_sole[device].holds(id);
}

void prof_begin(ada_ctx* ctx, int kid, cudaStream_t s) {
    Profiler& pr = ctx->prof;
    if (!pr.on || pr.n >= Profiler::MAXREC) return;
    if (pr.n >= pr.created) {
        cudaEventCreate(&pr.ev0[pr.n]);
        cudaEventCreate(&pr.ev1[pr.n]);
        pr.created = pr.n + 1;
    }
    pr.kid[pr.n] = kid;
    cudaEventRecord(pr.ev0[pr.n], s);
}

void prof_end(ada_ctx* ctx, cudaStream_t s) {
    Profiler& pr = ctx->prof;
    if (!pr.on || pr.n >= Profiler::MAXREC) return;
    cudaEventRecord(pr.ev1[pr.n], s);
    ++pr.n;
}

}  // namespace ada

extern "C" {

const char* ada_status_string(ada_status s) {
    switch (s) {
        case ADA_OK: return "ADA_OK";
        case ADA_ERR_INVALID_ARG: return "ADA_ERR_INVALID_ARG";
        case ADA_ERR_UNSUPPORTED: return "ADA_ERR_UNSUPPORTED";
        case ADA_ERR_WORKSPACE: return "ADA_ERR_WORKSPACE";
        case ADA_ERR_CUDA: return "ADA_ERR_CUDA";
        case ADA_ERR_BAD_INDEX_SET: return "ADA_ERR_BAD_INDEX_SET";
        case ADA_ERR_NONFINITE: return "ADA_ERR_NONFINITE";
        case ADA_ERR_TIMEOUT: return "ADA_ERR_TIMEOUT";
        case ADA_ERR_BAD_TAU: return "ADA_ERR_BAD_TAU";
    }
    return "ADA_ERR_UNKNOWN";
}

uint64_t ada_gram_op_count(int cascade, int64_t T, int64_t d, int64_t r) {
    if (T < 0 || d < 0 || r < 0) return 0;
    const uint64_t t = (uint64_t)T, dd = (uint64_t)d, rr = (uint64_t)r;
    if (!cascade) return t * t * dd;
    if (r > T) return 0;
    return rr * rr * dd + (t - rr) * rr * dd;
}

ada_status ada_create(ada_ctx** out, int device, int64_t maxB, int64_t maxT, int64_t maxd,
                      ada_dtype dt) {
    if (out == nullptr) return ADA_ERR_INVALID_ARG;
    *out = nullptr;
    if (maxB < 1 || maxT < 1 || maxd < 1 || (dt != ADA_F32 && dt != ADA_BF16))
        return ADA_ERR_INVALID_ARG;
    // the compaction packs three per-sequence counts into 21-bit fields of one word
    if (maxT > ADA_MAX_T || maxB * maxT > (int64_t)1 << 30) return ADA_ERR_INVALID_ARG;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev)
        return ADA_ERR_CUDA;
    DeviceGuard guard(device);
    ada_ctx* ctx = new (std::nothrow) ada_ctx();
    if (ctx == nullptr) return ADA_ERR_CUDA;
    ctx->device = device;
    ctx->maxB = maxB; ctx->maxT = maxT; ctx->maxd = maxd;
    ctx->dt = dt;
    ctx->es = dt == ADA_F32 ? 4 : 2;
    ctx->engine = ADA_ENGINE_AUTO;
    ctx->stage = nullptr; ctx->stage_bytes = 0; ctx->host_stream = nullptr;
    ctx->host_event = nullptr; ctx->host_ready = nullptr; ctx->host_out = false;
    ctx->attn_ws = nullptr; ctx->attn_ws_bytes = 0;
    ctx->map_cache = nullptr;
    ctx->tc_attr_set = false;
    ctx->cooperative = true;
    ctx->dep_launch = true;
    ctx->tc2_attr_set = false;
    ctx->short_attr_set = false;
    ctx->tc2_pairs = 0;
    ctx->compact_min_rows = 8192;
    ctx->max_parts = MAX_PARTS;
    cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, device);

    const size_t n_tok = (size_t)maxB * (size_t)maxT;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
    // role, g_tok, g_rep are contiguous so that one memset clears them
    const size_t o_role = take(n_tok * 4), o_gtok = take(n_tok * 4), o_grep = take(n_tok * 4);
    const size_t o_ctr = take(32);
    const size_t o_near = take(n_tok * 8);
    const size_t o_inv = take(n_tok * 4), o_invr = take(n_tok * 4);
    const size_t o_reff = take((size_t)maxB * 4), o_stat = take(32);
    const size_t o_xrep = take(n_tok * (size_t)maxd * ctx->es + 1024);
    // bf16: the rows outside a large inherited set, copied out for the cross step (Algorithm 1 line 6)
    const size_t o_ntok = take(dt == ADA_BF16 ? n_tok * 4 : 0);
    const size_t o_grept = take(dt == ADA_BF16 ? n_tok * 4 : 0);      // (cleared together with the one before it)
    const size_t o_xnon = take(dt == ADA_BF16 ? n_tok * (size_t)maxd * 2 + 1024 : 0);
    const size_t split_bytes = dt == ADA_F32 ? n_tok * (size_t)plane_len(maxd) * 6 + 1024 : 0;
    const size_t o_sx = take(split_bytes), o_sr = take(split_bytes);
    // one 256-column fp32 accumulator per SM
    ctx->part_bytes = (size_t)ctx->sm_count * 128 * 256 * 4;
    const size_t o_part = take(ctx->part_bytes);
    if (cudaMalloc(&ctx->ws, off) != cudaSuccess) {
        cudaGetLastError();
        delete ctx;
        return ADA_ERR_CUDA;
    }
    ctx->role = reinterpret_cast<int32_t*>(ctx->ws + o_role);
    ctx->g_tok = reinterpret_cast<unsigned*>(ctx->ws + o_gtok);
    ctx->g_rep = reinterpret_cast<unsigned*>(ctx->ws + o_grep);
    ctx->g_rep_tok = dt == ADA_BF16 ? reinterpret_cast<unsigned*>(ctx->ws + o_grept) : nullptr;
    ctx->inv_norm = reinterpret_cast<float*>(ctx->ws + o_inv);
    ctx->inv_rep = reinterpret_cast<float*>(ctx->ws + o_invr);
    ctx->r_eff = reinterpret_cast<int32_t*>(ctx->ws + o_reff);
    ctx->status = reinterpret_cast<unsigned*>(ctx->ws + o_stat);
    ctx->tile_ctr = reinterpret_cast<unsigned*>(ctx->ws + o_ctr);
    ctx->near_key = reinterpret_cast<unsigned long long*>(ctx->ws + o_near);
    ctx->Xrep = ctx->ws + o_xrep;
    ctx->Xnon = dt == ADA_BF16 ? ctx->ws + o_xnon : nullptr;
    ctx->non_tok = dt == ADA_BF16 ? reinterpret_cast<int32_t*>(ctx->ws + o_ntok) : nullptr;
    ctx->splitX = split_bytes ? ctx->ws + o_sx : nullptr;
    ctx->splitR = split_bytes ? ctx->ws + o_sr : nullptr;
    ctx->part_buf = reinterpret_cast<unsigned*>(ctx->ws + o_part);
    // A stream and events for the *_host calls: made here so that a context's first such call costs no
    // more than its second.  The fills run on that stream, which waits for nobody, and are waited for: the
    // first call may come on any stream, and none of them is ordered behind a fill.
    if (cudaStreamCreateWithFlags(&ctx->host_stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->host_event, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->host_ready, cudaEventDisableTiming) != cudaSuccess ||
        cudaMemsetAsync(ctx->ws, 0, o_xrep, ctx->host_stream) != cudaSuccess ||
        cudaMemsetAsync(ctx->part_buf, 0xFF, ctx->part_bytes, ctx->host_stream) != cudaSuccess ||
        (dt == ADA_BF16 && cudaMemsetAsync(ctx->ws + o_ntok, 0, o_xnon - o_ntok, ctx->host_stream) != cudaSuccess) ||
        cudaStreamSynchronize(ctx->host_stream) != cudaSuccess) {
        cudaGetLastError();
        ada_destroy(ctx);
        return ADA_ERR_CUDA;
    }
    ctx->map_cache = new_map_cache();
    *out = ctx;
    return ADA_OK;
}

ada_status ada_destroy(ada_ctx* ctx) {
    if (ctx == nullptr) return ADA_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    const unsigned long long mark = sole_mark(ctx->device);
    if (cudaDeviceSynchronize() == cudaSuccess) sole_idle(ctx->device, true, nullptr, mark);
    for (int i = 0; i < ctx->prof.created; ++i) {
        cudaEventDestroy(ctx->prof.ev0[i]);
        cudaEventDestroy(ctx->prof.ev1[i]);
    }
    if (ctx->stage) cudaFree(ctx->stage);
    if (ctx->attn_ws) cudaFree(ctx->attn_ws);
    if (ctx->host_stream) cudaStreamDestroy(ctx->host_stream);
    if (ctx->host_event) cudaEventDestroy(ctx->host_event);
    if (ctx->host_ready) cudaEventDestroy(ctx->host_ready);
    cudaFree(ctx->ws);
    delete_map_cache(ctx->map_cache);
    delete ctx;
    return ADA_OK;
}

ada_status ada_set_engine(ada_ctx* ctx, ada_engine e) {
    if (ctx == nullptr) return ADA_ERR_INVALID_ARG;
    if (e != ADA_ENGINE_AUTO && e != ADA_ENGINE_FFMA && e != ADA_ENGINE_TCGEN05 &&
        e != ADA_ENGINE_TCGEN05_PAIR)
        return ADA_ERR_INVALID_ARG;
    if ((e == ADA_ENGINE_TCGEN05 || e == ADA_ENGINE_TCGEN05_PAIR) && !gram_tc_available())
        return ADA_ERR_UNSUPPORTED;
    ctx->engine = e;
    return ADA_OK;
}

ada_status ada_set_row_compaction(ada_ctx* ctx, int64_t min_rows) {
    if (ctx == nullptr || min_rows < 1) return ADA_ERR_INVALID_ARG;
    ctx->compact_min_rows = min_rows > 0x7fffffff ? 0x7fffffff : (int)min_rows;
    return ADA_OK;
}

ada_status ada_set_cooperative(ada_ctx* ctx, int on) {
    if (ctx == nullptr) return ADA_ERR_INVALID_ARG;
    ctx->cooperative = on != 0;
    return ADA_OK;
}

ada_status ada_set_dependent_launch(ada_ctx* ctx, int on) {
    if (ctx == nullptr) return ADA_ERR_INVALID_ARG;
    ctx->dep_launch = on != 0;
    return ADA_OK;
}

ada_status ada_normalize(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                         int64_t ldx, ada_dtype dt, void* Xhat, float* inv_norm,
                         const int32_t* rep_idx, const int32_t* rep_cnt, void* Xrep,
                         void* stream) {
    ada_status st = check_common(ctx, X, B, T, d, ldx, dt);
    if (st != ADA_OK) return st;
    const bool gather = rep_idx != nullptr || rep_cnt != nullptr || Xrep != nullptr;
    if (gather && (rep_idx == nullptr || rep_cnt == nullptr || Xrep == nullptr))
        return ADA_ERR_INVALID_ARG;
    if ((Xhat != nullptr && !aligned16(Xhat)) || (Xrep != nullptr && !aligned16(Xrep)))
        return ADA_ERR_UNSUPPORTED;
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CU(launch_norm_gather(ctx, X, (int)B, (int)T, (int)d, ldx, T * ldx, dt, inv_norm, Xhat,
                          gather ? rep_idx : nullptr, rep_cnt, nullptr, nullptr, Xrep, ctx->inv_rep,
                          s));
    return ADA_OK;
}

// fp32 rows of X as bf16 planes in ctx->splitX (and their inverse norms)
static SplitJob split_job(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d, int64_t ldx, int64_t xb) {
    SplitJob j;
    memset(&j, 0, sizeof(j));
    j.X = static_cast<const float*>(X); j.ldx = ldx; j.xb = xb;
    j.T = (int)T; j.B = (int)B; j.d = (int)d; j.dpad = (int)plane_len(d);
    j.XP = static_cast<__nv_bfloat16*>(ctx->splitX);
    j.inv_norm = ctx->inv_norm;
    j.role = ctx->role; j.r_eff = ctx->r_eff;
    j.RP = static_cast<__nv_bfloat16*>(ctx->splitR);
    j.inv_rep = ctx->inv_rep;
    return j;
}

// Algorithm 1 lines 1-2 on bf16 rows, inside a pair-kernel launch
static GatherJob gather_job(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d, int64_t ldx, int64_t xb,
                            const int32_t* rep_in, const int32_t* rep_in_cnt) {
    GatherJob j;
    memset(&j, 0, sizeof(j));
    j.X = X; j.ldx = ldx; j.xb = xb;
    j.rep_in = rep_in; j.rep_in_cnt = rep_in_cnt;
    j.role = ctx->role; j.r_eff = ctx->r_eff; j.Xrep = ctx->Xrep; j.inv_rep = ctx->inv_rep;
    j.T = (int)T; j.d = (int)d; j.B = (int)B;
    j.Xnon = ctx->Xnon; j.non_tok = ctx->non_tok; j.inv_norm = ctx->inv_norm;
    j.compact_min_rows = ctx->compact_min_rows;
    return j;
}

// operands of `p` are rows of planes; the one-CTA kernel walks the six cross terms as one contraction
static void use_planes(GramProblem& p, const void* A, const void* Bm, int64_t T, int64_t d, bool pair) {
    const int64_t pl = plane_len(d);
    p.A = A; p.Bm = Bm;
    p.lda = p.ldb = 3 * pl;
    p.a_batch = p.b_batch = T * 3 * pl;
    p.planes = (int)pl;
    p.d = (int)(pair ? d : 6 * pl);
}

// Definition 1 for B independent problems; row (b, t) of X starts at element b * xb + t * ldx
static ada_status select_full_impl(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                                   int64_t ldx, int64_t xb, ada_dtype dt, double tau,
                                   int32_t* rep_idx, int32_t* rep_cnt, float* gamma, void* stream) {
    if (rep_idx == nullptr || rep_cnt == nullptr || !tau_ok(tau)) return ADA_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const float thr = (float)(1.0 - tau * tau);

    // the gamma scratch is zero on entry (workspace invariant kept by the compaction kernels)
    const bool split = use_split(ctx, dt), tc = use_tc(ctx, dt);
    const bool pair = (split || tc) && use_pair(ctx, B, T, d, dt, true);
    // bf16: the pair kernel (and the one-CTA kernel, for many rows of a long contraction) computes
    // the row norms itself, hidden behind the MMAs
    const bool fuse = tc && (pair || (d >= 2048 && B * T >= 4096 && xb == T * ldx));
    NormJob nj;
    nj.X = X; nj.ldx = ldx; nj.n_rows = B * T; nj.d = (int)d; nj.inv_norm = ctx->inv_norm;
    nj.batch = xb; nj.rows_per_seq = (int)T;
    SplitJob sj = split_job(ctx, X, B, T, d, ldx, xb);
    GramProblem p;
    memset(&p, 0, sizeof(p));
    p.A = X; p.Bm = X;
    p.lda = ldx; p.ldb = ldx;
    p.a_batch = xb; p.b_batch = xb;
    p.inv_a = ctx->inv_norm; p.inv_b = ctx->inv_norm;
    p.out = ctx->g_tok;
    p.n_dev = nullptr; p.n_host = (int)T;
    p.rows = (int)T; p.cap = (int)T; p.d = (int)d; p.B = (int)B;
    p.tri = 1;
    p.wait_norm_a = p.wait_norm_b = fuse ? 1 : 0;
    if (split) {   // 1/||x|| and the bf16 planes of X, inside the pair kernel's launch or before the other's
        use_planes(p, ctx->splitX, ctx->splitX, T, d, pair);
        if (!pair) CU(launch_split(ctx, sj, s));
    } else if (!fuse) {
        CU(launch_norm_gather(ctx, X, (int)B, (int)T, (int)d, ldx, xb, dt, ctx->inv_norm, nullptr,
                              nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, s));
    }
    if (pair) CU(launch_gram_tc2(ctx, &p, nullptr, fuse ? &nj : nullptr, nullptr, split ? &sj : nullptr, s));
    else if (split || tc) CU(launch_gram_tc(ctx, &p, nullptr, fuse ? &nj : nullptr, s));
    else CU(launch_gram_ffma(ctx, p, dt, s));
    CU(launch_compact_full(ctx, (int)B, (int)T, thr, rep_idx, rep_cnt, gamma, s));
    return ADA_OK;
}

ada_status ada_select_full(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                           int64_t ldx, ada_dtype dt, double tau, int32_t* rep_idx,
                           int32_t* rep_cnt, float* gamma, void* stream) {
    ada_status st = check_common(ctx, X, B, T, d, ldx, dt);
    if (st != ADA_OK) return st;
    return select_full_impl(ctx, X, B, T, d, ldx, T * ldx, dt, tau, rep_idx, rep_cnt, gamma, stream);
}

// heads interleaved inside each token's row: head j of token t starts at t * ldx + j * d_h
static ada_status check_heads(ada_ctx* ctx, const void* X, int64_t T, int64_t h, int64_t d_h,
                              int64_t ldx, ada_dtype dt) {
    ada_status st = check_common(ctx, X, h, T, d_h, ldx, dt);
    if (st != ADA_OK) return st;
    return ldx < h * d_h ? ADA_ERR_INVALID_ARG : ADA_OK;
}

ada_status ada_select_full_heads(ada_ctx* ctx, const void* X, int64_t T, int64_t h, int64_t d_h,
                                 int64_t ldx, ada_dtype dt, double tau, int32_t* rep_idx,
                                 int32_t* rep_cnt, float* gamma, void* stream) {
    ada_status st = check_heads(ctx, X, T, h, d_h, ldx, dt);
    if (st != ADA_OK) return st;
    return select_full_impl(ctx, X, h, T, d_h, ldx, d_h, dt, tau, rep_idx, rep_cnt, gamma, stream);
}

// Algorithm 1 for B independent problems; row (b, t) of X starts at element b * xb + t * ldx
static ada_status cascade_impl(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                               int64_t ldx, int64_t xb, ada_dtype dt, double tau,
                               const int32_t* rep_in, const int32_t* rep_in_cnt, int32_t* rep_out,
                               int32_t* rep_out_cnt, int32_t* add_idx, int32_t* add_cnt,
                               int32_t* rem_idx, int32_t* rem_cnt, float* gamma_rep,
                               float* gamma_cross, uint32_t flags, void* stream,
                               const TauUpdate* tu = nullptr) {
    if (rep_in == nullptr || rep_in_cnt == nullptr || rep_out == nullptr ||
        rep_out_cnt == nullptr || add_idx == nullptr || add_cnt == nullptr ||
        rem_idx == nullptr || rem_cnt == nullptr || !tau_ok(tau))
        return ADA_ERR_INVALID_ARG;
    if (rep_out == rep_in || (flags & ~ADA_CROSS_CAUSAL) != 0) return ADA_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const float thr = (float)(1.0 - tau * tau);
    TauUpdate tau_upd;
    memset(&tau_upd, 0, sizeof(tau_upd));
    if (tu != nullptr) tau_upd = *tu;

    // one attention head per sequence, or rows as short as that: the whole step in one launch
    if (ctx->engine == ADA_ENGINE_AUTO && tu == nullptr && use_tc(ctx, dt)) {
        const int ctas = step_short_ctas(ctx, B, T, d);
        if (ctas > 0) {
            CU(launch_step_short(ctx, ctas, X, (int)B, (int)T, (int)d, ldx, xb, thr, rep_in, rep_in_cnt, rep_out,
                                 rep_out_cnt, add_idx, add_cnt, rem_idx, rem_cnt, gamma_rep, gamma_cross,
                                 (flags & ADA_CROSS_CAUSAL) ? 1 : 0, s));
            return ADA_OK;
        }
    }

    // role map, gamma scratch and dependency counters are zero on entry (workspace invariant
    // kept by the compaction kernels).
    const bool split = use_split(ctx, dt);
    const bool fuse = use_tc(ctx, dt) || split;
    // On the pair kernel ONE Gram launch does lines 1-8.  Its spare warps validate the
    // inherited list, scatter the role map and gather the rows (lines 1-2; fp32: and make the bf16
    // planes); the r x r tiles (lines 3-5) and the cross tiles (lines 6-8) follow; for bf16 the
    // norms of X are made beside them and the row's own factor 1/||x_t|| is left to the
    // compaction.
    const bool inl = fuse && use_pair(ctx, B, T, d, dt, false);
    // otherwise lines 1-2 are a launch of their own: inverse norms of all rows, inherited list
    // validated, scattered into the role map and its rows gathered into Xrep; for long K the
    // one-CTA tensor-core launch computes line 1's row norms itself
    const bool fuse_norm = !inl && !split && fuse && d >= 2048 && B * T >= 4096 && xb == T * ldx;
    SplitJob sj = split_job(ctx, X, B, T, d, ldx, xb);
    sj.rep_in = rep_in; sj.rep_in_cnt = rep_in_cnt;
    if (split && !inl) CU(launch_split(ctx, sj, s));
    else if (!inl)
        CU(launch_norm_gather(ctx, X, (int)B, (int)T, (int)d, ldx, xb, dt, fuse_norm ? nullptr : ctx->inv_norm,
                              nullptr, rep_in, rep_in_cnt, ctx->role, ctx->r_eff, ctx->Xrep,
                              ctx->inv_rep, s));
    NormJob nj;
    nj.X = X; nj.ldx = ldx; nj.n_rows = B * T; nj.d = (int)d; nj.inv_norm = ctx->inv_norm;
    nj.batch = 0; nj.rows_per_seq = 0;
    GatherJob gj = gather_job(ctx, X, B, T, d, ldx, xb, rep_in, rep_in_cnt);
    // lines 3-4: r x r Gram among inherited reps, max over earlier ones
    GramProblem p;
    memset(&p, 0, sizeof(p));
    p.A = ctx->Xrep; p.Bm = ctx->Xrep;
    p.lda = d; p.ldb = d;
    p.a_batch = T * d; p.b_batch = T * d;
    p.inv_a = ctx->inv_rep; p.inv_b = ctx->inv_rep;
    p.out = ctx->g_rep;
    // (by token too: the compaction then reads everything of a token at once instead of by its position)
    const bool by_tok = inl && !split;
    p.out_tok = by_tok ? ctx->g_rep_tok : nullptr;
    p.col_token = rep_in;
    p.n_dev = inl ? rep_in_cnt : ctx->r_eff; p.n_host = 0;
    p.n_clamp = inl ? 1 : 0;
    p.rows = (int)T; p.cap = (int)T; p.d = (int)d; p.B = (int)B;
    p.tri = 1;
    if (!fuse) CU(launch_gram_ffma(ctx, p, dt, s));
    // lines 6-8: cross-Gram of all rows against the valid inherited reps
    GramProblem q;
    memset(&q, 0, sizeof(q));
    q.A = X; q.Bm = ctx->Xrep;
    q.lda = ldx; q.ldb = d;
    q.a_batch = xb; q.b_batch = T * d;
    q.inv_a = ctx->inv_norm; q.inv_b = ctx->inv_rep;
    q.out = ctx->g_tok;
    q.n_dev = p.n_dev; q.n_host = 0;
    q.n_clamp = p.n_clamp;
    q.rows = (int)T; q.cap = (int)T; q.d = (int)d; q.B = (int)B;
    q.tri = 0;
    q.col_gate = ctx->g_rep;
    q.thr_bits = 0;
    memcpy(&q.thr_bits, &thr, 4);
    q.tau_seq = tau_upd.tau_state;
    q.col_token = rep_in;
    q.row_role = ctx->role;
    q.causal = (flags & ADA_CROSS_CAUSAL) ? 1 : 0;
    q.wait_norm_a = fuse_norm ? 1 : 0;
    if (inl && !split) {
        q.defer_row = 1;
        q.inv_out = ctx->inv_norm;
        q.hb_rows = gram_tc2_hb_rows(ctx, (int)B, (int)T);
        if (q.hb_rows == 0) return ADA_ERR_CUDA;
    }
    if (split) {
        use_planes(p, ctx->splitR, ctx->splitR, T, d, inl);
        use_planes(q, ctx->splitX, ctx->splitR, T, d, inl);
    }
    if (inl) CU(launch_gram_tc2(ctx, &p, &q, nullptr, split ? nullptr : &gj, split ? &sj : nullptr, s));
    else if (fuse) CU(launch_gram_tc(ctx, &p, &q, fuse_norm ? &nj : nullptr, s));
    else CU(launch_gram_ffma(ctx, q, dt, s));
    // lines 5, 9, 10-11
    CU(launch_compact_cascade(ctx, (int)B, (int)T, thr, rep_out, rep_out_cnt, add_idx, add_cnt,
                              rem_idx, rem_cnt, gamma_rep, gamma_cross, tau_upd, q.defer_row != 0, by_tok, s));
    return ADA_OK;
}

ada_status ada_cascade_step_adaptive(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                                     int64_t ldx, ada_dtype dt, double* tau_state,
                                     const ada_tau_policy* policy, const int32_t* rep_in,
                                     const int32_t* rep_in_cnt, int32_t* rep_out,
                                     int32_t* rep_out_cnt, int32_t* add_idx, int32_t* add_cnt,
                                     int32_t* rem_idx, int32_t* rem_cnt, float* gamma_rep,
                                     float* gamma_cross, float* turnover, uint32_t flags,
                                     void* stream) {
    ada_status st = check_common(ctx, X, B, T, d, ldx, dt);
    if (st != ADA_OK) return st;
    if (tau_state == nullptr) return ADA_ERR_INVALID_ARG;
    TauUpdate tu;
    memset(&tu, 0, sizeof(tu));
    tu.tau_state = tau_state;
    tu.turnover = turnover;
    if (policy != nullptr) {
        // also rejects NaN in any field
        if (!(policy->gain >= 0.0) || !(policy->target_turnover >= 0.0) || !(policy->tau_min > 0.0) ||
            !(policy->tau_max < 1.0) || !(policy->tau_min <= policy->tau_max))
            return ADA_ERR_INVALID_ARG;
        tu.update = 1;
        tu.target = policy->target_turnover; tu.gain = policy->gain;
        tu.tau_min = policy->tau_min; tu.tau_max = policy->tau_max;
    }
    // the host-side tau of the fixed-threshold call is not used; 0.5 passes its range check
    return cascade_impl(ctx, X, B, T, d, ldx, T * ldx, dt, 0.5, rep_in, rep_in_cnt, rep_out,
                        rep_out_cnt, add_idx, add_cnt, rem_idx, rem_cnt, gamma_rep, gamma_cross,
                        flags, stream, &tu);
}

ada_status ada_cascade_step(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                            int64_t ldx, ada_dtype dt, double tau, const int32_t* rep_in,
                            const int32_t* rep_in_cnt, int32_t* rep_out, int32_t* rep_out_cnt,
                            int32_t* add_idx, int32_t* add_cnt, int32_t* rem_idx,
                            int32_t* rem_cnt, float* gamma_rep, float* gamma_cross,
                            uint32_t flags, void* stream) {
    ada_status st = check_common(ctx, X, B, T, d, ldx, dt);
    if (st != ADA_OK) return st;
    return cascade_impl(ctx, X, B, T, d, ldx, T * ldx, dt, tau, rep_in, rep_in_cnt, rep_out,
                        rep_out_cnt, add_idx, add_cnt, rem_idx, rem_cnt, gamma_rep, gamma_cross,
                        flags, stream);
}

ada_status ada_cascade_step_heads(ada_ctx* ctx, const void* X, int64_t T, int64_t h, int64_t d_h,
                                  int64_t ldx, ada_dtype dt, double tau, const int32_t* rep_in,
                                  const int32_t* rep_in_cnt, int32_t* rep_out,
                                  int32_t* rep_out_cnt, int32_t* add_idx, int32_t* add_cnt,
                                  int32_t* rem_idx, int32_t* rem_cnt, float* gamma_rep,
                                  float* gamma_cross, uint32_t flags, void* stream) {
    ada_status st = check_heads(ctx, X, T, h, d_h, ldx, dt);
    if (st != ADA_OK) return st;
    return cascade_impl(ctx, X, h, T, d_h, ldx, d_h, dt, tau, rep_in, rep_in_cnt, rep_out,
                        rep_out_cnt, add_idx, add_cnt, rem_idx, rem_cnt, gamma_rep, gamma_cross,
                        flags, stream);
}

ada_status ada_nearest_rep(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                           int64_t ldx, ada_dtype dt, const int32_t* rep_idx,
                           const int32_t* rep_cnt, int32_t* nearest_idx, float* nearest_gamma,
                           void* stream) {
    ada_status st = check_common(ctx, X, B, T, d, ldx, dt);
    if (st != ADA_OK) return st;
    if (rep_idx == nullptr || rep_cnt == nullptr || nearest_idx == nullptr) return ADA_ERR_INVALID_ARG;
    const bool split = dt == ADA_F32;
    if (!gram_tc_available() || (split && ctx->splitX == nullptr)) return ADA_ERR_UNSUPPORTED;
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool pair = use_pair(ctx, B, T, d, dt, false);
    // role map and keys are zero on entry (workspace invariant); the finish kernel clears them
    SplitJob sj = split_job(ctx, X, B, T, d, ldx, T * ldx);
    sj.rep_in = rep_idx; sj.rep_in_cnt = rep_cnt;
    GatherJob gj = gather_job(ctx, X, B, T, d, ldx, T * ldx, rep_idx, rep_cnt);
    gj.Xnon = nullptr;                // every row is wanted
    if (!pair) {
        if (split) CU(launch_split(ctx, sj, s));
        else
            CU(launch_norm_gather(ctx, X, (int)B, (int)T, (int)d, ldx, T * ldx, dt, ctx->inv_norm, nullptr, rep_idx,
                                  rep_cnt, ctx->role, ctx->r_eff, ctx->Xrep, ctx->inv_rep, s));
    }
    GramProblem q;
    memset(&q, 0, sizeof(q));
    q.A = X; q.Bm = ctx->Xrep;
    q.lda = ldx; q.ldb = d;
    q.a_batch = T * ldx; q.b_batch = T * d;
    q.inv_a = ctx->inv_norm; q.inv_b = ctx->inv_rep;
    q.out = ctx->g_tok;
    q.out_arg = ctx->near_key;
    q.n_dev = pair ? rep_cnt : ctx->r_eff; q.n_host = 0;
    q.n_clamp = pair ? 1 : 0;
    q.rows = (int)T; q.cap = (int)T; q.d = (int)d; q.B = (int)B;
    q.tri = 0;
    q.col_gate = ctx->g_rep;          // all zero: every column passes the gate
    q.thr_bits = 0xFFFFFFFFu;
    q.col_token = rep_idx;
    q.row_role = ctx->role;           // representatives are resolved by the finish kernel
    q.causal = 0;
    q.defer_row = 1;                  // which applies the row's own factor too
    if (split) use_planes(q, ctx->splitX, ctx->splitR, T, d, pair);
    else if (pair) {
        q.inv_out = ctx->inv_norm;
        q.hb_rows = gram_tc2_hb_rows(ctx, (int)B, (int)T);
        if (q.hb_rows == 0) return ADA_ERR_CUDA;
    }
    if (pair) CU(launch_gram_tc2(ctx, nullptr, &q, nullptr, split ? nullptr : &gj, split ? &sj : nullptr, s));
    else CU(launch_gram_tc(ctx, nullptr, &q, nullptr, s));
    CU(launch_nearest_finish(ctx, (int)B, (int)T, rep_idx, nearest_idx, nearest_gamma, s));
    return ADA_OK;
}

ada_status ada_attention_reps(ada_ctx* ctx, const void* Q, const void* K, const void* V, int64_t T,
                              int64_t h, int64_t d_h, int64_t ld, ada_dtype dt, const int32_t* rep_idx,
                              const int32_t* rep_cnt, const int32_t* nearest_idx, float* out,
                              int64_t ldo, uint32_t flags, void* stream) {
    if (ctx == nullptr || Q == nullptr || K == nullptr || V == nullptr || rep_idx == nullptr ||
        rep_cnt == nullptr || out == nullptr)
        return ADA_ERR_INVALID_ARG;
    if (T < 1 || h < 1 || d_h < 1 || ld < h * d_h || ldo < h * d_h || (flags & ~ADA_ATTN_CAUSAL) != 0)
        return ADA_ERR_INVALID_ARG;
    if (dt != ADA_F32 && dt != ADA_BF16) return ADA_ERR_INVALID_ARG;
    // bf16 operands on the tensor cores; head widths the two contractions' tiles cover
    if (dt != ADA_BF16 || ctx->dt != ADA_BF16 || d_h % 16 != 0 || d_h > 128 || !gram_tc_available())
        return ADA_ERR_UNSUPPORTED;
    if (T > ctx->maxT || h * d_h > ctx->maxd) return ADA_ERR_WORKSPACE;
    if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(out) || (ld * 2) % 16 != 0 ||
        (ldo * 4) % 16 != 0)
        return ADA_ERR_UNSUPPORTED;
    DeviceGuard guard(ctx->device);
    CU(launch_attention_reps(ctx, Q, K, V, (int)T, (int)h, (int)d_h, ld, rep_idx, rep_cnt, nearest_idx, out,
                             ldo, (flags & ADA_ATTN_CAUSAL) ? 1 : 0, static_cast<cudaStream_t>(stream)));
    return ADA_OK;
}

ada_status ada_device_status(ada_ctx* ctx, void* stream, int64_t* n_zero_norm_rows) {
    if (ctx == nullptr) return ADA_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned h[8];
    const unsigned long long mark = sole_mark(ctx->device);
    CU(cudaMemcpyAsync(h, ctx->status, sizeof(h), cudaMemcpyDeviceToHost, s));
    CU(cudaMemsetAsync(ctx->status, 0, sizeof(h), s));
    CU(cudaStreamSynchronize(s));
    sole_idle(ctx->device, false, s, mark);
    if (n_zero_norm_rows != nullptr) *n_zero_norm_rows = (int64_t)h[1];
    if (h[0] != 0) {
        // a faulted call may have left scratch behind: restore the workspace invariants
        CU(cudaMemsetAsync(ctx->role, 0, (size_t)((char*)ctx->inv_norm - (char*)ctx->role), s));
        CU(cudaMemsetAsync(ctx->part_buf, 0xFF, ctx->part_bytes, s));
        if (ctx->g_rep_tok != nullptr) CU(cudaMemsetAsync(ctx->g_rep_tok, 0, (size_t)ctx->maxB * ctx->maxT * 4, s));
        CU(cudaStreamSynchronize(s));
    }
    if (h[0] & ST_TIMEOUT) return ADA_ERR_TIMEOUT;
    if (h[0] & (ST_BAD_INDEX | ST_BAD_COUNT)) return ADA_ERR_BAD_INDEX_SET;
    if (h[0] & ST_NONFINITE) return ADA_ERR_NONFINITE;
    if (h[0] & ST_BAD_TAU) return ADA_ERR_BAD_TAU;
    return ADA_OK;
}

// ---------------------------------------------------------------------------
// host-buffer entry points
// ---------------------------------------------------------------------------
static ada_status ensure_stage(ada_ctx* ctx) {
    if (ctx->stage != nullptr) return ADA_OK;
    const size_t n_tok = (size_t)ctx->maxB * ctx->maxT;
    // X | 5 index lists | 2 gamma arrays | 4 count arrays
    const size_t bytes = align_up(n_tok * ctx->maxd * ctx->es, 256) + 7 * align_up(n_tok * 4, 256) +
                         4 * align_up((size_t)ctx->maxB * 4, 256);
    if (cudaMalloc(&ctx->stage, bytes) != cudaSuccess) {
        cudaGetLastError();
        return ADA_ERR_CUDA;
    }
    ctx->stage_bytes = bytes;
    return ADA_OK;
}

struct Stage {
    char* X;
    int32_t *l0, *l1, *l2, *l3;
    float *g0, *g1;
    int32_t *c0, *c1, *c2, *c3;
};

static Stage carve(ada_ctx* ctx) {
    const size_t n_tok = (size_t)ctx->maxB * ctx->maxT;
    const size_t lx = align_up(n_tok * ctx->maxd * ctx->es, 256), ll = align_up(n_tok * 4, 256),
                 lc = align_up((size_t)ctx->maxB * 4, 256);
    Stage st;
    char* p = ctx->stage;
    st.X = p; p += lx;
    st.l0 = (int32_t*)p; p += ll;
    st.l1 = (int32_t*)p; p += ll;
    st.l2 = (int32_t*)p; p += ll;
    st.l3 = (int32_t*)p; p += ll;
    st.g0 = (float*)p; p += ll;
    st.g1 = (float*)p; p += ll;
    p += ll;
    st.c0 = (int32_t*)p; p += lc;
    st.c1 = (int32_t*)p; p += lc;
    st.c2 = (int32_t*)p; p += lc;
    st.c3 = (int32_t*)p;
    return st;
}

// Outputs in pinned host memory are written by the compaction itself, through their device address: the
// call is bound by copying the activations in (16.8 MB at 50 GB/s), and eight small copies back, one
// after the other, added 25 us to it.  Anything else goes through the staging buffers.
struct HostOut {
    void* host;
    void* dev;        // where the kernels write
    size_t bytes;     // copied back afterwards; 0: nothing to copy
};
// Device address of a host range that kernels may store 4-byte words to, or NULL: pinned from its first to its
// last byte (part of a buffer may be registered), at consecutive device addresses, not read-only for the
// device, and aligned.  A copy takes, or refuses, what a store would fault on.
static void* mapped(void* host, size_t bytes) {
    cudaPointerAttributes at, end;
    unsigned flags = 0;
    if (reinterpret_cast<uintptr_t>(host) % 4 != 0) return nullptr;
    if (cudaPointerGetAttributes(&at, host) != cudaSuccess ||
        cudaPointerGetAttributes(&end, static_cast<char*>(host) + bytes - 1) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (at.type != cudaMemoryTypeHost || end.type != cudaMemoryTypeHost || at.devicePointer == nullptr ||
        static_cast<char*>(end.devicePointer) - static_cast<char*>(at.devicePointer) != (ptrdiff_t)(bytes - 1))
        return nullptr;
    if (cudaHostGetFlags(&flags, host) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return (flags & cudaHostRegisterReadOnly) != 0 ? nullptr : at.devicePointer;
}
// the staging buffers become the outputs' own memory where every output is mapped, and none overlaps
// another (copied back one after the other, the last one stays; written by kernels, a mixture would)
static void choose_outputs(ada_ctx* ctx, HostOut* out, int n) {
    void* m[8];
    for (int i = 0; i < n; ++i) {
        m[i] = nullptr;
        if (out[i].host == nullptr) continue;
        const uintptr_t lo = reinterpret_cast<uintptr_t>(out[i].host);
        for (int j = 0; j < i; ++j) {
            const uintptr_t other = reinterpret_cast<uintptr_t>(out[j].host);
            if (other != 0 && lo < other + out[j].bytes && other < lo + out[i].bytes) return;
        }
        m[i] = mapped(out[i].host, out[i].bytes);
        if (m[i] == nullptr) return;
    }
    for (int i = 0; i < n; ++i) { out[i].dev = m[i]; out[i].bytes = 0; }
    ctx->host_out = true;
}
static ada_status copy_back(HostOut* out, int n, cudaStream_t s) {
    for (int i = 0; i < n; ++i)
        if (out[i].host != nullptr && out[i].bytes > 0)
            CU(cudaMemcpyAsync(out[i].host, out[i].dev, out[i].bytes, cudaMemcpyDeviceToHost, s));
    CU(cudaStreamSynchronize(s));
    return ADA_OK;
}

ada_status ada_select_full_host(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                                ada_dtype dt, double tau, int32_t* rep_idx, int32_t* rep_cnt,
                                float* gamma, void* stream) {
    if (ctx == nullptr || X == nullptr || rep_idx == nullptr || rep_cnt == nullptr)
        return ADA_ERR_INVALID_ARG;
    if (B < 1 || T < 1 || d < 1) return ADA_ERR_INVALID_ARG;
    if (dt != ADA_F32 && dt != ADA_BF16) return ADA_ERR_INVALID_ARG;
    // before anything is copied: the copies below are sized by the context's element type
    if (dt != ctx->dt || (d * ctx->es) % 16 != 0) return ADA_ERR_UNSUPPORTED;
    if (B > ctx->maxB || T > ctx->maxT || d > ctx->maxd) return ADA_ERR_WORKSPACE;
    DeviceGuard guard(ctx->device);
    ada_status st = ensure_stage(ctx);
    if (st != ADA_OK) return st;
    Stage sg = carve(ctx);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t n_tok = (size_t)B * T;
    CU(cudaMemcpyAsync(sg.X, X, n_tok * d * ctx->es, cudaMemcpyHostToDevice, s));
    HostOut out[3] = {{rep_idx, sg.l0, n_tok * 4}, {rep_cnt, sg.c0, (size_t)B * 4}, {gamma, sg.g0, n_tok * 4}};
    choose_outputs(ctx, out, 3);
    st = ada_select_full(ctx, sg.X, B, T, d, d, dt, tau, (int32_t*)out[0].dev, (int32_t*)out[1].dev,
                         gamma ? (float*)out[2].dev : nullptr, s);
    ctx->host_out = false;
    return st != ADA_OK ? st : copy_back(out, 3, s);
}

ada_status ada_cascade_step_host(ada_ctx* ctx, const void* X, int64_t B, int64_t T, int64_t d,
                                 ada_dtype dt, double tau, const int32_t* rep_in,
                                 const int32_t* rep_in_cnt, int32_t* rep_out,
                                 int32_t* rep_out_cnt, int32_t* add_idx, int32_t* add_cnt,
                                 int32_t* rem_idx, int32_t* rem_cnt, float* gamma_rep,
                                 float* gamma_cross, uint32_t flags, void* stream) {
    if (ctx == nullptr || X == nullptr || rep_in == nullptr || rep_in_cnt == nullptr ||
        rep_out == nullptr || rep_out_cnt == nullptr || add_idx == nullptr ||
        add_cnt == nullptr || rem_idx == nullptr || rem_cnt == nullptr)
        return ADA_ERR_INVALID_ARG;
    if (B < 1 || T < 1 || d < 1) return ADA_ERR_INVALID_ARG;
    if (dt != ADA_F32 && dt != ADA_BF16) return ADA_ERR_INVALID_ARG;
    // before anything is copied: the copies below are sized by the context's element type
    if (dt != ctx->dt || (d * ctx->es) % 16 != 0) return ADA_ERR_UNSUPPORTED;
    if (B > ctx->maxB || T > ctx->maxT || d > ctx->maxd) return ADA_ERR_WORKSPACE;
    DeviceGuard guard(ctx->device);
    ada_status st = ensure_stage(ctx);
    if (st != ADA_OK) return st;
    Stage sg = carve(ctx);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t n_tok = (size_t)B * T;
    // the inherited lists travel beside the activations, on a stream of their own that joins the caller's
    // before and after: work queued on `stream` ahead of the call may still be filling them
    CU(cudaEventRecord(ctx->host_ready, s));
    CU(cudaStreamWaitEvent(ctx->host_stream, ctx->host_ready, 0));
    CU(cudaMemcpyAsync(sg.X, X, n_tok * d * ctx->es, cudaMemcpyHostToDevice, s));
    CU(cudaMemcpyAsync(sg.l0, rep_in, n_tok * 4, cudaMemcpyHostToDevice, ctx->host_stream));
    CU(cudaMemcpyAsync(sg.c0, rep_in_cnt, (size_t)B * 4, cudaMemcpyHostToDevice, ctx->host_stream));
    CU(cudaEventRecord(ctx->host_event, ctx->host_stream));
    CU(cudaStreamWaitEvent(s, ctx->host_event, 0));
    HostOut out[8] = {{rep_out, sg.l1, n_tok * 4}, {add_idx, sg.l2, n_tok * 4}, {rem_idx, sg.l3, n_tok * 4},
                      {rep_out_cnt, sg.c1, (size_t)B * 4}, {add_cnt, sg.c2, (size_t)B * 4},
                      {rem_cnt, sg.c3, (size_t)B * 4},
                      {gamma_rep, sg.g0, n_tok * 4}, {gamma_cross, sg.g1, n_tok * 4}};
    choose_outputs(ctx, out, 8);
    st = ada_cascade_step(ctx, sg.X, B, T, d, d, dt, tau, sg.l0, sg.c0, (int32_t*)out[0].dev, (int32_t*)out[3].dev,
                          (int32_t*)out[1].dev, (int32_t*)out[4].dev, (int32_t*)out[2].dev, (int32_t*)out[5].dev,
                          gamma_rep ? (float*)out[6].dev : nullptr, gamma_cross ? (float*)out[7].dev : nullptr, flags, s);
    ctx->host_out = false;
    return st != ADA_OK ? st : copy_back(out, 8, s);
}

ada_status ada_selftest_wait_timeout(ada_ctx* ctx, int limit_ms, void* stream) {
    if (ctx == nullptr || limit_ms < 1 || limit_ms > 2000) return ADA_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    CU(launch_selftest_wait(ctx, limit_ms, static_cast<cudaStream_t>(stream)));
    return ADA_OK;
}

int ada_selftest_launches_alone(int device, void* stream) {
    DeviceGuard guard(device);
    return sole_holds(device, static_cast<cudaStream_t>(stream)) ? 1 : 0;
}

ada_status ada_profile_enable(ada_ctx* ctx, int on) {
    if (ctx == nullptr) return ADA_ERR_INVALID_ARG;
    ctx->prof.on = on != 0;
    ctx->prof.n = 0;
    return ADA_OK;
}

int ada_profile_read(ada_ctx* ctx, const char** names, int64_t* launches, double* total_ms,
                     int cap) {
    if (ctx == nullptr) return 0;
    DeviceGuard guard(ctx->device);
    Profiler& pr = ctx->prof;
    int64_t cnt[K_COUNT] = {0};
    double ms[K_COUNT] = {0};
    for (int i = 0; i < pr.n; ++i) {
        cudaEventSynchronize(pr.ev1[i]);
        float t = 0.f;
        if (cudaEventElapsedTime(&t, pr.ev0[i], pr.ev1[i]) == cudaSuccess) {
            cnt[pr.kid[i]] += 1;
            ms[pr.kid[i]] += t;
        }
    }
    pr.n = 0;
    for (int k = 0; k < K_COUNT && k < cap; ++k) {
        if (names) names[k] = kKernelNames[k];
        if (launches) launches[k] = cnt[k];
        if (total_ms) total_ms[k] = ms[k];
    }
    return K_COUNT;
}

}  // extern "C"
