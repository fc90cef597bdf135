// One launch for a whole cascade step (Algorithm 1) over many short-row sequences: one attention
// head per sequence (Section 8.5), rows of at most 128 bf16 elements.
//
// A sequence belongs to a cluster of up to eight CTAs, and nothing in the step crosses sequences, so
// everything the steps of the algorithm wait for is an mbarrier arrival inside the cluster (about
// half a microsecond) instead of a grid boundary or a counter in global memory (two to three):
//   gather     the cluster's CTAs check the inherited list and copy its rows to Xrep, a share each
//              (lines 1-2); every CTA notes which of its own tokens are inherited
//   triangle   r x r Gram, row tiles of 128 representatives dealt to the CTAs (lines 3-4); the row
//              maxima go to a per-position scratch that all CTAs read after the second arrival
//   cross      a CTA owns consecutive 128-row tiles of X and takes them against chunks of 256
//              representatives (lines 6-8); a row's maximum stays in shared memory over the chunks, its norm
//              comes out of the tile that the MMA reads
//   lists      ballots over the CTA's tokens, totals exchanged through distributed shared memory, and
//              every CTA writes its part of the ascending lists (lines 5, 9-11)
// Warp 0 issues the TMA copies, warp 1 the MMAs, warps 2..9 do the rest: two sets of four (a warp per
// TMEM lane quadrant) that share every tile's columns, with two 128 x 256 accumulators, so that the
// next tile's MMAs run behind a tile's reading.
//
// What bounds it (T = 2048, 32 heads of 128, r = 410, one B200; 42.3 us as three launches, 26.0 so; in-kernel time
// stamps): 5 us until the rows are gathered, 1.5 us to the first MMA, 5 us for the triangle and its verdict,
// 10 us for eight cross tiles, 4 us for the lists, 1 us between launches.  A cross tile (128 x 256 x 128) takes
// 1.25 us where its MMAs need 0.55: the epilogue reads an accumulator in 0.75 us, a quarter of it column factors
// out of shared memory.
#include "gram_tc_dev.cuh"

namespace ada {

using namespace tc;

namespace {

constexpr int SS_THREADS = 320;
constexpr int SS_WORKERS = 256;                      // warps 2..9
constexpr int SS_COLS = 256;                         // representatives per chunk = accumulator columns
constexpr int SS_B_SLOT = SS_COLS * 128 * 2;         // two 64-element K blocks of 256 rows
constexpr int SS_A_SLOT = BM * 128 * 2;
constexpr int SS_CLUSTER = 8;                        // largest portable cluster
constexpr int SS_MAX_T = 2048;                       // tokens of a sequence (see step_short_ctas), and of a CTA
constexpr int SS_TAB = 1024;                         // representatives whose factors are passed through shared memory
static_assert(SS_MAX_T < 1 << 16, "positions fit role[]");
constexpr int SS_CHUNKS = SS_MAX_T / SS_COLS;

struct alignas(16) StepShared {
    unsigned long long a_full[2], a_empty[2], b_full[2], b_empty[2], t_full[2], t_empty[2], drain;
    // one arrival per CTA of the cluster: rows gathered; maxima of the triangle written; list totals written
    unsigned long long gathered, verdict, totals;
    unsigned long long staged;                       // column factors of a group of chunks
    unsigned tmem_base;
    int abort_flag[2];                               // why the CTA gives up (0: it does not); limit of its waits
    int tok0[SS_CHUNKS];                             // first token of every chunk
    alignas(16) float col_f[2][2 * SS_COLS];         // column factors (and tokens) of a group, in alternating buffers
    alignas(16) int col_t[2][2 * SS_COLS];
    float tab[SS_TAB];                               // cross factors of the first representatives, written by their owners
    unsigned long long off[SS_MAX_T / 32];           // counts, then exclusive offsets, by 32 tokens
    unsigned long long total[SS_CLUSTER];            // of every CTA of the cluster
    unsigned short role[SS_MAX_T];                   // this CTA's tokens: 0, or position + 1 in the inherited list
    unsigned mx[SS_MAX_T];                           // maxima (bit patterns): of its representatives, then of its tokens
    float inv[SS_MAX_T];                             // 1/||x_t||
};
constexpr int SS_SMEM = 2 * SS_B_SLOT + 2 * SS_A_SLOT + (int)sizeof(StepShared) + 1024;
static_assert(SS_SMEM <= 227 * 1024, "shared memory budget");

struct StepMaps {
    CUtensorMap x, ra, rb;      // rows of X and of Xrep in boxes of 128, rows of Xrep in boxes of 64
};
struct StepArgs {
    const __nv_bfloat16* X;
    int64_t ldx, xb;
    const int32_t *rep_in, *rep_in_cnt;
    __nv_bfloat16* Xrep;        // [B*T][d]
    float* inv_rep;             // [B*T] by position
    float* g_pos;               // [B*T] scratch: gamma_rep by position
    unsigned* status;
    int T, d, rows;             // rows: tokens per CTA, a multiple of 128
    float thr;
    int32_t *keep_idx, *keep_cnt, *add_idx, *add_cnt, *rem_idx, *rem_cnt;
    float *gamma_rep, *gamma_cross;
};

__device__ __forceinline__ unsigned ss_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned ss_map(unsigned addr, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void ss_arrive(unsigned cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// bounded wait for arrivals of the whole cluster; what the arriving threads wrote before is visible
__device__ __forceinline__ bool ss_wait(unsigned long long* bar, volatile int* abort_flag, int where) {
    unsigned polls = 0;
    unsigned long long t0 = 0;
    while (true) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(smem_u32(bar)), "r"(0u), "r"(20000u) : "memory");
        if (ok) return true;
        if ((++polls & 15u) == 0 && gives_up(&t0, abort_flag, where)) return false;
    }
}
__device__ __forceinline__ void ss_workers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(SS_WORKERS) : "memory"); }

// The CTA's tiles, in the order in which every role takes them: first the triangle (row tiles rank, rank + C, ..),
// then the cross tiles; in each, two chunks at a time (a group: both slots of the right operand), every row
// tile against both, so that a left operand is fetched once per group (for every chunk: 26.5 -> 27.1 us).
// Within a group a chunk that has something for a row tile has something for all later ones.
struct Walk {
    int n, nch, nrt, C, rank, tiles, t0, causal;
    // columns and chunks of the cross tiles.  Where every token is inherited no maximum of theirs is read, and one narrow
    // chunk is left, with which the row norms come (one such head beside 31 with 20 of 2048 tokens: 90 -> 57 us).
    int nx, nchx;
    const int* tok0;
    __device__ __forceinline__ int groups(int ph) const { return ph ? max((nchx + 1) >> 1, 1) : (nch + 1) >> 1; }
    __device__ __forceinline__ int first(int ph, int g) const {
        if (ph) return 0;
        const int lo = 4 * g;                            // (nothing of chunk 2g left of row tile 4g)
        return lo + ((rank - lo) % C + C) % C;
    }
    __device__ __forceinline__ int end(int ph) const { return ph ? tiles : nrt; }
    __device__ __forceinline__ int step(int ph) const { return ph ? 1 : C; }
    __device__ __forceinline__ int last(int ph) const {  // row tile; below first(): none
        return ph ? tiles - 1 : (nrt - 1 < rank ? -1 : nrt - 1 - (nrt - 1 - rank) % C);
    }
    // Anything for row tile x in chunk c?  Triangle: columns left of the tile's last row.  Under ADA_CROSS_CAUSAL: a
    // chunk whose first token is below the tile's last row (and chunk 0, with which the row norms come).  The second
    // chunk of a group only with the first, also where a rejected list does not ascend.
    __device__ __forceinline__ bool live(int ph, int c, int x) const {
        if (!ph) return c < nch && x >= 2 * c;
        const int lim = t0 + (x + 1) * BM;
        return c == 0 || (c < nchx && !(causal && (tok0[c] >= lim || (c > 1 && tok0[c & ~1] >= lim))));
    }
    __device__ __forceinline__ int cols(int ph, int c) const {
        return max(16, (min((ph ? nx : n) - c * SS_COLS, SS_COLS) + 15) & ~15);
    }
    // (nothing right of a triangular tile's last row)
    __device__ __forceinline__ int width(int ph, int c, int x) const {
        return ph ? cols(1, c) : min(cols(0, c), (x + 1) * BM - c * SS_COLS);
    }
    // Has a column to be compared with the row, or does the whole chunk lie before the tile?  (Causal: every
    // token of a chunk is below the next one's first.  Compared everywhere, a tile of a causal step took 1.6 us
    // instead of 1.25: 32 heads x 2048, r = 1024 58.0 -> 51.6, which three launches do in 69.)
    __device__ __forceinline__ bool mixed(int ph, int c, int x, int ncols) const {
        if (!ph) return c * SS_COLS + ncols > x * BM;
        return causal && !(c + 1 < nch && tok0[c + 1] <= t0 + x * BM);
    }
};

// CAUSAL: ADA_CROSS_CAUSAL.  (A parameter of the template, so that each form does without the other's code, which is
// fetched cold: 32 heads x 2048, r = 410 26.4 -> 26.0 us; r = 1024 47.3 -> 46.5, causal 51.7 -> 51.1.)
template <bool CAUSAL>
__global__ void __launch_bounds__(SS_THREADS, 1)
k_step_short(const __grid_constant__ StepMaps maps, const __grid_constant__ StepArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    unsigned char* const bs = smem;
    unsigned char* const as = smem + 2 * SS_B_SLOT;
    StepShared& sh = *reinterpret_cast<StepShared*>(smem + 2 * SS_B_SLOT + 2 * SS_A_SLOT);
    volatile int* abort_flag = sh.abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)ss_rank(), C = (int)gridDim.x, b = blockIdx.y;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.a_full[i], 1); mbar_init(&sh.a_empty[i], 5);     // MMAs retired; four warps have read their rows
            mbar_init(&sh.b_full[i], 1); mbar_init(&sh.b_empty[i], 1);
            mbar_init(&sh.t_full[i], 1); mbar_init(&sh.t_empty[i], SS_WORKERS / 32);
        }
        mbar_init(&sh.drain, 1); mbar_init(&sh.staged, SS_WORKERS / 32);
        mbar_init(&sh.gathered, C); mbar_init(&sh.verdict, C); mbar_init(&sh.totals, C);
        sh.abort_flag[0] = 0;
        sh.abort_flag[1] = wait_limit_units(false);  // (a cluster is placed whole: no CTA waits for one that cannot run)
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sh.tmem_base)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 32) { prefetch_map(&maps.x); prefetch_map(&maps.ra); prefetch_map(&maps.rb); }
    for (int i = threadIdx.x; i < a.rows; i += SS_THREADS) { sh.role[i] = 0; sh.mx[i] = 0u; sh.inv[i] = 0.f; }
    tcgen05_fence_before();
    __syncthreads();
    // (also: every CTA's barriers exist before another's arrivals)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    tcgen05_fence_after();
    const unsigned tmem_base = sh.tmem_base;
    // everything above is local to the cluster; from here on the predecessor's results are read
    grid_dep_wait();
    grid_dep_launch_next();

    const int T = a.T, d = a.d;
    const int64_t o = (int64_t)b * T;
    const int32_t* const list = a.rep_in + o;
    const int t0 = rank * a.rows;                    // this CTA's tokens: [t0, t0 + own)
    const int own = min(max(T - t0, 0), a.rows);
    int n = __ldg(a.rep_in_cnt + b);
    constexpr int U = 8;                             // rows of a lane group in flight (gather)
    int G = 1;                                       // lanes per row
    while (G < (d >> 3)) G <<= 1;
    const int R = 32 / G, sub = lane / G, gl = lane % G;
    const int g0 = (rank * (SS_WORKERS / 32) + (warp - 2)) * R, stride = C * (SS_WORKERS / 32) * R;
    int32_t idx[U], prev[U];
    if (warp >= 2) {
        // the first entries, beside the count and not after it
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = g0 + sub + u * stride;
            idx[u] = i < T ? __ldg(list + i) : -1;
            prev[u] = i < T && i > 0 ? __ldg(list + i - 1) : -1;
        }
    }
    if (n < 0 || n > T) {
        if (rank == 0 && threadIdx.x == 0) atomicOr(a.status, ST_BAD_COUNT);
        n = n < 0 ? 0 : T;
    }
    const int nkb = (d + BK - 1) / BK;               // 64-element K blocks (one or two)
    Walk w;
    w.n = n; w.nch = (n + SS_COLS - 1) / SS_COLS; w.nrt = (n + BM - 1) / BM;
    w.nx = n == T ? 1 : n; w.nchx = n == T ? 1 : w.nch;
    w.C = C; w.rank = rank; w.tiles = (own + BM - 1) / BM; w.t0 = t0; w.causal = CAUSAL ? 1 : 0;
    w.tok0 = sh.tok0;

    if (warp >= 2) {
        // ------------------------------------------------ gather, workers of all CTAs: a lane group of G per row
        const int wk = (int)threadIdx.x - 64;
        const int nvec = d >> 3;
        const __nv_bfloat16* Xs = a.X + (int64_t)b * a.xb;
        for (int i0 = g0 + sub; i0 - sub < n; i0 += U * stride) {
            uint4 x[U];
            if (i0 != g0 + sub) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = i0 + u * stride;
                    idx[u] = i < n ? __ldg(list + i) : -1;
                    prev[u] = i < n && i > 0 ? __ldg(list + i - 1) : -1;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u * stride;
                const bool ok = i < n && idx[u] >= 0 && idx[u] < T && prev[u] < idx[u];
                if (!ok && i < n && gl == 0) atomicOr(a.status, ST_BAD_INDEX);
                x[u] = make_uint4(0u, 0u, 0u, 0u);
                if (ok && gl < nvec) x[u] = __ldg(reinterpret_cast<const uint4*>(Xs + (int64_t)idx[u] * a.ldx) + gl);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u * stride;
                float ss = sumsq_bf16x8(x[u]);
                for (int q = G >> 1; q > 0; q >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, q);
                if (i >= n) continue;
                // (a rejected entry: a row of zeros whose column counts for nothing)
                if (gl < nvec) reinterpret_cast<uint4*>(a.Xrep + (o + i) * d)[gl] = x[u];
                if (gl == 0) a.inv_rep[o + i] = (ss <= 3.0e38f && ss > 0.f) ? 1.0f / sqrtf(ss) : 0.f;
            }
        }
        // the rows just written are read by TMA (async proxy), from every CTA of the cluster
        asm volatile("fence.proxy.async.global;" ::: "memory");
        if (wk < SS_CHUNKS && wk * SS_COLS < n) sh.tok0[wk] = __ldg(list + wk * SS_COLS);
        ss_workers_sync();
        // (the arrivals' release covers what the barrier ordered before it)
        if (wk < C) ss_arrive(ss_map(smem_u32(&sh.gathered), wk));
        // which of this CTA's tokens are inherited
        for (int i = wk; i < n; i += SS_WORKERS) {
            const unsigned t = (unsigned)(__ldg(list + i) - t0);
            if (t < (unsigned)own) sh.role[t] = (unsigned short)(i + 1);
        }
    }
    // (A wait that runs out only clears `ok`: the workers of a CTA meet at barriers without a limit, and each CTA
    // still owes the others its arrivals.  The status is raised at the end.)
    bool ok = ss_wait(&sh.gathered, abort_flag, 50);
    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (lane == 0 && ok) {
            asm volatile("fence.proxy.async.global;" ::: "memory");
            unsigned ka = 0, nb[2] = {0, 0};         // left operands so far; chunks through each slot
            for (int ph = 0; ph < 2 && ok; ++ph)
                for (int g = 0; g < w.groups(ph) && ok; ++g) {
                    const int x1 = w.last(ph);
                    for (int x = w.first(ph, g); x < w.end(ph) && ok; x += w.step(ph)) {
                        if (!w.live(ph, 2 * g, x) && !w.live(ph, 2 * g + 1, x)) continue;
                        const unsigned s = ka & 1u;
                        ok = mbar_wait(&sh.a_empty[s], ((ka >> 1) & 1u) ^ 1u, abort_flag, 52);
                        if (!ok) break;
                        mbar_expect_tx(&sh.a_full[s], (unsigned)(nkb * A_BYTES));
                        for (int kb = 0; kb < nkb; ++kb)
                            tma_load_3d(ph ? &maps.x : &maps.ra, &sh.a_full[s], as + s * SS_A_SLOT + kb * A_BYTES,
                                        kb * BK, (ph ? t0 : 0) + x * BM, b);
                        ++ka;
                        if (x != w.first(ph, g) && w.live(ph, 2 * g, x - w.step(ph))) continue;
                        // the group's chunks, behind the first left operand that meets them
                        for (int e = 0; e < 2 && ok; ++e) {
                            const int c = 2 * g + e;
                            if (!w.live(ph, c, x1)) continue;
                            const int nbox = (w.cols(ph, c) + BOX_N - 1) / BOX_N;
                            ok = mbar_wait(&sh.b_empty[e], (nb[e] & 1u) ^ 1u, abort_flag, 51);
                            if (!ok) break;
                            ++nb[e];
                            mbar_expect_tx(&sh.b_full[e], (unsigned)(nkb * nbox * BOX_BYTES));
                            for (int kb = 0; kb < nkb; ++kb)
                                for (int j = 0; j < nbox; ++j)
                                    tma_load_3d(&maps.rb, &sh.b_full[e],
                                                bs + e * SS_B_SLOT + kb * (SS_B_SLOT / 2) + j * BOX_BYTES, kb * BK,
                                                c * SS_COLS + j * BOX_N, b);
                        }
                    }
                }
            // every copy has to land before the CTA may exit
            const unsigned long long since = global_ns();
            for (unsigned s = 0; s < 2; ++s) {
                const unsigned ua = (ka + 1 - s) >> 1, ub = nb[s];                 // uses of slot s
                while (!((ua == 0 || mbar_try(&sh.a_full[s], (ua - 1) & 1u)) && (ub == 0 || mbar_try(&sh.b_full[s], (ub - 1) & 1u))))
                    if (past_limit(2 * (global_ns() - since), abort_flag)) { *abort_flag = 53; break; }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0 && ok) {
            unsigned k = 0, ka = 0, nb[2] = {0, 0};  // tiles, left operands, chunks through each slot
            for (int ph = 0; ph < 2 && ok; ++ph)
                for (int g = 0; g < w.groups(ph) && ok; ++g) {
                    const int x1 = w.last(ph);
                    bool seen[2] = {false, false};
                    for (int x = w.first(ph, g); x < w.end(ph) && ok; x += w.step(ph)) {
                        const unsigned s = ka & 1u;
                        bool any = false;
                        for (int e = 0; e < 2; ++e) {
                            const int c = 2 * g + e;
                            if (!w.live(ph, c, x)) continue;
                            if (!any) ok = mbar_wait(&sh.a_full[s], (ka >> 1) & 1u, abort_flag, 55);
                            if (ok && !seen[e]) ok = mbar_wait(&sh.b_full[e], nb[e] & 1u, abort_flag, 54);
                            any = seen[e] = true;
                            const unsigned p = k & 1u;
                            ok = ok && mbar_wait(&sh.t_empty[p], ((k >> 1) & 1u) ^ 1u, abort_flag, 56);
                            if (!ok) break;
                            tcgen05_fence_after();
                            const unsigned idesc = instr_desc(w.width(ph, c, x));
                            const unsigned long long adesc = smem_desc_sw128(smem_u32(as + s * SS_A_SLOT));
                            const unsigned long long bdesc = smem_desc_sw128(smem_u32(bs + e * SS_B_SLOT));
                            if (nkb == 2) umma_blocks<2>(tmem_base + p * SS_COLS, adesc, bdesc, A_BYTES, SS_B_SLOT / 2, idesc);
                            else umma_blocks<1>(tmem_base + p * SS_COLS, adesc, bdesc, 0, 0, idesc);
                            umma_commit(&sh.t_full[p]);
                            ++k;
                            if (x == x1) { umma_commit(&sh.b_empty[e]); ++nb[e]; }
                        }
                        if (any && ok) { umma_commit(&sh.a_empty[s]); ++ka; }
                    }
                }
            // all MMAs issued by this thread must retire before TMEM is freed
            umma_commit(&sh.drain);
            const unsigned long long since = global_ns();
            while (!mbar_try(&sh.drain, 0))
                if (past_limit(2 * (global_ns() - since), abort_flag)) { *abort_flag = 57; break; }
        }
    } else {
        // ------------------------------------------------ workers: epilogues, then the lists
        const int wk = (int)threadIdx.x - 64, wl = warp - 2;
        const int quad = warp & 3, set = wl >> 2;
        const int lrow = quad * 32 + lane;               // this thread's row of a tile
        constexpr int V = SS_MAX_T / SS_WORKERS;
        const int slices = (own + SS_WORKERS - 1) / SS_WORKERS;
        unsigned k = 0, ka = 0, staged = 0;              // tiles, left operands, groups so far
        float gp[V];                                     // gamma_rep of this thread's tokens, where they are inherited
        ok = __all_sync(0xffffffffu, ok);
        for (int ph = 0; ph < 2; ++ph) {
            for (int g = 0; g < w.groups(ph) && ok; ++g) {
                if (w.first(ph, g) >= w.end(ph)) continue;
                // column factors of the group's chunks, two per thread: 1/||x||, and 0 past the end and (cross) for a
                // representative that line 5 removed.  (A warp that stages the next group has seen this one
                // staged by all, so nobody still reads the buffer that it writes.)
                const float* const gs = sh.col_f[staged & 1u];
                const int* const gt = sh.col_t[staged & 1u];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int col = (2 * g + e) * SS_COLS + wk;
                    const bool live = col < n;
                    float v = 0.f;
                    if (ph && n <= SS_TAB) v = live ? sh.tab[col] : 0.f;
                    else if (live) {
                        v = __ldcg(a.inv_rep + o + col);
                        if (ph && !(__ldcg(a.g_pos + o + col) < a.thr)) v = 0.f;
                    }
                    sh.col_f[staged & 1u][e * SS_COLS + wk] = v;
                    if (ph == 0 || CAUSAL) sh.col_t[staged & 1u][e * SS_COLS + wk] = ph && live ? __ldg(list + col) : col;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.staged);
                ok = __all_sync(0xffffffffu, mbar_wait(&sh.staged, staged & 1u, abort_flag, 62));
                ++staged;
                for (int x = w.first(ph, g); x < w.end(ph) && ok; x += w.step(ph)) {
                    const int row = (ph ? t0 : 0) + x * BM + lrow;     // token, or position
                    const int at = (ph ? x : x / C) * BM + lrow;       // place in mx
                    bool any = false;
                    float m0 = 0.f, m1 = 0.f;
                    for (int e = 0; e < 2; ++e) {
                    const int c = 2 * g + e;
                    if (!w.live(ph, c, x)) continue;
                    const unsigned p = k & 1u, use = (k >> 1) & 1u;
                    ++k;
                    const float* const cs = gs + e * SS_COLS;
                    const int* const ct = gt + e * SS_COLS;
                    if (!any && (int)(ka & 1u) == set) {
                        const unsigned sa = ka & 1u;
                        if (ph && g == 0) {
                            // the row's norm, out of the tile that the MMA reads (the swizzle permutes 16-byte pieces of
                            // a row, which a sum of squares need not undo; lanes start at different pieces)
                            ok = __all_sync(0xffffffffu, mbar_wait(&sh.a_full[sa], (ka >> 1) & 1u, abort_flag, 58));
                            if (!ok) break;
                            float s0 = 0.f, s1 = 0.f;
                            for (int kb = 0; kb < nkb; ++kb) {
                                const unsigned char* rowp = as + sa * SS_A_SLOT + kb * A_BYTES + lrow * 128;
#pragma unroll
                                for (int j = 0; j < 8; j += 2) {
                                    s0 += sumsq_bf16x8(*reinterpret_cast<const uint4*>(rowp + (((j + lane) & 7) << 4)));
                                    s1 += sumsq_bf16x8(*reinterpret_cast<const uint4*>(rowp + (((j + 1 + lane) & 7) << 4)));
                                }
                            }
                            const float ss = s0 + s1;
                            if (row < T) {
                                float inv = 0.f;
                                if (!(ss <= 3.0e38f)) atomicOr(a.status, ST_NONFINITE);
                                else if (ss > 0.f) inv = 1.0f / sqrtf(ss);
                                else atomicAdd(a.status + 1, 1u);
                                sh.inv[at] = inv;
                            }
                            __syncwarp();
                        }
                        if (lane == 0) mbar_arrive(&sh.a_empty[sa]);
                    }
                    any = true;
                    ok = __all_sync(0xffffffffu, mbar_wait(&sh.t_full[p], use, abort_flag, 59));
                    if (!ok) break;
                    tcgen05_fence_after();
                    const int ncols = w.width(ph, c, x);
                    const bool need_cmp = w.mixed(ph, c, x, ncols);
                    const unsigned tbase = tmem_base + ((unsigned)(quad * 32) << 16) + p * SS_COLS;
                    auto consume = [&](const unsigned (&r)[32], int c0) {
                        if (!need_cmp) {
                            row_max32(r, cs + c0, m0, m1);
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; j += 4) {
                                const float4 f = *reinterpret_cast<const float4*>(cs + c0 + j);
                                const int4 t = *reinterpret_cast<const int4*>(ct + c0 + j);
                                if (t.x < row) m0 = fmaxf(m0, fabsf(__uint_as_float(r[j])) * f.x);
                                if (t.y < row) m1 = fmaxf(m1, fabsf(__uint_as_float(r[j + 1])) * f.y);
                                if (t.z < row) m0 = fmaxf(m0, fabsf(__uint_as_float(r[j + 2])) * f.z);
                                if (t.w < row) m1 = fmaxf(m1, fabsf(__uint_as_float(r[j + 3])) * f.w);
                            }
                        }
                    };
                    // the sets take alternate pieces of 32 columns, two in flight (rolled: the code is fetched cold)
#pragma unroll 1
                    for (int c0 = 32 * set; c0 < ncols; c0 += 128) {
                        unsigned r0[32], r1[32];
                        const bool two = c0 + 64 < ncols;
                        tmem_ld32_issue(tbase + c0, r0);
                        tmem_ld32_issue(tbase + c0 + 64, r1);          // (inside the accumulator whatever the width)
                        tmem_ld_wait(r0);
                        tmem_ld_wait(r1);
                        consume(r0, c0);
                        if (two) consume(r1, c0 + 64);
                    }
                    tcgen05_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh.t_empty[p]);
                    }
                    if (any) ++ka;
                    const float m = fmaxf(m0, m1);
                    if (m > 0.f && row < (ph ? T : n)) atomicMax(&sh.mx[at], __float_as_uint(m));
                }
            }
            if (ph) break;
            // gamma_rep of this CTA's representatives, and their factors in the cross tiles (line 5), for all CTAs
            const int mine = (w.nrt - rank + C - 1) / C * BM;          // row tiles of the triangle here, in rows
            float ir = 0.f;
            for (int i = wk; i - wk < mine; i += SS_WORKERS) {
                const int pos = ((i >> 7) * C + rank) * BM + (i & 127);
                const bool live = i < mine && pos < n;
                ir = live ? __ldcg(a.inv_rep + o + pos) : 0.f;
                if (i == wk) ss_workers_sync();                        // (the loads are under way)
                if (!live) continue;
                const unsigned m = sh.mx[i];
                const float g = m != 0u ? __uint_as_float(m) * ir : 0.f;
                a.g_pos[o + pos] = g;
                sh.mx[i] = 0u;
                if (n <= SS_TAB)
                    for (int q = 0; q < C; ++q)
                        asm volatile("st.shared::cluster.f32 [%0], %1;"
                                     ::"r"(ss_map(smem_u32(&sh.tab[pos]), q)), "f"(g < a.thr ? ir : 0.f) : "memory");
            }
            if (mine <= 0) ss_workers_sync();
            ss_workers_sync();
            if (wk < C) ss_arrive(ss_map(smem_u32(&sh.verdict), wk));
            ok = __all_sync(0xffffffffu, ss_wait(&sh.verdict, abort_flag, 60)) && ok;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int i = v * SS_WORKERS + wk;
                const int q = i < own ? sh.role[i] : 0;
                gp[v] = q > 0 ? __ldcg(a.g_pos + o + q - 1) : 0.f;
            }
        }
        ss_workers_sync();
        // ------------------------------------------------ lists (lines 5, 9-11 and Eq. 6); the three counts of a
        // sequence share a word (20 bits each)
        constexpr unsigned BITS = 20;
        constexpr unsigned MASK = (1u << BITS) - 1u;
        {
            unsigned bk[V], ba[V], br[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                bk[v] = ba[v] = br[v] = 0u;
                if (v >= slices) continue;
                const int i = v * SS_WORKERS + wk, t = t0 + i;
                bool keep = false, add = false, rem = false;
                if (i < own) {
                    float ga = 0.f, gb = 0.f;
                    if (sh.role[i] > 0) {
                        ga = gp[v];
                        keep = ga < a.thr;
                        rem = !keep;
                    } else {
                        // (an untouched entry is a maximum over nothing: 0 whatever the row's norm)
                        gb = sh.mx[i] != 0u ? __uint_as_float(sh.mx[i]) * sh.inv[i] : 0.f;
                        keep = add = gb < a.thr;
                    }
                    if (a.gamma_rep != nullptr) a.gamma_rep[o + t] = ga;
                    if (a.gamma_cross != nullptr) a.gamma_cross[o + t] = gb;
                }
                bk[v] = __ballot_sync(0xffffffffu, keep);
                ba[v] = __ballot_sync(0xffffffffu, add);
                br[v] = __ballot_sync(0xffffffffu, rem);
                if (lane == 0)
                    sh.off[v * (SS_WORKERS / 32) + wl] = (unsigned long long)__popc(bk[v]) |
                        ((unsigned long long)__popc(ba[v]) << BITS) | ((unsigned long long)__popc(br[v]) << (2 * BITS));
            }
            ss_workers_sync();
            if (warp == 2) {                             // lane l scans entries 2l and 2l + 1 (token order)
                static_assert(SS_MAX_T / 32 == 64, "two entries per lane");
                const int ne = slices * (SS_WORKERS / 32);
                const unsigned long long c0 = 2 * lane < ne ? sh.off[2 * lane] : 0ull, c1 = 2 * lane + 1 < ne ? sh.off[2 * lane + 1] : 0ull;
                unsigned long long incl = c0 + c1;
#pragma unroll
                for (int q = 1; q < 32; q <<= 1) {
                    const unsigned long long up = __shfl_up_sync(0xffffffffu, incl, q);
                    if (lane >= q) incl += up;
                }
                const unsigned long long total = __shfl_sync(0xffffffffu, incl, 31);
                sh.off[2 * lane] = incl - c0 - c1;
                sh.off[2 * lane + 1] = incl - c1;
                __syncwarp();
                if (lane < C) {                          // this CTA's total, to every CTA of the cluster
                    asm volatile("st.shared::cluster.u64 [%0], %1;"
                                 ::"r"(ss_map(smem_u32(&sh.total[rank]), lane)), "l"(total) : "memory");
                    ss_arrive(ss_map(smem_u32(&sh.totals), lane));
                }
            }
            if (__all_sync(0xffffffffu, ss_wait(&sh.totals, abort_flag, 61))) {
                unsigned long long base = 0, all = 0;
                for (int q = 0; q < C; ++q) {
                    const unsigned long long one = sh.total[q];
                    all += one;
                    if (q < rank) base += one;
                }
                const unsigned below = (1u << lane) - 1u;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    if (v >= slices) continue;
                    const int t = t0 + v * SS_WORKERS + wk;
                    const unsigned long long at = base + sh.off[v * (SS_WORKERS / 32) + wl];
                    if ((bk[v] >> lane) & 1u) a.keep_idx[o + (int)(at & MASK) + __popc(bk[v] & below)] = t;
                    if ((ba[v] >> lane) & 1u) a.add_idx[o + (int)((at >> BITS) & MASK) + __popc(ba[v] & below)] = t;
                    if ((br[v] >> lane) & 1u) a.rem_idx[o + (int)(at >> (2 * BITS)) + __popc(br[v] & below)] = t;
                }
                if (rank == 0 && wk == 0) {
                    a.keep_cnt[b] = (int)(all & MASK);
                    a.add_cnt[b] = (int)((all >> BITS) & MASK);
                    a.rem_cnt[b] = (int)(all >> (2 * BITS));
                }
            }
        }
    }

    tcgen05_fence_before();
    __syncthreads();
    // (no CTA leaves while another may still arrive on its barriers)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 1) {
        tcgen05_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    }
    if (threadIdx.x == 0 && sh.abort_flag[0] != 0) {
        atomicOr(a.status, ST_TIMEOUT);
        a.status[2] = 300u + (unsigned)sh.abort_flag[0];
    }
}

}  // namespace

// How many clusters of C CTAs (C = 1..8) run at once, per context.
static cudaError_t ensure_short(ada_ctx* ctx) {
    if (ctx->short_attr_set) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_step_short<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SS_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step_short<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SS_SMEM);
    if (e != cudaSuccess) { cudaGetLastError(); return e; }
    for (int C = 1; C <= SS_CLUSTER; ++C) {
        cudaLaunchConfig_t q;
        memset(&q, 0, sizeof(q));
        q.gridDim = dim3(C, ctx->sm_count);
        q.blockDim = dim3(SS_THREADS);
        q.dynamicSmemBytes = SS_SMEM;
        cudaLaunchAttribute qa[1];
        qa[0].id = cudaLaunchAttributeClusterDimension;
        qa[0].val.clusterDim.x = C; qa[0].val.clusterDim.y = 1; qa[0].val.clusterDim.z = 1;
        q.attrs = qa; q.numAttrs = 1;
        int at_once = 0;
        e = cudaOccupancyMaxActiveClusters(&at_once, k_step_short<false>, &q);
        if (e != cudaSuccess) { cudaGetLastError(); return e; }
        ctx->short_clusters[C] = at_once;
    }
    ctx->short_attr_set = true;
    return cudaSuccess;
}

// CTAs per sequence of the one-launch step, or 0: not this step.  As many as let all clusters run at once, at most
// eight (with one more round of clusters 16 heads x 2048 took 27.6 us instead of 17.0).
//
// A sequence has its cluster and no other CTA, while the tiles of the three launches go to all SMs: the one launch lasts as
// long as its largest set, the others as long as the average.  Both forms (d = 128; us, one launch / three) where all sets
// hold T/100, T/10, T/5, T/2 of the tokens, where one holds T/5, T/2, or all, the others T/100, and where they are
// spread evenly in the logarithm over T/100..T/5 and T/100..0.6 T:
//                  T/100       T/10        T/5         T/2       one T/5     one T/2      one T       ..T/5     ..0.6 T
//    8 x 1000   14.1/18.5   15.1/19.7   16.1/20.1   18.7/21.2   15.7/19.1   18.1/20.0   20.7/20.4   15.4/19.9   18.0/20.4
//   32 x 1000   15.9/22.9   17.1/24.7   18.6/26.1   22.9/32.5   17.2/23.5   21.0/23.9   27.8/24.0   17.2/24.8   27.8/29.2
//  100 x 1000   22.5/57.5   25.6/62.2   33.5/66.5   55.0/86.0   32.5/57.2   53.7/57.1   74.4/57.7   32.2/62.2   67.8/68.0
//   12 x 2048   15.4/21.7   17.9/24.0   20.8/27.2   30.9/34.5   19.9/22.6   29.6/23.1   36.9/25.6   19.5/24.3   29.7/29.0
//   16 x 2048   17.1/23.4   20.0/25.5   23.7/30.3   40.3/41.4   22.8/24.5   39.0/25.3   46.1/27.2   22.2/27.1   38.7/30.7
//   32 x 2048   18.4/29.4   22.0/34.2   26.9/42.1   47.1/61.8   25.1/30.0   45.1/30.7   56.6/33.4   25.4/34.8   58.2/42.3
//  148 x 2048   32.7/107    47.7/123    72.8/157    149/278     70.3/109    143/109     179/109     71.1/123    185/156
//   32 x 3000   20.8/35.4   29.5/49.2   44.0/59.4   82.8/103    41.8/36.4   80.3/37.7   92.8/40.7   41.4/45.1   96.6/61.7
// (ADA_CROSS_CAUSAL changes both by up to a sixth, and no comparison up to T/5.)  The set sizes live on the device, so the
// line is drawn where no set of up to a fifth of its sequence, whatever the others hold, makes the step slower: at 2048
// tokens.  Where one set is larger than that and the others are not, the three launches would be faster, by up to 1.5
// times at T/2.  (At 8192 tokens a single set of T/2 beside 31 small ones took 411 us instead of 87.)  Sharing such a head's tiles among all CTAs, counted out through global memory, was tried: 8192 tokens 411 -> 93,
// but 2048 tokens 45 -> 43, and its code costs every other step 0.5 to 5 %.
//
// Within that, used where its CTAs cover three fifths of the SMs, or have one row tile each (8 x 2048, r = T/2: 30.7 / 29.1;
// 2 x 1000, r = T/2: 18.2 / 18.6), and up to as many sequences as there are SMs (more rounds of clusters: not measured).
int step_short_ctas(ada_ctx* ctx, int64_t B, int64_t T, int64_t d) {
    if (d > 128 || T > SS_MAX_T || ensure_short(ctx) != cudaSuccess) return 0;
    const int64_t tiles = (T + BM - 1) / BM;
    for (int64_t C = SS_CLUSTER; C >= 1; --C) {
        if (C > tiles || ctx->short_clusters[C] < B) continue;
        const int64_t per = (tiles + C - 1) / C;                       // row tiles per CTA
        C = (tiles + per - 1) / per;                                   // (no CTA without rows)
        if (per > 1 && 5 * B * C < 3 * ctx->sm_count) return 0;
        return (int)C;
    }
    return 0;
}

cudaError_t launch_step_short(ada_ctx* ctx, int C, const void* X, int B, int T, int d, int64_t ldx, int64_t xb, float thr,
                              const int32_t* rep_in, const int32_t* rep_in_cnt, int32_t* rep_out, int32_t* rep_out_cnt,
                              int32_t* add_idx, int32_t* add_cnt, int32_t* rem_idx, int32_t* rem_cnt, float* gamma_rep,
                              float* gamma_cross, int causal, cudaStream_t s) {
    StepMaps maps;
    memset(&maps, 0, sizeof(maps));
    if (!make_map(ctx, &maps.x, X, d, T, B, ldx, xb, BM) ||
        !make_map(ctx, &maps.ra, ctx->Xrep, d, T, B, d, (int64_t)T * d, BM) ||
        !make_map(ctx, &maps.rb, ctx->Xrep, d, T, B, d, (int64_t)T * d, BOX_N))
        return cudaErrorInvalidValue;
    StepArgs a;
    a.X = static_cast<const __nv_bfloat16*>(X); a.ldx = ldx; a.xb = xb;
    a.rep_in = rep_in; a.rep_in_cnt = rep_in_cnt;
    a.Xrep = static_cast<__nv_bfloat16*>(ctx->Xrep); a.inv_rep = ctx->inv_rep; a.g_pos = ctx->inv_norm;
    a.status = ctx->status;
    a.T = T; a.d = d; a.rows = ((T + BM - 1) / BM + C - 1) / C * BM;
    a.thr = thr;
    a.keep_idx = rep_out; a.keep_cnt = rep_out_cnt;
    a.add_idx = add_idx; a.add_cnt = add_cnt; a.rem_idx = rem_idx; a.rem_cnt = rem_cnt;
    a.gamma_rep = gamma_rep; a.gamma_cross = gamma_cross;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(C, B);
    cfg.blockDim = dim3(SS_THREADS);
    cfg.dynamicSmemBytes = SS_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->dep_launch ? 2 : 1;
    prof_begin(ctx, K_STEP_SHORT, s);
    cudaError_t e = cudaLaunchKernelEx(&cfg, causal ? k_step_short<true> : k_step_short<false>, maps, a);
    if (e != cudaSuccess) cudaGetLastError();   // returned; the next launcher that asks must not find it again
    prof_end(ctx, s);
    return e;
}

}  // namespace ada
