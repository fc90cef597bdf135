// bf16 masked-Gram kernel for sm_100a, two-CTA form: the CTAs of a cluster of two
// (one per SM of a TPC) share one 256-row output tile.  Each CTA loads its own 128 rows
// of the left operand but only HALF of the right operand's columns; the leader CTA
// issues tcgen05.mma.cta_group::2 (M = 256), which reads both halves from the two shared
// memories and writes each CTA's 128 x N accumulator into its own TMEM.  Per CTA and
// K block that is 16 KiB + N*64 bytes of TMA traffic instead of 16 KiB + N*128: the
// one-CTA kernel is bound by what one SM can pull out of L2, this one by the tensor pipe.
//
// Same contract as the one-CTA kernel (out[i] = max_j |a_i.b_j| inv_a[i] inv_b[j] over the
// admissible j; Definition 1, Algorithm 1 lines 3-4 and 7-8; the Gram never leaves TMEM),
// same order of tiles (triangular segment first, cross epilogues wait for it); ten warps:
//   warp 0      plans the work (tile list, what is split along K), decodes the CTA's tiles into shared
//               memory and then is the TMA producer, in BOTH CTAs (completion bytes of both land on
//               the leader's mbarrier; no multicast is used)
//   warp 1      leader: MMA issuer; releases ring stages and hands over accumulators with
//               tcgen05.commit multicast to both CTAs.  Both CTAs: TMEM allocation
//   warps 2..9  first the preparation of a cascade step: Algorithm 1 lines 1-2 (list checked, role
//               map, rows copied to Xrep with their inverse norms; fp32: the bf16 planes of
//               every row), which loads and epilogues wait for; then the row norms of X with
//               plain loads behind the first main loops (in the streaming form out of
//               the left-operand tiles while those sit in shared memory, one thread per row,
//               so that X is read from memory exactly once); then the epilogue, each CTA on its own
//               128 rows, two warps per TMEM lane quadrant; the peer's returns the accumulator by
//               a remote arrive on the leader's mbarrier
// The cross segment's row maxima are published WITHOUT the factor 1/||x_t|| (it commutes with
// the maximum; the compaction applies it), so no epilogue waits for a norm.  When one column
// tile covers all representatives the step is bound by streaming X once: the row tiles are
// then cut shorter than 128 rows per CTA so that every SM pair streams a share.
//
// What bounds a launch (in-kernel time stamps, one B200): 8-9 us until the first MMA of a cascade step
// (preparation 4 us, arrival seen by every CTA 1.5 us, first copies 2-3 us, much of it instruction
// fetch: with a layer's activations passing through L2 between launches the code is cold), 0.6 us per
// 64 KB stage and SM in the main loop (L2 to SM), 2-3 us from the last accumulator to the
// maxima, 3-5 us when a tile was split.
// Every wait is bounded; the two CTAs meet at a cluster barrier before either frees TMEM
// or exits.
#include "gram_tc_dev.cuh"

namespace ada {

using namespace tc;

namespace {

constexpr int PM = 2 * BM;     // rows of a pair tile
// What a ring stage holds.  bf16 storage: two consecutive 64-element K blocks (each its own
// 128-byte-swizzled sub-tile), so that the per-stage costs -- barrier round trips, fences,
// commit -- are paid once per 128 K elements and the MMA issue stays ahead of the tensor pipe.
// fp32 storage: the three bf16 planes (hi, mid, lo) of ONE 64-element K block, from which the six
// leading cross terms are contracted: every plane is fetched once and used two or three times.
// Its tiles are at most 128 columns wide so that three stages fit the ring.
// Warps 2..9 do everything but copies and MMAs: preparation, row norms, epilogue.  (Twelve of them left
// 128 registers a thread and an epilogue that spilled, which cost more than the warps gave.)
constexpr int EPI_WARPS = 8;
constexpr int SUBS = EPI_WARPS / 4;            // warps per TMEM lane quadrant
constexpr int PAIR_THREADS = 64 + 32 * EPI_WARPS;
template <bool SPLIT>
struct Stage {
    static constexpr int NSUB = SPLIT ? 3 : 2;
    static constexpr int K = SPLIT ? BK : 2 * BK;          // K elements per stage
    static constexpr int MAXW = SPLIT ? BN / 2 : BN;       // widest tile (columns of the pair)
    static constexpr int TERMS = SPLIT ? 6 : 2;            // MMA groups per stage
    static constexpr bool ALT = !SPLIT;                     // may the two epilogue sets take alternate tiles?
    static constexpr int COLS = ALT ? MAXW : MAXW / SUBS;   // columns of a tile that one epilogue warp sees
    // sub-tiles of A and B multiplied by group t
    static __device__ __forceinline__ constexpr int ta(int t) { return SPLIT ? (t == 2 || t == 5 ? 1 : (t == 4 ? 2 : 0)) : t; }
    static __device__ __forceinline__ constexpr int tb(int t) { return SPLIT ? (t == 1 || t == 5 ? 1 : (t == 3 ? 2 : 0)) : t; }
};

// ---------------------------------------------------------------- PTX, pair forms
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of the same shared-memory location in CTA `rank` of this cluster
__device__ __forceinline__ unsigned map_to_cta(unsigned addr, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void mbar_arrive_remote(unsigned cluster_addr, unsigned count) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_addr), "r"(count)
                 : "memory");
}
// TMA load whose completion bytes go to the LEADER's barrier: bit 24 of a shared::cluster
// address selects the CTA within the pair, clearing it names the even (leader) CTA.
__device__ __forceinline__ void tma_load_3d_pair(const CUtensorMap* map, unsigned long long* bar,
                                                 void* dst, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<unsigned long long>(map)),
          "r"(smem_u32(bar) & 0xFEFFFFFFu), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
// The same for rows that no later copy of the launch reads: the first lines to leave L2.
__device__ __forceinline__ void tma_load_3d_pair_once(const CUtensorMap* map, unsigned long long* bar,
                                                      void* dst, int c0, int c1, int c2, unsigned long long policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5}], [%2], %6;"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<unsigned long long>(map)),
          "r"(smem_u32(bar) & 0xFEFFFFFFu), "r"(c0), "r"(c1), "r"(c2), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(unsigned tmem_d, unsigned long long adesc,
                                               unsigned long long bdesc, unsigned idesc,
                                               unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// commit: arrive on the barrier at this offset in BOTH CTAs once the MMAs issued so far retire
__device__ __forceinline__ void umma_commit_pair_both(unsigned long long* bar) {
    const unsigned short mask = 3;
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(smem_u32(bar)), "h"(mask)
        : "memory");
}
__device__ __forceinline__ void umma_commit_pair_local(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_u32(bar))
                 : "memory");
}
// instruction descriptor of the pair MMA: M = 256
__device__ __forceinline__ unsigned instr_desc_pair(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(PM >> 4) << 24);
}

// ---------------------------------------------------------------- tile list (256-row tiles)
// a / b for 0 <= a, 0 < b and quotients below 2^20: a float quotient is off by at most one there, and an
// integer division costs several times as much on the path to the first copy
__device__ __forceinline__ int quot(int a, int b) {
    int q = (int)__fdividef((float)a, (float)b);
    const int r = a - q * b;
    q += (r >= b) - (r < 0);
    return q;
}
constexpr int PLAN_B = 64;      // sequences whose lengths are kept in shared memory
// Work plan of a launch, made by one warp of every CTA.
struct Plan {
    int tiles0, total;          // triangular tiles; all tiles
    int tw;                     // column width of the triangular tiles
    int hrows;                  // rows of the left operand per CTA in cross tiles (128, or fewer: streaming form)
    int smem_norms, compact;      // row norms of X out of the tiles in shared memory (2: streaming form); cross tiles over Xnon
    int alt;                    // the two epilogue sets take alternate tiles
    int full, rem, parts;       // tiles dealt whole; tiles of the last round, each cut into `parts` K ranges
    int len[PLAN_B];            // sequence lengths (B <= PLAN_B)
};
__device__ __forceinline__ int seq_n_global(const GramProblem& p, int b) {
    int n = p.n_dev != nullptr ? p.n_dev[b] : p.n_host;
    if (p.n_clamp) n = min(max(n, 0), p.cap);
    return n;
}
__device__ __forceinline__ int seq_n(const GramProblem& p, const Plan& pl, int b) {
    return p.B <= PLAN_B ? pl.len[b] : seq_n_global(p, b);
}
// lower triangle in column tiles of width tw (256 or 128): row pair P (256 rows) needs the columns below (P + 1) 256
__device__ __forceinline__ int tri_tiles(int n, int tw) {
    const int M = (n + PM - 1) / PM;
    const int f = tw == PM ? 1 : 2;
    return M > 0 ? f * (M * (M - 1) / 2) + (tw == PM ? M : (n + BM - 1) / BM) : 0;
}
// column tiles of a cross problem with n columns, at most maxw wide.  With in-launch norms (inv_out)
// a sequence without columns still gets one (empty) column tile: its rows have to be read for
// their norms.
__device__ __forceinline__ void cross_cols(const GramProblem& p, int n, int maxw, int& nct, int& w) {
    nct = (n + maxw - 1) / maxw;
    if (nct == 0 && p.inv_out != nullptr && n == 0) nct = 1;
    w = nct > 0 ? max(32, (quot(n + nct - 1, nct) + 31) & ~31) : 0;    // each CTA holds w/2 columns: keep w/2 a multiple of 16
}
// rows of the cross segment's left operand for a sequence with n inherited tokens: all of
// X, or only the tokens outside the inherited set when those were copied out (compact)
__device__ __forceinline__ int cross_rows(const GramProblem& p, int n, bool compact) {
    return compact ? p.rows - n : p.rows;
}
__device__ __forceinline__ int seq_tiles(const GramProblem& p, int n, int maxw, int tw, int hrows, bool compact) {
    if (p.tri) return tri_tiles(n, tw);
    int nct, w;
    cross_cols(p, n, maxw, nct, w);
    return quot(cross_rows(p, n, compact) + 2 * hrows - 1, 2 * hrows) * nct;
}
template <bool SPLIT>
__device__ __forceinline__ bool decode_tile(const GramProblem& p, const Plan& pl, int id, Piece& t) {
    constexpr int MAXW = Stage<SPLIT>::MAXW;
    const int hrows = pl.hrows, tw = pl.tw;
    const bool compact = pl.compact != 0;
    for (int b = 0; b < p.B; ++b) {
        const int n = seq_n(p, pl, b);
        const int cnt = seq_tiles(p, n, MAXW, tw, hrows, compact);
        if (id >= cnt) { id -= cnt; continue; }
        t.b = b;
        t.n = n;
        int nc;
        if (p.tri) {
            const int f = tw == PM ? 1 : 2, M = (n + PM - 1) / PM;
            int mi = M - 1;
            if (id < f * (M * (M - 1) / 2)) {
                mi = (int)((sqrtf(8.0f * (float)(f == 1 ? id : id >> 1) + 1.0f) - 1.0f) * 0.5f);
                while (f * (mi * (mi + 1) / 2) > id) --mi;
                while (f * ((mi + 1) * (mi + 2) / 2) <= id) ++mi;
            }
            t.row0 = mi * PM;
            t.col0 = (id - f * (mi * (mi + 1) / 2)) * tw;
            t.m = n;
            nc = min(n - t.col0, tw);
        } else {
            int nct, w;
            cross_cols(p, n, MAXW, nct, w);
            const int q = quot(id, nct);
            t.row0 = q * 2 * hrows;
            t.col0 = (id - q * nct) * w;
            t.m = cross_rows(p, n, compact);
            nc = min(n - t.col0, w);
        }
        t.ncols = max(32, (nc + 31) & ~31);
        return true;
    }
    return false;
}
// per-CTA stage: the CTA's rows of A (a_bytes per 64-element K block, a multiple of 1024) and
// ncols/2 rows of B (in 64-row boxes, a 32-row one at the end where that is enough)
__device__ __forceinline__ int a_bytes_of(int hrows) { return (hrows * 128 + 1023) & ~1023; }
__device__ __forceinline__ int sub_bytes_pair(int a_bytes, int ncols) {
    const int half = ncols >> 1, rest = half % BOX_N;
    return a_bytes + half / BOX_N * BOX_BYTES + (rest == 0 ? 0 : (rest <= 32 ? BOX_BYTES / 2 : BOX_BYTES));
}
// Row norms of the cross segment's left operand (inv_out).  When one column tile covers all
// columns every row tile is loaded exactly once and the launch is bound by streaming them: the
// norms are then taken from the tiles in shared memory (`from_smem`; the stage release waits for
// the readers, which costs nothing while the tensor pipe idles).  With several column tiles the
// main loops are bound by the tensor pipe and by what an SM can draw from L2, a stage release
// that waits for readers slows them, and warps 2..9 read the rows with plain loads
// instead (X then stays resident in L2 between the column tiles anyway).
__device__ __forceinline__ bool norm_duty(const GramProblem& p, int col0, bool from_smem) {
    return from_smem && !p.tri && p.inv_out != nullptr && col0 == 0;
}
// Under ADA_CROSS_CAUSAL a cross tile whose first (lowest) column token is not below the
// tile's last row has no admissible (row, column) pair: every role skips it, so neither
// its loads nor its MMAs are issued.  Column tokens ascend with the column index.  (A tile
// that has to yield row norms is never skipped.)
__device__ __forceinline__ bool dead_tile(const GramProblem& p, const Piece& pc, int hrows, bool from_smem,
                                          bool compact) {
    if (p.tri || !p.causal || p.col_token == nullptr || pc.n <= 0 || norm_duty(p, pc.col0, from_smem)) return false;
    if (compact) return false;     // rows are compacted there: a row index is not a token index
    return p.col_token[(int64_t)pc.b * p.cap + pc.col0] >= pc.row0 + 2 * hrows;
}

struct GramMaps {
    CUtensorMap a[2];        // left operand, 128-row boxes
    CUtensorMap b[2], bt[2]; // right operand in 64-row boxes, and in 32-row boxes for a half-empty last one
    CUtensorMap ah;          // left operand of the cross segment in boxes of hb_rows rows
    CUtensorMap an;          // the rows outside a large inherited set (Xnon), 128-row boxes
};

// ---------------------------------------------------------------- work plan
// Tiles are dealt round-robin to the pairs.  What does not fill a last round -- everything, in a
// small problem -- is cut along K: each of its `rem` tiles goes to `parts` pairs, which exchange
// partial accumulators through L2 (see the epilogue): a pair's share shrinks from the whole
// chain to a part of it, and a wide tile split over K draws fewer bytes per SM than narrow tiles
// would.  Measured: full selection at T = 2048, d = 4096 31.0 -> 26.1 us, at T = 512, d = 768 fp32 30.2 ->
// 17.7 us, cascade steps at T = 2005, d = 4096 43 -> 31 us.
// How many shares a tile may have.  The tensor core's accumulator truncates, so a sum over d elements comes out too small,
// and cutting it in p shares takes part of that away: the same row moves by as much when the number of tiles around it
// changes, the split sum being the better one.  That is to stay below 1.5e-5 for bf16 (1e-5 for the six terms of fp32
// storage, whose contraction is cut earlier) whatever the scale of the rows.
// An accumulation loses in proportion to the unit in the last place of the running sum, so with elements of one scale a
// whole sum loses e d f of itself, f = 1/s - 2/(3 s^2) for a sum that ends at s (1 <= s < 2) in its binade: 1/3 at
// its ends, 3/8 at s = 4/3.  A share ends p times lower, at f': the row moves by e d (f - f'/p), at worst
// 0.19, 0.26, 0.28 e d for p = 2, 3, 4, which is 3/8 e d (1 - 1/p) within a few per cent, hence one limit on d (1 - 1/p).
// Measured e = 1.2e-8 .. 1.38e-8; largest shifts over rows of scale 0.7 .. 1.3: 1.32e-5 (d = 5120, p = 2), 1.34e-5 (4096, 3),
// 1.23e-5 (3640, 4); fp32 7.6e-6 (2136, 2), 6.9e-6 (1600, 3), 7.0e-6 (1424, 4).  Error against 64 bits at d = 4096: 4.3e-6 in
// three shares, 1.7e-5 whole.
template <bool SPLIT>
__device__ __forceinline__ bool shares_ok(int p, int d) {
    return (p - 1) * d <= (SPLIT ? MAX_SPLIT_D_F32 : MAX_SPLIT_D) / 2 * p;
}
// Limits of the plan's rules in stages of a bf16 tile: what a split has to save, the longest contraction whose
// norms come out of the tiles in shared memory, the longest whose epilogue sets take alternate tiles.  The last
// two count on whole tiles (ring_s below, the shares of pub_cnt): what they cover is never split.
constexpr int SPLIT_SAVES = 10, SMEM_NORM_STAGES = 8, ALT_STAGES = 12;
static_assert(ALT_STAGES - (ALT_STAGES + MAX_PARTS - 1) / MAX_PARTS < SPLIT_SAVES && SMEM_NORM_STAGES <= ALT_STAGES,
              "tiles read by alternate sets, or for their norms, are whole");
template <bool SPLIT>
__device__ __noinline__ void make_plan(Plan& pl, const GramProblem& seg0, const GramProblem& seg1, int nseg,
                                          bool maybe_compact, int npairs, int max_parts, int lane) {
    constexpr int MAXW = Stage<SPLIT>::MAXW;
    const GramProblem& cx = nseg > 1 ? seg1 : seg0;
    // both segments of a launch share the sequences: one read of every length
    bool one = !cx.tri, big = true;
    for (int b = lane; b < cx.B; b += 32) {
        const int n = seq_n_global(cx, b);
        if (b < PLAN_B) pl.len[b] = n;
        one = one && n <= MAXW;
        big = big && 5 * (int64_t)n >= 2 * (int64_t)cx.rows;
    }
    one = __all_sync(0xffffffffu, one);
    big = __all_sync(0xffffffffu, big);
    // streaming form: one column tile covers the columns of every sequence and the rows are many,
    // so the launch is one pass over the rows of A, and shorter row tiles put every pair to work.
    // Below 48 rows per CTA the right operand would be most of the traffic and splitting K is cheaper.  d = 4096,
    // 2 % representatives, new rows at every call, split against streaming form: T = 4096 (28 rows) 28.4
    // and 30.3 us, 6000 (41) 33.8 and 34.8, 7200 (50) 36.2 and 35.1, 8192 (57) 38.6 and 36.6, 10000 (69)
    // 43.8 and 40.7.  (With an X that the call before left in L2 the lines cross at 64 rows: 31.8 and
    // 36.1 at T = 8192.)
    const bool stream = !SPLIT && one && cx.hb_rows >= 48;
    const int hrows = stream && cx.hb_rows < BM ? cx.hb_rows : BM;
    const bool compact = !SPLIT && maybe_compact && big && !one;       // (compact_wanted)
    __syncwarp();
    int t256 = 0, t128 = 0, tc = 0;                 // triangular tiles by width, cross tiles
    for (int b = lane; b < cx.B; b += 32) {
        const int n = cx.B <= PLAN_B ? pl.len[b] : seq_n_global(cx, b);
        if (seg0.tri) { t256 += tri_tiles(n, PM); t128 += tri_tiles(n, BM); }
        if (!cx.tri) tc += seq_tiles(cx, n, MAXW, PM, hrows, compact);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        t256 += __shfl_xor_sync(0xffffffffu, t256, o);
        t128 += __shfl_xor_sync(0xffffffffu, t128, o);
        tc += __shfl_xor_sync(0xffffffffu, tc, o);
    }
    // The number of shares, for both widths of the triangular tiles at once: lane 8 w + q asks whether
    // q + 1 shares are possible with width w.  (Integer divisions are slow and the plan is on the
    // path to the first copy.)
    const int nst = ((SPLIT ? cx.planes : cx.d) + Stage<SPLIT>::K - 1) / Stage<SPLIT>::K;
    const int cand = (lane & 8) ? t128 + tc : t256 + tc, q1 = (lane & 7) + 1;
    const int rounds = quot(cand, npairs), rem = cand - rounds * npairs;
    // the exchange costs about 5 us: as much as six stages of fp32 planes, ten of bf16 (SPLIT_SAVES)
    const bool can = q1 == 1 || (!stream && q1 <= max_parts && shares_ok<SPLIT>(q1, cx.d) && rem > 0 && q1 * rem <= npairs && 2 * q1 <= nst &&
                                 nst - quot(nst + q1 - 1, q1) >= (SPLIT ? 6 : SPLIT_SAVES));
    const unsigned cans = __ballot_sync(0xffffffffu, can);
    const int parts256 = 32 - __clz(cans & 0xffu), parts128 = 32 - __clz((cans >> 8) & 0xffu);
    const int rounds256 = __shfl_sync(0xffffffffu, rounds + (rem > 0), 0), rounds128 = __shfl_sync(0xffffffffu, rounds + (rem > 0), 8);
    // cross epilogues wait for the triangle: half-width triangular tiles are done earlier, where that
    // costs neither a round nor a finer split
    const bool narrow = SPLIT || (nseg > 1 && rounds128 == rounds256 && parts128 >= parts256);
    const int the_rem = __shfl_sync(0xffffffffu, rem, narrow ? 8 : 0);
    if (lane == 0) {
        const int tiles0 = seg0.tri ? (narrow ? t128 : t256) : tc;
        const int total = nseg > 1 ? tiles0 + tc : tiles0;
        pl.tiles0 = tiles0; pl.total = total; pl.tw = narrow ? BM : PM; pl.hrows = hrows;
        // Norms out of the tiles in shared memory also for 385 to 1024 elements and at most two tiles a pair, where
        // the plain loads hold the epilogues up more than a late stage release does: steps over 4096 x 768,
        // r = 410, 19.5 -> 18.8 us, 4 x 2048 x 768, r = 410, 27.1 -> 25.6, 2 x 2048 x 512 18.9 -> 18.5; at
        // 1024 elements even (20.7), at 1536 slower (22.0 -> 23.7).
        pl.smem_norms = stream ? 2 : (!SPLIT && !cx.tri && nst >= 4 && nst <= SMEM_NORM_STAGES && total <= 2 * npairs && !compact) ? 1 : 0;
        pl.compact = compact ? 1 : 0;
        // Short contractions, many tiles: a tile's main loop is as short as the bookkeeping of its
        // epilogue (column factors, barriers, atomics: dependent round trips), so the two sets of
        // four warps take alternate tiles, one accumulator each, and one set's bookkeeping runs beside
        // the other's reading.  Otherwise both read every tile and its maxima are there sooner.  Steps, both
        // reading against alternating: 2 x 8192 x 768, r = 819, 39.7 -> 36.6 us; 8192 x 1024, r = 1638, 38.9 ->
        // 38.3; at 1536 elements, the longest that alternates, 46.0 -> 46.7.
        pl.alt = Stage<SPLIT>::ALT && !pl.smem_norms && nst <= ALT_STAGES && total > 2 * npairs ? 1 : 0;
        pl.parts = narrow ? parts128 : parts256;
        pl.rem = pl.parts > 1 ? the_rem : 0;
        pl.full = total - pl.rem;
    }
}
// Work item of a pair: a tile, or one share of a split tile's contraction, with all that the roles need to
// know about it.
struct alignas(16) Item {
    int row0, col0, ncols, b;   // ncols: multiple of 32
    int n, m, st0, st1;         // columns of the sequence, row bound, K stages [st0, st1)
    int kind;                   // 0: no more work, 1: tile, 2: nothing to do (dead tile)
    int seg, part, parts;
    int unit0;                  // first exchange slot of a split tile
    int ring;                   // stages of the ring at this tile's stage size
    int pad[2];
};
constexpr int ITEMS = 32;       // items decoded ahead, one per lane; later ones on the fly

// (200 KiB hold as many bf16 stages of every width as 208 would; the rest is column factors.)
template <bool SPLIT> struct Ring { static constexpr int BYTES = (SPLIT ? 216 : 200) * 1024; };

// Not inlined: the decoding is a few hundred instructions of integer arithmetic that would sit in
// the path of every role; run once, by 32 lanes side by side, it is read from shared memory.
template <bool SPLIT>
__device__ __noinline__ void decode_item(const GramProblem* seg0, const GramProblem* seg1, const Plan& pl, int pair,
                                         int npairs, int it, Item& w) {
    const int at = pair + it * npairs;
    int id = at, part = 0, parts = 1;
    w.kind = 0;
    if (at >= pl.full) {                            // pl.full is a multiple of npairs when anything is split
        const int u = at - pl.full;
        parts = pl.parts;
        if (u >= pl.rem * parts) return;
        const int tile = quot(u, parts);
        id = pl.full + tile;
        part = u - tile * parts;
    }
    const int sg = id < pl.tiles0 ? 0 : 1;
    const GramProblem& p = sg ? *seg1 : *seg0;
    Piece t;
    if (!decode_tile<SPLIT>(p, pl, id - (sg ? pl.tiles0 : 0), t)) return;
    const int nst = ((SPLIT ? p.planes : p.d) + Stage<SPLIT>::K - 1) / Stage<SPLIT>::K;
    w.row0 = t.row0; w.col0 = t.col0; w.ncols = t.ncols; w.b = t.b; w.n = t.n; w.m = t.m;
    w.st0 = 0; w.st1 = nst;
    if (parts > 1) { w.st0 = quot(nst * part, parts); w.st1 = quot(nst * (part + 1), parts); }
    w.seg = sg; w.part = part; w.parts = parts; w.unit0 = (id - pl.full) * parts;
    const int a_bytes = a_bytes_of(p.tri ? BM : pl.hrows);
    // the MMA reads 128 rows of A whatever was loaded: what it reads past a shorter tile stays inside the ring
    const int room = Ring<SPLIT>::BYTES - (A_BYTES - a_bytes), sb = Stage<SPLIT>::NSUB * sub_bytes_pair(a_bytes, t.ncols);
    w.ring = 0;
#pragma unroll
    for (int q = 1; q <= MAX_STAGES; ++q) w.ring += q * sb <= room;
    w.kind = dead_tile(p, t, pl.hrows, pl.smem_norms != 0, pl.compact != 0) ? 2 : 1;
}

// ---------------------------------------------------------------- the kernel
template <bool SPLIT>
struct alignas(16) SharedPair {
    unsigned long long full[MAX_STAGES];
    unsigned long long empty[MAX_STAGES];
    unsigned long long consumed[MAX_STAGES];   // MMAs of a norm-duty stage retired: its A tile may be read
    unsigned long long tmem_full[2];
    unsigned long long tmem_empty[2];
    unsigned long long drain;
    unsigned long long planned;                // the work plan is in shared memory
    // global counters seen complete by the thread that polls them for the CTA (for an epilogue set, where
    // those take alternate tiles): preparation, row norms, triangle
    unsigned long long prep_seen, norm_seen[SUBS], dep_seen[SUBS];
    unsigned pub_cnt;                          // epilogue warps that have published their share of a triangular tile
    unsigned tmem_base;
    int abort_flag[2];                         // why the CTA gives up (0: it does not); limit of its waits
    unsigned norm_cnt[MAX_STAGES];             // norm warps done with a stage
    unsigned long long normed;                 // the sums of squares of a tile's rows are in norm_part
    float norm_part[2][SUBS][BM];              // by tile parity and set
    Plan plan;
    // the launch's arguments once more: what is not inlined takes them by reference, and reading the
    // parameter space through a pointer is a trip to memory
    GramProblem seg[2];
    SplitJob split;
    GatherJob gather;
    NormJob norms;
    Item item[ITEMS];
    // column factors of a tile, per epilogue set (the chunks that it reads), in alternating buffers: each of
    // the set's four warps stages a quarter, `staged` completes when all have.  A warp is never more
    // than one tile ahead of another.
    unsigned long long staged[SUBS];
    alignas(16) float col_scale[SUBS][2][Stage<SPLIT>::COLS];
    alignas(16) int col_token[SUBS][2][Stage<SPLIT>::COLS];
};
template <bool SPLIT>
constexpr int smem_pair_bytes() { return Ring<SPLIT>::BYTES + (int)sizeof(SharedPair<SPLIT>) + 1024; }
static_assert(smem_pair_bytes<false>() <= 227 * 1024 && smem_pair_bytes<true>() <= 227 * 1024, "shared memory budget");
// partial accumulators: [tile][source part][CTA of the pair][32-column chunk][8 16-byte columns][128 rows]
constexpr int CHUNK_WORDS = BM * 32;
__device__ __forceinline__ int64_t chunk_at(int unit, int rank, int chunk) {
    return (((int64_t)unit * 2 + rank) * (BN / 32) + chunk) * CHUNK_WORDS;
}

// Adds one thread's 32 partial sums at src (16-byte columns, BM apart) to r once they have arrived, and
// marks the place empty again for the next launch.  An empty word holds a NaN pattern that no
// sum can produce, so every word says for itself whether it is there: no fence, no flag and no
// second round trip between the writer and the reader.
constexpr unsigned EMPTY_WORD = 0xFFFFFFFFu;
__device__ __forceinline__ void load_partials(const uint4* src, uint4 (&x)[8]) {
#pragma unroll
    for (int e = 0; e < 8; ++e)
        asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(x[e].x), "=r"(x[e].y), "=r"(x[e].z), "=r"(x[e].w) : "l"(src + e * BM) : "memory");
}
__device__ __forceinline__ bool take_partials(uint4* src, uint4 (&x)[8], unsigned (&r)[32], volatile int* abort_flag) {
    unsigned polls = 0;
    unsigned long long t0 = 0;
    while (true) {
        bool there = true;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            there = there && x[e].x != EMPTY_WORD && x[e].y != EMPTY_WORD && x[e].z != EMPTY_WORD && x[e].w != EMPTY_WORD;
        if (there) break;
        if ((++polls & 255u) == 0) {
            if (*abort_flag != 0) return false;
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (past_limit(now - t0, abort_flag)) { *abort_flag = 16; return false; }
        }
        load_partials(src, x);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        r[4 * e] = __float_as_uint(__uint_as_float(r[4 * e]) + __uint_as_float(x[e].x));
        r[4 * e + 1] = __float_as_uint(__uint_as_float(r[4 * e + 1]) + __uint_as_float(x[e].y));
        r[4 * e + 2] = __float_as_uint(__uint_as_float(r[4 * e + 2]) + __uint_as_float(x[e].z));
        r[4 * e + 3] = __float_as_uint(__uint_as_float(r[4 * e + 3]) + __uint_as_float(x[e].w));
        __stcg(src + e * BM, make_uint4(EMPTY_WORD, EMPTY_WORD, EMPTY_WORD, EMPTY_WORD));
    }
    return true;
}

template <typename T>
__device__ __forceinline__ void copy_args(T& dst, const T& src, int i, int n) {
    static_assert(sizeof(T) % 8 == 0, "copied in 8-byte words");
    for (; i < (int)(sizeof(T) / 8); i += n)
        reinterpret_cast<unsigned long long*>(&dst)[i] = reinterpret_cast<const unsigned long long*>(&src)[i];
}

// The copies of one tile in the streaming form: every row of the left operand is copied once per
// launch, so its lines are the first to leave L2.  Left to the default, a pass over an X larger than
// L2 threw out all that the next launch starts with -- code, right operand, arguments (step over
// T = 16384, d = 4096 with new rows each time: 45.5 -> 42.5 us; 4 x 4096: 41.5 -> 38.4;
// 8 x 2000, d = 1536: 26.9 -> 24.8).  Not inlined and rolled: the same loop beside, or with a
// choice of policy inside, the common one cost the pipelines 1-2 %.
struct Fed { unsigned fills, used; int s; bool ok; };
template <bool SPLIT>
__device__ __noinline__ Fed feed_once(const CUtensorMap* amap, const CUtensorMap* bmap, const CUtensorMap* btail,
                                      unsigned long long* full, unsigned long long* empty, volatile int* abort_flag,
                                      unsigned char* smem, int subb, int a_bytes, unsigned tx, int nbox, bool tail32,
                                      int a_row, int b_row, int wb, int nst, int ring, int s, unsigned fills) {
    unsigned long long policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    Fed f{fills, 0u, s, true};
    for (int st = 0; st < nst; ++st) {
        if (!mbar_wait(&empty[f.s], ((f.fills >> f.s) & 1u) ^ 1u, abort_flag, 1)) { f.ok = false; break; }
        unsigned char* su = smem + f.s * Stage<SPLIT>::NSUB * subb;
        if (tx != 0) mbar_expect_tx(&full[f.s], tx);
#pragma unroll 1
        for (int u = 0; u < Stage<SPLIT>::NSUB; ++u, su += subb) {
            const int k0 = st * Stage<SPLIT>::K + u * BK;
            tma_load_3d_pair_once(amap, &full[f.s], su, k0, a_row, wb, policy);
#pragma unroll 1
            for (int j = 0; j < nbox; ++j)
                tma_load_3d_pair(j == nbox - 1 && tail32 ? btail : bmap, &full[f.s], su + a_bytes + j * BOX_BYTES,
                                 k0, b_row + j * BOX_N, wb);
        }
        f.fills ^= 1u << f.s; f.used |= 1u << f.s;
        f.s = (f.s + 1 == ring) ? 0 : f.s + 1;
    }
    return f;
}

template <bool SPLIT>
__global__ void __launch_bounds__(PAIR_THREADS, 1)
k_gram_tc2(const __grid_constant__ GramMaps maps, const __grid_constant__ GramProblem seg0,
           const __grid_constant__ GramProblem seg1, const int nseg,
           const __grid_constant__ NormJob norms, const __grid_constant__ GatherJob gather,
           const __grid_constant__ SplitJob split, const int max_parts, const int wait_limit, unsigned* __restrict__ part_buf,
           unsigned* __restrict__ dep_ctr, unsigned* __restrict__ status) {
    using St = Stage<SPLIT>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    SharedPair<SPLIT>& sh = *reinterpret_cast<SharedPair<SPLIT>*>(smem + Ring<SPLIT>::BYTES);
    volatile int* abort_flag = sh.abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned rank = cluster_rank();            // 0 = leader
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(&sh.full[s], 1);
            mbar_init(&sh.empty[s], 1);
            mbar_init(&sh.consumed[s], 1);
            sh.norm_cnt[s] = 0u;
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&sh.tmem_full[a], 1);
            mbar_init(&sh.tmem_empty[a], 2 * EPI_WARPS);     // the epilogue warps of both CTAs
        }
        mbar_init(&sh.drain, 1);
        mbar_init(&sh.planned, 1);
        mbar_init(&sh.prep_seen, 1);
        mbar_init(&sh.normed, EPI_WARPS);
        for (int q = 0; q < SUBS; ++q) mbar_init(&sh.staged[q], 4);
        for (int q = 0; q < SUBS; ++q) { mbar_init(&sh.norm_seen[q], 1); mbar_init(&sh.dep_seen[q], 1); }
        sh.pub_cnt = 0u;
        sh.abort_flag[0] = 0;
        sh.abort_flag[1] = wait_limit;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sh.tmem_base)), "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    if (warp >= 2) {
        const int i = (int)threadIdx.x - 64, n = 32 * EPI_WARPS;
        copy_args(sh.seg[0], seg0, i, n);
        copy_args(sh.seg[1], seg1, i, n);
        if constexpr (SPLIT) copy_args(sh.split, split, i, n);
        else if (gather.X != nullptr) copy_args(sh.gather, gather, i, n);
        if (i == 0) {
            const GramProblem& cx = (nseg > 1) ? seg1 : seg0;
            if (norms.X != nullptr) {
                sh.norms = norms;
            } else {                                 // cascade step: the left operand of the cross segment
                sh.norms.X = cx.A; sh.norms.ldx = cx.lda; sh.norms.n_rows = (int64_t)cx.B * cx.rows; sh.norms.d = cx.d;
                sh.norms.inv_norm = cx.inv_out;
                sh.norms.batch = cx.a_batch; sh.norms.rows_per_seq = cx.rows;
            }
        }
    }
    if (threadIdx.x == 32) {                         // descriptors are fetched before the first copy needs them
        prefetch_map(&maps.a[0]); prefetch_map(&maps.b[0]); prefetch_map(&maps.bt[0]);
        prefetch_map(&maps.a[1]); prefetch_map(&maps.b[1]); prefetch_map(&maps.bt[1]);
        prefetch_map(&maps.ah); prefetch_map(&maps.an);
    }
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();          // the peer's barriers exist before anything signals them
    tcgen05_fence_after();
    const unsigned tmem_base = sh.tmem_base;
    const bool has_prep = SPLIT ? split.X != nullptr : gather.X != nullptr;
    // The work plan: before the predecessor's results are waited for where it does not depend on them (full
    // selection, T = 2048, d = 4096: 26.3 -> 25.2 us; one-CTA kernel, T = 512, d = 768: 14.1 -> 13.1).
    auto plan_work = [&]() {
        const bool maybe_compact = gather.X != nullptr && gather.Xnon != nullptr && gather.T >= gather.compact_min_rows;
        make_plan<SPLIT>(sh.plan, sh.seg[0], sh.seg[1], nseg, maybe_compact, npairs, max_parts, lane);
        __syncwarp();
        decode_item<SPLIT>(&sh.seg[0], &sh.seg[1], sh.plan, pair, npairs, lane, sh.item[lane]);
        __syncwarp();
        if (lane == 0) { __threadfence_block(); mbar_arrive(&sh.planned); }
        __syncwarp();
    };
    const bool early = (nseg > 1 ? seg1 : seg0).n_dev == nullptr;
    if (early && warp == 0) plan_work();
    // everything above is local to the CTA; from here on the predecessor's results are read
    grid_dep_wait();
    // (the compaction's blocks may take the SMs that fall idle first: they wait for this whole grid)
    grid_dep_launch_next();
    if (has_prep && warp >= 2) {
        // ------------------------------------------------ preparation, by every warp that is idle at
        // the start.  Items are dealt across the SMs first, so that a
        // short list is read by all of them.  One arrival per CTA.
        const int g = (warp - 2) * (int)gridDim.x + (int)blockIdx.x, nw = (int)gridDim.x * EPI_WARPS;
        if constexpr (!SPLIT) gather_rows(gather, sh.gather, g, nw, lane, status);
        else split_rows(sh.split, g, nw, lane, status);
        // the rows just written are read by TMA (async proxy) from other CTAs
        // (one fence for the whole device per CTA, after the barrier: it covers what the barrier ordered
        // before it)
        asm volatile("fence.proxy.async.global;" ::: "memory");
        asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
        if (threadIdx.x == 64) {
            __threadfence();
            atomicAdd(dep_ctr + 3, 1u);
        }
    }
    const unsigned prep_total = gridDim.x;
    if (!early && warp == 0) plan_work();
    // (made by warp 0 of the same CTA, which waits for nobody)
    const bool planned = __all_sync(0xffffffffu, mbar_wait(&sh.planned, 0, abort_flag, 18));
    const Plan& pl = sh.plan;
    const int tiles0 = pl.tiles0;
    const int hrows = pl.hrows;                          // rows per CTA of a cross tile
    const bool smem_norms = pl.smem_norms != 0;        // row norms out of the tiles in shared memory
    const bool compact = pl.compact != 0;                // cross tiles over the copied-out rows (Xnon)
    Item own;                                            // an item beyond the table

    auto item_at = [&](int it) __attribute__((always_inline)) -> const Item& {
        if (it < ITEMS) return sh.item[it];
        decode_item<SPLIT>(&sh.seg[0], &sh.seg[1], pl, pair, npairs, it, own);
        return own;
    };
    if (!planned) {
        // no work: on to the end, where the status is raised
    } else if (warp == 0) {
        // ------------------------------------------------ TMA producer (both CTAs)
        if (lane == 0) {
            unsigned fills = 0, used = 0, ever = 0;
            int cur_sb = 0, cur_nst = 0, s = 0;
            bool ok = true, prep_ok = !has_prep;
            for (int it = 0; ok; ++it) {
                const Item& w = item_at(it);
                if (w.kind == 0) break;
                if (w.kind == 2) continue;
                const int sg = w.seg;
                const GramProblem& p = sg ? seg1 : seg0;
                const int half = w.ncols >> 1, st0 = w.st0, st1 = w.st1, wb = w.b;
                // whole 64-row boxes, and for the rest a 32- or a 64-row one
                const int nbox = (half + BOX_N - 1) / BOX_N, rest = half % BOX_N;
                const bool tail32 = rest != 0 && rest <= 32;
                const int arows = p.tri ? BM : hrows;
                const int a_bytes = a_bytes_of(arows);
                const int subb = sub_bytes_pair(a_bytes, w.ncols);
                const int sb = St::NSUB * subb;
                const unsigned tx = (unsigned)(St::NSUB * (arows * 128 + nbox * BOX_BYTES - (tail32 ? BOX_BYTES / 2 : 0)));
                const CUtensorMap* amap = p.tri ? &maps.a[sg] : (compact ? &maps.an : (hrows != BM ? &maps.ah : &maps.a[sg]));
                if (sb != cur_sb) {
                    for (int q = 0; q < cur_nst && ok; ++q)
                        if ((used >> q) & 1u)
                            ok = mbar_wait(&sh.empty[q], ((fills >> q) & 1u) ^ 1u, abort_flag, 6);
                    if (!ok) break;
                    cur_sb = sb; cur_nst = w.ring; s = 0; used = 0;
                }
                const int a_row = w.row0 + (int)rank * arows;
                const int b_row = w.col0 + (int)rank * half;
                const int kstep = SPLIT ? p.planes : BK;          // from one sub-tile of a stage to the next
                if (!prep_ok) {
                    // the right operand (and the triangle's left operand) is made by the preparation;
                    // all of the above is ready by the time that ends
                    ok = wait_counter_1(dep_ctr + 3, prep_total, abort_flag, 12);
                    mbar_arrive(&sh.prep_seen);
                    asm volatile("fence.proxy.async.global;" ::: "memory");
                    prep_ok = true;
                    if (!ok) break;
                }
                if constexpr (!SPLIT) if (pl.smem_norms == 2 && !p.tri) {
                    // (streaming form: no share of K is cut, st0 = 0)
                    const Fed f = feed_once<SPLIT>(amap, &maps.b[sg], &maps.bt[sg], sh.full, sh.empty, abort_flag, smem,
                                            subb, a_bytes, rank == 0 ? 2u * tx : 0u, nbox, tail32, a_row, b_row, wb, st1, cur_nst, s, fills);
                    fills = f.fills; s = f.s; ok = f.ok;
                    used |= f.used; ever |= f.used;
                    continue;
                }
                for (int st = st0; st < st1; ++st) {
                    if (!mbar_wait(&sh.empty[s], ((fills >> s) & 1u) ^ 1u, abort_flag, 1)) { ok = false; break; }
                    unsigned char* sa = smem + s * sb;
                    // the leader's barrier counts the bytes of both CTAs
                    if (rank == 0) mbar_expect_tx(&sh.full[s], 2u * tx);
                    // K past the operand is zero-filled by the TMA unit (planes are padded with zeros)
#pragma unroll
                    for (int u = 0; u < St::NSUB; ++u) {
                        unsigned char* su = sa + u * subb;
                        const int k0 = st * St::K + u * kstep;
                        tma_load_3d_pair(amap, &sh.full[s], su, k0, a_row, wb);
                        for (int j = 0; j < nbox; ++j)
                            tma_load_3d_pair(j == nbox - 1 && tail32 ? &maps.bt[sg] : &maps.b[sg], &sh.full[s],
                                             su + a_bytes + j * BOX_BYTES, k0, b_row + j * BOX_N, wb);
                    }
                    fills ^= 1u << s; used |= 1u << s; ever |= 1u << s;
                    s = (s + 1 == cur_nst) ? 0 : s + 1;
                }
            }
            // drain: a stage's release (empty) implies its copy landed and was consumed
            for (int q = 0; q < MAX_STAGES; ++q) {
                if (!((ever >> q) & 1u)) continue;
                const unsigned ph = ((fills >> q) & 1u) ^ 1u;
                const unsigned long long t0 = global_ns();
                while (!mbar_try(&sh.empty[q], ph)) {
                    if (*abort_flag != 0 || past_limit(2 * (global_ns() - t0), abort_flag)) { *abort_flag = 7; break; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer (leader CTA only)
        if (lane == 0 && rank == 0) {
            unsigned uses = 0, tile_it = 0;
            int cur_sb = 0, cur_nst = 0, s = 0;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                const Item& w = item_at(it);
                if (w.kind == 0) break;
                if (w.kind == 2) continue;
                const GramProblem& p = w.seg ? seg1 : seg0;
                const int st0 = w.st0, st1 = w.st1;
                const int a_bytes = a_bytes_of(p.tri ? BM : hrows);
                const int subb = sub_bytes_pair(a_bytes, w.ncols);
                const int sb = St::NSUB * subb;
                if (sb != cur_sb) { cur_sb = sb; cur_nst = w.ring; s = 0; }
                const bool duty = norm_duty(p, w.col0, smem_norms);
                const unsigned acc = tile_it & 1u, acc_ph = (tile_it >> 1) & 1u;
                ++tile_it;
                if (!mbar_wait(&sh.tmem_empty[acc], acc_ph ^ 1u, abort_flag, 2)) { ok = false; break; }
                tcgen05_fence_after();
                const unsigned idesc = instr_desc_pair(w.ncols);
                const unsigned d_tmem = tmem_base + acc * BN;
                for (int st = st0; st < st1; ++st) {
                    if (!mbar_wait(&sh.full[s], (uses >> s) & 1u, abort_flag, 3)) { ok = false; break; }
                    tcgen05_fence_after();
                    const unsigned s_addr = smem_u32(smem + s * sb);
#pragma unroll
                    for (int t = 0; t < St::TERMS; ++t) {
                        const unsigned long long adesc = smem_desc_sw128(s_addr + St::ta(t) * subb);
                        const unsigned long long bdesc = smem_desc_sw128(s_addr + St::tb(t) * subb + a_bytes);
#pragma unroll
                        for (int k = 0; k < BK / UMMA_K; ++k)
                            umma_bf16_pair(d_tmem, adesc + 2 * k, bdesc + 2 * k, idesc, ((st - st0) | t | k) != 0);
                    }
                    // both producers may refill this stage -- after the norm warps have read the
                    // A tiles, where those yield the row norms
                    umma_commit_pair_both(duty ? &sh.consumed[s] : &sh.empty[s]);
                    uses ^= 1u << s;
                    s = (s + 1 == cur_nst) ? 0 : s + 1;
                }
                if (ok) umma_commit_pair_both(&sh.tmem_full[acc]);   // both epilogues may read
            }
            umma_commit_pair_local(&sh.drain);
            const unsigned long long t0 = global_ns();
            while (!mbar_try(&sh.drain, 0)) {
                if (past_limit(2 * (global_ns() - t0), abort_flag)) { *abort_flag = 8; break; }
            }
        }
    } else {
        // ------------------------------------------------ warps 2..9, both CTAs: row norms of X where
        // the launch makes them, then the epilogue.  A warp reaches the TMEM lanes 32 (warp % 4)..;
        // the two warps of a lane quadrant share a tile's 32-column chunks (sub, sub + 2, ..), so
        // that a finished accumulator is read out by eight warps.
        const int quad = warp & 3, sub = (warp - 2) >> 2;
        unsigned n_staged = 0;                       // tiles of this set so far
        const GramProblem& cx = (nseg > 1) ? seg1 : seg0;
        // 1/||x_t|| of every row of X with plain loads, behind the first main loops.  Full selection: at once, the
        // epilogues need them.  Cascade step with several column tiles: nothing in this launch waits
        // for them (the row factor is applied by the compaction), but everything waits for the
        // triangle, so its tiles go first.
        bool norms_due = norms.X != nullptr || (!cx.tri && cx.inv_out != nullptr && !smem_norms && !compact);
        // row norms out of the A tiles in shared memory (streaming form): thread lrow owns row lrow of the CTA's
        // tile, set `sub` the stage's K block `sub`, and both follow the ring exactly as the producer
        // fills it.  (The stage goes back to the producer behind them: with one set reading both K
        // blocks the ring turned over in 1.06 us per stage at T = 16384, r = 164.)
        static_assert(SPLIT || SUBS == St::NSUB, "a set per K block of a stage");
        const bool ring_norms = !SPLIT && smem_norms && !cx.tri && cx.inv_out != nullptr;
        unsigned n_normed = 0;
        unsigned cons = 0;
        int ring_sb = 0, ring_nst = 0, ring_s = 0;
        // every share of a triangular tile is published once by both CTAs
        const unsigned dep_total = 2u * (unsigned)(min(tiles0, pl.full) + max(tiles0 - pl.full, 0) * pl.parts);
        bool dep_ok = !(nseg > 1 && tiles0 > 0);
        bool norm_ok = norms.X == nullptr;           // row norms computed by this launch's norm warps
        bool prep_ok = !has_prep;
        const unsigned norm_total = (unsigned)(gridDim.x * EPI_WARPS);
        // the accumulator goes back to the leader's barrier
        const unsigned empty_addr[2] = {map_to_cta(smem_u32(&sh.tmem_empty[0]), 0),
                                        map_to_cta(smem_u32(&sh.tmem_empty[1]), 0)};
        const bool alt = pl.alt != 0;
        // Wait for a counter of the whole grid.  One thread per CTA (or epilogue set) polls it and the other warps wait in
        // shared memory: with every warp polling, the polls alone saturate the counter's L2 slice
        // and delay the very arrivals that they wait for (up to 9 us before the cross epilogues).
        auto await = [&](const unsigned* ctr, unsigned target, unsigned long long* seen, int where)
                         __attribute__((always_inline)) -> bool {
            seen += alt ? sub : 0;
            if (warp == 2 || (alt && warp == 6)) {
                const bool good = wait_counter(ctr, target, lane, abort_flag, where);
                if (lane == 0) mbar_arrive(seen);
                return good;
            }
            return __all_sync(0xffffffffu, mbar_wait(seen, 0, abort_flag, where)) && *abort_flag == 0;
        };
        unsigned tile_it = 0;
#pragma unroll 1
        for (int it = 0;; ++it) {
            const Item& w = item_at(it);
            if (norms_due && (norms.X != nullptr || w.kind == 0 || !(w.seg ? seg1 : seg0).tri)) {
                norm_rows(sh.norms, blockIdx.x * EPI_WARPS + (warp - 2), gridDim.x * EPI_WARPS, lane, dep_ctr + 1, status);
                norms_due = false;
            }
            if (w.kind == 0) break;
            if (w.kind == 2) continue;
            const int sg = w.seg, col0 = w.col0, ncols = w.ncols, row0 = w.row0;
            const GramProblem& p = sg ? seg1 : seg0;
            const unsigned acc = tile_it & 1u, acc_ph = (tile_it >> 1) & 1u;
            ++tile_it;
            const bool solo = alt && w.parts == 1;       // this set's tile alone
            if (solo && (int)acc != sub) continue;
            // the warp's chunks of 32 columns: cfirst, cfirst + cstep, .. below nch
            const int cfirst = solo ? 0 : sub, cstep = solo ? 1 : SUBS;
            float* cs = sh.col_scale[sub][n_staged & 1u];
            int* ct = sh.col_token[sub][n_staged & 1u];
            const int64_t o = (int64_t)w.b * p.cap;
            const int nch = ncols >> 5;
            const int arows = p.tri ? BM : hrows;
            const int lrow = quad * 32 + lane;           // this thread's row of the CTA's share of the tile
            const int row_base = row0 + (int)rank * arows;
            const int row = row_base + lrow;
            if (ring_norms) {
                const int nst = w.st1;                   // (nothing is split in this form)
                const int a_bytes = a_bytes_of(arows);
                const int subb = sub_bytes_pair(a_bytes, ncols);
                const int sb = St::NSUB * subb;
                if (sb != ring_sb) { ring_sb = sb; ring_nst = w.ring; ring_s = 0; }
                if (!norm_duty(p, col0, smem_norms)) {
                    ring_s = (ring_s + nst) % ring_nst;
                } else {
                    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
                    bool fine = true;
                    for (int st = 0; st < nst; ++st) {
                        fine = __all_sync(0xffffffffu, mbar_wait(&sh.consumed[ring_s], (cons >> ring_s) & 1u, abort_flag, 14));
                        if (!fine) break;
                        if (lrow < arows) {
                            // the 16-byte chunks of a row are permuted by the swizzle, which a sum
                            // of squares need not undo; lanes start at different chunks so that a
                            // warp's loads spread over all banks
                            const unsigned char* rowp = smem + ring_s * sb + sub * subb + lrow * 128;
                            uint4 x[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                x[j] = *reinterpret_cast<const uint4*>(rowp + (((j + lane) & 7) << 4));
                            s0 += sumsq_bf16x8(x[0]) + sumsq_bf16x8(x[4]);
                            s1 += sumsq_bf16x8(x[1]) + sumsq_bf16x8(x[5]);
                            s2 += sumsq_bf16x8(x[2]) + sumsq_bf16x8(x[6]);
                            s3 += sumsq_bf16x8(x[3]) + sumsq_bf16x8(x[7]);
                        }
                        __syncwarp();
                        // the last of the eight warps releases the stage to the producer
                        if (lane == 0) {
                            if (atomicAdd(&sh.norm_cnt[ring_s], 1u) == EPI_WARPS - 1) {
                                sh.norm_cnt[ring_s] = 0u;
                                mbar_arrive(&sh.empty[ring_s]);
                            }
                        }
                        cons ^= 1u << ring_s;
                        ring_s = (ring_s + 1 == ring_nst) ? 0 : ring_s + 1;
                    }
                    if (!fine) break;
                    float* part = sh.norm_part[n_normed & 1u][0];
                    part[sub * BM + lrow] = (s0 + s1) + (s2 + s3);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh.normed);
                    if (!__all_sync(0xffffffffu, mbar_wait(&sh.normed, n_normed & 1u, abort_flag, 17))) break;
                    ++n_normed;
                    if (sub == 0 && lrow < arows && row < w.m) {
                        const float ss = part[lrow] + part[BM + lrow];
                        float inv = 0.f;
                        if (!(ss <= 3.0e38f)) atomicOr(status, ST_NONFINITE);
                        else if (ss > 0.f) inv = 1.0f / sqrtf(ss);
                        else atomicAdd(status + 1, 1u);
                        p.inv_out[o + row] = inv;
                    }
                }
            }
            if (!prep_ok) {
                // the gathered rows' inverse norms (column factors, and the triangle's row factors)
                if (!__all_sync(0xffffffffu, mbar_wait(&sh.prep_seen, 0, abort_flag, 13))) break;
                prep_ok = true;
            }
            if (p.wait_norm_b && !norm_ok) {
                if (!await(dep_ctr + 1, norm_total, sh.norm_seen, 9)) break;
                norm_ok = true;
            }
            const unsigned thr_b = (!p.tri && p.tau_seq != nullptr) ? __float_as_uint(tau_threshold(__ldcg(p.tau_seq + w.b))) : p.thr_bits;
            bool row_live = lrow < arows && row < w.m;
            // the token this row belongs to: the row index itself, except over the copied-out rows
            // (an entry the gather did not write -- possible only with a rejected list -- is
            // never used as an index)
            int tokrow = row;
            if (compact && !p.tri && row_live) {
                tokrow = __ldcg(gather.non_tok + o + row);
                if ((unsigned)tokrow >= (unsigned)p.cap) { tokrow = row; row_live = false; }
            }
            const bool defer = !p.tri && p.defer_row != 0;   // the row's own factor is applied later
            // inherited reps are not candidates (with a deferred factor the compaction ignores them)
            const bool skip = row_live && !p.tri && !defer && p.row_role[o + row] != 0;
            const bool inv_early = defer || !(p.wait_norm_a && !norm_ok);
            float inv_row = defer ? 1.0f : ((row_live && inv_early) ? __ldcg(p.inv_a + o + row) : 0.f);
            const int rep_tok = !SPLIT && p.tri && p.out_tok != nullptr && row_live ? __ldg(p.col_token + o + row) : -1;
            const unsigned tbase = tmem_base + ((unsigned)(quad * 32) << 16) + acc * BN;
            int own0 = 0, own1 = nch;                    // chunks that this share of the tile answers for
            // Two steps: the column factors (for a cross tile they wait for the triangle's verdict), and for a
            // share of a split tile the exchange of partial sums.  What has to wait comes second.
            bool ok = true;
#pragma unroll 1
            for (int step = 0; step < 2; ++step) {
            if ((step == 0) != (p.tri != 0)) {
            if (w.parts > 1) {
                // A share of the contraction.  The tile's chunks are divided among its shares: each
                // writes its partial sums of the others' chunks to the exchange buffer (a row per
                // thread, 16-byte columns outermost: coalesced both ways) and adds the others' to its
                // own chunks, in a fixed order, in TMEM.  A cross tile does all this before it waits for
                // the triangle's verdict (pair kernel, T = 512, d = 768, fp32: 4 us of a 24 us step).
                const bool got = mbar_wait(&sh.tmem_full[acc], acc_ph, abort_flag, 4);
                ok = __all_sync(0xffffffffu, got);
                if (!ok) break;
                tcgen05_fence_after();
                own0 = quot(nch * w.part, w.parts); own1 = quot(nch * (w.part + 1), w.parts);
                const int unit0 = w.unit0;
#pragma unroll 1
                for (int c = sub; c < nch; c += SUBS) {
                    if (c >= own0 && c < own1) continue;
                    unsigned r0[32];
                    tmem_ld32_issue(tbase + 32 * c, r0);
                    tmem_ld_wait(r0);
                    uint4* dst = reinterpret_cast<uint4*>(part_buf + chunk_at(unit0 + w.part, rank, c)) + lrow;
#pragma unroll
                    for (int j = 0; j < 32; ++j) r0[j] = r0[j] == EMPTY_WORD ? 0x7FFFFFFFu : r0[j];   // another NaN
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        __stcg(dst + q * BM, make_uint4(r0[4 * q], r0[4 * q + 1], r0[4 * q + 2], r0[4 * q + 3]));
                }
                bool good = true;
#pragma unroll 1
                for (int c = sub; c < own1; c += SUBS) {
                    if (c < own0) continue;
                    uint4* const src = reinterpret_cast<uint4*>(part_buf + chunk_at(unit0, rank, c)) + lrow;
                    constexpr int STEP = 2 * (BN / 32) * CHUNK_WORDS / 4;        // from one share's slot to the next
                    unsigned r0[32];
                    tmem_ld32_issue(tbase + 32 * c, r0);
                    tmem_ld_wait(r0);
#pragma unroll 1
                    for (int q = 0; q < w.parts; ++q) {
                        if (q == w.part) continue;
                        uint4 x0[8];
                        load_partials(src + q * STEP, x0);
                        good = take_partials(src + q * STEP, x0, r0, abort_flag) && good;
                    }
                    tmem_st32(tbase + 32 * c, r0);
                }
                ok = __all_sync(0xffffffffu, good);
                if (!ok) break;
            }
            } else {
            if (sg == 1 && !dep_ok) {
                // every triangular tile of this launch first (line 5 before line 7)
                ok = await(dep_ctr, dep_total, sh.dep_seen, 5);
                if (!ok) break;
                dep_ok = true;
            }
            // Column factors: the set's chunks are dealt to its four warps.  (Columns past the tile are
            // clamped to its last one and discarded afterwards, so that no load hangs on a
            // data-dependent branch.)
            const int last = max(w.n - 1, 0);
#pragma unroll
            for (int e = 0; e < (St::COLS / 32 + 3) / 4; ++e) {
                const int c = cfirst + (quad + 4 * e) * cstep, col = col0 + 32 * c + lane;
                if (c >= nch) break;
                const int64_t from = o + min(col, last);
                const float f = __ldcg(p.inv_b + from);
                // representative removed at line 5 (written earlier in this launch: read at L2)
                const unsigned gate = p.tri ? 0u : __ldcg(p.col_gate + from);
                const int tk = !p.tri && p.causal ? __ldcg(p.col_token + from) : col;
                const bool live = col < w.n;
                const int at = 32 * (quad + 4 * e) + lane;
                cs[at] = (live && (p.tri || gate < thr_b)) ? f : 0.f;
                ct[at] = live ? tk : col;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.staged[sub]);
            }
            }
            if (!ok) break;
            {
                const bool got = mbar_wait(&sh.staged[sub], n_staged & 1u, abort_flag, 4);
                ++n_staged;
                if (!__all_sync(0xffffffffu, got)) break;
            }
            if (w.parts == 1) {
                const bool got = mbar_wait(&sh.tmem_full[acc], acc_ph, abort_flag, 4);
                if (!__all_sync(0xffffffffu, got)) break;
                tcgen05_fence_after();
            }
            const bool need_cmp = p.tri ? (col0 + ncols > row_base) : (p.causal != 0);
            const bool want_arg = (SPLIT || !p.tri) && p.out_arg != nullptr;
            float mx0 = 0.f, mx1 = 0.f;
            int arg = 0;                                     // nearest-representative mode: column of the maximum
            // 32 columns (chunk c) of this thread's row
            auto consume = [&](const unsigned (&r)[32], int c) __attribute__((always_inline)) {
                const float* csk = cs + (solo ? 32 * c : 32 * (c >> 1));
                if (want_arg) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) {           // ascending columns, strict '>': lowest index on ties
                        const float x = fabsf(__uint_as_float(r[j])) * csk[j];
                        if (x > mx0) { mx0 = x; arg = 32 * c + j; }
                    }
                } else if (!need_cmp) {
                    row_max32(r, csk, mx0, mx1);
                } else {
                    const int* ctk = ct + (solo ? 32 * c : 32 * (c >> 1));
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float4 f = *reinterpret_cast<const float4*>(csk + j);
                        const int4 t = *reinterpret_cast<const int4*>(ctk + j);
                        if (t.x < tokrow) mx0 = fmaxf(mx0, fabsf(__uint_as_float(r[j])) * f.x);
                        if (t.y < tokrow) mx1 = fmaxf(mx1, fabsf(__uint_as_float(r[j + 1])) * f.y);
                        if (t.z < tokrow) mx0 = fmaxf(mx0, fabsf(__uint_as_float(r[j + 2])) * f.z);
                        if (t.w < tokrow) mx1 = fmaxf(mx1, fabsf(__uint_as_float(r[j + 3])) * f.w);
                    }
                }
            };
            // (a warp whose 32 rows lie past a short tile's rows still joins the aligned loads; rolled
            // loops: the code of an epilogue is fetched cold in most launches)
#pragma unroll 1
            for (int c = cfirst; c < own1; c += cstep) {
                if (c < own0) continue;
                unsigned r0[32];
                tmem_ld32_issue(tbase + 32 * c, r0);
                tmem_ld_wait(r0);
                consume(r0, c);
            }
            float mx = fmaxf(mx0, mx1);
            tcgen05_fence_before();
            __syncwarp();
            // (a share is its pair's last item: nobody waits for its accumulator, and the arrive would
            // first wait for the stores above)
            if (lane == 0 && w.parts == 1) mbar_arrive_remote(empty_addr[acc], solo ? SUBS : 1);
            if (!inv_early && !norm_ok) {
                if (!await(dep_ctr + 1, norm_total, sh.norm_seen, 9)) break;
                norm_ok = true;
            }
            if (row_live && !skip) {
                if (!inv_early) inv_row = __ldcg(p.inv_a + o + row);
                mx *= inv_row;
                if (mx > 0.f) {
                    if (want_arg)
                        atomicMax(p.out_arg + o + tokrow, ((unsigned long long)__float_as_uint(mx) << 32) |
                                                              (unsigned long long)(0xFFFFFFFFu - (unsigned)(col0 + arg)));
                    else
                        atomicMax(p.out + o + tokrow, __float_as_uint(mx));
                }
            }
            if (sg == 0 && nseg > 1) {
                // publish: one arrival per CTA and tile, by the last of its warps, whose fence covers what
                // the others' orders before the shared counter
                __threadfence_block();
                __syncwarp();
                const unsigned share = solo ? SUBS : 1;
                if (lane == 0 && (atomicAdd(&sh.pub_cnt, share) + share) % EPI_WARPS == 0) {
                    __threadfence();
                    atomicAdd(dep_ctr, 1u);
                }
                // By token too, behind the arrival, since nobody in this launch waits for it: the compaction then reads all
                // that it needs of a token at once (2005 x 4096 chain of 28 796 -> 786 us; 8 x 2048 x 768 and 8192 x 4096 within
                // their spread, nothing for fp32, whose steps do without).  (An entry of a rejected list may be anything.)
                if (!SPLIT && mx > 0.f && (unsigned)rep_tok < (unsigned)p.cap) atomicMax(p.out_tok + o + rep_tok, __float_as_uint(mx));
            }
        }
    }

    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();          // neither CTA frees TMEM or exits while the other may still touch it
    if (warp == 1) {
        tcgen05_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                     "r"(TMEM_COLS)
                     : "memory");
    }
    if (threadIdx.x == 0 && sh.abort_flag[0] != 0) {
        atomicOr(status, ST_TIMEOUT);
        status[2] = 100u + (unsigned)sh.abort_flag[0];
    }
}

}  // namespace

static cudaError_t ensure_tc2(ada_ctx* ctx) {
    if (ctx->tc2_attr_set) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_gram_tc2<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         smem_pair_bytes<false>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_gram_tc2<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_pair_bytes<true>());
    if (e != cudaSuccess) { cudaGetLastError(); return e; }
    // how many clusters of two fit on the device at once
    cudaLaunchConfig_t q;
    memset(&q, 0, sizeof(q));
    q.gridDim = dim3(2 * (ctx->sm_count / 2));
    q.blockDim = dim3(PAIR_THREADS);
    q.dynamicSmemBytes = smem_pair_bytes<false>();
    cudaLaunchAttribute qa[1];
    qa[0].id = cudaLaunchAttributeClusterDimension;
    qa[0].val.clusterDim.x = 2; qa[0].val.clusterDim.y = 1; qa[0].val.clusterDim.z = 1;
    q.attrs = qa; q.numAttrs = 1;
    int nclusters = 0;
    e = cudaOccupancyMaxActiveClusters(&nclusters, k_gram_tc2<false>, &q);
    if (e != cudaSuccess || nclusters < 1) { cudaGetLastError(); return cudaErrorLaunchOutOfResources; }
    ctx->tc2_pairs = nclusters < ctx->sm_count / 2 ? nclusters : ctx->sm_count / 2;
    ctx->tc2_attr_set = true;
    return cudaSuccess;
}

// Rows of X per CTA for a cross-Gram whose columns fit one column tile (at most 256
// representatives per sequence): such a launch is one pass over X, so the row tiles are cut to
// give every SM pair but the ones that take the small triangular problems a share.  128 = the
// ordinary tile.  (0 if the kernel cannot be configured.)
int gram_tc2_hb_rows(ada_ctx* ctx, int B, int T) {
    if (ensure_tc2(ctx) != cudaSuccess) return 0;
    const int free_pairs = ctx->tc2_pairs - B;            // one triangular tile per sequence
    if (free_pairs < B) return BM;
    const int tiles_per_seq = free_pairs / B;
    int h = (T + 2 * tiles_per_seq - 1) / (2 * tiles_per_seq);
    if (h < 16) h = 16;
    return h >= BM ? BM : h;
}

// Pair-CTA launch.  tri and/or cross may be NULL; with both the cross epilogues wait in-kernel
// for the triangular segment (ctx->tile_ctr must be zero at launch).
cudaError_t launch_gram_tc2(ada_ctx* ctx, const GramProblem* tri, const GramProblem* cross,
                            const NormJob* norms, const GatherJob* gather, const SplitJob* split,
                            cudaStream_t s) {
    cudaError_t e0 = ensure_tc2(ctx);
    if (e0 != cudaSuccess) return e0;
    GramMaps maps;
    memset(&maps, 0, sizeof(maps));
    GramProblem segs[2];
    memset(segs, 0, sizeof(segs));
    int nseg = 0;
    const GramProblem* in[2] = {tri, cross};
    for (int i = 0; i < 2; ++i) {
        const GramProblem* p = in[i];
        if (p == nullptr) continue;
        const int n_cap = p->n_dev != nullptr ? p->cap : p->n_host;
        const int a_rows = p->tri ? n_cap : p->rows;
        if (n_cap <= 0 || a_rows <= 0) continue;
        const int width = p->planes > 0 ? 3 * p->planes : p->d;
        if (!make_map(ctx, &maps.a[nseg], p->A, width, p->tri ? p->cap : p->rows, p->B, p->lda, p->a_batch, BM) ||
            !make_map(ctx, &maps.b[nseg], p->Bm, width, p->cap, p->B, p->ldb, p->b_batch, BOX_N) ||
            !make_map(ctx, &maps.bt[nseg], p->Bm, width, p->cap, p->B, p->ldb, p->b_batch, BOX_N / 2))
            return cudaErrorInvalidValue;
        if (!p->tri && p->hb_rows > 0 && p->hb_rows < BM) {
            if (!make_map(ctx, &maps.ah, p->A, width, p->rows, p->B, p->lda, p->a_batch, p->hb_rows))
                return cudaErrorInvalidValue;
        } else {
            maps.ah = maps.a[nseg];
        }
        segs[nseg++] = *p;
    }
    if (nseg == 0) return cudaSuccess;
    if (nseg == 1) { maps.a[1] = maps.a[0]; maps.b[1] = maps.b[0]; maps.bt[1] = maps.bt[0]; segs[1] = segs[0]; segs[1].B = 0; }
    maps.an = maps.ah;
    if (gather != nullptr && gather->Xnon != nullptr && cross != nullptr && gather->T >= gather->compact_min_rows &&
        !make_map(ctx, &maps.an, gather->Xnon, cross->d, cross->rows, cross->B, cross->d, (int64_t)cross->cap * cross->d, BM))
        return cudaErrorInvalidValue;
    NormJob nj;
    memset(&nj, 0, sizeof(nj));
    if (norms != nullptr) nj = *norms;
    GatherJob gj;
    memset(&gj, 0, sizeof(gj));
    if (gather != nullptr) gj = *gather;
    SplitJob sj;
    memset(&sj, 0, sizeof(sj));
    if (split != nullptr) sj = *split;
    const bool planes = segs[0].planes > 0;
    int max_parts = ctx->part_buf != nullptr ? ctx->max_parts : 1;
    if (nseg == 1 && segs[0].tri && segs[0].n_dev == nullptr) {
        // tile count known here: a last round that is more than half full is not split
        const int M = (segs[0].n_host + PM - 1) / PM, f = planes ? 2 : 1;
        const int64_t tiles = (int64_t)segs[0].B * (f * (M * (M - 1) / 2) + (segs[0].n_host + PM / f - 1) / (PM / f));
        if (2 * (tiles % ctx->tc2_pairs) > ctx->tc2_pairs || tiles % ctx->tc2_pairs == 0) max_parts = 1;
    }
    const bool fused = nseg == 2;
    prof_begin(ctx, fused ? K_GRAM_TC_CASCADE : (segs[0].tri ? K_GRAM_TC_TRI : K_GRAM_TC_CROSS), s);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(2 * ctx->tc2_pairs);
    cfg.blockDim = dim3(PAIR_THREADS);
    cfg.dynamicSmemBytes = planes ? smem_pair_bytes<true>() : smem_pair_bytes<false>();
    cfg.stream = s;
    cudaLaunchAttribute attr[3];
    int na = 0;
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = 2; attr[na].val.clusterDim.y = 1; attr[na].val.clusterDim.z = 1;
    ++na;
    // CTAs wait on results of other CTAs (triangle before cross epilogues, the preparation before
    // everything, the row norms, the other shares of a split tile): all of them have to get to run
    const bool waits = fused || gj.X != nullptr || sj.X != nullptr || nj.X != nullptr || max_parts > 1;
    const bool coop = waits && coop_begin(ctx, s);
    if (coop) {
        attr[na].id = cudaLaunchAttributeCooperative;
        attr[na].val.cooperative = 1;
        ++na;
    }
    if (ctx->dep_launch) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    cudaError_t e = cudaLaunchKernelEx(&cfg, planes ? k_gram_tc2<true> : k_gram_tc2<false>, maps, segs[0], segs[1],
                                       nseg, nj, gj, sj, max_parts, wait_limit_units(ctx->cooperative && waits && !coop),
                                       ctx->part_buf, ctx->tile_ctr, ctx->status);
    if (waits) coop_end(ctx, coop);
    prof_end(ctx, s);
    return e;
}

}  // namespace ada
