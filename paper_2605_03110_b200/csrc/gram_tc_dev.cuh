// Device-side building blocks shared by the tcgen05 Gram kernels: tile constants, the
// shared-memory control block, PTX wrappers (mbarrier, TMA, tcgen05), descriptors.
#pragma once

#include <cuda.h>
#include <string.h>

#include "common.cuh"

namespace ada {
namespace tc {


static constexpr int BM = 128;          // accumulator rows per tile (TMEM lanes)
static constexpr int BN = 256;          // accumulator columns per tile
static constexpr int BK = 64;           // bf16 elements per K block = one 128-byte swizzle row
static constexpr int MAX_STAGES = 9;
static constexpr int RING_BYTES = 216 * 1024;               // TMA ring: 4 stages of a 256-wide tile ... 9 of a 64-wide one
static constexpr int UMMA_K = 16;
static constexpr int A_BYTES = BM * BK * 2;                 // 16 KiB
static constexpr int BOX_N = 64;                            // B rows per TMA box
static constexpr int BOX_BYTES = BOX_N * BK * 2;            // 8 KiB
static constexpr int NORM_WARPS = 8;
static constexpr int NUM_THREADS = 192 + 32 * NORM_WARPS;   // producer, MMA, 4 epilogue warps, norm warps
static constexpr int TMEM_COLS = 512;
// Has a wait that began at t0 reached its limit?  That is set per launch (launch_policy.h) and lies, in units of
// 2^20 ns, in the word behind a CTA's abort flag.
static __device__ __forceinline__ bool past_limit(unsigned long long elapsed_ns, const volatile int* abort_flag) {
    return (int)(elapsed_ns >> 20) > abort_flag[1];
}

// one output tile: `ncols` (multiple of 16, <= 256) columns from col0 of the 128-row tile at row0
struct Piece {
    int b, row0, col0, ncols, n, m;
};

// ---------------------------------------------------------------- PTX wrappers
static __device__ __forceinline__ unsigned smem_u32(const void* p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
static __device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
static __device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
static __device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
static __device__ __forceinline__ bool mbar_try(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
static __device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// One try that suspends the thread for up to about 20 us: a waiting warp then costs neither issue slots
// nor power (a dozen warps per SM polling through a 200 us main loop were measured to cost 3 %).
static __device__ __forceinline__ bool mbar_try_long(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}
// A wait that has polled in vain for a while: has the CTA been aborted, or this wait reached its limit?  (Out of
// line: a kernel has a dozen waits, and its code is fetched cold.  fp32 chain of twelve layers, T = 512:
// 253 us inlined, 244 so; per-head step 42.2 -> 42.0; sparse step at T = 16384 42.2 -> 41.8.)
static __device__ __noinline__ bool gives_up(unsigned long long* t0, volatile int* abort_flag, int where) {
    if (*abort_flag != 0) return true;
    const unsigned long long now = global_ns();
    if (*t0 == 0) *t0 = now;
    else if (past_limit(now - *t0, abort_flag)) {
        *abort_flag = where;
        return true;
    }
    return false;
}
// Bounded wait.  Returns false when the CTA is aborting (this or another wait ran out).
static __device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity,
                                          volatile int* abort_flag, int where) {
    unsigned polls = 0;
    unsigned long long t0 = 0;
    while (!mbar_try_long(bar, parity)) {
        // (the wall clock is a slow special register)
        if ((++polls & 15u) == 0 && gives_up(&t0, abort_flag, where)) return false;
    }
    return true;
}
static __device__ __forceinline__ void tma_load_3d(const CUtensorMap* map, unsigned long long* bar,
                                            void* dst, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<unsigned long long>(map)), "r"(smem_u32(bar)),
          "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
static __device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<unsigned long long>(map)) : "memory");
}
static __device__ __forceinline__ void tcgen05_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
static __device__ __forceinline__ void tcgen05_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
static __device__ __forceinline__ void umma_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_u32(bar))
                 : "memory");
}
static __device__ __forceinline__ void umma_bf16(unsigned tmem_d, unsigned long long adesc,
                                          unsigned long long bdesc, unsigned idesc,
                                          unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The MMAs of one tile over one or two 64-element K blocks (a_next, b_next: bytes from a block to the next; what
// lies past the operands' last element is zero).  Unrolled and without a condition per instruction: one
// thread's loop takes longer over an instruction than the tensor core does (128 x 256 x 16: 0.1 us against
// 0.067).  The first one overwrites the accumulator.  (Each instruction under a condition of its own, `if (16 q < d)`,
// gave wrong sums from the second one on.  The source does not show why, so that form is not used anywhere: blocks are
// contracted whole, here and in the loops of the other kernels, and only the first flag is ever a variable.)
template <int BLOCKS>
static __device__ __forceinline__ void umma_blocks(unsigned tmem_d, unsigned long long adesc, unsigned long long bdesc,
                                                   int a_next, int b_next, unsigned idesc) {
#pragma unroll
    for (int kb = 0; kb < BLOCKS; ++kb)
#pragma unroll
        for (int q = 0; q < BK / UMMA_K; ++q)
            umma_bf16(tmem_d, adesc + kb * (a_next >> 4) + 2 * q, bdesc + kb * (b_next >> 4) + 2 * q, idesc, (kb | q) != 0);
}
static __device__ __forceinline__ void tmem_ld32(unsigned taddr, float (&v)[32]) {
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        // the wait sits in the same statement so that no use of the registers can be
        // scheduled ahead of it
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// The same load as two statements.  After tmem_ld32_issue the registers are undefined; the
// wait takes them as in/out operands, so every use in the code that follows depends on it.
static __device__ __forceinline__ void tmem_ld32_issue(unsigned taddr, unsigned (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
static __device__ __forceinline__ void tmem_ld_wait(unsigned (&r)[32]) {
    asm volatile(
        "tcgen05.wait::ld.sync.aligned;"
        : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
          "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]),
          "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]),
          "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]),
          "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
        :
        : "memory");
}

// tcgen05.st of 32 columns of this warp's lanes
static __device__ __forceinline__ void tmem_st32(unsigned taddr, const unsigned (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n\t"
        "tcgen05.wait::st.sync.aligned;"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
// max(m, |a|, |b|) in one instruction
static __device__ __forceinline__ float max3_abs(float m, float a, float b) {
    float d;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(m), "f"(a), "f"(b));
    return d;
}
// Running maxima of |r[j]| * f[j] over 32 columns: two products per multiply, two candidates per maximum, i.e.
// one arithmetic instruction per column (the epilogues of short contractions are bound by them).
static __device__ __forceinline__ void row_max32(const unsigned (&r)[32], const float* f, float& m0, float& m1) {
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        const ulonglong2 ff = *reinterpret_cast<const ulonglong2*>(f + j);
        float a, b, c, d;
        asm("{\n\t.reg .b64 x, y;\n\t"
            "mov.b64 x, {%4, %5};\n\tmov.b64 y, {%6, %7};\n\t"
            "mul.rn.f32x2 x, x, %8;\n\tmul.rn.f32x2 y, y, %9;\n\t"
            "mov.b64 {%0, %1}, x;\n\tmov.b64 {%2, %3}, y;\n\t}"
            : "=f"(a), "=f"(b), "=f"(c), "=f"(d)
            : "r"(r[j]), "r"(r[j + 1]), "r"(r[j + 2]), "r"(r[j + 3]), "l"(ff.x), "l"(ff.y));
        m0 = max3_abs(m0, a, b);
        m1 = max3_abs(m1, c, d);
    }
}

// Shared-memory matrix descriptor of a K-major bf16 tile whose rows are 128 bytes wide and
// stored with the 128-byte swizzle: 8-row groups are 1024 bytes apart (stride byte offset),
// the leading byte offset is unused for swizzled K-major tiles, descriptor version 1.
static __device__ __forceinline__ unsigned long long smem_desc_sw128(unsigned addr) {
    unsigned long long d = 0;
    d |= (unsigned long long)((addr & 0x3FFFFu) >> 4);        // start address, 16-byte units
    d |= (unsigned long long)1 << 16;                         // leading byte offset (ignored)
    d |= (unsigned long long)(1024 >> 4) << 32;               // stride byte offset
    d |= (unsigned long long)1 << 46;                         // descriptor version (sm_100)
    d |= (unsigned long long)2 << 61;                         // layout: 128-byte swizzle
    return d;
}
// Instruction descriptor: D = fp32, A = B = bf16, both K-major, M = 128, N = n.
static __device__ __forceinline__ unsigned instr_desc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(BM >> 4) << 24);
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static inline EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        else
            cudaGetLastError();
    }
    return fn;
}

// 3-D map over a stack of K-major bf16 matrices: (k, row, sequence).
static inline bool encode_map(CUtensorMap* map, const void* base, int d, int rows, int B, int64_t ld,
                              int64_t batch, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (fn == nullptr) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)rows, (cuuint64_t)B};
    // the stride of the last dimension is unused when B == 1 but must still be legal
    const cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)(B > 1 ? batch : (int64_t)rows * ld) * 2};
    const cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The last tensor maps of a context: a call needs up to eight, most of them over the context's own
// workspace or a tensor that the caller passes again (a descriptor depends on address and shape
// only).  One context serves one stream at a time, so it has no lock; ctx->map_cache is NULL where a
// context may be used by several threads at once.
struct MapCache {
    static constexpr int N = 48;
    struct Key {
        const void* base;
        int64_t ld, batch;
        int d, rows, B, box_rows;
    } key[N];
    CUtensorMap map[N];
    int n = 0, next = 0;
};
static inline bool make_map(ada_ctx* ctx, CUtensorMap* map, const void* base, int d, int rows, int B, int64_t ld,
                            int64_t batch, int box_rows) {
    MapCache* c = static_cast<MapCache*>(ctx->map_cache);
    if (c == nullptr) return encode_map(map, base, d, rows, B, ld, batch, box_rows);
    for (int i = 0; i < c->n; ++i) {
        const MapCache::Key& k = c->key[i];
        if (k.base == base && k.d == d && k.rows == rows && k.B == B && k.ld == ld && k.batch == batch &&
            k.box_rows == box_rows) {
            *map = c->map[i];
            return true;
        }
    }
    if (!encode_map(map, base, d, rows, B, ld, batch, box_rows)) return false;
    const int at = c->next;
    c->key[at] = {base, ld, batch, d, rows, B, box_rows};
    c->map[at] = *map;
    c->next = at + 1 == MapCache::N ? 0 : at + 1;
    if (c->n < MapCache::N) ++c->n;
    return true;
}

// ---------------------------------------------------------------- in-launch row norms
// bf16 pairs are the halves of 32-bit words; a bf16 is the upper half of an fp32
static __device__ __forceinline__ float sumsq_bf16x8(const uint4& v) {
    float s = 0.f;
    const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xffff0000u);
        s = fmaf(lo, lo, s);
        s = fmaf(hi, hi, s);
    }
    return s;
}
static __device__ __forceinline__ float inv_of_sumsq(float ss, int lane, unsigned* status) {
    float inv = 0.f;
    if (!(ss <= 3.0e38f)) {
        if (lane == 0) atomicOr(status, ST_NONFINITE);
    } else if (ss > 0.f) {
        inv = 1.0f / sqrtf(ss);
    } else if (lane == 0) {
        atomicAdd(status + 1, 1u);
    }
    return inv;
}
// Executed by the norm warps of every CTA: warp `w` of `nw` takes rows w, w+nw, ...; when a
// warp has stored its last row it bumps the counter, so counter == nw means "all rows done".
static __device__ __forceinline__ void norm_rows(const NormJob& job, int w, int nw, int lane, unsigned* counter,
                                              unsigned* status) {
    const int nvec = job.d >> 3;
    const __nv_bfloat16* X = reinterpret_cast<const __nv_bfloat16*>(job.X);
    // (row counts fit 31 bits; a 32-bit division is several times cheaper)
    auto at = [&](int64_t row) {
        return job.rows_per_seq > 0 ? ((unsigned)row / (unsigned)job.rows_per_seq) * job.batch +
                                          ((unsigned)row % (unsigned)job.rows_per_seq) * job.ldx
                                    : row * job.ldx;
    };
    int64_t row = w;
    if (nvec <= 128) {
        // rows of at most 128 vectors: four rows, sixteen loads, in flight per lane
        for (; row + 3 * (int64_t)nw < job.n_rows; row += 4 * (int64_t)nw) {
            float ss[4];
            uint4 x[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4* src = reinterpret_cast<const uint4*>(X + at(row + i * (int64_t)nw));
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    x[i][q] = lane + 32 * q < nvec ? __ldg(src + lane + 32 * q) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                ss[i] = ((sumsq_bf16x8(x[i][0]) + sumsq_bf16x8(x[i][1])) + sumsq_bf16x8(x[i][2])) + sumsq_bf16x8(x[i][3]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < 4; ++i) ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], o);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float inv = inv_of_sumsq(ss[i], lane, status);
                if (lane == 0) job.inv_norm[row + i * (int64_t)nw] = inv;
            }
        }
    }
    for (; row < job.n_rows; row += nw) {
        const int64_t off = at(row);
        const uint4* src = reinterpret_cast<const uint4*>(X + off);
        // sixteen independent 128-bit loads in flight per lane: these few warps have to cover the
        // memory latency that a dedicated kernel would hide with occupancy
        float ss = 0.f;
        int v = lane;
        for (; v + 480 < nvec; v += 512) {
            uint4 x[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) x[q] = __ldg(src + v + 32 * q);
#pragma unroll
            for (int q = 0; q < 16; ++q) ss += sumsq_bf16x8(x[q]);
        }
        for (; v < nvec; v += 256) {
            uint4 x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                x[q] = v + 32 * q < nvec ? __ldg(src + v + 32 * q) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int q = 0; q < 8; ++q) ss += sumsq_bf16x8(x[q]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float inv = inv_of_sumsq(ss, lane, status);
        if (lane == 0) job.inv_norm[row] = inv;
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) atomicAdd(counter, 1u);
}
// Bounded, warp-uniform wait until a global counter reaches `target`.
static __device__ __forceinline__ bool wait_counter(const unsigned* counter, unsigned target, int lane,
                                                    volatile int* abort_flag, int where,
                                                    unsigned long long limit_ns = 0) {
    int good = 1;
    if (lane == 0) {
        const unsigned long long t0 = global_ns();
        unsigned seen;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
            if (seen >= target) break;
            if (*abort_flag != 0) { good = 0; break; }
            const unsigned long long dt = global_ns() - t0;
            if (limit_ns != 0 ? dt > limit_ns : past_limit(dt, abort_flag)) { *abort_flag = where; good = 0; break; }
            __nanosleep(64);
        }
    }
    return __shfl_sync(0xffffffffu, good, 0) != 0;
}

// ---------------------------------------------------------------- in-launch gather (cascade step)
// bounded wait of ONE thread until a global counter reaches `target`
static __device__ __forceinline__ bool wait_counter_1(const unsigned* counter, unsigned target,
                                               volatile int* abort_flag, int where) {
    const unsigned long long t0 = global_ns();
    unsigned seen;
    while (true) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
        if (seen >= target) return true;
        if (*abort_flag != 0) return false;
        if (past_limit(global_ns() - t0, abort_flag)) { *abort_flag = where; return false; }
        __nanosleep(64);
    }
}

// Is the complement of the inherited set copied out (below)?  Two fifths of the tokens or more in
// every sequence of a long batch, and more than one column tile (256) in one of them.  (Measured on
// the crossover sweep at r/T = 0.5: 1052 -> 699 us at T = 16384, 250 -> 217 us at T = 8192, but
// 87 -> 97 us at T = 4096, where the copy costs more than the saved tiles.)
static __device__ __forceinline__ bool compact_wanted(const GatherJob& gj, int lane) {
    if (gj.Xnon == nullptr || gj.T < gj.compact_min_rows) return false;
    bool one = true, big = true;
    for (int b = lane; b < gj.B; b += 32) {
        const int n = min(max(gj.rep_in_cnt[b], 0), gj.T);
        one = one && n <= BN;
        big = big && 5 * (int64_t)n >= 2 * (int64_t)gj.T;
    }
    return __all_sync(0xffffffffu, big) && !__all_sync(0xffffffffu, one);
}

// one warp: copy U rows of nvec 16-byte vectors (dst NULL: only read), V loads per lane and row in flight;
// ss: their sums of squares (all lanes)
template <int U, int V>
static __device__ __forceinline__ void copy_rows(const uint4* const (&src)[U], uint4* const (&dst)[U], int nvec, int lane,
                                                 float (&ss)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) ss[u] = 0.f;
    int v = lane;
    for (; v - lane + 32 * V <= nvec; v += 32 * V) {
        uint4 x[U][V];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int q = 0; q < V; ++q) x[u][q] = __ldg(src[u] + v + 32 * q);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int q = 0; q < V; ++q) {
                ss[u] += sumsq_bf16x8(x[u][q]);
                if (U == 1 || dst[u] != nullptr) dst[u][v + 32 * q] = x[u][q];
            }
    }
#pragma unroll 1
    for (; v - lane < nvec; v += 128) {
        uint4 x[U][4];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                x[u][q] = v + 32 * q < nvec ? __ldg(src[u] + v + 32 * q) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                ss[u] += sumsq_bf16x8(x[u][q]);
                if ((U == 1 || dst[u] != nullptr) && v + 32 * q < nvec) dst[u][v + 32 * q] = x[u][q];
            }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) ss[u] += __shfl_xor_sync(0xffffffffu, ss[u], o);
}

// Walks a warp through the entries of all sequences' lists: item -> (sequence b, entry i).  The counts are
// read 32 sequences at a time, one per lane (dozens of heads or a batch: one thread following
// them would be a chain of memory round trips).
struct ListCursor {
    const int32_t* counts;
    int T, B, lane, b0, mine, incl;
    bool first;
    int64_t base;                // items of the sequences before b0
    int32_t* r_eff;
    unsigned* status;
    int b, cnt, i;
    __device__ __forceinline__ ListCursor(const int32_t* c, int T_, int B_, bool first_, int32_t* re, int lane_,
                                          unsigned* st)
        : counts(c), T(T_), B(B_), lane(lane_), b0(0), first(first_), base(0), r_eff(re), status(st) { load(); }
    __device__ __forceinline__ void load() {
        mine = 0;
        if (b0 + lane < B) {
            mine = counts[b0 + lane];
            if (mine < 0 || mine > T) {
                if (first) atomicOr(status, ST_BAD_COUNT);
                mine = mine < 0 ? 0 : T;
            }
            if (first) r_eff[b0 + lane] = mine;
        }
        incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
    }
    // (items ascend from call to call)
    __device__ __forceinline__ bool find(int64_t item) {
        while (true) {
            const unsigned above = __ballot_sync(0xffffffffu, item - base < incl);
            if (above != 0u) {
                const int l = __ffs(above) - 1;
                b = b0 + l;
                cnt = __shfl_sync(0xffffffffu, mine, l);
                i = (int)(item - base) - __shfl_sync(0xffffffffu, incl - mine, l);
                return true;
            }
            base += __shfl_sync(0xffffffffu, incl, 31);
            b0 += 32;
            if (b0 >= B) return false;
            load();
        }
    }
};

// Entries of the inherited lists, warp `g` of `nw`, U at a time: entry i of sequence b is checked (in range,
// strictly above entry i-1), role[token] = i + 1, the raw row goes to Xrep[b, i] and its inverse
// norm to inv_rep[b, i]; a rejected entry gets inverse norm 0 (its column then counts for
// nothing) and raises the status.  copy: false when another pass copies the rows.
template <int U, int V>
static __device__ __forceinline__ void gather_entries(const GatherJob& gj, int g, int nw, int lane, bool copy,
                                                      unsigned* status) {
    const __nv_bfloat16* X = reinterpret_cast<const __nv_bfloat16*>(gj.X);
    __nv_bfloat16* Xrep = reinterpret_cast<__nv_bfloat16*>(gj.Xrep);
    // this warp's first entry is most often entry g of sequence 0: fetch it (and its
    // predecessor) beside the count instead of after it
    int32_t first_idx = 0, first_prev = -1;
    if (g < gj.T) {
        first_idx = __ldg(gj.rep_in + g);
        if (g > 0) first_prev = __ldg(gj.rep_in + g - 1);
    }
    ListCursor cur(gj.rep_in_cnt, gj.T, gj.B, g == 0, gj.r_eff, lane, status);
    int64_t item = g;
    bool more = true;
    while (more) {
        int b[U], i[U];
        int32_t idx[U], prev[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            b[u] = -1;
            if (more) more = cur.find(item);
            if (!more) continue;
            b[u] = cur.b; i[u] = cur.i;
            item += nw;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (b[u] < 0) continue;
            const int32_t* list = gj.rep_in + (int64_t)b[u] * gj.T;
            const bool spec = b[u] == 0 && i[u] == g;
            idx[u] = spec ? first_idx : __ldg(list + i[u]);
            prev[u] = i[u] == 0 ? -1 : (spec ? first_prev : __ldg(list + i[u] - 1));
        }
        const uint4* src[U];
        uint4* dst[U];
        bool ok[U], any = false;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            src[u] = reinterpret_cast<const uint4*>(X); dst[u] = nullptr;
            ok[u] = b[u] >= 0 && idx[u] >= 0 && idx[u] < gj.T && prev[u] < idx[u];
            if (b[u] < 0) continue;
            const int64_t prow = (int64_t)b[u] * gj.T + i[u];
            if (!ok[u] && lane == 0) { atomicOr(status, ST_BAD_INDEX); gj.inv_rep[prow] = 0.f; }
            if (!ok[u] || !copy) continue;
            any = true;
            src[u] = reinterpret_cast<const uint4*>(X + (int64_t)b[u] * gj.xb + (int64_t)idx[u] * gj.ldx);
            dst[u] = reinterpret_cast<uint4*>(Xrep + prow * (int64_t)gj.d);
        }
        if (!any) continue;
        float ss[U];
        copy_rows<U, V>(src, dst, gj.d >> 3, lane, ss);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (ok[u] && lane == 0) {
                gj.inv_rep[(int64_t)b[u] * gj.T + i[u]] = (ss[u] <= 3.0e38f && ss[u] > 0.f) ? 1.0f / sqrtf(ss[u]) : 0.f;
                gj.role[(int64_t)b[u] * gj.T + idx[u]] = i[u] + 1;
            }
    }
}

// How many of the ascending list's n entries lie below t: a 32-way search by the whole warp
static __device__ __forceinline__ int entries_below(const int32_t* list, int n, int t, int lane) {
    int lo = 0, hi = n;
    while (hi - lo > 32) {
        const int step = (hi - lo + 31) >> 5, at = lo + (lane + 1) * step - 1;
        const unsigned below = __ballot_sync(0xffffffffu, at < hi && __ldg(list + min(at, hi - 1)) < t);
        const int k = __popc(below);
        lo += k * step;
        hi = min(hi, lo + step);
        if (lo >= hi) return hi;
    }
    return lo + __popc(__ballot_sync(0xffffffffu, lo + lane < hi && __ldg(list + min(lo + lane, n - 1)) < t));
}

// Line 6's row set as a matrix of its own.  Line 6 builds the cross-Gram from the (T - r) tokens OUTSIDE
// the inherited set; when the set is large, streaming all T rows and masking the inherited ones
// wastes r/T of the loads and MMAs, so those rows are copied, in order, to Xnon (row t goes to t
// minus the number of inherited tokens before it), with their token index in non_tok and
// 1/||x_t|| in inv_norm, and the inherited ones to Xrep, in one pass over X: a warp takes runs of
// consecutive tokens of equal length.  (Dealt by gaps between list entries, the longest gap held
// everybody up: 56 us instead of 17 at T = 8192, r/T = 0.5, d = 1536.)
template <int U, int V>
static __device__ __forceinline__ void gather_all_rows(const GatherJob& gj, int g, int nw, int lane, unsigned* status) {
    const __nv_bfloat16* X = reinterpret_cast<const __nv_bfloat16*>(gj.X);
    __nv_bfloat16* Xrep = reinterpret_cast<__nv_bfloat16*>(gj.Xrep);
    __nv_bfloat16* Xnon = reinterpret_cast<__nv_bfloat16*>(gj.Xnon);
    const int run = min(32, (int)(((int64_t)gj.B * gj.T + nw - 1) / nw));
    const int runs = (gj.T + run - 1) / run;                       // per sequence
    for (int64_t it = g; it < (int64_t)gj.B * runs; it += nw) {
        const int b = (int)(it / runs), t0 = (int)(it % runs) * run, t1 = min(t0 + run, gj.T);
        const int32_t* list = gj.rep_in + (int64_t)b * gj.T;
        const int cnt = min(max(gj.rep_in_cnt[b], 0), gj.T);
        int pos = entries_below(list, cnt, t0, lane);
        const int32_t ahead = pos + lane < cnt ? __ldg(list + pos + lane) : -1;
        int used = 0;
        for (int t = t0; t < t1; t += U) {
            const uint4* src[U];
            uint4* dst[U];
            int at[U];                                             // >= 0: list position; < 0: -1 - row of Xnon
#pragma unroll
            for (int u = 0; u < U; ++u) {
                src[u] = reinterpret_cast<const uint4*>(X); dst[u] = nullptr;
                at[u] = 0;
                if (t + u >= t1) continue;
                const bool rep = used < 32 && __shfl_sync(0xffffffffu, ahead, used & 31) == t + u;
                at[u] = rep ? pos : -1 - max(t + u - pos, 0);
                if (rep) { ++pos; ++used; }
                src[u] = reinterpret_cast<const uint4*>(X + (int64_t)b * gj.xb + (int64_t)(t + u) * gj.ldx);
                dst[u] = reinterpret_cast<uint4*>(rep ? Xrep + ((int64_t)b * gj.T + at[u]) * (int64_t)gj.d
                                                      : Xnon + ((int64_t)b * gj.T + (-1 - at[u])) * (int64_t)gj.d);
            }
            float ss[U];
            copy_rows<U, V>(src, dst, gj.d >> 3, lane, ss);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (t + u >= t1) continue;
                const float inv = inv_of_sumsq(ss[u], lane, status);
                if (lane != 0) continue;
                const int64_t o = (int64_t)b * gj.T;
                gj.inv_norm[o + t + u] = inv;
                if (at[u] >= 0) { gj.inv_rep[o + at[u]] = inv; gj.role[o + t + u] = at[u] + 1; }
                else gj.non_tok[o + (-1 - at[u])] = t + u;
            }
        }
    }
}

// Algorithm 1 lines 1-2, by the preparation warps of all CTAs (warp `g` of `nw`).  (A single row at a time
// outside the copying-out form: a warp has one or two, and several at once cost more code, fetched
// cold, than they save.)
static __device__ __noinline__ void gather_compact(const GatherJob& gj, int g, int nw, int lane, unsigned* status) {
    gather_entries<1, 16>(gj, g, nw, lane, false, status);
    if (gj.d <= 1024) gather_all_rows<4, 4>(gj, g, nw, lane, status);
    else gather_all_rows<1, 16>(gj, g, nw, lane, status);
}
// (gs: the same job in shared memory.  The rare form is not inlined: a Gram launch fetches its
// instructions cold, and its start-up gets longer with every line of code between those it executes.)
static __device__ __forceinline__ void gather_rows(const GatherJob& gj, const GatherJob& gs, int g, int nw, int lane,
                                                   unsigned* status) {
    if (compact_wanted(gj, lane)) gather_compact(gs, g, nw, lane, status);
    else gather_entries<1, 16>(gj, g, nw, lane, true, status);
}

// ---------------------------------------------------------------- fp32 rows as three bf16 planes
static __device__ __forceinline__ void split3(float x, __nv_bfloat16& hi, __nv_bfloat16& mid, __nv_bfloat16& lo) {
    hi = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(hi);
    mid = __float2bfloat16_rn(r1);
    const float r2 = r1 - __bfloat162float(mid);
    lo = __float2bfloat16_rn(r2);
}
// one warp: planes of one row (each `dpad` elements, zeros past d), its sum of squares (all lanes)
static __device__ __forceinline__ float split_row(const float4* __restrict__ src, __nv_bfloat16* __restrict__ dst,
                                                  int d, int dpad, int lane) {
    float ss = 0.f;
    const int nvec = d >> 2, nout = dpad >> 2;                // d is a multiple of 4
    for (int v0 = lane; v0 < nout; v0 += 256) {
        float4 x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            x[q] = v0 + 32 * q < nvec ? __ldg(src + v0 + 32 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int v = v0 + 32 * q;
            if (v >= nout) break;
            const float xs[4] = {x[q].x, x[q].y, x[q].z, x[q].w};
            __align__(8) __nv_bfloat16 hi[4], mid[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                ss = fmaf(xs[e], xs[e], ss);
                split3(xs[e], hi[e], mid[e], lo[e]);
            }
            *reinterpret_cast<uint2*>(dst + v * 4) = *reinterpret_cast<const uint2*>(hi);
            *reinterpret_cast<uint2*>(dst + dpad + v * 4) = *reinterpret_cast<const uint2*>(mid);
            *reinterpret_cast<uint2*>(dst + 2 * dpad + v * 4) = *reinterpret_cast<const uint2*>(lo);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    return ss;
}
// Preparation of an fp32 call, warp `g` of `nw`: planes and inverse norms of every row of X, and of
// the rows of the inherited list (checked and scattered into the role map as in gather_rows).
static __device__ __noinline__ void split_rows(const SplitJob& sj, int g, int nw, int lane, unsigned* status) {
    const int64_t n_rows = (int64_t)sj.B * sj.T;
    const int64_t prow_len = 3 * (int64_t)sj.dpad;
    // list entries first: they hang on two more loads than the plain rows
    if (sj.rep_in != nullptr) {
        int64_t item = g;
        for (ListCursor cur(sj.rep_in_cnt, sj.T, sj.B, g == 0, sj.r_eff, lane, status); cur.find(item); item += nw) {
            const int b = cur.b, i = cur.i;
            const int32_t* list = sj.rep_in + (int64_t)b * sj.T;
            const int32_t idx = list[i];
            bool ok = idx >= 0 && idx < sj.T;
            if (ok && i > 0) ok = list[i - 1] < idx;
            const int64_t prow = (int64_t)b * sj.T + i;
            if (!ok) {
                if (lane == 0) { atomicOr(status, ST_BAD_INDEX); sj.inv_rep[prow] = 0.f; }
                continue;
            }
            const float ss = split_row(reinterpret_cast<const float4*>(sj.X + (int64_t)b * sj.xb + (int64_t)idx * sj.ldx),
                                       sj.RP + prow * prow_len, sj.d, sj.dpad, lane);
            if (lane == 0) {
                sj.inv_rep[prow] = (ss <= 3.0e38f && ss > 0.f) ? 1.0f / sqrtf(ss) : 0.f;
                sj.role[(int64_t)b * sj.T + idx] = i + 1;
            }
        }
    }
    // warps from the far end take the rows first, so that few warps have both kinds
    for (int64_t row = nw - 1 - g; row < n_rows; row += nw) {
        const int64_t b = row / sj.T, t = row % sj.T;
        const float ss = split_row(reinterpret_cast<const float4*>(sj.X + b * sj.xb + t * sj.ldx), sj.XP + row * prow_len,
                                   sj.d, sj.dpad, lane);
        if (lane == 0) {
            float inv = 0.f;
            if (!(ss <= 3.0e38f)) atomicOr(status, ST_NONFINITE);
            else if (ss > 0.f) inv = 1.0f / sqrtf(ss);
            else atomicAdd(status + 1, 1u);
            sj.inv_norm[row] = inv;
        }
    }
}

}  // namespace tc
}  // namespace ada
