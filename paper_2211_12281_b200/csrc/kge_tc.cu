// Tensor-core score block (5th-generation tensor cores: tcgen05.mma with the accumulator in
// tensor memory, operands staged in shared memory by TMA tensor copies).
//
//   C[M, N] = A[M, K] . B[N, K]^T      A, B bf16, K contiguous; fp32 accumulation
//
// Persistent CTAs (one per SM) each walk a run of 128 x 128 output tiles.  Warp 0 feeds a ring of
// shared-memory stages with TMA (one elected lane), warp 1 issues the MMAs (one elected lane)
// into one of the accumulators in tensor memory and owns the allocation, eight or sixteen more drain
// another accumulator meanwhile (a warp may only touch the 32 lanes of its own quarter; two or four warps
// share a quarter, 64 columns each) and apply the epilogue:
//   EPI_STORE   C = acc (the score block as a test reads it)
//   EPI_LOSS    no score leaves the chip: dL/dF up to a factor of the row as bf16, for the two backward contractions, and per row
//               and 64-column piece the sum of exponentials and the weighted loss sum of Section 3.1 "Loss Functions"; the
//               score is the contraction (DistMult, ComplEx) or, for TransE with p = 2, the
//               norm expansion -sqrt(max(|q|^2 + |t|^2 - 2 acc, 0))
//   EPI_GRAD    dL/dF of the rows, if any, whose scores lie too far from what EPI_LOSS took as their reference
// Every wait on a barrier is bounded; a wait that runs out records KGE_ERR_TIMEOUT, tells the
// other warps to stop, and the CTA still releases its tensor memory before it returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "kge_common.cuh"

namespace kge {

namespace {

constexpr int TC_BM = 128, TC_BN = 128, TC_BK = 64;      // BK bf16 = one 128-byte swizzle row
constexpr int TC_STAGES = 4;
constexpr int TC_EPI_WARPS = 8;                           // epilogue warps of the training kernels: TC_EPI_GROUPS per tensor-memory lane quarter
constexpr int TC_EPI_GROUPS = TC_EPI_WARPS / 4;
constexpr int TC_GRAD_STAGE_BYTES = 2048;                 // per epilogue warp: 32 rows x 32 bf16 columns on their way to memory
constexpr int TC_STORE_STAGE_BYTES = 4096;                // the same for EPI_STORE's 32 rows x 32 fp32 columns
constexpr int TC_PIECE = TC_BN / TC_EPI_GROUPS;           // columns of a 128-wide tile per piece of loss statistics
// The fused loss epilogues on 256-column tiles run on sixteen warps: 64 columns, one piece of statistics, per warp, as on 128-column tiles.
// Sixteen leave 96 registers per thread; the distance variants spill up to 20 bytes outside their loops.
constexpr int TC_FUSED_WARPS_256 = 16;
__host__ __device__ constexpr int tc_epi_warps(int epi, int bn = 128) {   // 1, 2 = the fused loss epilogues
    return ((epi & 3) == 1 || (epi & 3) == 2) && bn == 256 ? TC_FUSED_WARPS_256 : TC_EPI_WARPS;
}
__host__ __device__ constexpr int tc_threads(int epi, int bn = 128) { return 32 * (2 + tc_epi_warps(epi, bn)); }
constexpr uint32_t TC_A_BYTES = TC_BM * TC_BK * 2;
constexpr uint32_t TC_MN_GROUP_BYTES = 64 * TC_BK * 2;    // MN-major operand: 64 contiguous elements x 64 K rows per TMA box
__host__ __device__ constexpr uint32_t tc_stage_bytes(int bn) { return TC_A_BYTES + (uint32_t)bn * TC_BK * 2; }
__host__ __device__ constexpr size_t tc_smem_bytes(int bn) { return 1024 + (size_t)TC_STAGES * tc_stage_bytes(bn) + 256; }

enum { EPI_STORE = 0, EPI_LOSS = 1, EPI_GRAD = 2, EPI_L2 = 4, EPI_CE = 8,    // L2 / CE: flags of the fused loss epilogues
       EPI_A1 = 16 };   // log-sigmoid loss of a distance score with self-adversarial temperature exactly 1 (see tc_loss_chunk)

struct TcGemmParams {
    int M, N, K;
    int kb_per_split;                     // 64-wide slices of K per split
    int tiles_m, tiles_n, items;          // items = splits * tiles_m * tiles_n
    int bn;                               // columns per tile (128 or 256)
    float* C; int64_t ldc;
    int64_t split_stride;                 // floats between the output slabs of consecutive K splits
    const float *row_norm2, *col_norm2;   // norm expansion: |q_b|^2 [M], |t_n|^2 [N]
    int32_t* status;
    int wait_limit;                       // tries of a bounded barrier wait
    // fused loss epilogues (EPI_LOSS, EPI_GRAD): the score is acc, or for l2 != 0 the distance score above
    int l2, loss;
    float gamma, adv_temp, ce_c, loss_scale;
    int row_pieces;                       // pieces of TC_PIECE columns per row of stat_part
    float4* stat_part;                    // [M, row_pieces] per column piece: (base-2 reference, sum exp, weighted loss sum, -)
    const float2* row_stat;               // [M] EPI_LOSS: (base-2 reference, -); EPI_GRAD: (base-2 maximum, 1 / normaliser), 0: row is finished
    const int32_t* redo;                  // EPI_GRAD: whether there is any row to do
    uint16_t* Gb; int64_t ldg;            // [M, ldg] bf16 dL/dF (divided by the distance for l2)
};

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"(tm), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile written by TMA with the 128-byte
// swizzle: rows of 128 bytes, groups of 8 rows 1024 bytes apart, tile base 1024-byte aligned.
__device__ __forceinline__ uint64_t umma_desc_k_sw128(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);   // start address, 16-byte units
    d |= (uint64_t)1 << 16;                          // leading byte offset (not used by swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;                          // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                          // layout type: 128-byte swizzle
    return d;
}

// The same for an operand whose M (or N) index is the contiguous one ("MN-major"), as TMA leaves
// it from boxes of 64 contiguous elements x 64 K rows: inside a box a K row is 128 bytes, groups
// of 8 K rows are 1024 bytes apart (stride offset), the next 64 elements of M / N are one box
// (8192 bytes) further (leading offset).
__device__ __forceinline__ uint64_t umma_desc_mn_sw128(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(TC_MN_GROUP_BYTES >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor: D fp32, A and B bf16, M x N tile; a_mn / b_mn: that operand is MN-major.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int m, int n, bool a_mn = false, bool b_mn = false) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrives on the barrier once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// A CTA that gives up may not leave copies into its shared memory, or MMAs on its tensor memory, behind: these waits are bounded by
// the default limit even where a test has shortened the kernel's own.  (Where no wait ran out both are done when all warps are: asked
// for all the same, they cost nine launches of full-entity scoring 1.7 %, 39 queries x 432,015 x 128 218.8 -> 222.5 us.)
// The last copies into each of `stages` stages, of `issued` in all.
__device__ __forceinline__ void tc_settle_copies(uint64_t* full, int stages, int issued) {
    for (int r = max(0, issued - stages); r < issued; ++r) mbar_wait_idle(&full[r % stages], (r / stages) & 1, kDefaultWaitLimit);
}
// Every MMA this thread has issued; `done` is a barrier of its own.
__device__ __forceinline__ void tc_settle_mmas(uint64_t* done) {
    umma_commit(done);
    mbar_wait_idle(done, 0, kDefaultWaitLimit);
}
// An epilogue warp's wait for an accumulator, with one answer for all its lanes: false if it ran out or another warp gave up.
__device__ __forceinline__ bool tc_acc_ready(uint64_t* bar, uint32_t parity, int limit, volatile uint32_t* stop) {
    const bool ok = mbar_wait_bounded(bar, parity, limit) && !*stop;
    return __all_sync(0xffffffffu, ok);
}

// 32 consecutive fp32 columns of this thread's tensor-memory lane.
// (the registers are valid after tmem_ld_wait)
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Waits for this thread's outstanding tensor-memory loads; the registers pass through, so that nothing that uses them moves ahead.
__device__ __forceinline__ void tmem_ld_wait(float (&v)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]), "+f"(v[9]), "+f"(v[10]),
                   "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]), "+f"(v[16]), "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]),
                   "+f"(v[21]), "+f"(v[22]), "+f"(v[23]), "+f"(v[24]), "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29]), "+f"(v[30]),
                   "+f"(v[31])::"memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) { tmem_ld32_issue(taddr, v); tmem_ld_wait(); }

// Two columns.
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, float (&v)[2]) {
    uint32_t a, b;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n" : "=r"(a), "=r"(b) : "r"(taddr));
    tmem_ld_wait();
    v[0] = __uint_as_float(a); v[1] = __uint_as_float(b);
}

struct TcItem { int z, m0, n0; };   // K split, first row, first column

constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;
__device__ __forceinline__ float fast_exp2(float y) { float r; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y)); return r; }
__device__ __forceinline__ float fast_log2(float y) { float r; asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y)); return r; }
__device__ __forceinline__ float fast_rcp(float y) { float r; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y)); return r; }
__device__ __forceinline__ float fast_rsqrt(float y) { float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y)); return r; }

// Maximum of three in one instruction.
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// The fused epilogues evaluate one transcendental per special-function instruction: their
// inputs come from bf16 operands, so the approximate forms (relative error about 2^-22) are
// far inside the error of the scores, and an epilogue of a d = 128 contraction is bound by
// exactly these instructions.
// sigmoid(z)
__device__ __forceinline__ float tc_sigmoid(float z) {
    const float e = fast_exp2(-fabsf(z) * kLog2e);
    const float r = fast_rcp(1.f + e);
    return z >= 0.f ? r : e * r;
}

// Score of a pair from the accumulator: the contraction itself, or (L2) the distance score of
// the norm expansion, with the reciprocal distance the gradient needs (0 at distance 0).
template <bool L2>
__device__ __forceinline__ float tc_score_inv(const TcGemmParams& p, float acc, float rn, int col, float& inv) {
    if (!L2) { inv = 0.f; return acc; }
    const float s2 = fmaxf(rn + p.col_norm2[col] - 2.f * acc, 0.f);
    inv = s2 > 0.f ? fast_rsqrt(s2) : 0.f;
    return -s2 * inv;
}
template <bool L2>
__device__ __forceinline__ float tc_score(const TcGemmParams& p, float acc, float rn, int col) {
    float inv;
    return tc_score_inv<L2>(p, acc, rn, col, inv);
}


// Per-row inputs of an epilogue, read before the accumulator is waited for.
struct TcRowState {
    float rn;                 // squared norm of the row (norm expansion)
    float cn[2];              // fused loss, norm expansion: squared norms of this lane's column of each of the warp's chunks of 32
    float2 st;                // EPI_LOSS: the row's (base-2 reference, -); EPI_GRAD: (base-2 maximum, 1 / normaliser)
};
template <int EPI>
__device__ __forceinline__ TcRowState tc_row_state(const TcGemmParams& p, int row) {
    TcRowState r{0.f, {}, make_float2(0.f, 0.f)};
    if (row >= p.M) return r;
    if ((EPI & EPI_L2) != 0) r.rn = p.row_norm2[row];
    if ((EPI & 3) == EPI_LOSS || (EPI & 3) == EPI_GRAD) r.st = p.row_stat[row];
    return r;
}

// The loss in one pass over the scores.  Per row, dL/dF is a function of the score over the row's normaliser Z, which is known
// only when the row has been seen; so what is written is dL/dF without that factor, E = e(f) u(f) with e = 2^(y - ref), y the
// base-2 exponent (a f log2 e for the self-adversarial weights, (f + c) log2 e for the sampled softmax) and u the rest
// (sigmoid(gamma + f), the reciprocal distance), and the factor loss_scale / Z joins afterwards: dQ's rows are multiplied by
// it, and dT's contraction takes q_b times it as its operand (both see as many roundings to bf16 as with the factor in E).
// bf16 and fp32 share their exponent range, so any reference within it serves: `ref` is the larger y of two of the row's
// negatives (the gather kernel computes them), a lower bound of the maximum up to rounding and a constant.  A chunk of 32 scores that exceeds it
// by more than 2^TC_REF_SPAN takes its own maximum instead, which keeps the statistics in range, and the row is found by
// stats_combine_kernel and its E written again, over the true maximum and with the factor, by an EPI_GRAD launch that
// otherwise ends at once; so is a row whose scores all lie far below it (finish_low_row).  (Until then a pass for the statistics and one for the gradients, the scores recomputed: ComplEx
// softmax 4,096 x 16,384 x 256 34 + 53 us, TransE-L2 8,192 x 8,192 x 128 67 + 94 us.)
constexpr float TC_REF_SPAN = 80.f;
constexpr float TC_EXP_MIN = -126.f;      // below it an exponential is 0

// One chunk of 32 scores.  FULL: all 32 columns lie inside the problem (no per-element masking); otherwise the first `valid`
// do.  k0: the exponent's constant less the reference; cn: the columns' squared norms (shared memory, norm expansion).  Returns what was
// subtracted beyond the reference.
// A1 (distance scores f <= 0, log-sigmoid loss, temperature a = 1): with K = exp(gamma) 2^ref, exp(gamma + f) = K e =: t, so
// softplus(gamma + f) = log(1 + t) and sigmoid(gamma + f) = t / (1 + t): four special-function instructions per score
// (distance, exponential, logarithm, reciprocal).
// K is gone where it is below 2^-126; a chunk whose largest t would not be takes its own maximum too.
// An L2 score is at most 0, so only a row whose reference is far below (`low`) can exceed it by much, and the chunk's maximum
// is looked for only in a warp that holds such a row; the other scores' maximum is a tree of three-input maxima.
template <bool L2, bool CE, bool FULL, bool A1>
__device__ __forceinline__ float tc_loss_chunk(const TcGemmParams& p, const float (&v)[32], float rn, int ncol, int valid,
                                               float k1, float k0, float ref, bool low, const float* cn, float& z, float& l, uint32_t (&g2)[16]) {
    auto score = [&](int i, float& inv) {
        if (!L2) { inv = 0.f; return v[i]; }
        const float s2 = fmaxf(fmaf(-2.f, v[i], rn + cn[i]), 0.f);
        inv = s2 > 0.f ? fast_rsqrt(s2) : 0.f;
        return -s2 * inv;
    };
    float fm = -INFINITY;
    if (!L2) {
        float vm[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = FULL || 8 * j + i < valid ? v[8 * j + i] : -INFINITY;
            vm[j] = max3(max3(x[0], x[1], x[2]), max3(x[3], x[4], x[5]), fmaxf(x[6], x[7]));
        }
        fm = fmaxf(max3(vm[0], vm[1], vm[2]), vm[3]);
    } else if (__any_sync(0xffffffffu, low)) {      // the largest score is that of the smallest squared distance
        float sm = INFINITY;
#pragma unroll
        for (int i = 0; i < 32; ++i) if (FULL || i < valid) sm = fminf(sm, fmaxf(fmaf(-2.f, v[i], rn + cn[i]), 0.f));
        fm = sm > 0.f ? -sm * fast_rsqrt(sm) : 0.f;
    }
    const float ym = fmaf(fm, k1, k0);      // (k1 >= 0)
    float shift = ym > TC_REF_SPAN ? ym : 0.f;
    if (A1) {
        const float x = fmaf(p.gamma, kLog2e, ref);
        if (x < TC_EXP_MIN && x + ym >= TC_EXP_MIN) shift = ym;
    }
    const float kk = k0 - shift;
    const float kexp = A1 ? fast_exp2(fmaf(p.gamma, kLog2e, ref + shift)) : 0.f;
    float zv[4] = {0.f, 0.f, 0.f, 0.f}, lv[4] = {0.f, 0.f, 0.f, 0.f};
    auto one = [&](int i) {
        if (!FULL && i >= valid) return 0.f;
        float inv;
        const float f = score(i, inv);
        const float e = fast_exp2(fmaf(f, k1, kk));
        zv[i & 3] += e;
        float g = L2 ? e * inv : e;
        if (A1) {
            const float t = kexp * e, t1 = 1.f + t;
            lv[i & 3] = fmaf(e, fast_log2(t1), lv[i & 3]);
            g *= t * fast_rcp(t1);
        } else if (!CE) {
            // softplus(x) = max(x, 0) + log(1 + exp(-|x|)) and sigmoid(x) from one exponential
            const float x = p.gamma + f, w = fast_exp2(-fabsf(x) * kLog2e), w1 = 1.f + w, r = fast_rcp(w1);
            lv[i & 3] = fmaf(e, fmaf(fmaxf(x, 0.f), kLog2e, fast_log2(w1)), lv[i & 3]);
            g *= x >= 0.f ? r : w * r;
        }
        return g;
    };
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float a = one(2 * i), b = one(2 * i + 1);
        const __nv_bfloat162 pr = __floats2bfloat162_rn(a, b);
        g2[i] = *reinterpret_cast<const uint32_t*>(&pr);
    }
    z = (zv[0] + zv[1]) + (zv[2] + zv[3]);
    if (!CE) l = kLn2 * ((lv[0] + lv[1]) + (lv[2] + lv[3]));
    return shift;
}

// A warp's 32 rows x 32 columns of bf16 on their way to memory: through `stage` (2 KB of shared memory of its own), so that a store
// instruction writes whole 32-byte sectors, eight rows x 64 contiguous bytes instead of 16 bytes in each of 32 rows.  The 16-byte chunk c
// of row r sits at chunk c ^ ((r >> 1) & 3) of the row: both the row-wise writes and the 8-row reads then touch every bank once.
// `rows`: the rows (lanes) to be written; `valid`: columns inside the problem.
__device__ __forceinline__ void tc_put_bf16(const TcGemmParams& p, int row0, int ncol, int valid, uint32_t rows, const uint32_t (&g2)[16], uint4* stage) {
    const int lane = threadIdx.x & 31;
    if (valid == 32) {
        const int sw = (lane >> 1) & 3;
#pragma unroll
        for (int i = 0; i < 4; ++i) stage[lane * 4 + (i ^ sw)] = make_uint4(g2[4 * i], g2[4 * i + 1], g2[4 * i + 2], g2[4 * i + 3]);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = i * 8 + (lane >> 2), c = lane & 3;
            const uint4 val = stage[r * 4 + (c ^ ((r >> 1) & 3))];
            if (rows >> r & 1u) *reinterpret_cast<uint4*>(p.Gb + (int64_t)(row0 + r) * p.ldg + ncol + c * 8) = val;
        }
        __syncwarp();
    } else if (rows >> lane & 1u) {
        uint16_t* dst = p.Gb + (int64_t)(row0 + lane) * p.ldg + ncol;
#pragma unroll
        for (int i = 0; i < 32; ++i) if (i < valid) dst[i] = (uint16_t)(g2[i >> 1] >> ((i & 1) * 16));
    }
}

// This thread's 64 columns of one row.  `release`: called once the accumulator has been read.
template <bool L2, bool CE, bool A1, class Release>
__device__ __forceinline__ void tc_epilogue_loss(const TcGemmParams& p, const TcItem& it, int row, const TcRowState& rs, int col_off, uint32_t taddr, uint4* stage,
                                                 Release release) {
    static_assert(TC_PIECE == 64, "two chunks of 32 columns per piece");
    const bool rin = row < p.M;
    const float rn = rs.rn, ref = rs.st.x;
    const float k1 = CE ? kLog2e : p.adv_temp * kLog2e, k0 = (CE ? p.ce_c * kLog2e : 0.f) - ref;
    const bool low = L2 && (k0 > TC_REF_SPAN || (A1 && fmaf(p.gamma, kLog2e, ref) < TC_EXP_MIN));
    const uint32_t rows = __ballot_sync(0xffffffffu, rin);
    const int row0 = row - (int)(threadIdx.x & 31);
    float m = ref, z = 0.f, l = 0.f;
    auto chunk = [&](const float (&v)[32], int c0, float cnorm) {
        const int ncol = it.n0 + c0, valid = min(32, p.N - ncol);             // (the same for every lane; may be <= 0)
        if (valid <= 0) return;
        const float* cn = reinterpret_cast<const float*>(stage);
        if (L2) { reinterpret_cast<float*>(stage)[threadIdx.x & 31] = cnorm; __syncwarp(); }
        uint32_t g2[16];
        float cz, cl = 0.f, shift;
        if (valid == 32) shift = tc_loss_chunk<L2, CE, true, A1>(p, v, rn, ncol, valid, k1, k0, ref, low, cn, cz, cl, g2);
        else shift = tc_loss_chunk<L2, CE, false, A1>(p, v, rn, ncol, valid, k1, k0, ref, low, cn, cz, cl, g2);
        const float cm = ref + shift;
        if (cm == m) { z += cz; l += cl; }
        else {
            const float mm = fmaxf(m, cm), ra = fast_exp2(m - mm), rb = fast_exp2(cm - mm);
            z = z * ra + cz * rb; l = l * ra + cl * rb; m = mm;
        }
        if (L2) __syncwarp();
        tc_put_bf16(p, row0, ncol, valid, rows, g2, stage);
    };
    if (L2) {                                  // (both chunks at once spill here)
#pragma unroll 1
        for (int c = 0; c < TC_PIECE; c += 32) {
            float v[32];
            tmem_ld32(taddr + (uint32_t)c, v);
            if (c + 32 == TC_PIECE) release();
            chunk(v, col_off + c, c == 0 ? rs.cn[0] : rs.cn[1]);
        }
    } else {
        float v0[32], v1[32];
        tmem_ld32_issue(taddr, v0);            // both chunks are requested before the first is used
        tmem_ld32_issue(taddr + 32u, v1);
        tmem_ld_wait(v0); tmem_ld_wait(v1);
        release();                             // the next item is multiplied under this one's arithmetic
        chunk(v0, col_off, 0.f);
        chunk(v1, col_off + 32, 0.f);
    }
    const int piece = (it.n0 + col_off) / TC_PIECE;
    if (rin && piece < p.row_pieces) p.stat_part[(int64_t)row * p.row_pieces + piece] = make_float4(m, z, l, 0.f);
}

// The rows that EPI_LOSS could not finish: dL/dF from the recomputed score and the row's final (base-2 max, 1 / normaliser).
// A1: sigmoid(gamma + f) = t / (1 + t) with t = krow e, krow = exp(gamma) 2^max.
template <bool L2, bool CE, bool A1, class Release>
__device__ __forceinline__ void tc_epilogue_grad(const TcGemmParams& p, const TcItem& it, int row, const TcRowState& rs, int col_off, uint32_t taddr,
                                                 uint4* stage, Release release) {
    const uint32_t rows = __ballot_sync(0xffffffffu, row < p.M && rs.st.y != 0.f);
    if (rows == 0u) { release(); return; }
    const float k1 = CE ? kLog2e : p.adv_temp * kLog2e, k0 = (CE ? p.ce_c * kLog2e : 0.f) - rs.st.x;
    const float scale = p.loss_scale * rs.st.y;
    const float krow = A1 ? fast_exp2(fmaf(p.gamma, kLog2e, rs.st.x)) : 0.f;
    const float* cn = reinterpret_cast<const float*>(stage);
#pragma unroll 1
    for (int c = 0; c < TC_PIECE; c += 32) {
        float v[32];
        tmem_ld32(taddr + (uint32_t)c, v);
        if (c + 32 == TC_PIECE) release();
        const int ncol = it.n0 + col_off + c, valid = min(32, p.N - ncol);
        if (valid <= 0) continue;
        if (L2) { reinterpret_cast<float*>(stage)[threadIdx.x & 31] = c == 0 ? rs.cn[0] : rs.cn[1]; __syncwarp(); }
        uint32_t g2[16];
        auto one = [&](int i) {                          // (what lies outside the problem, or in a finished row, is not written)
            float f = v[i], inv = 1.f;
            if (L2) {
                const float s2 = fmaxf(fmaf(-2.f, v[i], rs.rn + cn[i]), 0.f);
                inv = s2 > 0.f ? fast_rsqrt(s2) : 0.f;
                f = -s2 * inv;
            }
            const float e = fast_exp2(fmaf(f, k1, k0));
            float g = scale * e;
            if (A1) { const float t = krow * e; g *= t * fast_rcp(1.f + t); }
            else if (!CE) g *= tc_sigmoid(p.gamma + f);
            return g * inv;
        };
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float a = one(2 * i), b = one(2 * i + 1);
            const __nv_bfloat162 pr = __floats2bfloat162_rn(a, b);
            g2[i] = *reinterpret_cast<const uint32_t*>(&pr);
        }
        if (L2) __syncwarp();
        tc_put_bf16(p, row - (int)(threadIdx.x & 31), ncol, valid, rows, g2, stage);
    }
}

// 1.0f if a > b, else 0.0f, in one instruction.
__device__ __forceinline__ float one_if_gt(float a, float b) {
    float r;
    asm("set.gt.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Largest float below x (x finite or -inf; -inf maps to itself).
__device__ __forceinline__ float float_below(float x) {
    if (x == 0.f) return __uint_as_float(0x80000001u);
    if (x == -INFINITY) return x;
    const uint32_t b = __float_as_uint(x);
    return __uint_as_float(x > 0.f ? b - 1u : b + 1u);
}

// Epilogue of one warp on one item: WIDTH columns [col_off, col_off + WIDTH) of the tile row held by
// this thread's tensor-memory lane (taddr points at the first of them).
template <int EPI, int WIDTH, class Release>
__device__ __forceinline__ void tc_epilogue(const TcGemmParams& p, const TcItem& it, int row, const TcRowState& rs, int col_off, uint32_t taddr, void* scratch, Release release) {
    static_assert((EPI & 3) == EPI_STORE || WIDTH == TC_PIECE, "the fused loss epilogues work on pieces of TC_PIECE columns");
    if ((EPI & 3) == EPI_LOSS || (EPI & 3) == EPI_GRAD) {
        uint4* stage = static_cast<uint4*>(scratch);
        if ((EPI & 3) == EPI_LOSS) tc_epilogue_loss<(EPI & EPI_L2) != 0, (EPI & EPI_CE) != 0, (EPI & EPI_A1) != 0>(p, it, row, rs, col_off, taddr, stage, release);
        else tc_epilogue_grad<(EPI & EPI_L2) != 0, (EPI & EPI_CE) != 0, (EPI & EPI_A1) != 0>(p, it, row, rs, col_off, taddr, stage, release);
        return;
    }
    float* const Cout = p.C + (int64_t)it.z * p.split_stride;
    const float rn = rs.rn;
#pragma unroll 1
    for (int c0 = col_off; c0 < col_off + WIDTH; c0 += 32) {
        float v[32];
        tmem_ld32(taddr + (uint32_t)(c0 - col_off), v);
        const int ncol = it.n0 + c0;
        if (EPI & EPI_L2) {   // the debug tap of the score block: the distance score of the norm expansion, as the fused epilogues form it
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = ncol + i < p.N ? tc_score<true>(p, v[i], rn, ncol + i) : 0.f;
        }
        if (ncol + 32 <= p.N && (p.ldc & 3) == 0) {
            // (warp-uniform) a lane holds 32 columns of its own row: stored as they are, every instruction would touch
            // 32 rows with 16 bytes each.  Through shared memory (128-byte rows, 16-byte pieces XOR-swizzled by row) an
            // instruction writes four rows' whole 128 bytes.
            float4* st = static_cast<float4*>(scratch);
            const int lane = threadIdx.x & 31, sw = lane & 7, row0 = row - lane;
#pragma unroll
            for (int i = 0; i < 8; ++i) st[lane * 8 + (i ^ sw)] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int r = j * 4 + (lane >> 3), c = lane & 7;
                const float4 val = st[r * 8 + (c ^ (r & 7))];
                if (row0 + r < p.M) *reinterpret_cast<float4*>(Cout + (int64_t)(row0 + r) * p.ldc + ncol + 4 * c) = val;
            }
            __syncwarp();
        } else if (row < p.M) {
            float* dst = Cout + (int64_t)row * p.ldc + ncol;
#pragma unroll
            for (int i = 0; i < 32; ++i) if (ncol + i < p.N) dst[i] = v[i];
        }
    }
    release();
}

// Work item = (K split, row tile, column tile), column tile fastest.  A CTA takes a contiguous
// run of items, so consecutive items mostly share their A rows (kept warm in L2).
__device__ __forceinline__ TcItem tc_item(const TcGemmParams& p, int64_t item) {
    const int tn = (int)(item % p.tiles_n), r = (int)(item / p.tiles_n);
    return TcItem{r / p.tiles_m, (r % p.tiles_m) * TC_BM, tn * p.bn};
}
// The same walk one item at a time: the divisions are paid once per CTA, not once per item and warp.
__device__ __forceinline__ void tc_item_next(const TcGemmParams& p, TcItem& it) {
    it.n0 += p.bn;
    if (it.n0 >= p.tiles_n * p.bn) {
        it.n0 = 0; it.m0 += TC_BM;
        if (it.m0 >= p.tiles_m * TC_BM) { it.m0 = 0; ++it.z; }
    }
}

// EPI_GRAD: the row tiles with a row to do, a bit for every `group` of them (in shared memory, every CTA finds them for itself); their items
// are dealt out to all CTAs in runs, like those of the other epilogues.
constexpr int TC_TODO_WORDS = 128;
__device__ __forceinline__ int tc_todo_group(const TcGemmParams& p) { return (p.tiles_m + 32 * TC_TODO_WORDS - 1) / (32 * TC_TODO_WORDS); }
// First set bit from `bit` on; there is one.
__device__ __forceinline__ int tc_todo_from(const uint32_t* todo, int bit) {
    int w = bit >> 5;
    uint32_t x = todo[w] & (~0u << (bit & 31));
    while (x == 0u) x = todo[++w];
    return 32 * w + __ffs(x) - 1;
}
__device__ __forceinline__ TcItem tc_todo_item(const TcGemmParams& p, const uint32_t* todo, int item) {
    const int group = tc_todo_group(p), tn = item % p.tiles_n, r = item / p.tiles_n;
    int bit = tc_todo_from(todo, 0);
    for (int k = r / group; k > 0; --k) bit = tc_todo_from(todo, bit + 1);
    return TcItem{0, (bit * group + r % group) * TC_BM, tn * p.bn};
}
// `more`: whether there is a next item.
__device__ __forceinline__ void tc_todo_next(const TcGemmParams& p, const uint32_t* todo, TcItem& it, bool more) {
    it.n0 += p.bn;
    if (it.n0 < p.tiles_n * p.bn || !more) return;
    const int group = tc_todo_group(p), tile = it.m0 / TC_BM + 1;
    it.n0 = 0;
    it.m0 = (tile % group != 0 ? tile : tc_todo_from(todo, tile / group) * group) * TC_BM;
}

// BN: columns per tile, 128 or 256.
template <int EPI, int BN = 128>
__global__ void __launch_bounds__(tc_threads(EPI, BN), 1) tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA,
                                                             const __grid_constant__ CUtensorMap tmB, TcGemmParams p) {
    constexpr uint32_t TC_STAGE_BYTES = tc_stage_bytes(BN);
    constexpr int NACC = 512 / BN;                      // fp32 accumulators in tensor memory, used in turn: all 512 columns
    constexpr uint32_t TC_TMEM_COLS = NACC * BN;
    constexpr int EW = tc_epi_warps(EPI, BN), EG = EW / 4, TC_THREADS = tc_threads(EPI, BN);
    constexpr int GCOLS = BN / EG;                      // columns per epilogue warp
    extern __shared__ unsigned char tc_smem_raw[];
    unsigned char* base = tc_smem_raw + ((1024u - (smem_u32(tc_smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(base + (size_t)TC_STAGES * TC_STAGE_BYTES);
    uint64_t* empty = full + TC_STAGES;
    uint64_t* acc_full = empty + TC_STAGES;    // [NACC] accumulator buffer written
    uint64_t* acc_empty = acc_full + NACC;       // [NACC] accumulator buffer drained by all epilogue warps
    uint64_t* done = acc_empty + NACC;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile uint32_t* stop = tmem_slot + 1;     // set by a warp whose wait ran out
    volatile uint32_t* filled = tmem_slot + 2;   // stages filled in all
    unsigned char* scratch_sm = base + (size_t)TC_STAGES * TC_STAGE_BYTES + 256;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ uint32_t todo[(EPI & 3) == EPI_GRAD ? TC_TODO_WORDS : 1];
    int items = p.items;
    if ((EPI & 3) == EPI_GRAD) {                        // (nothing in flight writes the flag)
        grid_dependency_wait();
        allow_dependents();
        if (*p.redo == 0) return;
        for (int i = threadIdx.x; i < TC_TODO_WORDS; i += TC_THREADS) todo[i] = 0u;
        __syncthreads();
        const int group = tc_todo_group(p), rows = group * TC_BM;
        for (int u = warp; u < (p.tiles_m + group - 1) / group; u += TC_THREADS / 32) {
            bool any = false;
            for (int64_t r = (int64_t)u * rows + lane, end = min((int64_t)(u + 1) * rows, (int64_t)p.M); r < end; r += 32) any = any || p.row_stat[r].y != 0.f;
            if (__any_sync(0xffffffffu, any) && lane == 0) atomicOr(&todo[u >> 5], 1u << (u & 31));
        }
        __syncthreads();
        int units = 0;
        for (int i = lane; i < TC_TODO_WORDS; i += 32) units += __popc(todo[i]);
        items = __reduce_add_sync(0xffffffffu, units) * group * p.tiles_n;
    }
    auto item_at = [&](int item) { return (EPI & 3) == EPI_GRAD ? tc_todo_item(p, todo, item) : tc_item(p, item); };
    auto item_next = [&](TcItem& it, bool more) { if ((EPI & 3) == EPI_GRAD) tc_todo_next(p, todo, it, more); else tc_item_next(p, it); };
    const int per_cta = (items + gridDim.x - 1) / gridDim.x;
    const int item_begin = blockIdx.x * per_cta;
    if ((EPI & 3) == EPI_GRAD && item_begin >= items) return;
    const int kb_total = (p.K + TC_BK - 1) / TC_BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < NACC; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], EW); }
        mbar_init(done, 1);
        *stop = 0;
        mbar_init_fence();
    }
    if (warp == 1) {   // one warp allocates both accumulator buffers and gives up the right to allocate more
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TC_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int item_end = min(items, item_begin + per_cta);
    if ((EPI & 3) == EPI_LOSS) grid_dependency_wait();     // (launched while the kernel before it drains)

    if (warp == 0) {
        if (lane == 0) {
            int ring = 0;    // slices issued so far: stage = ring % STAGES, phase = ring / STAGES
            // Without K splits and with a slice count that divides the ring, slice kb of every item
            // lands in the same stages, so the row tile that consecutive items share is still there from
            // the item before: it is fetched again only when it changes.  keep[s] = first row of the tile
            // held by stage s.
            const bool reuse = p.kb_per_split == kb_total && TC_STAGES % kb_total == 0;
            int keep[TC_STAGES];
#pragma unroll
            for (int s = 0; s < TC_STAGES; ++s) keep[s] = -1;
            TcItem it = item_at(item_begin);
            for (int item = item_begin; item < item_end && !*stop; ++item, item_next(it, item < item_end)) {
                const int kb0 = it.z * p.kb_per_split, nkb = min(p.kb_per_split, kb_total - kb0);
                for (int kb = 0; kb < nkb; ++kb, ++ring) {
                    const int s = ring % TC_STAGES;
                    if (!mbar_wait_idle(&empty[s], ((ring / TC_STAGES) & 1) ^ 1, p.wait_limit)) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); break; }
                    unsigned char* sa = base + (size_t)s * TC_STAGE_BYTES;
                    bool have = false;
#pragma unroll
                    for (int q = 0; q < TC_STAGES; ++q) if (q == s) { have = reuse && keep[q] == it.m0; keep[q] = it.m0; }
                    mbar_arrive_expect_tx(&full[s], have ? TC_STAGE_BYTES - TC_A_BYTES : TC_STAGE_BYTES);
                    const int k0 = (kb0 + kb) * TC_BK;
                    if (!have) tma_load_2d(sa, &tmA, k0, it.m0, &full[s]);
                    unsigned char* sb = sa + TC_A_BYTES;
#pragma unroll
                    for (int g = 0; g < BN / 128; ++g)   // boxes of 128 rows, one after the other
                        tma_load_2d(sb + g * (128 * TC_BK * 2), &tmB, k0, it.n0 + 128 * g, &full[s]);
                }
            }
            *filled = (uint32_t)ring;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(TC_BM, BN, false, false);
            int ring = 0;
            bool ok = true;
            TcItem it = item_at(item_begin);
            for (int item = item_begin, local = 0; item < item_end && ok && !*stop; ++item, ++local, item_next(it, item < item_end)) {
                const int nkb = min(p.kb_per_split, kb_total - it.z * p.kb_per_split);
                const int buf = local % NACC;
                // the epilogue warps must have drained this buffer (two items ago)
                if (!mbar_wait_idle(&acc_empty[buf], ((local / NACC) & 1) ^ 1, p.wait_limit)) { ok = false; break; }
                tc_fence_after();
                const uint32_t tmem_acc = tmem_base + (uint32_t)buf * BN;
                for (int kb = 0; kb < nkb; ++kb, ++ring) {
                    const int s = ring % TC_STAGES;
                    if (!mbar_wait_idle(&full[s], (ring / TC_STAGES) & 1, p.wait_limit)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(base + (size_t)s * TC_STAGE_BYTES);
#pragma unroll
                    for (int k = 0; k < TC_BK / 16; ++k) {   // one MMA covers 16 of K: 32 bytes of a K-major row, 16 rows MN-major
                        const uint64_t ad = umma_desc_k_sw128(sa + k * 32), bd = umma_desc_k_sw128(sa + TC_A_BYTES + k * 32);
                        umma_bf16(tmem_acc, ad, bd, idesc, (kb | k) != 0);
                    }
                    umma_commit(&empty[s]);            // the stage is free once these MMAs have read it
                }
                umma_commit(&acc_full[buf]);           // also after a failed wait, so the epilogue warps wake up
            }
            if (!ok) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); }
        }
    } else {
        const int quarter = warp & 3;                  // tensor-memory lanes this warp may read
        const int cgrp = (warp - 2) >> 2;              // which group of the tile's columns
        TcItem it = item_at(item_begin);
        for (int item = item_begin, local = 0; item < item_end; ++item, ++local) {
            if (local != 0) item_next(it, true);
            // what the epilogue needs of its row does not depend on the accumulator: fetched before the wait
            TcRowState rs = tc_row_state<EPI>(p, it.m0 + quarter * 32 + lane);
            if ((EPI & EPI_L2) != 0 && (EPI & 3) != EPI_STORE) {
#pragma unroll
                for (int i = 0; i < GCOLS / 32; ++i) {
                    const int col = it.n0 + cgrp * GCOLS + 32 * i + lane;
                    rs.cn[i] = col < p.N ? __ldg(p.col_norm2 + col) : 1.f;
                }
            }
            const int buf = local % NACC;
            const bool ok = tc_acc_ready(&acc_full[buf], (local / NACC) & 1, p.wait_limit, stop);
            tc_fence_after();
            if (!ok) { if (lane == 0) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); } break; }
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * BN + cgrp * GCOLS);
            // scratch after the barriers: 2 or 4 KB per epilogue warp for the stores of bf16 or fp32 tiles
            void* scratch = scratch_sm + (warp - 2) * ((EPI & 3) == EPI_STORE ? TC_STORE_STAGE_BYTES : TC_GRAD_STAGE_BYTES);
            tc_epilogue<EPI, GCOLS>(p, it, it.m0 + quarter * 32 + lane, rs, cgrp * GCOLS, taddr, scratch, [&] {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[buf]);
            });
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*stop) {
        if (lane == 0) {
            if (warp == 0) tc_settle_copies(full, TC_STAGES, (int)*filled);
            if (warp == 1) tc_settle_mmas(done);
        }
        __syncthreads();
    }
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TC_TMEM_COLS) : "memory");
}

// ------------------------------------------------------------------------------------------
// Both backward contractions of a step in one launch:
//   problem 0   dQ partial[z] = G . T     A = dL/dF read K-major,  B = negatives read MN-major
//   problem 1   dT partial[z] = G^T . Q   A = dL/dF read MN-major, B = queries read MN-major
// Launched one after the other, each gave every CTA a single item, so the pipeline fill, the drain
// of the accumulator and the launch were exposed twice (11-18 us of 41-47 us at B = 4096,
// N = 16384, d = 256).  Here the items of both problems form one list that the CTAs take in
// strides, two items per CTA at the shapes above, and the second item's MMAs run under the first
// item's drain (the accumulators are used in turn, as in tc_gemm_kernel).  Plain stores of fp32
// tiles; warp roles, barriers and bounded waits as in tc_gemm_kernel.
// ------------------------------------------------------------------------------------------
struct DualProb {
    int M, N, kb_total, kb_per_split, tiles_m, tiles_n, items;
    float* C; int64_t ldc, split_stride;
    // K in segments of seg_kb slices: the B operand's K coordinate starts over with every segment, and an MN-major
    // A operand moves a_seg_x columns to the right per segment instead of going on downwards (its segments lie
    // side by side in memory).  One segment = a plain contraction.
    int seg_kb, a_seg_x;
    // fold > 0: output column c goes to column c % fold of slab c / fold (slabs fold_stride floats apart)
    int fold; int64_t fold_stride;
    // XCOL: groups of 64 columns of B per tile; extra[split][row] receives the extra column
    int groups; float* extra;
};

// PAIR: the A operand has two K segments that meet the same slices of the B operand (two-term splits of dL/dF-like
// coefficients against one [x1 | x2] operand).  A stage then holds both segments' A tiles beside the one B tile and both
// are multiplied into the accumulator, so a B slice is fetched once instead of once per segment (a third fewer operand
// bytes per flop); K runs over one segment's slices.  Three stages instead of four fit.
// XCOL (norm expansion): the B operand has one more column than the output: ones in problem 0, the factor of every row of dL/dF
// as two bf16 terms in problem 1 (box tmX), which gives the sums of dL/dF over its rows and columns exactly as the contractions
// see it.  The box of 64 columns that holds it follows a tile's `groups` boxes; the last tile's MMAs are 16 columns wider
// for it.  The ones lie in shared memory from the start: problem 0's copies leave that box alone, and a CTA's items of problem 1
// come after those of problem 0.
// FORM: how the operands of both problems are read.  DUAL_STEP: as above.  DUAL_NT: A and B K-major (the encoder's two
// projections).  DUAL_TN: A and B MN-major (the encoder's two matrix gradients).
enum { DUAL_STEP = 0, DUAL_NT = 1, DUAL_TN = 2 };
template <int BN, bool PAIR = false, int FORM = DUAL_STEP, bool XCOL = false>
__global__ void __launch_bounds__(32 * (2 + TC_EPI_WARPS), 1) tc_gemm_dual_kernel(const __grid_constant__ CUtensorMap tmA0,
                                                                                    const __grid_constant__ CUtensorMap tmB0,
                                                                                    const __grid_constant__ CUtensorMap tmA1,
                                                                                    const __grid_constant__ CUtensorMap tmB1,
                                                                                    const __grid_constant__ CUtensorMap tmX,
                                                                                    DualProb q0, DualProb q1, int32_t* status, int wait_limit) {
    constexpr uint32_t A_BYTES = PAIR ? 2 * TC_A_BYTES : TC_A_BYTES;      // A tile(s) of a stage; the B tile follows
    constexpr uint32_t STAGE_BYTES = tc_stage_bytes(BN) + (PAIR ? TC_A_BYTES : 0u);
    constexpr int STAGES = PAIR ? 3 : TC_STAGES;
    constexpr int NACC = 512 / BN;
    constexpr uint32_t TMEM_COLS = NACC * BN;
    constexpr int EW = TC_EPI_WARPS, EG = EW / 4;
    extern __shared__ unsigned char tc_smem_raw[];
    unsigned char* base = tc_smem_raw + ((1024u - (smem_u32(tc_smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(base + (size_t)STAGES * STAGE_BYTES);
    uint64_t* empty = full + TC_STAGES;
    uint64_t* acc_full = empty + TC_STAGES;
    uint64_t* acc_empty = acc_full + NACC;
    uint64_t* done = acc_empty + NACC;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile uint32_t* stop = tmem_slot + 1;
    volatile uint32_t* filled = tmem_slot + 2;   // stages filled in all

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total = q0.items + q1.items;
    // item -> (problem, K split, first row, first column); column tile fastest inside a problem
    auto prob_of = [&](int item) { return item < q0.items ? 0 : 1; };
    auto item_of = [&](const DualProb& q, int local_item) {
        const int tn = local_item % q.tiles_n, r = local_item / q.tiles_n;
        return TcItem{r / q.tiles_m, (r % q.tiles_m) * TC_BM, tn * (XCOL ? 64 * q.groups : BN)};
    };
    auto last_tile = [&](const DualProb& q, const TcItem& it) { return it.n0 + 64 * q.groups >= q.N; };

    if (XCOL) {     // K row r of the box: 128 bytes, 16-byte piece c at c ^ (r & 7)
        for (int i = threadIdx.x; i < STAGES * 512; i += blockDim.x) {
            const int r = i >> 3 & 63, c = i & 7;
            *reinterpret_cast<uint4*>(base + (size_t)(i >> 9) * STAGE_BYTES + A_BYTES + q0.groups * TC_MN_GROUP_BYTES + r * 128 + c * 16) =
                make_uint4(c == (r & 7) ? 0x3F80u : 0u, 0u, 0u, 0u);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < NACC; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], EW); }
        mbar_init(done, 1);
        *stop = 0;
        mbar_init_fence();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    grid_dependency_wait();
    if (FORM != DUAL_STEP) allow_dependents();     // (in a step the SMs left over serve the id sort, not waiting CTAs)

    if (warp == 0) {
        if (lane == 0) {
            int ring = 0;
            for (int item = blockIdx.x; item < total && !*stop; item += gridDim.x) {
                const int which = prob_of(item);
                const DualProb q = which ? q1 : q0;
                const TcItem it = item_of(q, which ? item - q0.items : item);
                const CUtensorMap* ta = which ? &tmA1 : &tmA0;
                const CUtensorMap* tb = which ? &tmB1 : &tmB0;
                const int kb0 = it.z * q.kb_per_split, nkb = min(q.kb_per_split, q.kb_total - kb0);
                for (int kb = 0; kb < nkb; ++kb, ++ring) {
                    const int s = ring % STAGES;
                    if (!mbar_wait_idle(&empty[s], ((ring / STAGES) & 1) ^ 1, wait_limit)) { *stop = 1; set_status(status, KGE_ERR_TIMEOUT); break; }
                    unsigned char* sa = base + (size_t)s * STAGE_BYTES;
                    const bool load_x = XCOL && which && last_tile(q, it);
                    mbar_arrive_expect_tx(&full[s], XCOL ? A_BYTES + (uint32_t)(q.groups + (load_x ? 1 : 0)) * TC_MN_GROUP_BYTES : STAGE_BYTES);
                    const int kblk = kb0 + kb, seg = PAIR ? 0 : kblk / q.seg_kb;
                    const int k0 = kblk * TC_BK, kseg = (kblk - seg * q.seg_kb) * TC_BK;
#pragma unroll
                    for (int half = 0; half < (PAIR ? 2 : 1); ++half) {       // PAIR: both segments' A tiles of this slice
                        unsigned char* da = sa + half * TC_A_BYTES;
                        if (FORM == DUAL_TN || (FORM == DUAL_STEP && which)) {      // the contraction index as rows: two boxes of 64 output rows
#pragma unroll
                            for (int g = 0; g < TC_BM / 64; ++g)
                                tma_load_2d(da + g * TC_MN_GROUP_BYTES, ta, it.m0 + 64 * g + (PAIR ? half : seg) * q.a_seg_x, kseg, &full[s]);
                        } else {
                            tma_load_2d(da, ta, k0 + half * q.seg_kb * TC_BK, it.m0, &full[s]);
                        }
                    }
                    if (FORM == DUAL_NT) {
#pragma unroll
                        for (int g = 0; g < BN / 128; ++g) tma_load_2d(sa + A_BYTES + g * (128 * TC_BK * 2), tb, kseg, it.n0 + 128 * g, &full[s]);
                    } else if (XCOL) {
                        for (int g = 0; g < q.groups; ++g) tma_load_2d(sa + A_BYTES + g * TC_MN_GROUP_BYTES, tb, it.n0 + 64 * g, kseg, &full[s]);
                        if (load_x) tma_load_2d(sa + A_BYTES + q.groups * TC_MN_GROUP_BYTES, &tmX, 0, kseg, &full[s]);
                    } else {
#pragma unroll
                        for (int g = 0; g < BN / 64; ++g) tma_load_2d(sa + A_BYTES + g * TC_MN_GROUP_BYTES, tb, it.n0 + 64 * g, kseg, &full[s]);
                    }
                }
            }
            *filled = (uint32_t)ring;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc_k = umma_idesc_bf16(TC_BM, BN, false, FORM != DUAL_NT), idesc_mn = umma_idesc_bf16(TC_BM, BN, true, true);
            int ring = 0;
            bool ok = true;
            for (int item = blockIdx.x, local = 0; item < total && ok && !*stop; item += gridDim.x, ++local) {
                const int which = prob_of(item);
                const DualProb q = which ? q1 : q0;
                const TcItem it = item_of(q, which ? item - q0.items : item);
                const int nkb = min(q.kb_per_split, q.kb_total - it.z * q.kb_per_split);
                const int buf = local % NACC;
                const int cols = 64 * q.groups + (last_tile(q, it) ? 16 : 0);       // XCOL
                const uint32_t idesc = XCOL ? umma_idesc_bf16(TC_BM, cols, which != 0, true) : 0u;
                if (!mbar_wait_idle(&acc_empty[buf], ((local / NACC) & 1) ^ 1, wait_limit)) { ok = false; break; }
                tc_fence_after();
                const uint32_t tmem_acc = tmem_base + (uint32_t)buf * BN;
                for (int kb = 0; kb < nkb; ++kb, ++ring) {
                    const int s = ring % STAGES;
                    if (!mbar_wait_idle(&full[s], (ring / STAGES) & 1, wait_limit)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(base + (size_t)s * STAGE_BYTES);
#pragma unroll
                    for (int half = 0; half < (PAIR ? 2 : 1); ++half) {
#pragma unroll
                        for (int k = 0; k < TC_BK / 16; ++k) {
                            const uint32_t aa = sa + half * TC_A_BYTES;
                            const bool a_mn = FORM == DUAL_TN || (FORM == DUAL_STEP && which);
                            const uint64_t ad = a_mn ? umma_desc_mn_sw128(aa + k * 2048) : umma_desc_k_sw128(aa + k * 32);
                            const uint64_t bd = FORM == DUAL_NT ? umma_desc_k_sw128(sa + A_BYTES + k * 32) : umma_desc_mn_sw128(sa + A_BYTES + k * 2048);
                            umma_bf16(tmem_acc, ad, bd, XCOL ? idesc : (a_mn ? idesc_mn : idesc_k), (kb | k | half) != 0);
                        }
                    }
                    umma_commit(&empty[s]);
                }
                umma_commit(&acc_full[buf]);           // also after a failed wait, so the epilogue warps wake up
            }
            if (!ok) { *stop = 1; set_status(status, KGE_ERR_TIMEOUT); }
        }
    } else {
        const int quarter = warp & 3;                  // tensor-memory lanes this warp may read
        const int cgrp = (warp - 2) >> 2;              // which half of the tile's columns
        constexpr int COLS = BN / EG;
        float4* st = reinterpret_cast<float4*>(base + (size_t)STAGES * STAGE_BYTES + 256) + (size_t)(warp - 2) * (TC_STORE_STAGE_BYTES / 16);
        for (int item = blockIdx.x, local = 0; item < total; item += gridDim.x, ++local) {
            const int buf = local % NACC;
            const bool ok = tc_acc_ready(&acc_full[buf], (local / NACC) & 1, wait_limit, stop);
            tc_fence_after();
            if (!ok) { if (lane == 0) { *stop = 1; set_status(status, KGE_ERR_TIMEOUT); } break; }
            const int which = prob_of(item);
            const DualProb q = which ? q1 : q0;
            const TcItem it = item_of(q, which ? item - q0.items : item);
            const int row = it.m0 + quarter * 32 + lane;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * BN);
            float* const Cout = q.C + (int64_t)it.z * q.split_stride;
            // (XCOL: a tile's columns are fewer than BN; the groups of warps take them 32 by 32 in turn)
#pragma unroll 1
            for (int c0 = cgrp * (XCOL ? 32 : COLS); c0 < (XCOL ? 64 * q.groups : (cgrp + 1) * COLS); c0 += XCOL ? 32 * EG : 32) {
                float v[32];
                tmem_ld32(taddr + (uint32_t)c0, v);
                const int ncol = it.n0 + c0;
                float* piece = Cout + ncol;                    // column ncol of row 0 of this item's slab
                if (q.fold > 0) piece += (int64_t)(ncol / q.fold) * (q.fold_stride - q.fold);   // (32-column pieces never straddle a fold)
                if (ncol + 32 <= q.N && (q.ldc & 3) == 0) {    // (warp-uniform) through shared memory: four rows' whole 128 bytes per store instruction
                    const int sw = lane & 7, row0 = row - lane;
#pragma unroll
                    for (int i = 0; i < 8; ++i) st[lane * 8 + (i ^ sw)] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int r = j * 4 + (lane >> 3), c = lane & 7;
                        const float4 val = st[r * 8 + (c ^ (r & 7))];
                        if (row0 + r < q.M) *reinterpret_cast<float4*>(piece + (int64_t)(row0 + r) * q.ldc + 4 * c) = val;
                    }
                    __syncwarp();
                } else if (row < q.M) {
                    float* dst = piece + (int64_t)row * q.ldc;
#pragma unroll
                    for (int i = 0; i < 32; ++i) if (ncol + i < q.N) dst[i] = v[i];
                }
            }
            if (XCOL && cgrp == EG - 1 && last_tile(q, it)) {
                float x[2];
                tmem_ld2(taddr + (uint32_t)(64 * q.groups), x);
                if (row < q.M) q.extra[(int64_t)it.z * q.M + row] = x[0] + x[1];    // (problem 0: the second column is zero)
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*stop) {
        if (lane == 0) {
            if (warp == 0) tc_settle_copies(full, STAGES, (int)*filled);
            if (warp == 1) tc_settle_mmas(done);
        }
        __syncthreads();
    }
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
}

// ------------------------------------------------------------------------------------------
// C[M, N] = A . B^T in fp32 accuracy from bf16 operands: both operands arrive as three-term splits x = x1 + x2 + x3 laid
// out side by side, [x1 | x2 | x3] with `tstride` columns per term (K rounded up to 64, padding zero), and the six
// products a_i b_j with i + j <= 4 are accumulated in fp32 (what is left out is below 2^-25 relative).  A stage holds
// one 64-wide K slice of all three terms of both operands (6 x 16 KB), so every slice is fetched once for the up to
// three products it takes part in: half the operand bytes of the same products run as one long K (each term's slice would
// be fetched once per product).  128 x 128 tiles, two stages, four accumulators in turn; warp roles, barriers and bounded
// waits as in tc_gemm_kernel; fp32 tiles leave through shared memory (see tc_epilogue).
// ------------------------------------------------------------------------------------------
struct TermsParams {
    int M, N, kslices, tstride;     // kslices = tstride / 64
    int tiles_m, tiles_n, items;    // column tile fastest
    float* C; int64_t ldc;
    int32_t* status; int wait_limit;
};
constexpr uint32_t TT_TERM_BYTES = 128 * TC_BK * 2;           // one term's 128 x 64 bf16 tile
constexpr uint32_t TT_STAGE_BYTES = 6 * TT_TERM_BYTES;
constexpr int TT_STAGES = 2;
constexpr size_t TT_SMEM = 1024 + (size_t)TT_STAGES * TT_STAGE_BYTES + 256 + (size_t)TC_EPI_WARPS * TC_STORE_STAGE_BYTES;

__global__ void __launch_bounds__(32 * (2 + TC_EPI_WARPS), 1) tc_gemm_terms_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                                     const __grid_constant__ CUtensorMap tmB, TermsParams p) {
    constexpr int BN = 128, NACC = 512 / BN;
    constexpr uint32_t TMEM_COLS = 512;
    extern __shared__ unsigned char tc_smem_raw[];
    unsigned char* base = tc_smem_raw + ((1024u - (smem_u32(tc_smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(base + (size_t)TT_STAGES * TT_STAGE_BYTES);
    uint64_t* empty = full + TT_STAGES;
    uint64_t* acc_full = empty + TT_STAGES;
    uint64_t* acc_empty = acc_full + NACC;
    uint64_t* done = acc_empty + NACC;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile uint32_t* stop = tmem_slot + 1;
    volatile uint32_t* filled = tmem_slot + 2;   // stages filled in all
    float4* store_stage = reinterpret_cast<float4*>(base + (size_t)TT_STAGES * TT_STAGE_BYTES + 256);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < TT_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < NACC; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], TC_EPI_WARPS); }
        mbar_init(done, 1);
        *stop = 0;
        mbar_init_fence();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int ring = 0;
            for (int item = blockIdx.x; item < p.items && !*stop; item += gridDim.x) {
                const int m0 = (item / p.tiles_n) * TC_BM, n0 = (item % p.tiles_n) * BN;
                for (int ks = 0; ks < p.kslices; ++ks, ++ring) {
                    const int s = ring % TT_STAGES;
                    if (!mbar_wait_idle(&empty[s], ((ring / TT_STAGES) & 1) ^ 1, p.wait_limit)) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); break; }
                    unsigned char* sa = base + (size_t)s * TT_STAGE_BYTES;
                    mbar_arrive_expect_tx(&full[s], TT_STAGE_BYTES);
#pragma unroll
                    for (int t = 0; t < 3; ++t) {
                        tma_load_2d(sa + t * TT_TERM_BYTES, &tmA, t * p.tstride + ks * TC_BK, m0, &full[s]);
                        tma_load_2d(sa + (3 + t) * TT_TERM_BYTES, &tmB, t * p.tstride + ks * TC_BK, n0, &full[s]);
                    }
                }
            }
            *filled = (uint32_t)ring;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(TC_BM, BN, false, false);
            int ring = 0;
            bool ok = true;
            for (int item = blockIdx.x, local = 0; item < p.items && ok && !*stop; item += gridDim.x, ++local) {
                const int buf = local % NACC;
                if (!mbar_wait_idle(&acc_empty[buf], ((local / NACC) & 1) ^ 1, p.wait_limit)) { ok = false; break; }
                tc_fence_after();
                const uint32_t tmem_acc = tmem_base + (uint32_t)buf * BN;
                for (int ks = 0; ks < p.kslices; ++ks, ++ring) {
                    const int s = ring % TT_STAGES;
                    if (!mbar_wait_idle(&full[s], (ring / TT_STAGES) & 1, p.wait_limit)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(base + (size_t)s * TT_STAGE_BYTES);
#pragma unroll
                    for (int ta = 0; ta < 3; ++ta) {
#pragma unroll
                        for (int tb = 0; tb < 3; ++tb) {
                            if (ta + tb > 2) continue;          // the six products that matter (terms counted from 0)
#pragma unroll
                            for (int k = 0; k < TC_BK / 16; ++k) {
                                const uint64_t ad = umma_desc_k_sw128(sa + ta * TT_TERM_BYTES + k * 32);
                                const uint64_t bd = umma_desc_k_sw128(sa + (3 + tb) * TT_TERM_BYTES + k * 32);
                                umma_bf16(tmem_acc, ad, bd, idesc, (ks | ta | tb | k) != 0);
                            }
                        }
                    }
                    umma_commit(&empty[s]);
                }
                umma_commit(&acc_full[buf]);           // also after a failed wait, so the epilogue warps wake up
            }
            if (!ok) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); }
        }
    } else {
        const int quarter = warp & 3;                  // tensor-memory lanes this warp may read
        const int cgrp = (warp - 2) >> 2;              // which half of the tile's columns
        constexpr int COLS = BN / (TC_EPI_WARPS / 4);
        float4* st = store_stage + (size_t)(warp - 2) * (TC_STORE_STAGE_BYTES / 16);
        for (int item = blockIdx.x, local = 0; item < p.items; item += gridDim.x, ++local) {
            const int buf = local % NACC;
            const bool ok = tc_acc_ready(&acc_full[buf], (local / NACC) & 1, p.wait_limit, stop);
            tc_fence_after();
            if (!ok) { if (lane == 0) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); } break; }
            const int m0 = (item / p.tiles_n) * TC_BM, n0 = (item % p.tiles_n) * BN;
            const int row0 = m0 + quarter * 32, row = row0 + lane;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * BN + cgrp * COLS);
#pragma unroll 1
            for (int c0 = cgrp * COLS; c0 < (cgrp + 1) * COLS; c0 += 32) {
                float v[32];
                tmem_ld32(taddr + (uint32_t)(c0 - cgrp * COLS), v);
                const int ncol = n0 + c0;
                if (ncol + 32 <= p.N && (p.ldc & 3) == 0) {      // (warp-uniform) four rows' whole 128 bytes per store instruction
                    const int sw = lane & 7;
#pragma unroll
                    for (int i = 0; i < 8; ++i) st[lane * 8 + (i ^ sw)] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int r = j * 4 + (lane >> 3), c = lane & 7;
                        const float4 val = st[r * 8 + (c ^ (r & 7))];
                        if (row0 + r < p.M) *reinterpret_cast<float4*>(p.C + (int64_t)(row0 + r) * p.ldc + ncol + 4 * c) = val;
                    }
                    __syncwarp();
                } else if (row < p.M) {
                    float* dst = p.C + (int64_t)row * p.ldc + ncol;
#pragma unroll
                    for (int i = 0; i < 32; ++i) if (ncol + i < p.N) dst[i] = v[i];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*stop) {
        if (lane == 0) {
            if (warp == 0) tc_settle_copies(full, TT_STAGES, (int)*filled);
            if (warp == 1) tc_settle_mmas(done);
        }
        __syncthreads();
    }
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
}

// ------------------------------------------------------------------------------------------
// Full-entity scoring (Section 3.1 "Inference"): a score survives into the query's candidate list if it is ordered before the query's
// current k-th best under (score descending, entity id ascending); entities ordered before the true tail are counted for its rank.
//
// The queries stay and the entities pass by.  A CTA keeps MT tiles of 128 queries in shared memory and runs 256-entity tiles past them,
// 64 coordinates (32 KB) at a time through a ring; each (query tile, entity tile) is one accumulator of 256 columns, two in
// turn; the sixteen epilogue warps (32 queries x 64 entities each) take an accumulator into registers and hand it back before they
// look at it, so that its next tile is multiplied meanwhile.  What an epilogue needs of its queries (threshold, true tail's
// score and id) and its rank count are registers for hundreds of tiles.  With the entity tile kept and the
// queries passing by, as before, every tile read them from L2 and added its counts to shared memory: 39.8 ms for 15,000 x
// 8 M x 128, 3,000 cycles per 128 x 256 tile against the MMAs' 1,024, most of it latency.
// MT = 2 for rows of at most 128 coordinates halves the entity bytes a SM reads per score (32 bytes a clock at the
// MMAs' full rate); longer rows leave no room for the second tile's ring.
// The table is to be read from HBM once.  Few query groups: as many CTAs for each, the CTAs of one entity range side by side.  Many:
// all CTAs walk the table one superblock of some 32 MB after the other, each through its own contiguous run of the superblock's (query
// group, entity tile) pairs, query group slowest, so that a CTA changes queries rarely.  (300 queries x 1 M x 320, three groups:
// superblocks that give every CTA enough pairs are then larger than L2 and each group reads the table for itself, 399 us.)
// ------------------------------------------------------------------------------------------
constexpr int SCAN_BN = 256, SCAN_WARPS = 16, SCAN_THREADS = 32 * (2 + SCAN_WARPS), SCAN_RING_MAX = 8;
constexpr uint32_t SCAN_SLICE_BYTES = SCAN_BN * TC_BK * 2;
constexpr size_t SCAN_SMEM_MAX = 227 * 1024;

struct ScanParams {
    int M, N, slices, tiles_m, groups, tiles_n, sb_tiles, ring;     // groups of MT query tiles; tiles per superblock
    int ctas_per_group;                   // 0: superblocks
    int64_t n_base, id_base;              // first table row of this launch; the caller's id of table row 0 (sharded inference)
    const float *thr, *ftrue;             // [M] current k-th best score; score of the true tail
    const int32_t *thr_id, *tt;           // [M] its id; true tail ids (or NULL)
    int32_t *cand_cnt, *beat_tmp;         // [M] candidates appended in this launch; entities ordered before the true tail
    float* cand_score; int32_t* cand_id;  // [M, cand_cap]
    int cand_cap;
    int32_t* overflow;                    // set when a candidate list is full: the call's later launches do nothing
    int32_t* status; int wait_limit;
};

// One query as its lane holds it: k-th best score, score and id of the true tail, entities before it so far, and one candidate
// (score, id) on its way to the query's list (no score: -inf).
struct ScanRow {
    float thr, ft;
    int32_t tt, beat;
    float cand;
    int32_t cand_id;
};
// Puts the lanes' candidates into their lists.  All lanes at once: one wait for the atomics.
__device__ __forceinline__ void scan_flush(const ScanParams& p, ScanRow& r, int row) {
    if (r.cand != -INFINITY) {
        const int slot = atomicAdd(&p.cand_cnt[row], 1);
        if (slot < p.cand_cap) {
            p.cand_score[(int64_t)row * p.cand_cap + slot] = r.cand;
            p.cand_id[(int64_t)row * p.cand_cap + slot] = r.cand_id;
        } else {
            *p.overflow = 1;   // the host redoes this chunk in shorter pieces
        }
        r.cand = -INFINITY;
    }
    __syncwarp();
}

// Calls f(query group, entity tile) for this CTA's pairs until it returns false.
template <class F>
__device__ __forceinline__ void scan_walk(const ScanParams& p, F f) {
    if (p.ctas_per_group) {
        const int g = blockIdx.x / p.ctas_per_group, c = blockIdx.x % p.ctas_per_group;
        const int end = (int)((int64_t)p.tiles_n * (c + 1) / p.ctas_per_group);
        for (int e = (int)((int64_t)p.tiles_n * c / p.ctas_per_group); e < end; ++e)
            if (!f(g, e)) return;
        return;
    }
    for (int sb = 0; sb < p.tiles_n; sb += p.sb_tiles) {
        const int tiles = min(p.sb_tiles, p.tiles_n - sb);
        const int64_t pairs = (int64_t)p.groups * tiles;
        const int64_t begin = pairs * blockIdx.x / gridDim.x, end = pairs * (blockIdx.x + 1) / gridDim.x;
        int g = (int)(begin / tiles), e = (int)(begin % tiles);
        for (int64_t i = begin; i < end; ++i) {
            if (!f(g, sb + e)) return;
            if (++e == tiles) { e = 0; ++g; }
        }
    }
}

// 32 scores of query `row` against the entities [e0, e0 + 32) from tile column `ncol` on.  Within a run of entity ids that does not contain
// the reference id, "ordered before (f0, id0)" is a plain comparison: f >= f0 if the run lies below id0, f > f0 if above; f >= f0
// is written f > (largest float below f0).  `cut`: that bound of the true tail, unless the true tail is among the warp's ids
// (`exact`); n: the count so far, in floating point on four chains (exact, and the additions go to the FMA pipe).
template <bool FIRST>
__device__ __forceinline__ void scan_chunk(const ScanParams& p, float (&v)[32], ScanRow& r, int row, int ncol, float cut, bool exact, float (&n)[4]) {
    const int valid = p.N - ncol;                                      // the same for every lane
    if (valid <= 0) return;
    const int32_t e0 = (int32_t)(p.n_base + p.id_base + ncol);
    if (valid < 32) {
#pragma unroll
        for (int i = 0; i < 32; ++i) if (i >= valid) v[i] = -INFINITY;   // never counted, never a candidate
    }
    if (!exact) {
        if (p.tt) {
#pragma unroll
            for (int i = 0; i < 32; ++i) n[i & 3] += one_if_gt(v[i], cut);
        }
    } else if (r.tt >= 0) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int32_t e = e0 + i;
            if (e != r.tt && (v[i] > r.ft || (v[i] == r.ft && e < r.tt))) ++r.beat;
        }
    }
    if constexpr (FIRST) {     // (a chunk starts at a multiple of 32 columns: whole 128-byte pieces of the row's list)
        if (row < p.M) {
            float4* dst = reinterpret_cast<float4*>(p.cand_score + (int64_t)row * p.cand_cap + ncol);
#pragma unroll
            for (int i = 0; i < 8; ++i) dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
    } else {
        float vm[4];           // a tree of three-input maxima, not a chain of 31
#pragma unroll
        for (int j = 0; j < 4; ++j)
            vm[j] = max3(max3(v[8 * j], v[8 * j + 1], v[8 * j + 2]), max3(v[8 * j + 3], v[8 * j + 4], v[8 * j + 5]), fmaxf(v[8 * j + 6], v[8 * j + 7]));
        const float vmax = fmaxf(max3(vm[0], vm[1], vm[2]), vm[3]);
        // Rare once the threshold has tightened, but one warp of sixteen meets it at most tiles, and the tile waits for the slowest of
        // them.  So nothing here waits for memory: a lane keeps its candidate until the query's next one comes, and then the warp
        // hands all it holds to the lists (every candidate at once with an atomic of its own: 11.8 ms for 15,000 x 2 M x 128, the
        // MMAs alone 6.0).
        unsigned hits = 0u;
        if (!__any_sync(0xffffffffu, vmax >= r.thr)) return;
#pragma unroll
        for (int i = 0; i < 32; ++i) if (v[i] >= r.thr) hits |= 1u << i;
        if (valid < 32) hits &= (1u << valid) - 1u;
        // (the tensor map covers every query that fits the workspace: the scores of a row outside the call come from whatever an
        // earlier call left there, and no finite or infinite threshold is above +inf)
        if (row >= p.M) hits = 0u;
        else if (vmax == r.thr) {                  // only ties with the k-th best: before it with a smaller id
            const int before = p.thr_id[row] - e0;
            hits &= before >= 32 ? ~0u : (before <= 0 ? 0u : (1u << before) - 1u);
        }
        while (__any_sync(0xffffffffu, hits != 0u)) {
            if (hits != 0u) {
                const int at = __ffs(hits) - 1;
                float f = v[0];
#pragma unroll
                for (int i = 1; i < 32; ++i) if (at == i) f = v[i];
                // (the k-th best score itself: before it only with a smaller id)
                if (f == r.thr && !(e0 + at < p.thr_id[row])) hits &= hits - 1u;
                else if (r.cand == -INFINITY) { r.cand = f; r.cand_id = e0 + at; hits &= hits - 1u; }
            }
            if (__any_sync(0xffffffffu, hits != 0u)) scan_flush(p, r, row);
        }
    }
}

// FIRST: nothing is filtered yet, the scores go to the candidate lists in entity order.
template <int MT, bool FIRST>
__global__ void __launch_bounds__(SCAN_THREADS, 1) tc_scan_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, ScanParams p) {
    extern __shared__ unsigned char tc_smem_raw[];
    unsigned char* base = tc_smem_raw + ((1024u - (smem_u32(tc_smem_raw) & 1023u)) & 1023u);
    unsigned char* slice0 = base + (size_t)MT * p.slices * TC_A_BYTES;
    uint64_t* full = reinterpret_cast<uint64_t*>(slice0 + (size_t)p.ring * SCAN_SLICE_BYTES);
    uint64_t* empty = full + SCAN_RING_MAX;
    uint64_t* acc_full = empty + SCAN_RING_MAX;    // [2] accumulator written
    uint64_t* acc_empty = acc_full + 2;            // [2] accumulator read by all epilogue warps
    uint64_t* q_full = acc_empty + 2;              // query tiles loaded / no longer read by any MMA
    uint64_t* q_free = q_full + 1;
    uint64_t* done = q_free + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile uint32_t* stop = tmem_slot + 1;       // set by a warp whose wait ran out
    volatile uint32_t* filled = tmem_slot + 3;     // [2] slices and groups of query tiles fetched in all
    volatile uint32_t* given_up = tmem_slot + 2;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < SCAN_RING_MAX; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], SCAN_WARPS); }
        mbar_init(q_full, 1); mbar_init(q_free, 1); mbar_init(done, 1);
        *stop = 0;
        // after a list overflowed: no pairs (one thread's reading: the flag may change while this launch runs)
        *given_up = *reinterpret_cast<volatile int32_t*>(p.overflow) != 0;
        mbar_init_fence();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(2u * SCAN_BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const bool idle = *given_up != 0;

    if (idle) {
    } else if (warp == 0) {
        if (lane == 0) {
            int ring = 0, phase = 1, cur = -1, changes = 0, fills = 0;
            bool ok = true;
            scan_walk(p, [&](int g, int e) {
                if (*stop) return false;
                if (g != cur) {                    // other queries: every MMA on the ones before must be done
                    cur = g;
                    if (!mbar_wait_idle(q_free, (changes & 1) ^ 1, p.wait_limit)) { ok = false; return false; }
                    ++changes;
                    const int tiles = min(MT, p.tiles_m - g * MT);
                    mbar_arrive_expect_tx(q_full, (uint32_t)(tiles * p.slices) * TC_A_BYTES);
                    for (int t = 0; t < tiles; ++t)
                        for (int kb = 0; kb < p.slices; ++kb)
                            tma_load_2d(base + (size_t)(t * p.slices + kb) * TC_A_BYTES, &tmA, kb * TC_BK, (g * MT + t) * TC_BM, q_full);
                }
                for (int kb = 0; kb < p.slices; ++kb) {
                    if (!mbar_wait_idle(&empty[ring], phase, p.wait_limit)) { ok = false; return false; }
                    mbar_arrive_expect_tx(&full[ring], SCAN_SLICE_BYTES);
                    unsigned char* dst = slice0 + (size_t)ring * SCAN_SLICE_BYTES;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        tma_load_2d(dst + h * (128 * TC_BK * 2), &tmB, kb * TC_BK, (int)p.n_base + e * SCAN_BN + 128 * h, &full[ring]);
                    if (++ring == p.ring) { ring = 0; phase ^= 1; }
                    ++fills;
                }
                return true;
            });
            if (!ok) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); }
            filled[0] = (uint32_t)fills; filled[1] = (uint32_t)changes;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(TC_BM, SCAN_BN, false, false);
            int ring = 0, phase = 0, cur = -1, changes = 0;
            int uses[2] = {0, 0}, turn = 0;
            bool ok = true;
            scan_walk(p, [&](int g, int e) {
                if (*stop) return false;
                if (g != cur) {
                    if (cur >= 0) umma_commit(q_free);
                    cur = g;
                    if (!mbar_wait_idle(q_full, changes & 1, p.wait_limit)) { ok = false; return false; }
                    ++changes;
                }
                const int tiles = min(MT, p.tiles_m - g * MT);
                int s = ring, ph = phase;
#pragma unroll
                for (int t = 0; t < MT; ++t) {
                    if (t >= tiles) break;
                    const int buf = MT == 1 ? turn : t;
                    const int used = buf ? uses[1]++ : uses[0]++;
                    if (!mbar_wait_idle(&acc_empty[buf], (used & 1) ^ 1, p.wait_limit)) { ok = false; return false; }
                    tc_fence_after();
                    s = ring; ph = phase;
                    for (int kb = 0; kb < p.slices; ++kb) {
                        // (the second query tile finds the slices that the first waited for)
                        if (!mbar_wait_idle(&full[s], ph, p.wait_limit)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t sa = smem_u32(base + (size_t)(t * p.slices + kb) * TC_A_BYTES);
                        const uint32_t sb = smem_u32(slice0 + (size_t)s * SCAN_SLICE_BYTES);
#pragma unroll
                        for (int k = 0; k < TC_BK / 16; ++k)
                            umma_bf16(tmem_base + (uint32_t)buf * SCAN_BN, umma_desc_k_sw128(sa + k * 32), umma_desc_k_sw128(sb + k * 32), idesc, (kb | k) != 0);
                        if (t + 1 == tiles) umma_commit(&empty[s]);
                        if (++s == p.ring) { s = 0; ph ^= 1; }
                    }
                    umma_commit(&acc_full[buf]);       // also after a failed wait, so the epilogue warps wake up
                    if (!ok) return false;
                }
                ring = s; phase = ph; turn ^= 1;
                return true;
            });
            if (!ok) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); }
        }
    } else {
        const int quarter = warp & 3, col0 = ((warp - 2) >> 2) * 64;            // (a warp reads the lanes of its own quarter only)
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col0;
        int cur = -1, turn = 0;
        uint32_t parity = 0;                       // bit b: parity of accumulator b's next full phase
        ScanRow rows[MT];
#pragma unroll
        for (int t = 0; t < MT; ++t) rows[t] = ScanRow{INFINITY, INFINITY, -1, 0, -INFINITY, 0};
        auto row_of = [&](int g, int t) { return (g * MT + t) * TC_BM + quarter * 32 + lane; };
        auto hand_over = [&] {
#pragma unroll
            for (int t = 0; t < MT; ++t) {
                if (rows[t].beat > 0) atomicAdd(&p.beat_tmp[row_of(cur, t)], rows[t].beat);
                scan_flush(p, rows[t], row_of(cur, t));
            }
        };
        bool ok = true;
        scan_walk(p, [&](int g, int e) {
            if (g != cur) {
                if (cur >= 0) hand_over();
                cur = g;
#pragma unroll
                for (int t = 0; t < MT; ++t) {
                    // rows outside the problem stay in the loop (the warp votes need every lane): no true tail, a threshold that only +inf reaches
                    const int row = row_of(g, t);
                    rows[t] = ScanRow{INFINITY, INFINITY, -1, 0, -INFINITY, 0};
                    if (row < p.M) {
                        rows[t].thr = p.thr[row];
                        if (p.tt) { rows[t].ft = p.ftrue[row]; rows[t].tt = p.tt[row]; }
                    }
                }
            }
            const int32_t id0 = (int32_t)(p.n_base + p.id_base + e * SCAN_BN + col0);
#pragma unroll 1
            for (int t = 0; t < MT; ++t) {                 // (one copy of the code: the rows change places)
                if (MT == 2) { const ScanRow x = rows[0]; rows[0] = rows[MT - 1]; rows[MT - 1] = x; }
                if (g * MT + t >= p.tiles_m) continue;
                ScanRow& r = rows[MT - 1];
                const int acc = MT == 1 ? turn : t;
                const bool exact = __any_sync(0xffffffffu, r.tt >= id0 && r.tt < id0 + 64);
                const float cut = r.tt < 0 ? INFINITY : (r.tt >= id0 + 64 ? float_below(r.ft) : r.ft);
                ok = tc_acc_ready(&acc_full[acc], parity >> acc & 1u, p.wait_limit, stop);
                parity ^= 1u << acc;
                tc_fence_after();
                if (!ok) return false;
                float va[32], vb[32];
                tmem_ld32_issue(taddr + (uint32_t)(acc * SCAN_BN), va);
                tmem_ld32_issue(taddr + (uint32_t)(acc * SCAN_BN + 32), vb);
                tmem_ld_wait(va); tmem_ld_wait(vb);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[acc]);
                float n[4] = {0.f, 0.f, 0.f, 0.f};
                scan_chunk<FIRST>(p, va, r, row_of(g, t), e * SCAN_BN + col0, cut, exact, n);
                scan_chunk<FIRST>(p, vb, r, row_of(g, t), e * SCAN_BN + col0 + 32, cut, exact, n);
                r.beat += (int)((n[0] + n[1]) + (n[2] + n[3]));
            }
            turn ^= 1;
            return true;
        });
        // (after a wait that ran out the call has failed, and `rows` may be in the order of the other tile: nothing of them is handed over)
        if (ok && cur >= 0) hand_over();
        if (!ok && lane == 0) { *stop = 1; set_status(p.status, KGE_ERR_TIMEOUT); }
    }
    tc_fence_before();
    __syncthreads();
    if (*stop) {
        if (lane == 0) {
            if (warp == 0) {
                tc_settle_copies(full, p.ring, (int)filled[0]);
                if (filled[1] > 0) mbar_wait_idle(q_full, (filled[1] - 1) & 1, kDefaultWaitLimit);
            }
            if (warp == 1) tc_settle_mmas(done);
        }
        __syncthreads();
    }
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2u * SCAN_BN) : "memory");
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

}  // namespace

// Tensor map of a row-major bf16 matrix [rows, cols] with leading dimension ld (ld % 8 == 0,
// base 16-byte aligned) read in boxes of box_rows rows x 64 columns with the 128-byte swizzle
// (128 rows for a K-major operand tile, 64 for an MN-major one); what a box covers beyond the
// matrix reads as zero.
int tc_make_operand_map(kge_handle* h, void* map_out, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) { std::snprintf(h->cuda_err, sizeof(h->cuda_err), "cuTensorMapEncodeTiled is not available from this driver"); return KGE_ERR_CUDA; }
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(static_cast<CUtensorMap*>(map_out), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base),
                          dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { std::snprintf(h->cuda_err, sizeof(h->cuda_err), "cuTensorMapEncodeTiled failed with code %d", (int)r); return KGE_ERR_CUDA; }
    return KGE_OK;
}

int tc_make_f32_tile_map(kge_handle* h, void* map_out, const void* base, int64_t rows, int64_t cols) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) { std::snprintf(h->cuda_err, sizeof(h->cuda_err), "cuTensorMapEncodeTiled is not available from this driver"); return KGE_ERR_CUDA; }
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 4};
    const cuuint32_t box[2] = {32, 64};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(static_cast<CUtensorMap*>(map_out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base),
                          dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { std::snprintf(h->cuda_err, sizeof(h->cuda_err), "cuTensorMapEncodeTiled failed with code %d", (int)r); return KGE_ERR_CUDA; }
    return KGE_OK;
}

namespace {

// One warp per positive merges the per-piece statistics of its row (and the positive score, which the sampled softmax
// normalises over too) into the per-positive loss, dL/df+ and the row's factor loss_scale / Z, and multiplies the row of the dT
// contraction's operand by it.  A row with a piece that left its reference (see tc_loss_chunk), or with no score anywhere near it,
// keeps its operand and a factor of one; its (max, 1 / Z) go to the launch that writes its dL/dF.
struct CombineParams {
    const float4* stat_part; int pieces; int B;
    const float* fpos;
    int loss; float gamma, ce_c, loss_scale;
    float2* row_stat; float *Lrow, *gpos;
    float* row_scale;                     // [B] what a row of dL/dF is still to be multiplied by
    const float4* Q; uint2* Qb; int d4;   // [B, d] query vectors; their bf16 copies
    uint32_t* Xq;                         // norm expansion: [B, 64] bf16, the factor as two terms beside the operand's columns, or NULL
    int32_t* redo;
    const uint2* Tb; int N;               // [N, d] bf16 copies of the negatives
    const float *qn2, *tn2;               // squared norms, norm expansion only
    float k1, k0;                         // base-2 exponent of a score: k1 f + k0
};

// What a row leaves behind, from its (base-2 maximum, sum of exponentials, weighted loss sum): the operand's factor, the loss, dL/df+.
// `good`: its dL/dF stands up to the factor loss_scale / z; otherwise it is left to the second round.
__device__ __forceinline__ void finish_row(const CombineParams& p, int b, int lane, float fp, float m, float z, float l, bool good) {
    const float scale = good ? p.loss_scale / z : 1.f;
    if (good)
        for (int c = lane; c < p.d4; c += 32) {
            const float4 q = p.Q[(int64_t)b * p.d4 + c];
            const __nv_bfloat162 lo = __floats2bfloat162_rn(scale * q.x, scale * q.y), hi = __floats2bfloat162_rn(scale * q.z, scale * q.w);
            p.Qb[(int64_t)b * p.d4 + c] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        }
    if (p.Xq) {
        const __nv_bfloat16 hi = __float2bfloat16_rn(scale), lo = __float2bfloat16_rn(scale - __bfloat162float(hi));
        p.Xq[(int64_t)b * 32 + lane] = lane == 0 ? (uint32_t)__bfloat16_as_ushort(hi) | (uint32_t)__bfloat16_as_ushort(lo) << 16 : 0u;
    }
    if (lane != 0) return;
    if (p.loss == KGE_LOSS_SAMPLED_SOFTMAX) {
        const float epos = exp2f(fp * kLog2e - m);
        p.Lrow[b] = -fp + (m + log2f(z)) * 0.6931471805599453f;
        p.gpos[b] = p.loss_scale * (epos / z - 1.f);
    } else {
        const float zp = -(p.gamma + fp), ep = expf(-fabsf(zp)), rp = 1.f / (1.f + ep);   // once per row: the exact forms
        const float sp = fmaxf(zp, 0.f) + log1pf(ep), sg = zp >= 0.f ? rp : ep * rp;
        p.Lrow[b] = sp + l / z;
        p.gpos[b] = -p.loss_scale * sg;
    }
    p.row_scale[b] = scale;
    p.row_stat[b] = make_float2(m, good ? 0.f : 1.f / z);
    if (!good) *p.redo = 1;
}

// A row whose scores all lie so far below its reference that their exponentials are gone: the reference comes from the unrounded
// rows, and with norms or a temperature far beyond the usual the score block can be 2^126 below it.  The warp goes over the row's
// scores itself.  (Called last and with nothing to keep, so that the other rows' registers do not pay for it: called from the middle of
// the kernel, 0.9 to 1.4 us of a step at 4,096 x 16,384 and 8,192 x 8,192.)
__device__ __noinline__ void finish_low_row(const CombineParams& p, int b, int lane, float fp) {
    const bool ce = p.loss == KGE_LOSS_SAMPLED_SOFTMAX;
    const uint2* q = p.Qb + (int64_t)b * p.d4;
    const float rn = p.Xq ? p.qn2[b] : 0.f;
    float m = -INFINITY, z = 0.f, l = 0.f;
    for (int n = lane; n < p.N; n += 32) {
        const uint2* t = p.Tb + (int64_t)n * p.d4;
        float acc = 0.f;
        auto two = [&](uint32_t x, uint32_t y) {
            acc = fmaf(__uint_as_float(x << 16), __uint_as_float(y << 16), acc);
            acc = fmaf(__uint_as_float(x & 0xffff0000u), __uint_as_float(y & 0xffff0000u), acc);
        };
        for (int c = 0; c < p.d4; ++c) { const uint2 x = q[c], y = t[c]; two(x.x, y.x); two(x.y, y.y); }
        const float f = p.Xq ? -sqrtf(fmaxf(rn + p.tn2[n] - 2.f * acc, 0.f)) : acc, y = fmaf(f, p.k1, p.k0);
        if (y > m) { const float r = exp2f(m - y); z *= r; l *= r; m = y; }
        const float e = exp2f(y - m);
        z += e;
        if (!ce) l += e * softplusf(p.gamma + f);
    }
    float top = warp_max(m);
    const float r = m == -INFINITY ? 0.f : exp2f(m - top);
    z = warp_sum(z * r); l = warp_sum(l * r);
    if (ce) {                  // the positive score, which the sampled softmax normalises over too
        const float mm = fmaxf(top, fp * kLog2e);
        z = z * exp2f(top - mm) + exp2f(fp * kLog2e - mm);
        top = mm;
    }
    finish_row(p, b, lane, fp, top, z, l, false);
}

__global__ void __launch_bounds__(256, 8) stats_combine_kernel(const __grid_constant__ CombineParams p) {
    const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    grid_dependency_wait();
    allow_dependents();
    if (b >= p.B) return;
    const float4* row = p.stat_part + (int64_t)b * p.pieces;
    const float fp = p.fpos[b], ref = p.row_stat[b].x;
    const bool ce = p.loss == KGE_LOSS_SAMPLED_SOFTMAX;
    // the pieces carry their references and exponent sums in base 2 (exponent times log2 e)
    float m = -INFINITY;
    bool good = true;
    for (int j = lane; j < p.pieces; j += 32) { const float x = row[j].x; m = fmaxf(m, x); good = good && x == ref; }
    m = warp_max(m);
    good = __all_sync(0xffffffffu, good);
    if (ce && !good) m = fmaxf(m, fp * kLog2e);        // (a good row's reference is within 2^1 of it or above)
    float z = 0.f, l = 0.f;
    for (int j = lane; j < p.pieces; j += 32) {
        const float4 s = row[j];
        const float r = exp2f(s.x - m);
        z += s.y * r; l += s.z * r;
    }
    z = warp_sum(z); l = warp_sum(l);
    if (ce) z += exp2f(fp * kLog2e - m);
    if (z < 0x1p-40f) finish_low_row(p, b, lane, fp);  // (at 2^-40 the weights that matter are still 2^60 above the smallest number)
    else finish_row(p, b, lane, fp, m, z, l, good && z < INFINITY);
}

}  // namespace

namespace {
template <int EPI, int BN = 128>
cudaError_t launch_gemm_inst(const unsigned char* tmA, const unsigned char* tmB, const TcGemmParams& p, int num_sms, cudaStream_t s) {
    constexpr size_t smem = tc_smem_bytes(BN) + (size_t)tc_epi_warps(EPI, BN) * ((EPI & 3) == EPI_STORE ? TC_STORE_STAGE_BYTES : TC_GRAD_STAGE_BYTES);
    static DeviceOnce configured;
    const cudaError_t e = once_per_device(configured, [] {
        return cudaFuncSetAttribute(tc_gemm_kernel<EPI, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (e != cudaSuccess) return e;
    if ((EPI & 3) == EPI_LOSS || (EPI & 3) == EPI_GRAD)
        return launch_dependent(tc_gemm_kernel<EPI, BN>, dim3(std::min(p.items, num_sms)), dim3(tc_threads(EPI, BN)), smem, s,
                                *reinterpret_cast<const CUtensorMap*>(tmA), *reinterpret_cast<const CUtensorMap*>(tmB), p);
    tc_gemm_kernel<EPI, BN><<<std::min(p.items, num_sms), tc_threads(EPI, BN), smem, s>>>(
        *reinterpret_cast<const CUtensorMap*>(tmA), *reinterpret_cast<const CUtensorMap*>(tmB), p);
    return cudaSuccess;
}

// Scores Q . T^T with the fused loss epilogue, in tiles of BN columns.
template <int BN>
cudaError_t launch_loss_bn(bool l2, bool ce, kge_handle* h, const TcGemmParams& p, cudaStream_t s) {
    // the shared-exponential form of the log-sigmoid distance epilogue: temperature exactly 1, exp(gamma) finite
    if (l2 && !ce && p.adv_temp == 1.f && p.gamma <= 80.f) return launch_gemm_inst<EPI_LOSS | EPI_L2 | EPI_A1, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
    switch ((l2 ? 2 : 0) | (ce ? 1 : 0)) {
        case 0: return launch_gemm_inst<EPI_LOSS, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
        case 1: return launch_gemm_inst<EPI_LOSS | EPI_CE, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
        case 2: return launch_gemm_inst<EPI_LOSS | EPI_L2, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
        default: return launch_gemm_inst<EPI_LOSS | EPI_L2 | EPI_CE, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
    }
}
// The rows that launch could not finish: hardly ever more than a look at the flag.
template <int BN>
cudaError_t launch_redo_bn(bool l2, bool ce, kge_handle* h, const TcGemmParams& p, cudaStream_t s) {
    if (l2 && !ce && p.adv_temp == 1.f && p.gamma <= 80.f) return launch_gemm_inst<EPI_GRAD | EPI_L2 | EPI_A1, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
    switch ((l2 ? 2 : 0) | (ce ? 1 : 0)) {
        case 0: return launch_gemm_inst<EPI_GRAD, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
        case 1: return launch_gemm_inst<EPI_GRAD | EPI_CE, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
        case 2: return launch_gemm_inst<EPI_GRAD | EPI_L2, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
        default: return launch_gemm_inst<EPI_GRAD | EPI_L2 | EPI_CE, BN>(h->tm_q, h->tm_t, p, h->num_sms, s);
    }
}
}  // namespace

// Forward of the tensor-core path without the B x N score block ever leaving the chip: scores -> dL/dF up to a factor per row, as
// bf16, and per-piece statistics; merge per row -> loss, dL/df+, the factor; the rows that take another round, if any.
int launch_tc_forward(kge_handle* h, cudaStream_t s) {
    const kge_config& c = h->cfg;
    Workspace& w = h->ws;
    TcGemmParams p{};
    p.M = c.batch; p.N = c.num_neg; p.K = c.dim;
    p.kb_per_split = (p.K + TC_BK - 1) / TC_BK; p.split_stride = 0;
    // 256-column tiles halve the operand bytes fetched per score (the row tile is shared by twice
    // the columns); narrow problems keep 128 so that the tiles still spread over the SMs
    p.bn = (p.N >= 1024 && (int64_t)((p.M + TC_BM - 1) / TC_BM) * ((p.N + 255) / 256) >= h->num_sms) ? 256 : TC_BN;
    p.tiles_m = (p.M + TC_BM - 1) / TC_BM; p.tiles_n = (p.N + p.bn - 1) / p.bn; p.items = p.tiles_m * p.tiles_n;
    p.row_pieces = TC_EPI_GROUPS * ((p.N + TC_BN - 1) / TC_BN);
    p.C = nullptr; p.ldc = 0;
    p.row_norm2 = w.qn2; p.col_norm2 = w.tn2;
    p.status = w.status; p.wait_limit = h->wait_limit;
    p.l2 = h->kind == KIND_L2; p.loss = c.loss;
    p.gamma = c.gamma; p.adv_temp = c.adv_temp; p.ce_c = c.ce_correction; p.loss_scale = c.loss_scale;
    p.stat_part = reinterpret_cast<float4*>(w.stat_part); p.row_stat = reinterpret_cast<const float2*>(w.row_stat);
    p.Gb = w.Gb; p.ldg = (c.num_neg + 7) / 8 * 8;
    p.redo = w.status + TC_REDO_FLAG;
    const bool ce = c.loss == KGE_LOSS_SAMPLED_SOFTMAX;
    if (h->capture_scores) {
        // debug tap: this path never stores the score block, so an extra contraction writes it (fp32 [B, N]) with the
        // same mainloop and, for the norm expansion, the same score formula as the fused epilogues
        TcGemmParams cp = p;
        cp.bn = TC_BN; cp.tiles_n = (p.N + TC_BN - 1) / TC_BN; cp.items = cp.tiles_m * cp.tiles_n;
        cp.C = h->capture_scores; cp.ldc = p.N;
        if (p.l2) KGE_CUDA_CHECK(h, (launch_gemm_inst<EPI_STORE | EPI_L2, 128>(h->tm_q, h->tm_t, cp, h->num_sms, s)));
        else KGE_CUDA_CHECK(h, (launch_gemm_inst<EPI_STORE, 128>(h->tm_q, h->tm_t, cp, h->num_sms, s)));
        KGE_LAUNCH_CHECK(h);
    }
    stage_begin(h, ST_BLOCK, s);
    KGE_CUDA_CHECK(h, p.bn == 256 ? launch_loss_bn<256>(p.l2 != 0, ce, h, p, s) : launch_loss_bn<128>(p.l2 != 0, ce, h, p, s));
    stage_end(h, ST_BLOCK, s);
    KGE_LAUNCH_CHECK(h);
    stage_begin(h, ST_LOSS, s);
    CombineParams cp{p.stat_part, p.row_pieces, p.M, w.fpos, c.loss, c.gamma, c.ce_correction, c.loss_scale,
                     reinterpret_cast<float2*>(w.row_stat), w.Lrow, w.gpos, w.Grow, reinterpret_cast<const float4*>(w.Q),
                     reinterpret_cast<uint2*>(w.Qb), c.dim / 4, p.l2 ? reinterpret_cast<uint32_t*>(w.Xq) : nullptr, w.status + TC_REDO_FLAG,
                     reinterpret_cast<const uint2*>(w.Tb), c.num_neg, w.qn2, w.tn2, ce ? kLog2e : c.adv_temp * kLog2e, ce ? c.ce_correction * kLog2e : 0.f};
    KGE_CUDA_CHECK(h, launch_dependent(stats_combine_kernel, dim3((p.M * 32 + 255) / 256), dim3(256), 0, s, cp));
    KGE_LAUNCH_CHECK(h);
    KGE_CUDA_CHECK(h, p.bn == 256 ? launch_redo_bn<256>(p.l2 != 0, ce, h, p, s) : launch_redo_bn<128>(p.l2 != 0, ce, h, p, s));
    KGE_LAUNCH_CHECK(h);
    stage_end(h, ST_LOSS, s);
    return KGE_OK;
}

namespace {
// bn: columns per tile.
DualProb dual_prob(int M, int N, int K, int split, float* C, int64_t ldc, int bn) {
    DualProb q{};
    q.M = M; q.N = N;
    q.kb_total = (K + TC_BK - 1) / TC_BK;
    q.kb_per_split = (q.kb_total + split - 1) / split;
    q.tiles_m = (M + TC_BM - 1) / TC_BM; q.tiles_n = (N + bn - 1) / bn;
    q.items = q.tiles_m * q.tiles_n * ((q.kb_total + q.kb_per_split - 1) / q.kb_per_split);
    q.C = C; q.ldc = ldc; q.split_stride = (int64_t)M * ldc;
    q.seg_kb = q.kb_total; q.a_seg_x = 0; q.fold = 0; q.fold_stride = 0;
    q.groups = bn / 64; q.extra = nullptr;
    return q;
}
template <int BN, bool PAIR = false, int FORM = DUAL_STEP, bool XCOL = false>
cudaError_t launch_gemm_dual(kge_handle* h, const unsigned char* tmA0, const unsigned char* tmB0, const unsigned char* tmA1,
                             const unsigned char* tmB1, const DualProb& q0, const DualProb& q1, cudaStream_t s, const unsigned char* tmX = nullptr) {
    constexpr size_t smem = (PAIR ? 1024 + (size_t)3 * (tc_stage_bytes(BN) + TC_A_BYTES) + 256 : tc_smem_bytes(BN)) +
                            (size_t)TC_EPI_WARPS * TC_STORE_STAGE_BYTES;      // + the epilogue warps' store staging
    static DeviceOnce configured;
    const cudaError_t e = once_per_device(configured, [] {
        return cudaFuncSetAttribute(tc_gemm_dual_kernel<BN, PAIR, FORM, XCOL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (e != cudaSuccess) return e;
    // as few CTAs as give the same number of rounds: SMs left over serve the id sort that runs beside this launch
    const int total = q0.items + q1.items;
    const int rounds = (total + h->num_sms - 1) / h->num_sms;
    const int grid = (total + rounds - 1) / rounds;
    return launch_dependent(tc_gemm_dual_kernel<BN, PAIR, FORM, XCOL>, dim3(grid), dim3(32 * (2 + TC_EPI_WARPS)), smem, s,
                            *reinterpret_cast<const CUtensorMap*>(tmA0), *reinterpret_cast<const CUtensorMap*>(tmB0),
                            *reinterpret_cast<const CUtensorMap*>(tmA1), *reinterpret_cast<const CUtensorMap*>(tmB1),
                            *reinterpret_cast<const CUtensorMap*>(tmX ? tmX : tmB1), q0, q1, h->ws.status, h->wait_limit);
}
}  // namespace

// The feature-projection encoder's contractions, both roles in one launch.
//   C0[M0, N] = A0[M0, K] . B0[N, K]^T and C1[M1, N] = A1[M1, K] . B1[N, K]^T   (K-major: tensor maps with 128-row boxes)
int launch_tc_dual_nt(kge_handle* h, const unsigned char* tmA0, const unsigned char* tmB0, const unsigned char* tmA1, const unsigned char* tmB1,
                      int M0, int M1, int N, int K, float* C0, float* C1, cudaStream_t s) {
    const DualProb q0 = dual_prob(M0, N, K, 1, C0, N, 128), q1 = dual_prob(M1, N, K, 1, C1, N, 128);
    KGE_CUDA_CHECK(h, (launch_gemm_dual<128, false, DUAL_NT>(h, tmA0, tmB0, tmA1, tmB1, q0, q1, s)));
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}
//   C0[split0][M, N] = A0[K0, M]^T . B0[K0, N] over K slices of each split, and C1 likewise (MN-major: 64-row boxes)
int launch_tc_dual_tn(kge_handle* h, const unsigned char* tmA0, const unsigned char* tmB0, const unsigned char* tmA1, const unsigned char* tmB1,
                      int M, int N, int K0, int K1, int split0, int split1, float* C0, float* C1, cudaStream_t s) {
    const int bn = tc_backward_tile_cols(N);
    const DualProb q0 = dual_prob(M, N, K0, split0, C0, N, bn), q1 = dual_prob(M, N, K1, split1, C1, N, bn);
    KGE_CUDA_CHECK(h, bn == 256 ? (launch_gemm_dual<256, false, DUAL_TN>(h, tmA0, tmB0, tmA1, tmB1, q0, q1, s))
                                : (launch_gemm_dual<128, false, DUAL_TN>(h, tmA0, tmB0, tmA1, tmB1, q0, q1, s)));
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}
//   C[M, N] = A . B^T with fp32 accuracy from three-term bf16 splits [x1 | x2 | x3] of both operands (`tstride` columns per
//   term, a multiple of 64 with zero padding; tensor maps with 128-row boxes over [rows, 3 tstride])
int launch_tc_gemm_terms(kge_handle* h, const unsigned char* tmA, const unsigned char* tmB, int M, int N, int tstride, float* C,
                         int64_t ldc, cudaStream_t s) {
    TermsParams p{};
    p.M = M; p.N = N; p.tstride = tstride; p.kslices = tstride / TC_BK;
    p.tiles_m = (M + TC_BM - 1) / TC_BM; p.tiles_n = (N + 127) / 128; p.items = p.tiles_m * p.tiles_n;
    p.C = C; p.ldc = ldc; p.status = h->ws.status; p.wait_limit = h->wait_limit;
    static DeviceOnce configured;
    KGE_CUDA_CHECK(h, once_per_device(configured, [] {
        return cudaFuncSetAttribute(tc_gemm_terms_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TT_SMEM);
    }));
    tc_gemm_terms_kernel<<<std::min(p.items, h->num_sms), 32 * (2 + TC_EPI_WARPS), TT_SMEM, s>>>(
        *reinterpret_cast<const CUtensorMap*>(tmA), *reinterpret_cast<const CUtensorMap*>(tmB), p);
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}
bool tc_negatives_direct(const kge_handle* h) {
    // (with the regulariser on, the chain kernel still has a term to add to every negative's row)
    return h->cfg.prec == KGE_PREC_BF16_TC && h->kind == KIND_DOT && h->split_t == 1 && !(h->cfg.reg_lambda > 0.f);
}

// Columns per tile of a backward contraction whose output rows are `cols` wide.
int tc_backward_tile_cols(int cols) { return cols > 128 ? 256 : 128; }

// 64-column groups per tile and tiles of a backward contraction of the norm expansion, whose last tile needs room for one more
// group (see tc_gemm_dual_kernel): at most three groups in a tile of 256 columns.
static int tc_xcol_groups(int cols) { const int g = (cols + 63) / 64, tiles = (g + 2) / 3; return (g + tiles - 1) / tiles; }
// Column tiles of a backward contraction; `xcol`: of the norm expansion.
int tc_backward_col_tiles(int cols, bool xcol) {
    const int bn = xcol ? 64 * tc_xcol_groups(cols) : tc_backward_tile_cols(cols);
    return (cols + bn - 1) / bn;
}

// Column pieces per 128-wide tile for which the fused forward keeps separate statistics.
int tc_pieces_per_tile() { return TC_EPI_GROUPS; }

// The two backward contractions on tensor cores, from the bf16 dL/dF the forward left behind.
// No operand is transposed in memory: an operand whose contraction index is its row index is
// read MN-major.
//   dQ partial[split] = G . T      A = Gb [B, N] (K-major),          B operand = Tb [N, d] (MN-major)
//   dT partial[split] = G^T . Q    A = Gb [B, N] read MN-major,      B operand = Qb [B, d] (MN-major)
// The K splits land in the same partial buffers the CUDA-core path uses and are added in
// ascending order by the chain kernel.
int launch_tc_backward(kge_handle* h, cudaStream_t s, cudaStream_t side) {
    const kge_config& c = h->cfg;
    Workspace& w = h->ws;
    const int B = c.batch, N = c.num_neg, d = c.dim;
    (void)side;
    // one split and no correction term: the negatives' rows are final, so they go where the update reads them
    float* dT_out = tc_negatives_direct(h) ? w.grad_ent + (size_t)2 * B * d : w.dTpart;
    const bool xcol = h->kind == KIND_L2;
    const int bn = xcol ? 64 * tc_xcol_groups(d) : tc_backward_tile_cols(d);
    DualProb q0 = dual_prob(B, d, N, h->split_q, w.dQpart, d, bn), q1 = dual_prob(N, d, B, h->split_t, dT_out, d, bn);
    q0.extra = w.xsum_q; q1.extra = w.Cpart;
    stage_begin(h, ST_ACCUM_Q, s);        // (both contractions: the profile reports them as one stage)
    if (xcol)
        KGE_CUDA_CHECK(h, bn > 64 ? (launch_gemm_dual<256, false, DUAL_STEP, true>(h, h->tm_g, h->tm_t64, h->tm_g64, h->tm_q64, q0, q1, s, h->tm_x64))
                                  : (launch_gemm_dual<128, false, DUAL_STEP, true>(h, h->tm_g, h->tm_t64, h->tm_g64, h->tm_q64, q0, q1, s, h->tm_x64)));
    else
        KGE_CUDA_CHECK(h, bn == 256 ? launch_gemm_dual<256>(h, h->tm_g, h->tm_t64, h->tm_g64, h->tm_q64, q0, q1, s)
                                    : launch_gemm_dual<128>(h, h->tm_g, h->tm_t64, h->tm_g64, h->tm_q64, q0, q1, s));
    stage_end(h, ST_ACCUM_Q, s);
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}

// TransH on the fp32 path: the two contractions of the backward whose coefficient is one number per pair,
//   dW_b += sum_n c_bn t_n      and      dT_n += sum_b c_bn w_b,
// from bf16 two-term splits x = x1 + x2 of all three operands.  With the splits side by side, [c1 | c2] over K and
// [x1 | x2] over the output columns, one pass forms c1 x1 + c2 x1 in the left half of a tile and c1 x2 + c2 x2 in
// the right half: all four products, accumulated in fp32; the halves (and the K splits) land in slabs of their own
// behind the CUDA-core kernels' slabs and the chain kernel adds them in order.
int th_contract_slabs(const kge_handle* h) { return h->th_tc ? 2 * h->th_gsplit : 0; }

int launch_th_contract_gemm(kge_handle* h, cudaStream_t s) {
    const kge_config& c = h->cfg;
    Workspace& w = h->ws;
    const int B = c.batch, N = c.num_neg, d = c.dim;
    const int Np = (N + 63) / 64 * 64, Bp = (B + 63) / 64 * 64;
    const int bn = tc_backward_tile_cols(2 * d);
    // (K runs over one segment: both segments' tiles of c travel in one stage, see tc_gemm_dual_kernel<BN, PAIR>)
    DualProb q0 = dual_prob(B, 2 * d, Np, h->th_gsplit, w.dWpart + (size_t)h->split_q * B * d, d, bn);
    DualProb q1 = dual_prob(N, 2 * d, Bp, h->th_gsplit, w.dTpart + (size_t)h->split_t * N * d, d, bn);
    q0.seg_kb = Np / TC_BK; q0.a_seg_x = 0;
    q1.seg_kb = Bp / TC_BK; q1.a_seg_x = Np;
    q0.fold = q1.fold = d;
    q0.fold_stride = (int64_t)B * d; q0.split_stride = 2 * q0.fold_stride;
    q1.fold_stride = (int64_t)N * d; q1.split_stride = 2 * q1.fold_stride;
    KGE_CUDA_CHECK(h, bn == 256 ? (launch_gemm_dual<256, true>(h, h->tm_cs, h->tm_ts64, h->tm_cs64, h->tm_ws64, q0, q1, s))
                                : (launch_gemm_dual<128, true>(h, h->tm_cs, h->tm_ts64, h->tm_cs64, h->tm_ws64, q0, q1, s)));
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}


namespace {
__global__ void __launch_bounds__(256) cast_bf16_kernel(const float4* src, uint2* dst, int64_t n4) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 v = src[i];
        const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        dst[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    }
}
}  // namespace

// bf16 copy of `count` floats (count % 4 == 0, both 16-byte aligned).
int launch_cast_bf16(kge_handle* h, const float* src, uint16_t* dst, int64_t count, cudaStream_t s) {
    const int64_t n4 = count / 4;
    const int grid = (int)std::min<int64_t>((n4 + 255) / 256, (int64_t)h->num_sms * 16);
    cast_bf16_kernel<<<std::max(grid, 1), 256, 0, s>>>(reinterpret_cast<const float4*>(src), reinterpret_cast<uint2*>(dst), n4);
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}

// One chunk of full-entity scoring on tensor cores: the bf16 query vectors against the bf16
// rows [e_lo, e_hi) of the entity table, survivors appended to the candidate lists.
int launch_tc_infer_chunk(kge_handle* h, int nq, int64_t e_lo, int64_t e_hi, const int32_t* true_tails, int64_t id_base, int first, cudaStream_t s) {
    const Workspace& w = h->ws;
    ScanParams p{};
    p.M = nq; p.N = (int)(e_hi - e_lo);
    p.slices = (h->cfg.dim + TC_BK - 1) / TC_BK;
    p.tiles_m = (nq + TC_BM - 1) / TC_BM; p.tiles_n = (p.N + SCAN_BN - 1) / SCAN_BN;
    // two query tiles per CTA where that still gives every SM a pair (500 queries x 10,000 x 128: 103.7 us with two, 92.7 with one;
    // 257 x 1,000 57.1 and 49.7, which 128 x 256 tiles with the entities kept took 48.1 for; 700 x 150,000 189 and 184)
    const int mt = p.slices <= 2 && p.tiles_m > 1 && (int64_t)((p.tiles_m + 1) / 2) * p.tiles_n >= h->num_sms ? 2 : 1;
    p.groups = (p.tiles_m + mt - 1) / mt;
    const size_t fixed = 1024 + 256 + (size_t)mt * p.slices * TC_A_BYTES;
    p.ring = (int)std::min<size_t>(SCAN_RING_MAX, (SCAN_SMEM_MAX - fixed) / SCAN_SLICE_BYTES);
    int grid = (int)std::min<int64_t>((int64_t)p.groups * p.tiles_n, h->num_sms);
    // CTAs of their own for every group where that leaves at most one in sixteen idle
    const int per_group = std::min(h->num_sms / p.groups, p.tiles_n);
    p.ctas_per_group = per_group > 0 && (per_group == p.tiles_n || per_group * p.groups * 16 >= h->num_sms * 15) ? per_group : 0;
    if (p.ctas_per_group) grid = p.ctas_per_group * p.groups;
    // superblocks of about 32 MB, but at least 32 pairs per CTA in each
    const int64_t tile_bytes = (int64_t)SCAN_BN * h->cfg.dim * 2;
    const int64_t sb = std::max<int64_t>((int64_t)(32 << 20) / tile_bytes, ((int64_t)32 * grid + p.groups - 1) / p.groups);
    const int64_t n_sb = (p.tiles_n + sb - 1) / sb;
    p.sb_tiles = (int)((p.tiles_n + n_sb - 1) / n_sb);
    p.status = w.status; p.wait_limit = h->wait_limit;
    p.n_base = e_lo; p.id_base = id_base;
    p.thr = w.thr; p.thr_id = w.thr_id; p.ftrue = w.iftrue; p.tt = true_tails;
    p.cand_cnt = w.cand_cnt; p.beat_tmp = w.beat_tmp; p.cand_score = w.cand_score; p.cand_id = w.cand_id;
    p.cand_cap = kCandCap; p.overflow = w.status + 1;
    static DeviceOnce configured;
    KGE_CUDA_CHECK(h, once_per_device(configured, [] {
        cudaError_t e = cudaSuccess;
        for (auto k : {tc_scan_kernel<1, false>, tc_scan_kernel<1, true>, tc_scan_kernel<2, false>, tc_scan_kernel<2, true>})
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SCAN_SMEM_MAX);
        return e;
    }));
    // (the table's tensor map covers all rows; the kernel offsets its row coordinate by n_base)
    auto kernel = mt == 2 ? (first ? tc_scan_kernel<2, true> : tc_scan_kernel<2, false>) : (first ? tc_scan_kernel<1, true> : tc_scan_kernel<1, false>);
    kernel<<<grid, SCAN_THREADS, fixed + (size_t)p.ring * SCAN_SLICE_BYTES, s>>>(*reinterpret_cast<const CUtensorMap*>(h->tm_iq),
                                                                                 *reinterpret_cast<const CUtensorMap*>(h->tm_eb), p);
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}

}  // namespace kge
