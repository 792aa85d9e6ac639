// Feature-projection encoder (Section 3.1 "Encoder", Eq. 1): e = e_S + M e_F, with M = M_H for heads and M_T for
// tails and negatives.  Around the unchanged scoring step:
//   forward   gather the bf16 feature rows of the batch's 2B + N slots; P = F_slots . M^T on tensor cores (the
//             (B + N) |e_F| d term of the paper's cost model); the gather kernel of the step adds P to the rows it reads
//   backward  the slots' gradient rows (dL/de, which are also the shallow rows' gradients) rounded to bf16;
//             dM_H = dE_heads^T . F_heads, dM_T = dE_tails+negs^T . F_tails+negs as split-K contractions (both operands
//             read MN-major, nothing transposed in memory); one dense optimiser step per matrix that adds the K
//             splits in ascending order
#include <cmath>

#include <cuda_bf16.h>

#include "kge_sample.cuh"

namespace kge {

namespace {

struct PrepareParams {
    const uint16_t* feat; int F8;        // [E, F] bf16 features, F / 8 16-byte words per row
    int64_t E;
    const int32_t *heads, *tails, *negs;
    int B, N;
    uint16_t* out;                       // [2B+N, F]
    const float4 *MH, *MT; uint2* Mb;    // the matrices and their bf16 copies, m4 float4 each (MT: NULL when shared)
    int64_t m4;
    int pos_ctas, neg_ctas;
    int fused_sample, slots_per_bucket;
    SampleParams sp;
    int32_t* status;
};

__device__ __forceinline__ void copy_row(uint4* dst, const uint4* src, int n, int lane) {
    for (int c0 = 0; c0 < n; c0 += 128) {        // four loads in flight per lane
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { const int c = c0 + 32 * u + lane; if (c < n) v[u] = src[c]; }
#pragma unroll
        for (int u = 0; u < 4; ++u) { const int c = c0 + 32 * u + lane; if (c < n) dst[c] = v[u]; }
    }
}

// Everything the projection reads, in one launch (the sampling, the gather and two casts took a launch each, 18 us at
// B = 512, N = 1024, d = 256, F = 768): CTAs [0, pos_ctas) the feature rows of eight positives' heads and tails (a warp
// each; with fused_sample it draws its positive first), then those of eight negatives each, then the bf16 copies of the matrices.
__global__ void __launch_bounds__(256) encoder_prepare_kernel(PrepareParams p) {
    extern __shared__ uint64_t bucket_wcum[];   // fused sampling: cumulative weights of this CTA's buckets
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int blk = blockIdx.x;
    grid_dependency_wait();
    allow_dependents();
    const uint4* feat = reinterpret_cast<const uint4*>(p.feat);
    uint4* out = reinterpret_cast<uint4*>(p.out);
    if (blk < p.pos_ctas) {
        const int b = blk * 8 + warp;
        int32_t ih, ir, it;
        if (p.fused_sample) {
            stage_bucket_weights(p.sp, p.slots_per_bucket, blk * 8, bucket_wcum);
            __syncthreads();
            if (b >= p.B) return;
            if (lane == 0) {
                sample_positive_staged(p.sp, p.slots_per_bucket, blk * 8, b, bucket_wcum, ih, ir, it);
                p.sp.heads[b] = ih; p.sp.rels[b] = ir; p.sp.tails[b] = it;
            }
            ih = __shfl_sync(0xffffffffu, ih, 0); it = __shfl_sync(0xffffffffu, it, 0);
        } else {
            if (b >= p.B) return;
            ih = p.heads[b]; it = p.tails[b];
        }
        copy_row(out + (int64_t)b * p.F8, feat + checked_id(ih, p.E, p.status) * p.F8, p.F8, lane);
        copy_row(out + (int64_t)(p.B + b) * p.F8, feat + checked_id(it, p.E, p.status) * p.F8, p.F8, lane);
        return;
    }
    blk -= p.pos_ctas;
    if (blk < p.neg_ctas) {
        const int n = blk * 8 + warp;
        if (n >= p.N) return;
        int32_t neg;
        if (p.fused_sample) { neg = sample_negative(p.sp, n); if (lane == 0) p.sp.negs[n] = neg; }
        else neg = p.negs[n];
        copy_row(out + (int64_t)(2 * p.B + n) * p.F8, feat + checked_id(neg, p.E, p.status) * p.F8, p.F8, lane);
        return;
    }
    blk -= p.neg_ctas;
    const int64_t i = (int64_t)blk * 256 + threadIdx.x, all = p.MT ? 2 * p.m4 : p.m4;
    if (i >= all) return;
    const float4 v = i < p.m4 ? p.MH[i] : p.MT[i - p.m4];
    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    p.Mb[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

struct DenseMat {
    float* M; float* state;            // [rows, width]; Adam [rows, 2 width] (m | v); row-wise Adagrad [rows]
    const float* part; int splits;     // [splits][rows, width] partial gradients, added in ascending order
    const float* part2; int splits2;   // a second set (shared matrix: both roles), or NULL
};
struct DenseStep {
    DenseMat mat[2];
    int rows, width, opt;
    float lr, beta1, beta2, eps, corr1, corr2;
};

// One CTA per row of a matrix, CTAs [rows, 2 rows) the second matrix's: bound by reading the splits (one warp per row and
// a launch per matrix, a load after every addition, took 32 us per matrix at 256 x 768).
__global__ void __launch_bounds__(256) dense_step_kernel(DenseStep p) {
    __shared__ float red[8];
    const DenseMat m = p.mat[(int)blockIdx.x >= p.rows ? 1 : 0];
    const int row = (int)blockIdx.x % p.rows, tid = threadIdx.x;
    grid_dependency_wait();
    const int64_t slab = (int64_t)p.rows * p.width;
    auto sum = [&](const float* first, int n, float g) {         // eight loads in flight, added in ascending order
        for (int z0 = 0; z0 < n; z0 += 8) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = z0 + i < n ? first[(z0 + i) * slab] : 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) if (z0 + i < n) g += v[i];
        }
        return g;
    };
    auto grad = [&](int c) {
        const int64_t at = (int64_t)row * p.width + c;
        const float g = sum(m.part + at, m.splits, 0.f);
        return m.part2 ? sum(m.part2 + at, m.splits2, g) : g;
    };
    float* mrow = m.M + (int64_t)row * p.width;
    if (p.opt == KGE_OPT_SGD) {
        for (int c = tid; c < p.width; c += 256) mrow[c] -= p.lr * grad(c);
    } else if (p.opt == KGE_OPT_ADAM) {
        float* m1 = m.state + (int64_t)row * 2 * p.width;
        float* m2 = m1 + p.width;
        for (int c = tid; c < p.width; c += 256) {
            const float g = grad(c);
            const float a = p.beta1 * m1[c] + (1.f - p.beta1) * g, v = p.beta2 * m2[c] + (1.f - p.beta2) * g * g;
            m1[c] = a; m2[c] = v;
            mrow[c] -= p.lr * (a / p.corr1) / (sqrtf(v / p.corr2) + p.eps);
        }
    } else {
        float ss = 0.f;
        for (int c = tid; c < p.width; c += 256) { const float g = grad(c); ss += g * g; }
        ss = warp_sum(ss);
        if ((tid & 31) == 0) red[tid >> 5] = ss;
        __syncthreads();
        ss = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) ss += red[i];
        const float acc = m.state[row] + ss / (float)p.width;
        __syncthreads();               // every thread has read the old state
        if (tid == 0) m.state[row] = acc;
        const float stepv = p.lr / (sqrtf(acc) + p.eps);
        for (int c = tid; c < p.width; c += 256) mrow[c] -= stepv * grad(c);
    }
}

}  // namespace

int encoder_make_maps(kge_handle* h) {
    const kge_config& c = h->cfg;
    const Workspace& w = h->ws;
    const int64_t B = c.batch, N = c.num_neg, d = c.dim, F = c.feat_dim;
    int rc = tc_make_operand_map(h, h->tm_fh, w.Fb, B, F, F, 128);
    if (rc == KGE_OK) rc = tc_make_operand_map(h, h->tm_ft, w.Fb + B * F, B + N, F, F, 128);
    if (rc == KGE_OK) rc = tc_make_operand_map(h, h->tm_mh, w.Mb, d, F, F, 128);
    if (rc == KGE_OK) rc = tc_make_operand_map(h, h->tm_mt, w.Mb + d * F, d, F, F, 128);
    if (rc == KGE_OK) rc = tc_make_operand_map(h, h->tm_gh64, w.Gslot, B, d, d, 64);
    if (rc == KGE_OK) rc = tc_make_operand_map(h, h->tm_gt64, w.Gslot + B * d, B + N, d, d, 64);
    if (rc == KGE_OK) rc = tc_make_operand_map(h, h->tm_fh64, w.Fb, B, F, F, 64);
    if (rc == KGE_OK) rc = tc_make_operand_map(h, h->tm_ft64, w.Fb + B * F, B + N, F, F, 64);
    return rc;
}

int launch_encoder_forward(kge_handle* h, const int32_t* heads, const int32_t* tails, const int32_t* negs, bool fused_sample, uint64_t step, cudaStream_t s) {
    const kge_config& c = h->cfg;
    const Workspace& w = h->ws;
    const int B = c.batch, N = c.num_neg, d = c.dim, F = c.feat_dim;
    PrepareParams p{};
    p.feat = h->feat; p.F8 = F / 8; p.E = c.num_entities;
    p.heads = heads; p.tails = tails; p.negs = negs; p.B = B; p.N = N; p.out = w.Fb;
    p.MH = reinterpret_cast<const float4*>(h->MH); p.MT = c.feat_shared ? nullptr : reinterpret_cast<const float4*>(h->MT);
    p.Mb = reinterpret_cast<uint2*>(w.Mb); p.m4 = (int64_t)d * F / 4;
    p.pos_ctas = (B + 7) / 8; p.neg_ctas = (N + 7) / 8;
    p.fused_sample = fused_sample ? 1 : 0;
    p.slots_per_bucket = B / (c.head_part < 0 ? c.num_parts * c.num_parts : c.num_parts);
    p.sp = make_sample_params(h, step);
    p.sp.heads = w.heads; p.sp.rels = w.rels; p.sp.tails = w.tails; p.sp.negs = w.negs;
    p.status = w.status;
    const int64_t cast_ctas = ((p.MT ? 2 : 1) * p.m4 + 255) / 256;
    KGE_CUDA_CHECK(h, launch_dependent(encoder_prepare_kernel, dim3((unsigned)(p.pos_ctas + p.neg_ctas + cast_ctas)), dim3(256),
                                       fused_sample ? (size_t)fused_sample_smem(c.num_relations, p.slots_per_bucket) : 0, s, p));
    KGE_LAUNCH_CHECK(h);
    return launch_tc_dual_nt(h, h->tm_fh, h->tm_mh, h->tm_ft, c.feat_shared ? h->tm_mh : h->tm_mt, B, B + N, d, F, w.proj,
                             w.proj + (size_t)B * d, s);
}

int launch_encoder_backward(kge_handle* h, uint64_t step, float lr, cudaStream_t s) {
    const kge_config& c = h->cfg;
    const Workspace& w = h->ws;
    const int B = c.batch, N = c.num_neg, d = c.dim, F = c.feat_dim;
    if (tc_negatives_direct(h)) {       // the negatives' rows were written by a contraction; the others' bf16 copies came with the rows
        const int rc = launch_cast_bf16(h, w.grad_ent + (size_t)2 * B * d, w.Gslot + (size_t)2 * B * d, (int64_t)N * d, s);
        if (rc != KGE_OK) return rc;
    }
    auto real_splits = [](int K, int split) { const int kb = (K + 63) / 64, per = (kb + split - 1) / split; return (kb + per - 1) / per; };
    const int nH = real_splits(B, h->split_mh), nT = real_splits(B + N, h->split_mt);
    float* partH = w.dMpart;
    float* partT = w.dMpart + (size_t)h->split_mh * d * F;
    const int rc = launch_tc_dual_tn(h, h->tm_gh64, h->tm_fh64, h->tm_gt64, h->tm_ft64, d, F, B, B + N, h->split_mh, h->split_mt, partH, partT, s);
    if (rc != KGE_OK) return rc;
    DenseStep p{};
    p.rows = d; p.width = F; p.opt = c.opt;
    p.lr = lr; p.beta1 = c.beta1; p.beta2 = c.beta2; p.eps = c.eps;
    p.corr1 = (float)(1.0 - std::pow((double)c.beta1, (double)(step + 1)));
    p.corr2 = (float)(1.0 - std::pow((double)c.beta2, (double)(step + 1)));
    if (c.feat_shared) {
        p.mat[0] = DenseMat{h->MH, h->MH_state, partH, nH, partT, nT};
    } else {
        p.mat[0] = DenseMat{h->MH, h->MH_state, partH, nH, nullptr, 0};
        p.mat[1] = DenseMat{h->MT, h->MT_state, partT, nT, nullptr, 0};
    }
    KGE_CUDA_CHECK(h, launch_dependent(dense_step_kernel, dim3(c.feat_shared ? d : 2 * d), dim3(256), 0, s, p));
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}

}  // namespace kge
