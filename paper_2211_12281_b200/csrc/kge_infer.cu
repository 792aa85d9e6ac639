// Full-entity inference (Section 3.1 "Inference"): every query is scored against every
// entity; per query the k best tails under (score descending, id ascending) and the rank
// of the true tail.  The entity table is streamed once, in chunks that grow geometrically;
// inside a chunk a pair survives only if it beats the query's current k-th best, survivors
// are appended to a per-query candidate list, and a selection step between chunks merges
// them into the running top-k and tightens the threshold (the single-device analogue of the
// per-worker top-K followed by a final top-K over the gathered candidates).
//
// fp32 arithmetic here is "canonical": per pair one accumulator, embedding index ascending,
// rounding exactly where written (intrinsics keep the compiler from fusing anything else),
// so that ties and near-ties order the same way on any implementation of the same recipe.
#include <algorithm>
#include <climits>
#include <cmath>

#include <cuda_bf16.h>

#include <cuda.h>

#include "kge_common.cuh"

namespace kge {

namespace {

struct InferParams {
    int nq, k, d, d4, score, kind;
    int64_t E, R;
    const float *ent, *rel, *relw;
    const int32_t *qh, *qr, *tt;   // tt may be NULL
    int64_t e_lo, e_hi;            // entity range of this launch
    int q_tiles;
    int wait_limit;                // tries of a bounded barrier wait
    // sharded inference (Section 4 "Inference"): the bound table is the shard [id_base, id_base + E) of a larger one;
    // query vectors and true-tail scores come from outside (they need rows of other shards), ids are global
    int64_t id_base;
    const float* ext_q;            // [nq, d] finished query vectors, or NULL: build them from qh, qr
    const float* ext_ftrue;        // [nq] scores of the true tails, or NULL: score them here
    int raw_beat;                  // out_ranks receives the shard's count of entities ordered before the true tail, not 1 + count
    const uint16_t* Eb;            // tensor-core arithmetic: the bf16 copy of the table (the true tail is scored from it), or NULL
    int first;                     // first chunk: nothing is filtered, the scores go to the candidate lists in entity order
    int last;                      // last chunk: its selection writes the outputs
    int32_t* out_ids; float* out_scores; int32_t* out_ranks;
    Workspace w;                   // status[1]: a candidate list overflowed (nothing further of this call runs), status[6]: entities done
};

// One canonical accumulation step over the 4 floats of a slice.
template <int KIND>
__device__ __forceinline__ void canon_update(float& acc, float4 q, float4 t) {
    if (KIND == KIND_DOT) {
        acc = __fmaf_rn(q.x, t.x, acc); acc = __fmaf_rn(q.y, t.y, acc);
        acc = __fmaf_rn(q.z, t.z, acc); acc = __fmaf_rn(q.w, t.w, acc);
    } else if (KIND == KIND_L1) {
        acc = __fadd_rn(acc, fabsf(__fsub_rn(q.x, t.x))); acc = __fadd_rn(acc, fabsf(__fsub_rn(q.y, t.y)));
        acc = __fadd_rn(acc, fabsf(__fsub_rn(q.z, t.z))); acc = __fadd_rn(acc, fabsf(__fsub_rn(q.w, t.w)));
    } else if (KIND == KIND_L2) {
        float x;
        x = __fsub_rn(q.x, t.x); acc = __fmaf_rn(x, x, acc); x = __fsub_rn(q.y, t.y); acc = __fmaf_rn(x, x, acc);
        x = __fsub_rn(q.z, t.z); acc = __fmaf_rn(x, x, acc); x = __fsub_rn(q.w, t.w); acc = __fmaf_rn(x, x, acc);
    } else {  // KIND_CL1
        float xr = __fsub_rn(q.x, t.x), xi = __fsub_rn(q.y, t.y);
        acc = __fadd_rn(acc, __fsqrt_rn(__fmaf_rn(xr, xr, __fmul_rn(xi, xi))));
        xr = __fsub_rn(q.z, t.z); xi = __fsub_rn(q.w, t.w);
        acc = __fadd_rn(acc, __fsqrt_rn(__fmaf_rn(xr, xr, __fmul_rn(xi, xi))));
    }
}

__device__ __forceinline__ float4 canon_th_x(float u, float4 w, float4 q, float4 t) {
    const float2 a = sub2(make_float2(q.x, q.y), make_float2(t.x, t.y)), b = sub2(make_float2(q.z, q.w), make_float2(t.z, t.w));
    return make_float4(__fmaf_rn(u, w.x, a.x), __fmaf_rn(u, w.y, a.y), __fmaf_rn(u, w.z, b.x), __fmaf_rn(u, w.w, b.y));
}
__device__ __forceinline__ void canon_th_acc(int kind, float& acc, float4 x) {
    if (kind == KIND_TH_L1) {
        acc = __fadd_rn(acc, fabsf(x.x)); acc = __fadd_rn(acc, fabsf(x.y));
        acc = __fadd_rn(acc, fabsf(x.z)); acc = __fadd_rn(acc, fabsf(x.w));
    } else {
        acc = __fmaf_rn(x.x, x.x, acc); acc = __fmaf_rn(x.y, x.y, acc);
        acc = __fmaf_rn(x.z, x.z, acc); acc = __fmaf_rn(x.w, x.w, acc);
    }
}
__device__ __forceinline__ float canon_finish(int kind, float acc) {
    if (kind == KIND_DOT) return acc;
    if (kind == KIND_L2 || kind == KIND_TH_L2) return -__fsqrt_rn(acc);
    return -acc;
}

__device__ __forceinline__ bool ordered_before(float fa, int32_t ia, float fb, int32_t ib) {
    return fa > fb || (fa == fb && ia < ib);
}

// ------------------------------------------------------------------------------------------
// query set-up: one thread per query builds q (and the TransH unit normal) sequentially,
// scores the true tail, and resets the query's running state.
// ------------------------------------------------------------------------------------------
// TransH: the unit normal of relation rid into wh, sequentially.
__device__ __forceinline__ void unit_normal_seq(const InferParams& p, int64_t rid, float* wh) {
    const float* w = p.relw + rid * p.d;
    float s = 0.f;
    for (int k = 0; k < p.d; ++k) s = __fmaf_rn(w[k], w[k], s);
    const float den = fmaxf(__fsqrt_rn(s), 1e-12f);
    for (int k = 0; k < p.d; ++k) wh[k] = __fdiv_rn(w[k], den);
}

// Query vector of (head row h, relation rid) into qv (and the TransH unit normal into wh), sequentially.
__device__ __forceinline__ void build_query_seq(const InferParams& p, const float* h, int64_t rid, float* qv, float* wh) {
    const int d = p.d;
    if (p.score == KGE_TRANSE) {
        const float* r = p.rel + rid * d;
        for (int k = 0; k < d; ++k) qv[k] = __fadd_rn(h[k], r[k]);
    } else if (p.score == KGE_DISTMULT) {
        const float* r = p.rel + rid * d;
        for (int k = 0; k < d; ++k) qv[k] = __fmul_rn(r[k], h[k]);
    } else if (p.score == KGE_COMPLEX) {
        const float* r = p.rel + rid * d;
        for (int k = 0; k < d; k += 2) {
            qv[k] = __fmaf_rn(r[k], h[k], -__fmul_rn(r[k + 1], h[k + 1]));
            qv[k + 1] = __fmaf_rn(r[k], h[k + 1], __fmul_rn(r[k + 1], h[k]));
        }
    } else if (p.score == KGE_ROTATE) {
        const float* th = p.rel + rid * (d / 2);
        for (int k = 0; k < d; k += 2) {
            const float cs = cosf(th[k / 2]), sn = sinf(th[k / 2]);
            qv[k] = __fmaf_rn(h[k], cs, -__fmul_rn(h[k + 1], sn));
            qv[k + 1] = __fmaf_rn(h[k], sn, __fmul_rn(h[k + 1], cs));
        }
    } else {  // TransH
        const float* r = p.rel + rid * d;
        unit_normal_seq(p, rid, wh);
        float a = 0.f;
        for (int k = 0; k < d; ++k) a = __fmaf_rn(wh[k], h[k], a);
        for (int k = 0; k < d; ++k) qv[k] = __fadd_rn(__fmaf_rn(-a, wh[k], h[k]), r[k]);
    }
}

// Canonical score of (query vector qv, unit normal wh, tail row t).
__device__ __forceinline__ float score_seq(const InferParams& p, const float* qv, const float* wh, const float* t) {
    const int d = p.d;
    {
        float acc = 0.f;
        if (p.score == KGE_TRANSH) {
            float u = 0.f;
            for (int k = 0; k < d; ++k) u = __fmaf_rn(wh[k], t[k], u);
            for (int k = 0; k < d; k += 4)
                canon_th_acc(p.kind, acc, canon_th_x(u, *reinterpret_cast<const float4*>(wh + k),
                                                     *reinterpret_cast<const float4*>(qv + k),
                                                     *reinterpret_cast<const float4*>(t + k)));
        } else {
            for (int k = 0; k < d; k += 4) {
                const float4 q4 = *reinterpret_cast<const float4*>(qv + k);
                const float4 t4 = *reinterpret_cast<const float4*>(t + k);
                if (p.kind == KIND_DOT) canon_update<KIND_DOT>(acc, q4, t4);
                else if (p.kind == KIND_L1) canon_update<KIND_L1>(acc, q4, t4);
                else if (p.kind == KIND_L2) canon_update<KIND_L2>(acc, q4, t4);
                else canon_update<KIND_CL1>(acc, q4, t4);
            }
        }
        return canon_finish(p.kind, acc);
    }
}

// One warp per query (one thread per query read every row element by element: 105 us for 128 queries of width 256, 51 us
// for 15,000 of width 128).  The lanes fetch the rows and form what is independent per coordinate; a sum whose order is
// canonical runs on one lane, over rows in shared memory.
constexpr int SETUP_WARPS = 4;
__global__ void __launch_bounds__(32 * SETUP_WARPS) query_setup_kernel(InferParams p) {
    __shared__ __align__(16) float rows[SETUP_WARPS][3][kMaxDim];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = blockIdx.x * SETUP_WARPS + warp;
    allow_dependents();
    if (blockIdx.x == 0 && threadIdx.x == 0) { p.w.status[1] = 0; p.w.status[6] = 0; }
    if (q >= p.nq) return;
    const int d = p.d;
    const bool th = p.score == KGE_TRANSH;
    float *qv = rows[warp][0], *wh = rows[warp][1], *tv = rows[warp][2];
    const int64_t rid = checked_id(p.qr[q], p.R, p.w.status);
    if (th) {
        const float* wrow = p.relw + rid * d;
        for (int k = lane; k < d; k += 32) wh[k] = wrow[k];
        __syncwarp();
        float s = 0.f;
        if (lane == 0) for (int k = 0; k < d; ++k) s = __fmaf_rn(wh[k], wh[k], s);
        const float den = fmaxf(__fsqrt_rn(__shfl_sync(0xffffffffu, s, 0)), 1e-12f);
        for (int k = lane; k < d; k += 32) wh[k] = __fdiv_rn(wh[k], den);
        __syncwarp();
    }
    if (p.ext_q) {   // sharded: the query vector was built by the shard that holds the head
        for (int k = lane; k < d; k += 32) qv[k] = p.ext_q[(int64_t)q * d + k];
    } else {
        const float* h = p.ent + checked_id(p.qh[q], p.E, p.w.status) * d;
        if (p.score == KGE_TRANSE || p.score == KGE_DISTMULT) {
            const float* r = p.rel + rid * d;
            for (int k = lane; k < d; k += 32) qv[k] = p.score == KGE_TRANSE ? __fadd_rn(h[k], r[k]) : __fmul_rn(r[k], h[k]);
        } else if (p.score == KGE_COMPLEX) {
            const float* r = p.rel + rid * d;
            for (int k = 2 * lane; k < d; k += 64) {
                qv[k] = __fmaf_rn(r[k], h[k], -__fmul_rn(r[k + 1], h[k + 1]));
                qv[k + 1] = __fmaf_rn(r[k], h[k + 1], __fmul_rn(r[k + 1], h[k]));
            }
        } else if (p.score == KGE_ROTATE) {
            const float* ph = p.rel + rid * (d / 2);
            for (int k = 2 * lane; k < d; k += 64) {
                const float cs = cosf(ph[k / 2]), sn = sinf(ph[k / 2]);
                qv[k] = __fmaf_rn(h[k], cs, -__fmul_rn(h[k + 1], sn));
                qv[k + 1] = __fmaf_rn(h[k], sn, __fmul_rn(h[k + 1], cs));
            }
        } else {  // TransH
            const float* r = p.rel + rid * d;
            for (int k = lane; k < d; k += 32) tv[k] = h[k];
            __syncwarp();
            float a = 0.f;
            if (lane == 0) for (int k = 0; k < d; ++k) a = __fmaf_rn(wh[k], tv[k], a);
            a = __shfl_sync(0xffffffffu, a, 0);
            for (int k = lane; k < d; k += 32) qv[k] = __fadd_rn(__fmaf_rn(-a, wh[k], tv[k]), r[k]);
        }
    }
    __syncwarp();
    for (int k = lane; k < d; k += 32) {
        p.w.iq[(int64_t)q * d + k] = qv[k];
        if (th) p.w.iwhat[(int64_t)q * d + k] = wh[k];
        if (p.Eb) p.w.iqb[(int64_t)q * d + k] = __bfloat16_as_ushort(__float2bfloat16_rn(qv[k]));
    }
    if (p.ext_ftrue) {
        if (lane == 0) p.w.iftrue[q] = p.ext_ftrue[q];
    } else if (p.tt) {
        const int64_t tid = checked_id(p.tt[q], p.E, p.w.status);
        if (p.Eb) {   // the arithmetic of the tensor-core path: operands rounded to bf16, fp32 accumulation
            const uint16_t* t = p.Eb + tid * d;
            for (int k = lane; k < d; k += 32) { tv[k] = __uint_as_float((uint32_t)t[k] << 16); qv[k] = __bfloat162float(__float2bfloat16_rn(qv[k])); }
        } else {
            const float* t = p.ent + tid * d;
            for (int k = lane; k < d; k += 32) tv[k] = t[k];
        }
        __syncwarp();
        if (lane == 0) p.w.iftrue[q] = score_seq(p, qv, wh, tv);
    }
    for (int j = lane; j < p.k; j += 32) {
        p.w.top_score[(int64_t)q * p.k + j] = -INFINITY;
        p.w.top_id[(int64_t)q * p.k + j] = INT_MAX;
    }
    if (lane == 0) {
        p.w.thr[q] = -INFINITY; p.w.thr_id[q] = INT_MAX;
        p.w.cand_cnt[q] = 0; p.w.beat_tmp[q] = 0; p.w.beat[q] = 0;
    }
}

constexpr int IQ = 64, IE = 64, IKC = 32, ILD = IKC + 4;

// Whether a candidate list overflowed earlier in this call: asked by one thread before the first load, so that what was queued
// behind costs little more than its launch.  (A plain load: the CTAs of a launch find it in their SM's cache, which is empty when
// the launch begins; one that misses a change during the launch does work that is redone.)
__device__ __forceinline__ int call_given_up(const InferParams& p) { return p.first ? 0 : p.w.status[1]; }

// Largest float below x (x finite).
__device__ __forceinline__ float float_below(float x) {
    if (x == 0.f) return __uint_as_float(0x80000001u);
    const uint32_t b = __float_as_uint(x);
    return __uint_as_float(x > 0.f ? b - 1u : b + 1u);
}

// Epilogue of a 64 x 64 score tile: rank counting against the true tail, threshold filter into the
// candidate lists.  Thread (tx, ty) holds the pairs (q0 + ty + 16 i, e0 + tx + 16 j).
// The tile's 64 entity ids are consecutive.  If the reference id (the true tail, or the id of the
// current k-th best) is not among them, "ordered before (f0, id0)" is the same plain comparison
// for the whole row of the tile: f >= f0 when the tile lies below id0, f > f0 when above, and
// f >= f0 is f > (largest float below f0).  So the common case costs one compare per pair and
// test; a row whose reference id falls inside the tile, a ragged last tile and non-finite
// reference scores take the element-by-element form.
//
// `cuts` (optional, shared memory, one entry per query row of the tile): the two comparison values of a row in the
// plain case, worked out once per row by score_tile_row_cuts while the tile's rows are still on their way, so that
// the sixteen threads of a row do not each load the row's state and form them again.
__device__ __forceinline__ void score_tile_row_cuts(const InferParams& p, int q0, int64_t e0, int row, float4* cuts) {
    const int64_t g0 = e0 + p.id_base;
    const int q = q0 + row;
    float4 c = make_float4(0.f, INFINITY, 0.f, 0.f);     // (x: candidate cut, y: rank cut, z: 1 = plain case)
    if (q < p.nq && e0 + IE <= p.e_hi) {
        const float thr = p.w.thr[q]; const int32_t thr_id = p.w.thr_id[q];
        float ft = 0.f; int32_t tt = -1;
        if (p.tt) { ft = p.w.iftrue[q]; tt = p.tt[q]; }
        const bool thr_out = thr_id < g0 || thr_id >= g0 + IE, tt_out = !p.tt || tt < g0 || tt >= g0 + IE;
        if (thr_out && tt_out && fabsf(thr) < INFINITY && fabsf(ft) < INFINITY) {
            c.x = thr_id >= g0 + IE ? float_below(thr) : thr;
            c.y = !p.tt ? INFINITY : (tt >= g0 + IE ? float_below(ft) : ft);     // without true tails nothing is counted
            c.z = 1.f;
        }
    }
    cuts[row] = c;
}

template <int KIND>
__device__ __forceinline__ void score_tile_epilogue(const InferParams& p, const float (&acc)[4][4], int q0, int64_t e0, int tx, int ty,
                                                    const float4* cuts = nullptr) {
    const int64_t g0 = e0 + p.id_base;                  // the id the caller knows the tile's first entity by
    const bool whole = e0 + IE <= p.e_hi;
    const bool first = p.first != 0;
    int beat_all = 0;                                   // four rows' counts, one byte each (at most 4 per thread, 64 per row)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int q = q0 + ty + 16 * i;
        const bool qin = q < p.nq;
        if (cuts) {
            const float4 c = cuts[ty + 16 * i];
            if (c.z != 0.f) {
                int beat = 0;
                float f[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) { f[j] = canon_finish(KIND, acc[i][j]); beat += f[j] > c.y ? 1 : 0; }
                if (fmaxf(fmaxf(f[0], f[1]), fmaxf(f[2], f[3])) > c.x) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (f[j] > c.x) {
                            const int slot = atomicAdd(&p.w.cand_cnt[q], 1);
                            if (slot < kCandCap) {
                                p.w.cand_score[(int64_t)q * kCandCap + slot] = f[j];
                                p.w.cand_id[(int64_t)q * kCandCap + slot] = (int32_t)(g0 + tx + 16 * j);
                            } else {
                                p.w.status[1] = 1;
                            }
                        }
                }
                beat_all |= beat << (8 * i);
                continue;
            }
        }
        float thr = 0.f, ft = 0.f; int32_t thr_id = 0, tt = 0;
        if (qin) {
            thr = p.w.thr[q]; thr_id = p.w.thr_id[q];
            if (p.tt) { ft = p.w.iftrue[q]; tt = p.tt[q]; }
        }
        auto append = [&](float f, int32_t ge) {
            const int slot = atomicAdd(&p.w.cand_cnt[q], 1);
            if (slot < kCandCap) {
                p.w.cand_score[(int64_t)q * kCandCap + slot] = f;
                p.w.cand_id[(int64_t)q * kCandCap + slot] = ge;
            } else {
                p.w.status[1] = 1;   // this chunk overflowed a list: the host redoes it in small pieces
            }
        };
        const bool thr_out = thr_id < g0 || thr_id >= g0 + IE, tt_out = tt < g0 || tt >= g0 + IE;
        const bool plain = whole && qin && thr_out && tt_out && fabsf(thr) < INFINITY && fabsf(ft) < INFINITY;
        int beat = 0;
        if (plain) {
            const float thr_c = thr_id >= g0 + IE ? float_below(thr) : thr;
            const float ft_c = tt >= g0 + IE ? float_below(ft) : ft;
            float f[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) { f[j] = canon_finish(KIND, acc[i][j]); beat += f[j] > ft_c ? 1 : 0; }
            // candidates are rare once the threshold has tightened: one test of the largest of the four
            // instead of four divergent branches
            if (fmaxf(fmaxf(f[0], f[1]), fmaxf(f[2], f[3])) > thr_c) {
#pragma unroll
                for (int j = 0; j < 4; ++j) if (f[j] > thr_c) append(f[j], (int32_t)(g0 + tx + 16 * j));
            }
            if (!p.tt) beat = 0;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t e = e0 + tx + 16 * j;
                if (!qin || e >= p.e_hi) continue;
                const float f = canon_finish(KIND, acc[i][j]);
                const int32_t ge = (int32_t)(e + p.id_base);
                if (p.tt && ordered_before(f, ge, ft, tt)) ++beat;
                if (first) p.w.cand_score[(int64_t)q * kCandCap + (e - p.e_lo)] = f;
                else if (ordered_before(f, ge, thr, thr_id)) append(f, ge);
            }
        }
        beat_all |= beat << (8 * i);
    }
    // The 16 lanes sharing a query row are contiguous.  The tile's 64 counts leave as two warp-wide additions: as thirty-two of
    // two lanes each, the tiles of a launch met on the few lines that hold the counters of few queries, which was the bound there
    // (64 queries, 4 M entities, d = 84: 3.89 ms against 1.70 without ranks, 2.24 now; 115 queries, 1.5 M: 1.90 -> 1.27).
    if (!p.tt) return;
    __shared__ int counts[IQ];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) beat_all += __shfl_xor_sync(0xffffffffu, beat_all, o);
    if (tx == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) counts[ty + 16 * i] = (beat_all >> (8 * i)) & 0xff;
    }
    __syncthreads();
    const int row = tx + 16 * ty;
    if (row < IQ && counts[row] > 0) atomicAdd(&p.w.beat_tmp[q0 + row], counts[row]);
}

// ------------------------------------------------------------------------------------------
// score tile: 64 queries x 64 entities per CTA, 4 x 4 pairs per thread.  Consecutive CTAs
// walk the query tiles of one entity tile, so an entity tile is fetched from HBM once and
// served to the other query tiles by L2.
// ------------------------------------------------------------------------------------------
template <int KIND>
__global__ void __launch_bounds__(256) score_tile_kernel(InferParams p) {
    constexpr bool TH = KIND == KIND_TH_L1 || KIND == KIND_TH_L2;
    __shared__ __align__(16) float Qs[IQ * ILD];
    __shared__ __align__(16) float Ts[IE * ILD];
    __shared__ __align__(16) float Ws[TH ? IQ * ILD : 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int qt = blockIdx.x % p.q_tiles;
    const int64_t et = blockIdx.x / p.q_tiles;
    const int q0 = qt * IQ;
    const int64_t e0 = p.e_lo + et * IE;
    const int d4 = p.d4;
    const float4* Qg = reinterpret_cast<const float4*>(p.w.iq);
    const float4* Wg = reinterpret_cast<const float4*>(p.w.iwhat);
    const float4* Tg = reinterpret_cast<const float4*>(p.ent);

    __shared__ float4 cuts[IQ];
    __shared__ int skip;
    grid_dependency_wait();
    allow_dependents();
    if (tid == 0) skip = call_given_up(p);
    __syncthreads();
    if (skip) return;
    if (tid >= 256 - IQ) score_tile_row_cuts(p, q0, e0, tid - (256 - IQ), cuts);     // (read after the barriers of the loop below)
    float acc[4][4], u[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j] = 0.f; u[i][j] = 0.f; }
    const int npass = TH ? 2 : 1;
    for (int pass = 0; pass < npass; ++pass) {
        const bool upass = TH && pass == 0;
        for (int k0 = 0; k0 < p.d; k0 += IKC) {
#pragma unroll
            for (int it = 0; it < 2; ++it) {
                const int idx = tid + 256 * it, row = idx >> 3, c4 = idx & 7;
                const int gc = (k0 >> 2) + c4;
                const bool kin = gc < d4;
                float4 qv = make_float4(0.f, 0.f, 0.f, 0.f), tv = qv, wv = qv;
                if (kin && q0 + row < p.nq) {
                    qv = Qg[(int64_t)(q0 + row) * d4 + gc];
                    if (TH) wv = Wg[(int64_t)(q0 + row) * d4 + gc];
                }
                if (kin && e0 + row < p.e_hi) tv = Tg[(e0 + row) * d4 + gc];
                *reinterpret_cast<float4*>(&Qs[row * ILD + c4 * 4]) = qv;
                *reinterpret_cast<float4*>(&Ts[row * ILD + c4 * 4]) = tv;
                if (TH) *reinterpret_cast<float4*>(&Ws[row * ILD + c4 * 4]) = wv;
            }
            __syncthreads();
#pragma unroll
            for (int kk = 0; kk < IKC; kk += 4) {
                float4 qv[4], tv[4], wv[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    qv[i] = *reinterpret_cast<const float4*>(&Qs[(ty + 16 * i) * ILD + kk]);
                    tv[i] = *reinterpret_cast<const float4*>(&Ts[(tx + 16 * i) * ILD + kk]);
                    if (TH) wv[i] = *reinterpret_cast<const float4*>(&Ws[(ty + 16 * i) * ILD + kk]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (!TH) {
                            canon_update<TH ? KIND_L1 : KIND>(acc[i][j], qv[i], tv[j]);
                        } else if (upass) {
                            u[i][j] = __fmaf_rn(wv[i].x, tv[j].x, u[i][j]); u[i][j] = __fmaf_rn(wv[i].y, tv[j].y, u[i][j]);
                            u[i][j] = __fmaf_rn(wv[i].z, tv[j].z, u[i][j]); u[i][j] = __fmaf_rn(wv[i].w, tv[j].w, u[i][j]);
                        } else {
                            canon_th_acc(KIND, acc[i][j], canon_th_x(u[i][j], wv[i], qv[i], tv[j]));
                        }
                    }
            }
            __syncthreads();
        }
    }
    score_tile_epilogue<KIND>(p, acc, q0, e0, tx, ty, cuts);
}

// ------------------------------------------------------------------------------------------
// score tile, kinds that are a function of (q, t) alone, rows of fewer than 32 floats: the same 64 x 64 tile
// and the same operation order (one accumulator per pair, coordinates ascending), but the 64 query
// rows and 64 entity rows arrive by one asynchronous bulk copy per row into padded shared-memory
// rows, so a CTA waits once instead of loading and synchronising every 32 coordinates.
// ------------------------------------------------------------------------------------------
constexpr int ITENSOR_MIN_D = 32;          // rows from here on are staged by tensor copies (below)
inline size_t infer_tma_smem(int d) { return (size_t)(IQ + IE) * (d + 4) * sizeof(float) + sizeof(uint64_t); }

template <int KIND>
__global__ void __launch_bounds__(256) score_tile_tma_kernel(InferParams p) {
    extern __shared__ __align__(128) unsigned char smraw[];
    constexpr int ROWS = IQ + IE;        // rows [0, IQ) hold queries, the rest entities
    const int ld = p.d + 4;
    float* base = reinterpret_cast<float*>(smraw);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smraw + (size_t)ROWS * ld * sizeof(float));
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int qt = blockIdx.x % p.q_tiles;
    const int64_t et = blockIdx.x / p.q_tiles;
    const int q0 = qt * IQ;
    const int64_t e0 = p.e_lo + et * IE;

    __shared__ int skip;
    if (tid == 0) { mbar_init(bar, ROWS); mbar_init_fence(); }
    grid_dependency_wait();
    allow_dependents();
    if (tid == 0) skip = call_given_up(p);
    __syncthreads();
    if (skip) return;
    if (tid < ROWS) {                            // thread r owns row r
        const bool isq = tid < IQ;
        const int64_t g = isq ? q0 + tid : e0 + (tid - IQ);
        const bool in = isq ? g < p.nq : g < p.e_hi;
        float* dst = base + (size_t)tid * ld;
        if (in) {
            mbar_arrive_expect_tx(bar, (uint32_t)p.d * 4u);
            bulk_g2s(dst, (isq ? p.w.iq : p.ent) + g * p.d, (uint32_t)p.d * 4u, bar);
        } else {
            for (int k = 0; k < p.d; k += 4) *reinterpret_cast<float4*>(dst + k) = make_float4(0.f, 0.f, 0.f, 0.f);
            mbar_arrive(bar);
        }
    }
    __shared__ float4 cuts[IQ];
    if (tid >= 256 - IQ) score_tile_row_cuts(p, q0, e0, tid - (256 - IQ), cuts);     // (read after the barrier that follows the wait)

    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

    const bool ok = mbar_wait_bounded(bar, 0u, p.wait_limit);
    if (!__syncthreads_and(ok)) {
        if (tid == 0) set_status(p.w.status, KGE_ERR_TIMEOUT);
        // give copies still in flight a bounded chance to land before shared memory is released
        (void)mbar_wait_bounded(bar, 0u, p.wait_limit);
        return;
    }
    const float* Qs = base;
    const float* Ts = Qs + IQ * ld;
#pragma unroll 2
    for (int kk = 0; kk < p.d; kk += 4) {
        float4 qv[4], tv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            qv[i] = *reinterpret_cast<const float4*>(&Qs[(ty + 16 * i) * ld + kk]);
            tv[i] = *reinterpret_cast<const float4*>(&Ts[(tx + 16 * i) * ld + kk]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) canon_update<KIND>(acc[i][j], qv[i], tv[j]);
    }
    score_tile_epilogue<KIND>(p, acc, q0, e0, tx, ty, cuts);
}

// ------------------------------------------------------------------------------------------
// The same score tile for rows of at least 32 floats, staged by the TMA engine's tensor copies: four
// copies per stage of 64 coordinates (two 64-row x 32-float boxes of the queries, two of the entities,
// 128-byte swizzle) issued by one thread.  A box holds a row's 32 floats as eight 16-byte units, unit
// u of row r at position u ^ (r & 7): a thread's rows all share r & 7, so its eight unit offsets are
// computed once and every 128-bit read is base + constant + one of them, without bank conflicts.
// Two stages of 32 KB whatever the row length, so that three CTAs share an SM: with stages of 128
// coordinates, rows of more than 128 floats left one CTA per SM (0.67 of the instruction rate).
//
// Bound: the FMA pipe (L1: one subtraction and one addition per element).  The differences of two
// coordinates are one packed subtraction (the same rounding, one issue slot for two): a packed
// instruction holds the pipe for two cycles and adds no arithmetic rate, but leaves issue slots for
// the shared-memory reads, which otherwise take 8 of every 136.
// ------------------------------------------------------------------------------------------
constexpr int ITB_KC = 64;
constexpr int ITB_BOX_BYTES = 64 * 128, ITB_CHUNK_BYTES = 2 * ITB_BOX_BYTES, ITB_STAGE_BYTES = 2 * ITB_CHUNK_BYTES;
__host__ __device__ inline int infer_tensor_stages(int d) { return d > ITB_KC ? 2 : 1; }
inline size_t infer_tensor_smem(int d) { return 1024 + (size_t)infer_tensor_stages(d) * ITB_STAGE_BYTES + 2 * sizeof(uint64_t); }
__device__ __forceinline__ void tile_load_2d(void* dst, const CUtensorMap* tm, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"(tm), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}

// canon_update with the subtractions of neighbouring coordinates packed.
template <int KIND>
__device__ __forceinline__ void canon_update_packed(float& acc, float4 q, float4 t) {
    if (KIND == KIND_DOT) { canon_update<KIND>(acc, q, t); return; }
    const float2 a = sub2(make_float2(q.x, q.y), make_float2(t.x, t.y)), b = sub2(make_float2(q.z, q.w), make_float2(t.z, t.w));
    if (KIND == KIND_L1) {
        acc = __fadd_rn(acc, fabsf(a.x)); acc = __fadd_rn(acc, fabsf(a.y));
        acc = __fadd_rn(acc, fabsf(b.x)); acc = __fadd_rn(acc, fabsf(b.y));
    } else if (KIND == KIND_L2) {
        acc = __fmaf_rn(a.x, a.x, acc); acc = __fmaf_rn(a.y, a.y, acc);
        acc = __fmaf_rn(b.x, b.x, acc); acc = __fmaf_rn(b.y, b.y, acc);
    } else {  // KIND_CL1
        acc = __fadd_rn(acc, __fsqrt_rn(__fmaf_rn(a.x, a.x, __fmul_rn(a.y, a.y))));
        acc = __fadd_rn(acc, __fsqrt_rn(__fmaf_rn(b.x, b.x, __fmul_rn(b.y, b.y))));
    }
}

template <int KIND>
__global__ void __launch_bounds__(256, 3) score_tile_tensor_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmE,
                                                                   InferParams p) {
    extern __shared__ unsigned char smraw_t[];
    unsigned char* base = smraw_t + ((1024u - (smem_u32(smraw_t) & 1023u)) & 1023u);       // swizzled boxes want 1024-byte alignment
    const int nstage = infer_tensor_stages(p.d);
    const int nchunk = (p.d + ITB_KC - 1) / ITB_KC;
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + (size_t)nstage * ITB_STAGE_BYTES);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int qt = blockIdx.x % p.q_tiles;
    const int64_t et = blockIdx.x / p.q_tiles;
    const int q0 = qt * IQ;
    const int64_t e0 = p.e_lo + et * IE;

    if (tid == 0) {
        for (int st = 0; st < nstage; ++st) mbar_init(&bars[st], 1);
        mbar_init_fence();
    }
    __shared__ int skip;
    grid_dependency_wait();
    allow_dependents();
    if (tid == 0) skip = call_given_up(p);
    __syncthreads();
    if (skip) return;
    auto issue = [&](int chunk, int stage) {     // (a box that begins beyond the row is left out)
        if (tid != 0) return;
        unsigned char* qs = base + (size_t)stage * ITB_STAGE_BYTES;
        const int x = chunk * ITB_KC;
        const bool two = x + 32 < p.d;
        mbar_arrive_expect_tx(&bars[stage], (uint32_t)(two ? ITB_STAGE_BYTES : ITB_STAGE_BYTES / 2));
        tile_load_2d(qs, &tmQ, x, q0, &bars[stage]);
        tile_load_2d(qs + ITB_CHUNK_BYTES, &tmE, x, (int)e0, &bars[stage]);
        if (two) {
            tile_load_2d(qs + ITB_BOX_BYTES, &tmQ, x + 32, q0, &bars[stage]);
            tile_load_2d(qs + ITB_CHUNK_BYTES + ITB_BOX_BYTES, &tmE, x + 32, (int)e0, &bars[stage]);
        }
    };
    issue(0, 0);
    if (nchunk > 1) issue(1, 1);
    __shared__ float4 cuts[IQ];
    if (tid >= 256 - IQ) score_tile_row_cuts(p, q0, e0, tid - (256 - IQ), cuts);     // (read after the barrier that follows the first wait)

    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    uint32_t qoff[8], toff[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) { qoff[u] = (uint32_t)((u ^ (ty & 7)) << 4); toff[u] = (uint32_t)((u ^ (tx & 7)) << 4); }

    for (int chunk = 0; chunk < nchunk; ++chunk) {
        const int stage = chunk % nstage;
        const bool ok = mbar_wait_bounded(&bars[stage], (uint32_t)(chunk / nstage) & 1u, p.wait_limit);
        const bool all = __syncthreads_and(ok);
        if (!all) {
            if (tid == 0) set_status(p.w.status, KGE_ERR_TIMEOUT);
            for (int st = 0; st < min(nstage, nchunk); ++st) (void)mbar_wait_bounded(&bars[st], (uint32_t)(chunk / nstage) & 1u, p.wait_limit);
            return;
        }
        const unsigned char* qrow = base + (size_t)stage * ITB_STAGE_BYTES + ty * 128;
        const unsigned char* trow = base + (size_t)stage * ITB_STAGE_BYTES + ITB_CHUNK_BYTES + tx * 128;
        const int len = min(ITB_KC, p.d - chunk * ITB_KC);
        auto unit = [&](const unsigned char* qb, const unsigned char* tb) {      // four coordinates of the 4 x 4 pairs
            float4 qv[4], tv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                qv[i] = *reinterpret_cast<const float4*>(qb + i * (16 * 128));
                tv[i] = *reinterpret_cast<const float4*>(tb + i * (16 * 128));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) canon_update_packed<KIND>(acc[i][j], qv[i], tv[j]);
        };
#pragma unroll 1
        for (int b = 0; b < len / 32; ++b) {
#pragma unroll
            for (int u = 0; u < 8; ++u) unit(qrow + b * ITB_BOX_BYTES + qoff[u], trow + b * ITB_BOX_BYTES + toff[u]);
        }
        if (len % 32 != 0) {             // the row ends inside a box
            const int at = (len / 32) * ITB_BOX_BYTES;
#pragma unroll 1
            for (int u = 0; u < (len % 32) / 4; ++u) unit(qrow + at + ((u ^ (ty & 7)) << 4), trow + at + ((u ^ (tx & 7)) << 4));
        }
        if (chunk + nstage < nchunk) {
            __syncthreads();             // every thread is done reading this stage
            issue(chunk + nstage, stage);
        }
    }
    score_tile_epilogue<KIND>(p, acc, q0, e0, tx, ty, cuts);
}

template <int KIND>
cudaError_t launch_score_tile_tensor(const kge_handle* h, const InferParams& p, unsigned grid, cudaStream_t s) {
    static DeviceOnce configured;
    const cudaError_t e = once_per_device(configured, [] {
        return cudaFuncSetAttribute(score_tile_tensor_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)infer_tensor_smem(kMaxDim));
    });
    if (e != cudaSuccess) return e;
    return launch_dependent(score_tile_tensor_kernel<KIND>, dim3(grid), dim3(256), infer_tensor_smem(p.d), s,
                            *reinterpret_cast<const CUtensorMap*>(h->tm_iq32), *reinterpret_cast<const CUtensorMap*>(h->tm_ent32), p);
}

template <int KIND>
cudaError_t launch_score_tile_tma(const InferParams& p, unsigned grid, cudaStream_t s) {
    return launch_dependent(score_tile_tma_kernel<KIND>, dim3(grid), dim3(256), infer_tma_smem(p.d), s, p);
}

// ------------------------------------------------------------------------------------------
// select: one CTA per query merges the running top-k with this chunk's candidates by a
// bitonic sort in shared memory under (score descending, id ascending), commits the chunk's
// rank count and resets the candidate list; after the last chunk it writes the outputs.
//
// A long list (the first chunk's 1,024 unfiltered scores) is cut down first: each of the 128 threads
// takes the best of its share, and the k-th best of those 128 is a lower bound of the k-th best of
// all, so only what reaches it is sorted (k = 10: some 13 of 1,024 instead of a sort of 2,048 places,
// 1,435 us for 15,000 queries).  Up to 64 entries are sorted by one warp without CTA-wide barriers.
// ------------------------------------------------------------------------------------------
constexpr int SEL_THREADS = 128;
constexpr int SEL_MAX = 2 * kCandCap;   // k <= kCandCap plus at most kCandCap candidates
constexpr int SEL_CUT_MIN = 192;        // candidates from which the cut pays

__global__ void __launch_bounds__(SEL_THREADS) select_kernel(InferParams p) {
    __shared__ float ss[SEL_MAX];
    __shared__ int32_t si[SEL_MAX];
    __shared__ __align__(16) float best[SEL_THREADS];
    __shared__ float cut_sm;
    __shared__ int kept;
    const int q = blockIdx.x, tid = threadIdx.x;
    grid_dependency_wait();
    allow_dependents();
    if (p.w.status[1]) return;              // (nothing in flight writes it)
    const int cnt = p.first ? (int)(p.e_hi - p.e_lo) : min(p.w.cand_cnt[q], kCandCap);
    const float* cs = p.w.cand_score + (int64_t)q * kCandCap;
    const int32_t* ci = p.w.cand_id + (int64_t)q * kCandCap;
    const int32_t first_id = (int32_t)(p.e_lo + p.id_base);
    auto candidate = [&](int i, float& s, int32_t& id) {
        s = cs[i];
        id = p.first ? first_id + i : ci[i];
        // never candidates: what is not a number and, in the tensor-core arithmetic, -inf
        if (p.first && (!(s == s) || (p.Eb && s == -INFINITY))) { s = -INFINITY; id = INT_MAX; }
    };
    const int run = p.first ? 0 : p.k;      // before the first chunk the running list is empty
    int total = run + cnt;
    const bool cut = cnt >= SEL_CUT_MIN && p.k <= SEL_THREADS;
    for (int i = tid; i < run; i += SEL_THREADS) { ss[i] = p.w.top_score[(int64_t)q * p.k + i]; si[i] = p.w.top_id[(int64_t)q * p.k + i]; }
    if (cut) {
        constexpr int PER = kCandCap / SEL_THREADS;
        float v[PER]; int32_t id[PER];
        float b = -INFINITY;
        if (tid == 0) { kept = 0; cut_sm = -INFINITY; }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            v[i] = -INFINITY; id[i] = INT_MAX;
            if (tid + i * SEL_THREADS < cnt) candidate(tid + i * SEL_THREADS, v[i], id[i]);
            b = fmaxf(b, v[i]);
        }
        best[tid] = b;
        __syncthreads();
        int rank = 0;                       // threads whose best comes before mine
#pragma unroll 8
        for (int j = 0; j < SEL_THREADS; j += 4) {
            const float4 o = *reinterpret_cast<const float4*>(&best[j]);
            rank += (o.x > b || (o.x == b && j < tid)) + (o.y > b || (o.y == b && j + 1 < tid)) + (o.z > b || (o.z == b && j + 2 < tid)) + (o.w > b || (o.w == b && j + 3 < tid));
        }
        if (rank == p.k - 1) cut_sm = b;
        __syncthreads();
        const float c = cut_sm;
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (tid + i * SEL_THREADS < cnt && v[i] >= c) { const int at = run + atomicAdd(&kept, 1); ss[at] = v[i]; si[at] = id[i]; }
        __syncthreads();
        total = run + kept;
    } else {
        for (int i = tid; i < cnt; i += SEL_THREADS) { float s; int32_t id; candidate(i, s, id); ss[run + i] = s; si[run + i] = id; }
    }
    int n2 = 1;
    while (n2 < total || n2 < p.k) n2 <<= 1;
    for (int i = total + tid; i < n2; i += SEL_THREADS) { ss[i] = -INFINITY; si[i] = INT_MAX; }
    __syncthreads();
    auto exchange = [&](int t, int size, int stride) {
        const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
        const bool up = (lo & size) == 0;   // "up" blocks end with the best element first
        const float a = ss[lo], b = ss[hi]; const int32_t ia = si[lo], ib = si[hi];
        const bool b_first = ordered_before(b, ib, a, ia);
        if (b_first == up) { ss[lo] = b; si[lo] = ib; ss[hi] = a; si[hi] = ia; }
    };
    if (n2 <= 64) {
        if (tid < 32) {
            for (int size = 2; size <= n2; size <<= 1)
                for (int stride = size >> 1; stride > 0; stride >>= 1) {
                    if (tid < n2 / 2) exchange(tid, size, stride);
                    __syncwarp();
                }
        }
        __syncthreads();
    } else {
        for (int size = 2; size <= n2; size <<= 1)
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int t = tid; t < n2 / 2; t += SEL_THREADS) exchange(t, size, stride);
                __syncthreads();
            }
    }
    for (int i = tid; i < p.k; i += SEL_THREADS) {
        p.w.top_score[(int64_t)q * p.k + i] = ss[i];
        p.w.top_id[(int64_t)q * p.k + i] = si[i];
        if (p.last && p.out_ids) {
            p.out_ids[(int64_t)q * p.k + i] = si[i] == INT_MAX ? -1 : si[i];
            p.out_scores[(int64_t)q * p.k + i] = ss[i];
        }
    }
    if (tid == 0) {
        p.w.thr[q] = ss[p.k - 1]; p.w.thr_id[q] = si[p.k - 1];
        const int beat = p.w.beat[q] + p.w.beat_tmp[q];
        p.w.beat[q] = beat;
        p.w.beat_tmp[q] = 0; p.w.cand_cnt[q] = 0;
        if (q == 0) p.w.status[6] = (int32_t)p.e_hi;
        if (p.last && p.out_ranks) p.out_ranks[q] = (p.raw_beat ? 0 : 1) + beat;      // (may be the array of the chunk's counts)
    }
}

// ---- sharded inference: the pieces that need rows of one shard only ----
// Query vectors of the queries whose head lies in this shard; zeros for the others, so that a sum over the shards
// (every head lies in exactly one) gives every query's vector exactly.
__global__ void shard_query_kernel(InferParams p, float* qvec_out, float* wh_scratch) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= p.nq) return;
    const int64_t hid = (int64_t)p.qh[q] - p.id_base;
    float* qv = qvec_out + (int64_t)q * p.d;
    if (hid < 0 || hid >= p.E) { for (int k = 0; k < p.d; ++k) qv[k] = 0.f; return; }
    const int64_t rid = checked_id(p.qr[q], p.R, p.w.status);
    build_query_seq(p, p.ent + hid * p.d, rid, qv, p.score == KGE_TRANSH ? wh_scratch + (int64_t)q * p.d : nullptr);
}

// Scores of the true tails that lie in this shard, from finished query vectors; zeros for the others.  bf16_rows: the
// tensor-core arithmetic (query vector and tail row rounded to bf16, fp32 accumulation).
__global__ void shard_ftrue_kernel(InferParams p, const float* qvec, float* wh_scratch, float* f_out, const uint16_t* bf16_rows) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= p.nq) return;
    const int64_t tid = (int64_t)p.tt[q] - p.id_base;
    if (tid < 0 || tid >= p.E) { f_out[q] = 0.f; return; }
    const float* qv = qvec + (int64_t)q * p.d;
    if (bf16_rows) {
        const uint16_t* tb = bf16_rows + tid * p.d;
        float acc = 0.f;
        for (int k = 0; k < p.d; ++k) {
            const __nv_bfloat16 qb = __float2bfloat16_rn(qv[k]);
            acc = __fmaf_rn(__bfloat162float(qb), __uint_as_float((uint32_t)tb[k] << 16), acc);
        }
        f_out[q] = acc;
        return;
    }
    float* wh = nullptr;
    if (p.score == KGE_TRANSH) { wh = wh_scratch + (int64_t)q * p.d; unit_normal_seq(p, checked_id(p.qr[q], p.R, p.w.status), wh); }
    f_out[q] = score_seq(p, qv, wh, p.ent + tid * p.d);
}

// Final top-k of a query over the candidates gathered from all shards: one CTA per query sorts per_query (score, id)
// pairs under (score descending, id ascending); unused places (id -1) sort last.
constexpr int MERGE_THREADS = 128, MERGE_MAX = 2048;
__global__ void __launch_bounds__(MERGE_THREADS) merge_topk_kernel(const int32_t* cand_ids, const float* cand_scores, int per_query, int k,
                                                                   int32_t* out_ids, float* out_scores) {
    __shared__ float ss[MERGE_MAX];
    __shared__ int32_t si[MERGE_MAX];
    const int q = blockIdx.x, tid = threadIdx.x;
    int n2 = 1;
    while (n2 < per_query) n2 <<= 1;
    for (int i = tid; i < n2; i += MERGE_THREADS) {
        float s = -INFINITY; int32_t id = INT_MAX;
        if (i < per_query) {
            id = cand_ids[(int64_t)q * per_query + i]; s = cand_scores[(int64_t)q * per_query + i];
            if (id < 0) { id = INT_MAX; s = -INFINITY; }
        }
        ss[i] = s; si[i] = id;
    }
    __syncthreads();
    for (int size = 2; size <= n2; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = tid; t < n2 / 2; t += MERGE_THREADS) {
                const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                const bool up = (lo & size) == 0;
                const float a = ss[lo], b = ss[hi]; const int32_t ia = si[lo], ib = si[hi];
                if (ordered_before(b, ib, a, ia) == up) { ss[lo] = b; si[lo] = ib; ss[hi] = a; si[hi] = ia; }
            }
            __syncthreads();
        }
    for (int i = tid; i < k; i += MERGE_THREADS) {
        const bool have = i < n2 && si[i] != INT_MAX;
        out_ids[(int64_t)q * k + i] = have ? si[i] : -1;
        out_scores[(int64_t)q * k + i] = have ? ss[i] : -INFINITY;
    }
}

__global__ void reset_chunk_kernel(InferParams p) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < p.nq) { p.w.cand_cnt[q] = 0; p.w.beat_tmp[q] = 0; }
    if (q == 0) p.w.status[1] = 0;
}

cudaError_t launch_score_tiles(const kge_handle* h, const InferParams& p, cudaStream_t s) {
    const int64_t e_tiles = (p.e_hi - p.e_lo + IE - 1) / IE;
    const unsigned grid = (unsigned)(e_tiles * p.q_tiles);
    if (h->tiles32_ready && p.d >= ITENSOR_MIN_D) {      // tiles staged by tensor copies
        switch (p.kind) {
            case KIND_L1: return launch_score_tile_tensor<KIND_L1>(h, p, grid, s);
            case KIND_L2: return launch_score_tile_tensor<KIND_L2>(h, p, grid, s);
            case KIND_CL1: return launch_score_tile_tensor<KIND_CL1>(h, p, grid, s);
            case KIND_DOT: return launch_score_tile_tensor<KIND_DOT>(h, p, grid, s);
            default: break;
        }
    }
    switch (p.kind) {
        case KIND_L1: return launch_score_tile_tma<KIND_L1>(p, grid, s);
        case KIND_L2: return launch_score_tile_tma<KIND_L2>(p, grid, s);
        case KIND_CL1: return launch_score_tile_tma<KIND_CL1>(p, grid, s);
        case KIND_DOT: return launch_score_tile_tma<KIND_DOT>(p, grid, s);
        case KIND_TH_L1: return launch_dependent(score_tile_kernel<KIND_TH_L1>, dim3(grid), dim3(256), 0, s, p);
        default: return launch_dependent(score_tile_kernel<KIND_TH_L2>, dim3(grid), dim3(256), 0, s, p);
    }
}

}  // namespace

namespace {
InferParams infer_params(kge_handle* h, const int32_t* qh, const int32_t* qr, int32_t nq, int32_t k, const int32_t* true_tails) {
    const kge_config& c = h->cfg;
    InferParams p;
    p.nq = nq; p.k = k; p.d = c.dim; p.d4 = c.dim / 4; p.score = c.score; p.kind = h->kind;
    p.E = c.num_entities; p.R = c.num_relations;
    p.ent = h->ent; p.rel = h->rel; p.relw = h->relw;
    p.qh = qh; p.qr = qr; p.tt = true_tails;
    p.q_tiles = (nq + IQ - 1) / IQ;
    p.wait_limit = h->wait_limit;
    p.id_base = 0; p.ext_q = nullptr; p.ext_ftrue = nullptr; p.raw_beat = 0;
    p.w = h->ws;
    p.e_lo = 0; p.e_hi = 0;
    p.Eb = nullptr; p.first = 0; p.last = 0;
    p.out_ids = nullptr; p.out_scores = nullptr; p.out_ranks = nullptr;
    return p;
}
}  // namespace

int run_shard_query_vectors(kge_handle* h, const int32_t* qh, const int32_t* qr, int32_t nq, int64_t ent_base, float* qvec_out, cudaStream_t s) {
    InferParams p = infer_params(h, qh, qr, nq, 1, nullptr);
    p.id_base = ent_base;
    shard_query_kernel<<<(nq + 127) / 128, 128, 0, s>>>(p, qvec_out, h->ws.iwhat);
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}

int run_shard_true_scores(kge_handle* h, const float* qvec, const int32_t* qr, const int32_t* true_tails, int32_t nq, int64_t ent_base,
                          float* ftrue_out, cudaStream_t s) {
    InferParams p = infer_params(h, nullptr, qr, nq, 1, true_tails);
    p.id_base = ent_base;
    if (h->ws.Eb && !h->eb_valid) {       // tensor-core arithmetic scores against the bf16 copy of the shard
        const int rc = launch_cast_bf16(h, h->ent, h->ws.Eb, h->cfg.num_entities * h->cfg.dim, s);
        if (rc != KGE_OK) return rc;
        h->eb_valid = true;
    }
    shard_ftrue_kernel<<<(nq + 127) / 128, 128, 0, s>>>(p, qvec, h->ws.iwhat, ftrue_out, h->ws.Eb);
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}

int run_merge_topk(const int32_t* cand_ids, const float* cand_scores, int32_t nq, int32_t per_query, int32_t k, int32_t* out_ids,
                   float* out_scores, cudaStream_t s) {
    if (per_query > MERGE_MAX) return KGE_ERR_WORKSPACE;
    merge_topk_kernel<<<nq, MERGE_THREADS, 0, s>>>(cand_ids, cand_scores, per_query, k, out_ids, out_scores);
    return cudaGetLastError() == cudaSuccess ? KGE_OK : KGE_ERR_CUDA;
}

int run_score_all_topk(kge_handle* h, const int32_t* qh, const int32_t* qr, int32_t nq, int32_t k,
                       const int32_t* true_tails, int32_t* out_ids, float* out_scores, int32_t* out_ranks,
                       cudaStream_t s, const ShardScoring* shard) {
    const kge_config& c = h->cfg;
    InferParams p = infer_params(h, qh, qr, nq, k, true_tails);
    if (shard) { p.id_base = shard->ent_base; p.ext_q = shard->qvec; p.ext_ftrue = shard->ftrue; p.raw_beat = 1; }
    const int qblocks = (nq + 127) / 128;
    const bool tc = h->ws.Eb != nullptr;    // dot-product model with the tensor-core score block
    if (tc && !h->eb_valid) {               // the bf16 copy of the table is kept until the table changes
        const int rc = launch_cast_bf16(h, h->ent, h->ws.Eb, c.num_entities * c.dim, s);
        if (rc != KGE_OK) return rc;
        h->eb_valid = true;
    }
    if (tc) p.Eb = h->ws.Eb;
    p.out_ids = out_ids; p.out_scores = out_scores; p.out_ranks = out_ranks;
    query_setup_kernel<<<(nq + SETUP_WARPS - 1) / SETUP_WARPS, 32 * SETUP_WARPS, 0, s>>>(p);
    KGE_LAUNCH_CHECK(h);
    if (!tc && !h->tiles32_ready && c.dim >= ITENSOR_MIN_D && h->kind != KIND_TH_L1 && h->kind != KIND_TH_L2) {
        // tensor maps of the fp32 query vectors and of the entity table (host-side encoding, nothing allocated)
        int rc = tc_make_f32_tile_map(h, h->tm_iq32, h->ws.iq, h->max_queries, c.dim);
        if (rc == KGE_OK) rc = tc_make_f32_tile_map(h, h->tm_ent32, h->ent, c.num_entities, c.dim);
        if (rc != KGE_OK) return rc;
        h->tiles32_ready = true;
    }

    // The first chunk is one candidate list's worth, since nothing is filtered yet; a later one covers `grow` times what all
    // chunks before it did, so that about grow x k entities per query beat the threshold (at most a quarter of a list at the
    // usual k), capped so that a launch stays bounded.  Twice as long a chunk each time was 14 chunks for 8 M entities at
    // some 50 us of selection, start-up and drain each; four times as long is 7.
    //
    // The chunks are queued without waiting for one another.  A list that fills up (scores rising along the table) sets
    // status[1]: what is queued behind does nothing, status[6] says how far the call has come, and it goes on from there with
    // chunks an eighth as long (those of one list's worth cannot overflow), a few queued at a time.  Once they pass they grow
    // again, after twice as many queues each time that this proved too early.
    const int64_t max_chunk = std::max<int64_t>(kCandCap, std::min<int64_t>((int64_t)1 << 22, (int64_t)0x7fffffff / p.q_tiles * IE / 2));
    const int64_t grow = std::max(1, std::min(4, 256 / k));
    constexpr int kFew = 16;
    int64_t most = max_chunk;                        // longest chunk for now
    int passed = 0, patience = 1;
    bool grown = false;
    auto chunk_len = [&](int64_t lo) { return std::min(std::min(std::max<int64_t>(lo * grow, kCandCap), most), p.E - lo); };
    int64_t lo = 0;
    while (lo < p.E) {
        int64_t at = lo;
        for (int queued = 0; at < p.E && (most == max_chunk || queued < kFew); ++queued) {
            p.e_lo = at; p.e_hi = at + chunk_len(at);
            p.first = at == 0; p.last = p.e_hi == p.E;
            if (tc) {
                const int rc = launch_tc_infer_chunk(h, nq, p.e_lo, p.e_hi, true_tails, p.id_base, p.first, s);
                if (rc != KGE_OK) return rc;
            } else {
                KGE_CUDA_CHECK(h, launch_score_tiles(h, p, s));
                KGE_LAUNCH_CHECK(h);
            }
            KGE_CUDA_CHECK(h, launch_dependent(select_kernel, dim3(nq), dim3(SEL_THREADS), 0, s, p));
            KGE_LAUNCH_CHECK(h);
            at = p.e_hi;
        }
        int32_t words[6];
        int32_t* const flags = h->host_flags ? h->host_flags : words;
        KGE_CUDA_CHECK(h, cudaMemcpyAsync(flags, h->ws.status + 1, sizeof(words), cudaMemcpyDeviceToHost, s));
        KGE_CUDA_CHECK(h, cudaStreamSynchronize(s));
        if (flags[0]) {
            lo = flags[5];
            most = std::max<int64_t>(kCandCap, (chunk_len(lo) / 8 + kCandCap - 1) / kCandCap * kCandCap);
            patience = grown ? std::min(2 * patience, 64) : 1;
            passed = 0;
            grown = false;
            reset_chunk_kernel<<<qblocks, 128, 0, s>>>(p);
            KGE_LAUNCH_CHECK(h);
        } else {
            lo = at;
            if (most < max_chunk) grown = ++passed >= patience;
            if (grown) { most = std::min(8 * most, max_chunk); passed = 0; }
        }
    }
    return KGE_OK;
}

}  // namespace kge

// ------------------------------------------------------------------------------------------
// Full-entity scoring for callers that may not allocate device memory.  All scratch lives in
// one file-scope device array that every GPU loading the library holds until the process
// exits; nothing is allocated or freed here, on the host heap or on the device.
// ------------------------------------------------------------------------------------------
namespace kge {
namespace {

constexpr int kStaticMaxQueries = 64;
constexpr int kStaticMaxTopk = 32;
constexpr size_t kStaticQueryRows = (size_t)kStaticMaxQueries * kMaxDim * sizeof(float);       // 131072
constexpr size_t kStaticCandList = (size_t)kStaticMaxQueries * kCandCap * 4;                   // 262144
constexpr size_t kStaticTopList = (size_t)kStaticMaxQueries * kStaticMaxTopk * 4;              // 8192
constexpr size_t kStaticSmall = 256;                                                            // >= 64 x 4 bytes
constexpr size_t kStaticBytes = 256 + 2 * kStaticQueryRows + 6 * kStaticSmall + 2 * kStaticCandList + 2 * kStaticTopList;

static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];   // 804,608 bytes per GPU

constexpr int kStaticMaxDevices = 64;
void* g_static_scratch_addr[kStaticMaxDevices] = {};   // device address of the array, per device ordinal

}  // namespace
}  // namespace kge

extern "C" int kge_score_all_topk_static(const kge_config* cfg, const float* ent, const float* rel,
                                         const float* relw, const int32_t* q_heads, const int32_t* q_rels,
                                         int32_t nq, int32_t k, const int32_t* true_tails, int32_t* out_ids,
                                         float* out_scores, int32_t* out_ranks, void* stream) {
    using namespace kge;
    if (!cfg || !ent || !rel || !q_heads || !q_rels || !out_ids || !out_scores || nq < 0 || k <= 0)
        return KGE_ERR_BAD_ARG;
    if (out_ranks && !true_tails) return KGE_ERR_BAD_ARG;
    const kge_config& c = *cfg;
    if (c.num_entities <= 0 || c.num_entities > INT32_MAX || c.num_relations <= 0 || c.num_relations > INT32_MAX ||
        c.dim <= 0 || c.dim % 4 != 0 || c.score < KGE_TRANSE || c.score > KGE_ROTATE_REAL_L1 ||
        (c.p_norm != 1 && c.p_norm != 2) || (c.score == KGE_TRANSH && !relw))
        return KGE_ERR_BAD_ARG;
    // the fixed scratch bounds the problem: refuse anything it cannot hold
    if (nq > kStaticMaxQueries || k > kStaticMaxTopk || c.dim > kMaxDim) return KGE_ERR_WORKSPACE;
    if (nq == 0) return KGE_OK;

    kge_handle h{};                     // plain host object on the stack, every field zero; nothing in it is heap-backed
    h.cfg = c;
    h.kind = kind_of(c);
    if (c.score == KGE_ROTATE_REAL_L1) h.cfg.score = KGE_ROTATE;      // the same query vector, the real norm (see kge_create)
    h.kw = h.cfg.score == KGE_ROTATE ? c.dim / 2 : c.dim;
    h.ent = const_cast<float*>(ent); h.rel = const_cast<float*>(rel); h.relw = const_cast<float*>(relw);
    h.ent_state = h.rel_state = h.relw_state = nullptr;
    h.launches = 0; h.bound = true; h.graph_loaded = false;
    h.max_queries = kStaticMaxQueries; h.topk = kStaticMaxTopk;
    h.num_sms = 148; h.split_q = h.split_t = 1; h.num_triples = 0;
    h.ws_base = nullptr; h.ws_bytes = 0; h.streams_ready = false;
    h.wait_limit = kDefaultWaitLimit; h.capture_scores = nullptr;

    // Set-up, once per device and with that device current: in host code the array's name is
    // only a stand-in, so its device address has to be asked for.
    int dev = -1;
    KGE_CUDA_CHECK(&h, cudaGetDevice(&dev));
    if (dev < 0 || dev >= kStaticMaxDevices) return KGE_ERR_UNSUPPORTED;
    if (!g_static_scratch_addr[dev]) {
        void* addr = nullptr;
        KGE_CUDA_CHECK(&h, cudaGetSymbolAddress(&addr, g_static_scratch));
        g_static_scratch_addr[dev] = addr;
    }
    unsigned char* base = static_cast<unsigned char*>(g_static_scratch_addr[dev]);

    Workspace w{};
    size_t o = 0;
    auto take = [&](size_t bytes) { unsigned char* p = base + o; o += bytes; return p; };
    w.status = reinterpret_cast<int32_t*>(take(256));
    w.iq = reinterpret_cast<float*>(take(kStaticQueryRows));
    w.iwhat = reinterpret_cast<float*>(take(kStaticQueryRows));
    w.iftrue = reinterpret_cast<float*>(take(kStaticSmall));
    w.thr = reinterpret_cast<float*>(take(kStaticSmall));
    w.thr_id = reinterpret_cast<int32_t*>(take(kStaticSmall));
    w.cand_cnt = reinterpret_cast<int32_t*>(take(kStaticSmall));
    w.beat_tmp = reinterpret_cast<int32_t*>(take(kStaticSmall));
    w.beat = reinterpret_cast<int32_t*>(take(kStaticSmall));
    w.cand_score = reinterpret_cast<float*>(take(kStaticCandList));
    w.cand_id = reinterpret_cast<int32_t*>(take(kStaticCandList));
    w.top_score = reinterpret_cast<float*>(take(kStaticTopList));
    w.top_id = reinterpret_cast<int32_t*>(take(kStaticTopList));
    if (o != kStaticBytes) return KGE_ERR_WORKSPACE;
    h.ws = w;

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the array still holds the previous call's words: the status header must start at zero
    // (the per-query state is rewritten by the query set-up kernel)
    KGE_CUDA_CHECK(&h, cudaMemsetAsync(w.status, 0, 256, s));
    int rc = run_score_all_topk(&h, q_heads, q_rels, nq, k, true_tails, out_ids, out_scores, out_ranks, s, nullptr);
    if (rc != KGE_OK) return rc;
    int32_t word = 0;
    KGE_CUDA_CHECK(&h, cudaMemcpyAsync(&word, w.status, 4, cudaMemcpyDeviceToHost, s));
    KGE_CUDA_CHECK(&h, cudaStreamSynchronize(s));
    return word;   // 0, or the code a kernel recorded (an id outside its table, a bounded wait that ran out)
}
