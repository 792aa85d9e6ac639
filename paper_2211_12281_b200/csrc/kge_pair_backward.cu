// Backward of the score block for the distance kinds whose pair is a function of (q, t) alone, both sides
// in one pass:  dQ_b = sum_n G_bn df/dq,  dT_n = sum_b G_bn df/dt  (TransE, RotatE; fp32 on CUDA cores).
//
// Bound: the arithmetic pipes.  Both sides need the same function of q_b - t_n, so a pass of its own for
// each (as the dot products have, whose two sides share nothing) computes it twice: per element and both
// sides 4 -> 3 instructions for p = 1 (compare, two predicated additions) and p = 2 (difference, two
// multiply-adds), per complex modulus 16 + 2 -> 10 + 1 (the special-function root once).
//
// A thread owns one float4 column of PB_R query rows: rows and their sums stay in registers.  Threads are
// numbered (row group, column) without padding, so a row width that is no multiple of 128 floats leaves
// only the remainder of the CTA idle (d = 200: 250 of 256 threads; a warp per row left 14 of 64 lanes idle and, for
// d > 128, two slices per lane at half the occupancy).  The rows of the other side arrive C at a time by one
// bulk copy into a double buffer; every group leaves its share of their gradients in shared memory, and
// after the chunk the groups' shares are added in order into the CTA's own slab of dT.
//
// A CTA works on a rectangle: the query rows [q_begin, q_end), a tile of PB_R x groups rows at a time, against its
// columns.  Every column range gives one slab of dQ, every row range one of dT; the chain kernel adds the slabs in
// order.  No atomics: results are bit-reproducible.
//
// Measured against a pass per side: TransE p = 1, 1024 x 1024 x 128 31.4 -> 25.1 us, 4096 x 4096 389 -> 362; p = 2, 4096 x 4096
// 410 -> 330; 512 x 1024 x 256 36 -> 25; RotatE moduli 600 x 1500 x 200 118 -> 56, 2048 x 2048 x 200 500 -> 236.  Rows of fewer
// than 32 floats keep the pass per side: a group is then so narrow that a thread would stage sixteen or more weights per chunk.
#include <algorithm>

#include "kge_common.cuh"

namespace kge {

namespace {

constexpr int PB_R = 8;              // query rows per thread
constexpr int PB_MIN_D4 = 8;         // narrower rows: too few threads share a chunk's weights

struct PairBackParams {
    const float4 *Q, *T;             // [B, d4], [N, d4]
    const float* G;                  // [B, N] dL/dF (p = 2: divided by the distance)
    int B, N, d4, groups;
    int q_rows, n_cols;              // rectangle of a CTA
    float4 *dQ, *dT;                 // [column ranges][B, d4], [row ranges][N, d4]
    float* Csum;                     // [row ranges][N] sums of G over the rows (p = 1)
    int32_t* status;
    int wait_limit;
};

__device__ __forceinline__ void add_both_if_gt(float& aq, float& at, float q, float t, float w) {
    asm("{\n .reg .pred p;\n setp.gt.f32 p, %2, %3;\n @p add.f32 %0, %0, %4;\n @p add.f32 %1, %1, %4;\n}\n" : "+f"(aq), "+f"(at) : "f"(q), "f"(t), "f"(w));
}
// One float4 column of a pair.  p = 1: both sides collect P = sum of the weights of the pairs with q > t (the chain kernel
// forms (row sum) - 2 P and 2 P - (column sum)).  Otherwise aq += w df/dq and at collects w df/dq as well, which is -w df/dt:
// p = 2 with w = G / distance; moduli with one special-function reciprocal root per complex component (relative error
// 2^-22; a zero modulus has both parts zero, so the finite factor from the floor contributes nothing).
template <int KIND>
__device__ __forceinline__ void pair_back(float4& aq, float4& at, float4 q, float4 t, float w) {
    if (KIND == KIND_L1) {
        add_both_if_gt(aq.x, at.x, q.x, t.x, w); add_both_if_gt(aq.y, at.y, q.y, t.y, w);
        add_both_if_gt(aq.z, at.z, q.z, t.z, w); add_both_if_gt(aq.w, at.w, q.w, t.w, w);
        return;
    }
    const float2 a = sub2(make_float2(t.x, t.y), make_float2(q.x, q.y)), b = sub2(make_float2(t.z, t.w), make_float2(q.z, q.w));
    float wa = w, wb = w;
    if (KIND == KIND_CL1) {
        wa *= approx_rsqrt(fmaxf(fmaf(a.x, a.x, a.y * a.y), 1e-37f));
        wb *= approx_rsqrt(fmaxf(fmaf(b.x, b.x, b.y * b.y), 1e-37f));
    }
    aq.x = fmaf(wa, a.x, aq.x); aq.y = fmaf(wa, a.y, aq.y); aq.z = fmaf(wb, b.x, aq.z); aq.w = fmaf(wb, b.y, aq.w);
    at.x = fmaf(wa, a.x, at.x); at.y = fmaf(wa, a.y, at.y); at.z = fmaf(wb, b.x, at.z); at.w = fmaf(wb, b.y, at.w);
}

__host__ __device__ inline int pb_chunk(int d4) { return d4 > 64 ? 8 : 16; }
inline int pb_groups(int B, int d4) { return std::min({256 / d4, std::max(8, 64 / d4), (B + PB_R - 1) / PB_R}); }
inline int pb_threads(int d4, int groups) { return (groups * d4 + 31) / 32 * 32; }
inline size_t pb_smem(int d4, int groups) {
    const int C = pb_chunk(d4);
    return (size_t)2 * C * d4 * 16 + (size_t)groups * C * d4 * 16 + (size_t)2 * C * (PB_R * groups + 4) * 4 + 2 * sizeof(uint64_t);
}

// C: rows of the other side per chunk; WPT: weights of a chunk a thread brings in; D4: the row width when 256 threads are
// whole groups of it (addresses and the groups' reduction are then constants: 4.5 -> 4.1 instructions per element at p = 1), or 0.
template <int KIND, int C, int WPT, int D4>
__global__ void __launch_bounds__(256, 2) pair_backward_kernel(PairBackParams p) {
    extern __shared__ __align__(128) unsigned char pb_smem_raw[];
    const int d4 = D4 ? D4 : p.d4, G = D4 ? 256 / (D4 ? D4 : 1) : p.groups, QT = PB_R * G, ldw = QT + 4;
    float4* Bs = reinterpret_cast<float4*>(pb_smem_raw);                   // [2][C][d4]
    float4* slab = Bs + 2 * C * d4;                                        // [G][C][d4] the groups' shares of dT
    float* Gs = reinterpret_cast<float*>(slab + (size_t)G * C * d4);       // [2][C][ldw]
    uint64_t* bars = reinterpret_cast<uint64_t*>(Gs + 2 * C * ldw);

    const int tid = threadIdx.x, nthr = D4 ? 256 : blockDim.x;
    const int g = tid / d4, c = tid - g * d4;
    const bool active = g < G;
    const int n0 = blockIdx.x * p.n_cols, n1 = min(p.N, n0 + p.n_cols);
    const int q_begin = blockIdx.y * p.q_rows, q_end = min(p.B, q_begin + p.q_rows);
    const int chunks = (n1 - n0 + C - 1) / C, tiles = (q_end - q_begin + QT - 1) / QT;

    if (tid == 0) { mbar_init(&bars[0], 1); mbar_init(&bars[1], 1); mbar_init_fence(); }
    __syncthreads();
    grid_dependency_wait();
    allow_dependents();

    auto issue_rows = [&](int ch, int buf) {         // thread 0 only
        const int first = n0 + ch * C;
        const uint32_t bytes = (uint32_t)min(C, n1 - first) * (uint32_t)d4 * 16u;
        mbar_arrive_expect_tx(&bars[buf], bytes);
        bulk_g2s(Bs + (size_t)buf * C * d4, p.T + (int64_t)first * d4, bytes, &bars[buf]);
    };
    float greg[WPT];
    auto load_weights = [&](int tile, int ch) {
#pragma unroll
        for (int e = 0; e < WPT; ++e) {
            const int idx = tid + nthr * e, cc = idx % C, rr = idx / C;
            const int b = q_begin + tile * QT + rr, n = n0 + ch * C + cc;
            greg[e] = (rr < QT && b < q_end && n < n1) ? p.G[(int64_t)b * p.N + n] : 0.f;
        }
    };
    auto store_weights = [&](int buf) {
#pragma unroll
        for (int e = 0; e < WPT; ++e) {
            const int idx = tid + nthr * e, cc = idx % C, rr = idx / C;
            if (rr < QT) Gs[(buf * C + cc) * ldw + rr] = greg[e];
        }
    };
    float4 A[PB_R], acc[PB_R];
    auto load_rows = [&](int tile) {
#pragma unroll
        for (int i = 0; i < PB_R; ++i) {
            const int b = q_begin + tile * QT + g * PB_R + i;
            A[i] = (active && b < q_end) ? p.Q[(int64_t)b * d4 + c] : make_float4(0.f, 0.f, 0.f, 0.f);
            acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };

    if (tid == 0) issue_rows(0, 0);
    load_weights(0, 0);
    load_rows(0);
    store_weights(0);
    int tile = 0, ch = 0;
    for (int it = 0; it < tiles * chunks; ++it) {
        const int cur = it & 1;
        const bool more = it + 1 < tiles * chunks, tile_ends = ch + 1 == chunks;
        if (more) {
            if (tid == 0) issue_rows(tile_ends ? 0 : ch + 1, cur ^ 1);
            load_weights(tile_ends ? tile + 1 : tile, tile_ends ? 0 : ch + 1);
        }
        const bool ok = mbar_wait_bounded(&bars[cur], (uint32_t)(it >> 1) & 1u, p.wait_limit);
        if (!__syncthreads_and(ok)) {
            if (tid == 0) set_status(p.status, KGE_ERR_TIMEOUT);
            (void)mbar_wait_bounded(&bars[cur ^ 1], (uint32_t)((it + 1) >> 1) & 1u, p.wait_limit);
            return;
        }
        const int first = n0 + ch * C, ccmax = min(C, n1 - first);
        const float* Gc = Gs + cur * C * ldw;
        if (active) {
            const float4* Bc = Bs + (size_t)cur * C * d4 + c;
            float4* out = slab + (size_t)g * C * d4 + c;
            const float* gp = Gc + g * PB_R;
            // rolled: unrolled, the compiler holds the next iteration's operands in a second register set and copies them over
#pragma unroll 1
            for (int cc = 0; cc < ccmax; ++cc, Bc += d4, out += d4, gp += ldw) {
                const float4 w0 = *reinterpret_cast<const float4*>(gp), w1 = *reinterpret_cast<const float4*>(gp + 4);
                const float4 t = *Bc;
                float4 dt = make_float4(0.f, 0.f, 0.f, 0.f);
                pair_back<KIND>(acc[0], dt, A[0], t, w0.x); pair_back<KIND>(acc[1], dt, A[1], t, w0.y);
                pair_back<KIND>(acc[2], dt, A[2], t, w0.z); pair_back<KIND>(acc[3], dt, A[3], t, w0.w);
                pair_back<KIND>(acc[4], dt, A[4], t, w1.x); pair_back<KIND>(acc[5], dt, A[5], t, w1.y);
                pair_back<KIND>(acc[6], dt, A[6], t, w1.z); pair_back<KIND>(acc[7], dt, A[7], t, w1.w);
                *out = dt;
            }
        }
        if (KIND == KIND_L1) {       // the weights' column sums, a warp per column
            for (int cc = tid >> 5; cc < ccmax; cc += nthr >> 5) {
                float v = 0.f;
                for (int r = tid & 31; r < QT; r += 32) v += Gc[cc * ldw + r];
                v = warp_sum(v);
                float* dst = p.Csum + (int64_t)blockIdx.y * p.N + first + cc;
                if ((tid & 31) == 0) *dst = tile == 0 ? v : *dst + v;
            }
        }
        if (more) store_weights(cur ^ 1);
        __syncthreads();
        // the groups' shares in ascending order, onto what the row range's earlier tiles left
        constexpr float SIGN = KIND == KIND_L1 ? 1.f : -1.f;
        float4* dst = p.dT + ((int64_t)blockIdx.y * p.N + first) * d4;
        for (int i = tid; i < ccmax * d4; i += nthr) {
            float4 s = tile == 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : dst[i];
            const float4* v = slab + i;
            if (D4) {
#pragma unroll
                for (int k = 0; k < (D4 ? 256 / (D4 ? D4 : 1) : 1); ++k) {
                    const float4 u = v[k * C * D4];
                    s.x += SIGN * u.x; s.y += SIGN * u.y; s.z += SIGN * u.z; s.w += SIGN * u.w;
                }
            } else {
#pragma unroll 2
                for (int k = 0; k < G; ++k, v += C * d4) {
                    const float4 u = *v;
                    s.x += SIGN * u.x; s.y += SIGN * u.y; s.z += SIGN * u.z; s.w += SIGN * u.w;
                }
            }
            dst[i] = s;
        }
        if (tile_ends) {
            if (active) {
#pragma unroll
                for (int i = 0; i < PB_R; ++i) {
                    const int b = q_begin + tile * QT + g * PB_R + i;
                    if (b < q_end) p.dQ[((int64_t)blockIdx.x * p.B + b) * d4 + c] = acc[i];
                }
            }
            if (more) load_rows(tile + 1);
            ++tile; ch = 0;
        } else {
            ++ch;
        }
    }
}

template <int KIND, int C, int WPT, int D4>
cudaError_t launch_inst(const PairBackParams& p, dim3 grid, cudaStream_t s) {
    static DeviceOnce configured;
    const cudaError_t e = once_per_device(configured, [] {
        return cudaFuncSetAttribute(pair_backward_kernel<KIND, C, WPT, D4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024);
    });
    if (e != cudaSuccess) return e;
    return launch_dependent(pair_backward_kernel<KIND, C, WPT, D4>, grid, dim3(pb_threads(p.d4, p.groups)), pb_smem(p.d4, p.groups), s, p);
}
template <int KIND>
cudaError_t launch_kind(const PairBackParams& p, dim3 grid, cudaStream_t s) {
    if (p.d4 == 32 && p.groups == 8) return launch_inst<KIND, 16, 4, 32>(p, grid, s);
    if (p.d4 == 64 && p.groups == 4) return launch_inst<KIND, 16, 2, 64>(p, grid, s);
    if (p.d4 > 64) return launch_inst<KIND, 8, 1, 0>(p, grid, s);
    return p.d4 >= 32 ? launch_inst<KIND, 16, 4, 0>(p, grid, s) : launch_inst<KIND, 16, 16, 0>(p, grid, s);
}

}  // namespace

bool pair_backward_serves(const kge_handle* h) {
    return h->cfg.prec == KGE_PREC_FP32 && (h->kind == KIND_L1 || h->kind == KIND_L2 || h->kind == KIND_CL1) && h->cfg.dim / 4 >= PB_MIN_D4;
}

// Column ranges (split_q: slabs of dQ) and row ranges (split_t: slabs of dT).  The CTAs of one wave fill the GPU; among the
// divisions that do, the one whose longest CTA plus the slabs' traffic is shortest: a chunk row costs about 0.11 us per
// CTA and SM-resident CTA pair at 256 threads (moduli 0.24), a tile's start about 24 such rows, a slab is written and read at some
// 5 TB/s.  More than 64 column ranges, where the rows leave places for them, have to gain more than the chain kernel's rounds over their
// slabs cost (eight slabs a round, some 1.2 us): 64 x 16,384 x 128 in 64 ranges 126 us a step (RotatE 207), in 128 113 (151), in 256 126
// (129); 64 x 4,096 x 128 in 64 ranges 56 us, in 128 60 (RotatE 81 and 76).
void pair_backward_split(int kind, int B, int N, int d4, int num_sms, int* split_q, int* split_t) {
    const int groups = pb_groups(B, d4), threads = pb_threads(d4, groups), q_tiles = (B + PB_R * groups - 1) / (PB_R * groups);
    const int ctas_per_sm = std::max(1, std::min({65536 / (threads * 128), (int)(224 * 1024 / (pb_smem(d4, groups) + 1024)), 16}));
    const int slots = num_sms * ctas_per_sm;
    const double width = ctas_per_sm * (threads / 256.0), slab_us = d4 * 32.0 / 5e6;
    double best = 1e30;
    *split_q = *split_t = 1;
    for (int sq = 1; sq <= std::min(q_tiles, 64); ++sq) {
        const int tiles = (q_tiles + sq - 1) / sq, rows = (q_tiles + tiles - 1) / tiles;             // row ranges that are not empty
        if (rows != sq) continue;
        const int want = std::max(1, std::min({slots / rows, 64, (N + 15) / 16}));
        const int per = (N + want - 1) / want, cols = (N + per - 1) / per;
        const int waves = (rows * cols + slots - 1) / slots;
        const double us = 0.11 * width * waves * tiles * (per + 24) + ((double)rows * N + (double)cols * B) * slab_us;
        if (us < best) { best = us; *split_q = cols; *split_t = rows; }
    }
    const int cols64 = *split_q, rows = *split_t, tiles = (q_tiles + rows - 1) / rows;
    double gain = 0.0;
    for (int want = std::min(slots / rows, (N + 15) / 16); want > 64; want /= 2) {
        const int per = (N + want - 1) / want, cols = (N + per - 1) / per;
        const double us = (kind == KIND_CL1 ? 0.24 : 0.11) * width * tiles * ((N + cols64 - 1) / cols64 - per) - (double)(cols - cols64) * B * slab_us -
                          1.2 * ((cols + 7) / 8 - (cols64 + 7) / 8);
        if (us > gain) { gain = us; *split_q = cols; }
    }
}

int launch_pair_backward(kge_handle* h, cudaStream_t s) {
    const kge_config& c = h->cfg;
    const Workspace& w = h->ws;
    PairBackParams p;
    p.Q = reinterpret_cast<const float4*>(w.Q); p.T = reinterpret_cast<const float4*>(w.Tneg); p.G = w.F;
    p.B = c.batch; p.N = c.num_neg; p.d4 = c.dim / 4; p.groups = pb_groups(c.batch, p.d4);
    const int tile_rows = PB_R * p.groups, q_tiles = (p.B + tile_rows - 1) / tile_rows;
    p.q_rows = (q_tiles + h->split_t - 1) / h->split_t * tile_rows;
    p.n_cols = (p.N + h->split_q - 1) / h->split_q;
    p.dQ = reinterpret_cast<float4*>(w.dQpart); p.dT = reinterpret_cast<float4*>(w.dTpart); p.Csum = w.Cpart;
    p.status = w.status; p.wait_limit = h->wait_limit;
    const dim3 grid(h->split_q, h->split_t);
    KGE_CUDA_CHECK(h, h->kind == KIND_L1 ? launch_kind<KIND_L1>(p, grid, s) : (h->kind == KIND_L2 ? launch_kind<KIND_L2>(p, grid, s) : launch_kind<KIND_CL1>(p, grid, s)));
    KGE_LAUNCH_CHECK(h);
    return KGE_OK;
}

}  // namespace kge
