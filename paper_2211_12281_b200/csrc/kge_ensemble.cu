// Power-rank ensemble (Section 3.2 "Ensemble", Eq. 2): M models each give a top-K list of tails per
// query; an entity's ensemble score is the sum over the models of a rank-based score,
//     s_m(t) = -sgn(p) k^p            if t is the k-th entry of model m's list (k = 1 .. K)
//              -[p > 0] (K + 1)^p     if t is not in model m's list,
// and the query's final prediction is the top-n entities by s(t) (ties: smaller entity id first).
// Only entities that occur in some list can reach the top (an entity in no list has the lowest
// possible score and every list holds K >= n distinct entities), so the candidates of a query are
// the union of its M lists.
//
// One thread block per query gathers the union in a hash table in shared memory, models in ascending
// blocks: a block's entries are inserted in any order (the position of an entity in each of the
// block's models is one byte of the entity's cell words), then every entity adds its rank scores
// model by model in ascending order (an absent model contributes the absent score at its place in
// that order), in fp64; n rounds of a block-wide maximum then pick the result.  The rank scores k^p
// come from a table the caller fills with kge_ensemble_rank_scores, so the sums are plain IEEE
// additions of given numbers in a fixed order: the result does not depend on any device math library.
// A query whose union does not fit the table, or with an entity twice in one list, is left to a second
// launch, which has a larger table and, behind that, a sort of all entries by (entity id, model, position).
#include <algorithm>
#include <cmath>

#include "kge_common.cuh"

namespace kge {
namespace {

constexpr int ENS_THREADS = 512;            // the sort
constexpr int ENS_MAX_ENTRIES = 16384;      // M * K per query (85 models x top-100 = 8,500 fits)
constexpr int ENS_MAX_K = 254;              // positions are kept as bytes (position + 1); longer lists are sorted
constexpr int ENS_LEFT = -2;                // first output id of a query the first launch left to the second

struct EnsParams {
    const int32_t* lists;      // [M, nq, K]
    const double* table;       // [K + 1]: rank scores of positions 1 .. K, then the absent score
    int M, nq, K, top_n, n2;   // n2 = M * K rounded up to a power of two
    int32_t* out_ids; double* out_scores;
    int log2_slots;            // first launch: slots of the hash table
    uint32_t inv_k;            // ceil(2^32 / K): e / K = umulhi(e, inv_k) for every entry index e of a block of models; 0: K = 1
};

__device__ __forceinline__ bool ens_before(double sa, int32_t ia, double sb, int32_t ib) { return sa > sb || (sa == sb && ia < ib); }

// ------------------------------------------------------------------------------------------
// Hash form.  Shared memory per slot: entity id, fp64 sum, MB position bytes, one entry of the list of
// occupied slots.  The cell words of a slot lie `slots` words apart, so that the slots a warp touches
// (random, one model) spread over the banks.
// Returns false (all threads) if the union does not fit or a list names an entity twice.
// ------------------------------------------------------------------------------------------
template <int MB>
constexpr size_t ens_slot_bytes() { return sizeof(double) + sizeof(int32_t) + MB + sizeof(uint16_t); }
template <int MB>
inline size_t ens_hash_smem(int slots, int K) { return (size_t)slots * ens_slot_bytes<MB>() + (size_t)(K + 1) * sizeof(double); }

// Order-preserving map of a double to an unsigned integer (no NaN).
__device__ __forceinline__ uint64_t ens_ordered(double s) {
    const uint64_t b = (uint64_t)__double_as_longlong(s);
    return (b >> 63) ? ~b : b | 0x8000000000000000ull;
}
__device__ __forceinline__ double ens_unordered(uint64_t k) {
    return __longlong_as_double((long long)((k >> 63) ? k & 0x7fffffffffffffffull : ~k));
}

template <int MB>
__device__ bool ens_hash_query(const EnsParams& p, const int q, const int log2_slots, unsigned char* smem) {
    constexpr int WORDS = MB / 4;
    const int slots = 1 << log2_slots, tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
    double* sum = reinterpret_cast<double*>(smem);                              // [slots]
    double* tab = sum + slots;                                                  // [K + 1] absent score, then positions 1 .. K
    int32_t* key = reinterpret_cast<int32_t*>(tab + p.K + 1);                   // [slots] entity id or -1
    uint32_t* cell = reinterpret_cast<uint32_t*>(key + slots);                  // [WORDS][slots] bytes: position + 1 in the block's models
    uint16_t* used = reinterpret_cast<uint16_t*>(cell + (size_t)WORDS * slots); // [slots] occupied slots, in order of arrival
    __shared__ int n_used, bad;
    __shared__ uint64_t red_s[2][32];
    __shared__ int32_t red_i[2][32];
    for (int i = tid; i < slots; i += nthr) key[i] = -1;
    for (int i = tid; i < slots * WORDS; i += nthr) cell[i] = 0u;
    for (int i = tid; i <= p.K; i += nthr) tab[i] = p.table[i == 0 ? p.K : i - 1];
    if (tid == 0) { n_used = 0; bad = 0; }
    __syncthreads();
    const double absent = tab[0];
    double before = 0.0;                    // an entity's sum over the models ahead of the block it first appears in
    int seen = 0;                           // occupied slots after the blocks so far
    for (int m0 = 0; m0 < p.M; m0 += MB) {
        const int mb = min(MB, p.M - m0), entries = mb * p.K;
        const int32_t* src = p.lists + ((int64_t)m0 * p.nq + q) * p.K;
        const int64_t step = (int64_t)(p.nq - 1) * p.K;                         // list m + 1 begins `step` further than list m ends
        for (int e0 = 0; e0 < entries; e0 += 4 * nthr) {
            int32_t id[4];
            int ml[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {                                       // four loads in flight
                const int e = e0 + u * nthr + tid;
                ml[u] = p.inv_k ? (int)__umulhi((uint32_t)e, p.inv_k) : e;
                id[u] = e < entries ? src[e + ml[u] * step] : -1;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                // the warp probes together: left to themselves, the lanes that need one probe more run the rest of the body on their own
                const int e = e0 + u * nthr + tid, want = id[u];
                uint32_t h = (uint32_t)want * 0x9E3779B1u >> (32 - log2_slots);
                int32_t k = want < 0 ? want : *reinterpret_cast<volatile int32_t*>(key + h);       // (unused places of a list hold -1)
                bool need = k != want;
                for (int probe = 0; probe < slots && __any_sync(0xffffffffu, need); ++probe) {
                    if (need && k == -1) {
                        k = atomicCAS(key + h, -1, want);
                        if (k == -1) { used[atomicAdd(&n_used, 1)] = (uint16_t)h; k = want; }
                    }
                    need = need && k != want;
                    if (need) {
                        h = (h + 1) & (uint32_t)(slots - 1);
                        k = *reinterpret_cast<volatile int32_t*>(key + h);
                        need = k != want;
                    }
                    if ((probe & 15) == 15 && __any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&bad))) break;
                }
                const uint32_t sh = (uint32_t)(ml[u] & 3) * 8u;
                if (want >= 0 && (need || (atomicAdd(&cell[(ml[u] >> 2) * slots + h], (uint32_t)(e - ml[u] * p.K + 1) << sh) >> sh & 0xffu) != 0u)) bad = 1;
            }
            // (by vote: the lanes read the flag at different times, and those that stay vote with the whole warp again)
            if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&bad))) break;
        }
        __syncthreads();
        if (bad) return false;
        const int total = n_used;
        for (int i = tid; i < total; i += nthr) {
            const int h = used[i];
            double s = i < seen ? sum[h] : before;
            for (int w = 0; 4 * w < mb; ++w) {
                const uint32_t c = cell[w * slots + h];
                cell[w * slots + h] = 0u;
                if (c == 0u && absent == 0.0) continue;                         // (s is never -0: adding 0 leaves it as it is)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (4 * w + j < mb) s += tab[c >> (8 * j) & 0xffu];
            }
            sum[h] = s;
        }
        seen = total;
        if (absent != 0.0) for (int m = 0; m < mb; ++m) before += absent;
        __syncthreads();
    }
    // a thread's best candidate stays in registers until it is taken
    auto best_of_mine = [&](uint64_t& bs, int32_t& bi, int& bp) {
        bs = 0; bi = INT32_MAX; bp = -1;
        for (int i = tid; i < seen; i += nthr) {
            const int h = used[i];
            if (key[h] < 0) continue;
            const uint64_t s = ens_ordered(sum[h]);
            if (bp < 0 || s > bs || (s == bs && key[h] < bi)) { bs = s; bi = key[h]; bp = h; }
        }
    };
    uint64_t bs; int32_t bi; int bp;
    best_of_mine(bs, bi, bp);
    // warp maximum under (score descending, id ascending): the score's two halves, then the id
    auto warp_best = [&](uint64_t s, int32_t id, uint64_t& os, int32_t& oi) {
        const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(s >> 32));
        const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(s >> 32) == hi ? (uint32_t)s : 0u);
        os = (uint64_t)hi << 32 | lo;
        oi = __reduce_min_sync(0xffffffffu, s == os ? id : INT32_MAX);
    };
    uint64_t ws; int32_t wi;                // the warp's best
    warp_best(bs, bi, ws, wi);
    for (int r = 0; r < p.top_n; ++r) {
        if (lane == 0) { red_s[r & 1][warp] = ws; red_i[r & 1][warp] = wi; }
        __syncthreads();
        uint64_t s; int32_t id;
        warp_best(lane < nwarps ? red_s[r & 1][lane] : 0ull, lane < nwarps ? red_i[r & 1][lane] : INT32_MAX, s, id);   // (every warp for itself)
        const bool have = s != 0ull;                                            // (no score maps to 0)
        if (tid == 0) {
            p.out_ids[(int64_t)q * p.top_n + r] = have ? id : -1;               // fewer candidates than places: -1 and -inf
            if (p.out_scores) p.out_scores[(int64_t)q * p.top_n + r] = have ? ens_unordered(s) : -INFINITY;
        }
        if (have && s == ws && id == wi) {                                      // taken (ids are distinct: one warp, one thread)
            if (bp >= 0 && bi == id) { key[bp] = -1; best_of_mine(bs, bi, bp); }
            __syncwarp();
            warp_best(bs, bi, ws, wi);
        }
    }
    return true;
}

// First launch: one CTA per query, 16 models at a time, at most 1,024 slots (31 KB: seven CTAs per SM).  85 x top-100 lists of
// 15,000 queries: 36.7 ms as a sort, 0.93 ms with 32 models at a time (four CTAs), 0.87 with 8, 0.81 with 16; 128 threads 1.00 ms.
// Bound by instruction issue (about 48,000 warp instructions a query, 74 % of the slots), not by the 510 MB of lists (78 us).
constexpr int ENS_MB = 16, ENS_MAX_LOG2 = 10;
template <int MB>
__global__ void __launch_bounds__(256) ensemble_hash_kernel(EnsParams p) {
    extern __shared__ __align__(16) unsigned char ens_smem[];
    allow_dependents();
    if (!ens_hash_query<MB>(p, blockIdx.x, p.log2_slots, ens_smem) && threadIdx.x == 0) p.out_ids[(int64_t)blockIdx.x * p.top_n] = ENS_LEFT;
}

// The general form: all entries of query q sorted by (entity id, model, position) in shared memory.
__device__ void ens_sort_query(const EnsParams& p, const int q, unsigned char* ens_smem) {
    uint64_t* key = reinterpret_cast<uint64_t*>(ens_smem);                      // [n2] (id, model, position); later the candidates' scores
    int32_t* cid = reinterpret_cast<int32_t*>(key + p.n2);                      // [n2] candidate id at the first entry of its run, else -1
    __shared__ double red_s[ENS_THREADS / 32];
    __shared__ int32_t red_i[ENS_THREADS / 32], red_pos[ENS_THREADS / 32];
    __shared__ int32_t win_pos;
    const int tid = threadIdx.x, n = p.M * p.K;
    for (int i = tid; i < p.n2; i += ENS_THREADS) {
        uint64_t k = ~0ull;
        if (i < n) {
            const int m = i / p.K, pos = i - m * p.K;
            const int32_t id = p.lists[((int64_t)m * p.nq + q) * p.K + pos];
            if (id >= 0) k = ((uint64_t)(uint32_t)id << 32) | ((uint64_t)m << 16) | (uint64_t)pos;   // unused places of a list hold -1
        }
        key[i] = k;
    }
    __syncthreads();
    for (int size = 2; size <= p.n2; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = tid; t < p.n2 / 2; t += ENS_THREADS) {
                const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                const bool up = (lo & size) == 0;
                const uint64_t x = key[lo], y = key[hi];
                if ((x > y) == up) { key[lo] = y; key[hi] = x; }
            }
            __syncthreads();
        }
    // runs of equal ids: mark their first entries (reads only)
    for (int i = tid; i < p.n2; i += ENS_THREADS) {
        const uint64_t k = key[i];
        const bool head = k != ~0ull && (i == 0 || (key[i - 1] >> 32) != (k >> 32));
        cid[i] = head ? (int32_t)(k >> 32) : -1;
    }
    __syncthreads();
    // every run is summed by the thread of its first entry, which then keeps the score in that entry's place
    const double absent = p.table[p.K];
    for (int i = tid; i < p.n2; i += ENS_THREADS) {
        if (cid[i] < 0) continue;
        const uint32_t id = (uint32_t)cid[i];
        int j = i;
        double s = 0.0;
        for (int m = 0; m < p.M; ++m) {
            bool present = false;
            while (j < p.n2 && (uint32_t)(key[j] >> 32) == id && (int)((key[j] >> 16) & 0xffffu) == m) {
                s += p.table[key[j] & 0xffffu];
                present = true; ++j;
            }
            if (!present) s += absent;
        }
        key[i] = (uint64_t)__double_as_longlong(s);
    }
    __syncthreads();
    for (int r = 0; r < p.top_n; ++r) {
        double bs = -INFINITY; int32_t bi = INT32_MAX, bp = -1;
        for (int i = tid; i < p.n2; i += ENS_THREADS) {
            const int32_t id = cid[i];
            if (id < 0) continue;
            const double s = __longlong_as_double((long long)key[i]);
            if (bp < 0 || ens_before(s, id, bs, bi)) { bs = s; bi = id; bp = i; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double os = __shfl_xor_sync(0xffffffffu, bs, o);
            const int32_t oi = __shfl_xor_sync(0xffffffffu, bi, o), op = __shfl_xor_sync(0xffffffffu, bp, o);
            if (op >= 0 && (bp < 0 || ens_before(os, oi, bs, bi))) { bs = os; bi = oi; bp = op; }
        }
        if ((tid & 31) == 0) { red_s[tid >> 5] = bs; red_i[tid >> 5] = bi; red_pos[tid >> 5] = bp; }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < ENS_THREADS / 32; ++w)
                if (red_pos[w] >= 0 && (bp < 0 || ens_before(red_s[w], red_i[w], bs, bi))) { bs = red_s[w]; bi = red_i[w]; bp = red_pos[w]; }
            p.out_ids[(int64_t)q * p.top_n + r] = bp >= 0 ? bi : -1;          // fewer candidates than places: -1 and -inf
            if (p.out_scores) p.out_scores[(int64_t)q * p.top_n + r] = bp >= 0 ? bs : -INFINITY;
            win_pos = bp;
        }
        __syncthreads();
        if (tid == 0 && win_pos >= 0) cid[win_pos] = -1;                       // taken
        __syncthreads();
    }
}

// Lists of more than ENS_MAX_K places: every query takes the general form.
__global__ void __launch_bounds__(ENS_THREADS) ensemble_sort_kernel(EnsParams p) {
    extern __shared__ __align__(16) unsigned char ens_smem[];
    ens_sort_query(p, blockIdx.x, ens_smem);
}

// Second launch: the queries the first one left (usually none), shared out over the CTAs.
constexpr int ENS_BIG_MB = 8, ENS_BIG_LOG2 = 13;      // 8,192 slots, eight models at a time: 180 KB
__global__ void __launch_bounds__(ENS_THREADS) ensemble_left_kernel(EnsParams p) {
    extern __shared__ __align__(16) unsigned char ens_smem[];
    __shared__ int32_t todo[ENS_THREADS];
    __shared__ int n_todo;
    grid_dependency_wait();
    for (int64_t base = blockIdx.x; base < p.nq; base += (int64_t)gridDim.x * ENS_THREADS) {
        __syncthreads();
        if (threadIdx.x == 0) n_todo = 0;
        __syncthreads();
        const int64_t q = base + (int64_t)gridDim.x * threadIdx.x;
        if (q < p.nq && p.out_ids[q * p.top_n] == ENS_LEFT) todo[atomicAdd(&n_todo, 1)] = (int32_t)q;
        __syncthreads();
        const int n = n_todo;
        for (int i = 0; i < n; ++i) {
            __syncthreads();
            const bool done = ens_hash_query<ENS_BIG_MB>(p, todo[i], ENS_BIG_LOG2, ens_smem);
            __syncthreads();
            if (!done) ens_sort_query(p, todo[i], ens_smem);
        }
    }
}

}  // namespace
}  // namespace kge

extern "C" {

int kge_ensemble_rank_scores(double power, int32_t k_list, double* table) {
    if (!table || k_list <= 0 || power == 0.0 || !std::isfinite(power)) return KGE_ERR_BAD_ARG;
    const double sign = power > 0.0 ? 1.0 : -1.0;
    for (int32_t k = 1; k <= k_list; ++k) table[k - 1] = -sign * std::pow((double)k, power);
    table[k_list] = power > 0.0 ? -std::pow((double)k_list + 1.0, power) : 0.0;
    return KGE_OK;
}

int kge_ensemble_topk(const int32_t* lists, int32_t num_models, int32_t nq, int32_t k_list, const double* table,
                      int32_t top_n, int32_t* out_ids, double* out_scores, void* stream) {
    using namespace kge;
    if (!lists || !table || !out_ids || num_models <= 0 || nq < 0 || k_list <= 0 || top_n <= 0) return KGE_ERR_BAD_ARG;
    if (num_models > 65535 || k_list > 65535) return KGE_ERR_UNSUPPORTED;
    if ((int64_t)num_models * k_list > ENS_MAX_ENTRIES) return KGE_ERR_WORKSPACE;
    if (nq == 0) return KGE_OK;
    EnsParams p;
    p.lists = lists; p.table = table; p.M = num_models; p.nq = nq; p.K = k_list; p.top_n = top_n;
    p.n2 = 2;
    while (p.n2 < num_models * k_list) p.n2 <<= 1;
    p.out_ids = out_ids; p.out_scores = out_scores;
    const size_t sort_smem = (size_t)p.n2 * (sizeof(uint64_t) + sizeof(int32_t));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    static DeviceOnce configured;
    cudaError_t e = once_per_device(configured, [] {
        constexpr int sort_max = (int)(ENS_MAX_ENTRIES * (sizeof(uint64_t) + sizeof(int32_t)));
        static_assert((1 << ENS_BIG_LOG2) * ens_slot_bytes<ENS_BIG_MB>() + (ENS_MAX_K + 1) * sizeof(double) <= sort_max, "the larger table fits where the sort does");
        cudaError_t e0 = cudaFuncSetAttribute(ensemble_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_max);
        if (e0 == cudaSuccess) e0 = cudaFuncSetAttribute(ensemble_left_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_max);
        if (e0 == cudaSuccess) e0 = cudaFuncSetAttribute(ensemble_hash_kernel<ENS_MB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         (int)ens_hash_smem<ENS_MB>(1 << ENS_MAX_LOG2, ENS_MAX_K));
        return e0;
    });
    if (e != cudaSuccess) return KGE_ERR_CUDA;
    if (k_list > ENS_MAX_K) {
        ensemble_sort_kernel<<<nq, ENS_THREADS, sort_smem, s>>>(p);
        return cudaGetLastError() == cudaSuccess ? KGE_OK : KGE_ERR_CUDA;
    }
    p.inv_k = (uint32_t)((((uint64_t)1 << 32) + k_list - 1) / k_list);
    p.log2_slots = 5;
    while (p.log2_slots < ENS_MAX_LOG2 && 2 << p.log2_slots < 3 * num_models * k_list) ++p.log2_slots;
    const int threads = p.log2_slots >= 9 ? 256 : (p.log2_slots >= 7 ? 128 : 64);
    ensemble_hash_kernel<ENS_MB><<<nq, threads, ens_hash_smem<ENS_MB>(1 << p.log2_slots, k_list), s>>>(p);
    if (cudaGetLastError() != cudaSuccess) return KGE_ERR_CUDA;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return KGE_ERR_CUDA;
    const size_t big_smem = std::max(sort_smem, ens_hash_smem<ENS_BIG_MB>(1 << ENS_BIG_LOG2, k_list));
    e = launch_dependent(ensemble_left_kernel, dim3((unsigned)std::min(nq, sms)), dim3(ENS_THREADS), big_smem, s, p);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? KGE_OK : KGE_ERR_CUDA;
}

}  // extern "C"
