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
// A query whose union would fill more than three quarters of the table is left to a second launch, which
// gathers it in a larger table, as many passes over the lists as its entries can need: a pass takes the
// entities whose hash falls into its part, so every sum keeps its order.  A query with an entity twice in
// one list (and lists of more than 254 places) is left to a third, which sorts all entries by (entity id, model, position).
#include <algorithm>
#include <cmath>

#include "kge_common.cuh"

namespace kge {
namespace {

constexpr int ENS_THREADS = 1024;           // at most
constexpr int ENS_MAX_ENTRIES = 16384;      // M * K per query (85 models x top-100 = 8,500 fits)
constexpr int ENS_MAX_K = 254;              // positions are kept as bytes (position + 1); longer lists are sorted
constexpr int ENS_LEFT = -2, ENS_SORT = -3;    // first output id of a query left to the second launch (too large a union) or to the sort

struct EnsParams {
    const int32_t* lists;      // [M, nq, K]
    const double* table;       // [K + 1]: rank scores of positions 1 .. K, then the absent score
    int M, nq, K, top_n, n2;   // n2 = M * K rounded up to a power of two
    int32_t* out_ids; double* out_scores;
    int log2_slots;            // first launch: slots of the hash table
    int left_log2, log2_parts; // second launch: slots of its table, passes over the lists
    int sort_here;             // second launch: its memory holds the sort too
    uint32_t inv_k;            // ceil(2^32 / K): e / K = umulhi(e, inv_k) for every entry index e of a block of models; 0: K = 1
    uint32_t inv_quads;        // the same for the quads of a list, ceil(K / 4); 0: one
};

__device__ __forceinline__ bool ens_before(double sa, int32_t ia, double sb, int32_t ib) { return sa > sb || (sa == sb && ia < ib); }

// ------------------------------------------------------------------------------------------
// Hash form.  Shared memory per slot: entity id, fp64 sum, MB position bytes, one entry of the list of
// occupied slots.  The cell words of a slot lie `slots` words apart, so that the slots a warp touches
// (random, one model) spread over the banks.
// A table that may overflow is given up at three quarters of its slots, after the block of models that takes it
// beyond or where a probe grows long: linear probing costs tens of steps per entry from there on (thousands near the
// last slot: 85 lists of 100 random ids for 15,000 queries took 134 ms that way, the sort alone 37).
// ------------------------------------------------------------------------------------------
template <int MB>
constexpr size_t ens_slot_bytes() { return sizeof(double) + sizeof(int32_t) + MB + sizeof(uint16_t); }
template <int MB>
constexpr size_t ens_hash_smem(int slots, int K) { return (size_t)slots * ens_slot_bytes<MB>() + (size_t)(K + 1) * sizeof(double); }
enum { ENS_BAD_FULL = 1, ENS_BAD_TWICE = 2 };

// Order-preserving map of a double to an unsigned integer (no NaN).
__device__ __forceinline__ uint64_t ens_ordered(double s) {
    const uint64_t b = (uint64_t)__double_as_longlong(s);
    return (b >> 63) ? ~b : b | 0x8000000000000000ull;
}
__device__ __forceinline__ double ens_unordered(uint64_t k) {
    return __longlong_as_double((long long)((k >> 63) ? k & 0x7fffffffffffffffull : ~k));
}

// The table of the entities of query q whose hash falls into part `part` of 2^log2_parts.
template <int MB>
struct EnsTable {
    double* sum;          // [slots]
    double* tab;          // [K + 1] absent score, then positions 1 .. K
    int32_t* key;         // [slots] entity id or -1
    uint32_t* cell;       // [MB / 4][slots] bytes: position + 1 in the block's models
    uint16_t* used;       // [slots] occupied slots, in order of arrival
    int n;                // of them

    __device__ EnsTable(unsigned char* smem, int slots, int K)
        : sum(reinterpret_cast<double*>(smem)), tab(sum + slots), key(reinterpret_cast<int32_t*>(tab + K + 1)),
          cell(reinterpret_cast<uint32_t*>(key + slots)), used(reinterpret_cast<uint16_t*>(cell + (size_t)(MB / 4) * slots)), n(0) {}

    // 0, or (all threads) why the table was given up: more than `limit` entities, or an entity twice in one list.
    __device__ int gather(const EnsParams& p, const int q, const int log2_slots, const int limit, const int part, const int log2_parts) {
        constexpr int WORDS = MB / 4;
        const int slots = 1 << log2_slots, tid = threadIdx.x, nthr = blockDim.x;
        __shared__ int n_used, twice;
        for (int i = tid; i < slots; i += nthr) key[i] = -1;
        for (int i = tid; i < slots * WORDS; i += nthr) cell[i] = 0u;
        for (int i = tid; i <= p.K; i += nthr) tab[i] = p.table[i == 0 ? p.K : i - 1];
        if (tid == 0) { n_used = 0; twice = 0; }
        __syncthreads();
        const double absent = tab[0];
        double before = 0.0;                    // an entity's sum over the models ahead of the block it first appears in
        int seen = 0;                           // occupied slots after the blocks so far
        for (int m0 = 0; m0 < p.M; m0 += MB) {
            const int mb = min(MB, p.M - m0), entries = mb * p.K;
            const int32_t* src = p.lists + ((int64_t)m0 * p.nq + q) * p.K;
            const int64_t step = (int64_t)(p.nq - 1) * p.K;                     // list m + 1 begins `step` further than list m ends
            for (int e0 = 0; e0 < entries; e0 += 4 * nthr) {
                int32_t id[4];
                int ml[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {                                   // four loads in flight
                    const int e = e0 + u * nthr + tid;
                    ml[u] = p.inv_k ? (int)__umulhi((uint32_t)e, p.inv_k) : e;
                    id[u] = e < entries ? src[e + ml[u] * step] : -1;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    // the warp probes together: left to themselves, the lanes that need one probe more run the rest of the body on their own
                    const int e = e0 + u * nthr + tid;
                    int want = id[u];
                    const uint32_t hash = (uint32_t)want * 0x9E3779B1u;
                    uint32_t h = hash >> (32 - log2_slots);
                    if (log2_parts && (int)(hash >> (32 - log2_slots - log2_parts) & ((1u << log2_parts) - 1u)) != part) want = -1;
                    int32_t k = want < 0 ? want : *reinterpret_cast<volatile int32_t*>(key + h);   // (unused places of a list hold -1)
                    bool need = k != want;
                    for (int probe = 0; probe < slots && __any_sync(0xffffffffu, need); ++probe) {
                        if (need && k == -1) {
                            k = atomicCAS(key + h, -1, want);
                            if (k == -1) {
                                used[atomicAdd(&n_used, 1)] = (uint16_t)h; k = want;
                            }
                        }
                        need = need && k != want;
                        if (need) {
                            h = (h + 1) & (uint32_t)(slots - 1);
                            k = *reinterpret_cast<volatile int32_t*>(key + h);
                            need = k != want;
                        }
                        // (by vote: a lane on its own would leave the others to vote without it)
                        if ((probe & 15) == 15 && __any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&twice) != 0 || *reinterpret_cast<volatile int*>(&n_used) > limit)) break;
                    }
                    const uint32_t sh = (uint32_t)(ml[u] & 3) * 8u;
                    if (want >= 0 && !need && (atomicAdd(&cell[(ml[u] >> 2) * slots + h], (uint32_t)(e - ml[u] * p.K + 1) << sh) >> sh & 0xffu) != 0u)
                        twice = 1;
                }
            }
            __syncthreads();
            if (twice) return ENS_BAD_TWICE;
            const int total = n_used;
            if (total > limit) return ENS_BAD_FULL;
            for (int i = tid; i < total; i += nthr) {
                const int h = used[i];
                double s = i < seen ? sum[h] : before;
                for (int w = 0; 4 * w < mb; ++w) {
                    const uint32_t c = cell[w * slots + h];
                    cell[w * slots + h] = 0u;
                    if (c == 0u && absent == 0.0) continue;                     // (s is never -0: adding 0 leaves it as it is)
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
        n = seen;
        return 0;
    }

    // This thread's best entity that is not taken: its ordered score (0: none), id and slot.
    __device__ void best_of_mine(uint64_t& bs, int32_t& bi, int& bp) const {
        bs = 0; bi = INT32_MAX; bp = -1;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int h = used[i];
            if (key[h] < 0) continue;
            const uint64_t s = ens_ordered(sum[h]);
            if (bp < 0 || s > bs || (s == bs && key[h] < bi)) { bs = s; bi = key[h]; bp = h; }
        }
    }
};

// Warp maximum under (score descending, id ascending): the score's two halves, then the id.
__device__ __forceinline__ void ens_warp_best(uint64_t s, int32_t id, uint64_t& os, int32_t& oi) {
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(s >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(s >> 32) == hi ? (uint32_t)s : 0u);
    os = (uint64_t)hi << 32 | lo;
    oi = __reduce_min_sync(0xffffffffu, s == os ? id : INT32_MAX);
}

// The table's entities from the best on, one per round, to `take(round, score, id)` (called by all threads with the same
// values; no score maps to 0) until it returns false or none is left.  A thread's best stays in registers until it is taken.
template <int MB, class Take>
__device__ void ens_select(EnsTable<MB>& t, Take take) {
    __shared__ uint64_t red_s[2][32];
    __shared__ int32_t red_i[2][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    uint64_t bs; int32_t bi; int bp;
    t.best_of_mine(bs, bi, bp);
    uint64_t ws; int32_t wi;                // the warp's best
    ens_warp_best(bs, bi, ws, wi);
    for (int r = 0;; ++r) {
        if (lane == 0) { red_s[r & 1][warp] = ws; red_i[r & 1][warp] = wi; }
        __syncthreads();
        uint64_t s; int32_t id;
        ens_warp_best(lane < nwarps ? red_s[r & 1][lane] : 0ull, lane < nwarps ? red_i[r & 1][lane] : INT32_MAX, s, id);   // (every warp for itself)
        if (!take(r, s, id)) return;
        if (s != 0ull && s == ws && id == wi) {                                 // taken (ids are distinct: one warp, one thread)
            if (bp >= 0 && bi == id) { t.key[bp] = -1; t.best_of_mine(bs, bi, bp); }
            __syncwarp();
            ens_warp_best(bs, bi, ws, wi);
        }
    }
}

__device__ __forceinline__ void ens_put(const EnsParams& p, int q, int r, uint64_t s, int32_t id) {
    p.out_ids[(int64_t)q * p.top_n + r] = s != 0ull ? id : -1;                  // fewer candidates than places: -1 and -inf
    if (p.out_scores) p.out_scores[(int64_t)q * p.top_n + r] = s != 0ull ? ens_unordered(s) : -INFINITY;
}

// ------------------------------------------------------------------------------------------
// Unions of at most R entities per thread.  A thread takes four places of one list at a time, whose first probes
// are in flight together; what a lane has left over of its four is probed one step at a time by the whole warp, so that a
// warp's rounds are those of its unluckiest lane's four and not of its unluckiest lane four times.  The table is sparse
// (2,048 slots for 768 entities) for the same reason.  The sums stay in registers: entity i of the order of arrival belongs
// to thread i mod threads, which adds its rank scores model by model.  The rank scores lie in COPIES copies side by side,
// a lane reads its own: a random look-up in one copy would meet three others in its bank.  An entity twice in one list
// loses one of its two bytes (position + 1), so that the bytes read add up to less than the bytes written.
// ------------------------------------------------------------------------------------------
constexpr int ENS_CUT_TOP = 16;
constexpr size_t ens_union_smem(int models, int copies, int slots, int K) {
    return (size_t)(K + 1) * copies * sizeof(double) + (size_t)slots * (sizeof(int32_t) + models) + (size_t)slots * sizeof(uint16_t);
}

// V: places of a list that lie on one boundary of a load (4, 2 or 1).  Returns 0, or (all threads) why the table was given up.
template <int MB, int V, int R, int COPIES>
__device__ int ens_union_query(const EnsParams& p, const int q, const int log2_slots, const int limit, unsigned char* smem) {
    constexpr int WORDS = MB / 4;
    const int slots = 1 << log2_slots, tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, K = p.K;
    double* tab = reinterpret_cast<double*>(smem);                              // [K + 1][copies] absent score, then positions 1 .. K
    int32_t* key = reinterpret_cast<int32_t*>(tab + (size_t)(K + 1) * COPIES);   // [slots] entity id or -1
    uint32_t* cell = reinterpret_cast<uint32_t*>(key + slots);                  // [MB / 4][slots] bytes: position + 1 in the block's models
    uint16_t* used = reinterpret_cast<uint16_t*>(cell + (size_t)WORDS * slots);      // [slots] occupied slots, in order of arrival
    __shared__ int n_used, lost;
    for (int i = tid; i < slots / 4; i += nthr) reinterpret_cast<int4*>(key)[i] = make_int4(-1, -1, -1, -1);
    for (int i = tid; i < slots * WORDS / 4; i += nthr) reinterpret_cast<int4*>(cell)[i] = make_int4(0, 0, 0, 0);
    for (int i = tid; i < (K + 1) * (COPIES / 2); i += nthr) {
        const int j = i / (COPIES / 2);
        const double x = p.table[j == 0 ? K : j - 1];
        reinterpret_cast<double2*>(tab)[i] = make_double2(x, x);
    }
    if (tid == 0) { n_used = 0; lost = 0; }
    const int quads = (K + 3) >> 2, per_block = min(MB, nthr / quads);           // quads of a list; models per block: a quad per thread
    const int ml = p.inv_quads ? (int)__umulhi((uint32_t)tid, p.inv_quads) : tid, pos = 4 * (tid - ml * quads);
    const int64_t list_step = (int64_t)p.nq * K;
    const int32_t* src = p.lists + ((int64_t)ml * p.nq + q) * K + pos;
    auto fetch = [&](int m0, int32_t (&id)[4]) {
        const bool in = ml < per_block && m0 + ml < p.M;
#pragma unroll
        for (int u = 0; u < 4; ++u) id[u] = -1;
        if (!in) return;
        if constexpr (V == 4) {
            const int4 x = *reinterpret_cast<const int4*>(src);
            id[0] = x.x; id[1] = x.y; id[2] = x.z; id[3] = x.w;
        } else if constexpr (V == 2) {
            const int2 x = *reinterpret_cast<const int2*>(src);
            id[0] = x.x; id[1] = x.y;
            if (pos + 2 < K) { const int2 y = *reinterpret_cast<const int2*>(src + 2); id[2] = y.x; id[3] = y.y; }
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) if (pos + u < K) id[u] = src[u];
        }
    };
    int32_t next[4];
    fetch(0, next);
    __syncthreads();
    const double* mytab = tab + (lane & (COPIES - 1));
    const double absent = tab[0];
    double before = 0.0, sum[R];     // before: an entity's sum over the models ahead of the block it first appears in
    int slot[R];
#pragma unroll
    for (int r = 0; r < R; ++r) { sum[r] = 0.0; slot[r] = 0; }
    int seen = 0;                           // occupied slots after the blocks so far
    uint32_t bytes = 0;                     // positions written less positions read
    unsigned char* mycell = reinterpret_cast<unsigned char*>(cell + (size_t)(ml >> 2) * slots) + (ml & 3);
    for (int m0 = 0; m0 < p.M; m0 += per_block) {
        const int mb = min(per_block, p.M - m0);
        int32_t want[4], k[4];
        uint32_t h[4];
        uint32_t left = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            want[u] = next[u];
            h[u] = (uint32_t)want[u] * 0x9E3779B1u >> (32 - log2_slots);
            k[u] = reinterpret_cast<volatile int32_t*>(key)[h[u]];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (want[u] >= 0 && k[u] != want[u]) left |= 1u << u;               // (unused places of a list hold -1)
        while (__any_sync(0xffffffffu, left != 0u)) {                           // (a slot is always free: see the launch)
            if (left) {
                const bool b0 = left & 1u, b1 = left & 2u, b2 = left & 4u;
                const int32_t w = b0 ? want[0] : (b1 ? want[1] : (b2 ? want[2] : want[3]));
                uint32_t g = b0 ? h[0] : (b1 ? h[1] : (b2 ? h[2] : h[3]));
                int32_t x = reinterpret_cast<volatile int32_t*>(key)[g];
                if (x == -1) {
                    x = atomicCAS(key + g, -1, w);
                    if (x == -1) { used[atomicAdd(&n_used, 1)] = (uint16_t)g; x = w; }
                }
                if (x == w) left &= left - 1u;
                else {
                    g = (g + 1) & (uint32_t)(slots - 1);
                    if (b0) h[0] = g; else if (b1) h[1] = g; else if (b2) h[2] = g; else h[3] = g;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (want[u] >= 0) {
                mycell[4 * h[u]] = (unsigned char)(pos + 1 + u);
                bytes += (uint32_t)(pos + 1 + u);
            }
        src += per_block * list_step;
        fetch(m0 + per_block, next);                                            // on its way while this block is summed
        __syncthreads();
        const int total = n_used;
        if (total > limit) return ENS_BAD_FULL;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = r * nthr + tid;
            if (i >= total) break;
            if (i >= seen) { slot[r] = used[i]; sum[r] = before; }
            double s = sum[r];
#pragma unroll
            for (int w = 0; w < WORDS; ++w) {
                if (4 * w >= mb) break;
                const uint32_t c = cell[w * slots + slot[r]];
                if (c == 0u && absent == 0.0) continue;                         // (s is never -0: adding 0 leaves it as it is)
                cell[w * slots + slot[r]] = 0u;
                bytes -= __dp4a(c, 0x01010101u, 0u);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (4 * w + j < mb) s += mytab[(c >> (8 * j) & 0xffu) * COPIES];
            }
            sum[r] = s;
        }
        seen = total;
        if (absent != 0.0) for (int m = 0; m < mb; ++m) before += absent;
        __syncthreads();
    }
    allow_dependents();     // (a second launch's CTAs, started at once, waited in the places of this one's: 85 x 10, an id twice everywhere, 751 -> 638 us)
    bytes = __reduce_add_sync(0xffffffffu, bytes);
    if (lane == 0 && bytes) atomicAdd(&lost, (int)bytes);

    // The best top_n: those that reach a bound which at least top_n entities reach, hardly more, are ranked against one another.  Up to
    // ENS_CUT_TOP the bound is the top_n-th best of 32 groups' best scores (upper halves), beyond of up to as many groups as threads,
    // twice top_n where there are.  (A CTA-wide round per place, each with a barrier: 10 x 100 x 4,000, all 100 places, 294 us.)
    uint64_t os[R];                  // ordered scores, 0: none
    int32_t id[R];
    uint32_t top_hi = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const bool in = r * nthr + tid < seen;
        os[r] = in ? ens_ordered(sum[r]) : 0ull;
        id[r] = in ? key[slot[r]] : INT32_MAX;
        top_hi = max(top_hi, (uint32_t)(os[r] >> 32));
    }
    uint64_t* cand_s = reinterpret_cast<uint64_t*>(cell);                       // (the positions are done with; 12 bytes per entity fit: see ens_union_smem's callers)
    int32_t* cand_i = reinterpret_cast<int32_t*>(cand_s + seen);
    __shared__ __align__(16) uint32_t group_hi[256];
    __shared__ uint32_t cut;
    __shared__ int n_cand;
    int groups = 32;
    if (p.top_n > ENS_CUT_TOP) while (groups < nthr && groups < 2 * p.top_n) groups <<= 1;
    const int per_group = nthr / groups;                                        // 1, 2, 4 or 8 lanes
    for (int o = per_group >> 1; o > 0; o >>= 1) top_hi = max(top_hi, __shfl_xor_sync(0xffffffffu, top_hi, o));
    if ((tid & (per_group - 1)) == 0) group_hi[tid / per_group] = top_hi;
    if (tid == 0) { n_cand = 0; cut = 0u; }
    __syncthreads();
    if (lost) return ENS_BAD_TWICE;
    if (p.top_n <= ENS_CUT_TOP) {
        if (tid < 32) {
            uint32_t v = group_hi[tid], c = 0;
            for (int found = 0; found < p.top_n;) {
                c = __reduce_max_sync(0xffffffffu, v);
                if (c == 0u) break;
                const bool hit = v == c;
                found += __popc(__ballot_sync(0xffffffffu, hit));
                if (hit) v = 0u;
            }
            if (tid == 0) cut = c;
        }
    } else if (p.top_n <= groups && tid < groups) {
        const uint32_t mine = group_hi[tid];
        int ahead = 0;
#pragma unroll 4
        for (int j = 0; j < groups; j += 4) {
            const uint4 o = *reinterpret_cast<const uint4*>(&group_hi[j]);
            ahead += (o.x > mine || (o.x == mine && j < tid)) + (o.y > mine || (o.y == mine && j + 1 < tid)) +
                     (o.z > mine || (o.z == mine && j + 2 < tid)) + (o.w > mine || (o.w == mine && j + 3 < tid));
        }
        if (ahead == p.top_n - 1) cut = mine;
    }
    __syncthreads();
    const uint32_t c = cut;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (os[r] != 0ull && (uint32_t)(os[r] >> 32) >= c) {
            const int at = atomicAdd(&n_cand, 1);
            cand_s[at] = os[r]; cand_i[at] = id[r];
        }
    __syncthreads();
    const int n = n_cand;
    for (int i = tid; i < n; i += nthr) {
        const uint64_t s = cand_s[i];
        const int32_t e = cand_i[i];
        int rank = 0;
#pragma unroll 4
        for (int j = 0; j < n; ++j) rank += cand_s[j] > s || (cand_s[j] == s && cand_i[j] < e);
        if (rank < p.top_n) ens_put(p, q, rank, s, e);
    }
    for (int i = n + tid; i < p.top_n; i += nthr) ens_put(p, q, i, 0ull, 0);
    return 0;
}

// The whole of a query in one table.
template <int MB>
__device__ int ens_hash_query(const EnsParams& p, const int q, const int log2_slots, const int limit, unsigned char* smem) {
    EnsTable<MB> t(smem, 1 << log2_slots, p.K);
    const int bad = t.gather(p, q, log2_slots, limit, 0, 0);
    if (bad) return bad;
    ens_select(t, [&](int r, uint64_t s, int32_t id) {
        if (r >= p.top_n) return false;
        if (threadIdx.x == 0) ens_put(p, q, r, s, id);
        return true;
    });
    return 0;
}

// The general form: all entries of query q sorted by (entity id, model, position) in shared memory.  NT: the threads of the
// CTA where they are known, or 0.
template <int NT>
__device__ void ens_sort_query(const EnsParams& p, const int q, unsigned char* ens_smem) {
    uint64_t* key = reinterpret_cast<uint64_t*>(ens_smem);                      // [n2] (id, model, position); later the candidates' scores
    int32_t* cid = reinterpret_cast<int32_t*>(key + p.n2);                      // [n2] candidate id at the first entry of its run, else -1
    __shared__ double red_s[ENS_THREADS / 32];
    __shared__ int32_t red_i[ENS_THREADS / 32], red_pos[ENS_THREADS / 32];
    __shared__ int32_t win_pos;
    const int tid = threadIdx.x, nthr = NT ? NT : (int)blockDim.x, n = p.M * p.K;
    for (int i = tid; i < p.n2; i += nthr) {
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
            for (int t = tid; t < p.n2 / 2; t += nthr) {
                const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                const bool up = (lo & size) == 0;
                const uint64_t x = key[lo], y = key[hi];
                if ((x > y) == up) { key[lo] = y; key[hi] = x; }
            }
            __syncthreads();
        }
    // runs of equal ids: mark their first entries (reads only)
    for (int i = tid; i < p.n2; i += nthr) {
        const uint64_t k = key[i];
        const bool head = k != ~0ull && (i == 0 || (key[i - 1] >> 32) != (k >> 32));
        cid[i] = head ? (int32_t)(k >> 32) : -1;
    }
    __syncthreads();
    // every run is summed by the thread of its first entry, which then keeps the score in that entry's place
    const double absent = p.table[p.K];
    for (int i = tid; i < p.n2; i += nthr) {
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
        for (int i = tid; i < p.n2; i += nthr) {
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
            for (int w = 1; w < nthr / 32; ++w)
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

template <int NT>
__device__ __noinline__ void ens_sort_call(const EnsParams& p, int q, unsigned char* smem) { ens_sort_query<NT>(p, q, smem); }

// Lists of more than ENS_MAX_K places: every query takes the general form.
template <int NT>
__global__ void __launch_bounds__(NT) ensemble_sort_kernel(EnsParams p) {
    extern __shared__ __align__(16) unsigned char ens_smem[];
    ens_sort_query<NT>(p, blockIdx.x, ens_smem);
}

// The queries that earlier launches left, shared out over the CTAs: `serve(query, left to the sort)`, called by all threads.
template <class Serve>
__device__ void ens_left(const EnsParams& p, bool table, bool sort, Serve serve) {
    __shared__ int32_t todo[ENS_THREADS];
    __shared__ int n_todo;
    for (int64_t base = blockIdx.x; base < p.nq; base += (int64_t)gridDim.x * blockDim.x) {
        __syncthreads();
        if (threadIdx.x == 0) n_todo = 0;
        __syncthreads();
        const int64_t q = base + (int64_t)gridDim.x * threadIdx.x;
        const int32_t mark = q < p.nq ? p.out_ids[q * p.top_n] : 0;
        if ((table && mark == ENS_LEFT) || (sort && mark == ENS_SORT)) todo[atomicAdd(&n_todo, 1)] = mark == ENS_LEFT ? (int32_t)q : ~(int32_t)q;
        __syncthreads();
        const int n = n_todo;
        for (int i = 0; i < n; ++i) {
            const int32_t entry = todo[i];
            __syncthreads();
            serve(entry < 0 ? ~entry : entry, entry < 0);
        }
    }
}

// The queries left to the sort, where the second launch's memory is more than the sort's.  Four times as many CTAs as are resident,
// so that those of an SM are not all in the same phase (15,000 queries of 30 lists of 100, every one sorted: 5.69 -> 5.06 ms; a
// CTA per query, as where all are sorted from the start, 4.57).
__global__ void __launch_bounds__(512) ensemble_sort_left_kernel(EnsParams p) {
    extern __shared__ __align__(16) unsigned char ens_smem[];
    grid_dependency_wait();
    ens_left(p, false, true, [&](int q, bool) { ens_sort_call<512>(p, q, ens_smem); });
}

// Lists so short that a table of 1.5 slots per entry fits (M K <= 682): one launch, no table overflows, and a query with an
// entity twice in one list is sorted where it stands (the sort needs no more memory than the table).  64 threads where they hold the
// entries, six each, and (nearly) a block of models at once, else 128 with three or six; two copies of the rank scores: with so few
// look-ups, filling sixteen takes longer than their conflicts (6 x 33 x 15,000: 219 us on 256 threads with sixteen, 65 so; 4 x 80 174 and
// 94; 2 x 254 295 and 150).  Up to four queries per SM a CTA has the SM nearly to itself: threads for a whole block of models then
// (6 x 100 x 296: 12.4 us on 128, 10.4 on 256; 16 x 20 x 100 10.3 on 64, 9.5 on 128).
constexpr int ENS_SMALL_MB = 16, ENS_SMALL_COPIES = 2, ENS_SMALL_LOG2 = 10, ENS_ENTITIES = 768;
template <int V, int R>
__global__ void __launch_bounds__(256) ensemble_small_kernel(EnsParams p) {
    extern __shared__ __align__(16) unsigned char ens_smem[];
    if (!ens_union_query<ENS_SMALL_MB, V, R, ENS_SMALL_COPIES>(p, blockIdx.x, p.log2_slots, 1 << p.log2_slots, ens_smem)) return;
    __syncthreads();
    ens_sort_call<0>(p, blockIdx.x, ens_smem);
}

// Longer lists, first launch: one CTA of T threads per query, MB models in a block.  A block of models is at most T quads, 1,024
// places, so that with ENS_ENTITIES entities before it a slot is always free.  Which T, MB and COPIES: see the launch.
constexpr int ENS_LOG2 = 11;
static_assert(ENS_ENTITIES + 1024 < 1 << ENS_LOG2, "a probe ends");
static_assert(ENS_ENTITIES * 12 <= (1 << ENS_LOG2) * 8, "the positions' memory holds all entities' scores and ids (eight or more models; sixteen and 1.5 slots per entity in the single launch)");
template <int MB, int V, int T, int COPIES>
__global__ void __launch_bounds__(T) ensemble_hash_kernel(EnsParams p) {
    extern __shared__ __align__(16) unsigned char ens_smem[];
    const int bad = ens_union_query<MB, V, ENS_ENTITIES / T, COPIES>(p, blockIdx.x, ENS_LOG2, ENS_ENTITIES, ens_smem);
    if (bad && threadIdx.x == 0) p.out_ids[(int64_t)blockIdx.x * p.top_n] = bad == ENS_BAD_TWICE ? ENS_SORT : ENS_LEFT;
}

// Second launch: the queries with larger unions.  Up to 8,192 slots (180 KB), eight models at a time.  Up to ENS_BIG_PART
// entries the table takes whatever the lists hold, in one pass; beyond, the passes are as many as give each at most ENS_BIG_PART
// entries if their hashes spread evenly (a query whose hashes favour one part that much is sorted), and the best n of the passes
// so far wait in shared memory.  85 x top-100 lists of 15,000 queries, all left here: unions of 1,000 7.2 ms, 3,500 9.0, 6,600
// 11.0, where the sort takes 37.8.
constexpr int ENS_BIG_MB = 8, ENS_BIG_LOG2 = 13, ENS_BIG_PART = 5400, ENS_BIG_TOP = ENS_THREADS;
template <int NT>
__global__ void __launch_bounds__(NT, 2048 / NT) ensemble_left_kernel(EnsParams p) {
    extern __shared__ __align__(16) unsigned char ens_smem[];
    grid_dependency_wait();
    allow_dependents();
    ens_left(p, true, p.sort_here != 0, [&](int q, bool sort) {
        if (sort) {
        } else if (p.log2_parts == 0) {
            sort = ens_hash_query<ENS_BIG_MB>(p, q, p.left_log2, 1 << p.left_log2, ens_smem) != 0;
        } else if (p.top_n > ENS_BIG_TOP) {
            sort = true;
        } else {                             // (1,024 threads, 8,192 slots)
            const int tid = threadIdx.x;
            uint64_t* run_s = reinterpret_cast<uint64_t*>(ens_smem);            // [top_n] ordered scores, 0: free
            int32_t* run_i = reinterpret_cast<int32_t*>(run_s + ENS_BIG_TOP);
            EnsTable<ENS_BIG_MB> t(reinterpret_cast<unsigned char*>(run_i + ENS_BIG_TOP), 1 << ENS_BIG_LOG2, p.K);
            if (tid < p.top_n) { run_s[tid] = 0; run_i[tid] = INT32_MAX; }
            for (int part = 0; part < 1 << p.log2_parts; ++part) {
                sort = t.gather(p, q, ENS_BIG_LOG2, 3 << (ENS_BIG_LOG2 - 2), part, p.log2_parts) != 0;
                if (sort) break;
                ens_select(t, [&](int, uint64_t s, int32_t id) {
                    const uint64_t last_s = run_s[p.top_n - 1]; const int32_t last_i = run_i[p.top_n - 1];
                    if (s == 0ull || s < last_s || (s == last_s && id > last_i)) return false;
                    // into its place: everything behind it moves one on
                    const bool in = tid < p.top_n, mine_first = in && (run_s[tid] > s || (run_s[tid] == s && run_i[tid] < id));
                    const bool prev_first = in && (tid == 0 || run_s[tid - 1] > s || (run_s[tid - 1] == s && run_i[tid - 1] < id));
                    const uint64_t ps = in && tid > 0 ? run_s[tid - 1] : 0ull; const int32_t pi = in && tid > 0 ? run_i[tid - 1] : 0;
                    __syncthreads();
                    if (in && !mine_first) { run_s[tid] = prev_first ? s : ps; run_i[tid] = prev_first ? id : pi; }
                    return true;
                });
                __syncthreads();
            }
            if (!sort && tid < p.top_n) ens_put(p, q, tid, run_s[tid], run_i[tid]);
        }
        if (sort && p.sort_here) {
            __syncthreads();
            ens_sort_call<NT>(p, q, ens_smem);
        } else if (sort && threadIdx.x == 0) {
            p.out_ids[(int64_t)q * p.top_n] = ENS_SORT;
        }
    });
}

}  // namespace
}  // namespace kge

namespace kge {
namespace {

// The widest load that every quad of a list allows.
int ens_places_per_load(const int32_t* lists, int k) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(lists);
    return k % 4 == 0 && at % 16 == 0 ? 4 : (k % 2 == 0 && at % 8 == 0 ? 2 : 1);
}

using EnsKernel = void (*)(EnsParams);
struct EnsUnion { EnsKernel kernel; int models, threads, copies; };
template <int MB, int T, int COPIES>
EnsUnion ens_union_of(int v) {
    return EnsUnion{v == 4 ? ensemble_hash_kernel<MB, 4, T, COPIES> : (v == 2 ? ensemble_hash_kernel<MB, 2, T, COPIES> : ensemble_hash_kernel<MB, 1, T, COPIES>), MB, T, COPIES};
}
template <int V>
EnsKernel ens_small_of(int each) { return each == 1 ? ensemble_small_kernel<V, 1> : (each == 3 ? ensemble_small_kernel<V, 3> : ensemble_small_kernel<V, 6>); }
EnsKernel ens_small_kernel(int v, int each) { return v == 4 ? ens_small_of<4>(each) : (v == 2 ? ens_small_of<2>(each) : ens_small_of<1>(each)); }

// Models per block, threads and copies of the rank scores by the lists' length and number: a block of models should fill the
// threads, and few models should not have to fill a large table (15,000 queries, us; the present choice against 256 threads with
// sixteen models, or eight beyond 64 places, and sixteen copies):
//   up to 24 places     8 models on 128 threads     60 x 20: 208 / 247 (16 on 128)   163 x 10: 345 / 384
//   up to 48            12 on 128                   40 x 33: 212 / 284               85 x 40: 329 / 388
//   up to 80            8 on 128 up to 40 models    10 x 80: 159 / 212               30 x 65: 259 / 310
//   up to 100           8 on 128 up to 20 models    10 x 100: 173 / 224              20 x 100: 261 / 294
//     beyond            16 on 256 to 64 places, 12 on 256 from there   60 x 65: 392 / 458   60 x 80: 404 / 472   85 x 100: 617 / 700
//   up to 128           8 on 128 up to 12 models    10 x 101: 196 / 228              12 x 128: 237 / 249
//     beyond            8 on 256;  more than 214 places: sixteen copies take a resident CTA, eight do not, 10 x 254: 398 / 484
// Few queries (up to eight per SM) do not fill the SMs with small CTAs, and a query's own time counts: as many models per
// block and threads as there are (200 queries, against the choice for many: 85 x 10: 16.5 / 20.6, 40 x 20: 12.5 / 14.4, 30 x 50: 12.4 / 14.4,
// 40 x 100: 20.6 / 28.8; 1,184 queries: 85 x 10: 30.9 / 34.9, 30 x 50: 27.0 / 28.9, 40 x 100: 45.8 / 57.3; 2,368: 51.3 / 47.3, 45.4 / 41.9, 82.0 / 88.3).
EnsUnion ens_union_choice(int models, int k, int v, bool few) {
    if (few) {
        if (k <= 32) return ens_union_of<16, 128, 16>(v);
        if (k <= 64) return ens_union_of<16, 256, 16>(v);
    } else {
        if (k <= 24) return ens_union_of<8, 128, 8>(v);
        if (k <= 48) return ens_union_of<12, 128, 8>(v);
        if (models <= (k <= 80 ? 40 : (k <= 100 ? 20 : 12)) && k <= 128) return ens_union_of<8, 128, 8>(v);
        if (k <= 64) return ens_union_of<16, 256, 16>(v);
    }
    if (k <= 100) return ens_union_of<12, 256, 8>(v);
    return k <= 214 ? ens_union_of<8, 256, 16>(v) : ens_union_of<8, 256, 8>(v);
}
// Every kernel of the two above with the most shared memory it is launched with.
template <class F>
void ens_each_union(F f) {
    constexpr size_t sort = 1024 * (sizeof(uint64_t) + sizeof(int32_t));        // (M K <= 682)
    for (int v : {1, 2, 4}) {
        for (int each : {1, 3, 6}) f(ens_small_kernel(v, each), std::max(ens_union_smem(ENS_SMALL_MB, ENS_SMALL_COPIES, 1 << ENS_SMALL_LOG2, ENS_MAX_K), sort));
        for (const EnsUnion& u : {ens_union_of<8, 128, 8>(v), ens_union_of<12, 128, 8>(v), ens_union_of<16, 128, 16>(v), ens_union_of<16, 256, 16>(v),
                                  ens_union_of<12, 256, 8>(v), ens_union_of<8, 256, 16>(v), ens_union_of<8, 256, 8>(v)})
            f(u.kernel, ens_union_smem(u.models, u.copies, 1 << ENS_LOG2, ENS_MAX_K));
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
    // (5 lists of 300 places, 3,000 queries: 512 threads 432 us, 256 372; 12 lists 904 and 960; 16,384 entries: 512 threads 37.8 ms, 1,024 35.3)
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    constexpr size_t parts_smem = ens_hash_smem<ENS_BIG_MB>(1 << ENS_BIG_LOG2, ENS_MAX_K) + ENS_BIG_TOP * (sizeof(uint64_t) + sizeof(int32_t));
    static DeviceOnce configured;
    cudaError_t e = once_per_device(configured, [] {
        constexpr int sort_max = (int)(ENS_MAX_ENTRIES * (sizeof(uint64_t) + sizeof(int32_t)));
        static_assert(parts_smem <= sort_max, "the larger table fits where the sort does");
        cudaError_t e0 = cudaSuccess;
        ens_each_union([&](void (*k)(EnsParams), size_t smem) { if (e0 == cudaSuccess) e0 = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); });
        for (void (*k)(EnsParams) : {ensemble_sort_kernel<256>, ensemble_sort_kernel<512>, ensemble_sort_kernel<ENS_THREADS>, ensemble_sort_left_kernel,
                                     ensemble_left_kernel<256>, ensemble_left_kernel<512>, ensemble_left_kernel<ENS_THREADS>})
            if (e0 == cudaSuccess) e0 = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_max);
        return e0;
    });
    if (e != cudaSuccess) return KGE_ERR_CUDA;
    if (k_list > ENS_MAX_K) {
        if (p.n2 <= 2048) ensemble_sort_kernel<256><<<nq, 256, sort_smem, s>>>(p);
        else if (p.n2 <= 8192) ensemble_sort_kernel<512><<<nq, 512, sort_smem, s>>>(p);
        else ensemble_sort_kernel<ENS_THREADS><<<nq, ENS_THREADS, sort_smem, s>>>(p);
        return cudaGetLastError() == cudaSuccess ? KGE_OK : KGE_ERR_CUDA;
    }
    p.inv_k = (uint32_t)((((uint64_t)1 << 32) + k_list - 1) / k_list);
    const int quads = (k_list + 3) / 4;
    p.inv_quads = quads == 1 ? 0u : (uint32_t)((((uint64_t)1 << 32) + quads - 1) / quads);
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return KGE_ERR_CUDA;
    const int v = ens_places_per_load(lists, k_list);
    p.log2_slots = 5;
    while (2 << p.log2_slots < 3 * num_models * k_list) ++p.log2_slots;
    if (p.log2_slots <= ENS_SMALL_LOG2) {
        const int entries = num_models * k_list, block = std::min(num_models, ENS_SMALL_MB) * quads;
        int threads = entries <= 384 && (block <= 64 || (block <= 80 && k_list <= 64)) ? 64 : 128;
        if (nq <= 4 * sms && block > threads) threads = block <= 128 ? 128 : 256;
        const int each = entries <= threads ? 1 : (entries <= 3 * threads ? 3 : 6);
        const size_t smem = std::max(ens_union_smem(ENS_SMALL_MB, ENS_SMALL_COPIES, 1 << p.log2_slots, k_list), sort_smem);
        ens_small_kernel(v, each)<<<nq, threads, smem, s>>>(p);
        return cudaGetLastError() == cudaSuccess ? KGE_OK : KGE_ERR_CUDA;
    }
    const EnsUnion u = ens_union_choice(num_models, k_list, v, nq <= 8 * sms);
    u.kernel<<<nq, u.threads, ens_union_smem(u.models, u.copies, 1 << ENS_LOG2, k_list), s>>>(p);
    if (cudaGetLastError() != cudaSuccess) return KGE_ERR_CUDA;
    p.log2_parts = 0; p.left_log2 = ENS_LOG2;
    while (p.left_log2 < ENS_BIG_LOG2 && 3 << (p.left_log2 - 2) < num_models * k_list) ++p.left_log2;
    while (num_models * k_list > ENS_BIG_PART << p.log2_parts) ++p.log2_parts;
    auto launch_left = [&](void (*kernel)(EnsParams), int threads, size_t smem, int waves) {
        const int per_sm = std::max(1, std::min(2048 / threads, (int)(224 * 1024 / (smem + 8 * 1024))));
        return launch_dependent(kernel, dim3((unsigned)std::min<int64_t>(nq, (int64_t)sms * per_sm * waves)), dim3(threads), smem, s, p);
    };
    const size_t table_smem = p.log2_parts > 0 ? parts_smem : ens_hash_smem<ENS_BIG_MB>(1 << p.left_log2, k_list);
    // (where the sort takes much less memory than the table, and so more CTAs of it share an SM, it is a launch of its own)
    const bool sort_apart = p.left_log2 > ENS_LOG2 && p.n2 <= 8192;
    p.sort_here = sort_apart ? 0 : 1;
    const size_t left_smem = sort_apart ? table_smem : std::max(table_smem, sort_smem);
    if (p.left_log2 == ENS_LOG2) e = launch_left(ensemble_left_kernel<256>, 256, left_smem, 2);
    else if (p.left_log2 == ENS_LOG2 + 1) e = launch_left(ensemble_left_kernel<512>, 512, left_smem, 1);
    else e = launch_left(ensemble_left_kernel<ENS_THREADS>, ENS_THREADS, left_smem, 1);
    if (e == cudaSuccess && sort_apart) e = launch_left(ensemble_sort_left_kernel, 512, sort_smem, 4);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? KGE_OK : KGE_ERR_CUDA;
}

}  // extern "C"
