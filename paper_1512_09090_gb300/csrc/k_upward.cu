// Upward search of PHAST (Section 2): from each source s, distances in the
// upward graph G_up = (V, {(u,v) in E u E+ : rank(u) < rank(v)}), pruned at the
// query's limit tau.
//
// One CTA per lane.  Every upward arc ends at a strictly higher CH level, so
// G_up is a DAG and a frontier-based Bellman-Ford over it converges after as
// many rounds as the longest shortest upward path has arcs: each round relaxes
// the out-arcs of every vertex whose label improved in the previous round, a warp
// per vertex, or half a warp where the round has more vertices than warps (upper
// vertices have 11 arcs; half a warp throughout took twice as long for a source of
// thousands of arcs, 8,100: 284 us, now 155, and 7% longer on 4M vertices, 64
// searches: 221 us, now 206; a warp throughout 235).  Labels live in an
// open-addressing hash table in shared memory (vertex -> label) with two bitmaps
// of the vertices queued for the next round (the rounds use them in turn); a
// search space too large for it is redone with the same structures in global
// memory.  Dropping labels above tau is exact because lengths are non-negative:
// every prefix of a path of length <= tau is itself <= tau.
//
// Bound by latency: a chain of rounds (about 90 on 18M vertices).  So a round has
// one load from global memory in its chain -- an arc record says where its head's
// own arcs start, and the last arc of a vertex is marked -- and one CTA barrier.
// With the arc range looked up first and three barriers a round: 0.19 ms for one search
// on 18M vertices, 64 searches 0.47; without, 0.18 and 0.36.  (Five other batches, half
// a warp per vertex throughout: 0.223 and 0.319, now 0.206 and 0.300.)
#include "iso_device.cuh"

namespace {

using namespace isod;

constexpr int kThreads = 1024;
constexpr int kSmemSlots = 16384;  // power of two; at most half of them occupied

constexpr int kSmemFrontier = 3072;  // frontier entries in shared memory (the rest in global memory)
constexpr int kGroup = 16;           // threads per frontier vertex where a warp each is not enough
constexpr int kOverflow = 1 << 28;   // frontier size that says the table overflowed

struct Table {
    int32_t* key;        // vertex or -1
    uint32_t* dist;      // label
    uint32_t* queued[2]; // bitmaps: slot is in the frontier of an even / odd round
    uint2* fr[2];        // frontiers {slot, first arc}: entries below fcap ...
    uint2* more[2];      // ... and those from fcap on, minus fcap
    uint32_t mask;       // slots - 1
    int limit;           // maximum occupied slots, and frontier entries
    int fcap;
};

// key, dist, two bitmaps, two frontiers
__host__ __device__ constexpr size_t table_words(size_t slots, size_t fcap) {
    return slots + slots + 2 * (slots / 32) + 4 * fcap;
}

__device__ __forceinline__ int find_or_insert(const Table& t, int32_t v, int* s_used) {
    uint32_t s = ((uint32_t)v * 0x9E3779B1u) & t.mask;
    for (uint32_t probe = 0; probe <= t.mask; ++probe) {
        const int32_t k = atomicCAS(&t.key[s], -1, v);
        if (k == v) return (int)s;
        if (k == -1) {
            if (atomicAdd(s_used, 1) < t.limit) return (int)s;
            // The search is given up after this round.  The slot is freed again: full to the
            // last one, the table would be walked whole for every further vertex of the round
            // (9 s a batch with a source of 40,000 arcs, now 20 ms, the larger tables included).
            *(volatile int32_t*)&t.key[s] = -1;
            return -1;
        }
        s = (s + 1) & t.mask;
    }
    return -1;
}

__device__ __forceinline__ Table carve(uint32_t* base, uint32_t slots, uint32_t fcap) {
    Table t;
    t.key = (int32_t*)base;
    t.dist = base + slots;
    t.queued[0] = base + 2 * slots;
    t.queued[1] = t.queued[0] + slots / 32;
    t.fr[0] = (uint2*)(t.queued[1] + slots / 32);
    t.fr[1] = t.fr[0] + fcap;
    t.more[0] = t.more[1] = nullptr;
    t.mask = slots - 1;
    t.limit = (int)(slots / 2);
    t.fcap = (int)fcap;
    return t;
}

// Runs the search with table t.  Returns false if the table overflowed.
__device__ bool search(const Table& t, const UpParams& p, int32_t s, uint32_t tau, int lane) {
    __shared__ int s_used, s_nfr[3], s_out, s_core;
    const uint32_t slots = t.mask + 1;
    for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x) {
        t.key[i] = -1;
        t.dist[i] = kInf;
    }
    for (uint32_t i = threadIdx.x; i < 2 * (slots / 32); i += blockDim.x) t.queued[0][i] = 0;
    if (threadIdx.x == 0) { s_used = 0; s_out = 0; s_core = 0; }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int sl = find_or_insert(t, s, &s_used);
        const uint32_t a = __ldg(p.up_off + s);
        t.dist[sl] = 0;
        t.fr[0][0] = make_uint2((uint32_t)sl, a);
        s_nfr[0] = a < __ldg(p.up_off + s + 1) ? 1 : 0;
        s_nfr[1] = 0;
    }
    __syncthreads();
    int nfr;
    for (int r = 0;; ++r) {
        nfr = s_nfr[r % 3];  // (nobody changes it in this round)
        if (nfr == 0 || nfr >= kOverflow) break;
        if (threadIdx.x == 0) s_nfr[(r + 2) % 3] = 0;  // last read in round r - 1
        const int gs = nfr > kThreads / 32 ? kGroup : 32;  // threads per frontier vertex
        const int gl = threadIdx.x & (gs - 1);
        const unsigned peers = gs == 32 ? 0xFFFFFFFFu : 0xFFFFu << (threadIdx.x & 16);  // the group's of the warp
        uint2* cur = t.fr[r & 1];
        uint2* nxt = t.fr[(r + 1) & 1];
        for (int f0 = 0;;) {
            const int n = min(nfr - f0, t.fcap);
            for (int f = threadIdx.x / gs; f < n; f += kThreads / gs) {
                const uint2 me = cur[f];
                const int su = (int)me.x;
                // the vertex leaves its queue; an improvement in this round re-queues it in the other one
                if (gl == 0) atomicAnd(&t.queued[r & 1][su >> 5], ~(1u << (su & 31)));
                const uint32_t du = *((volatile uint32_t*)&t.dist[su]);
                const int4* at = p.up_arc + (me.y + gl);
                int4 next = __ldg(at);  // (the array goes on for a group past its end)
                for (;;) {
                    const int4 arc = next;
                    const unsigned last = __ballot_sync(peers, arc.w != 0) & peers;
                    if (!last) next = __ldg(at += gs);  // (a long list: on its way meanwhile)
                    const bool mine = !last || (threadIdx.x & 31) <= __ffs(last) - 1;
                    const uint32_t nd = du + (uint32_t)arc.y;
                    if (mine && nd <= tau) {
                        const int sx = find_or_insert(t, arc.x, &s_used);
                        if (sx < 0) {
                            atomicMax(&s_nfr[(r + 1) % 3], kOverflow);
                        } else if (nd < atomicMin(&t.dist[sx], nd) && arc.z != -1) {
                            const uint32_t bit = 1u << (sx & 31);
                            if (!(atomicOr(&t.queued[(r + 1) & 1][sx >> 5], bit) & bit)) {
                                const int i = atomicAdd(&s_nfr[(r + 1) % 3], 1);
                                const uint2 x = make_uint2((uint32_t)sx, (uint32_t)arc.z);
                                if (i < t.fcap) nxt[i] = x;
                                else if (i < t.limit) t.more[(r + 1) & 1][i - t.fcap] = x;
                                else atomicMax(&s_nfr[(r + 1) % 3], kOverflow);
                            }
                        }
                    }
                    if (last) break;
                    __syncwarp(peers);
                }
            }
            // (rare: the part of the frontier that the shared one did not hold takes its place)
            f0 += t.fcap;
            if (f0 >= nfr) break;
            __syncthreads();
            for (int f = threadIdx.x; f < min(nfr - f0, t.fcap); f += kThreads) cur[f] = t.more[r & 1][f0 - t.fcap + f];
            __syncthreads();
        }
        __syncthreads();
    }
    if (nfr >= kOverflow) return false;
    if (p.direct) {
        // labels go straight into their row slots (other lanes own the other
        // slots); those of the top core [0, core_n), which the sweep resolves
        // per lane, go to the lane's pair list instead
        int2* core = p.pairs + (size_t)lane * p.cap;
        for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x) {
            const int32_t v = t.key[i];
            if (v >= 0) {
                if (v < p.core_n) {
                    core[atomicAdd(&s_core, 1)] = make_int2(v, (int)t.dist[i]);
                } else {
                    p.d[(size_t)v * p.K + lane] = t.dist[i];
                    atomicOr(p.upmask + v, 1ull << lane);
                    p.upflag[v] = 1;
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) s_out = s_core;
    } else {
        int2* out = p.pairs + (size_t)lane * p.cap;
        for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x) {
            const int32_t v = t.key[i];
            if (v >= 0) out[atomicAdd(&s_out, 1)] = make_int2(v, (int)t.dist[i]);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) p.cnt[lane] = s_out;
    return true;
}

__host__ __device__ constexpr size_t iso_upward_table_words_of(size_t gcap) { return table_words(gcap, gcap / 2); }

__global__ void __launch_bounds__(kThreads) k_upward(UpParams p) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int lane = blockIdx.x;
    const int32_t src = p.src[lane];
    const int32_t tau = p.tau[lane];
    if (src < 0) {                                   // idle lane
        if (threadIdx.x == 0) p.cnt[lane] = 0;
        return;
    }
    if (src >= p.n || tau < 0 || tau > p.tau_max) {
        if (threadIdx.x == 0) { p.cnt[lane] = 0; atomicCAS(p.status, kStOk, kStBadInput); }
        return;
    }
    const int32_t s = p.pos[src];
    uint32_t* base = p.gtab + (size_t)lane * iso_upward_table_words_of(p.gcap);
    // A table in shared memory holds all its vertices as one frontier too: what goes past
    // the shared part lies where the global table would be.  (Source of 7,000 arcs to
    // vertices with arcs of their own: 575 us when such a search was redone in global
    // memory for its frontier, now 189.)  Not where the pairs cannot hold every label.
    const bool fits = (p.direct || p.cap >= kSmemSlots / 2) && p.gcap >= kSmemSlots / 2;
    if (fits) {
        Table t = carve(smem, kSmemSlots, kSmemFrontier);
        t.more[0] = (uint2*)base;
        t.more[1] = t.more[0] + (kSmemSlots / 2 - kSmemFrontier);
        if (search(t, p, s, (uint32_t)tau, lane)) return;
    }
    // Too large for shared memory: the same search on this lane's global table.
    __syncthreads();
    if (!search(carve(base, (uint32_t)p.gcap, (uint32_t)p.gcap / 2), p, s, (uint32_t)tau, lane)) {
        if (threadIdx.x == 0) { p.cnt[lane] = 0; atomicCAS(p.status, kStOk, kStUpOverflow); }
    }
}

}  // namespace

size_t iso_upward_table_words(size_t gcap) { return iso_upward_table_words_of(gcap); }

cudaError_t iso_launch_upward(const isod::UpParams& p, int K, cudaStream_t s) {
    const size_t smem = table_words(kSmemSlots, kSmemFrontier) * 4;  // 180 KB
    static std::atomic<unsigned long long> attr{0};
    if (cudaError_t e = iso_smem_attr_once(k_upward, (int)smem, attr)) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(K);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributePriority;
    at[0].val.priority = iso_high_priority();
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_upward, p);
}
