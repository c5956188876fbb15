// Isochrone edge emission (Section 3): an arc between u and h is an isochrone
// edge for lane i iff exactly one of them is in range, i.e. iff bit i of mask[u]
// XOR mask[h] is set.  Vertex pairs (emit_pairs.cpp: both arcs of a two-way road at
// once) are visited in BFS order of their owners.  A CTA collects the edges it
// finds in shared memory and takes room in the lists with one atomicAdd per query
// for about a thousand of them.
//
// Then k_sort_gather sorts each lane's ids ascending (bucket sort in shared
// memory, several CTAs per lane) and writes them to the contiguous output at the
// lane's offset; CTA 0 also writes the offsets.
#include "iso_device.cuh"

namespace {

using namespace isod;

template <int K> struct MaskOf { using T = uint8_t; };
template <> struct MaskOf<16> { using T = uint16_t; };
template <> struct MaskOf<32> { using T = uint32_t; };
template <> struct MaskOf<64> { using T = unsigned long long; };

constexpr int kEmitThreads = 256;
constexpr int kEmitBatch = 2;     // rounds of 32 pairs whose loads a warp has in flight together
constexpr int kEmitBuffer = 2048; // edges a CTA collects before it takes room in the lists
constexpr int kSortThreads = 1024;
constexpr int kSortSmem = 16384;  // ids bucketed in shared memory (64 KB): two sorting CTAs fit an SM

// Bound by latency: two dependent loads per pair (head, then its mask: 8 bytes
// anywhere in a few stretches of the mask array).  Two rounds of 32 pairs in flight
// per warp and all the warps an SM holds (64); the appends must not wait for a
// counter each: one atomicAdd per warp, query and round (half a million of them on
// 64 counters in two cache lines) kept the kernel at 0.32 ms however many warps it
// had.  18M vertices, 64 queries (1.2M edges): 0.52 ms arc by arc with those
// atomics, now 0.22 (0.35 GB to move); one query 0.34, now 0.15.
template <int K>
__global__ void __launch_bounds__(kEmitThreads, 8) k_emit(EmitParams p) {
    using MaskT = typename MaskOf<K>::T;
    // bits of lanes that exist: a mask word holds at least 8 bits, and after a
    // failed sweep it may hold anything
    constexpr unsigned long long kLanes = K >= 64 ? ~0ull : ((1ull << K) - 1ull);
    __shared__ int s_id[kEmitBuffer];       // edges found: arc id ...
    __shared__ uint32_t s_to[kEmitBuffer];  // ... and query << 24 | place among the query's
    __shared__ int s_n, s_cnt[K], s_base[K];
    // a failed batch (bad input, upward overflow, timeout) is reported by the
    // host; its masks may be stale, so nothing is emitted
    if (*(volatile const int32_t*)p.status != kStOk) return;
    const MaskT* mask = static_cast<const MaskT*>(p.mask);
    const unsigned lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < K; i += kEmitThreads) s_cnt[i] = 0;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    auto flush = [&]() {  // (the whole CTA)
        for (int i = threadIdx.x; i < K; i += kEmitThreads)
            s_base[i] = s_cnt[i] ? atomicAdd(p.ecnt + i, s_cnt[i]) : 0;
        __syncthreads();
        const int n = min(s_n, kEmitBuffer);
        for (int e = threadIdx.x; e < n; e += kEmitThreads) {
            if (s_to[e] == 0xFFFFFFFFu) continue;  // the buffer ended inside a pair
            const int i = (int)(s_to[e] >> 24), q = s_base[i] + (int)(s_to[e] & 0xFFFFFFu);
            if (q < p.ecap) p.ebuf[(size_t)i * p.ecap + q] = s_id[e];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < K; i += kEmitThreads) s_cnt[i] = 0;
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
    };
    // a CTA takes kEmitThreads consecutive owners at a time, a warp 32 of them; a
    // warp's pairs are one contiguous range
    for (int64_t c0 = (int64_t)blockIdx.x * kEmitThreads; c0 < p.n; c0 += (int64_t)gridDim.x * kEmitThreads) {
        const int u0 = (int)min(c0 + (threadIdx.x & ~31u), (int64_t)p.n);
        const int u = min(u0 + (int)lane, p.n);
        const uint32_t my_off = __ldg(p.off + u);           // start of owner u0+lane's pairs
        const uint32_t a0 = __shfl_sync(0xffffffffu, my_off, 0);
        const uint32_t a1 = __ldg(p.off + min(u0 + 32, p.n));
        const unsigned long long mu_lane =
            u < p.n ? (unsigned long long)mask[__ldg(p.owner + u)] : 0ull;
        // kEmitBatch rounds of 32 pairs at a time: all their heads, then all the
        // heads' masks are in flight together
        for (uint32_t base0 = a0; base0 < a1; base0 += 32 * kEmitBatch) {
            unsigned long long mh[kEmitBatch];
            {
                int32_t hd[kEmitBatch];
#pragma unroll
                for (int r = 0; r < kEmitBatch; ++r) {
                    const uint32_t a = base0 + 32 * r + lane;
                    hd[r] = a < a1 ? __ldg(p.head + a) : -1;
                }
#pragma unroll
                for (int r = 0; r < kEmitBatch; ++r) mh[r] = hd[r] >= 0 ? (unsigned long long)mask[hd[r]] : 0ull;
            }
            unsigned long long left[kEmitBatch] = {};  // queries whose edges found no room in the buffer
            int2 id[kEmitBatch];
#pragma unroll
            for (int r = 0; r < kEmitBatch; ++r) {
                const uint32_t base = base0 + 32 * r;
                if (base >= a1) break;  // warp-uniform
                const uint32_t a = base + lane;
                // owner of pair a: the last lane t whose first pair is <= a
                int lo = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const uint32_t o = __shfl_sync(0xffffffffu, my_off, lo + step);
                    if (lo + step < 32 && o <= a) lo += step;
                }
                const unsigned long long mu = __shfl_sync(0xffffffffu, mu_lane, lo);
                unsigned long long x = a < a1 ? (mu ^ mh[r]) & kLanes : 0ull;
                if (x == 0) continue;
                id[r] = __ldg(p.ids + a);
                const int each = id[r].y >= 0 ? 2 : 1;
                // (a full buffer's counter stands still, so it cannot wrap)
                const bool full = *(volatile int*)&s_n >= kEmitBuffer;
                for (int slot = full ? kEmitBuffer : atomicAdd(&s_n, each * __popcll(x)); x; x &= x - 1, slot += each) {
                    if (slot + each > kEmitBuffer) {
                        if (slot < kEmitBuffer) s_to[slot] = 0xFFFFFFFFu;
                        left[r] = x;
                        break;
                    }
                    const int i = __ffsll((long long)x) - 1;
                    const uint32_t to = (uint32_t)i << 24 | (uint32_t)atomicAdd(&s_cnt[i], each);
                    s_id[slot] = id[r].x;
                    s_to[slot] = to;
                    if (each == 2) {
                        s_id[slot + 1] = id[r].y;
                        s_to[slot + 1] = to + 1;
                    }
                }
            }
            unsigned long long some = 0;
#pragma unroll
            for (int r = 0; r < kEmitBatch; ++r) some |= left[r];
            if (!__any_sync(0xffffffffu, some != 0)) continue;
            // No room left: straight to the lists, the warp's edges of a query together and
            // the queries' counters side by side, two a thread.  (20M edges of 64 queries on
            // 1M vertices, most of them this way: 3.7 ms with an atomicAdd per pair and
            // query, one after another, now 0.26.)
#pragma unroll
            for (int r = 0; r < kEmitBatch; ++r) {
                const unsigned long long x = left[r];
                const bool both = x && id[r].y >= 0;
                const unsigned long long any = (unsigned long long)__reduce_or_sync(0xffffffffu, (uint32_t)(x >> 32)) << 32 |
                                               __reduce_or_sync(0xffffffffu, (uint32_t)x);
                int take[2] = {0, 0};  // edges of queries lane and 32 + lane, then their places
                for (unsigned long long q = any; q; q &= q - 1) {
                    const int i = __ffsll((long long)q) - 1;
                    const bool mine = (x >> i) & 1ull;
                    const int n = __popc(__ballot_sync(0xffffffffu, mine)) + __popc(__ballot_sync(0xffffffffu, mine && both));
                    if ((i & 31) == (int)lane) take[i >> 5] = n;
                }
                if (take[0]) take[0] = atomicAdd(p.ecnt + lane, take[0]);
                if (take[1]) take[1] = atomicAdd(p.ecnt + 32 + lane, take[1]);
                for (unsigned long long q = any; q; q &= q - 1) {
                    const int i = __ffsll((long long)q) - 1;
                    const bool mine = (x >> i) & 1ull;
                    const unsigned before = (1u << lane) - 1u;
                    const int at = __shfl_sync(0xffffffffu, i < 32 ? take[0] : take[1], i & 31) +
                                   __popc(__ballot_sync(0xffffffffu, mine) & before) +
                                   __popc(__ballot_sync(0xffffffffu, mine && both) & before);
                    int32_t* const dst = p.ebuf + (size_t)i * p.ecap;
                    if (mine && at < p.ecap) dst[at] = id[r].x;
                    if (mine && both && at + 1 < p.ecap) dst[at + 1] = id[r].y;
                }
            }
        }
        // The decision is the barrier's own result, so that it is one for the whole CTA: a
        // thread that read s_n after the barrier could see what a faster warp has added in
        // the next round.  (Each thread reads after its own appends, the last to append
        // reads the final count, and the count only grows: some thread's answer is true
        // iff the final count's is.)
        if (__syncthreads_or(*(volatile int*)&s_n > kEmitBuffer / 2)) flush();
    }
    flush();
}

// `parts` CTAs per lane (the fewer lanes, the more).  Ids are distinct and in
// [0, m); fine(id) maps them to [0, 2^14) without ever decreasing (one
// multiplication; below 2^14 ids it is the id itself), its top bits are the part
// and the next ones a bucket of the part.  CTA (lane, part) reads the lane's list
// twice: to count the ids of every part and of its own buckets, and, after a scan,
// to scatter its own ids into their buckets in shared memory.  Small buckets
// (about four ids) are then sorted by one thread each (insertion sort), larger
// ones by a warp or the whole CTA (every id's place is the number of smaller ids
// in its bucket; a thread alone took up to 40 us for 64 ids: one list of 1,006 ids
// in two runs of neighbours among 2M, 45 us, now 16).  The ranking loops' registers
// (48) leave one CTA per SM: held to 32, crowded lists took up to 2.7 times as long
// and spread ones no less.  The parts' sorted lists are consecutive pieces of the lane's.  CTA 0
// also writes the offsets.  A lane one of whose parts would not fit shared memory
// is sorted by its part-0 CTA alone with the list in global memory.
//
// Bound by latency (5 MB of ids): two passes over the longest list.  18M vertices,
// 64 queries (1.2M ids): 0.20 ms with three passes, two 64-bit divisions an id and
// a ten-step scan, now 0.058; one query (15,000 ids) 0.061 with four CTAs, now 0.028.
constexpr int kFineBits = 14;
constexpr int kMaxBuckets = 4096;
constexpr int kSmallBucket = 16;
constexpr int kWarpBucket = 128;
constexpr int kMaxBigBuckets = 256;  // big buckets listed for the whole-CTA ranking
constexpr int kMaxParts = 16;

__device__ __forceinline__ uint32_t fine_of(uint32_t id, uint32_t mult) { return mult ? __umulhi(id, mult) : id; }

__global__ void __launch_bounds__(kSortThreads) k_sort_gather(GatherParams p) {
    extern __shared__ int32_t sbuf[];
    int32_t* s_hist = sbuf + kSortSmem;           // [kMaxBuckets + 1]
    int32_t* s_cur = s_hist + kMaxBuckets + 1;    // [kMaxBuckets]
    __shared__ long long s_off;
    __shared__ int s_pc[kMaxParts], s_warp[kSortThreads / 32], s_nbig, s_big[kMaxBigBuckets];
    const int lane = blockIdx.x >> p.part_bits;
    int part = (int)blockIdx.x & ((1 << p.part_bits) - 1);
    const int tid = threadIdx.x, warp = tid >> 5, wl = tid & 31;
    if (*(volatile const int32_t*)p.status != kStOk) return;  // failed batch: the host reports it
    // list sizes and offsets (at most 64 lanes): two lanes a thread of warp 0
    if (warp == 0) {
        const long long c0 = 2 * wl < p.k ? min(p.ecnt[2 * wl], p.ecap) : 0;
        const long long c1 = 2 * wl + 1 < p.k ? min(p.ecnt[2 * wl + 1], p.ecap) : 0;
        long long sum = c0 + c1;
        for (int o = 1; o < 32; o <<= 1) {
            const long long up = __shfl_up_sync(0xffffffffu, sum, o);
            if (wl >= o) sum += up;
        }
        if (blockIdx.x == 0) {
            if (wl == 0) p.out_off[0] = 0;
            if (2 * wl < p.k) p.out_off[2 * wl + 1] = sum - c1;
            if (2 * wl + 1 < p.k) p.out_off[2 * wl + 2] = sum;
        }
        if (lane / 2 == wl) s_off = lane & 1 ? sum - c1 : sum - c1 - c0;
    }
    if (tid < kMaxParts) s_pc[tid] = 0;
    if (tid == 0) s_nbig = 0;
    if (lane >= p.k) return;
    const int cnt = min(p.ecnt[lane], p.ecap);
    if (cnt == 0) return;
    const int32_t* seg = p.ebuf + (size_t)lane * p.ecap;
    // buckets per part: about four ids each if all of the list lies in one part, which it
    // does where ids follow the map.  Made for lists spread over the parts, buckets of such
    // ids held up to sixteen times as many, and ranking them takes the square: 3,000
    // neighbouring ids of 2M in 64 lists 223 us, now 49; one list on 1M vertices with ids in
    // the order of the map, limit 3,600, 60, now 17; spread ids 16 and 12 as before.
    int lg = 0;
    while (lg < kFineBits - p.part_bits && (1 << lg) < kMaxBuckets && (4 << lg) < cnt) ++lg;
    int pbits = p.part_bits;
    int32_t* B = sbuf;
    int my = 0, below = 0;
    for (int pass = 0;; ++pass) {
        // (second pass: a part is too large, the lane is sorted as one by this CTA)
        const int nb = 1 << lg, shift = kFineBits - pbits - lg;
        for (int i = tid; i < nb; i += kSortThreads) s_hist[i] = 0;
        __syncthreads();
        for (int i0 = tid; i0 < cnt; i0 += 4 * kSortThreads) {
            uint32_t x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = i0 + k * kSortThreads < cnt ? (uint32_t)seg[i0 + k * kSortThreads] : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (i0 + k * kSortThreads >= cnt) break;
                const int f = (int)fine_of(x[k], p.mult) >> shift, q = f >> lg;
                if (q == part) atomicAdd(&s_hist[f & (nb - 1)], 1);
                // the other parts' counts: one atomic per warp and part
                if (pass == 0) {
                    const unsigned peers = __match_any_sync(__activemask(), q);
                    if (wl == __ffs(peers) - 1) atomicAdd(&s_pc[q], __popc(peers));
                }
            }
        }
        __syncthreads();
        if (pass == 1) { my = cnt; below = 0; break; }
        bool whole = false;
        for (int q = 0; q < (1 << pbits); ++q) {
            whole = whole || s_pc[q] > kSortSmem;
            if (q < part) below += s_pc[q];
        }
        my = s_pc[part];
        if (!whole) break;
        if (part != 0) return;
        B = p.tmp + (size_t)lane * p.ecap;
        pbits = 0;
        lg = 12;
        __syncthreads();
    }
    if (my == 0) return;
    const int nb = 1 << lg, shift = kFineBits - pbits - lg;
    int32_t* out = p.out + s_off + below;
    // exclusive scan of the nb counts (nb <= kMaxBuckets, at most four per thread)
    {
        const int per = (nb + kSortThreads - 1) / kSortThreads, b0 = tid * per;
        int sum = 0;
        for (int i = b0; i < min(b0 + per, nb); ++i) sum += s_hist[i];
        int run = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, run, o);
            if (wl >= o) run += up;
        }
        if (wl == 31) s_warp[warp] = run;
        __syncthreads();
        int acc = run - sum;
        for (int w = 0; w < warp; ++w) acc += s_warp[w];
        for (int i = b0; i < min(b0 + per, nb); ++i) {
            const int c = s_hist[i];
            s_hist[i] = acc;
            s_cur[i] = acc;
            acc += c;
        }
        if (tid == 0) s_hist[nb] = my;
    }
    __syncthreads();
    for (int i0 = tid; i0 < cnt; i0 += 4 * kSortThreads) {
        uint32_t x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = i0 + k * kSortThreads < cnt ? (uint32_t)seg[i0 + k * kSortThreads] : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int f = (int)fine_of(x[k], p.mult) >> shift;
            if (i0 + k * kSortThreads < cnt && f >> lg == part) B[atomicAdd(&s_cur[f & (nb - 1)], 1)] = (int32_t)x[k];
        }
    }
    __syncthreads();
    bool more = false;  // a bucket that is not small
    for (int bb = tid; bb < nb; bb += kSortThreads) {
        const int blo = s_hist[bb], bhi = s_hist[bb + 1];
        if (bhi - blo > kSmallBucket) {
            more = true;
            if (bhi - blo > kWarpBucket) {
                const int q = atomicAdd(&s_nbig, 1);
                if (q < kMaxBigBuckets) s_big[q] = bb;
            }
            continue;
        }
        for (int i = blo + 1; i < bhi; ++i) {
            const int32_t x = B[i];
            int j = i - 1;
            while (j >= blo && B[j] > x) { B[j + 1] = B[j]; --j; }
            B[j + 1] = x;
        }
    }
    more = __syncthreads_or(more);
    // sorted buckets go out together (coalesced); the others' places are written over
    for (int i = tid; i < my; i += kSortThreads) out[i] = B[i];
    if (!more) return;
    __syncthreads();
    // buckets of middling size are ranked by a warp each, of the 32 its threads look at
    // (neighbours, which are crowded together, go to different warps)
    for (int b0 = 0; b0 < nb; b0 += kSortThreads) {
        const int bb = b0 + wl * (kSortThreads / 32) + warp;
        const int blo = bb < nb ? s_hist[bb] : 0, c = bb < nb ? s_hist[bb + 1] - blo : 0;
        for (unsigned mid = __ballot_sync(0xffffffffu, c > kSmallBucket && c <= kWarpBucket); mid; mid &= mid - 1) {
            const int lo = __shfl_sync(0xffffffffu, blo, __ffs(mid) - 1);
            const int hi = lo + __shfl_sync(0xffffffffu, c, __ffs(mid) - 1);
            for (int i = lo + wl; i < hi; i += 32) {
                const int32_t x = B[i];
                int r = 0;
                for (int j = lo; j < hi; ++j) r += B[j] < x;
                out[lo + r] = x;
            }
        }
    }
    // big ones by the whole CTA, from the list of them or, if it overflowed, bucket by bucket
    const int nbig = s_nbig;
    for (int t = 0; t < (nbig <= kMaxBigBuckets ? nbig : nb); ++t) {
        const int bb = nbig <= kMaxBigBuckets ? s_big[t] : t;
        const int blo = s_hist[bb], bhi = s_hist[bb + 1];
        if (bhi - blo <= kWarpBucket) continue;
        for (int i = blo + tid; i < bhi; i += kSortThreads) {
            const int32_t x = B[i];
            int r = 0;
            for (int j = blo; j < bhi; ++j) r += B[j] < x;
            out[blo + r] = x;
        }
    }
}

// Labels to the caller's layout (query-major, original vertex order): a CTA takes
// VT consecutive original vertices, reads their label rows (16 bytes a thread,
// whole rows) through shared memory and writes each query's VT labels as one run.
// Bound by HBM: every label read and written once (4 * K * n bytes each way).  A
// thread per vertex writing one label per query at a time, as before, put every
// label into a sector of its own: the call for 64 queries with distances on 1M
// vertices took 2.76 ms, now 0.80.
template <int K>
__global__ void __launch_bounds__(256) k_dist(DistParams p) {
    constexpr int VT = K >= 16 ? 2048 / K : 256;
    constexpr int Q = K >= 4 ? K / 4 : 1;  // pieces of a row: four labels, or the only one
    __shared__ uint32_t t[K][VT + 1];
    for (int64_t o0 = (int64_t)blockIdx.x * VT; o0 < p.n; o0 += (int64_t)gridDim.x * VT) {
        const int nv = (int)min((int64_t)VT, p.n - o0);
        for (int i = threadIdx.x; i < nv * Q; i += 256) {
            const int v = i / Q, q = i % Q;
            const uint32_t* row = p.d + (size_t)__ldg(p.pos + o0 + v) * K;
            if constexpr (K >= 4) {
                const uint4 x = __ldcg(reinterpret_cast<const uint4*>(row) + q);
                t[4 * q][v] = x.x; t[4 * q + 1][v] = x.y; t[4 * q + 2][v] = x.z; t[4 * q + 3][v] = x.w;
            } else {
                t[0][v] = __ldcg(row);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < p.k * VT; i += 256)
            if (i % VT < nv) p.out[(size_t)(i / VT) * p.n + o0 + i % VT] = (int32_t)t[i / VT][i % VT];
        __syncthreads();
    }
}

// Vertices in range (Section 3's other output: the set of vertices in range),
// as one bitset over original vertex ids per query: a warp takes 32
// consecutive original ids, reads each one's in-range mask through its sweep
// position, and for every query i writes the 32-bit word whose bit t is bit i
// of vertex (v0 + t)'s mask (one ballot per query; lane i % 32 stores it).
template <int K>
__global__ void k_range(RangeParams p) {
    using MaskT = typename MaskOf<K>::T;
    const MaskT* mask = static_cast<const MaskT*>(p.mask);
    const int lane = threadIdx.x & 31;
    const int warps = (int)(gridDim.x * blockDim.x) >> 5;
    for (int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); (int64_t)w * 32 < p.n; w += warps) {
        const int v = w * 32 + lane;
        const unsigned long long m = v < p.n ? (unsigned long long)mask[__ldg(p.pos + v)] : 0ull;
        for (int i = 0; i < p.k; ++i) {
            const unsigned word = __ballot_sync(0xffffffffu, (m >> i) & 1ull);
            if (lane == (i & 31)) p.out[(size_t)i * p.words + w] = word;
        }
    }
}

}  // namespace

cudaError_t iso_launch_range(const isod::RangeParams& p, int K, cudaStream_t s) {
    const int grid = 1024;
    switch (K) {
        case 1: k_range<1><<<grid, 256, 0, s>>>(p); break;
        case 4: k_range<4><<<grid, 256, 0, s>>>(p); break;
        case 8: k_range<8><<<grid, 256, 0, s>>>(p); break;
        case 16: k_range<16><<<grid, 256, 0, s>>>(p); break;
        case 32: k_range<32><<<grid, 256, 0, s>>>(p); break;
        case 64: k_range<64><<<grid, 256, 0, s>>>(p); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t iso_launch_emit(const isod::EmitParams& p, int K, int grid, cudaStream_t s) {
    switch (K) {
        case 1: k_emit<1><<<grid, kEmitThreads, 0, s>>>(p); break;
        case 4: k_emit<4><<<grid, kEmitThreads, 0, s>>>(p); break;
        case 8: k_emit<8><<<grid, kEmitThreads, 0, s>>>(p); break;
        case 16: k_emit<16><<<grid, kEmitThreads, 0, s>>>(p); break;
        case 32: k_emit<32><<<grid, kEmitThreads, 0, s>>>(p); break;
        case 64: k_emit<64><<<grid, kEmitThreads, 0, s>>>(p); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t iso_launch_sort_gather(const isod::GatherParams& params, int K, cudaStream_t s) {
    const int smem = (kSortSmem + 2 * kMaxBuckets + 1) * 4;
    static std::atomic<unsigned long long> attr{0};
    if (cudaError_t e = iso_smem_attr_once(k_sort_gather, smem, attr)) return e;
    GatherParams p = params;
    // about 256 CTAs, which two per SM hold at once
    p.part_bits = K >= 64 ? 2 : K >= 32 ? 3 : 4;
    p.mult = p.m > (1 << kFineBits) ? (uint32_t)((1ull << (32 + kFineBits)) / (unsigned long long)p.m) : 0u;
    k_sort_gather<<<K << p.part_bits, kSortThreads, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t iso_launch_dist(const isod::DistParams& p, cudaStream_t s) {
    const int grid = 2048;
    switch (p.K) {
        case 1: k_dist<1><<<grid, 256, 0, s>>>(p); break;
        case 4: k_dist<4><<<grid, 256, 0, s>>>(p); break;
        case 8: k_dist<8><<<grid, 256, 0, s>>>(p); break;
        case 16: k_dist<16><<<grid, 256, 0, s>>>(p); break;
        case 32: k_dist<32><<<grid, 256, 0, s>>>(p); break;
        case 64: k_dist<64><<<grid, 256, 0, s>>>(p); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}
