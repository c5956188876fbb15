// PHAST scanning phase (Section 2) for K queries at once, pruned at tau, tile by
// tile out of shared memory.
//
// Same computation as k_sweep_tma.cu: d[v,i] = min(up_i(v), min over downward
// arcs (u,v) of d[u,i] + len(u,v)), 0x7FFFFFFF when that exceeds tau_i; uint32
// sums never wrap (labels <= 0x7FFFFFFF, lengths <= 0x7FFFFFFE).
//
// The plan (tiles.cpp) cuts the vertices below the per-lane core into tiles of
// several levels each.  A persistent CTA takes a tile at a time:
//   - the tile's record (own vertices, arcs, rows it needs) comes by one bulk
//     copy, started while the tile before it is swept;
//   - the label rows of sources outside the tile are copied into shared memory
//     (cp.async, 16 bytes a thread, all of them in flight at once);
//   - the own vertices are swept phase by phase, a CTA barrier after each, a
//     group of TPV threads per vertex with two 16-byte quads of lanes per thread;
//     rows read inside the tile go to shared memory, rows read by other tiles
//     to global memory, and every vertex's in-range mask to global memory.
// Restricted sweeps: a tile that landmark bounds show out of range for every query
// (k_skip.cu) fetches no rows and sweeps nothing.  Tiles are compact, so their bounds
// skip more than those of the chunk schedule's strips: one query with limit 3,600 on
// 4M vertices skips 9,339 to 9,632 of 9,902 tiles (three sources); the call took 0.87 ms
// over chunks, 0.44 now.
// Tiles of one tier are independent; a grid barrier separates the tiers (18M
// vertices: 27 at 64 lanes, 17 at one).  All waits are bounded (status word).
//
// Bound: latency.  A tile of 50 vertices takes a CTA about 5 us, of which the rows
// from outside are a third and five phases the rest (a phase: a serial chain of
// shared-memory reads per four arcs of its largest vertex).  The sweep step (with
// k_core, default core) on 18M vertices, one GB300: 64 lanes 2.44 ms (chunk schedule
// 3.72), 32 lanes 1.66 (2.39), 16 lanes 1.24 (2.03), 8 lanes 1.10 (1.93), 4 lanes 0.90
// (1.34), one lane 0.79 (1.27); 1M: 64 lanes 0.30 (0.48), one lane 0.17 (0.35).
#include "sweep_device.cuh"

namespace {

// A thread's lanes of a row: LPT = 4 consecutive ones, or two quads, `sub` and
// `sub + TPV` of the row's, so that neighbouring threads' 16-byte accesses are
// neighbours.  (K = 32 and 16: two or four vertices share an access of eight
// threads; every other one takes its quads in the opposite order, which spreads
// them over the banks.)  Element i is lane lane_at(i).
template <int LPT> struct Lanes { uint32_t x[LPT]; };

__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

// Byte offsets of the thread's (first and second) quad in a row.
template <int K, int TPV>
struct Place {
    static constexpr int LPT = K / TPV;
    uint32_t o1, o2;
    __device__ __forceinline__ Place(int sub, int lane) {
        const bool flip = LPT == 8 && TPV < 8 && ((lane / TPV) & 1);
        o1 = LPT == 1 ? 0u : 16u * (uint32_t)(sub + (flip ? TPV : 0));
        o2 = K == 64 ? o1 + 128u : 16u * (uint32_t)(sub + (flip ? 0 : TPV));
    }
    __device__ __forceinline__ int lane_at(int i) const { return (int)((i < 4 ? o1 : o2) / 4) + (i & 3); }
};

template <int K, int TPV>
__device__ __forceinline__ Lanes<K / TPV> lds_lanes(uint32_t row, const Place<K, TPV>& at) {
    Lanes<K / TPV> r;
    if constexpr (K / TPV == 1) {
        r.x[0] = lds32(row);
    } else {
        const uint4 v = lds128(row + at.o1);
        r.x[0] = v.x; r.x[1] = v.y; r.x[2] = v.z; r.x[3] = v.w;
        if constexpr (K / TPV == 8) {
            const uint4 u = lds128(row + at.o2);
            r.x[4] = u.x; r.x[5] = u.y; r.x[6] = u.z; r.x[7] = u.w;
        }
    }
    return r;
}

template <int K, int TPV>
__device__ __forceinline__ void st_lanes(uint32_t* row, const Place<K, TPV>& at, const Lanes<K / TPV>& r) {
    if constexpr (K / TPV == 1) {
        *row = r.x[0];
    } else {
        *reinterpret_cast<uint4*>(row + at.o1 / 4) = make_uint4(r.x[0], r.x[1], r.x[2], r.x[3]);
        if constexpr (K / TPV == 8)
            *reinterpret_cast<uint4*>(row + at.o2 / 4) = make_uint4(r.x[4], r.x[5], r.x[6], r.x[7]);
    }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const uint32_t* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t* a) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr int kThreads = 128;
constexpr int kCtasPerSm = 5;     // most that the limits below leave room for

constexpr int kUpRows = 16;       // rows for upward labels (more flagged vertices read theirs in place)
constexpr int kInPlace = kUpRows + 1;

// Dynamic shared memory: two record buffers, the label rows (the tile's, then
// kUpRows more), a byte per own vertex (0: no upward label, 1 + i: in row i of
// the latter, kInPlace: in its global row), 16-byte aligned each.
struct TileSmem {
    int rows_at, flags_at, bytes;
};
// Grid-wide barrier of the CTA: arrivals add up in one counter (zeroed per batch),
// round r is over at (r + 1) * CTAs.  Bounded like grid_sync, and like it false, the
// same on every thread, once the kernel has failed.  Against grid_sync's arrival
// counter and generation word, one atomic round trip less for each of the barriers:
// the sweep step took 0.184 ms instead of 0.193 on 1M vertices (one lane, a core of
// 19,000), 1.23 instead of 1.25 on 18M (16 lanes).
__device__ bool tier_sync(const SweepParams& p, uint32_t& round) {
    __shared__ int s_ok;
    __syncthreads();
    ++round;
    if (threadIdx.x == 0) {
        const uint32_t want = round * (gridDim.x + (uint32_t)p.bar_extra);
        int ok = *(volatile int32_t*)p.status == kStOk;
        if (ok) {
            fence_acq_rel_gpu();
            asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
            const unsigned long long t0 = global_ns();
            for (uint32_t it = 0; ld_relaxed_u32(p.bar) < want; ++it) {
                if ((it & 15) == 15) {
                    if (*(volatile int32_t*)p.status != kStOk) { ok = 0; break; }
                    if (global_ns() - t0 > (unsigned long long)p.timeout_ns || it > (1u << 28)) {
                        atomicCAS(p.status, kStOk, kStTimeout);
                        ok = 0;
                        break;
                    }
                }
            }
            fence_acq_rel_gpu();
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <int K>
__host__ __device__ inline TileSmem tile_smem(const TileLimits& lim) {
    TileSmem s;
    s.rows_at = 2 * lim.blob_bytes;
    s.flags_at = s.rows_at + (((lim.rows + kUpRows) * K * 4 + 15) & ~15);
    s.bytes = s.flags_at + ((lim.blob_bytes / 8 + 15) & ~15);  // (a vertex record has 8 bytes)
    return s;
}

// Arcs a round of the sweep's inner loop.  With eight lanes a thread, the arithmetic
// that spare arcs cost weighs more than the rounds (18M, 64 lanes: 2.51 ms with two,
// 2.57 with four; 16 lanes 1.25 and 1.30); with one or four, the rounds' latency.
__host__ __device__ constexpr int kTileArcs(int K) { return K >= 8 ? 2 : 4; }

template <int K, int TPV>
__global__ void __launch_bounds__(kThreads, kCtasPerSm) k_tiles(SweepParams p) {
    constexpr int LPT = K / TPV;
    constexpr int ARCS = kTileArcs(K);
    static_assert(TPV == (int)sizeof(typename MaskOf<K>::T), "a thread writes one byte of the mask word");
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ unsigned long long full[2];
    __shared__ int s_off[kTileMaxTiers + 1];
    __shared__ int s_up, s_up_v[kUpRows];
    const TileSmem lay = tile_smem<K>(p.tile_lim);
    uint32_t* const rows = reinterpret_cast<uint32_t*>(smem + lay.rows_at);
    uint8_t* const flags = smem + lay.flags_at;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int sub = tid % TPV;
    const Place<K, TPV> at(sub, lane);

    if (p.trace && tid == 0 && blockIdx.x == 0 && p.core_levels == 0)
        p.trace[0] = p.trace[p.L + 1] = (long long)global_ns();
    if (tid == 0) {
        mbar_init(&full[0], 1);
        mbar_init(&full[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    uint32_t tau[LPT];
#pragma unroll
    for (int i = 0; i < LPT; ++i) {
        const int32_t t = p.tau[at.lane_at(i)];
        tau[i] = t < 0 ? 0u : (uint32_t)t;
    }
    for (int i = tid; i <= p.tiers; i += kThreads) s_off[i] = __ldg(p.tile_off + i);
    if (tid == 0) s_up = 0;
    __syncthreads();

    // tiles of this CTA: blockIdx.x, + gridDim.x, ... of every tier.  Each one's
    // record is fetched while the one before it is swept, across tiers too (it
    // holds graph data only).  Thread 0 also reads a tile's place one tile ahead.
    int next_t = 0, next_q = (int)blockIdx.x - (int)gridDim.x;  // the tile to fetch next
    uint2 next_at = make_uint2(0u, 0u);
    bool next_skip = false;  // (restricted sweep) it is out of range for every lane
    auto advance = [&]() {
        next_q += (int)gridDim.x;
        while (next_t < p.tiers && next_q >= s_off[next_t + 1] - s_off[next_t]) {
            ++next_t;
            next_q = (int)blockIdx.x;
        }
        if (next_t < p.tiers) {
            if (tid == 0) next_at = __ldg(p.tile_dir + s_off[next_t] + next_q);
            next_skip = p.skip && __ldg(p.skip + s_off[next_t] + next_q);
        }
    };
    auto fetch = [&](int b) {  // (thread 0)
        mbar_expect_tx(&full[b], next_at.y);
        bulk_load(smem + (size_t)b * p.tile_lim.blob_bytes, p.tile_blob + next_at.x, next_at.y, &full[b]);
    };
    advance();
    int done = 0;            // tiles swept
    int cur_t = next_t;      // tier of tile `done`
    bool cur_skip = next_skip;
    bool in_flight = false;  // thread 0: the copy of its record is on its way
    if (tid == 0 && next_t < p.tiers) { fetch(0); in_flight = true; }
    advance();

    // labels of the per-lane core as rows and masks, complete after the first barrier
    bool ok = true;
    uint32_t round = 0;  // grid barriers passed
    if (p.core_levels > 0) {
        core_rows<K, kThreads>(p, tid);
        if (p.tiers > 0 || p.bar_extra > 0) ok = tier_sync(p, round);
    }
    for (int t = 0; ok && t < p.tiers; ++t) {
        while (cur_t == t) {
            const int b = done & 1;
            // its record is here; every thread of the CTA goes on or none
            if (!__syncthreads_and(mbar_wait(&full[b], (uint32_t)(done >> 1) & 1u, p))) { ok = false; break; }
            ++done;
            in_flight = false;
            const uint32_t* rec = reinterpret_cast<const uint32_t*>(smem + (size_t)b * p.tile_lim.blob_bytes);
            const int n_ext = (int)rec[0], n_own = (int)rec[1], phases = (int)rec[2];
            const uint2* vert = reinterpret_cast<const uint2*>(rec + rec[3]);
            const uint2* arcs = reinterpret_cast<const uint2*>(rec + rec[4]);
            const uint32_t* ext = rec + kTileHeader + phases;
            // rows from outside (final: written before the last grid barrier)
            const bool skip = cur_skip;
            if (skip) {
                // (no rows are needed)
            } else if constexpr (K >= 4) {  // a thread keeps to its piece of the rows
                constexpr int Q = K / 4;
                const uint32_t* const src = p.d + 4 * (tid % Q);
                uint32_t dst = sa(rows) + 16u * (uint32_t)tid;
#pragma unroll 4
                for (int r = tid / Q; r < n_ext; r += kThreads / Q, dst += 16u * kThreads)
                    cp_async16(dst, src + (size_t)ext[r] * K);
            } else {
                for (int i0 = tid; i0 < n_ext; i0 += 4 * kThreads) {  // four loads in flight
                    uint32_t x[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        x[k] = i0 + k * kThreads < n_ext ? __ldcg(p.d + ext[i0 + k * kThreads]) : 0u;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (i0 + k * kThreads < n_ext) rows[i0 + k * kThreads] = x[k];
                }
            }
            // the next tile's record
            if (tid == 0 && next_t < p.tiers) { fetch(b ^ 1); in_flight = true; }
            cur_t = next_t;
            cur_skip = next_skip;
            advance();
            if (skip) {
                // empty masks, and kInf rows where other tiles read them (the bounds exclude
                // upward labels here; a flag is cleared regardless)
                for (int i = tid; i < n_own; i += kThreads) {
                    const int v = (int)(vert[i].x & ~kTileStore);
                    static_cast<typename MaskOf<K>::T*>(p.mask)[v] = 0;
                    if ((vert[i].x & kTileStore) || p.write_all) {
                        uint32_t* const row = p.d + (size_t)v * K;
                        if constexpr (K >= 4) {
#pragma unroll
                            for (int q = 0; q < K / 4; ++q)
                                reinterpret_cast<uint4*>(row)[q] = make_uint4(kInf, kInf, kInf, kInf);
                        } else {
                            *row = kInf;
                        }
                    }
                    if (__ldcg(p.upflag + v)) { p.upflag[v] = 0; p.upmask[v] = 0ull; }
                }
                continue;
            }
            // upward labels of own vertices: a row each, kInf in the lanes whose search did not get there
            bool up = false;
            constexpr int FLAGS = K >= 32 ? 1 : 4;  // flags in flight per thread
            for (int i0 = tid; i0 < n_own; i0 += FLAGS * kThreads) {
                int v[FLAGS], f[FLAGS];
#pragma unroll
                for (int k = 0; k < FLAGS; ++k) {
                    const int i = i0 + k * kThreads;
                    v[k] = i < n_own ? (int)(vert[i].x & ~kTileStore) : -1;
                    f[k] = v[k] >= 0 ? __ldcg(p.upflag + v[k]) : 0;
                }
#pragma unroll
                for (int k = 0; k < FLAGS; ++k) {
                    if (f[k]) {
                        up = true;
                        f[k] = min(atomicAdd(&s_up, 1) + 1, kInPlace);
                        if (f[k] < kInPlace) s_up_v[f[k] - 1] = v[k];
                    }
                    if (v[k] >= 0) flags[i0 + k * kThreads] = (uint8_t)f[k];
                }
            }
            if constexpr (K >= 4) cp_async_wait();
            up = __syncthreads_or(up);
            if (up) {
                constexpr int Q = K >= 4 ? K / 4 : 1;  // pieces of a row: four lanes, or the only one
                for (int i = tid; i < min(s_up, kUpRows) * Q; i += kThreads) {
                    const int v = s_up_v[i / Q], l = 4 * (i % Q);
                    const unsigned long long um = __ldcg(p.upmask + v) >> l;
                    uint32_t* const dst = rows + (p.tile_lim.rows + i / Q) * K + l;
                    const uint32_t* const src = p.d + (size_t)v * K + l;
                    if constexpr (K >= 4) {
                        uint4 x = __ldcg(reinterpret_cast<const uint4*>(src));
                        x.x = um & 1ull ? x.x : kInf;
                        x.y = um & 2ull ? x.y : kInf;
                        x.z = um & 4ull ? x.z : kInf;
                        x.w = um & 8ull ? x.w : kInf;
                        *reinterpret_cast<uint4*>(dst) = x;
                    } else {
                        const uint32_t x = __ldcg(src);
                        *dst = um & 1ull ? x : kInf;
                    }
                }
                __syncthreads();
            }
            // phases: the next one's vertex record is read before the barrier that ends
            // the phase in front of it
            const uint32_t rows_a = sa(rows), arcs_a = sa(arcs);
            int hi = (int)rec[kTileHeader];
            int j = tid / TPV;  // (at most kThreads / TPV vertices a phase)
            uint2 me = vert[j];  // (garbage from the record's later parts where j >= hi)
            uint32_t e = vert[j + 1].y;
            for (int ph = 0; ph < phases; ++ph) {
                if (j - lane / TPV < hi) {  // (uniform over the warp: some vertex is its)
                    const bool valid = j < hi;
                    const int v = (int)(me.x & ~kTileStore);
                    Lanes<LPT> acc;
#pragma unroll
                    for (int i = 0; i < LPT; ++i) acc.x[i] = kInf;
                    // Labels above tau need no clamp here: they only ever give labels above
                    // tau, and acc stays <= kInf, so that sums cannot wrap.
                    const uint32_t end = valid ? arcs_a + 8u * (e & 0xFFFFu) : 0u;
#pragma unroll 1
                    for (uint32_t a = arcs_a + 8u * (me.y & 0xFFFFu); a < end; a += 8u * ARCS) {
                        uint4 q[ARCS / 2];
                        Lanes<LPT> r[ARCS];
#pragma unroll
                        for (int k = 0; k < ARCS / 2; ++k) q[k] = lds128(a + 16u * k);
#pragma unroll
                        for (int k = 0; k < ARCS / 2; ++k) {
                            r[2 * k] = lds_lanes<K, TPV>(rows_a + q[k].x * (K * 4), at);
                            r[2 * k + 1] = lds_lanes<K, TPV>(rows_a + q[k].z * (K * 4), at);
                        }
#pragma unroll
                        for (int k = 0; k < ARCS / 2; ++k) {
#pragma unroll
                            for (int i = 0; i < LPT; ++i) acc.x[i] = __viaddmin_u32(r[2 * k].x[i], q[k].y, acc.x[i]);
#pragma unroll
                            for (int i = 0; i < LPT; ++i) acc.x[i] = __viaddmin_u32(r[2 * k + 1].x[i], q[k].w, acc.x[i]);
                        }
                    }
                    const int f = up && valid ? flags[j] : 0;
                    if (f == kInPlace) {  // only the lanes marked in upmask hold this batch's values
                        const unsigned long long um = __ldcg(p.upmask + v);
#pragma unroll
                        for (int i = 0; i < LPT; ++i) {
                            const int l = at.lane_at(i);
                            if ((um >> l) & 1ull) acc.x[i] = min(acc.x[i], __ldcg(p.d + (size_t)v * K + l));
                        }
                    } else if (f) {
                        const Lanes<LPT> r = lds_lanes<K, TPV>(rows_a + (uint32_t)(p.tile_lim.rows + f - 1) * (K * 4), at);
#pragma unroll
                        for (int i = 0; i < LPT; ++i) acc.x[i] = min(acc.x[i], r.x[i]);
                    }
                    const uint32_t slot = me.y >> 16;
                    if (valid && slot != kTileNoRow) st_lanes<K, TPV>(rows + slot * K, at, acc);
                    // out-of-range bits: the sign of tau - label (both below 2^31), last element first
                    uint32_t bits = 0;
#pragma unroll
                    for (int i = LPT - 1; i >= 0; --i) bits = __funnelshift_l(tau[i] - acc.x[i], bits, 1);
                    if (valid && ((me.x & kTileStore) || p.write_all)) {
                        if (p.write_all) {  // distances are returned: out-of-range labels as kInf
#pragma unroll
                            for (int i = 0; i < LPT; ++i)
                                if (acc.x[i] > tau[i]) acc.x[i] = kInf;
                        }
                        st_lanes<K, TPV>(p.d + (size_t)v * K, at, acc);
                    }
                    // one byte of the mask word per thread: with two quads, a thread and its
                    // neighbour swap a nibble each, the even one gets the lower quads' byte
                    bits = ~bits;
                    int byte = sub;
                    if constexpr (LPT == 8) {
                        if (at.o1 > at.o2) bits = (bits >> 4 & 0xFu) | bits << 4;  // lower quad first
                    }
                    if constexpr (LPT == 8 && TPV > 1) {
                        const uint32_t other = __shfl_xor_sync(0xffffffffu, bits, 1);
                        bits = sub & 1 ? (other >> 4 & 0xFu) | (bits & 0xF0u) : (bits & 0xFu) | (other & 0xFu) << 4;
                        byte = sub / 2 + (sub & 1) * (TPV / 2);
                    }
                    if (valid) static_cast<uint8_t*>(p.mask)[(size_t)v * TPV + byte] = (uint8_t)(bits & ((1u << LPT) - 1u));
                }
                if (ph + 1 < phases) {
                    j = hi + tid / TPV;
                    hi = (int)rec[kTileHeader + ph + 1];
                    me = vert[j];
                    e = vert[j + 1].y;
                }
                __syncthreads();
            }
            if (up) {  // the upward labels are used up
                for (int i = tid; i < n_own; i += kThreads)
                    if (flags[i]) {
                        const int v = (int)(vert[i].x & ~kTileStore);
                        p.upflag[v] = 0;
                        p.upmask[v] = 0ull;
                    }
                if (tid == 0) s_up = 0;
            }
        }
        if (ok && (t + 1 < p.tiers || p.bar_extra > 0)) ok = tier_sync(p, round);
        if (ok && p.trace)
            for (int j = tid; j < p.L; j += kThreads)
                if (p.level_tier[j] == t) atomicMax((unsigned long long*)p.trace + 1 + j, global_ns());
    }
    // a record copy still on its way lands before the CTA exits
    if (tid == 0 && in_flight) mbar_wait(&full[done & 1], (uint32_t)(done >> 1) & 1u, p);
}

constexpr int kMaxSmem = 224 * 1024;  // dynamic shared memory a CTA may ask for (static arrays come on top)

template <int K, int TPV>
int occupancy(const TileLimits& lim) {
    static std::atomic<unsigned long long> attr{0};
    const int bytes = tile_smem<K>(lim).bytes;
    int blocks = 0;
    if (iso_smem_attr_once(k_tiles<K, TPV>, kMaxSmem, attr) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_tiles<K, TPV>, kThreads, bytes) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return blocks;
}

template <int K, int TPV>
cudaError_t launch(const SweepParams& p, int grid, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    if (cudaError_t e = iso_smem_attr_once(k_tiles<K, TPV>, kMaxSmem, attr)) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = (size_t)tile_smem<K>(p.tile_lim).bytes;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_tiles<K, TPV>, p);
}

#define ISO_TILE_CASES(X) X(1, 1) X(4, 1) X(8, 1) X(16, 2) X(32, 4) X(64, 8)

}  // namespace

TileLimits iso_tile_limits(int K) {
    // CTAs per SM: five at 64, 16 and 8 lanes, four at 32 and 4, three at one (by shared
    // memory, 37 to 64 KB each, and at 8 lanes by registers).  A tile costs mostly latency (rows from
    // outside 1.4 us, 0.5 us a phase), so tiles in flight count for more than large
    // tiles, except with one lane, where a tile's own work is small.  18M vertices with a
    // core of 19,000, ms of the whole sweep step: 64 lanes, rows 100 (5 CTAs) 2.58, 120 2.61, 156
    // (4 CTAs) 2.71, 80 (6 CTAs) 2.62; comp 16 2.58, 12 2.58, 8 2.64.  16 lanes: rows
    // 300 1.25, 400 1.27, 220 1.35.  8 lanes: rows 400 1.12, 600 1.14.  One lane: 24 KB
    // records 0.83, 16 KB 0.89, 10 KB 0.90; comp 64 instead of 32 0.367 for 0.373 on 4M,
    // 0.178 for 0.184 on 1M.
    TileLimits l{};
    switch (K) {
        case 64: l.rows = 100; l.blob_bytes = 6144; l.comp = 16; break;
        case 32: l.rows = 200; l.blob_bytes = 8192; l.comp = 16; break;
        case 16: l.rows = 300; l.blob_bytes = 10240; l.comp = 16; break;
        case 8: l.rows = 400; l.blob_bytes = 10240; l.comp = 24; break;
        case 4: l.rows = 1000; l.blob_bytes = 14336; l.comp = 32; break;
        default: l.rows = 2500; l.blob_bytes = 24576; l.comp = 64; break;
    }
    l.arcs = kTileArcs(K);
    l.width = kThreads / (K >= 8 ? K / 8 : 1);
    return l;
}

int iso_tiles_occupancy(int K, const TileLimits& lim) {
#define X(k, t) if (K == k) return occupancy<k, t>(lim);
    ISO_TILE_CASES(X)
#undef X
    return 0;
}

cudaError_t iso_launch_tiles(const isod::SweepParams& p, int K, int grid, cudaStream_t s) {
#define X(k, t) if (K == k) return launch<k, t>(p, grid, s);
    ISO_TILE_CASES(X)
#undef X
    return cudaErrorInvalidValue;
}
