// Device parts shared by the persistent sweep kernels (k_sweep_tma.cu,
// k_tiles.cu): mask words, mbarriers and bulk copies, the bounded grid barrier,
// and the label rows of the per-lane core.
#pragma once

#include "iso_device.cuh"

namespace {

using namespace isod;

template <int K> struct MaskOf { using T = uint8_t; };
template <> struct MaskOf<16> { using T = uint16_t; };
template <> struct MaskOf<32> { using T = uint32_t; };
template <> struct MaskOf<64> { using T = unsigned long long; };

__device__ __forceinline__ uint32_t sa(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sa(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* b, uint32_t tx) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sa(b)), "r"(tx) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sa(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(sa(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Non-blocking probe of phase `parity` (try_wait may suspend the thread for a
// while; a polling loop that also watches other things must not).
__device__ __forceinline__ bool mbar_test_wait(unsigned long long* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(sa(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, unsigned long long* b) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     sa(dst)),
                 "l"(src), "r"(bytes), "r"(sa(b))
                 : "memory");
}

// Bounded wait for phase `parity` of barrier b.  false = gave up (status set).
__device__ inline bool mbar_wait(unsigned long long* b, uint32_t parity, const SweepParams& p) {
    if (mbar_try_wait(b, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(b, parity)) return true;
        if ((it & 63) == 0) {
            if (*(volatile int32_t*)p.status != kStOk) return false;
            if (global_ns() - t0 > (unsigned long long)p.timeout_ns || it > (1u << 28)) {
                atomicCAS(p.status, kStOk, kStTimeout);
                return false;
            }
        }
    }
}

__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Grid-wide barrier of the whole CTA (the launch is cooperative, so every CTA
// is resident): an arrival counter that the last arriver resets before it
// advances a generation word the others poll.  (A barrier on one ever-growing
// counter, one release-add to arrive and acquire-polling to wait, passed the
// grid-synchronous levels about 70 us sooner on the 18M graph but left the
// chunk phase that follows it 0.6 ms slower, with relaxed polling as well;
// this one is kept.)  Bounded: gives up, recording kStTimeout, after the
// timeout (bar_extra adds arrivals that never come, for the tests).  Returns
// false, the same on every thread of the CTA, if the kernel has failed.
__device__ inline bool grid_sync(const SweepParams& p) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        volatile int32_t* st = p.status;
        volatile uint32_t* gen = p.bar + 1;
        if (*st != kStOk) {
            ok = 0;
        } else {
            const uint32_t g0 = *gen;
            fence_acq_rel_gpu();
            const uint32_t want = gridDim.x + (uint32_t)p.bar_extra;
            if (atomicAdd(p.bar, 1u) + 1u == want) {
                atomicExch(p.bar, 0u);
                fence_acq_rel_gpu();
                atomicAdd(p.bar + 1, 1u);
            } else {
                const unsigned long long t0 = global_ns();
                for (uint32_t it = 0; *gen == g0; ++it) {
                    if ((it & 15) == 15) {
                        if (*st != kStOk) { ok = 0; break; }
                        if (global_ns() - t0 > (unsigned long long)p.timeout_ns || it > (1u << 28)) {
                            atomicCAS(p.status, kStOk, kStTimeout);
                            ok = 0;
                            break;
                        }
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

// Label rows and in-range masks of the core vertices from k_core's lane-major
// output (final, clamped labels).  A thread takes eight lanes of one vertex (all
// of them if K < 8): the threads of a warp read the same lane of 32 neighbouring
// vertices (coalesced), and each writes 32 bytes of its row and the byte of the
// mask word whose bit i is set iff lane i's label is not kInf.
template <int K, int THREADS>
__device__ void core_rows(const SweepParams& p, int tid) {
    constexpr int LPT = K >= 8 ? 8 : K;
    constexpr int TPV = K / LPT;
    const int cn = p.core_n;
    const int blocks = (cn + 31) / 32 * 32;  // vertices, rounded up to whole warps
    for (long long i = (long long)blockIdx.x * THREADS + tid; i < (long long)blocks * TPV; i += (long long)gridDim.x * THREADS) {
        const int v = (int)(i / (32 * TPV)) * 32 + (int)(i & 31), part = (int)(i >> 5) % TPV;
        if (v >= cn) continue;
        const uint32_t* src = p.core_out + (size_t)(part * LPT) * cn + v;
        uint32_t x[LPT], bits = 0;
#pragma unroll
        for (int l = 0; l < LPT; ++l) x[l] = __ldcg(src + (size_t)l * cn);
#pragma unroll
        for (int l = 0; l < LPT; ++l) bits |= (uint32_t)(x[l] != kInf) << l;
        uint32_t* row = p.d + (size_t)v * K + part * LPT;
        if constexpr (LPT >= 4) {
#pragma unroll
            for (int l = 0; l < LPT; l += 4)
                reinterpret_cast<uint4*>(row)[l / 4] = make_uint4(x[l], x[l + 1], x[l + 2], x[l + 3]);
        } else {
            row[0] = x[0];
        }
        static_cast<uint8_t*>(p.mask)[(size_t)v * TPV + part] = (uint8_t)bits;
    }
}

}  // namespace
