// PTX wrappers shared by the tcgen05 kernels: mbarrier, TMA, tcgen05 fences / commit / MMA, operand descriptors.
#pragma once
#include "common.cuh"

namespace {

constexpr long long WAIT_LIMIT_CYCLES = 4000000000ll;   // about two seconds

// ---- PTX wrappers ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Non-blocking test of a phase.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false when the limit expired or another role of this CTA already gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status,
                                          long long limit_cycles = WAIT_LIMIT_CYCLES) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    int spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 255) == 0) {
            if (*abort_flag) return false;
            if (clock64() - t0 > limit_cycles) {
                *abort_flag = 1;
                atomicExch(status, VIASD_EDEVICE);
                return false;
            }
        }
    }
    return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y) : "memory");
}

// The same for data that is read once per pass (weights, the committed K/V): its lines are the first to leave L2
// again.  Without the hint a layer's 0.4 GB of weights push everything else out of the 126 MB L2 - the partials and
// activations the split tiles hand over, and the kernels' own instructions, whose refetch from HBM was a good part
// of every launch's fixed cost.
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "l"(pol) : "memory");
}

// ---- arrival counters in global memory: `arrivals` releases, then `readers` acknowledgements, the last of which leaves the
// counter at zero for the next launch (inc wraps).  None of it returns a value: an atomic that told the last reader to
// clear the counter was a trip to L2 between the last arrival and the first sum of every split tile.
__device__ __forceinline__ void counter_arrive(int *ctr, int arrivals, int readers) {
    asm volatile("red.release.gpu.global.inc.u32 [%0], %1;" ::"l"(ctr), "r"(arrivals + readers - 1) : "memory");
}
__device__ __forceinline__ void counter_ack(int *ctr, int arrivals, int readers) {
    asm volatile("red.relaxed.gpu.global.inc.u32 [%0], %1;" ::"l"(ctr), "r"(arrivals + readers - 1) : "memory");
}
// One thread waits, bounded, and acknowledges.  A wait that gave up acknowledges too, and its caller goes on as if it had
// not: every CTA then takes the same barriers, arrivals and acknowledgements whatever expired, so nobody is left in a barrier
// and the counter comes back to zero (what is computed meanwhile is void, as the status word says).
__device__ __forceinline__ void counter_wait(int *ctr, int arrivals, int readers, volatile int *abort_flag, int *status) {
    auto arrived = [&]() { int v; asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory"); return v; };
    const long long t0 = clock64();
    while (arrived() < arrivals) {
        if (*abort_flag || clock64() - t0 > WAIT_LIMIT_CYCLES) { *abort_flag = 1; atomicExch(status, VIASD_EDEVICE); break; }
    }
    counter_ack(ctr, arrivals, readers);
}

// ---- single-thread instructions of a warp in step -----------------------------------------------
// tcgen05.mma and the TMA instructions take their operands from uniform registers.  The compiler only keeps descriptors and
// addresses there when it can see that the warp is in step and one thread executes them: the branch to the role on a warp
// number that went through a shuffle, the instructions under elect.sync.  Then an MMA issues every 10 cycles; under
// `if (lane == 0)` the operands are moved over each time, 48 - 63 cycles per MMA (N = 16: 49 -> 40 cycles per MMA with A in
// shared memory, 49 -> 11 with A in TMEM; N = 64: 48 -> 47 and 48 -> 33; N = 128: 65 either way, as long as nothing else
// sits between the MMAs).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}
template <typename T>
__device__ __forceinline__ T uniform(T x) { return (T)__shfl_sync(0xffffffffu, x, 0); }

// Zeroes rows [from, to) of a K or V tile that TMA has brought (two halves of 128-byte rows, `half` bytes apart), by a warp, and
// hands them on to the tensor cores.  Keys past the end of a sequence have weight zero, but what a cache holds there
// may never have been written, and 0 x NaN is not 0.
__device__ __forceinline__ void zero_tile_rows(uint32_t tile, uint32_t half, int from, int to, int lane) {
#pragma unroll 1
    for (int i = from * 8 + lane; i < to * 8; i += 32) {
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(tile + (uint32_t)i * 16u), "r"(0) : "memory");
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(tile + half + (uint32_t)i * 16u), "r"(0) : "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
}

// ---- the same for a whole warp in step ---------------------------------------------------------
// Loops that feed TMA and the tensor cores, run by all lanes of their warp with the instruction itself predicated to one
// lane.  Inside an `if (lane == 0)` the compiler keeps addresses, coordinates and descriptors in per-thread registers and
// moves each of them over to the uniform registers these instructions take: about 60 cycles per tcgen05.mma of the pair
// kernel, 500 for a box of four, where a uniform loop takes 300.  (The one-CTA kernel, two boxes per stage, gains nothing.)
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    int spins = 0;
    while (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) {
        if ((++spins & 255) == 0) {
            const bool late = clock64() - t0 > WAIT_LIMIT_CYCLES;
            if (late && (threadIdx.x & 31) == 0) { *abort_flag = 1; atomicExch(status, VIASD_EDEVICE); }
            if (__any_sync(0xffffffffu, late || *abort_flag)) return false;
        }
    }
    return true;
}
__device__ __forceinline__ void mbar_expect_tx_if(uint32_t on, uint32_t bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %0, 0;\n\t"
                 "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%1], %2;\n\t}" ::"r"(on), "r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// K-major operand tile, 128-byte swizzle, rows 128 bytes apart, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}

}  // namespace
