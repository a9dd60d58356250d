// The Newton evaluations of a solve by the warps of a CTA or of a cluster: the warps' sums
// go to the leader, which takes the step and says whether the solve ends.  pt_kernels.cu
// compiles it for the device; tests/exchange_warps.cpp runs one CTA's warps on the host in
// several orders, with exchanges that never arrive among them.
#pragma once

#include <climits>

#include "pt_internal.h"

namespace pt {

#ifdef __CUDACC__
// mbarrier and cluster-push primitives (PTX).  A push st.async's 16 bytes into
// the same variable of another CTA `rank` of the cluster and completes 16 bytes
// of the transaction count of that CTA's barrier; a CTA's own warps store their
// entries locally and arrive on the barrier; the receiver arms its barrier with
// the bytes it expects from the other CTAs and waits on the phase parity.
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive_expect(unsigned long long* bar, unsigned bytes) {
    asm volatile(
        "{\n\t.reg .b64 st;\n\t"
        "mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_addr(bar)),
        "r"(bytes)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile(
        "{\n\t.reg .b64 st;\n\t"
        "mbarrier.arrive.release.cta.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_test_wait(unsigned long long* bar, unsigned parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void cluster_push16(float* dst, unsigned long long* bar, unsigned rank, float4 v) {
    uint32_t d, b;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(smem_addr(dst)), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(smem_addr(bar)), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(d),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(b)
                 : "memory");
}
#endif

// A CTA gives up waiting for its cluster's Newton sums after this many cycles
// (about 2 s); the kernel then reports PT_ERR_TIMEOUT through its statistics.
constexpr long long kExchangeWaitCycles = 1ll << 32;

constexpr int kGaveUp = 8;  // in ns.done: the wait ran out

// A CTA's place in its cluster (the CTAs that share one item): kp CTAs, and the
// exchanges made so far (equal in every thread of the cluster; nseq < 0 in every thread
// of a CTA that gave up).
struct Team {
    int kp, rank;
    int cseq, nseq;
};

// Evaluations until the leader (warp ld of the CTA's nw; this thread is lane `lane` of warp
// w) ends the solve, at most maxit; returns how many there were, the same in every thread.
// sums() gives the warp's sums in every lane; step(cs, last) takes the step on the entries
// of slot cs and returns 0, or what ns.done is to say where the solve ends (always when
// last).
//
// kClus: every warp pushes its sums into every CTA and only the leader waits for them, so
// that wait is all that keeps the leader behind the other warps' reads of ns.done.  When it
// runs out, the solve therefore ends at the barrier that follows, and later solves make no
// exchange and no evaluation (0 is returned).
template <bool kClus, typename NS, typename Sums, typename Step>
__device__ __forceinline__ int newton_evaluations(int maxit, int w, int lane, int nw, int ld, NS& ns, Team& tm, Sums sums,
                                                  Step step) {
    if (kClus && tm.nseq < 0) return 0;
    int evals = 0;
    for (int it = 0; it < maxit; ++it) {
        const float4 v = sums();
        const int xe = tm.nseq++, cs = kClus ? xe & 1 : 0;
        if constexpr (kClus) {
            // Slot cs is free in every CTA: a warp pushes exchange xe only after its
            // CTA's leader received all of exchange xe - 1, which every CTA pushed
            // after its own leader had read exchange xe - 2 (the last use of cs).
            // Every lane holds the warp's sums: lane r pushes them to CTA r.
            float* slot = &ns.cxr[cs][tm.rank * nw + w][0];
            if (lane == tm.rank) {
                *reinterpret_cast<float4*>(slot) = v;  // this CTA's own copy
                mbar_arrive(&ns.mbx[cs]);
            } else if (lane < tm.kp) {
                cluster_push16(slot, &ns.mbx[cs], (unsigned)lane, v);
            }
            // no block barrier here: only the leader needs the sums
        } else {
            if (lane == 0) *reinterpret_cast<float4*>(&ns.cxr[0][w][0]) = v;
            __syncthreads();
        }
        ++evals;
        if (w == ld) {
            bool gone = false;
            if constexpr (kClus) {
                // wait (bounded) until the slot holds all kp x nw pushes of this exchange
                if (lane == 0) mbar_arrive_expect(&ns.mbx[cs], (unsigned)((tm.kp - 1) * nw * 16));
                bool ok = false;
                const long long tw = clock64();
                while (!ok) {
                    ok = mbar_test_wait(&ns.mbx[cs], (unsigned)(xe >> 1) & 1u);
                    if (!ok && clock64() - tw > kExchangeWaitCycles) break;
                }
                gone = __any_sync(0xffffffffu, !ok);
                if (gone && lane == 0) ns.abort_ = 1;
            }
            const int end = step(cs, gone || it + 1 == maxit);
            if (lane == 0) ns.done = end | (gone ? kGaveUp : 0);
        }
        __syncthreads();
        if (const int end = ns.done) {
            if (kClus && (end & kGaveUp)) tm.nseq = INT_MIN;
            break;
        }
    }
    return evals;
}

}  // namespace pt
