// Inline-PTX wrappers for the tensor-core kernels (sm_103a): mbarriers,
// bounded waits, TMA tensor loads, tcgen05 MMA / commit / TMEM loads and
// stores, and the shared-memory operand descriptors.  Each wrapper is one
// instruction (or a short fixed sequence) written from the PTX ISA.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <cstdlib>

namespace gbcorr {
namespace tc {

constexpr int kStatusTimeout = 2;   // device status word: a bounded wait gave up


__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// What a wait orders besides the arrivals themselves: memory written by this
// CTA, memory written anywhere in the cluster, or nothing (tcgen05 operations
// on either side of it are ordered by their own fences).
enum WaitSem { kAcquireCta, kAcquireCluster, kRelaxedCluster };

template <WaitSem SEM = kAcquireCta>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
#define GBCORR_TRY_WAIT(sem)                                                              \
    asm volatile(                                                                         \
        "{\n\t.reg .pred p;\n\t"                                                          \
        "mbarrier.try_wait.parity" sem ".shared::cta.b64 p, [%1], %2;\n\t"                \
        "selp.u32 %0, 1, 0, p;\n\t}"                                                      \
        : "=r"(ok)                                                                        \
        : "r"(bar), "r"(parity)                                                           \
        : "memory")
    if (SEM == kAcquireCluster)
        GBCORR_TRY_WAIT(".acquire.cluster");
    else if (SEM == kRelaxedCluster)
        GBCORR_TRY_WAIT(".relaxed.cluster");
    else
        GBCORR_TRY_WAIT("");
#undef GBCORR_TRY_WAIT
    return ok != 0;
}

// The address in CTA `rank` of the cluster of this CTA's shared-memory address.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// Arrive at a barrier of another CTA of the cluster (its cluster_addr), for
// tcgen05 operations that tc_fence_before has ordered before it.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// The same, announcing `bytes` of TMA copies.  It publishes nothing else: the
// copies' own completion on the barrier releases what they wrote.
__device__ __forceinline__ void mbar_expect_tx_cluster(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(bar),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void st_cluster(uint32_t addr, int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Bounded wait on phase `parity` of `bar`.  Returns false on timeout or when
// another role has already given up (the shared abort word is set); on
// timeout it sets the abort word and records kStatusTimeout in `status`.
template <WaitSem SEM = kAcquireCta>
__device__ __forceinline__ bool wait_bar_t(uint32_t bar, uint32_t parity, volatile int* abort_word,
                                           unsigned long long timeout_ns, int* status) {
    if (mbar_try_wait<SEM>(bar, parity)) return true;
    unsigned long long t0 = 0;
    for (uint32_t n = 0;; ++n) {
        if (mbar_try_wait<SEM>(bar, parity)) return true;
        if (*abort_word) return false;
        if ((n & 63) == 63) {
            const unsigned long long now = globaltimer();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > timeout_ns) {
                *abort_word = 1;
                *static_cast<volatile int*>(status) = kStatusTimeout;   // may be host memory
                __threadfence_system();
                return false;
            }
        }
    }
}

// Box (all frames of one k-tile, rows c1 .., channel c2, plane-and-tile c3)
// of the tile-major workspace.  CG 2: the barrier (a cluster_addr) may be the
// other CTA's of the pair.
template <int CG = 1>
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c1, int c2, int c3) {
    if (CG == 1)
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
            "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(0), "r"(c1), "r"(c2), "r"(c3)
            : "memory");
    else
        asm volatile(
            "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
            "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(0), "r"(c1), "r"(c2), "r"(c3)
            : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor of a K-major tile row layout, low word:
// start address and the (unused) leading offset in 16-byte units; adding to
// it moves the start.  High word: 8-row groups 512 bytes apart and the 64-byte
// swizzle (layout type 4 at bits 61-63) for 64-byte rows (FP16 modes), 1024
// and the 128-byte swizzle (2) for 128-byte rows (FP8); descriptor version 1
// at bits 46-47.
__device__ __forceinline__ uint32_t op_desc_lo(uint32_t saddr) { return (saddr & 0x3FFFFu) >> 4 | 1u << 16; }

template <int MODE>
__device__ __forceinline__ uint64_t op_desc(uint32_t lo) {
    constexpr uint32_t hi = MODE == 2 ? 1024u >> 4 | 1u << 14 | 2u << 29 : 512u >> 4 | 1u << 14 | 4u << 29;
    return (uint64_t)hi << 32 | lo;
}

// One lane of a converged warp, the same one each time.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// CG: CTAs that share the MMA (cta_group::1 or ::2, issued by rank 0 of the
// pair; the descriptors hold in both CTAs).
template <int MODE, int CG>
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                    uint32_t accumulate) {
#define GBCORR_MMA(group, kind)                                                          \
    asm volatile(                                                                        \
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"                                \
        "tcgen05.mma.cta_group::" group ".kind::" kind " [%0], %1, %2, %3, p;\n\t}" ::"r"( \
            d_tmem),                                                                     \
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)                              \
        : "memory")
    if (MODE == 2) {
        if (CG == 1)
            GBCORR_MMA("1", "f8f6f4");
        else
            GBCORR_MMA("2", "f8f6f4");
    } else {
        if (CG == 1)
            GBCORR_MMA("1", "f16");
        else
            GBCORR_MMA("2", "f16");
    }
#undef GBCORR_MMA
}

// Arrives at the barrier (CG 2: at this offset in both CTAs of the pair) once
// the MMAs issued so far are done.
template <int CG>
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    if (CG == 1)
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
            : "memory");
    else
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
            " [%0], %1;" ::"r"(bar),
            "h"((uint16_t)3)
            : "memory");
}

__device__ __forceinline__ void tma_store_5d(const CUtensorMap* map, uint32_t src, int c0, int c1,
                                             int c2, int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];" ::"l"(map),
        "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                   "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld_wait() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]),
                   "r"(v[6]), "r"(v[7])
                 : "memory");
}

__device__ __forceinline__ void tmem_st_wait() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// cuTensorMapEncodeTiled from the driver, through the runtime's entry-point
// query (no driver import library is linked); nullptr when there is none.
// Any thread may be the first to ask.
inline PFN_cuTensorMapEncodeTiled_v12000 get_encoder() {
    static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> known{nullptr};
    PFN_cuTensorMapEncodeTiled_v12000 fn = known.load(std::memory_order_acquire);
    if (fn) return fn;
    if (std::getenv("CORR_TEST_NO_TENSOR_MAPS")) return nullptr;      // test hook
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    known.store(fn, std::memory_order_release);
    return fn;
}

}  // namespace tc
}  // namespace gbcorr
