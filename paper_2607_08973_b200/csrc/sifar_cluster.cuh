/*
 * sifar_cluster.cuh - distributed shared memory of a thread-block cluster as the place where the ranks of a chunk
 * meet: addresses, tagged 16-byte slots, asynchronous stores that count themselves on the receiver's mbarrier, and
 * bounded waits.
 *
 * One hop between two CTAs, 128 threads each with a 16-byte unit of their own, measured on B200 (cycles at 1.92 GHz):
 *   tagged slot through the L2 (st_slot / ld_slot)                     632
 *   plain stores, CTA barrier, st.release flag through the L2    1900-2500
 *   tagged slot in the receiver's shared memory                        422
 *   st.async counted by the receiver's mbarrier                        365
 *   plain remote stores, then a remote mbarrier arrive (release)       708
 *
 * 16-byte tagged slots rest on single-copy atomicity of .b128 accesses, here in shared memory as elsewhere in the L2
 * (8.2e8 reads against concurrent remote stores: none torn).
 */
#ifndef SIFAR_CLUSTER_CUH
#define SIFAR_CLUSTER_CUH

#include "sifar_internal.cuh"
#include "sifar_reduce.cuh"

namespace sifar {

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

/* Address of the same shared-memory location in CTA `cta` of the cluster. */
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t cta)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
    return r;
}

/* All threads of all CTAs of the cluster (threads need not be converged). */
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

/* One 16-byte slot into another CTA's shared memory / out of this CTA's own. */
__device__ __forceinline__ void st_cluster_slot(uint32_t addr, uint4 v)
{
    asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%0, %1, %2, %3};\n\tst.relaxed.cluster.shared::cluster.b128 [%4], q;\n\t}"
                 :: "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(addr) : "memory");
}

__device__ __forceinline__ uint4 ld_shared_slot(uint32_t addr)
{
    uint4 v;
    asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.cluster.shared::cta.b128 q, [%4];\n\tmov.b128 {%0, %1, %2, %3}, q;\n\t}"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t ld_shared_tag(uint32_t slot)
{
    uint32_t v;
    asm volatile("ld.relaxed.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(slot + 12u) : "memory");
    return v;
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(mbar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

/* The receiver's own arrival: the phase completes when `bytes` bytes have been stored on top of it. */
__device__ __forceinline__ void mbar_expect(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cta.shared::cta.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes) : "memory");
}

/* Arrival on an mbarrier of any CTA of the cluster; what this thread did before is ordered before it. */
__device__ __forceinline__ void mbar_arrive_remote(uint32_t mbar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" :: "r"(mbar) : "memory");
}

/* 16 bytes into another CTA's shared memory, counted on an mbarrier of that CTA when they have landed. */
__device__ __forceinline__ void st_async_vec(uint32_t addr, uint4 v, uint32_t mbar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 :: "r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(mbar) : "memory");
}

/* One look at a phase, which may last up to a microsecond. */
__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(mbar), "r"(parity), "r"(1000u) : "memory");
    return ok != 0u;
}

/* Bounded wait for a phase.  Records SIFAR_ERR_TIMEOUT when the limit passes and gives up when somebody has failed. */
__device__ __forceinline__ bool mbar_wait_or_fail(uint32_t mbar, uint32_t parity, DevState *st, int *host_status,
                                                  unsigned long long timeout_ns)
{
    Deadline d;
    for (;;) {
        if (mbar_try(mbar, parity)) return true;
        if (d.expired(timeout_ns)) { fail(st, host_status, SIFAR_ERR_TIMEOUT); return false; }
        if ((d.polls % 64u) == 0u && ld_relaxed_u32(&st->status) != 0u) return false;
    }
}

/* Takes `bytes` off what the current phase waits for, as if they had been stored. */
__device__ __forceinline__ void mbar_complete_tx(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" :: "r"(mbar), "r"(bytes) : "memory");
}

/*
 * After a failure: waits until counted stores that are still on their way have landed, so that the CTA may leave.
 * `coming` bytes of the phase have been or will be stored, `expected` were armed (or, `armed` false, none yet).  The
 * phase is brought to exactly what is coming and then completes with the last of it; with everything that was expected
 * coming, or the phase complete already, nothing is changed.  A store takes well below a microsecond, so the limit is
 * there for the loop alone; running into it is counted as one more wait that timed out.
 */
constexpr unsigned long long kDrainLimitNs = 1000000ull;

__device__ __forceinline__ void mbar_drain(uint32_t mbar, uint32_t parity, bool armed, uint32_t expected, uint32_t coming,
                                           DevState *st)
{
    if (armed) {
        if (coming < expected) mbar_complete_tx(mbar, expected - coming);
    } else if (coming) {
        mbar_expect(mbar, coming);
    } else {
        return;
    }
    Deadline d;
    while (!mbar_try(mbar, parity))
        if (d.expired(kDrainLimitNs)) { atomicAdd(&st->stats[kStatTimeouts], 1ull); return; }
}

__device__ __forceinline__ void st_cluster_u32(uint32_t addr, uint32_t v)
{
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}

/* Time limit of a loop that polls shared memory: a poll takes some 30 cycles, 20 ns more in take_box_slots, so the clock is
   read on every 64th (after 1 to 3 us) and the context's status looked at on every 1024th (after 16 to 40 us). */
struct LocalDeadline {
    unsigned long long t0 = 0;
    unsigned polls = 0;
    __device__ __forceinline__ bool gives_up(DevState *st, int *host_status, unsigned long long timeout_ns)
    {
        if ((++polls % 64u) != 1u) return false;
        const unsigned long long now = globaltimer_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > timeout_ns) { fail(st, host_status, SIFAR_ERR_TIMEOUT); return true; }
        return (polls % 1024u) == 1u && polls > 1u && ld_relaxed_u32(&st->status) != 0u;
    }
};

/*
 * Slots of P ranks in this CTA's shared memory, [rank][kBoxStride]: the stride is one slot more than the CTA has
 * threads, so that one lane per rank can look at the same slot of all ranks without bank conflicts.
 */
constexpr int kBoxThreads = 128;
constexpr uint32_t kBoxStride = kBoxThreads + 1;

/*
 * Speculative read of slot threadIdx.x of every rank (all 32 lanes of the warp call): lane r < P first polls the tag of
 * rank r's copy of the warp's last slot, then every lane loads its P slots, and those whose tag is not `e` are loaded
 * again until they are (a sender's warp stores its 32 slots with one instruction, so that is rare).  Polling one word
 * per rank instead of P slots per lane leaves the shared-memory ports to the arriving stores, and the pause between two
 * looks leaves issue slots to the warps that compute (one reader, P = 8, 64 steps: 8 KB 63.9 -> 62.2 us, 32 KB 82.1 ->
 * 79.2; P = 3 fp32 4 KB 51.3 -> 49.1; P = 1 level, 1 us either way by size; a pause of 100 ns, or one in the producers' polls
 * too, is slower).  `reloads` counts looks
 * that found a stale slot.  False (on all lanes): time limit, or somebody has failed.
 */
template <int P>
__device__ __forceinline__ bool take_box_slots(uint4 (&x)[P], uint32_t box, uint32_t e, uint32_t forced, DevState *st,
                                               int *host_status, unsigned long long timeout_ns, unsigned &reloads)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t mine = box + threadIdx.x * 16u;
    bool ok = true;
    if (lane < (uint32_t)P) {
        const uint32_t last = box + (lane * kBoxStride + (threadIdx.x | 31u)) * 16u;
        LocalDeadline d;
        while (ld_shared_tag(last) != e) {
            if (d.gives_up(st, host_status, timeout_ns)) { ok = false; break; }
            __nanosleep(20);
        }
        reloads += d.polls;
    }
    if (!__all_sync(0xFFFFFFFFu, ok)) return false;
    for (uint32_t round = 0;; ++round) {
        uint32_t wrong = 0;
#pragma unroll
        for (int r = 0; r < P; ++r) x[r] = ld_shared_slot(mine + (uint32_t)r * kBoxStride * 16u);
#pragma unroll
        for (int r = 0; r < P; ++r) wrong |= x[r].w ^ e;
        if (wrong) {
            LocalDeadline d;
            for (;;) {
                uint32_t stale = 0;
#pragma unroll
                for (int r = 0; r < P; ++r) stale |= (uint32_t)(!slot_valid(x[r], e)) << r;
                if (stale == 0u) break;
                reloads += __popc(stale);
                if (d.gives_up(st, host_status, timeout_ns)) { ok = false; break; }
#pragma unroll
                for (int r = 0; r < P; ++r)
                    if (stale & (1u << r)) x[r] = ld_shared_slot(mine + (uint32_t)r * kBoxStride * 16u);
            }
        }
        ok = __all_sync(0xFFFFFFFFu, ok);
        /* forced retries (the retry-latency experiment): a read that found every slot valid is made again */
        if (!ok || round == forced) return ok;
        reloads += P;
    }
}

}  /* namespace sifar */
#endif
