/*
 * sifar_chain_cluster.cu - the persistent decode-step chains of small grids: the CTAs that own one chunk form a
 * thread-block cluster, and the ranks of that chunk meet in its distributed shared memory.
 *
 * A decode payload of 8 KB per rank is six chunks; what a step costs there is not bytes but dependent hops between
 * CTAs, one per arrow:
 *     rank stores its partial -> reader sees it, sums -> next operation takes the result -> ...
 * A hop through the L2 takes 632 cycles with tagged slots and about 2000 with a released flag; into another CTA's
 * shared memory it takes 365-422 (sifar_cluster.cuh).  Chunks do not talk to each other, so a cluster is all that has
 * to be resident together, and the hardware guarantees that: no cooperative launch, and the next run's prologue may
 * start while this one's last step drains (programmatic launch).
 *
 * The protocol is the mode's own, chunk by chunk; where it lives changes:
 *   SPECULATIVE     a slot {12 B, call number} is stored into the reader's shared memory, parity e & 1; the reader
 *                   loads, validates tags, loads stale ones again.
 *   DUALBUF         a plain 16-byte vector is stored into the reader's buffer of parity e & 1; the arrival flags are
 *                   the transaction count of an mbarrier per warp of the reader: it completes when the 32 vectors of
 *                   all P ranks have landed.
 *   BARRIER_ONESHOT one buffer; top barrier: one mbarrier per chunk counts every vector of every rank; bottom
 *                   barrier: every reading warp arrives on the writers' done mbarrier after its loads, and a writer
 *                   waits for all of them before it stores the next partial.
 */
#include <cstdlib>

#include "sifar_internal.cuh"
#ifdef SIFAR_SLOT_S8X2
#error "the decode-step chains are written for the default slot format; the fallback format is built for libsifar only"
#endif
#include "sifar_chain.cuh"
#include "sifar_cluster.cuh"
#include "sifar_gen.cuh"

namespace sifar {

constexpr uint32_t kWarpsPerCta = kChainThreads / 32;
static_assert(kChainThreads == kBoxThreads, "one slot per thread");

__device__ __forceinline__ void gdc_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void gdc_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }

/*
 * How many steps of this run the warps of every CTA of the cluster have made counted stores for, in the receiver's shared
 * memory: as many as a whole run has, unless a warp gave up and said otherwise before it came to the cluster's last barrier.
 */
template <uint32_t SENDERS>
struct Stored { uint32_t steps[SENDERS][kWarpsPerCta]; };

/* Zero tags in `slots` slots of shared memory, mbarriers ready, every CTA of the cluster past this point. */
template <uint32_t SENDERS>
__device__ __forceinline__ void cluster_prologue(uint4 *box, uint32_t slots, unsigned long long (*top)[kWarpsPerCta],
                                                 unsigned long long (*hand)[kWarpsPerCta], unsigned long long *done,
                                                 uint32_t done_count, Stored<SENDERS> &stored, uint32_t steps)
{
    for (uint32_t i = threadIdx.x; i < slots; i += kChainThreads) box[i] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x < SENDERS * kWarpsPerCta) (&stored.steps[0][0])[threadIdx.x] = steps;
    if (threadIdx.x < 2 * kWarpsPerCta) {
        mbar_init(smem_addr(&top[0][0] + threadIdx.x), 1u);
        if (hand) mbar_init(smem_addr(&hand[0][0] + threadIdx.x), 1u);
        if (threadIdx.x == 0) mbar_init(smem_addr(done), done_count);
        mbar_init_fence();
    }
    __syncthreads();
    cluster_sync();
}

/*
 * After the last step.  A store into a CTA that has left would be an error, so nobody leaves before all are done.  Plain
 * remote stores and arrivals have been performed by then; counted ones need not have been.  Where every wait came to
 * its end they have all been waited for; true: somebody gave up, and what is still on its way to this CTA is to be
 * waited for (mbar_drain).  (Whoever gave up has seen the context's status set before it came to the barrier.)
 */
__device__ __forceinline__ bool cluster_epilogue(DevState *st)
{
    __syncwarp();
    cluster_sync();
    return ld_relaxed_u32(&st->status) != 0u;
}

/* Bytes that the warps [w0, w1) of the senders [r0, r1) have stored for step d (512 per warp). */
template <uint32_t SENDERS>
__device__ __forceinline__ uint32_t stored_bytes(const Stored<SENDERS> &stored, uint32_t r0, uint32_t r1, uint32_t w0,
                                                 uint32_t w1, uint32_t d)
{
    uint32_t bytes = 0;
    for (uint32_t r = r0; r < r1; ++r)
        for (uint32_t w = w0; w < w1; ++w) bytes += (stored.steps[r][w] > d) ? 512u : 0u;
    return bytes;
}

/*
 * The partials that may still be on their way to a reader after a failure (one lane of a warp calls).  The warp has armed
 * `armed` phases: the last of them may be incomplete, and stores of the step after it may have been made (its writers
 * wait for this reader's result or for one of the barriers before they go further).  Both barriers: one mbarrier for the
 * whole chunk, which warp 0 arms.
 */
template <bool BARRIER, uint32_t SENDERS>
__device__ __forceinline__ void drain_partials(unsigned long long (*top)[kWarpsPerCta], const Stored<SENDERS> &stored,
                                               uint32_t r0, uint32_t r1, uint32_t warp, uint32_t warps, uint32_t armed,
                                               uint32_t e0, uint32_t steps, DevState *st)
{
    if (BARRIER && warp != 0u) return;
    for (uint32_t d = armed ? armed - 1u : 0u; d <= armed && d < steps; ++d) {
        if constexpr (BARRIER)
            mbar_drain(smem_addr(&top[0][0]), d & 1u, d < armed, (r1 - r0) * warps * 512u,
                       stored_bytes(stored, r0, r1, 0u, warps, d), st);
        else
            mbar_drain(smem_addr(&top[(e0 + 1u + d) & 1u][warp]), (d >> 1) & 1u, d < armed, (r1 - r0) * 512u,
                       stored_bytes(stored, r0, r1, warp, warp + 1u, d), st);
    }
}

template <int DT, int P, int MODE, bool TRACE>
__global__ void __launch_bounds__(kChainThreads, 6) k_chain_cluster(const PersistArgs a)
{
    constexpr bool no_ar = (MODE == kModeNoAllreduce);
    constexpr bool spec = (MODE == SIFAR_SPECULATIVE);
    constexpr bool barrier = (MODE == SIFAR_BARRIER_ONESHOT);
    constexpr bool slot_units = spec || no_ar;                        /* 12-byte units with a tag, else 16-byte vectors */
    constexpr int NW = slot_units ? 3 : 4;
    constexpr int NE = NW * ((DT == SIFAR_BF16) ? 2 : 1);
    constexpr uint32_t kRoles = no_ar ? P : P + 1;
    constexpr uint32_t kBoxSlots = (2 * P * kBoxStride > 2 * kChainThreads) ? 2 * P * kBoxStride : 2 * kChainThreads;
    /* the reader's box: [parity][rank][kBoxStride] partials; a producer's box: [parity][thread] results */
    __shared__ __align__(16) uint4 s_box[kBoxSlots];
    __shared__ unsigned long long s_top[2][kWarpsPerCta], s_hand[2][kWarpsPerCta], s_done;
    __shared__ Stored<kRoles> s_stored;                               /* by role: results of the reader, partials of the ranks */
    __shared__ int s_last;

    DevState *st = a.st;
    const uint32_t role = cluster_rank();
    const uint32_t chunk = blockIdx.x / kRoles;
    const bool is_reader = !no_ar && role == 0u;
    const uint32_t rank = no_ar ? role : role - 1u;                   /* of a producer */
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const size_t n = (size_t)a.n;
    /* whole warps of units, as in k_chain: units past the last element carry zeros, rows have room for them */
    const size_t nunits = ((n + NE - 1) / NE + 31) / 32 * 32;
    const size_t n_io = nunits * NE;
    const size_t unit0 = (size_t)chunk * kChainThreads;
    const uint32_t units = (nunits - unit0 < (size_t)kChainThreads) ? (uint32_t)(nunits - unit0) : (uint32_t)kChainThreads;
    const bool active = threadIdx.x < units;                          /* warp-uniform */
    const size_t u = unit0 + threadIdx.x;
    const uint32_t box = smem_addr(s_box);
    cluster_prologue(s_box, kBoxSlots, s_top, s_hand, &s_done, units / 32u, s_stored, a.steps);
    constexpr bool counted = !slot_units;                             /* stores counted on mbarriers */
    uint32_t gave_up = a.steps;                                       /* the step this warp did not get through */
    unsigned reloads = 0;
    /* results are stamped by the warps that publish them (rank 0's without all-reduce): the warps of a chunk are
       pipelines of their own, a chunk is complete with the last of them */
    const bool stamper = lane == 0u && (no_ar ? rank == 0u : is_reader);
    unsigned long long *my_stamps = a.stamps + ((size_t)chunk * kWarpsPerCta + warp) * (a.steps + 1u);
    const bool tracer = TRACE && a.trace != nullptr && chunk == 0u;
#define SIFAR_TRACE(slot, who) do { if (TRACE && tracer && (who)) a.trace[(size_t)s * kTraceSlots + (slot)] = globaltimer_ns(); } while (0)

    /* the same shared memory in the other CTAs: a producer's partials go to the reader, results to the producers */
    const uint32_t top_at = smem_addr(s_top) - box, hand_at = smem_addr(s_hand) - box, done_at = smem_addr(&s_done) - box;
    uint32_t peer[P];
#pragma unroll
    for (uint32_t q = 0; q < (uint32_t)P; ++q) peer[q] = cluster_map(box, no_ar ? role : is_reader ? q + 1u : 0u);
    Gen g;
    float z[NE];
    if (!is_reader && active) {
        /* the seeded half of the first step needs nothing from anybody */
        const uint32_t t = a.e0 + 1u - a.base_epoch;
        g = make_gen(a.w, rank, t);
        unit_noise<DT, NW>(g, t == 1u, u * NE, z);
    }
    gdc_wait();                                                       /* the run before this one is over */
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        /* what this launch really runs with, for sifar_chain_geometry */
        uint32_t cluster_ctas;
        asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cluster_ctas));
        a.cs->seen[0] = 1u; a.cs->seen[1] = cluster_ctas; a.cs->seen[2] = (spec || MODE == SIFAR_DUALBUF) ? 1u : 0u;
    }
    if (stamper) my_stamps[0] = globaltimer_ns();

    for (uint32_t s = 0; s < a.steps && active; ++s) {
        const uint32_t e = a.e0 + 1u + s;
        const uint32_t t = e - a.base_epoch;
        const uint32_t p = e & 1u;
        const bool last = (s + 1u == a.steps);
        /* results of a run's last step cross to the next run in global memory */
        const size_t ho_sets = no_ar ? (size_t)P : 1u, ho_mine = no_ar ? (size_t)rank : 0u;
        uint4 *ho_cur = a.handoff + ((size_t)p * ho_sets + ho_mine) * a.handoff_stride;
        const uint4 *ho_prev = a.handoff + ((size_t)(p ^ 1u) * ho_sets + ho_mine) * a.handoff_stride;
        if (last) gdc_launch_dependents();
        bool ok = true;
        const unsigned before = reloads;
        if (is_reader) {
            /* ---------------- the pulling side ---------------- */
            SIFAR_TRACE(0, threadIdx.x == 0);
            const uint32_t in = box + (barrier ? 0u : p) * P * kBoxStride * 16u;
            uint4 x[P];
            if constexpr (spec) {
                ok = take_box_slots<P>(x, in, e, a.poll.forced, st, a.host_status, a.timeout_ns, reloads);
            } else {
                if constexpr (barrier) {
                    if (threadIdx.x == 0) mbar_expect(smem_addr(&s_top[0][0]), P * units * 16u);
                    ok = mbar_wait_or_fail(smem_addr(&s_top[0][0]), s & 1u, st, a.host_status, a.timeout_ns);
                } else {
                    if (lane == 0u) mbar_expect(smem_addr(&s_top[p][warp]), P * 512u);
                    ok = mbar_wait_or_fail(smem_addr(&s_top[p][warp]), (s >> 1) & 1u, st, a.host_status, a.timeout_ns);
                }
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (ok) {
#pragma unroll
                    for (int r = 0; r < P; ++r) x[r] = ld_shared_slot(in + (r * kBoxStride + threadIdx.x) * 16u);
                }
            }
            if (!ok) { gave_up = s; break; }
            SIFAR_TRACE(1, threadIdx.x == 0);
            SIFAR_TRACE(38 + warp, spec && lane == 0u);
            if constexpr (barrier) {
                /* bottom barrier, reader side: this warp has read its share of the single buffer */
                __syncwarp();
                if (!last && lane < (uint32_t)P) mbar_arrive_remote(cluster_map(box, lane + 1u) + done_at);
                SIFAR_TRACE(28, threadIdx.x == 0);
            }
            const uint4 v = sum_vec<DT, P>(x, !slot_units);
            SIFAR_TRACE(2, threadIdx.x == 0);
            SIFAR_TRACE(3, threadIdx.x == 0);
            /* to the next producers (the critical path of the chain), then into the caller's ring */
            if (!last) {
                const uint32_t out = (p * kChainThreads + threadIdx.x) * 16u;
#pragma unroll
                for (uint32_t q = 0; q < (uint32_t)P; ++q) {
                    if constexpr (spec) st_cluster_slot(peer[q] + out, make_uint4(v.x, v.y, v.z, e));
                    else st_async_vec(peer[q] + out, v, peer[q] + hand_at + (p * kWarpsPerCta + warp) * 8u);
                }
            } else if (!barrier) {
                handoff_store<NW>(ho_cur, u, v, e);
            }
            char *row = a.ring + (size_t)((t - 1u) % a.ring_len) * a.ring_stride;
            if constexpr (slot_units) store_slot_result<DT>(row, u, n_io, v);
            else store_vec_result<DT>(row, u, n_io, v);
            if (spec && __any_sync(0xFFFFFFFFu, reloads != before) && lane == 0u) st_relaxed_u32(&a.retry_steps[s], 1u);
            if (TRACE && spec && tracer && threadIdx.x == 0) a.trace[(size_t)s * kTraceSlots + 29] = reloads - before;
        } else {
            /* ---------------- rank `rank`'s next operation ---------------- */
            const bool first = (t == 1u);
            uint32_t pw[NW], w[NW];
#pragma unroll
            for (int j = 0; j < NW; ++j) pw[j] = 0u;
            if (s > 0u) {
                const uint32_t mine = box + ((p ^ 1u) * kChainThreads + threadIdx.x) * 16u;
                uint4 v;
                if constexpr (slot_units) {
                    LocalDeadline d;
                    for (;;) {
                        v = ld_shared_slot(mine);
                        if (slot_valid(v, e - 1u)) break;
                        if (d.gives_up(st, a.host_status, a.timeout_ns)) { ok = false; break; }
                    }
                } else {
                    const uint32_t bar = smem_addr(&s_hand[p ^ 1u][warp]);
                    if (lane == 0u) mbar_expect(bar, 512u);
                    ok = mbar_wait_or_fail(bar, ((s - 1u) >> 1) & 1u, st, a.host_status, a.timeout_ns);
                    /* bottom barrier, writer side: the chunk's readers are done with the single buffer */
                    if (barrier && ok)
                        ok = mbar_wait_or_fail(smem_addr(&s_done), (s - 1u) & 1u, st, a.host_status, a.timeout_ns);
                    v = ld_shared_slot(mine);
                }
                pw[0] = v.x; pw[1] = v.y; pw[2] = v.z;
                if (NW == 4) pw[NW - 1] = v.w;
            } else if (!first) {
                if constexpr (barrier) {
                    const char *prev = a.ring + (size_t)((t + a.ring_len - 2u) % a.ring_len) * a.ring_stride;
                    const uint4 v = ld_slot(reinterpret_cast<const uint4 *>(prev) + u);
                    pw[0] = v.x; pw[1] = v.y; pw[2] = v.z; pw[NW - 1] = v.w;
                } else {
                    ok = handoff_wait<NW>(ho_prev, u, e - 1u, pw, st, a.host_status, a.timeout_ns);
                }
            }
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) { gave_up = s; break; }
            SIFAR_TRACE(4 + 3 * rank, threadIdx.x == 0);
            if (a.w.delay_max_ns != 0u) spin_ns(gen_delay_ns(a.w, rank, t));      /* seeded skew */
            unit_apply<DT, NW>(g, first, pw, u * NE, n, z, w);
            if constexpr (no_ar) {
                /* to itself: the next step of this thread */
                if (!last) st_cluster_slot(peer[0] + (p * kChainThreads + threadIdx.x) * 16u, make_uint4(w[0], w[1], w[2], e));
                else handoff_store<3>(ho_cur, u, make_uint4(w[0], w[1], w[2], 0u), e);
            } else {
                const uint32_t to = peer[0] + (((barrier ? 0u : p) * P + rank) * kBoxStride + threadIdx.x) * 16u;
                if constexpr (spec) st_cluster_slot(to, make_uint4(w[0], w[1], w[2], e));
                else st_async_vec(to, make_uint4(w[0], w[1], w[2], w[NW - 1]),
                                  peer[0] + top_at + (barrier ? 0u : (p * kWarpsPerCta + warp) * 8u));
            }
            SIFAR_TRACE(5 + 3 * rank, threadIdx.x == 0);
            SIFAR_TRACE(6 + 3 * rank, !slot_units && threadIdx.x == 0);
            SIFAR_TRACE(42 + warp, rank == 0u && lane == 0u);
            if (!last) {
                gen_step(g, t + 1u);
                unit_noise<DT, NW>(g, false, u * NE, z);
                /* here, while the partial is on its way, not below the next wait */
#pragma unroll
                for (int k = 0; k < NE; ++k) asm volatile("" : "+f"(z[k]));
            }
        }
        if (stamper) my_stamps[s + 1u] = globaltimer_ns();
    }
#undef SIFAR_TRACE
    /* A warp that gave up in step s has stored for the s steps before it; the reader has armed step s as well, a
       producer the results of the s steps before it.  A whole run hands over all results but the last. */
    if (counted && gave_up != a.steps && lane < (is_reader ? (uint32_t)P : 1u))
        st_cluster_u32(cluster_map(smem_addr(&s_stored.steps[role][warp]), is_reader ? lane + 1u : 0u), gave_up);
    const bool failed = cluster_epilogue(st);
    if (counted && failed && active && lane == 0u) {
        if (is_reader) {
            drain_partials<barrier>(s_top, s_stored, 1u, kRoles, warp, units / 32u, gave_up == a.steps ? gave_up : gave_up + 1u,
                                    a.e0, a.steps, st);
        } else {
            const uint32_t armed = gave_up == a.steps ? a.steps - 1u : gave_up;
            for (uint32_t d = armed ? armed - 1u : 0u; d <= armed && d + 1u < a.steps; ++d)
                mbar_drain(smem_addr(&s_hand[(a.e0 + 1u + d) & 1u][warp]), (d >> 1) & 1u, d < armed, 512u,
                           stored_bytes(s_stored, 0u, 1u, warp, warp + 1u, d), st);
        }
    }
    /* leave: mis-speculation counters, then the last CTA out publishes the call number */
    const unsigned warp_reloads = __reduce_add_sync(0xFFFFFFFFu, reloads);
    if (warp_reloads && lane == 0u) atomicAdd(&st->stats[kStatSlotReloads], (unsigned long long)warp_reloads);
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t left = atom_add_acq_rel_u32(&a.cs->exit_count, 1u) + 1u;
        s_last = (left == a.exit_base + gridDim.x && !no_ar && ld_relaxed_u32(&st->status) == 0u);
    }
    __syncthreads();
    if (s_last) {
        if constexpr (spec) {
            unsigned long long part = 0;
            for (uint32_t s = threadIdx.x; s < a.steps; s += kChainThreads) {
                part += ld_relaxed_u32(&a.retry_steps[s]);
                st_relaxed_u32(&a.retry_steps[s], 0u);
            }
            if (part) atomicAdd(&st->stats[kStatCallsWithRetry], part);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            atomicAdd(&st->stats[kStatCalls], (unsigned long long)a.steps);
            st_release_u32(&st->epoch, a.e0 + a.steps);
        }
    }
}

/*
 * The chain with P readers in the same way: every rank stores its partial into the shared memory of all P CTAs of the
 * chunk and reduces what has landed in its own.  The seeded half of the next operation is computed while the partials
 * are on their way.
 */
template <int DT, int P, int MODE>
__global__ void __launch_bounds__(kChainThreads, 6) k_sym_cluster(const SymArgs a)
{
    constexpr bool no_ar = (MODE == kModeNoAllreduce);
    constexpr bool spec = (MODE == SIFAR_SPECULATIVE);
    constexpr bool barrier = (MODE == SIFAR_BARRIER_ONESHOT);
    constexpr int NW = spec ? 3 : 4;
    constexpr int NE = NW * ((DT == SIFAR_BF16) ? 2 : 1);
    constexpr uint32_t kBoxSlots = (barrier ? 1 : 2) * P * kBoxStride;
    __shared__ __align__(16) uint4 s_box[kBoxSlots];                  /* [parity][rank][kBoxStride] */
    __shared__ unsigned long long s_top[2][kWarpsPerCta], s_done;
    __shared__ Stored<P> s_stored;
    __shared__ int s_last;

    DevState *st = a.st;
    const uint32_t rank = cluster_rank();
    const uint32_t chunk = blockIdx.x / (uint32_t)P;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const size_t n = (size_t)a.n;
    const size_t nunits = ((n + NE - 1) / NE + 31) / 32 * 32;
    const size_t n_io = nunits * NE;
    const size_t unit0 = (size_t)chunk * kChainThreads;
    const uint32_t units = (nunits - unit0 < (size_t)kChainThreads) ? (uint32_t)(nunits - unit0) : (uint32_t)kChainThreads;
    const bool active = threadIdx.x < units;
    const size_t u = unit0 + threadIdx.x;
    const uint32_t box = smem_addr(s_box);
    char *my_ring = a.rings + (size_t)rank * a.ring_len * a.ring_stride;
    cluster_prologue(s_box, kBoxSlots, s_top, nullptr, &s_done, (uint32_t)P * (units / 32u), s_stored, a.steps);
    constexpr bool counted = !spec && !no_ar;                         /* stores counted on mbarriers */
    uint32_t stored = a.steps, armed = a.steps;                       /* steps that this warp has stored, waited for */
    const bool stamper = lane == 0u;
    unsigned long long *my_stamps = a.stamps + (((size_t)rank * a.C + chunk) * kWarpsPerCta + warp) * (a.steps + 1u);
    const uint32_t top_at = smem_addr(s_top) - box, done_at = smem_addr(&s_done) - box;
    uint32_t peer[P];                                                 /* the readers, not everybody the same one first */
#pragma unroll
    for (uint32_t j = 0; j < (uint32_t)P; ++j) peer[j] = cluster_map(box, (rank + 1u + j) % (uint32_t)P);
    unsigned reloads = 0;
    uint32_t prevw[NW];                                               /* this thread's unit of the previous result */
#pragma unroll
    for (int j = 0; j < NW; ++j) prevw[j] = 0u;
    Gen g;
    float z[NE];
    const uint32_t t0 = a.e0 + 1u - a.base_epoch;
    if (active) {
        g = make_gen(a.w, rank, t0);
        unit_noise<DT, NW>(g, t0 == 1u, u * NE, z);
    }
    gdc_wait();
    if (stamper) my_stamps[0] = globaltimer_ns();
    if (active && t0 != 1u) {
        /* the run before left it in the rank's own row (without all-reduce: in the rank's buffer) */
        const char *prev = no_ar ? a.plain + ((size_t)(a.e0 & 1u) * P + rank) * a.plain_stride
                                 : my_ring + (size_t)((t0 + a.ring_len - 2u) % a.ring_len) * a.ring_stride;
        const uint32_t *p32 = reinterpret_cast<const uint32_t *>(prev) + u * NW;
#pragma unroll
        for (int j = 0; j < NW; ++j) prevw[j] = ld_relaxed_u32(p32 + j);
    }

    for (uint32_t s = 0; s < a.steps && active; ++s) {
        const uint32_t e = a.e0 + 1u + s;
        const uint32_t t = e - a.base_epoch;
        const uint32_t p = e & 1u;
        const bool last = (s + 1u == a.steps);
        if (last) gdc_launch_dependents();
        bool ok = true;
        if constexpr (barrier) {
            /* bottom barrier, writer side: all P readers are done with the single buffer (Section 3.1, phase 3) */
            if (s > 0u) ok = mbar_wait_or_fail(smem_addr(&s_done), (s - 1u) & 1u, st, a.host_status, a.timeout_ns);
            if (!__all_sync(0xFFFFFFFFu, ok)) { stored = armed = s; break; }
        }
        if (a.w.delay_max_ns != 0u) spin_ns(gen_delay_ns(a.w, rank, t));          /* seeded skew between the ranks */
        /* ---- the rank's operation, stored for every reader ---- */
        uint32_t w[NW];
        unit_apply<DT, NW>(g, t == 1u, prevw, u * NE, n, z, w);
        if constexpr (no_ar) {
#pragma unroll
            for (int j = 0; j < NW; ++j) prevw[j] = w[j];
            if (last) st_slot(reinterpret_cast<uint4 *>(a.plain + ((size_t)p * P + rank) * a.plain_stride) + u,
                              make_uint4(w[0], w[1], w[2], w[NW - 1]));
        } else {
            const uint32_t to = (((barrier ? 0u : p) * P + rank) * kBoxStride + threadIdx.x) * 16u;
            const uint32_t bar = top_at + (barrier ? 0u : (p * kWarpsPerCta + warp) * 8u);
#pragma unroll
            for (uint32_t j = 0; j < (uint32_t)P; ++j) {
                if constexpr (spec) st_cluster_slot(peer[j] + to, make_uint4(w[0], w[1], w[2], e));
                else st_async_vec(peer[j] + to, make_uint4(w[0], w[1], w[2], w[NW - 1]), peer[j] + bar);
            }
        }
        if (!last) {
            gen_step(g, t + 1u);
            unit_noise<DT, NW>(g, false, u * NE, z);
#pragma unroll
            for (int k = 0; k < NE; ++k) asm volatile("" : "+f"(z[k]));
        }
        /* ---- pull what all P ranks have stored and reduce in rank order ---- */
        if constexpr (!no_ar) {
            const uint32_t in = box + (barrier ? 0u : p) * P * kBoxStride * 16u;
            const unsigned before = reloads;
            uint4 x[P];
            if constexpr (spec) {
                ok = take_box_slots<P>(x, in, e, a.poll.forced, st, a.host_status, a.timeout_ns, reloads);
            } else {
                if constexpr (barrier) {
                    if (threadIdx.x == 0) mbar_expect(smem_addr(&s_top[0][0]), P * units * 16u);
                    ok = mbar_wait_or_fail(smem_addr(&s_top[0][0]), s & 1u, st, a.host_status, a.timeout_ns);
                } else {
                    if (lane == 0u) mbar_expect(smem_addr(&s_top[p][warp]), P * 512u);
                    ok = mbar_wait_or_fail(smem_addr(&s_top[p][warp]), (s >> 1) & 1u, st, a.host_status, a.timeout_ns);
                }
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (ok) {
#pragma unroll
                    for (int r = 0; r < P; ++r) x[r] = ld_shared_slot(in + (r * kBoxStride + threadIdx.x) * 16u);
                }
            }
            if (!ok) { stored = armed = s + 1u; break; }
            if constexpr (barrier) {
                /* bottom barrier, reader side: this warp's loads of the chunk have returned */
                __syncwarp();
                if (!last && lane < (uint32_t)P) mbar_arrive_remote(cluster_map(box, lane) + done_at);
            }
            const uint4 o = sum_vec<DT, P>(x, !spec);
            prevw[0] = o.x; prevw[1] = o.y; prevw[2] = o.z;
            if (NW == 4) prevw[NW - 1] = o.w;
            char *row = my_ring + (size_t)((t - 1u) % a.ring_len) * a.ring_stride;
            if constexpr (spec) store_slot_result<DT>(row, u, n_io, o);
            else store_vec_result<DT>(row, u, n_io, o);
            /* a rank mis-speculated in this step if any of its threads had to load a slot again */
            if (spec && __any_sync(0xFFFFFFFFu, reloads != before) && lane == 0u)
                st_relaxed_u32(&a.retry_marks[(size_t)rank * a.steps + s], 1u);
        }
        if (stamper) my_stamps[s + 1u] = globaltimer_ns();
    }
    if (counted && stored != a.steps && lane < (uint32_t)P)
        st_cluster_u32(cluster_map(smem_addr(&s_stored.steps[rank][warp]), lane), stored);
    const bool failed = cluster_epilogue(st);
    if (counted && failed && active && lane == 0u)
        drain_partials<barrier>(s_top, s_stored, 0u, (uint32_t)P, warp, units / 32u, armed, a.e0, a.steps, st);
    /* leave: statistics, then the last CTA out books the run and publishes the call number */
    const unsigned warp_reloads = __reduce_add_sync(0xFFFFFFFFu, reloads);
    if (warp_reloads && lane == 0u) atomicAdd(&st->stats[kStatSlotReloads], (unsigned long long)warp_reloads);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const uint32_t left = atom_add_acq_rel_u32(&a.cs->exit_count, 1u) + 1u;
        s_last = (left == a.exit_base + gridDim.x && !no_ar && ld_relaxed_u32(&st->status) == 0u);
    }
    __syncthreads();
    if (s_last) book_sym_run<P>(a, spec);
}

/* ------------------------------------------------------------------------ */
/* host side                                                                 */
/* ------------------------------------------------------------------------ */
static cudaLaunchConfig_t cluster_config(cudaLaunchAttribute *attr, int cluster, size_t clusters, int threads, cudaStream_t stream)
{
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * (size_t)cluster));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <int DT, int P, bool TRACE>
static const void *chain_cluster_p(int mode)
{
    switch (mode) {
    case SIFAR_BARRIER_ONESHOT: return (const void *)k_chain_cluster<DT, P, SIFAR_BARRIER_ONESHOT, TRACE>;
    case SIFAR_DUALBUF:         return (const void *)k_chain_cluster<DT, P, SIFAR_DUALBUF, TRACE>;
    case SIFAR_SPECULATIVE:     return (const void *)k_chain_cluster<DT, P, SIFAR_SPECULATIVE, TRACE>;
    default:                    return (const void *)k_chain_cluster<DT, P, kModeNoAllreduce, false>;
    }
}

template <int DT, int P>
static const void *sym_cluster_p(int mode)
{
    switch (mode) {
    case SIFAR_BARRIER_ONESHOT: return (const void *)k_sym_cluster<DT, P, SIFAR_BARRIER_ONESHOT>;
    case SIFAR_DUALBUF:         return (const void *)k_sym_cluster<DT, P, SIFAR_DUALBUF>;
    case SIFAR_SPECULATIVE:     return (const void *)k_sym_cluster<DT, P, SIFAR_SPECULATIVE>;
    case kModeNoAllreduce:      return (const void *)k_sym_cluster<DT, P, kModeNoAllreduce>;
    default:                    return nullptr;
    }
}

template <int DT>
static const void *chain_cluster_dt(int P, int mode, bool trace)
{
    /* the traced build exists for the shapes of the workload list only */
    if (trace && P == 8) return chain_cluster_p<DT, 8, true>(mode);
    if (trace && P == 2) return chain_cluster_p<DT, 2, true>(mode);
    switch (P) {
    case 1: return chain_cluster_p<DT, 1, false>(mode);
    case 2: return chain_cluster_p<DT, 2, false>(mode);
    case 3: return chain_cluster_p<DT, 3, false>(mode);
    case 4: return chain_cluster_p<DT, 4, false>(mode);
    case 5: return chain_cluster_p<DT, 5, false>(mode);
    case 6: return chain_cluster_p<DT, 6, false>(mode);
    case 7: return chain_cluster_p<DT, 7, false>(mode);
    default: return chain_cluster_p<DT, 8, false>(mode);
    }
}

template <int DT>
static const void *sym_cluster_dt(int P, int mode)
{
    switch (P) {
    case 1: return sym_cluster_p<DT, 1>(mode);
    case 2: return sym_cluster_p<DT, 2>(mode);
    case 3: return sym_cluster_p<DT, 3>(mode);
    case 4: return sym_cluster_p<DT, 4>(mode);
    case 5: return sym_cluster_p<DT, 5>(mode);
    case 6: return sym_cluster_p<DT, 6>(mode);
    case 7: return sym_cluster_p<DT, 7>(mode);
    default: return sym_cluster_p<DT, 8>(mode);
    }
}

const void *chain_cluster_kernel(int dtype, int P, int mode, bool trace)
{
    return dtype == SIFAR_BF16 ? chain_cluster_dt<SIFAR_BF16>(P, mode, trace) : chain_cluster_dt<SIFAR_F32>(P, mode, trace);
}

const void *sym_cluster_kernel(int dtype, int P, int mode)
{
    return dtype == SIFAR_BF16 ? sym_cluster_dt<SIFAR_BF16>(P, mode) : sym_cluster_dt<SIFAR_F32>(P, mode);
}

/* Asked for the default placement; by load the device holds as many clusters or more (reported on B200, default / by load:
   nine CTAs 93 / 96, seven 142 / 148, five 168 / 174, three 284 / 296). */
bool cluster_fits(const void *kernel, int cluster, size_t clusters)
{
    if (!kernel) return false;
    cudaError_t err = cudaSuccess;
    if (cluster > 8) err = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = cluster_config(attr, cluster, clusters, kChainThreads, nullptr);
    int most = 0;
    if (err == cudaSuccess) err = cudaOccupancyMaxActiveClusters(&most, kernel, &cfg);
    if (err != cudaSuccess) { cudaGetLastError(); return false; }
    return (size_t)most >= clusters;
}

bool chain_dependent_launches()
{
    static const bool on = !(getenv("SIFAR_CHAIN_PDL") && atoi(getenv("SIFAR_CHAIN_PDL")) == 0);
    return on;
}

cudaError_t launch_clusters(const void *kernel, int cluster, size_t clusters, cudaStream_t stream, void **params, bool dependent,
                            bool by_load)
{
    cudaLaunchAttribute attr[3];
    cudaLaunchConfig_t cfg = cluster_config(attr, cluster, clusters, kChainThreads, stream);
    if (by_load) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterSchedulingPolicyPreference;
        attr[cfg.numAttrs++].val.clusterSchedulingPolicyPreference = cudaClusterSchedulingPolicyLoadBalancing;
    }
    if (dependent && chain_dependent_launches()) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    return cudaLaunchKernelExC(&cfg, kernel, params);
}

}  /* namespace sifar */
