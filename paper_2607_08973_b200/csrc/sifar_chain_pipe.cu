/*
 * sifar_chain_pipe.cu - the persistent speculative chain on grids whose threads own several units per step: the units
 * of a thread are chains of their own, taken in turn.
 *
 * k_chain lets a producer compute the seeded halves of all its units, wait, and then take and store them one after the
 * other; a CTA of the reader does the same, and both end a step at a CTA barrier.  At 512 KB per rank and P = 8 the
 * generator's 3.6 us of integer arithmetic and the 4 us of dependent trips through the L2 came one after the other,
 * everywhere at the same time.  Units do not depend on one another, so here a producer takes, stores and prepares one
 * unit, then the next: while unit 0 travels to its reader and back, the thread computes the seeded halves of the others,
 * and the next unit's hand-over word is loaded before the arithmetic that hides the load.  No CTA barrier, no flag.
 * What is left is instructions (issue slots 77 % busy at 512 KB, the integer pipe 64 %), so those were counted: the kind of
 * the workload is looked at once per unit, whole units are not masked, index arithmetic has 32 bits, the look at the
 * P tags is one word.
 * Readers have fewer units per thread than producers where there is room (their trip per unit, about 1800 cycles under
 * load, is what a reader waits for and does little in), but not one alone: a reader needs something to do while it waits
 * (P = 8: at 240 KB per rank two units per reader thread took 14 % less time than one, at 512 KB 7 % less than four).
 * us per 120 steps at P = 8, bf16, 512 KB per rank: k_chain 1007, this kernel 787; other sizes at kPipeMinPairs, and where few
 * ranks give a thread too little to do, at pipe_pays().
 */
#include "sifar_internal.cuh"
#ifdef SIFAR_SLOT_S8X2
#error "the decode-step chains are written for the default slot format; the fallback format is built for libsifar only"
#endif
#include "sifar_chain.cuh"
#include "sifar_gen.cuh"

namespace sifar {

constexpr uint32_t kPipeWarps = kChainThreads / 32;

template <int DT, int P, bool TRACE>
__global__ void __launch_bounds__(kChainThreads, 6) k_chain_pipe(const PersistArgs a)
{
    constexpr int NE = 3 * ((DT == SIFAR_BF16) ? 2 : 1);              /* elements of a slot */
    DevState *st = a.st;
    const bool is_reader = blockIdx.x < a.C;                          /* readers first, then the producers rank by rank */
    const uint32_t K = is_reader ? a.K : a.prod_K;
    const uint32_t rank = is_reader ? 0u : (blockIdx.x - a.C) / a.prod_C;
    const uint32_t chunk = is_reader ? blockIdx.x : (blockIdx.x - a.C) % a.prod_C;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    /* 32-bit element and unit numbers: payloads have at most 2^31 elements.  Whole warps of units, as in k_chain: units
       past the last element carry zeros, rows have room for them. */
    const uint32_t n = (uint32_t)a.n;
    const uint32_t nunits = ((n + NE - 1) / NE + 31u) / 32u * 32u;
    const uint32_t unit0 = chunk * (uint32_t)kChainThreads * K + threadIdx.x;
    /* units of this thread; the same for all lanes of a warp */
    const uint32_t after = unit0 >= nunits ? 0u : (nunits - unit0 + kChainThreads - 1u) / kChainThreads;
    const uint32_t mine = after < K ? after : K;
    /* the seeded halves of the next step, by unit */
    __shared__ float s_z[kPipeParked][NE][kChainThreads];
    __shared__ int s_last;
    if (blockIdx.x == 0 && threadIdx.x == 0) { a.cs->seen[0] = 0u; a.cs->seen[1] = 1u; a.cs->seen[2] = 1u; a.cs->seen[3] = 1u; }
    unsigned reloads = 0;
    unsigned long long *my_stamps = a.stamps + ((size_t)chunk * kPipeWarps + warp) * (a.steps + 1u);
    const bool stamper = is_reader && lane == 0u;
    if (stamper) my_stamps[0] = globaltimer_ns();
    const bool tracer = TRACE && a.trace != nullptr && chunk == 0u;
#define SIFAR_TRACE(slot, who) do { if (TRACE && tracer && (who)) a.trace[(size_t)s * kTraceSlots + (slot)] = globaltimer_ns(); } while (0)

    if (is_reader) {
        bool ok = true;
        uint32_t seen = a.e0;                                          /* lane r: tag of rank r's copy of the warp's first slot */
        const auto slots_of = [&](uint32_t r, uint32_t parity) {
            return reinterpret_cast<const uint4 *>(a.slots + ((size_t)parity * P + r) * a.slot_stride);
        };
        const auto store_row = [](char *to, uint32_t u, const uint4 &v) {
            uint32_t *dst = reinterpret_cast<uint32_t *>(to) + (size_t)u * 3u;
            dst[0] = v.x; dst[1] = v.y; dst[2] = v.z;
        };
        for (uint32_t s = 0; s < a.steps && ok && mine; ++s) {
            const uint32_t e = a.e0 + 1u + s;
            const uint32_t p = e & 1u;
            char *row = a.ring + (size_t)((e - a.base_epoch - 1u) % a.ring_len) * a.ring_stride;
            uint4 *ho = a.handoff + (size_t)p * a.handoff_stride;
            const uint4 *src[P];
#pragma unroll
            for (int r = 0; r < P; ++r) src[r] = slots_of((uint32_t)r, p);
            const unsigned before = reloads;
            SIFAR_TRACE(0, threadIdx.x == 0);
#pragma unroll 1
            for (uint32_t k = 0; k < mine; ++k) {
                const uint32_t u = unit0 + k * kChainThreads;
                /* ahead of its producers: one lane per rank waits, the other slots are left alone meanwhile */
                if (a.poll.sentinel && __any_sync(0xFFFFFFFFu, lane < (uint32_t)P && seen != e))
                    ok = sentinel_wait<P>(src, u - lane, e, a.timeout_ns, reloads);
                uint4 x[P];
#pragma unroll
                for (int r = 0; r < P; ++r) x[r] = ld_slot(src[r] + u);
                /* a look at the unit that comes next travels beside these */
                if (a.poll.sentinel && lane < (uint32_t)P) {
                    const bool more = k + 1u < mine;
                    const uint4 *next = slots_of(lane, more ? p : p ^ 1u) + ((more ? u + kChainThreads : unit0) - lane);
                    seen = ld_relaxed_u32(&next->w);
                }
                uint32_t wrong = a.poll.forced;
#pragma unroll
                for (int r = 0; r < P; ++r) wrong |= x[r].w ^ e;
                if (wrong != 0u && ok)
                    ok = validate_slot<P>(x, src, u, e, a.timeout_ns, a.poll, reloads,
                                          (TRACE && tracer && threadIdx.x == 0 && k == 0u) ? a.trace + (size_t)s * kTraceSlots + 30 : nullptr);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) { if (lane == 0u) fail(st, a.host_status, SIFAR_ERR_TIMEOUT); break; }
                SIFAR_TRACE(1, k == 0u && threadIdx.x == 0);
                SIFAR_TRACE(38 + warp, k == 0u && lane == 0u);
                const uint4 v = sum_vec<DT, P>(x, false);
                handoff_store<3>(ho, u, v, e);
                store_row(row, u, v);
            }
            if (!ok) break;
            SIFAR_TRACE(2, threadIdx.x == 0);
            SIFAR_TRACE(3, threadIdx.x == 0);
            if (TRACE && tracer && threadIdx.x == 0) a.trace[(size_t)s * kTraceSlots + 29] = reloads - before;
            if (__any_sync(0xFFFFFFFFu, reloads != before) && lane == 0u) st_relaxed_u32(&a.retry_steps[s], 1u);
            if (stamper) my_stamps[s + 1u] = globaltimer_ns();
        }
    } else if (mine) {
        const uint32_t t0 = a.e0 + 1u - a.base_epoch;
        Gen g = make_gen(a.w, rank, t0);
        float z[NE];
        /* the seeded half of unit k for the step that g stands at, into its place */
        const auto park = [&](uint32_t k, bool opening) {
            const uint32_t i0 = (unit0 + k * kChainThreads) * NE;
            if (!opening && g.kind == 0) {
#pragma unroll
                for (int q = 0; q < NE; ++q) z[q] = __fmul_rn(gen_gauss(g, i0 + q), g.sigma);
#pragma unroll
                for (int q = 0; q < NE; ++q) s_z[k][q][threadIdx.x] = z[q];
            } else {
                /* the first step of a chain and the other kinds in little code */
#pragma unroll 1
                for (uint32_t q = 0; q < (uint32_t)NE; ++q) {
                    float y[1];
                    unit_noise<SIFAR_F32, 1>(g, opening, i0 + q, y);
                    s_z[k][q][threadIdx.x] = y[0];
                }
            }
        };
#pragma unroll 1
        for (uint32_t k = 0; k < mine; ++k) park(k, t0 == 1u);
        bool ok = true;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (t0 != 1u) v = ld_slot(a.handoff + (size_t)(a.e0 & 1u) * a.handoff_stride + unit0);
        for (uint32_t s = 0; s < a.steps && ok; ++s) {
            const uint32_t e = a.e0 + 1u + s;
            const uint32_t t = e - a.base_epoch;
            const uint32_t p = e & 1u;
            const bool first = (t == 1u), last = (s + 1u == a.steps);
            const uint4 *ho_prev = a.handoff + (size_t)(p ^ 1u) * a.handoff_stride;
            const uint4 *ho_cur = a.handoff + (size_t)p * a.handoff_stride;
            uint4 *dst = reinterpret_cast<uint4 *>(a.slots + ((size_t)p * P + rank) * a.slot_stride);
            const uint32_t delay_ns = gen_delay_ns(a.w, rank, t);
            gen_step(g, t + 1u);
#pragma unroll 1
            for (uint32_t k = 0; k < mine; ++k) {
                const uint32_t u = unit0 + k * kChainThreads;
                if (!first) {
                    Deadline d;
                    while (!slot_valid(v, e - 1u)) {
                        v = ld_slot(ho_prev + u);
                        if (slot_valid(v, e - 1u)) break;
                        if (d.expired(a.timeout_ns)) { fail(st, a.host_status, SIFAR_ERR_TIMEOUT); ok = false; break; }
                        if ((d.polls % 64u) == 0u && ld_relaxed_u32(&st->status) != 0u) { ok = false; break; }
                    }
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                }
                SIFAR_TRACE(4 + 3 * rank, k == 0u && threadIdx.x == 0);
                if (k == 0u) spin_ns(delay_ns);                        /* seeded skew, before anything is stored */
                const uint32_t pw[3] = {v.x, v.y, v.z};
                uint32_t w[3];
#pragma unroll
                for (int q = 0; q < NE; ++q) z[q] = s_z[k][q][threadIdx.x];
                if ((u + 1u) * NE <= n) unit_apply<DT, 3>(g, first, pw, 0, NE, z, w);      /* a whole unit: nothing to mask */
                else unit_apply<DT, 3>(g, first, pw, u * NE, n, z, w);
                store_slot(dst, u, w[0], w[1], w[2], e);
                /* the previous result of the unit that comes next is on its way while this unit's next seeded half is computed */
                if (k + 1u < mine) { if (!first) v = ld_slot(ho_prev + u + kChainThreads); }
                else if (!last) v = ld_slot(ho_cur + unit0);
                if (!last) park(k, false);
            }
            SIFAR_TRACE(42 + warp, rank == 0u && lane == 0u);
            SIFAR_TRACE(5 + 3 * rank, threadIdx.x == 0);
        }
    }
#undef SIFAR_TRACE
    /* leave: mis-speculation counters, then the last CTA out books the run and publishes the call number */
    const unsigned warp_reloads = __reduce_add_sync(0xFFFFFFFFu, reloads);
    if (warp_reloads && lane == 0u) atomicAdd(&st->stats[kStatSlotReloads], (unsigned long long)warp_reloads);
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t left = atom_add_acq_rel_u32(&a.cs->exit_count, 1u) + 1u;
        s_last = (left == a.exit_base + gridDim.x && ld_relaxed_u32(&st->status) == 0u);
    }
    __syncthreads();
    if (s_last) {
        unsigned long long part = 0;
        for (uint32_t s = threadIdx.x; s < a.steps; s += kChainThreads) {
            part += ld_relaxed_u32(&a.retry_steps[s]);
            st_relaxed_u32(&a.retry_steps[s], 0u);
        }
        if (part) atomicAdd(&st->stats[kStatCallsWithRetry], part);
        __syncthreads();
        if (threadIdx.x == 0) {
            atomicAdd(&st->stats[kStatCalls], (unsigned long long)a.steps);
            st_release_u32(&st->epoch, a.e0 + a.steps);
        }
    }
}

template <int DT, bool TRACE>
static const void *pipe_dt(int P)
{
    switch (P) {
    case 1: return (const void *)k_chain_pipe<DT, 1, false>;
    case 2: return (const void *)k_chain_pipe<DT, 2, TRACE>;
    case 3: return (const void *)k_chain_pipe<DT, 3, false>;
    case 4: return (const void *)k_chain_pipe<DT, 4, false>;
    case 5: return (const void *)k_chain_pipe<DT, 5, false>;
    case 6: return (const void *)k_chain_pipe<DT, 6, false>;
    case 7: return (const void *)k_chain_pipe<DT, 7, false>;
    default: return (const void *)k_chain_pipe<DT, 8, TRACE>;
    }
}

const void *chain_pipe_kernel(int dtype, int P, bool trace)
{
    /* the traced build exists for the shapes of the workload list only */
    if (dtype == SIFAR_BF16) return trace ? pipe_dt<SIFAR_BF16, true>(P) : pipe_dt<SIFAR_BF16, false>(P);
    return trace ? pipe_dt<SIFAR_F32, true>(P) : pipe_dt<SIFAR_F32, false>(P);
}

}  /* namespace sifar */
