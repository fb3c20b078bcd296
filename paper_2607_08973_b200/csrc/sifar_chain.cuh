/*
 * sifar_chain.cuh - what the persistent decode-step kernels share: their arguments, the flags of a chunk, and the
 * hand-over of a result through tagged words in global memory.
 */
#ifndef SIFAR_CHAIN_CUH
#define SIFAR_CHAIN_CUH

#include "sifar_internal.cuh"
#include "sifar_reduce.cuh"
#include "sifar_workload.h"

namespace sifar {

constexpr int kModeNoAllreduce = SIFAR_CHAIN_NO_ALLREDUCE;
constexpr int kChainThreads = 128;
constexpr int kTraceSlots = 48;         /* 0-3 reducer, 4 + 3r .. 6 + 3r rank r's producer, 28 done flags */

struct __align__(128) ChunkFlags {
    uint32_t ready;                 /* call number whose result chunk is published (flag form of the hand-over) */
    uint32_t pad0[7];
    uint32_t arrive[2][8];          /* per parity, per rank: this chunk of the rank's partial stored */
    uint32_t done[8];               /* per rank: the chunk's reducer has finished reading call e (bottom barrier) */
};

struct __align__(128) ChainDev {
    uint32_t exit_count;            /* CTAs that left the kernel (monotonic)                        */
    uint32_t seen[4];               /* written by CTA 0 of the last run: role layout (1 = clustered), CTAs per
                                       cluster as the hardware reports them, form of the hand-over (1 = tagged),
                                       [3] by k_chain_pipe alone (1 = units in turn) */
    uint32_t pad0[27];
};

struct PersistArgs {
    DevState *st;
    int *host_status;
    unsigned long long timeout_ns;
    sifar_workload w;
    unsigned long long n;
    char *plain;                    /* [parity][rank] plain buffers */
    unsigned long long plain_stride;
    char *slots;                    /* [parity][rank] slot buffers  */
    unsigned long long slot_stride;
    char *ring;
    unsigned long long ring_stride;
    uint32_t ring_len;
    uint32_t e0;                    /* calls completed before this run     */
    uint32_t base_epoch;
    uint32_t steps;
    uint32_t C;                     /* chunks = reducer CTAs               */
    uint32_t K;                     /* units per thread and step           */
    uint32_t prod_C, prod_K;        /* k_chain_pipe: the same for the producers (C, K: the readers) */
    uint32_t exit_base;
    uint32_t placed;                /* k_chain: one cluster per chunk, for placement only */
    PollShape poll;
    ChainDev *cs;
    ChunkFlags *chunks;
    unsigned long long *stamps;     /* C x pipes x (steps + 1): start of the run and every published result, per chunk
                                       (k_chain, one pipe) or per warp of its reader (k_chain_cluster) */
    unsigned long long *trace;      /* NULL, or steps x kTraceSlots phase stamps of chunk 0 (see sifar_workload.h) */
    uint32_t *retry_steps;          /* steps: 1 if any CTA re-loaded a slot in that step */
    uint4 *handoff;                 /* [parity][unit]: the result as the next producers take it over (see
                                       handoff_store), or NULL: one result-ready flag per chunk instead */
    unsigned long long handoff_stride;   /* 16-byte words per parity */
};

/*
 * Hand-over of a result unit from the chunk's reducer to the P producers of the next step.  The next operation
 * of a rank consumes the all-reduce result on the same GPU (Section 3.1: stream order there); in this one-reader
 * emulation reducer and producers are different CTAs, so the result has to cross.  It crosses the way the partials
 * do in the speculative mode: data and call number in one 16-byte store, validated by the reader, who polls the
 * unit it needs and nothing else - no CTA-wide barrier, no fence, no flag, no second round trip for the data.
 * The other form, one ready flag per chunk (barrier, release; acquire poll by thread 0, barrier, then the loads),
 * costs 0.3-2 us more per step up to 128 KB per rank at P = 8; it is kept for large dual-buffered grids (handoff_max_pairs),
 * where eight times as many threads polling data lines as there are units slow the reducers' stores by as much as the
 * flag costs, and for the large speculative ones that do not run k_chain_pipe (pipe_pays).  With both barriers neither form is needed: the done flags
 * of the bottom barrier follow the result stores.  The chain without all-reduce uses the words too: every rank
 * hands its partial to itself.
 * NW = 3 result words (a 12-byte unit: speculative mode, chain without all-reduce): {w0, w1, w2, tag}.  NW = 4
 * (a 16-byte vector of the dual-buffered mode): two stores {w0, tag, w1, tag}, {w2, tag, w3, tag}, each valid by
 * itself.
 */
template <int NW>
__device__ __forceinline__ void handoff_store(uint4 *base, size_t u, const uint4 &v, uint32_t tag)
{
    if (NW == 3) {
        st_slot(base + u, make_uint4(v.x, v.y, v.z, tag));
    } else {
        st_slot(base + 2 * u, make_uint4(v.x, tag, v.y, tag));
        st_slot(base + 2 * u + 1, make_uint4(v.z, tag, v.w, tag));
    }
}

/* Polls until unit u carries `tag` (bounded; also gives up when the context already carries an error). */
template <int NW>
__device__ __forceinline__ bool handoff_wait(const uint4 *base, size_t u, uint32_t tag, uint32_t (&w)[NW], DevState *st,
                                             int *host_status, unsigned long long timeout_ns)
{
    Deadline d;
    for (;;) {
        if (NW == 3) {
            const uint4 a = ld_slot(base + u);
            if (a.w == tag) { w[0] = a.x; w[1] = a.y; w[2] = a.z; return true; }
        } else {
            const uint4 a = ld_slot(base + 2 * u), b = ld_slot(base + 2 * u + 1);
            if (a.y == tag && a.w == tag && b.y == tag && b.w == tag) {
                w[0] = a.x; w[1] = a.z; w[2] = b.x; w[NW - 1] = b.z;
                return true;
            }
        }
        if (d.expired(timeout_ns)) { fail(st, host_status, SIFAR_ERR_TIMEOUT); return false; }
        if ((d.polls % 64u) == 0u && ld_relaxed_u32(&st->status) != 0u) return false;
    }
}


/* ------------------------------------------------------------------------ */
/* the chain with P readers                                                  */
/* ------------------------------------------------------------------------ */
/* Flags of one chunk: what the P CTAs that own it tell each other. */
struct __align__(128) SymFlags {
    uint32_t arrive[2][8];          /* [parity][rank]: chunk of the rank's partial of call e stored      */
    uint32_t pad0[16];
    uint32_t done[8];               /* [rank]: the rank's reader has finished reading the chunk of call e */
    uint32_t pad1[24];
};

struct __align__(128) SymDev {
    uint32_t exit_count;            /* CTAs that left the kernel (monotonic over runs) */
    uint32_t pad[31];
};

struct SymArgs {
    DevState *st;
    int *host_status;
    unsigned long long timeout_ns;
    sifar_workload w;
    unsigned long long n;
    char *plain;                    /* [parity][rank] plain buffers */
    unsigned long long plain_stride;
    char *slots;                    /* [parity][rank] slot buffers  */
    unsigned long long slot_stride;
    char *rings;                    /* [rank][ring_len] result rows */
    unsigned long long ring_stride;
    uint32_t ring_len;
    uint32_t e0;                    /* calls completed before this run */
    uint32_t base_epoch;
    uint32_t steps;
    uint32_t C, K;
    uint32_t exit_base;
    PollShape poll;
    SymDev *cs;
    SymFlags *flags;                /* C */
    unsigned long long *stamps;     /* [rank][chunk][warp][steps + 1] */
    uint32_t *retry_marks;          /* [rank][steps]: 1 if the rank re-loaded a slot in that step */
    unsigned long long *rank_retries; /* [P] cumulative (rank, step) pairs with a re-load */
};

/* Last CTA out of a run of the chain with P readers: the retry marks are summed and cleared, the run is booked. */
template <int P>
__device__ __forceinline__ void book_sym_run(const SymArgs &a, bool marks)
{
    DevState *st = a.st;
    if (marks) {
        unsigned long long any_steps = 0;
        for (uint32_t s = threadIdx.x; s < a.steps; s += blockDim.x) {
            uint32_t any = 0;
            for (int r = 0; r < P; ++r) {
                const uint32_t m = ld_relaxed_u32(&a.retry_marks[(size_t)r * a.steps + s]);
                if (m) {
                    atomicAdd(&a.rank_retries[r], 1ull);
                    st_relaxed_u32(&a.retry_marks[(size_t)r * a.steps + s], 0u);
                }
                any |= m;
            }
            any_steps += any ? 1ull : 0ull;
        }
        if (any_steps) atomicAdd(&st->stats[kStatCallsWithRetry], any_steps);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(&st->stats[kStatCalls], (unsigned long long)a.steps);
        st_release_u32(&st->epoch, a.e0 + a.steps);
    }
}

/* The kernels of small grids, whose ranks meet in a cluster's shared memory (sifar_chain_cluster.cu): one unit per
   thread, kChainThreads threads per CTA.  sym_cluster_kernel() is NULL for modes that have no such form. */
const void *chain_cluster_kernel(int dtype, int P, int mode, bool trace);
const void *sym_cluster_kernel(int dtype, int P, int mode);
/* The speculative chain whose threads take several units in turn (sifar_chain_pipe.cu), and how many at most. */
constexpr uint32_t kPipeParked = 8;
const void *chain_pipe_kernel(int dtype, int P, bool trace);
/* false: SIFAR_CHAIN_PDL=0 when this was first asked for */
bool chain_dependent_launches();
/* Can the device hold `clusters` clusters of `cluster` CTAs of the kernel at once? */
bool cluster_fits(const void *kernel, int cluster, size_t clusters);
/* `dependent`: the kernel does a prologue of its own and then waits for what precedes it on the stream.  `by_load`: the
   CTAs go where the fewest are (cluster_by_load). */
cudaError_t launch_clusters(const void *kernel, int cluster, size_t clusters, cudaStream_t stream, void **params, bool dependent,
                            bool by_load);

}  /* namespace sifar */
#endif
