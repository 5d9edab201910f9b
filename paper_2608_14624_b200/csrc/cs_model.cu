// Transition Learner and Survival Scorer state: transition counting (Algorithm 1,
// ObserveTouch), Eq. 3 normalisation with row arg-max (Eq. 5 / Eq. 10), predictability
// (Eq. 2) and gate (Eq. 11), threshold graph (Eq. 7), BFS hop table and survival scores
// (Eq. 8).  The model is tiny (A <= 1024), so these kernels are latency-bound: the design
// goal is few launches and no host round trip, not bandwidth.
#include <mutex>
#include <stddef.h>

#include <cooperative_groups.h>

#include "cs_common.cuh"

namespace cg = cooperative_groups;

#define OBS_THREADS 1024
#define ROW_THREADS 256
#define OBS_FUSED_MAX 256u     // events up to which a batch is applied inside the refresh launch (one per thread)
static_assert(OBS_FUSED_MAX <= 256, "the refresh kernel stages one event per thread");

// ---------------------------------------------------------------------------------------------
// Initial state of Algorithm 1: zero counts, no current agent; plus the recency table.
// ---------------------------------------------------------------------------------------------
__global__ void cs_init_kernel(cs_workspace ws, uint32_t A, uint32_t n_chains, uint32_t gtab_len, float lambda,
                               float delta)
{
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    for (uint32_t i = tid; i < A * A; i += nth) ws.C[i] = 0;
    for (uint32_t i = tid; i < A; i += nth) ws.rowsum[i] = 0;
    for (uint32_t i = tid; i < n_chains; i += nth) ws.cur[i] = CS_AGENT_NONE;
    for (uint32_t i = tid; i < CS_HIST_BINS; i += nth) ws.hist[i] = 0;
    for (uint32_t i = tid; i < gtab_len; i += nth) ws.gtab[i] = cs_recency(lambda, delta, i);
    if (tid == 0) {
        cs_scalars z;
        memset(&z, 0, sizeof(z));
        z.last_agent = CS_AGENT_NONE;
        z.a_star = 0xFFFFFFFFu;
        z.sel_T[0] = z.sel_T[1] = z.sel_T[2] = z.sel_T[3] = ~0ull;
        *ws.sc = z;
    }
}

// The recency factor must not increase with age for the select's age-limit prefilter to be exact.
// exp() is monotone mathematically; this checks the table that was actually produced.
__global__ void cs_gtab_check_kernel(cs_workspace ws, uint32_t gtab_len, uint32_t age_sat, float lambda, float delta)
{
    __shared__ int s_bad;
    if (threadIdx.x == 0) s_bad = (gtab_len != age_sat) ? 1 : 0;
    __syncthreads();
    const float g_sat = cs_recency(lambda, delta, age_sat);
    for (uint32_t i = threadIdx.x; i < gtab_len; i += blockDim.x) {
        const float next = (i + 1 < gtab_len) ? ws.gtab[i + 1] : g_sat;
        if (next > ws.gtab[i]) s_bad = 1;
    }
    __syncthreads();
    if (threadIdx.x == 0) ws.sc->gtab_monotone = s_bad ? 0u : 1u;
}

// ---------------------------------------------------------------------------------------------
// Transition counting over one long batch of events, one thread-block cluster.  The update is sequential per chain
// (each event's predecessor is the previous non-warmup event of the same chain, in this batch or carried in cur[]),
// but the counter increments commute, so every event is handled by its own thread once its predecessor is known.
// The batch is walked in rounds of one event per thread of the cluster, every CTA holding a consecutive share:
//   * inside a warp the predecessor comes from one match over the lanes' chains;
//   * inside a CTA a hash table gives, for every chain of the share, the set of warps that hold one of its events
//     (a 32-bit mask): the nearest earlier warp is searched for it, 32 events, one thread per (warp, chain);
//   * the first event of a chain in a share looks the chain up in the tables of the CTAs before it through distributed
//     shared memory, nearest first, and takes cur[] when none of them has it.  The last event of a chain in a share
//     writes cur[] when no later CTA has the chain.
// Counts gather in shared memory where the count matrix fits there (global atomics on the A * A addresses of a few
// agents queue up in L2) and reach the matrix once per call.  Integer adds make the result independent of the order.
//
// Bound by latency: the work of a round is a few hundred instructions per thread between two cluster barriers.
// 20,000 events of 64 chains, 12 agents: 427 us as one CTA that walked the batch 1,024 events at a time and searched
// predecessors event by event; 9.4 us like this (two rounds on 16 CTAs).
// ---------------------------------------------------------------------------------------------
#define OBS_MAX_CLUSTER 16
#define OBS_HASH (2u * OBS_THREADS)
#define OBS_NO_CHAIN 0xFFFFFFFFu
#define OBS_SMEM_AGENTS 64u            // up to this many agents the batch's counts gather in shared memory

struct ObsShare {                      // what the other CTAs of the cluster read
    uint32_t h_chain[OBS_HASH];        // chains of this CTA's share (open addressing), OBS_NO_CHAIN: empty
    uint16_t h_last[OBS_HASH];         // agent of the chain's last live event in the share
    uint16_t agent[OBS_THREADS];       // the share's agents, CS_AGENT_NONE where an event is skipped
    int last_at;                       // the share's last live event, -1: none
};

__device__ __forceinline__ uint32_t obs_slot(uint32_t chain) { return (chain * 0x9E3779B1u) >> 21; }
static_assert(OBS_HASH == 1u << 11, "obs_slot() takes the top bits of a 32-bit product");

// Slot of a chain in a (possibly remote) table, OBS_HASH when it is not there.
__device__ __forceinline__ uint32_t obs_find(const uint32_t *h_chain, uint32_t chain)
{
    for (uint32_t s = obs_slot(chain), n = 0; n < OBS_HASH; s = (s + 1u) & (OBS_HASH - 1u), ++n) {
        const uint32_t v = h_chain[s];
        if (v == chain) return s;
        if (v == OBS_NO_CHAIN) break;
    }
    return OBS_HASH;
}

__global__ void __launch_bounds__(OBS_THREADS)
cs_observe_kernel(cs_workspace ws, uint32_t A, uint32_t n_chains, const uint32_t *__restrict__ chain,
                  const uint16_t *__restrict__ agent, const uint8_t *__restrict__ evflags, uint32_t n_events,
                  const uint32_t *__restrict__ n_events_dev)
{
    __shared__ ObsShare sh;
    __shared__ uint32_t h_warps[OBS_HASH];                       // warps that hold an event of the slot's chain
    __shared__ __align__(16) uint32_t s_chain[OBS_THREADS];      // OBS_NO_CHAIN marks an event that is skipped
    __shared__ uint32_t s_C[OBS_SMEM_AGENTS * OBS_SMEM_AGENTS], s_row[OBS_SMEM_AGENTS];
    cs_wait_for_predecessor();
    cs_release_successor();
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (n_events_dev) n_events = min(n_events, *n_events_dev);   // device-resident count (graph replay)
    const uint32_t rounds = (n_events + CL * OBS_THREADS - 1) / (CL * OBS_THREADS);
    const uint32_t share = rounds ? (n_events + rounds * CL - 1) / (rounds * CL) : 0u;      // events per CTA and round
    // (a CTA on its own needs no cluster barriers, and with one round nothing it looks up in cur[] changes before it does)
    const auto everywhere = [&] { if (CL > 1) cluster.sync(); else __syncthreads(); };
    const bool local = A <= OBS_SMEM_AGENTS;
    if (local) {
        for (uint32_t i = tid; i < A * A; i += OBS_THREADS) s_C[i] = 0;
        if (tid < A) s_row[tid] = 0;
    }
    uint32_t n_skipped = 0, n_new = 0;
    for (uint32_t rd = 0; rd < rounds; ++rd) {
        const uint32_t e = (rd * CL + rank) * share + tid;
        uint32_t c = OBS_NO_CHAIN, a = CS_AGENT_NONE;
        if (tid < share && e < n_events) {
            c = chain[e];
            a = agent[e];
            const bool warm = evflags && (evflags[e] & CS_EV_WARMUP);
            uint32_t bad = 0;
            if (!warm && a >= A) bad |= CS_ST_BAD_AGENT;
            if (!warm && c >= n_chains) bad |= CS_ST_BAD_CHAIN;
            if (bad) atomicOr(&ws.sc->status, bad);
            if (warm || bad) { c = OBS_NO_CHAIN; a = CS_AGENT_NONE; ++n_skipped; }
        }
        const bool live = a != CS_AGENT_NONE;
        uint32_t carried = CS_AGENT_NONE;                        // in flight during the searches below
        if (live && rounds == 1u) carried = cs_ld_cg_pinned(ws.cur + c);
        s_chain[tid] = c;
        sh.agent[tid] = (uint16_t)a;
        for (uint32_t i = tid; i < OBS_HASH; i += OBS_THREADS) { sh.h_chain[i] = OBS_NO_CHAIN; h_warps[i] = 0; }
        if (tid == 0) sh.last_at = -1;
        // inside the warp: the events of this lane's chain, the one before it, whether it is the warp's last of the chain
        const uint32_t same = __match_any_sync(0xFFFFFFFFu, c);
        const uint32_t before = same & ((1u << lane) - 1u);
        const uint32_t a_before = __shfl_sync(0xFFFFFFFFu, a, before ? 31 - __clz(before) : (int)lane);
        uint32_t prev = (live && before) ? a_before : CS_AGENT_NONE;
        const bool last_in_warp = live && (same >> lane) == 1u;
        __syncthreads();
        uint32_t slot = 0;
        if (last_in_warp) {
            slot = obs_slot(c);
            for (;;) {                                           // ends: the table has twice as many slots as events
                const uint32_t was = atomicCAS(&sh.h_chain[slot], OBS_NO_CHAIN, c);
                if (was == OBS_NO_CHAIN || was == c) break;
                slot = (slot + 1u) & (OBS_HASH - 1u);
            }
            atomicOr(&h_warps[slot], 1u << warp);
        }
        slot = __shfl_sync(0xFFFFFFFFu, slot, 31 - __clz(same));        // the whole group learns its chain's slot
        const int newest_of_warp = __reduce_max_sync(0xFFFFFFFFu, live ? (int)tid : -1);
        if (lane == 0 && newest_of_warp >= 0) atomicMax(&sh.last_at, newest_of_warp);
        __syncthreads();
        const uint32_t wm = live ? h_warps[slot] : 0u;
        bool need_far = false;                                   // no event of the chain before this one in the share
        if (live && !before) {
            const uint32_t wb = wm & ((1u << warp) - 1u);
            if (wb) {
                const uint32_t w = 31u - __clz(wb);
                const uint4 *q = (const uint4 *)(s_chain + 32u * w);
                int at = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {                    // the last match is the one wanted
                    const uint4 v = q[i];
                    if (v.x == c) at = 4 * i;
                    if (v.y == c) at = 4 * i + 1;
                    if (v.z == c) at = 4 * i + 2;
                    if (v.w == c) at = 4 * i + 3;
                }
                prev = sh.agent[32u * w + at];
            } else {
                need_far = true;
            }
        }
        const bool last_in_cta = last_in_warp && (wm >> warp) == 1u;
        if (last_in_cta) sh.h_last[slot] = (uint16_t)a;
        everywhere();                                            // every table of the cluster is complete
        if (need_far) {
            for (int r = (int)rank - 1; r >= 0 && prev == CS_AGENT_NONE; --r) {
                const ObsShare *o = cluster.map_shared_rank(&sh, r);
                const uint32_t s = obs_find(o->h_chain, c);
                if (s < OBS_HASH) prev = o->h_last[s];
            }
            if (prev == CS_AGENT_NONE) prev = rounds == 1u ? carried : (uint32_t)__ldcg(&ws.cur[c]);
        }
        bool writes_cur = last_in_cta;
        for (uint32_t r = rank + 1; r < CL && writes_cur; ++r)
            if (obs_find(cluster.map_shared_rank(&sh, r)->h_chain, c) < OBS_HASH) writes_cur = false;
        uint32_t newest = CS_AGENT_NONE;
        if (rank == 0 && tid == 0)
            for (int r = (int)CL - 1; r >= 0 && newest == CS_AGENT_NONE; --r) {
                const ObsShare *o = cluster.map_shared_rank(&sh, r);
                if (o->last_at >= 0) newest = o->agent[o->last_at];
            }
        if (live && prev != CS_AGENT_NONE && prev != a) {
            ++n_new;
            if (local) {
                atomicAdd(&s_C[prev * A + a], 1u);
                atomicAdd(&s_row[prev], 1u);
            } else {
                atomicAdd(&ws.C[prev * A + a], 1u);
                atomicAdd(&ws.rowsum[prev], 1u);
            }
        }
        everywhere();                                            // every read of cur[] and of the tables precedes the writes below
        if (writes_cur) ws.cur[c] = (uint16_t)a;
        if (newest != CS_AGENT_NONE) ws.sc->last_agent = newest;
    }
    __syncthreads();
    if (local) {
        for (uint32_t i = tid; i < A * A; i += OBS_THREADS) {
            const uint32_t v = s_C[i];
            if (v) atomicAdd(&ws.C[i], v);
        }
        if (tid < A && s_row[tid]) atomicAdd(&ws.rowsum[tid], s_row[tid]);
    }
    n_new = __reduce_add_sync(0xFFFFFFFFu, n_new);
    n_skipped = __reduce_add_sync(0xFFFFFFFFu, n_skipped);
    if (lane == 0 && n_new) {
        atomicAdd(&ws.sc->n_transitions, n_new);
        atomicAdd((unsigned long long *)&ws.cnt->transitions_counted, (unsigned long long)n_new);
    }
    if (lane == 0 && n_skipped) atomicAdd((unsigned long long *)&ws.cnt->events_skipped, (unsigned long long)n_skipped);
    if (rank == 0 && tid == 0) atomicAdd((unsigned long long *)&ws.cnt->events_seen, (unsigned long long)n_events);
}

// ---------------------------------------------------------------------------------------------
// BFS over the bit-matrix graph from a set of source bits, then Eq. 8, by the first W warps of a CTA (all of their threads
// call; W = words of a row, KW = words it is compiled for).  The search PULLS: thread v holds row v of the TRANSPOSED
// adjacency matrix (the predecessors of v; row[], zero for a thread without a node) in registers and at every level ANDs it
// with the frontier.  A level is then W broadcast loads and ANDs per node, all nodes in parallel, one ballot per warp
// for the next frontier and ONE barrier -- whatever the frontier size, with no atomics and no divergent loops; up to 32
// agents one warp does it without any barrier.  (A push over the frontier's nodes, each ORing its adjacency row into the next
// frontier, was tried: one warp at it takes 80 cycles per node; a CTA at it from global memory, one dependent trip to L2 per
// word of every row, took most of the 92 us of a refresh of 1,024 agents.)
// s_front: 2 * PULL_MAX_WORDS words, the first half the source bits, ordered before this call.  Uses hardware barrier 1.
// ---------------------------------------------------------------------------------------------
#define PULL_MAX_WORDS (CS_MAX_AGENTS / 32u)
template <int KW>
__device__ __forceinline__ void cs_bfs_pull(const uint32_t (&row)[KW], uint32_t A, uint32_t W, uint32_t *s_front,
                                            uint16_t *hops, float *fsurv, uint32_t e_max, float delta)
{
    const uint32_t v = threadIdx.x, lane = v & 31;
    uint32_t my_hops = CS_HOP_NONE;
    if (KW == 1) {
        uint32_t front = s_front[0], seen = front;
        if ((seen >> lane) & 1u) my_hops = 0;
        for (uint32_t level = 1; front; ++level) {
            const bool fresh = (row[0] & front) != 0u && !((seen >> lane) & 1u);
            front = __ballot_sync(0xFFFFFFFFu, fresh);
            seen |= front;
            if (fresh) my_hops = level;
        }
    } else {
        bool seen = v >= A || ((s_front[v >> 5] >> lane) & 1u);
        if (v < A && seen) my_hops = 0;
        for (uint32_t level = 1; level <= A; ++level) {
            const uint32_t *cur = s_front + ((level & 1u) ? 0u : PULL_MAX_WORDS);
            uint32_t *nxt = s_front + ((level & 1u) ? PULL_MAX_WORDS : 0u);
            uint32_t hit = 0;
#pragma unroll
            for (int w = 0; w < KW; ++w) hit |= row[w] & cur[w];          // (words past W: zero rows)
            const bool fresh = hit != 0u && !seen;
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, fresh);
            if (lane == 0) nxt[v >> 5] = word;
            if (fresh) { seen = true; my_hops = level; }
            uint32_t any;
            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                         : "=r"(any)
                         : "r"((uint32_t)fresh), "r"(W * 32u)
                         : "memory");
            if (!any) break;
        }
    }
    if (v < A) {
        hops[v] = (uint16_t)my_hops;
        fsurv[v] = cs_survival_of(my_hops, e_max, delta);
    }
}

// Deterministic block reductions: a fixed butterfly inside each warp, then the warp sums added in warp order, so the
// result does not depend on scheduling.  s_red: one entry per warp (two for the pair form).
template <typename T>
__device__ T cs_block_sum(T v, T *s_red)
{
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    __syncthreads();                                       // an earlier result may still be being read
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    T r = s_red[0];
    for (uint32_t w = 1; w < n_warps; ++w) r += s_red[w];
    return r;
}

// ---------------------------------------------------------------------------------------------
// The refresh of everything derived from the counts: Eq. 3 in canonical fp32 (one rounding per operation, no FMA), every
// row's arg-max, adjacency bits (Eq. 7) and entropy term, then Eq. 2 / Eq. 11 over all rows and the cached search of
// Eq. 7 / 8.
//
// A refresh is a chain of dependent steps on a few hundred kilobytes, so what counts is the number of trips to L2 and of
// barriers between its first load and its last store -- and, once a row has a warp of its own, the instructions an SM has to
// issue for its rows (about a thousand per row: 32 rows per CTA were slower than 16).  Every warp fetches its row, the row's
// sum and -- redundantly per CTA -- the batch of events at once, and what has to meet (column sums of Eq. 2, the transposed
// adjacency matrix for the search, entropies, arg-max) does so in one of them:
//   * up to 32 agents: one CTA;
//   * up to 256: one thread-block cluster, 8 or 16 rows per CTA, meeting in the first CTA's shared memory;
//   * more: the whole GPU, 8 rows per CTA, meeting in global memory (cs_refresh_wide_kernel).
// That CTA then runs the search on some of its warps and the sums of Eq. 2 on others.
//
// Rows are sparse: entries with a zero count all have the same P = eps / n_i, so one logarithm stands for all of them, the
// entries with a count are compacted (one per lane), and their share of the column sums is one number per row with the
// differences on top.  A row no event of a small batch starts at keeps its P and arg-max; only what depends on the total
// number of transitions is recomputed.  Column sums are 2^-60 fixed point: integer addition commutes, so they are
// bit-identical from run to run whatever the order of the atomics.
//
// Measured (back to back in a CUDA graph, us per refresh) against one CTA per row with a "last CTA done" epilogue over
// global atomics and, above 256 agents, a search that pushed from global memory:
//   agents / events      4/1   12/5   12/256   30/8   64/64   128/64   256/64   256/256   400/64   1,024/64
//   before               7.7   8.4    14.8     8.7    12.3    11.9     10.9     21.9      35.8     93.4
//   now                  4.0   4.4    6.9      5.4    6.4     6.7      8.5      10.3      13.9     17.8
// ---------------------------------------------------------------------------------------------
#define RW_ROWS 8u                                        // rows per CTA of the kernel for many agents
#define RW_COLS 256u                                      // columns of a row per warp
template <int KW> struct RfShape {                        // KW: words of an adjacency row the kernel is compiled for
    static constexpr uint32_t COLS = KW * 32u;
    static constexpr uint32_t WARPS = KW == 8 ? 16u : 32u;                           // most warps of a CTA
    static constexpr uint32_t CTAS = KW == 1 ? 1u : (KW == 8 ? 16u : 4u);                    // most partial sums: CTAs, or warps of the last one
    static constexpr int CHUNK = KW < 8 ? KW : 8;                                    // words of a row in registers at a time
};
template <int KW> struct RfShared {
    unsigned long long q[RfShape<KW>::COLS];                        // column sums: this CTA's, in the end everybody's
    unsigned long long base[RfShape<KW>::CTAS];                     // what every column gets from a CTA's zero-count entries
    double hc[RfShape<KW>::CTAS];                                   // sum over a CTA's rows of n_i * (row entropy)
    double row_hc[32];
    unsigned long long row_base[32];
    double red[32];
    __align__(16) uint32_t ev_chain[OBS_FUSED_MAX];                 // the batch: chain of event e (read as 16-byte words),
    uint16_t ev_agent[OBS_FUSED_MAX];                               // its agent (CS_AGENT_NONE: skipped),
    uint16_t ev_prev[OBS_FUSED_MAX];                                // and the agent it follows when that is a counted transition
    uint32_t adj[RfShape<KW>::COLS];                                // bit i: this CTA's row i has an edge to the column
    uint32_t adjT[KW == 32 ? 1 : KW][KW == 32 ? 1 : RfShape<KW>::COLS];              // transposed matrix, word by word
    uint32_t nz_v[RfShape<KW>::WARPS][32];                          // per warp: entries of its row that have a count, gathered
    uint16_t nz_j[RfShape<KW>::WARPS][32];                          // so that every lane works on one
    uint16_t amax[KW == 32 ? 1 : RfShape<KW>::COLS];
    float best_v[KW == 32 ? 32 : 1];                                // KW = 32: what the four warps of a row found
    uint32_t best_i[KW == 32 ? 32 : 1];
    uint32_t front[2 * PULL_MAX_WORDS];
    int last_live;
    bool last_cta;
    uint8_t succ[OBS_FUSED_MAX];                                    // 1: a later live event of the batch has the same chain
};
static_assert(CS_MAX_AGENTS <= 4u * RW_COLS && CS_MAX_AGENTS <= 128u * RW_ROWS, "four warps per row, four warps of CTA sums");
static_assert(sizeof(RfShared<8>) <= 48 * 1024 && sizeof(RfShared<32>) <= 48 * 1024, "the default shared-memory limit");
static_assert(offsetof(RfShared<1>, ev_chain) % 16 == 0 && offsetof(RfShared<8>, ev_chain) % 16 == 0 &&
              offsetof(RfShared<32>, ev_chain) % 16 == 0, "read as 16-byte words");

__device__ __forceinline__ double cs_xlogx(double x) { return x * log(x); }

// A small batch of events is applied by the refresh, by every CTA to its own rows: each CTA finds every event's predecessor (in
// the batch, else the chain's current agent) as cs_observe_kernel does.  What is shared -- cur[], the last agent, the totals and
// the counters -- is written by rf_finish(), in the one CTA that runs it, after every CTA has read it.
template <class Shared>
__device__ __forceinline__ void rf_read_batch(Shared &sm, const cs_workspace &ws, uint32_t A, uint32_t n_chains,
                                              const uint32_t *__restrict__ ev_chain_in, const uint16_t *__restrict__ ev_agent_in,
                                              const uint8_t *__restrict__ ev_flags, uint32_t n_events, bool first, bool count_skipped,
                                              uint32_t &n_new, uint32_t &n_skipped)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (n_events) {
        uint32_t ch = OBS_NO_CHAIN, a = CS_AGENT_NONE, before = CS_AGENT_NONE;
        if (tid < n_events) {
            ch = ev_chain_in[tid];
            a = ev_agent_in[tid];
            const bool warm = ev_flags && (ev_flags[tid] & CS_EV_WARMUP);
            uint32_t bad = 0;
            if (!warm && a >= A) bad |= CS_ST_BAD_AGENT;
            if (!warm && ch >= n_chains) bad |= CS_ST_BAD_CHAIN;
            if (bad && first) atomicOr(&ws.sc->status, bad);
            if (warm || bad) { a = CS_AGENT_NONE; ch = OBS_NO_CHAIN; }
            else before = cs_ld_cg_pinned(ws.cur + ch);        // in flight during the search below
        }
        const bool live = a != CS_AGENT_NONE;
        if (tid < OBS_FUSED_MAX) { sm.ev_chain[tid] = ch; sm.ev_agent[tid] = (uint16_t)a; }
        uint32_t same = 0;
        int newest = -1;
        if (32u * warp < n_events) {                           // (whole warps)
            newest = __reduce_max_sync(0xFFFFFFFFu, live ? (int)tid : -1);
            same = __match_any_sync(0xFFFFFFFFu, ch) & ((1u << lane) - 1u);
        }
        __syncthreads();
        if (lane == 0 && newest >= 0) atomicMax(&sm.last_live, newest);
        bool counted = false;
        if (live) {
            int p = same ? (int)(warp * 32u) + 31 - __clz(same) : -1;
            for (int w = (int)warp - 1; w >= 0 && p < 0; --w) {          // earlier warps, nearest first
                const uint4 *q = (const uint4 *)(sm.ev_chain + 32 * w);
#pragma unroll
                for (int u = 0; u < 8; ++u) {                            // the last match is the one wanted
                    const uint4 v = q[u];
                    if (v.x == ch) p = 32 * w + 4 * u;
                    if (v.y == ch) p = 32 * w + 4 * u + 1;
                    if (v.z == ch) p = 32 * w + 4 * u + 2;
                    if (v.w == ch) p = 32 * w + 4 * u + 3;
                }
            }
            if (p >= 0) { before = sm.ev_agent[p]; sm.succ[p] = 1; }
            counted = before != CS_AGENT_NONE && before != a;
        }
        if (tid < OBS_FUSED_MAX) sm.ev_prev[tid] = (uint16_t)(counted ? before : CS_AGENT_NONE);
        n_new = (uint32_t)__syncthreads_count(counted);
        if (count_skipped) n_skipped = (uint32_t)__syncthreads_count(tid < n_events && !live);
    } else {
        __syncthreads();
    }
}

// The current agent of every chain that has one, as bits of front[] (zero before; whole CTA).  Many chains: eight to a load, four loads
// together, and an agent that another chain has brought costs a look, not an atomic.  Only in kernels of their own (ALL): the refresh
// waits for its instructions, and this code in its middle took 0.75 us from every refresh of few agents that never entered it.
__device__ __forceinline__ void rf_sources_of_chains(uint32_t *front, const uint16_t *cur, uint32_t A, uint32_t n_chains)
{
    const uint32_t tid = threadIdx.x, n_threads = blockDim.x;
    auto source = [&](uint32_t a) {
        if (a < A && !((*(volatile uint32_t *)&front[a >> 5] >> (a & 31)) & 1u)) atomicOr(&front[a >> 5], 1u << (a & 31));
    };
    if (n_chains <= 4u * n_threads) {
        for (uint32_t x = tid; x < n_chains; x += n_threads) source(__ldcg(&cur[x]));
        return;
    }
    const uint32_t n8 = n_chains / 8u;
    for (uint32_t x0 = tid; x0 < n8; x0 += 4u * n_threads) {
        uint4 v[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) v[u] = cs_ld_cg_pinned((const uint4 *)cur + min(x0 + u * n_threads, n8 - 1u));
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            if (x0 + u * n_threads >= n8) break;
            source(v[u].x & 0xFFFFu); source(v[u].x >> 16); source(v[u].y & 0xFFFFu); source(v[u].y >> 16);
            source(v[u].z & 0xFFFFu); source(v[u].z >> 16); source(v[u].w & 0xFFFFu); source(v[u].w >> 16);
        }
    }
    if (tid < (n_chains & 7u)) source(__ldcg(&cur[(n_chains & ~7u) + tid]));
}

// What the one CTA does that has everything: the batch's effect on the shared state, the sums of Eq. 2 and the search.  row:
// thread v's words of the transposed adjacency matrix; base[] and hc[] have n_parts numbers each.
template <int KW, bool ALL>
__device__ __forceinline__ void rf_finish(RfShared<KW> &sm, const cs_workspace &ws, const uint32_t (&row)[KW], uint32_t A, uint32_t W,
                                          uint32_t n_parts, uint32_t n_events, uint32_t n_new, uint32_t n_skipped, uint32_t n_total,
                                          uint32_t la, float r_min, uint32_t e_max, float delta, uint32_t n_chains)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31, n_threads = blockDim.x;
    if (n_events) {
        // the batch's effect on what all CTAs share
        const uint32_t a = tid < n_events ? sm.ev_agent[tid] : CS_AGENT_NONE;
        if (a != CS_AGENT_NONE && !sm.succ[tid]) ws.cur[sm.ev_chain[tid]] = (uint16_t)a;   // the chain's last live event of the batch
        if (sm.last_live >= 0) la = sm.ev_agent[sm.last_live];
        if (tid == 0) {
            ws.sc->last_agent = la;
            ws.sc->n_transitions = n_total;
            atomicAdd((unsigned long long *)&ws.cnt->events_seen, (unsigned long long)n_events);
            if (n_skipped) atomicAdd((unsigned long long *)&ws.cnt->events_skipped, (unsigned long long)n_skipped);
            if (n_new) atomicAdd((unsigned long long *)&ws.cnt->transitions_counted, (unsigned long long)n_new);
        }
    }
    if (ALL) {
        // sources: the current agent of every chain that has one (all live sessions)
        __syncthreads();
        rf_sources_of_chains(sm.front, ws.cur, A, n_chains);
        __syncthreads();
    }
    // The search by the first W warps; the sums of Eq. 2 by the warps behind them, side by side, where the CTA has enough of
    // them, else by the same warps first.
    const uint32_t sum0 = 2u * W * 32u <= n_threads ? W * 32u : 0u;       // first thread of the sums
    if (tid >= sum0 && tid < sum0 + W * 32u) {
        const uint32_t j = tid - sum0;
        double Hm = 0.0;
        if (n_total && j < A) {
            unsigned long long qf = sm.q[j % RfShape<KW>::COLS];
            for (uint32_t r = 0; r < n_parts; ++r) qf += sm.base[r];
            const double q = (double)qf * (1.0 / 1152921504606846976.0);
            if (q > 0.0) Hm = -cs_xlogx(q);
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) Hm += __shfl_xor_sync(0xFFFFFFFFu, Hm, d);
        if (lane == 0) sm.red[j >> 5] = Hm;
        asm volatile("bar.sync 2, %0;" ::"r"(W * 32u) : "memory");
        if (KW == 32 && j < 32u) {                             // (32 additions one after the other would be a microsecond)
            double v = j < W ? sm.red[j] : 0.0;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
            if (j == 0) sm.red[0] = v;
        }
        if (j == 0) {
            double Hc = 0.0, Hs = 0.0;
            for (uint32_t r = 0; r < n_parts; ++r) Hc -= sm.hc[r];
            for (uint32_t w = 0; w < (KW == 32 ? 1u : W); ++w) Hs += sm.red[w];
            double R = 0.0;
            if (n_total && Hs > 0.0) R = 1.0 - Hc / (double)n_total / Hs;
            const float Rf = (float)R;
            ws.sc->R = Rf;
            ws.sc->gate = (Rf >= r_min) ? 1u : 0u;
            ws.sc->a_star = la < A ? (uint32_t)(KW == 32 ? cs_ld_cg_pinned(ws.amax + la) : sm.amax[KW == 32 ? 0u : la]) : 0xFFFFFFFFu;    // Eq. 10, for the prefetch ranking
        }
        CS_STAMP(ws, CS_PS_REFRESH_SUMS_DONE, j == 0);
    }
    if (tid < 32u * W) {
        if (!ALL) {
            if (tid == 0 && la < A) sm.front[la >> 5] = 1u << (la & 31);
            asm volatile("bar.sync 1, %0;" ::"r"(W * 32u) : "memory");
        }
        cs_bfs_pull<KW>(row, A, W, sm.front, ws.hops, ws.fsurv, e_max, delta);
    }
    CS_STAMP(ws, CS_PS_REFRESH_END, tid == 0);
}

// blockDim.x / 32 rows per CTA, a warp each: 8, 16 or 32 in the one CTA (KW = 1), 8 or 16 in each of up to 16 (KW = 8).
template <int KW, bool ALL>
__global__ void __launch_bounds__(RfShape<KW>::WARPS * 32u)
cs_refresh_kernel(cs_workspace ws, uint32_t A, uint32_t W, float eps, float tau, float r_min, uint32_t e_max, float delta,
                  uint32_t n_chains, const uint32_t *__restrict__ ev_chain_in,
                  const uint16_t *__restrict__ ev_agent_in, const uint8_t *__restrict__ ev_flags, uint32_t n_events,
                  const uint32_t *__restrict__ n_events_dev, uint32_t every_row)
{
    constexpr uint32_t COLS = RfShape<KW>::COLS;
    constexpr int CHUNK = RfShape<KW>::CHUNK;
    static_assert(CHUNK == KW, "a row is one chunk");
    __shared__ RfShared<KW> sm;
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_threads = blockDim.x, rows = n_threads >> 5;
    CS_STAMP(ws, CS_PS_REFRESH_ENTRY, blockIdx.x == 0 && tid == 0);
    if (tid < COLS) {
        sm.q[tid] = 0;
        sm.adj[tid] = 0;
#pragma unroll
        for (int w = 0; w < KW; ++w) sm.adjT[w][tid] = 0;                  // (bits past the last row)
    }
    if (tid == 0) sm.last_live = -1;
    if (tid < OBS_FUSED_MAX) sm.succ[tid] = 0;
    if (tid < 2 * PULL_MAX_WORDS) sm.front[tid] = 0;
    if (KW > 1) asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");             // waited for below
    cs_wait_for_predecessor();
    CS_STAMP(ws, CS_PS_REFRESH_WAITED, blockIdx.x == 0 && tid == 0);
    cs_release_successor();

    // ---- everything that depends on nothing, in one trip ---------------------------------------------------------
    if (n_events_dev) n_events = min(n_events, cs_ld_cg_pinned(n_events_dev));
    const uint32_t i = rank * rows + warp;                     // this warp's row
    uint32_t c[CHUNK];
#pragma unroll
    for (int k = 0; k < CHUNK; ++k) {
        const uint32_t j = lane + 32u * k;
        c[k] = 0;
        if (i < A && j < A) c[k] = cs_ld_cg_pinned(ws.C + i * A + j);
    }
    uint32_t n_i = cs_ld_cg_pinned(ws.rowsum + (i < A ? i : 0u));
    uint32_t n_total = cs_ld_cg_pinned(&ws.sc->n_transitions);
    const uint32_t la = cs_ld_cg_pinned(&ws.sc->last_agent);
    uint32_t n_new = 0, n_skipped = 0;
    rf_read_batch(sm, ws, A, n_chains, ev_chain_in, ev_agent_in, ev_flags, n_events, rank == 0, rank == 0, n_new, n_skipped);
    n_total += n_new;
    if (KW > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");                // every CTA has started and cleared its sums

    double row_hc = 0.0;
    unsigned long long row_base = 0;
    const double inv_total = n_total ? 1.0 / (double)n_total : 0.0;
    if (i < A) {                                               // (whole warps)
        uint32_t n_add = 0;
        if (n_new)
            for (uint32_t e0 = 0; e0 < n_events; e0 += 32u) {
                uint32_t hits = __ballot_sync(0xFFFFFFFFu, e0 + lane < n_events && sm.ev_prev[e0 + lane] == i);
                n_add += __popc(hits);
                for (; hits; hits &= hits - 1u) {
                    const uint32_t j = sm.ev_agent[e0 + __ffs(hits) - 1];
#pragma unroll
                    for (int k = 0; k < CHUNK; ++k)
                        if (j == lane + 32u * k) ++c[k];
                }
            }
        n_i += n_add;
        const bool write = every_row || n_add;
        const double pi_fix = (double)n_i * inv_total * 1152921504606846976.0;      // pi_i * 2^60
        const float den = __fadd_rn((float)n_i, __fmul_rn((float)A, eps));
        const float p0 = __fdiv_rn(__fadd_rn(0.0f, eps), den);              // every entry with a zero count
        const bool p0_edge = p0 >= tau;
        const long long base_fix = __double2ll_rn(pi_fix * (double)p0);
        float bestv = -1.0f;
        uint32_t besti = 0xFFFFFFFFu, n_nz = 0, n_list = 0;
        double h = 0.0;
        uint32_t *lv = sm.nz_v[warp];
        uint16_t *lj = sm.nz_j[warp];
        // up to 32 entries that have a count, one per lane; in the lane behind them, the last time, those that have none
        auto take = [&](uint32_t n, bool last) {
            __syncwarp();
            const bool mine = lane < n;
            const uint32_t v = mine ? lv[lane] : 0u, j = mine ? lj[lane] : 0u;
            const float p = mine ? __fdiv_rn(__fadd_rn((float)v, eps), den) : p0;
            const double pd = (double)p, t = cs_xlogx(pd);
            if (mine) {
                if (write) {
                    ws.P[(size_t)i * A + j] = p;
                    ws.C[(size_t)i * A + j] = v;
                }
                if (p > bestv) { bestv = p; besti = j; }                       // strict: the lowest j among equals stays
                if (p >= tau) atomicOr(&sm.adj[j], 1u << warp);
                if (n_i) atomicAdd(&sm.q[j], (unsigned long long)(__double2ll_rn(pi_fix * pd) - base_fix));
                h += t;
            } else if (last && lane == n) {
                h += (double)(A - n_nz) * t;
            }
            __syncwarp();
        };
        // the entries that have a count go to the list, a word of 32 columns at a time; the rest is uniform
        uint32_t words = 0;
#pragma unroll
        for (int k = 0; k < CHUNK; ++k) {
            if (32u * k >= A) break;
            const uint32_t j = lane + 32u * k;
            if (__any_sync(0xFFFFFFFFu, c[k] != 0u)) words |= 1u << k;
            if (write && j < A) ws.P[(size_t)i * A + j] = p0;
            if (p0_edge && j < A && c[k] == 0u) atomicOr(&sm.adj[j], 1u << warp);
        }
        __syncwarp();                                                          // (an entry's P is written again by another lane)
#pragma unroll 1
        for (; words; words &= words - 1u) {
            const uint32_t k = __ffs(words) - 1u;
            uint32_t v = c[0];
#pragma unroll
            for (int u = 1; u < CHUNK; ++u) v = k == (uint32_t)u ? c[u] : v;
            const uint32_t b = __ballot_sync(0xFFFFFFFFu, v != 0u), n_b = __popc(b);
            if (n_list + n_b > 32u) { take(n_list, false); n_list = 0; }
            if (v) {
                const uint32_t at = n_list + __popc(b & ((1u << lane) - 1u));
                lv[at] = v;
                lj[at] = (uint16_t)(lane + 32u * k);
            }
            n_list += n_b;
            n_nz += n_b;
        }
#pragma unroll 1
        do {                                                                   // (twice when the list is full: the last lane has to be free)
            take(n_list, n_list < 32u);
            n_list = n_list == 32u ? 0u : 33u;
        } while (n_list != 33u);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const float v = __shfl_xor_sync(0xFFFFFFFFu, bestv, d);
            const uint32_t x = __shfl_xor_sync(0xFFFFFFFFu, besti, d);
            if (v > bestv || (v == bestv && x < besti)) { bestv = v; besti = x; }
            h += __shfl_xor_sync(0xFFFFFFFFu, h, d);
        }
        const uint32_t am = bestv > p0 ? besti : 0u;          // no entry above the zero-count ones: all are equal, the lowest wins
        if (lane == 0) {
            if (write) ws.amax[i] = (uint16_t)am;
            if (n_add) ws.rowsum[i] = n_i;
            cluster.map_shared_rank(sm.amax, 0)[i] = (uint16_t)am;
        }
        row_hc = (double)n_i * h;
        row_base = n_i ? (unsigned long long)base_fix : 0ull;
    }
    if (lane == 0) { sm.row_hc[warp] = row_hc; sm.row_base[warp] = row_base; }
    __syncthreads();
    CS_STAMP(ws, CS_PS_REFRESH_ROWS_DONE, blockIdx.x == 0 && tid == 0);

    // ---- everything meets in the first CTA -----------------------------------------------------------------------------
    RfShared<KW> *first = cluster.map_shared_rank(&sm, 0);
    if (tid < A) {
        const uint32_t bits = sm.adj[tid];
        if (KW == 8 && rank && sm.q[tid]) atomicAdd(&first->q[tid], sm.q[tid]);
        // this CTA's rows are 32, 16 or 8 bits of a word
        if (rows == 32u) first->adjT[0][tid] = bits;
        else if (rows == 16u) ((uint16_t *)&first->adjT[rank / 2u % KW][tid])[rank & 1u] = (uint16_t)bits;
        else ((uint8_t *)&first->adjT[rank / 4u % KW][tid])[rank & 3u] = (uint8_t)bits;
    }
    if (warp == rows - 1u) {
        double s = lane < rows ? sm.row_hc[lane] : 0.0;
        unsigned long long b = lane < rows ? sm.row_base[lane] : 0ull;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
            b += __shfl_xor_sync(0xFFFFFFFFu, b, d);
        }
        if (lane == 0) { first->hc[rank] = s; first->base[rank] = b; }
    }
    if (KW > 1) cluster.sync();
    else __syncthreads();
    if (rank != 0) return;
    CS_STAMP(ws, CS_PS_REFRESH_LAST_CTA, tid == 0);
    uint32_t row[KW];                                         // thread v: the predecessors of agent v
#pragma unroll
    for (int w = 0; w < KW; ++w) {
        row[w] = 0;
        if ((uint32_t)w < W && tid < A) {
            row[w] = sm.adjT[w][tid];
            ws.adjT[(size_t)w * A + tid] = row[w];            // for searches from explicit sources
        }
    }

    rf_finish<KW, ALL>(sm, ws, row, A, W, CL, n_events, n_new, n_skipped, n_total, la, r_min, e_max, delta, n_chains);
}

// The same for many agents (KW = 32): bound by the scan of the rows -- a megabyte and more of counts -- so they are spread over the
// whole GPU, 8 rows per CTA, a row's 256-column quarters by a warp each.  Column sums meet in global memory (atomics, only of
// columns some row of the CTA has a count in); 8 rows are one byte of every word of the transposed matrix, which their CTA stores
// whole (words of rows past the last one stay zero, as the workspace is made).  The CTA that is done last does the rest.
// A cluster of 16 CTAs with 32 or 64 rows each took 17.1 us for 400 agents, 28.8 for 600 and 35.3 for 1,024, most of it for
// issuing four chunks per row; this takes 13.9, 15.6 and 17.8: 5.8 the rows, 2.7 the meeting, 4 the sums, up to 4.5 the search.
// (For 256 agents or fewer the meeting in global memory costs more than it gives: 13.3 us instead of 8.5.)
template <bool ALL>
__global__ void __launch_bounds__(1024)
cs_refresh_wide_kernel(cs_workspace ws, uint32_t A, uint32_t W, float eps, float tau, float r_min, uint32_t e_max, float delta,
                       uint32_t n_chains, const uint32_t *__restrict__ ev_chain_in,
                       const uint16_t *__restrict__ ev_agent_in, const uint8_t *__restrict__ ev_flags, uint32_t n_events,
                       const uint32_t *__restrict__ n_events_dev, uint32_t every_row)
{
    constexpr int CHUNK = RfShape<32>::CHUNK;
    static_assert(CHUNK * 32u == RW_COLS, "a warp's columns are one chunk");
    __shared__ RfShared<32> sm;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    CS_STAMP(ws, CS_PS_REFRESH_ENTRY, blockIdx.x == 0 && tid == 0);
    sm.q[tid] = 0;
    sm.adj[tid] = 0;
    if (tid == 0) sm.last_live = -1;
    if (tid < OBS_FUSED_MAX) sm.succ[tid] = 0;
    if (tid < 2 * PULL_MAX_WORDS) sm.front[tid] = 0;
    cs_wait_for_predecessor();
    CS_STAMP(ws, CS_PS_REFRESH_WAITED, blockIdx.x == 0 && tid == 0);
    cs_release_successor();

    if (n_events_dev) n_events = min(n_events, cs_ld_cg_pinned(n_events_dev));
    const uint32_t r = warp >> 2, i = blockIdx.x * RW_ROWS + r, col0 = (warp & 3u) * RW_COLS;
    const uint32_t n_cols = i < A && col0 < A ? min(A - col0, RW_COLS) : 0u;
    uint32_t c[CHUNK];
#pragma unroll
    for (int k = 0; k < CHUNK; ++k) {
        const uint32_t j = lane + 32u * k;
        c[k] = 0;
        if (j < n_cols) c[k] = cs_ld_cg_pinned(ws.C + (size_t)i * A + col0 + j);
    }
    uint32_t n_i = cs_ld_cg_pinned(ws.rowsum + (i < A ? i : 0u));
    uint32_t n_total = cs_ld_cg_pinned(&ws.sc->n_transitions);
    const uint32_t la = cs_ld_cg_pinned(&ws.sc->last_agent);
    uint32_t n_new = 0, n_skipped = 0;
    rf_read_batch(sm, ws, A, n_chains, ev_chain_in, ev_agent_in, ev_flags, n_events, blockIdx.x == 0, true, n_new, n_skipped);
    n_total += n_new;
    const double inv_total = n_total ? 1.0 / (double)n_total : 0.0;

    float bestv = -1.0f;
    uint32_t besti = 0xFFFFFFFFu, n_add = 0;
    double h = 0.0;
    long long base_fix = 0;
    float p0 = 0.0f;
    if (n_cols) {                                              // (whole warps)
        if (n_new)
            for (uint32_t e0 = 0; e0 < n_events; e0 += 32u) {
                uint32_t hits = __ballot_sync(0xFFFFFFFFu, e0 + lane < n_events && sm.ev_prev[e0 + lane] == i);
                n_add += __popc(hits);
                for (; hits; hits &= hits - 1u) {
                    const uint32_t j = sm.ev_agent[e0 + __ffs(hits) - 1] - col0;
#pragma unroll
                    for (int k = 0; k < CHUNK; ++k)
                        if (j == lane + 32u * k) ++c[k];
                }
            }
        n_i += n_add;
        const bool write = every_row || n_add;
        const double pi_fix = (double)n_i * inv_total * 1152921504606846976.0;      // pi_i * 2^60
        const float den = __fadd_rn((float)n_i, __fmul_rn((float)A, eps));
        p0 = __fdiv_rn(__fadd_rn(0.0f, eps), den);                                  // every entry with a zero count
        const bool p0_edge = p0 >= tau;
        base_fix = __double2ll_rn(pi_fix * (double)p0);
        uint32_t n_nz = 0, n_list = 0, words = 0;
        uint32_t *lv = sm.nz_v[warp];
        uint16_t *lj = sm.nz_j[warp];
        auto take = [&](uint32_t n, bool last) {               // (as in cs_refresh_kernel)
            __syncwarp();
            const bool mine = lane < n;
            const uint32_t v = mine ? lv[lane] : 0u, j = mine ? lj[lane] : 0u;
            const float p = mine ? __fdiv_rn(__fadd_rn((float)v, eps), den) : p0;
            const double pd = (double)p, t = cs_xlogx(pd);
            if (mine) {
                if (write) {
                    ws.P[(size_t)i * A + j] = p;
                    ws.C[(size_t)i * A + j] = v;
                }
                if (p > bestv) { bestv = p; besti = j; }                       // strict: the lowest j among equals stays
                if (p >= tau) atomicOr(&sm.adj[j], 1u << r);
                if (n_i) atomicAdd(&sm.q[j], (unsigned long long)(__double2ll_rn(pi_fix * pd) - base_fix));
                h += t;
            } else if (last && lane == n) {
                h += (double)(n_cols - n_nz) * t;
            }
            __syncwarp();
        };
#pragma unroll
        for (int k = 0; k < CHUNK; ++k) {
            const uint32_t j = lane + 32u * k;
            if (__any_sync(0xFFFFFFFFu, c[k] != 0u)) words |= 1u << k;
            if (write && j < n_cols) ws.P[(size_t)i * A + col0 + j] = p0;
            if (p0_edge && j < n_cols && c[k] == 0u) atomicOr(&sm.adj[col0 + j], 1u << r);
        }
        __syncwarp();                                                          // (an entry's P is written again by another lane)
#pragma unroll 1
        for (; words; words &= words - 1u) {
            const uint32_t k = __ffs(words) - 1u;
            uint32_t v = c[0];
#pragma unroll
            for (int u = 1; u < CHUNK; ++u) v = k == (uint32_t)u ? c[u] : v;
            const uint32_t b = __ballot_sync(0xFFFFFFFFu, v != 0u), n_b = __popc(b);
            if (n_list + n_b > 32u) { take(n_list, false); n_list = 0; }
            if (v) {
                const uint32_t at = n_list + __popc(b & ((1u << lane) - 1u));
                lv[at] = v;
                lj[at] = (uint16_t)(col0 + lane + 32u * k);
            }
            n_list += n_b;
            n_nz += n_b;
        }
#pragma unroll 1
        do {                                                                   // (twice when the list is full: the last lane has to be free)
            take(n_list, n_list < 32u);
            n_list = n_list == 32u ? 0u : 33u;
        } while (n_list != 33u);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const float v = __shfl_xor_sync(0xFFFFFFFFu, bestv, d);
            const uint32_t x = __shfl_xor_sync(0xFFFFFFFFu, besti, d);
            if (v > bestv || (v == bestv && x < besti)) { bestv = v; besti = x; }
            h += __shfl_xor_sync(0xFFFFFFFFu, h, d);
        }
    }
    if (lane == 0) {
        sm.best_v[warp] = bestv;
        sm.best_i[warp] = besti;
        sm.row_hc[warp] = (double)n_i * h;
        sm.row_base[warp] = (warp & 3u) == 0 && n_i ? (unsigned long long)base_fix : 0ull;
    }
    __syncthreads();
    CS_STAMP(ws, CS_PS_REFRESH_ROWS_DONE, blockIdx.x == 0 && tid == 0);
    if ((warp & 3u) == 0 && lane == 0 && n_cols) {             // the row's arg-max, from its four quarters in order
        for (uint32_t u = 1; u < 4u; ++u)
            if (sm.best_v[warp + u] > bestv) { bestv = sm.best_v[warp + u]; besti = sm.best_i[warp + u]; }
        if (every_row || n_add) ws.amax[i] = (uint16_t)(bestv > p0 ? besti : 0u);   // (all entries equal: the lowest wins)
        if (n_add) ws.rowsum[i] = n_i;
    }
    if (tid < A) {
        if (sm.q[tid]) atomicAdd(ws.qsum + tid, sm.q[tid]);
        ((uint8_t *)(ws.adjT + (size_t)(blockIdx.x / 4u) * A + tid))[blockIdx.x & 3u] = (uint8_t)sm.adj[tid];
    }
    if (warp == 31u) {
        double s = sm.row_hc[lane];
        unsigned long long b = sm.row_base[lane];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
            b += __shfl_xor_sync(0xFFFFFFFFu, b, d);
        }
        if (lane == 0) { ws.cta_hc[blockIdx.x] = s; ws.cta_base[blockIdx.x] = b; }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) sm.last_cta = atomicAdd(&ws.sc->refresh_ticket, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (!sm.last_cta) return;
    __threadfence();
    CS_STAMP(ws, CS_PS_REFRESH_LAST_CTA, tid == 0);
    const unsigned long long q = tid < A ? cs_ld_cg_pinned(ws.qsum + tid) : 0ull;
    unsigned long long base = tid < gridDim.x ? cs_ld_cg_pinned(ws.cta_base + tid) : 0ull;
    double hc = tid < gridDim.x ? __longlong_as_double((long long)cs_ld_cg_pinned((const unsigned long long *)ws.cta_hc + tid)) : 0.0;
    uint32_t row[32];                                         // thread v: the predecessors of agent v
#pragma unroll
    for (int w = 0; w < 32; ++w) row[w] = ((uint32_t)w < W && tid < A) ? cs_ld_cg_pinned(ws.adjT + (size_t)w * A + tid) : 0u;
    if (warp < 4u) {                                          // (at most 128 CTAs; one number per warp is left to add up)
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            hc += __shfl_xor_sync(0xFFFFFFFFu, hc, d);
            base += __shfl_xor_sync(0xFFFFFFFFu, base, d);
        }
        if (lane == 0) { sm.hc[warp] = hc; sm.base[warp] = base; }
    }
    if (tid < A) {
        sm.q[tid] = q;
        ws.qsum[tid] = 0;
    }
    if (tid == 0) ws.sc->refresh_ticket = 0;
    __syncthreads();
    rf_finish<32, ALL>(sm, ws, row, A, W, 4u, n_events, n_new, n_skipped, n_total, la, r_min, e_max, delta, n_chains);
}

// BFS + Eq. 8 from explicit sources into the temporary tables (cs_score_blocks with sources): one thread per agent.
template <int KW>
__global__ void __launch_bounds__(KW * 32)
cs_survival_kernel(cs_workspace ws, uint32_t A, uint32_t W, const uint16_t *__restrict__ sources, uint32_t n_sources,
                   uint32_t e_max, float delta)
{
    __shared__ uint32_t s_front[2 * PULL_MAX_WORDS];
    const uint32_t tid = threadIdx.x;
    uint32_t row[KW];
    cs_wait_for_predecessor();
    cs_release_successor();
#pragma unroll
    for (int w = 0; w < KW; ++w) row[w] = ((uint32_t)w < W && tid < A) ? cs_ld_cg_pinned(ws.adjT + (size_t)w * A + tid) : 0u;
    for (uint32_t i = tid; i < 2 * PULL_MAX_WORDS; i += blockDim.x) s_front[i] = 0;
    __syncthreads();
    for (uint32_t s = tid; s < n_sources; s += blockDim.x) {
        const uint32_t a = sources[s];
        if (a < A) atomicOr(&s_front[a >> 5], 1u << (a & 31));
        else atomicOr(&ws.sc->status, CS_ST_BAD_SOURCE);
    }
    __syncthreads();
    cs_bfs_pull<KW>(row, A, W, s_front, ws.hops_tmp, ws.fsurv_tmp, e_max, delta);
}

// ---------------------------------------------------------------------------------------------
// Exact survival probability of Eq. 6 for every agent.  The unit mass at the current agent a0 is pushed through K steps
// of the chain with column a removed (mass that reaches a leaves the vector); what is left after K steps never visited a:
//     v_0 = e_{a0};  v_{t+1}[j] = sum_i v_t[i] P[i][j] (j != a), v_{t+1}[a] = 0;
//     p = sum_t sum_i v_t[i] P[i][a]  (= 1 - sum_j v_K[j]).
// The probability is accumulated as the mass absorbed at the target step by step (no 1 - x cancellation, so small
// probabilities keep full relative accuracy), in fp64 over the canonical fp32 matrix.  The paper treats this as too
// expensive for its per-request runtime and uses the hop proxy of Eq. 8; here it is an alternative scorer.
//
// A step for all targets is a product V (targets x agents) * P with another column zeroed in every row, so it is tiled
// like one: a cluster advances 8 targets together and splits the columns among its CTAs (every CTA keeps the whole of V
// for its targets in shared memory, [agent][target], and its columns of the new V go to every CTA of the cluster through
// distributed shared memory); inside a CTA a warp owns 64 columns (two per lane, 16 accumulators) and a slice of the
// agents summed over, so that 16 warps stay busy however few the columns; the slices' partial sums meet in shared memory.
// P comes from global memory (a CTA on its own finds its columns in its L1 in the later steps; a cluster barrier makes L1 forget
// them).  The last step needs column a only: one dot product per target, one warp each.
//
// Bound by the fp64 pipe for many agents (2 A^3 (K - 2) operations), by latency for few.  256 agents, K = 4: 62.7 us with
// one CTA per 8 targets that walked the matrix column by column (32 CTAs, one serial chain of 256 loads per step),
// 13.4 us per call like this (128 CTAs).  Few agents, one CTA, K = 32, with cluster barriers / with its own: 4 agents 42 / 17 us,
// 12 44 / 25, 64 85 / 42.
// ---------------------------------------------------------------------------------------------
#define XS_TARGETS 8u
#define XS_THREADS 512u
#define XS_WARPS (XS_THREADS / 32u)
#define XS_PART_ROW 68u                  // 64 columns of one target, padded: the reduction reads without bank conflicts
#define XS_MAX_CLUSTER 8u                // the portable limit
static size_t xs_smem_bytes(uint32_t A)
{
    return (2 * (size_t)A * XS_TARGETS + XS_WARPS * XS_TARGETS * XS_PART_ROW) * sizeof(double);
}

template <bool ONE>          // one CTA does all columns of its targets; else a cluster shares them
__global__ void __launch_bounds__(XS_THREADS, 1)
cs_exact_survival_kernel(cs_workspace ws, uint32_t A, uint32_t a0_arg, uint32_t K, uint32_t n_cols, float delta,
                         float *__restrict__ psurv_out, float *__restrict__ fsurv_out)
{
    extern __shared__ __align__(16) double s_xs[];
    double *const v_all = s_xs;                                    // [2][A][XS_TARGETS]
    double *const part = s_xs + 2 * (size_t)A * XS_TARGETS;        // [XS_WARPS][XS_TARGETS][XS_PART_ROW]
    __shared__ double s_hit[XS_TARGETS];
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t base = (blockIdx.x / CL) * XS_TARGETS;          // this cluster's targets
    const uint32_t col0 = rank * n_cols, col1 = min(col0 + n_cols, A);
    const float *__restrict__ P = ws.P;
    cs_wait_for_predecessor();
    cs_release_successor();
    const uint32_t a0 = a0_arg == CS_AGENT_NONE ? ws.sc->last_agent : a0_arg;
    const bool any = a0 < A && K > 0;
    auto owner = [&](uint32_t a) { return a >= col0 && a < col1; };  // this CTA holds column a
    if (tid < XS_TARGETS) s_hit[tid] = (any && base + tid < A) ? (double)P[(size_t)a0 * A + base + tid] : 0.0;
    if (any) {
        // step 1: every target starts from the unit mass at a0, i.e. from row a0 of the matrix
        for (uint32_t e = tid; e < A * XS_TARGETS; e += XS_THREADS) {
            const uint32_t j = e / XS_TARGETS, m = e % XS_TARGETS;
            v_all[e] = j == base + m ? 0.0 : (double)P[(size_t)a0 * A + j];
        }
        // (no slice of fewer than eight agents, because the slices' sums are added up one after the other: 64 agents, K = 32 41.5 us, with
        // four 50.8)
        const uint32_t col_warps = (n_cols + 63u) / 64u, slices = min(XS_WARPS / col_warps, max(2u, (A + 7u) / 8u));
        const uint32_t cw = warp % col_warps, sl = warp / col_warps;
        // (a CTA on its own keeps to its own barrier: a cluster's makes its L1 forget the matrix)
        const auto everywhere = [&] { if (ONE) __syncthreads(); else cluster.sync(); };
        everywhere();                                              // (also: every CTA has started before its memory is written)
        uint32_t cur = 0;
        for (uint32_t t = 1; t + 1 < K; ++t) {
            const double *v = v_all + (size_t)cur * A * XS_TARGETS;
            double *const nxt = v_all + (size_t)(cur ^ 1u) * A * XS_TARGETS;
            cur ^= 1u;
            if (sl < slices) {
                const uint32_t j0 = col0 + cw * 64u + lane, j1 = j0 + 32u, i_end = (sl + 1u) * A / slices;
                const float *p0 = P + (j0 < col1 ? j0 : 0u), *p1 = P + (j1 < col1 ? j1 : 0u);    // (columns past the end: unused)
                double acc0[XS_TARGETS], acc1[XS_TARGETS];
#pragma unroll
                for (uint32_t m = 0; m < XS_TARGETS; ++m) acc0[m] = acc1[m] = 0.0;
#pragma unroll 8
                for (uint32_t i = sl * A / slices; i < i_end; ++i) {
                    const double x0 = (double)__ldg(p0 + (size_t)i * A), x1 = (double)__ldg(p1 + (size_t)i * A);
                    const double2 *vi = (const double2 *)(v + (size_t)i * XS_TARGETS);
#pragma unroll
                    for (uint32_t h = 0; h < XS_TARGETS / 2; ++h) {
                        const double2 y = vi[h];
                        acc0[2 * h] = fma(y.x, x0, acc0[2 * h]);
                        acc0[2 * h + 1] = fma(y.y, x0, acc0[2 * h + 1]);
                        acc1[2 * h] = fma(y.x, x1, acc1[2 * h]);
                        acc1[2 * h + 1] = fma(y.y, x1, acc1[2 * h + 1]);
                    }
                }
                double *o = part + (size_t)warp * XS_TARGETS * XS_PART_ROW + lane;
#pragma unroll
                for (uint32_t m = 0; m < XS_TARGETS; ++m) { o[m * XS_PART_ROW] = acc0[m]; o[m * XS_PART_ROW + 32u] = acc1[m]; }
            }
            __syncthreads();
            for (uint32_t e = tid; e < (col1 > col0 ? col1 - col0 : 0u) * XS_TARGETS; e += XS_THREADS) {
                const uint32_t jc = e / XS_TARGETS, m = e % XS_TARGETS, j = col0 + jc;
                const double *q = part + (size_t)(jc / 64u) * XS_TARGETS * XS_PART_ROW + m * XS_PART_ROW + jc % 64u;
                double sum = 0.0;
                for (uint32_t u = 0; u < slices; ++u) sum += q[(size_t)u * col_warps * XS_TARGETS * XS_PART_ROW];
                if (j == base + m) { s_hit[m] += sum; sum = 0.0; }   // (one thread per target)
                if (ONE)
                    nxt[(size_t)j * XS_TARGETS + m] = sum;
                else
                    for (uint32_t r = 0; r < CL; ++r) cluster.map_shared_rank(nxt, r)[(size_t)j * XS_TARGETS + m] = sum;
            }
            everywhere();                                          // the new V is complete everywhere; `part` is free again
        }
        if (K > 1 && warp < XS_TARGETS && base + warp < A && owner(base + warp)) {
            const double *v = v_all + (size_t)cur * A * XS_TARGETS + warp;
            double sum = 0.0;
            for (uint32_t i = lane; i < A; i += 32u) sum = fma(v[(size_t)i * XS_TARGETS], (double)__ldg(P + (size_t)i * A + base + warp), sum);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
            if (lane == 0) s_hit[warp] += sum;
        }
    }
    __syncthreads();
    if (tid < XS_TARGETS && base + tid < A && owner(base + tid)) {
        if (psurv_out) psurv_out[base + tid] = (float)s_hit[tid];
        if (fsurv_out) fsurv_out[base + tid] = (float)(s_hit[tid] + (double)delta);
    }
}

// ---------------------------------------------------------------------------------------------
// The same table with one product less.  A path's first visit to a splits its later ones off: with g_n = P^n[a0][a] and d_n = P^n[a][a],
//     f_n = g_n - sum_{t < n} f_t d_{n-t}   is the probability that step n is the first at a, and p = f_1 + ... + f_K.
// All of g and d come from the columns w_n = P^n[:, a], which are the same product for every start and with nothing removed:
//     g_n = w_n[a0], d_n = w_n[a] for n <= K - 2;  g_{K-1} = r_1 w_{K-2}, g_K = r_2 w_{K-2}, d_{K-1} = P[a, :] w_{K-2},
// r_1 and r_2 being rows a0 of P and P^2.  So w_{K-2} is enough, K - 3 products; r_2 is summed up from the tiles of P that the first of them brings.
// The differences lose nothing that p has: every term of f_n is at most p, so what f_n is off by, before it goes on, is at most n roundings of p,
// and it goes on as e_n = delta_n - sum e_t d_{n-t}, which the renewal equation sums to at most twice the deltas' sum.
//
// (Against extended precision, matrices of 4 to 256 agents, dense, sparse, nearly a chain, agents that mostly follow themselves, and of entries from 1e-12
// to 1: relative to p, the way above is within 3e-15 and this one within 1e-14, and after the rounding to fp32 the largest errors are the same to three digits, 6e-8.)
//
// Clusters as above, but a warp multiplies 16 rows by a slice of the agents with matrix instructions (m16n8k8; rows of the new w by the agents summed
// over, times 8 targets), so that few slices are left to add up and the vectors are read from shared memory once for 16 rows.  Bound by the fp64 pipe
// (64 rows, 256 agents, 8 targets: 2.1 us at 32 multiply-adds per clock and SM) and, as much again, by the exchange between two products.  us per call, products above /
// here: K = 4 65 agents 8.3 / 7.3, 128 9.5 / 8.2, 256 13.5 / 10.9, 400 36.7 / 28.7; K = 6 13.2 / 10.2, 15.1 / 13.5, 22.0 / 19.7, 67.8 / 53.9.  Warps of 64
// rows and short slices: 256 agents 11.9; two chains of instructions per warp 11.2.
// Fewer steps than four have no product to save (r_2 costs what it saves with three: 400 agents 21.4 / 23.8), and one CTA's agents (64 at most) are
// bound by the steps' latency (12 agents 4.4 / 4.5, six steps 5.9 / 7.0): they go as above.
// ---------------------------------------------------------------------------------------------
#define XS_ROWS 16u                      // rows of a warp's tile
#define XS_DEEP 4u                       // instructions of eight agents whose part of the matrix is in flight
#define XS_ROWS_PAD 18u                  // 16 rows of one target, padded: written and summed without bank conflicts
#define XS_RENEWAL_STEPS 32u             // a lane per step in the end
#define XS_SMEM_MOST (227u * 1024u - 256u)
static size_t xs_renewal_smem(uint32_t A, uint32_t cl)
{
    return (2 * (size_t)A * XS_TARGETS + XS_WARPS * XS_TARGETS * XS_ROWS_PAD + (cl + 1u) * (size_t)A + XS_WARPS * 32u + 2u * XS_TARGETS * XS_RENEWAL_STEPS) * sizeof(double);
}
// c += a b: 16 x 8 by 8 x 8.  Lane l: a rows l/4 (a0, a2) and l/4 + 8 (a1, a3), columns l%4 (a0, a1) and l%4 + 4 (a2, a3); b rows l%4 and
// l%4 + 4, column l/4; c rows l/4 (c0, c1) and l/4 + 8 (c2, c3), columns 2 (l%4) and 2 (l%4) + 1.
__device__ __forceinline__ void mma_f64(double (&c)[4], double a0, double a1, double a2, double a3, double b0, double b1)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3]) : "d"(a0), "d"(a1), "d"(a2), "d"(a3), "d"(b0), "d"(b1));
}
// A probability of the matrix times 2^-896: a float's bits in a double's place, which costs no conversion and is exact for every finite float, denormal ones
// too (the smoothing keeps entries above 0, about eps / n of a row).  The vectors that it is
// multiplied with are kept times 2^896.  (A product of 64 rows, 256 agents and 8 targets 0.3 us less.)
#define XS_UP 0x1p896
#define XS_DOWN 0x1p-896
__device__ __forceinline__ double scaled_down(float x)
{
    const uint32_t b = __float_as_uint(x);
    return __hiloint2double((int)(b >> 3), (int)(b << 29));
}
__device__ __forceinline__ double warp_sum(double x)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, d);
    return x;
}

__global__ void __launch_bounds__(XS_THREADS, 1)
cs_renewal_survival_kernel(cs_workspace ws, uint32_t A, uint32_t a0_arg, uint32_t K, uint32_t n_rows, float delta,
                           float *__restrict__ psurv_out, float *__restrict__ fsurv_out)
{
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t row_warps = (n_rows + XS_ROWS - 1u) / XS_ROWS;            // (at most 16)
    extern __shared__ __align__(16) double s_xs[];
    double *const w_all = s_xs;                                    // [2][A][XS_TARGETS]
    double *const part = w_all + 2 * (size_t)A * XS_TARGETS;       // [XS_WARPS][XS_TARGETS][XS_ROWS_PAD]
    double *const r2_part = part + XS_WARPS * XS_TARGETS * XS_ROWS_PAD;      // [XS_WARPS][32]: r_2 over some of the CTA's rows,
    double *const r2 = r2_part + XS_WARPS * 32u;                   // [CL][A]: over all of each CTA's
    double *const r1 = r2 + (size_t)CL * A;                        // [A]
    double *const s_g = r1 + A, *const s_d = s_g + XS_TARGETS * XS_RENEWAL_STEPS;      // [XS_TARGETS][XS_RENEWAL_STEPS]
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t base = (blockIdx.x / CL) * XS_TARGETS;          // this cluster's targets
    const uint32_t row0 = min(rank * n_rows, A), row1 = min(row0 + n_rows, A);
    const float *__restrict__ P = ws.P;
    // this CTA holds the rows of the target that is this warp's
    const uint32_t a = base + warp;
    const bool mine = warp < XS_TARGETS && a < A && a >= row0 && a < row1;
    cs_wait_for_predecessor();
    cs_release_successor();
    const uint32_t a0 = a0_arg == CS_AGENT_NONE ? ws.sc->last_agent : a0_arg;
    double p = 0.0;
    if (a0 < A) {
        for (uint32_t e = tid; e < A * XS_TARGETS; e += XS_THREADS) {
            const uint32_t j = e / XS_TARGETS, m = e % XS_TARGETS;
            w_all[e] = base + m < A ? (double)P[(size_t)j * A + base + m] * XS_UP : 0.0;
        }
        for (uint32_t j = tid; j < A; j += XS_THREADS) r1[j] = (double)P[(size_t)a0 * A + j];
        const uint32_t slices = XS_WARPS / row_warps, rw = warp % row_warps, sl = warp / row_warps;
        const uint32_t groups = (A + 7u) / 8u, i_first = sl * groups / slices * 8u, i_end = sl < slices ? min((sl + 1u) * groups / slices * 8u, A) : i_first;
        const uint32_t row = lane / 4u, depth = lane % 4u, j0 = row0 + rw * XS_ROWS + row;               // a lane's place in the operands
        float next[XS_DEEP][4];                                    // of the matrix, on its way
        const auto ask = [&](uint32_t i0) {
#pragma unroll
            for (uint32_t x = 0; x < XS_DEEP; ++x)
#pragma unroll
                for (uint32_t q = 0; q < 4u; ++q) {
                    const uint32_t i = i0 + 8u * x + depth + 4u * (q >> 1), j = j0 + 8u * (q & 1u);
                    next[x][q] = i < i_end && j < row1 ? __ldg(P + (size_t)j * A + i) : 0.0f;
                }
        };
        ask(i_first);
        float own[8];                                              // the target's row of the matrix
#pragma unroll
        for (uint32_t h = 0; h < 8u; ++h) own[h] = mine && lane + 32u * h < A ? __ldg(P + (size_t)a * A + lane + 32u * h) : 0.0f;
        cluster.sync();                                            // (also: every CTA has started before its memory is written)
        uint32_t cur = 0;
        const auto note = [&](uint32_t n) {                        // w_{n + 1} at a0 and at its own target
            const double *w = w_all + (size_t)cur * A * XS_TARGETS;
            if (tid < XS_TARGETS && base + tid < A) {
                s_g[tid * XS_RENEWAL_STEPS + n] = w[(size_t)a0 * XS_TARGETS + tid] * XS_DOWN;
                s_d[tid * XS_RENEWAL_STEPS + n] = w[(size_t)(base + tid) * XS_TARGETS + tid] * XS_DOWN;
            }
        };
        for (uint32_t t = 0; t + 3u < K; ++t) {
            const double *w = w_all + (size_t)cur * A * XS_TARGETS;
            double *const nxt = w_all + (size_t)(cur ^ 1u) * A * XS_TARGETS;
            note(t);
            if (sl < slices) {
                double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
                for (uint32_t i0 = i_first; i0 < i_end; i0 += 8u * XS_DEEP) {
                    float now[XS_DEEP][4];
#pragma unroll
                    for (uint32_t x = 0; x < XS_DEEP; ++x)
#pragma unroll
                        for (uint32_t q = 0; q < 4u; ++q) now[x][q] = next[x][q];
                    if (i0 + 8u * XS_DEEP < i_end) ask(i0 + 8u * XS_DEEP);
                    else if (t + 4u < K) ask(i_first);             // (the next product's)
#pragma unroll
                    for (uint32_t x = 0; x < XS_DEEP; ++x) {
                        const uint32_t i = i0 + 8u * x + depth;
                        if (i0 + 8u * x < i_end)                   // (past the end: times zero)
                            mma_f64(acc, scaled_down(now[x][0]), scaled_down(now[x][1]), scaled_down(now[x][2]), scaled_down(now[x][3]),
                                    w[(size_t)min(i, A - 1u) * XS_TARGETS + row], w[(size_t)min(i + 4u, A - 1u) * XS_TARGETS + row]);
                    }
                }
                double *o = part + (size_t)warp * XS_TARGETS * XS_ROWS_PAD + row;
#pragma unroll
                for (uint32_t q = 0; q < 4u; ++q) o[(2u * depth + (q & 1u)) * XS_ROWS_PAD + 8u * (q >> 1)] = acc[q];
            }
            // r_2 over this CTA's rows, which the products above have brought to its L1: 32 agents per warp, what warps are over share the rows
            const uint32_t chunks = (A + 31u) / 32u, sharers = max(1u, XS_WARPS / chunks), share = warp / chunks;
            if (t == 0u && share < sharers)
                for (uint32_t c = warp % chunks; c < chunks; c += XS_WARPS) {
                    const uint32_t i = min(32u * c + lane, A - 1u), j_end = row0 + (row1 - row0) * (share + 1u) / sharers;
                    double s0 = 0.0, s1 = 0.0;
                    uint32_t j = row0 + (row1 - row0) * share / sharers;
#pragma unroll 8
                    for (; j + 1u < j_end; j += 2u) {
                        s0 = fma(r1[j], scaled_down(__ldg(P + (size_t)j * A + i)), s0);
                        s1 = fma(r1[j + 1u], scaled_down(__ldg(P + (size_t)(j + 1u) * A + i)), s1);
                    }
                    if (j < j_end) s0 = fma(r1[j], scaled_down(__ldg(P + (size_t)j * A + i)), s0);
                    if (sharers > 1u) r2_part[32u * warp + lane] = s0 + s1;
                    else if (32u * c + lane < A)
                        for (uint32_t r = 0; r < CL; ++r) cluster.map_shared_rank(r2, r)[(size_t)rank * A + i] = s0 + s1;
                }
            __syncthreads();
            for (uint32_t e = tid; e < (row1 - row0) * XS_TARGETS; e += XS_THREADS) {
                const uint32_t jc = e / XS_TARGETS, m = e % XS_TARGETS;
                const double *q = part + (size_t)(jc / XS_ROWS) * XS_TARGETS * XS_ROWS_PAD + m * XS_ROWS_PAD + jc % XS_ROWS;
                double sum = 0.0;
#pragma unroll 4
                for (uint32_t u = 0; u < slices; ++u) sum += q[(size_t)u * row_warps * XS_TARGETS * XS_ROWS_PAD];
                for (uint32_t r = 0; r < CL; ++r) cluster.map_shared_rank(nxt, r)[(size_t)(row0 + jc) * XS_TARGETS + m] = sum * XS_UP;
            }
            if (t == 0u && sharers > 1u)
                for (uint32_t i = tid; i < A; i += XS_THREADS) {
                    double sum = 0.0;
                    for (uint32_t u = 0; u < sharers; ++u) sum += r2_part[32u * (u * chunks + i / 32u) + i % 32u];
                    for (uint32_t r = 0; r < CL; ++r) cluster.map_shared_rank(r2, r)[(size_t)rank * A + i] = sum;
                }
            cluster.sync();                                        // the new w is complete everywhere; `part` is free again
            cur ^= 1u;
        }
        note(K - 3u);
        __syncthreads();
        if (mine) {
            const double *w = w_all + (size_t)cur * A * XS_TARGETS + warp;
            double x1 = 0.0, x2 = 0.0, x3 = 0.0;
#pragma unroll 1
            for (uint32_t i0 = 0; i0 < A; i0 += 256u)
#pragma unroll
                for (uint32_t h = 0; h < 8u; ++h) {
                    const uint32_t i = i0 + lane + 32u * h;
                    if (i >= A) continue;
                    const double y = w[(size_t)i * XS_TARGETS];
                    double r = 0.0;
                    for (uint32_t c = 0; c < CL; ++c) r += r2[(size_t)c * A + i];
                    x1 = fma(r1[i], y * XS_DOWN, x1);
                    x2 = fma(r, y, x2);                            // (r_2 is scaled down)
                    x3 = fma(scaled_down(i0 ? __ldg(P + (size_t)a * A + i) : own[h]), y, x3);
                }
            x1 = warp_sum(x1);
            x2 = warp_sum(x2);
            x3 = warp_sum(x3);
            // step lane + 1: its g, from which the steps before it are taken in turn, and its d
            double f = lane + 2u < K ? s_g[warp * XS_RENEWAL_STEPS + lane] : x2, d = lane + 2u < K ? s_d[warp * XS_RENEWAL_STEPS + lane] : x3;
            if (lane + 2u == K) f = x1;
            for (uint32_t n = 0; n < K; ++n) {
                const double f_n = __shfl_sync(0xFFFFFFFFu, f, n), d_n = __shfl_sync(0xFFFFFFFFu, d, (lane - n - 1u) & 31u);
                p += f_n;
                if (lane > n) f = fma(-f_n, d_n, f);
            }
        }
    }
    if (mine && lane == 0) {
        if (psurv_out) psurv_out[a] = (float)p;
        if (fsurv_out) fsurv_out[a] = (float)(p + (double)delta);
    }
}

int cs_launch_exact_survival(cs_ctx *ctx, uint32_t a0, uint32_t K, float *psurv_out, float *fsurv_out, cudaStream_t s)
{
    const cs_params &p = ctx->p;
    static std::mutex mu;
    static bool opted[64];                                  // shared-memory opt-in, once per process and device
    {
        std::lock_guard<std::mutex> lock(mu);
        if (ctx->device < 0 || ctx->device >= 64) return CS_EINVAL;
        if (!opted[ctx->device]) {
            const int most = (int)xs_smem_bytes(CS_MAX_AGENTS);
            cudaError_t e = cudaFuncSetAttribute(cs_exact_survival_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(cs_exact_survival_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(cs_renewal_survival_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)XS_SMEM_MOST);
            if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
            opted[ctx->device] = true;
        }
    }
    // as many CTAs per cluster as give each at least 64 columns and still fit one wave
    const uint32_t n_clusters = (p.n_agents + XS_TARGETS - 1) / XS_TARGETS;
    uint32_t cl = 1;
    while (cl < XS_MAX_CLUSTER && p.n_agents > 64u * cl && 2u * cl * n_clusters <= (uint32_t)ctx->sm_count) cl *= 2;
    const uint32_t n_cols = (p.n_agents + cl - 1) / cl;
    const size_t smem = xs_renewal_smem(p.n_agents, cl);
    if (cl > 1u && n_cols <= XS_WARPS * XS_ROWS && K >= 4u && K <= XS_RENEWAL_STEPS && smem <= XS_SMEM_MOST) {
        cs_launch_chained_clusters(cs_renewal_survival_kernel, n_clusters * cl, cl, XS_THREADS, smem, s, ctx->ws, p.n_agents, a0, K, n_cols, p.delta,
                                   psurv_out, fsurv_out);
        return cs_check_launch(ctx);
    }
    cs_launch_chained_clusters(cl == 1u ? cs_exact_survival_kernel<true> : cs_exact_survival_kernel<false>, n_clusters * cl, cl > 1u ? cl : 0u,
                               XS_THREADS, xs_smem_bytes(p.n_agents), s, ctx->ws, p.n_agents, a0, K, n_cols, p.delta, psurv_out, fsurv_out);
    return cs_check_launch(ctx);
}

// ---------------------------------------------------------------------------------------------
// Restores learner state saved with cs_get_model(): counts, per-chain current agents, last agent.
// Row sums and the transition total are recomputed from the counts (one CTA per row; integer
// atomics, so the total does not depend on arrival order).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(ROW_THREADS)
cs_import_kernel(cs_workspace ws, uint32_t A, uint32_t n_chains, const uint32_t *__restrict__ C_in,
                 const uint16_t *__restrict__ cur_in, uint32_t last_agent)
{
    __shared__ uint32_t s_red[ROW_THREADS];
    const uint32_t tid = threadIdx.x;
    if (blockIdx.x == 0) {
        if (tid == 0) { ws.sc->last_agent = last_agent < A ? last_agent : CS_AGENT_NONE; }
        for (uint32_t c = tid; c < n_chains; c += ROW_THREADS) {
            const uint32_t a = cur_in ? cur_in[c] : CS_AGENT_NONE;
            ws.cur[c] = (uint16_t)(a < A ? a : CS_AGENT_NONE);
        }
    }
    for (uint32_t i = blockIdx.x; i < A; i += gridDim.x) {
        uint32_t part = 0;
        for (uint32_t j = tid; j < A; j += ROW_THREADS) {
            const uint32_t v = (i == j) ? 0u : C_in[i * A + j];      // a self transition is never counted
            ws.C[i * A + j] = v;
            part += v;
        }
        const uint32_t n_i = cs_block_sum<uint32_t>(part, s_red);
        if (tid == 0) {
            ws.rowsum[i] = n_i;
            atomicAdd(&ws.sc->n_transitions, n_i);
        }
    }
}

int cs_launch_import(cs_ctx *ctx, const uint32_t *C_in, const uint16_t *cur_in, uint32_t last_agent, cudaStream_t s)
{
    const cs_params &p = ctx->p;
    cudaError_t e = cudaMemsetAsync(&ctx->ws.sc->n_transitions, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
    const uint32_t grid = p.n_agents < 2u * (uint32_t)ctx->sm_count ? p.n_agents : 2u * (uint32_t)ctx->sm_count;
    cs_import_kernel<<<grid, ROW_THREADS, 0, s>>>(ctx->ws, p.n_agents, p.n_chains, C_in, cur_in, last_agent);
    int rc = cs_check_launch(ctx);
    if (rc != CS_OK) return rc;
    return cs_launch_observe(ctx, nullptr, nullptr, nullptr, 0, s);      // refresh everything derived from the counts
}

// ---------------------------------------------------------------------------------------------
int cs_launch_init(cs_ctx *ctx, cudaStream_t s)
{
    const cs_params &p = ctx->p;
    cs_init_kernel<<<64, 256, 0, s>>>(ctx->ws, p.n_agents, p.n_chains, ctx->gtab_len, p.lambda, p.delta);
    int rc = cs_check_launch(ctx);
    if (rc != CS_OK) return rc;
    cs_gtab_check_kernel<<<1, 256, 0, s>>>(ctx->ws, ctx->gtab_len, ctx->age_sat, p.lambda, p.delta);
    if ((rc = cs_check_launch(ctx)) != CS_OK) return rc;
    return cs_launch_observe(ctx, nullptr, nullptr, nullptr, 0, s);
}

// Largest cluster (a power of two) a kernel can run as on a device, 0 when the driver would not say that any fits; asked once per
// process and device, with that device current.
struct ClusterLimit {
    std::mutex mu;
    int known[64];                                            // 0: not asked yet
    template <class Kernel> uint32_t get(int device, Kernel kernel, int most, int threads)
    {
        if (device < 0 || device >= 64) return 0;
        std::lock_guard<std::mutex> lock(mu);
        if (!known[device]) known[device] = cs_probe_cluster(kernel, most, threads, 0, 1);
        return known[device] > 0 ? (uint32_t)known[device] : 0u;
    }
};
static uint32_t obs_cluster_limit(int device)
{
    static ClusterLimit limit;
    return limit.get(device, cs_observe_kernel, OBS_MAX_CLUSTER, OBS_THREADS);
}
static uint32_t refresh_cluster_limit(int device)
{
    static ClusterLimit limit[2];
    const uint32_t last = limit[0].get(device, cs_refresh_kernel<8, false>, RfShape<8>::CTAS, RfShape<8>::WARPS * 32);
    const uint32_t all = limit[1].get(device, cs_refresh_kernel<8, true>, RfShape<8>::CTAS, RfShape<8>::WARPS * 32);
    return last < all ? last : all;
}

int cs_launch_observe(cs_ctx *ctx, const uint32_t *chain, const uint16_t *agent, const uint8_t *evflags,
                      uint32_t n_events, cudaStream_t s)
{
    const cs_params &p = ctx->p;
    const bool fused = n_events <= OBS_FUSED_MAX;             // small batches ride along with the refresh
    if (n_events && !fused) {
        // one event per thread and round: no more CTAs than the batch fills
        const uint32_t most = obs_cluster_limit(ctx->device);
        uint32_t cl = 1;
        while (cl < most && cl * OBS_THREADS < n_events) cl <<= 1;
        cs_launch_chained_clusters(cs_observe_kernel, cl, cl > 1u ? cl : 0u, OBS_THREADS, 0, s, ctx->ws, p.n_agents, p.n_chains, chain, agent,
                                   evflags, n_events, ctx->step_n_events_dev);
        int rc = cs_check_launch(ctx);
        if (rc != CS_OK) return rc;
    }
    const bool all = ctx->source_mode == CS_SOURCES_ALL_CHAINS;
    if (!fused) chain = nullptr, agent = nullptr, evflags = nullptr;
    const uint32_t n_fused = fused ? n_events : 0u;
    const uint32_t *n_fused_dev = fused ? ctx->step_n_events_dev : nullptr;
    const uint32_t every_row = n_fused ? 0u : 1u;            // a row keeps its P when no event of a small batch starts at it
    const auto launch = [&](auto kernel, uint32_t ctas, uint32_t cluster, uint32_t warps) {
        cs_launch_chained_clusters(kernel, ctas, cluster, warps * 32u, 0, s, ctx->ws, p.n_agents, ctx->W, p.eps, p.tau, p.r_min,
                                   p.e_max, p.delta, p.n_chains, chain, agent, evflags, n_fused, n_fused_dev, every_row);
    };
    const uint32_t most = refresh_cluster_limit(ctx->device);
    if (p.n_agents <= 32) {
        // one CTA of as many warps as there are rows, at least one thread per event of a small batch
        launch(all ? cs_refresh_kernel<1, true> : cs_refresh_kernel<1, false>, 1u, 1u, p.n_agents <= 8 ? 8u : (p.n_agents <= 16 ? 16u : 32u));
    } else if (p.n_agents <= RfShape<8>::COLS && p.n_agents <= RfShape<8>::WARPS * most) {
        // few rows per CTA (64 agents: 8.8 us with 32, 7.4 with 16, 6.8 with 8), as far as the cluster goes
        const uint32_t rows = p.n_agents <= 8u * most ? 8u : RfShape<8>::WARPS;
        uint32_t cl = 2;
        while (cl * rows < p.n_agents) cl <<= 1;
        launch(all ? cs_refresh_kernel<8, true> : cs_refresh_kernel<8, false>, cl, cl, rows);
    } else {
        launch(all ? cs_refresh_wide_kernel<true> : cs_refresh_wide_kernel<false>, (p.n_agents + RW_ROWS - 1u) / RW_ROWS, 0u, 32u);
    }
    return cs_check_launch(ctx);
}

int cs_launch_survival(cs_ctx *ctx, const uint16_t *sources, uint32_t n_sources, cudaStream_t s)
{
    const cs_params &p = ctx->p;
    const dim3 block(32u * ctx->W);
    const auto launch = [&](auto kernel) {
        cs_launch_chained(kernel, 1, block, 0, s, ctx->ws, p.n_agents, ctx->W, sources, n_sources, p.e_max, p.delta);
    };
    if (ctx->W == 1) launch(cs_survival_kernel<1>);
    else if (ctx->W <= 8) launch(cs_survival_kernel<8>);
    else launch(cs_survival_kernel<32>);
    return cs_check_launch(ctx);
}
