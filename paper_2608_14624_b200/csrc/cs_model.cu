// Transition Learner and Survival Scorer state: transition counting (Algorithm 1,
// ObserveTouch), Eq. 3 normalisation with row arg-max (Eq. 5 / Eq. 10), predictability
// (Eq. 2) and gate (Eq. 11), threshold graph (Eq. 7), BFS hop table and survival scores
// (Eq. 8).  The model is tiny (A <= 1024), so these kernels are latency-bound: the design
// goal is few launches and no host round trip, not bandwidth.
#include <mutex>

#include <cooperative_groups.h>

#include "cs_common.cuh"

namespace cg = cooperative_groups;

#define OBS_THREADS 1024
#define ROW_THREADS 256
#define OBS_FUSED_MAX 256u     // events up to which a batch is applied inside the refresh launch (one per thread)
static_assert(OBS_FUSED_MAX == ROW_THREADS, "the refresh kernel stages one event per thread");

// ---------------------------------------------------------------------------------------------
// Initial state of Algorithm 1: zero counts, no current agent; plus the recency table.
// ---------------------------------------------------------------------------------------------
__global__ void cs_init_kernel(cs_workspace ws, uint32_t A, uint32_t n_chains, uint32_t gtab_len, float lambda,
                               float delta)
{
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    for (uint32_t i = tid; i < A * A; i += nth) ws.C[i] = 0;
    for (uint32_t i = tid; i < A; i += nth) { ws.rowsum[i] = 0; ws.qfix[i] = 0; }
    for (uint32_t i = tid; i < n_chains; i += nth) ws.cur[i] = CS_AGENT_NONE;
    for (uint32_t i = tid; i < CS_HIST_BINS; i += nth) ws.hist[i] = 0;
    for (uint32_t i = tid; i <= CS_MAX_SPLITTERS; i += nth) CS_BCOUNT(ws, i) = 0;
    for (uint32_t i = tid; i < gtab_len; i += nth) ws.gtab[i] = cs_recency(lambda, delta, i);
    if (tid == 0) {
        cs_scalars z;
        memset(&z, 0, sizeof(z));
        z.last_agent = CS_AGENT_NONE;
        z.a_star = 0xFFFFFFFFu;
        z.sel_hint[0] = z.sel_hint[1] = z.sel_hint[2] = z.sel_hint[3] = 0xFFFFFFFFu;
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
        cluster.sync();                                          // every table of the cluster is complete
        if (need_far) {
            for (int r = (int)rank - 1; r >= 0 && prev == CS_AGENT_NONE; --r) {
                const ObsShare *o = cluster.map_shared_rank(&sh, r);
                const uint32_t s = obs_find(o->h_chain, c);
                if (s < OBS_HASH) prev = o->h_last[s];
            }
            if (prev == CS_AGENT_NONE) prev = __ldcg(&ws.cur[c]);
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
        cluster.sync();                                          // every read of cur[] and of the tables precedes the writes below
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
// BFS over the bit-matrix graph from a set of source bits, then Eq. 8.  Runs inside one CTA.
// s_front: 64 words (two frontiers, used in turn), s_visit / s_next: 32 words each, s_hops: one entry per agent.
//
// Up to one agent per thread the search PULLS: thread v holds row v of the TRANSPOSED adjacency matrix (the
// predecessors of v; kept up to date in global memory by the refresh, fetched ahead of time into registers) and at
// every level ANDs it with the frontier.  A level is then W broadcast loads and ANDs per node, all nodes in
// parallel, one ballot per warp for the next frontier and ONE barrier -- whatever the frontier size, with no
// atomics and no divergent loops.  (A push over the frontier's nodes by one warp was tried: lanes that walk
// different frontier words run one after the other, 80 cycles per node.  So was a transpose built in shared memory
// by this CTA: 3 us of shared-memory atomics.)
// More agents take the level-synchronous push from global memory: a node of the current frontier ORs its adjacency
// row into the next frontier (shared-memory atomics), two barriers per level.
// ---------------------------------------------------------------------------------------------
#define BFS_ROW_WORDS 8u                   // words of a row when the search pulls (one agent per thread: 256 agents)
struct BfsRow { uint32_t w[BFS_ROW_WORDS]; };
__device__ __forceinline__ bool cs_bfs_pulls(uint32_t A) { return A <= ROW_THREADS; }

// Row threadIdx.x of the transposed adjacency matrix, fetched so that the trip to global memory overlaps whatever
// the caller does in between (zero where the search will not pull, or for a thread without a node).
__device__ __forceinline__ void cs_bfs_load_row(const uint32_t *adjT, uint32_t A, uint32_t W, BfsRow &row)
{
    if (!cs_bfs_pulls(A)) {
#pragma unroll
        for (uint32_t w = 0; w < BFS_ROW_WORDS; ++w) row.w[w] = 0u;
        return;
    }
    const bool mine = threadIdx.x < A;
    const uint32_t *r = adjT + (mine ? threadIdx.x * W : 0u);          // (always a valid address; unused words are masked)
#pragma unroll
    for (uint32_t w = 0; w < BFS_ROW_WORDS; ++w) row.w[w] = cs_ld_cg_pinned(r + (w < W ? w : 0u));
#pragma unroll
    for (uint32_t w = 0; w < BFS_ROW_WORDS; ++w)
        if (!mine || w >= W) row.w[w] = 0u;
}

__device__ __forceinline__ void cs_bfs_survival(const uint32_t *__restrict__ adj, uint32_t A, uint32_t W, const BfsRow &rowT,
                                                uint32_t *s_front, uint32_t *s_visit, uint32_t *s_next, uint16_t *s_hops,
                                                uint16_t *hops, float *fsurv, uint32_t e_max, float delta)
{
    // on entry s_front[0 .. 32) holds the source bits and s_front[32 .. 64) zeroes (synchronised by the caller)
    const uint32_t tid = threadIdx.x;
    if (cs_bfs_pulls(A)) {
        const uint32_t v = tid;                                       // blockDim.x >= A
        bool seen = v >= A || ((s_front[v >> 5] >> (v & 31)) & 1u);
        uint32_t my_hops = (v < A && seen) ? 0u : CS_HOP_NONE;
        for (uint32_t level = 1; level <= A; ++level) {
            const uint32_t *cur = s_front + ((level & 1u) ? 0u : 32u);
            uint32_t *nxt = s_front + ((level & 1u) ? 32u : 0u);
            uint32_t hit = 0;
#pragma unroll
            for (uint32_t w = 0; w < BFS_ROW_WORDS; ++w) hit |= rowT.w[w] & cur[w];
            const bool fresh = hit != 0u && !seen;
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, fresh);
            if ((tid & 31u) == 0) nxt[tid >> 5] = word;
            if (fresh) { seen = true; my_hops = level; }
            if (!__syncthreads_or(fresh)) break;
        }
        if (v < A) s_hops[v] = (uint16_t)my_hops;
    } else {
        for (uint32_t a = tid; a < A; a += blockDim.x)
            s_hops[a] = ((s_front[a >> 5] >> (a & 31)) & 1u) ? 0 : CS_HOP_NONE;
        if (tid < W) { s_visit[tid] = s_front[tid]; s_next[tid] = 0; }
        __syncthreads();
        for (uint32_t level = 1; level <= A; ++level) {
            for (uint32_t node = tid; node < A; node += blockDim.x) {
                if ((s_front[node >> 5] >> (node & 31)) & 1u) {
                    for (uint32_t w = 0; w < W; ++w) {
                        const uint32_t v = __ldcg(&adj[node * W + w]);
                        if (v) atomicOr(&s_next[w], v);
                    }
                }
            }
            __syncthreads();
            uint32_t acc = 0;
            if (tid < W) {
                acc = s_next[tid] & ~s_visit[tid];
                s_next[tid] = 0;
                s_front[tid] = acc;
                s_visit[tid] |= acc;
                uint32_t bits = acc;
                while (bits) {
                    const uint32_t b2 = tid * 32 + (__ffs(bits) - 1);
                    bits &= bits - 1;
                    if (b2 < A) s_hops[b2] = (uint16_t)level;
                }
            }
            if (!__syncthreads_or(acc != 0)) break;
        }
    }
    __syncthreads();
    for (uint32_t a = tid; a < A; a += blockDim.x) {
        const uint32_t h = s_hops[a];
        const uint32_t m = h < e_max ? h : e_max;          // CS_HOP_NONE > e_max by construction
        const double ptilde = 1.0 - (double)m / (double)e_max;
        hops[a] = (uint16_t)h;
        fsurv[a] = (float)(ptilde + (double)delta);
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

__device__ void cs_block_sum2(double &a, double &b, double *s_red)
{
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        a += __shfl_xor_sync(0xFFFFFFFFu, a, d);
        b += __shfl_xor_sync(0xFFFFFFFFu, b, d);
    }
    __syncthreads();
    if (lane == 0) { s_red[warp] = a; s_red[32 + warp] = b; }
    __syncthreads();
    a = s_red[0];
    b = s_red[32];
    for (uint32_t w = 1; w < n_warps; ++w) { a += s_red[w]; b += s_red[32 + w]; }
}

// ---------------------------------------------------------------------------------------------
// One CTA per row i: Eq. 3 in canonical fp32 (one rounding per operation, no FMA), the row's
// arg-max, its adjacency bits (Eq. 7) and its entropy term.  The last CTA to finish then
// computes Eq. 2 / Eq. 11 over all rows and refreshes the cached BFS / Eq. 8 tables.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(ROW_THREADS)
cs_normalise_kernel(cs_workspace ws, uint32_t A, uint32_t W, float eps, float tau, float r_min, uint32_t e_max,
                    float delta, uint32_t all_chains, uint32_t n_chains, const uint32_t *__restrict__ ev_chain,
                    const uint16_t *__restrict__ ev_agent, const uint8_t *__restrict__ ev_flags, uint32_t n_events,
                    const uint32_t *__restrict__ n_events_dev)
{
    __shared__ uint32_t s_evc[OBS_FUSED_MAX];        // the batch: chain of event e,
    __shared__ uint16_t s_eva[OBS_FUSED_MAX];        // its agent (CS_AGENT_NONE: skipped),
    __shared__ uint16_t s_evp[OBS_FUSED_MAX];        // and the agent it follows when that is a counted transition
    __shared__ uint8_t s_succ[OBS_FUSED_MAX];        // 1: a later live event of the batch has the same chain
    __shared__ uint32_t s_add[CS_MAX_AGENTS];        // what the batch adds to the row being worked on
    __shared__ int s_last_live;
    __shared__ double s_red[64];
    __shared__ float s_bestv[ROW_THREADS / 32];
    __shared__ uint32_t s_besti[ROW_THREADS / 32];
    __shared__ uint32_t s_front[64], s_visit[32], s_next[32];
    __shared__ uint16_t s_hops[CS_MAX_AGENTS];
    __shared__ bool s_is_last;
    const uint32_t tid = threadIdx.x;
    CS_STAMP(ws, CS_PS_REFRESH_ENTRY, blockIdx.x == 0 && tid == 0);
    cs_wait_for_predecessor();
    CS_STAMP(ws, CS_PS_REFRESH_WAITED, blockIdx.x == 0 && tid == 0);
    cs_release_successor();

    // ---- a small batch of events is applied here, by every CTA to the rows it owns, instead of by a launch of its
    // own: each CTA stages the batch, finds every event's predecessor (in the batch, else the chain's current agent)
    // exactly as cs_observe_kernel does, and adds the transitions that start at row i to row i.  What is shared --
    // cur[], the last agent, the totals and the counters -- is written by the last CTA, after every CTA has read it.
    if (n_events_dev) n_events = min(n_events, *n_events_dev);
    uint32_t n_new = 0, n_skipped = 0;
    if (n_events) {
        uint32_t c = 0, a = CS_AGENT_NONE;
        if (tid == 0) s_last_live = -1;
        if (tid < n_events) {
            c = ev_chain[tid];
            a = ev_agent[tid];
            const bool warm = ev_flags && (ev_flags[tid] & CS_EV_WARMUP);
            uint32_t bad = 0;
            if (!warm && a >= A) bad |= CS_ST_BAD_AGENT;
            if (!warm && c >= n_chains) bad |= CS_ST_BAD_CHAIN;
            if (bad && blockIdx.x == 0) atomicOr(&ws.sc->status, bad);
            if (warm || bad) a = CS_AGENT_NONE;
        }
        s_evc[tid] = c;
        s_eva[tid] = (uint16_t)a;
        s_succ[tid] = 0;
        __syncthreads();
        const bool live = tid < n_events && a != CS_AGENT_NONE;
        uint32_t prev = CS_AGENT_NONE;
        if (live) {
            int j = (int)tid - 1;
            for (; j >= 0; --j)
                if (s_evc[j] == c && s_eva[j] != CS_AGENT_NONE) { prev = s_eva[j]; break; }
            if (j < 0) prev = ws.cur[c];
            else s_succ[j] = 1;                                // event j is not the last of its chain in this batch
            atomicMax(&s_last_live, (int)tid);
        }
        const bool counted = live && prev != CS_AGENT_NONE && prev != a;
        s_evp[tid] = (uint16_t)(counted ? prev : CS_AGENT_NONE);
        n_new = (uint32_t)__syncthreads_count(counted);
        n_skipped = (uint32_t)__syncthreads_count(tid < n_events && a == CS_AGENT_NONE);
    }
    // Column sums q_j = sum_i pi_i P_ij of Eq. 2 are accumulated by the row CTAs in 2^-60 fixed
    // point with integer atomics: integer addition commutes, so the sum is bit-identical from run
    // to run whatever order the CTAs finish in (a float atomic would not be).
    const uint32_t n_total = ws.sc->n_transitions + n_new;
    const uint32_t fill = ws.sc->adjT_cur ^ 1u;              // every CTA reads this before the last one flips it
    uint32_t *adjT_fill = ws.adjT + (size_t)fill * A * W, *adjT_clear = ws.adjT + (size_t)(fill ^ 1u) * A * W;
    const double inv_total = n_total ? 1.0 / (double)n_total : 0.0;
    for (uint32_t i = blockIdx.x; i < A; i += gridDim.x) {
        uint32_t n_i = ws.rowsum[i];
        // transitions of the batch that start at agent i
        const bool mine = n_events && tid < n_events && s_evp[tid] == i;
        const uint32_t row_new = n_events ? (uint32_t)__syncthreads_count(mine) : 0u;
        if (row_new) {
            for (uint32_t j = tid; j < A; j += ROW_THREADS) s_add[j] = 0;
            __syncthreads();
            if (mine) atomicAdd(&s_add[s_eva[tid]], 1u);
            __syncthreads();
            n_i += row_new;
            if (tid == 0) ws.rowsum[i] = n_i;
        }
        const double pi_fix = (double)n_i * inv_total * 1152921504606846976.0;      // pi_i * 2^60
        const float den = __fadd_rn((float)n_i, __fmul_rn((float)A, eps));
        // Most entries of a row have a zero count and therefore the same P = eps / den: their contribution to the
        // column sums is one number per row, added once to a scalar instead of A times to A columns; a column with a
        // count gets the difference on top.  Integer arithmetic, so the sums are bit for bit what A atomics per row gave.
        const long long base_fix = __double2ll_rn(pi_fix * (double)__fdiv_rn(__fadd_rn(0.0f, eps), den));
        if (tid == 0 && n_i) atomicAdd(&ws.sc->qbase, (unsigned long long)base_fix);
        float bestv = -1.0f;
        uint32_t besti = 0xFFFFFFFFu;
        double h = 0.0;
        for (uint32_t j0 = 0; j0 < A; j0 += ROW_THREADS) {       // A is padded to whole warps for the ballot
            const uint32_t j = j0 + tid;
            bool edge = false;
            if (j < A) {
                uint32_t cij = ws.C[i * A + j];
                if (row_new && s_add[j]) { cij += s_add[j]; ws.C[i * A + j] = cij; }
                const float p = __fdiv_rn(__fadd_rn((float)cij, eps), den);
                ws.P[i * A + j] = p;
                if (p > bestv) { bestv = p; besti = j; }         // strict: the lowest j among equals stays
                const double pd = (double)p;
                h += pd * log(pd);
                edge = p >= tau;
                if (n_i && cij) atomicAdd(&ws.qfix[j], (unsigned long long)(__double2ll_rn(pi_fix * pd) - base_fix));
            }
            const uint32_t bits = __ballot_sync(0xFFFFFFFFu, edge);
            if ((tid & 31) == 0 && (j >> 5) < W) ws.adj[i * W + (j >> 5)] = bits;
            if (edge) atomicOr(&adjT_fill[j * W + (i >> 5)], 1u << (i & 31));      // the transpose: i precedes j
        }
        for (uint32_t w = tid; w < W; w += ROW_THREADS) adjT_clear[i * W + w] = 0;  // for the refresh after this one
        // arg-max (max value, then min index) and the entropy term: a butterfly inside each warp, then the warp results
        // combined in warp order by thread 0
        const uint32_t lane = tid & 31, warp = tid >> 5;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const float v = __shfl_xor_sync(0xFFFFFFFFu, bestv, d);
            const uint32_t x = __shfl_xor_sync(0xFFFFFFFFu, besti, d);
            if (v > bestv || (v == bestv && x < besti)) { bestv = v; besti = x; }
            h += __shfl_xor_sync(0xFFFFFFFFu, h, d);
        }
        __syncthreads();                                         // the partials of the row before have been read
        if (lane == 0) { s_bestv[warp] = bestv; s_besti[warp] = besti; s_red[warp] = h; }
        __syncthreads();
        if (tid == 0) {
            float bv = s_bestv[0];
            uint32_t bi = s_besti[0];
            double hs = s_red[0];
            for (uint32_t w = 1; w < ROW_THREADS / 32; ++w) {
                if (s_bestv[w] > bv || (s_bestv[w] == bv && s_besti[w] < bi)) { bv = s_bestv[w]; bi = s_besti[w]; }
                hs += s_red[w];
            }
            ws.amax[i] = (uint16_t)bi;
            ws.rowH[i] = hs;
        }
    }

    CS_STAMP(ws, CS_PS_REFRESH_ROWS_DONE, blockIdx.x == 0 && tid == 0);
    // ---- last CTA done: global quantities ---------------------------------------------------------
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const uint32_t t = atomicAdd(&ws.sc->ticket0, 1u);
        s_is_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_is_last) return;
    __threadfence();
    CS_STAMP(ws, CS_PS_REFRESH_LAST_CTA, tid == 0);

    BfsRow rowT;                                                         // in flight during the sums
    cs_bfs_load_row(adjT_fill, A, W, rowT);
    // the operands of Eq. 2 (the first ROW_THREADS of each array) travel with it, so that the sums below start on data
    // that has arrived instead of on a trip of their own
    const uint32_t t0_ = tid < A ? tid : 0u;
    const uint32_t pre_rowsum = cs_ld_cg_pinned(ws.rowsum + t0_);
    const unsigned long long pre_rowH = cs_ld_cg_pinned((const unsigned long long *)ws.rowH + t0_);
    const unsigned long long pre_qfix = cs_ld_cg_pinned(ws.qfix + t0_);
    const unsigned long long qbase = cs_ld_cg_pinned(&ws.sc->qbase);
    uint32_t la = cs_ld_cg_pinned(&ws.sc->last_agent);
    if (n_events) {
        // the batch's effect on what all CTAs share (every other CTA is done reading it)
        const uint32_t a = tid < n_events ? s_eva[tid] : CS_AGENT_NONE;
        if (a != CS_AGENT_NONE) {
            if (!s_succ[tid]) ws.cur[s_evc[tid]] = (uint16_t)a;       // the chain's last live event of the batch
        }
        if (all_chains) __threadfence();                      // (cur[] is read back below when every chain is a source)
        if (s_last_live >= 0) la = s_eva[s_last_live];
        if (tid == 0) {
            ws.sc->last_agent = la;
            ws.sc->n_transitions = n_total;
            atomicAdd((unsigned long long *)&ws.cnt->events_seen, (unsigned long long)n_events);
            if (n_skipped) atomicAdd((unsigned long long *)&ws.cnt->events_skipped, (unsigned long long)n_skipped);
            if (n_new) atomicAdd((unsigned long long *)&ws.cnt->transitions_counted, (unsigned long long)n_new);
        }
    }
    if (tid < 64) s_front[tid] = (tid < 32 && !all_chains && la < A && (la >> 5) == tid) ? (1u << (la & 31)) : 0u;
    // Eq. 10's arg-max successor of the (now final) last agent: asked for here, used by thread 0 after the sums
    const uint32_t a_star_pre = (tid == 0 && la < A) ? (uint32_t)cs_ld_cg_pinned(ws.amax + la) : 0xFFFFFFFFu;
    const uint32_t N = n_total;
    double Hc = 0.0, Hm = 0.0;
    if (N > 0) {
        const double invN = 1.0 / (double)N;
        for (uint32_t i = tid; i < A; i += ROW_THREADS) {
            const uint32_t rs = i == tid ? pre_rowsum : __ldcg(&ws.rowsum[i]);
            const double rh = i == tid ? __longlong_as_double((long long)pre_rowH) : __ldcg(&ws.rowH[i]);
            Hc -= ((double)rs * invN) * rh;
        }
        for (uint32_t j = tid; j < A; j += ROW_THREADS) {
            const unsigned long long qf = j == tid ? pre_qfix : __ldcg(&ws.qfix[j]);
            const double q = (double)(qf + qbase) * (1.0 / 1152921504606846976.0);
            if (q > 0.0) Hm -= q * log(q);
        }
    }
    for (uint32_t j = tid; j < A; j += ROW_THREADS) ws.qfix[j] = 0;      // ready for the next refresh
    __syncthreads();                                                     // (every thread has read qbase)
    if (tid == 0) ws.sc->qbase = 0;
    cs_block_sum2(Hc, Hm, s_red);
    CS_STAMP(ws, CS_PS_REFRESH_SUMS_DONE, tid == 0);                                        // (its barriers also order s_front's zeroes)
    if (tid == 0) {
        double R = 0.0;
        if (N > 0 && Hm > 0.0) R = 1.0 - Hc / Hm;
        const float Rf = (float)R;
        ws.sc->R = Rf;
        ws.sc->gate = (Rf >= r_min) ? 1u : 0u;
        ws.sc->a_star = a_star_pre;                           // Eq. 10, for the prefetch ranking
        ws.sc->adjT_cur = fill;
        ws.sc->ticket0 = 0;
    }
    if (all_chains) {
        // sources: the current agent of every chain that has one (all live sessions)
        for (uint32_t ch = tid; ch < n_chains; ch += ROW_THREADS) {
            const uint32_t a = __ldcg(&ws.cur[ch]);
            if (a < A) atomicOr(&s_front[a >> 5], 1u << (a & 31));
        }
    }
    __syncthreads();
    cs_bfs_survival(ws.adj, A, W, rowT, s_front, s_visit, s_next, s_hops, ws.hops, ws.fsurv, e_max, delta);
    CS_STAMP(ws, CS_PS_REFRESH_END, tid == 0);
}

// BFS + Eq. 8 from explicit sources into the temporary tables (cs_score_blocks with sources).
__global__ void __launch_bounds__(ROW_THREADS)
cs_survival_kernel(cs_workspace ws, uint32_t A, uint32_t W, const uint16_t *__restrict__ sources, uint32_t n_sources,
                   uint32_t e_max, float delta)
{
    __shared__ uint32_t s_front[64], s_visit[32], s_next[32];
    __shared__ uint16_t s_hops[CS_MAX_AGENTS];
    const uint32_t tid = threadIdx.x;
    BfsRow rowT;
    cs_bfs_load_row(ws.adjT + (size_t)ws.sc->adjT_cur * A * W, A, W, rowT);
    if (tid < 64) s_front[tid] = 0;
    __syncthreads();
    for (uint32_t s = tid; s < n_sources; s += ROW_THREADS) {
        const uint32_t a = sources[s];
        if (a < A) atomicOr(&s_front[a >> 5], 1u << (a & 31));
        else atomicOr(&ws.sc->status, CS_ST_BAD_SOURCE);
    }
    __syncthreads();
    cs_bfs_survival(ws.adj, A, W, rowT, s_front, s_visit, s_next, s_hops, ws.hops_tmp, ws.fsurv_tmp, e_max, delta);
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
// P comes from global memory; a CTA's columns stay in its L1 for the later steps.  The last step needs column a only: one
// dot product per target, one warp each.
//
// Bound by the fp64 pipe for many agents (2 A^3 (K - 2) operations), by latency for few.  256 agents, K = 4: 62.7 us with
// one CTA per 8 targets that walked the matrix column by column (32 CTAs, one serial chain of 256 loads per step),
// 13.7 us per call like this (128 CTAs).
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
        cluster.sync();                                            // (also: every CTA has started before its memory is written)
        const uint32_t col_warps = (n_cols + 63u) / 64u, slices = XS_WARPS / col_warps;
        const uint32_t cw = warp % col_warps, sl = warp / col_warps;
        uint32_t cur = 0;
        for (uint32_t t = 1; t + 1 < K; ++t) {
            const double *v = v_all + (size_t)cur * A * XS_TARGETS;
            if (sl < slices) {
                const uint32_t j0 = col0 + cw * 64u + lane, j1 = j0 + 32u;
                const float *p0 = P + (j0 < col1 ? j0 : 0u), *p1 = P + (j1 < col1 ? j1 : 0u);    // (columns past the end: unused)
                const uint32_t i_end = (uint32_t)((unsigned long long)(sl + 1u) * A / slices);
                double acc0[XS_TARGETS], acc1[XS_TARGETS];
#pragma unroll
                for (uint32_t m = 0; m < XS_TARGETS; ++m) acc0[m] = acc1[m] = 0.0;
#pragma unroll 8
                for (uint32_t i = (uint32_t)((unsigned long long)sl * A / slices); i < i_end; ++i) {
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
            double *nxt = v_all + (size_t)(cur ^ 1u) * A * XS_TARGETS;
            for (uint32_t e = tid; e < (col1 > col0 ? col1 - col0 : 0u) * XS_TARGETS; e += XS_THREADS) {
                const uint32_t jc = e / XS_TARGETS, m = e % XS_TARGETS, j = col0 + jc;
                const double *q = part + (size_t)(jc / 64u) * XS_TARGETS * XS_PART_ROW + m * XS_PART_ROW + jc % 64u;
                double sum = 0.0;
                for (uint32_t u = 0; u < slices; ++u) sum += q[(size_t)u * col_warps * XS_TARGETS * XS_PART_ROW];
                if (j == base + m) { s_hit[m] += sum; sum = 0.0; }   // (one thread per target)
                for (uint32_t r = 0; r < CL; ++r) cluster.map_shared_rank(nxt, r)[(size_t)j * XS_TARGETS + m] = sum;
            }
            cluster.sync();                                        // the new V is complete everywhere; `part` is free again
            cur ^= 1u;
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

int cs_launch_exact_survival(cs_ctx *ctx, uint32_t a0, uint32_t K, float *psurv_out, float *fsurv_out, cudaStream_t s)
{
    const cs_params &p = ctx->p;
    static std::mutex mu;
    static bool opted[64];                                  // shared-memory opt-in, once per process and device
    {
        std::lock_guard<std::mutex> lock(mu);
        if (ctx->device < 0 || ctx->device >= 64) return CS_EINVAL;
        if (!opted[ctx->device]) {
            const cudaError_t e = cudaFuncSetAttribute(cs_exact_survival_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)xs_smem_bytes(CS_MAX_AGENTS));
            if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
            opted[ctx->device] = true;
        }
    }
    // as many CTAs per cluster as give each at least 64 columns and still fit one wave
    const uint32_t n_clusters = (p.n_agents + XS_TARGETS - 1) / XS_TARGETS;
    uint32_t cl = 1;
    while (cl < XS_MAX_CLUSTER && p.n_agents > 64u * cl && 2u * cl * n_clusters <= (uint32_t)ctx->sm_count) cl *= 2;
    const uint32_t n_cols = (p.n_agents + cl - 1) / cl;
    cs_launch_chained_clusters(cs_exact_survival_kernel, n_clusters * cl, cl, XS_THREADS, xs_smem_bytes(p.n_agents), s, ctx->ws,
                               p.n_agents, a0, K, n_cols, p.delta, psurv_out, fsurv_out);
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

// Largest cluster (a power of two) the observe kernel can run as on a device; asked once per process and device, with
// that device current.
static int obs_cluster_limit(int device)
{
    static std::mutex mu;
    static int known[64];                                     // 0: not asked yet
    if (device < 0 || device >= 64) return 1;
    std::lock_guard<std::mutex> lock(mu);
    if (!known[device]) known[device] = cs_probe_cluster(cs_observe_kernel, OBS_MAX_CLUSTER, OBS_THREADS, 0, 1);
    return known[device];
}

int cs_launch_observe(cs_ctx *ctx, const uint32_t *chain, const uint16_t *agent, const uint8_t *evflags,
                      uint32_t n_events, cudaStream_t s)
{
    const cs_params &p = ctx->p;
    const bool fused = n_events <= OBS_FUSED_MAX;             // small batches ride along with the refresh
    if (n_events && !fused) {
        // one event per thread and round: no more CTAs than the batch fills
        const int most = obs_cluster_limit(ctx->device);
        if (most < 1) { ctx->last_cuda_error = (int)cudaErrorInvalidClusterSize; return CS_ECUDA; }
        uint32_t cl = 1;
        while ((int)cl < most && cl * OBS_THREADS < n_events) cl <<= 1;
        cs_launch_chained_clusters(cs_observe_kernel, cl, cl, OBS_THREADS, 0, s, ctx->ws, p.n_agents, p.n_chains, chain, agent,
                                   evflags, n_events, ctx->step_n_events_dev);
        int rc = cs_check_launch(ctx);
        if (rc != CS_OK) return rc;
    }
    const uint32_t grid = p.n_agents < 2u * (uint32_t)ctx->sm_count ? p.n_agents : 2u * (uint32_t)ctx->sm_count;
    cs_launch_chained(cs_normalise_kernel, grid, ROW_THREADS, 0, s, ctx->ws, p.n_agents, ctx->W, p.eps, p.tau, p.r_min,
                      p.e_max, p.delta, ctx->source_mode == CS_SOURCES_ALL_CHAINS ? 1u : 0u, p.n_chains,
                      fused ? chain : (const uint32_t *)nullptr, fused ? agent : (const uint16_t *)nullptr,
                      fused ? evflags : (const uint8_t *)nullptr, fused ? n_events : 0u,
                      fused ? (const uint32_t *)ctx->step_n_events_dev : (const uint32_t *)nullptr);
    return cs_check_launch(ctx);
}

int cs_launch_survival(cs_ctx *ctx, const uint16_t *sources, uint32_t n_sources, cudaStream_t s)
{
    const cs_params &p = ctx->p;
    cs_survival_kernel<<<1, ROW_THREADS, 0, s>>>(ctx->ws, p.n_agents, ctx->W, sources, n_sources, p.e_max, p.delta);
    return cs_check_launch(ctx);
}
