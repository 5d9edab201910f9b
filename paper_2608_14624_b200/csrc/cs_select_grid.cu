// Selects over a large index in ONE launch on the whole GPU: a kernel of one CTA per SM that reads the index once for up to
// three lists (GPU-tier victims, host-tier victims, prefetch candidates), with grid barriers in place of kernel boundaries.  Same key,
// same eligibility rules, same exact ordered output as the launch chain of cs_select.cu, whose six launches per list it replaces.
//
//   1 scan     every entry's key is compared with the key that the previous call of the kind left for its list.  Candidates go to the list
//              of all candidates and, by the bucket boundaries that the previous call left as well, straight into the bucket they belong to.
//   2 finish   after ONE grid barrier: a warp per bucket ranks its keys by counting and stores their ids; larger buckets go round in parts
//              of eight keys.  Whoever places every step-th key stores it as a boundary for the next call: exact quantiles of this call's
//              order, up to 2.25 lists from its beginning, because a list's entries are usually gone by then.
//
// The boundaries decide nothing but the sizes of the buckets.  Where they do not hold -- a bucket of more than SG_BUCKET_MAX keys, too few
// keys below the last boundary, the first calls -- the candidates are ordered by a ranked sample instead (cs_select_buckets.cuh; two more
// barriers), and where the remembered key does not, a histogram and a collect pass come first (two more).  Both are remembered as scores and
// ages: their last_access moves on with the clock.
//
// Bound by latency up to a few million entries: the prologue's loads, a barrier and the finish's loads take 1 to 1.5 us each, a bucket's
// ranking 2; beyond that by the scan's instructions (about 200 per 128 entries; 64,000,000 entries at 119 us are 4.8 TB/s, where the chain's scan,
// which compares last_access alone for most entries, has 5.0).  Loads are asynchronous copies by each thread for itself, three steps of four
// entries ahead: bulk copies into a ring, with a producer warp, took 187 to 330 us for 64,000,000 entries, two steps at a time 10 % longer,
// four steps 2 % and 22 KiB of shared memory, which keeps the CTA off SMs where a compaction's runs.  Times beside those of the routes that it
// replaces stand at select_route() (cs_select.cu).
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "cs_select_buckets.cuh"

#define SG_THREADS 512u
#define SG_WARPS (SG_THREADS / 32u)
#define SG_STAGES 3u                   // steps in flight per warp
#define SG_QUEUE 64u                   // candidates of a warp that wait: 32 and 32 new ones
#define SG_STEP 24u                    // keys of a bucket aimed at, as long as CS_BUCKETS buckets hold the list
#define SG_BUCKET_WARP 96u             // largest bucket that one warp ranks, three keys per lane
#define SG_KEYS 128u                   // keys that a warp holds at a time
#define SG_BUCKET_MAX 1536u            // largest bucket that is counted.  (Index that moves, 1,000,000 entries, lists of 10,000 and 2,000, bench.py's metadata-scale loop
                                       // replayed from a graph: 1,024 keys 49.3 us, this 46.2, 2,048 45.2, 3,072 44.8; but where a list of 2,000 has come to lie in one
                                       // bucket, which the sample then ranks without a barrier more, 45.0, 44.6, 49.3, 48.9.  Larger ones divided among the CTAs by a sample of their own, so that
                                       // nearly no list goes on to the ranked sample: as fast or slower, 36 to 43 us for one list of 10,000, 50 to 65 for one of 30,000)
#define SG_MAP 512u                    // parts of larger buckets per CTA
#define SG_WAIT_LIMIT (1u << 23)       // polls of a grid barrier (seconds)
#define SG_PATIENCE 64u                // polls (about 50 us) between two looks for shares that nobody has begun
static_assert(SG_THREADS == CS_BUCKETS, "one bucket per thread");

// Candidates that a call should find (as cs_ahead(); a few thousand more cost less here than the shortest list's key that no longer holds).
__device__ __forceinline__ uint32_t sg_ahead(uint32_t k) { return 3u * k + 8192u; }

struct GridArgs {
    SelArgs a;                         // the index, the clock and the tables; tier, k, bins and the like are per list
    cs_workspace ws[3];                // by list: 0 GPU victims, 1 host victims, 2 prefetch; tables and scalars are the same in each
    uint32_t k[3], bin_lo[3], bin_shift[3];
    uint32_t *ids[3], *n_out[3];
    uint32_t want, speculate;          // lists wanted, one bit each; 0: nothing is remembered
    uint32_t give_up;                  // the barrier (1 ..) whose waits run out at once; SG_LATE: CTAs that start late; 0: neither
};

__host__ __device__ inline size_t sg_table_bytes(uint32_t A, uint32_t gtab_len)
{
    return (size_t)A * 8 + ((size_t)gtab_len + 1) * 4;
}
// Boundaries of the buckets and the candidates on their way out; the histograms of a miss lie over both.
struct ScanShared {
    u64 b_km[3][CS_BUCKETS + 1], q_km[SG_WARPS][SG_QUEUE];
    uint32_t b_id[3][CS_BUCKETS + 1], q_id[SG_WARPS][SG_QUEUE];
    uint8_t q_list[SG_WARPS][SG_QUEUE];
};
union ScanOrHist {
    ScanShared s;
    uint32_t hist[3][CS_HIST_BINS];
};
struct FinishShared {
    uint4 key[SG_WARPS][SG_KEYS];      // id, low and high word of a warp's keys
    uint32_t off[3][CS_BUCKETS], cnt[3][CS_BUCKETS];
    uint32_t map[SG_MAP];              // parts of larger buckets that are this CTA's: list, bucket, which keys
};
struct SampleShared {
    u64 km[FEW_MAX];
    uint32_t id[FEW_MAX];
};
struct PlaceShared {
    u64 s_km[CS_SAMPLE], b_km[CS_BUCKETS];
    uint32_t s_id[CS_SAMPLE], b_id[CS_BUCKETS];
};
// A thread's own steps on their way in; the ordering steps lie over it.
struct TileShared {
    uint4 la[SG_STAGES][SG_THREADS];
    uint2 ag[SG_STAGES][SG_THREADS], dp[SG_STAGES][SG_THREADS];
    uint32_t fl[SG_STAGES][SG_THREADS], rf[SG_STAGES][SG_THREADS], tk[SG_STAGES][SG_THREADS];
};
union StepShared {
    TileShared tile;
    FinishShared finish;
    SampleShared sample;
    PlaceShared place;
};

// Words of a list that every thread of a CTA looks at.
struct ListShared {
    u64 bound;                         // key up to which the scan collects; after a miss, the collect pass
    uint32_t known, nb;                // a key is remembered; buckets whose boundaries are
    uint32_t then, moves;              // the clock when they were; 1: the key is of the same call
    uint32_t c, n_elig, n_out, spec;   // candidates, eligible entries, length of the list, 1: the remembered key held
    uint32_t b0;                       // threshold bin of a miss
    uint32_t bad_at, ranked;           // first bucket offset from which on nothing can be ranked; keys that can be
    uint32_t refresh;                  // 1: too few for the next call's boundaries, which a sample gives then
    uint32_t step, next_nb, end;       // boundaries for the next call: every step-th key, next_nb buckets, the last of which ends at place `end`
    uint32_t cap, epoch, now;          // keys of a bucket's region; the set of words in use; the clock
};

// A CTA's shared memory, before the tables ([A] survival factor and anchor length, [gtab_len + 1] recency factors).  Every function finds it by
// itself: a pointer to it that has been handed over is a generic one.
struct CtaShared {
    StepShared step;
    ScanOrHist u;
    ListShared list[3];
    uint32_t part[4 * 64], elig[3], bad[3], words[4], scalar[5];
    uint32_t ok, lost;                 // a barrier's outcome; 1: this CTA's share is another's
    uint32_t n_own, pad;               // shares of this CTA: its own and those it has taken over
    uint16_t own[CS_GRID_MAX_CTAS];
};
extern __shared__ __align__(128) unsigned char sg_smem[];
#define SH (*(CtaShared *)sg_smem)
static_assert(sizeof(CtaShared) % 8 == 0, "the tables begin with pairs of words");

static size_t sg_smem_bytes(uint32_t A, uint32_t gtab_len) { return sizeof(CtaShared) + sg_table_bytes(A, gtab_len); }

struct Sg {                            // what the passes over the index share
    cs_grid_state *g;
    uint32_t now, a_star, epoch;
    uint32_t share;                    // whose part of the index
    uint32_t agent, gtab;              // shared-memory addresses of the tables
    bool whole_table;                  // the recency table covers every age before saturation; its last entry is the saturated factor
    bool depth;                        // the walks bring the depths
};

// ---- grid barrier -----------------------------------------------------------------------------------------------------------------
// The work is cut into gridDim.x shares, share x meant for CTA x.  A barrier counts shares, not CTAs: nobody waits for a CTA that has not
// started.  A CTA that has waited long at the first barrier takes over shares that nobody has begun, with all that belongs to them until
// the end of the launch; a CTA that finds its share taken leaves.  So a launch goes on with whatever SMs it gets -- other kernels may hold some
// for as long as they like -- and from the first barrier on every share is at a running CTA.  (Selects of 1,000,000 entries beside back-to-back
// compactions: 106 to 118 us each where every CTA had to find a place, 40 so.)
//
// A share's CTA adds one to its word when it starts, once in every launch, and so learns the launch's number, and whether the share is still its own;
// who takes a share over swaps that word for one that carries the launch's mark.
//
// All CTAs pass a barrier or none does: a wait that runs out marks the word unless everything is done, in one step with that look at it, and
// who comes late finds the mark.  The words are used once per launch, in two sets by turns: the CTA with share 0 clears the other set after the first
// barrier, when the launch before is over and nobody can be in the next one.
#define SG_GIVEN_UP 0x80000000u
enum : uint32_t { SG_FAILED = 0xFFFFFFFEu, SG_PASSED = 0xFFFFFFFFu };
__device__ __forceinline__ bool share_is_free(u64 taken, uint32_t number) { return (uint32_t)taken == number && (uint32_t)(taken >> 32) != ~number; }
// done: shares to be counted; take_over: shares may still be without a CTA.  Returns SG_PASSED, SG_FAILED or a share that is this CTA's now.
__device__ __noinline__ uint32_t grid_barrier(const GridArgs &ga, cs_grid_state *g, uint32_t number, uint32_t which, uint32_t done, bool take_over)
{
    __syncthreads();
    if (threadIdx.x < 32u) {
        const uint32_t lane = threadIdx.x, G = gridDim.x;
        uint32_t *word = g->bar[number & 1u][which], v = 0, polls = 0, share = SG_PASSED;
        if (lane == 0) {
            if (ga.give_up == which + 1u) atomicOr(word, SG_GIVEN_UP);
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(word), "r"(done) : "memory");
        }
        for (;;) {
            if (lane == 0) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
            v = __shfl_sync(0xFFFFFFFFu, v, 0);
            if (v >= G) break;                                 // (everything, or the mark)
            if (++polls % SG_PATIENCE == 0u && take_over) {
                for (uint32_t x0 = 0; x0 < G && share == SG_PASSED; x0 += 32u) {
                    const uint32_t x = x0 + lane;
                    const u64 taken = x < G ? __ldcg(g->taken + x) : ~0ull;
                    const uint32_t free = __ballot_sync(0xFFFFFFFFu, x < G && share_is_free(taken, number));
                    if (!free) continue;
                    const uint32_t one = __ffs(free) - 1u;
                    uint32_t mine = 0;
                    if (lane == one) mine = atomicCAS(g->taken + x, taken, (u64)~number << 32 | number) == taken ? 1u : 0u;
                    if (__shfl_sync(0xFFFFFFFFu, mine, one)) share = x0 + one;
                }
                if (share != SG_PASSED) break;
            }
            if (lane == 0 && polls > SG_WAIT_LIMIT) atomicCAS(word, v, v | SG_GIVEN_UP);
            if (polls > 4096u) __nanosleep(256);
        }
        if (lane == 0) {
            SH.ok = share != SG_PASSED ? share : (v & SG_GIVEN_UP ? SG_FAILED : SG_PASSED);
            if (share != SG_PASSED) SH.own[SH.n_own++] = (uint16_t)share;
        }
    }
    __syncthreads();
    return SH.ok;
}
// A barrier behind the first one.
__device__ __forceinline__ bool all_here(const GridArgs &ga, cs_grid_state *g, uint32_t epoch, uint32_t which)
{
    return grid_barrier(ga, g, epoch, which, SH.n_own, false) == SG_PASSED;
}

// A wait has run out, and every CTA with a share comes here once its own work up to that barrier is done.  The last one leaves empty lists, the status
// that says why, and nothing that a later call would trip over: no counts in the histograms, nothing remembered.
__device__ __noinline__ void give_up(const GridArgs &ga, cs_grid_state *g)
{
    const uint32_t tid = threadIdx.x;
    __threadfence();
    __syncthreads();
    if (tid == 0) SH.ok = atomicAdd(&g->failed, SH.n_own) + SH.n_own == gridDim.x ? 1u : 0u;
    __syncthreads();
    if (!SH.ok) return;
    __threadfence();
    for (uint32_t l = 0; l < 3u; ++l) {
        if (!((ga.want >> l) & 1u)) continue;
        for (uint32_t i = tid; i < ga.k[l]; i += SG_THREADS) ga.ids[l][i] = CS_ID_NONE;
        for (uint32_t i = tid; i < CS_HIST_BINS; i += SG_THREADS) ga.ws[l].hist[i] = 0;
        if (tid == 0) {
            *ga.n_out[l] = 0;
            g->rem_n[l] = 0;
            ga.ws[0].sc->sel_T[l] = ~0ull;
        }
    }
    if (tid == 0) {
        g->failed = 0;
        atomicOr(&ga.ws[0].sc->status, CS_ST_TIMEOUT);
    }
}

// cs_selftest_select_wait(): a CTA that starts late, once its share is another's (or some tenths of a second have gone by).
#define SG_LATE 6u
__device__ __noinline__ void late_start(cs_grid_state *g)
{
    if (threadIdx.x == 0) {
        const uint32_t number = (uint32_t)__ldcg(g->taken + blockIdx.x);
        for (uint32_t polls = 0; polls < 200000u && share_is_free(__ldcg(g->taken + blockIdx.x), number); ++polls) __nanosleep(256);
    }
    __syncthreads();
}

// The other set of words is the next launch's.
__device__ __noinline__ void prepare_next_launch(cs_grid_state *g, uint32_t epoch)
{
    const uint32_t tid = threadIdx.x, other = epoch ^ 1u;
    for (uint32_t l = 0; l < 3u; ++l) g->count[other][l][tid * CS_BCOUNT_STRIDE] = 0;
    if (tid < 8u) g->bar[other][tid][0] = 0;
    if (tid < 3u) { g->list[other][tid].c_scan = 0; g->list[other][tid].c_collect = 0; g->list[other][tid].eligible = 0; }
}

// Loads of the tables by shared-memory address.
__device__ __forceinline__ uint32_t lds_table(uint32_t at)
{
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at));
    return v;
}
__device__ __forceinline__ uint2 lds_table2(uint32_t at)
{
    uint2 v;
    asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(at));
    return v;
}
template <int BYTES> __device__ __forceinline__ void copy_in(void *to, const void *from)
{
    if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from), "n"(BYTES) : "memory");
}

// ---- the index, a quad per thread and step ------------------------------------------------------------------------------------------------
struct Quad4 {                         // four consecutive entries
    uint4 la;
    uint2 ag, dp;
    uint32_t rf, fl, tk;
};

// Quad q of the index into this thread's place of a stage (q beyond the last whole quad: nothing); one group.
__device__ __forceinline__ void quad_ask(const GridArgs &ga, const Sg &s, uint32_t q, uint32_t stage)
{
    if (q < ga.a.n / 4u) {
        TileShared &t = SH.step.tile;
        const uint32_t tid = threadIdx.x;
        copy_in<16>(&t.la[stage][tid], (const uint4 *)ga.a.la + q);
        copy_in<8>(&t.ag[stage][tid], (const uint2 *)ga.a.agent + q);
        copy_in<4>(&t.fl[stage][tid], (const uint32_t *)ga.a.flags + q);
        copy_in<4>(&t.rf[stage][tid], (const uint32_t *)ga.a.ref + q);
        if (ga.a.ntok) copy_in<4>(&t.tk[stage][tid], (const uint32_t *)ga.a.ntok + q);
        if (s.depth) copy_in<8>(&t.dp[stage][tid], (const uint2 *)ga.a.depth + q);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
// The first steps of a walk.  (Every thread copies for itself only: no barrier, no wait for anybody else.)
__device__ __forceinline__ void walk_start(const GridArgs &ga, const Sg &s)
{
    const uint32_t q = s.share * SG_THREADS + threadIdx.x;
#pragma unroll
    for (uint32_t i = 0; i < SG_STAGES; ++i) quad_ask(ga, s, q + i * gridDim.x * SG_THREADS, i);
}
__device__ __forceinline__ void walk_drain() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Calls f(quad, id of its first entry, valid entries as flags) for every quad of this thread (walk_start() before), whole warps; the index's
// last one to three entries come as a quad of their own.
template <class F>
__device__ __forceinline__ void walk(const GridArgs &ga, const Sg &s, F f)
{
    const uint32_t tid = threadIdx.x, n_quads = ga.a.n / 4u, stride = gridDim.x * SG_THREADS, no_sizes = 0x01010101u * ga.a.block_tokens;
    uint32_t q = s.share * SG_THREADS + tid, stage = 0;
    bool tail = (ga.a.n & 3u) != 0u && s.share == gridDim.x - 1u && tid >= SG_THREADS - 32u;
    for (;;) {
        const bool step = (q & ~31u) < n_quads;                // (whole warps)
        Quad4 Q;
        uint32_t id0, valid;
        if (step) {
            asm volatile("cp.async.wait_group %0;" ::"n"(SG_STAGES - 1) : "memory");
            const TileShared &t = SH.step.tile;
            Q.la = t.la[stage][tid];
            Q.ag = t.ag[stage][tid];
            Q.fl = t.fl[stage][tid];
            Q.rf = t.rf[stage][tid];
            Q.tk = ga.a.ntok ? t.tk[stage][tid] : no_sizes;
            Q.dp = s.depth ? t.dp[stage][tid] : make_uint2(0u, 0u);
            id0 = 4u * q;
            valid = q < n_quads ? 0x80808080u : 0u;
            if (!valid) Q.ag = make_uint2(0u, 0u);             // (nothing has been copied there)
        } else {
            if (!tail) break;
            tail = false;
            id0 = ga.a.n & ~3u;
            valid = 0;
            uint32_t la[4] = {}, ag[4] = {}, dp[4] = {};
            Q.fl = Q.rf = Q.tk = 0;
#pragma unroll
            for (uint32_t x = 0; x < 3; ++x) {
                const uint32_t id = id0 + x;
                if ((tid & 31) == 0u && id < ga.a.n) {
                    valid |= 0x80u << (8 * x);
                    la[x] = __ldg(ga.a.la + id);
                    ag[x] = __ldg(ga.a.agent + id);
                    if (s.depth) dp[x] = __ldg(ga.a.depth + id);
                    Q.fl |= (uint32_t)__ldg(ga.a.flags + id) << (8 * x);
                    Q.rf |= (uint32_t)__ldg(ga.a.ref + id) << (8 * x);
                    Q.tk |= (ga.a.ntok ? (uint32_t)__ldg(ga.a.ntok + id) : ga.a.block_tokens) << (8 * x);
                }
            }
            Q.la = make_uint4(la[0], la[1], la[2], 0u);
            Q.ag = make_uint2(ag[0] | ag[1] << 16, ag[2]);
            Q.dp = make_uint2(dp[0] | dp[1] << 16, dp[2]);
            __syncwarp();
        }
        if (step) {
            quad_ask(ga, s, q + SG_STAGES * stride, stage);
            q += stride;
            stage = stage + 1u == SG_STAGES ? 0u : stage + 1u;
        }
        f(Q, id0, valid);
    }
    walk_drain();                                              // (empty groups)
}

// Which of a quad's entries each list may take as far as flags and reference counts tell: 0x80 in an entry's byte.
static_assert(CS_FLAG_VALID == 1 && CS_FLAG_PINNED == 2 && CS_FLAG_TIER_HOST == 4 && CS_FLAG_OTHER_COPY == 8, "bit positions below");
__device__ __forceinline__ uint32_t quad_free(const Quad4 &Q, uint32_t valid)           // valid, not pinned, unreferenced
{
    return zero_bytes(((Q.fl & 0x03030303u) ^ 0x01010101u) | Q.rf) & valid;
}
__device__ __forceinline__ uint32_t quad_host(const Quad4 &Q) { return (Q.fl << 5) & 0x80808080u; }
__device__ __forceinline__ uint32_t quad_copy(const Quad4 &Q) { return (Q.fl << 4) & 0x80808080u; }
__device__ __forceinline__ uint32_t quad_u16(const uint2 &v, int r) { return ((r < 2 ? v.x : v.y) >> ((r & 1) * 16)) & 0xFFFFu; }

// Sets `flag` in `to` where a <= b: a compare and a predicated OR.
__device__ __forceinline__ void mark_le(uint32_t &to, uint32_t flag, u64 a, u64 b)
{
    asm("{\n\t.reg .pred p;\n\tsetp.le.u64 p, %1, %2;\n\t@p or.b32 %0, %0, %3;\n\t}" : "+r"(to) : "l"(a), "l"(b), "r"(flag));
}
struct Keys { uint32_t gtab_len, A, prefer, a_star; };
// Score bits of a quad's entries, all of agents in range (two roundings, never an FMA).  t: survival factor and anchor length of each.
template <bool PF>
__device__ __forceinline__ void quad_scores(const GridArgs &ga, const Sg &s, const Keys &K, const Quad4 &Q, const uint32_t (&ag)[4], uint2 (&t)[4], uint32_t (&bits)[4])
{
    uint32_t g[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        if (PF) t[x] = lds_table2(s.agent + 8u * ag[x]);
        else t[x].x = lds_table(s.agent + 8u * ag[x]);
        const uint32_t la = u4_word(Q.la, x);
        g[x] = lds_table(s.gtab + 4u * min(max(s.now, la) - la, K.gtab_len));
    }
    if (!s.whole_table) {                                      // (a decay so slow that the table ends before saturation)
#pragma unroll 1
        for (uint32_t x = 0; x < 4u; ++x) {
            const uint32_t la = u4_word(Q.la, x), age = max(s.now, la) - la;
            if (age < K.gtab_len || age >= ga.a.age_sat) continue;
            const uint32_t v = __float_as_uint(cs_recency(ga.a.lambda, ga.a.delta, age));
            if (x == 0u) g[0] = v;
            else if (x == 1u) g[1] = v;
            else if (x == 2u) g[2] = v;
            else g[3] = v;
        }
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
        bits[x] = __float_as_uint(__fmul_rn(__fmul_rn(__uint_as_float(t[x].x), __uint_as_float(g[x])), (float)((Q.tk >> (8 * x)) & 0xFFu)));
}
__device__ __forceinline__ u64 victim_key(const Keys &K, uint32_t bits, uint32_t la, uint32_t copy)      // copy: 1 with a copy on the other tier
{
    return (u64)(K.prefer ? (bits << 1) | (copy ^ 1u) : bits) << 32 | la;
}
__device__ __forceinline__ u64 prefetch_key(const Keys &K, uint32_t bits, uint32_t la, uint32_t agent)
{
    return (u64)((agent == K.a_star ? 0u : 0x80000000u) | (~bits & 0x7FFFFFFFu)) << 32 | (uint32_t)~la;
}

// One candidate per participating lane, whole warps: to the end of its list's candidates (the scan's or the collect pass's) and, where the
// list has boundaries, into its bucket.
__device__ __noinline__ void candidates_out(const GridArgs &ga, cs_grid_state *g, uint32_t epoch, bool cand, uint32_t l, u64 km, uint32_t id, uint32_t collected)
{
    const uint32_t lane = threadIdx.x & 31;
    const ScanShared &u = SH.u.s;
    const ListShared *const list = SH.list;
    if (!cand) l = 3u;
    const uint32_t m0 = __ballot_sync(0xFFFFFFFFu, l == 0u), m1 = __ballot_sync(0xFFFFFFFFu, l == 1u), m2 = __ballot_sync(0xFFFFFFFFu, l == 2u);
    const uint32_t m_lane = lane == 0u ? m0 : (lane == 1u ? m1 : (lane == 2u ? m2 : 0u)), mine = l == 0u ? m0 : (l == 1u ? m1 : m2);
    uint32_t base = 0, b = 0xFFFFFFFFu, slot = 0;
    if (m_lane) base = atomicAdd(collected ? &g->list[epoch][lane].c_collect : &g->list[epoch][lane].c_scan, __popc(m_lane));
    const uint32_t nb = cand && !collected ? list[l].nb : 0u;
    if (nb && less96(km, id, u.b_km[l][nb], u.b_id[l][nb])) {
        b = 0;                                                 // the last bucket that starts at or below the key
        for (uint32_t step = 1u << (31 - __clz(nb)); step > 0; step >>= 1)
            if (b + step < nb && !less96(km, id, u.b_km[l][b + step], u.b_id[l][b + step])) b += step;
        slot = atomicAdd(&g->count[epoch][l][b * CS_BCOUNT_STRIDE], 1u);
    }
    const uint32_t at = __shfl_sync(0xFFFFFFFFu, base, l < 3u ? l : 0u) + __popc(mine & ((1u << lane) - 1u));
    if (cand && at < ga.a.max_blocks) {
        ga.ws[l].cand_km[at] = km;
        ga.ws[l].cand_id[at] = id;
    }
    if (b != 0xFFFFFFFFu && slot < list[l].cap) {
        ga.ws[l].sort_km[(size_t)b * list[l].cap + slot] = km;
        ga.ws[l].sort_id[(size_t)b * list[l].cap + slot] = id;
    }
    __syncwarp();
}

// ---- 1 scan ---------------------------------------------------------------------------------------------------------------------------
// Candidates of a warp gather in its queue, whichever list they are for.
__device__ __forceinline__ void queue_out(const GridArgs &ga, const Sg &s, uint32_t &n, uint32_t collected)
{
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ScanShared &u = SH.u.s;
    __syncwarp();
    for (uint32_t i0 = 0; i0 < n; i0 += 32u) {
        const uint32_t i = i0 + lane;
        const bool have = i < n;
        const u64 km = have ? u.q_km[warp][i] : 0ull;
        const uint32_t id = have ? u.q_id[warp][i] : 0u, l = have ? u.q_list[warp][i] : 0u;
        candidates_out(ga, s.g, s.epoch, have, l, km, id, collected);
    }
    n = 0;
}
__device__ __forceinline__ void queue_one(const GridArgs &ga, const Sg &s, uint32_t &n, bool cand, uint32_t l, u64 km, uint32_t id, uint32_t collected)     // whole warps
{
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, cand), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (cand) {
        const uint32_t at = n + __popc(b & ((1u << lane) - 1u));
        SH.u.s.q_km[warp][at] = km;
        SH.u.s.q_id[warp][at] = id;
        SH.u.s.q_list[warp][at] = (uint8_t)l;
    }
    n += __popc(b);
    if (n > SG_QUEUE - 32u) queue_out(ga, s, n, collected);
}

// TIERS: tiers whose victims are wanted, PF: the prefetch list.
//
// Every entry's key, compared with its list's remembered one.  Bound by the instructions issued per entry: HBM leaves a scheduler 200 issue
// slots per warp and quad (128 entries) of a large index.  (One compare of last_access with its agent's cut, as in cs_sel_fast_kernel, saves
// two table look-ups and two products per entry, but blocks of another size, one in twenty, then need a second look with queues of their own
// and the cuts 1 to 3 us of searching before the first compare.)
template <int TIERS, bool PF>
__device__ __forceinline__ void scan_index(const GridArgs &ga, const Sg &s, uint32_t want, uint32_t collected)       // collected: 1 for the pass after a histogram
{
    const Keys K = {ga.a.gtab_len, ga.a.A, ga.a.prefer_copy, s.a_star};
    const uint32_t lane = threadIdx.x & 31;
    const bool host_tier = (ga.want & 2u) != 0;                                             // (TIERS == 1: the tier)
    const uint32_t pat = host_tier ? 0x05050505u : 0x01010101u;
    const uint32_t open_g = want & 1u ? 0xFFFFFFFFu : 0u, open_h = want & 2u ? 0xFFFFFFFFu : 0u;      // (lists without a key are not scanned for)
    const u64 T_g = SH.list[TIERS == 1 && host_tier ? 1 : 0].bound, T_h = SH.list[1].bound, T_p = SH.list[2].bound;
    uint32_t n = 0, elig_g = 0, elig_h = 0, elig_p = 0;
    walk(ga, s, [&](const Quad4 &Q, uint32_t id0, uint32_t valid) {
        uint32_t v_e = 0, p_e = 0, host = 0, copy = quad_copy(Q);
        if (TIERS == 1 && !PF) {
            v_e = zero_bytes(((Q.fl & 0x07070707u) ^ pat) | Q.rf) & valid & (host_tier ? open_h : open_g);
        } else {
            const uint32_t free = quad_free(Q, valid);
            host = quad_host(Q);
            if (TIERS) v_e = (free & host & open_h) | (free & ~host & open_g);
            if (PF) p_e = want & 4u ? free & host & ~copy : 0u;
        }
        uint32_t ag[4] = {Q.ag.x & 0xFFFFu, Q.ag.x >> 16, Q.ag.y & 0xFFFFu, Q.ag.y >> 16};
        const uint32_t most = __vmaxu2(Q.ag.x, Q.ag.y);
        if (max(most & 0xFFFFu, most >> 16) >= K.A) {              // an entry of no agent is reported, and in no list
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                if (ag[x] < K.A) continue;
                const uint32_t flag = 0x80u << (8 * x);
                if ((v_e | p_e) & flag) atomicOr(&ga.ws[0].sc->status, CS_ST_BAD_AGENT);
                v_e &= ~flag;
                p_e &= ~flag;
                ag[x] = 0;
            }
        }
        uint32_t bits[4], cand_v = 0, cand_p = 0, inside = 0;
        uint2 t[4];
        quad_scores<PF>(ga, s, K, Q, ag, t, bits);
        if (TIERS) {
            uint32_t pr[4] = {bits[0], bits[1], bits[2], bits[3]};
            if (K.prefer) {                                        // (a victim key's first word; as victim_key() has it)
#pragma unroll
                for (int x = 0; x < 4; ++x) pr[x] = (bits[x] << 1) | ((~copy >> (8 * x + 7)) & 1u);
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const uint32_t flag = 0x80u << (8 * x);
                mark_le(cand_v, flag, (u64)pr[x] << 32 | u4_word(Q.la, x), TIERS == 2 && host & flag ? T_h : T_g);
            }
        }
        if (PF) {
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const uint32_t flag = 0x80u << (8 * x);
                mark_le(inside, flag, (u64)quad_u16(Q.dp, x) + 1ull, (u64)t[x].y);
                mark_le(cand_p, flag, prefetch_key(K, bits[x], u4_word(Q.la, x), ag[x]), T_p);
            }
        }
        if (PF) p_e &= inside;
        if (TIERS == 2) { elig_h += __popc(v_e & host); elig_g += __popc(v_e & ~host); }
        else if (TIERS == 1) elig_g += __popc(v_e);
        if (PF) elig_p += __popc(p_e);
        cand_v &= v_e;
        cand_p &= p_e;
        while (__any_sync(0xFFFFFFFFu, (cand_v | cand_p) != 0u)) {             // one entry per lane and round
            const bool have = (cand_v | cand_p) != 0u, pf = cand_v == 0u;
            const uint32_t w = pf ? cand_p : cand_v, x = w ? (uint32_t)(__ffs(w) - 1) >> 3 : 0u, flag = w & (0u - w);
            const uint32_t la = u4_word(Q.la, x), b = x == 0u ? bits[0] : (x == 1u ? bits[1] : (x == 2u ? bits[2] : bits[3]));
            const uint32_t g = x == 0u ? ag[0] : (x == 1u ? ag[1] : (x == 2u ? ag[2] : ag[3])), tier = TIERS == 2 ? (host & flag ? 1u : 0u) : (host_tier ? 1u : 0u);
            const u64 km = PF && pf ? prefetch_key(K, b, la, g) : victim_key(K, b, la, copy & flag ? 1u : 0u);
            if (pf) cand_p &= ~flag;
            else cand_v &= ~flag;
            queue_one(ga, s, n, have, PF && pf ? 2u : tier, km, id0 + x, collected);
        }
    });
    if (n) queue_out(ga, s, n, collected);
    if (collected) return;
    if (TIERS == 1 && host_tier) { elig_h = elig_g; elig_g = 0; }
    const uint32_t g = __reduce_add_sync(0xFFFFFFFFu, elig_g), h = __reduce_add_sync(0xFFFFFFFFu, elig_h),
                   p = __reduce_add_sync(0xFFFFFFFFu, elig_p);
    if (lane == 0) {
        if (g) atomicAdd(SH.elig + 0, g);
        if (h) atomicAdd(SH.elig + 1, h);
        if (p) atomicAdd(SH.elig + 2, p);
    }
}

// ---- a miss: a histogram of all keys ----------------------------------------------------------------------------------------------------
// Then the scan again, below the histogram's threshold.  (4,000,000 entries, one list, all together 66 us; a loop over entries and lists that did
// both passes 105, the chain's 70.)
struct Bins { uint32_t bin_lo, bin_shift; };
// Adjacent entries of a thread often share a bin: they are counted once.
struct BinRun { uint32_t at, n; };
__device__ __forceinline__ void bin_count(BinRun &r, bool take, uint32_t at)
{
    if (take && at != r.at) {
        if (r.n) atomicAdd(SH.u.hist[0] + r.at, r.n);
        r.at = at;
        r.n = 0;
    }
    if (take) ++r.n;
}
template <int TIERS, bool PF>
__device__ __forceinline__ void count_index(const GridArgs &ga, const Sg &s, uint32_t lists)
{
    const Keys K = {ga.a.gtab_len, ga.a.A, ga.a.prefer_copy, s.a_star};
    const Bins victims = {ga.bin_lo[0], ga.bin_shift[0]}, prefetch = {ga.bin_lo[2], ga.bin_shift[2]};
    const uint32_t open_g = lists & 1u ? 0xFFFFFFFFu : 0u, open_h = lists & 2u ? 0xFFFFFFFFu : 0u, open_p = lists & 4u ? 0xFFFFFFFFu : 0u;
    BinRun of_v = {0u, 0u}, of_p = {0u, 0u};
    walk(ga, s, [&](const Quad4 &Q, uint32_t, uint32_t valid) {
        const uint32_t free = quad_free(Q, valid), host = quad_host(Q), copy = quad_copy(Q);
        uint32_t v_e = (free & host & open_h) | (free & ~host & open_g), p_e = PF ? free & host & ~copy & open_p : 0u, bits[4], ag[4];
        uint2 t[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            ag[x] = quad_u16(Q.ag, x);
            if (ag[x] < K.A) continue;
            const uint32_t flag = 0x80u << (8 * x);
            if ((v_e | p_e) & flag) atomicOr(&ga.ws[0].sc->status, CS_ST_BAD_AGENT);
            v_e &= ~flag;
            p_e &= ~flag;
            ag[x] = 0;
        }
        quad_scores<PF>(ga, s, K, Q, ag, t, bits);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const uint32_t flag = 0x80u << (8 * x), la = u4_word(Q.la, x);
            if (TIERS)
                bin_count(of_v, (v_e & flag) != 0u, (host & flag ? CS_HIST_BINS : 0u) +
                          bin_of<false>(victims, (uint32_t)(victim_key(K, bits[x], la, copy & flag ? 1u : 0u) >> 32)));
            if (PF)
                bin_count(of_p, (p_e & flag) != 0u && quad_u16(Q.dp, x) < t[x].y, 2u * CS_HIST_BINS +
                          bin_of<true>(prefetch, (uint32_t)(prefetch_key(K, bits[x], la, ag[x]) >> 32)));
        }
    });
    if (of_v.n) atomicAdd(SH.u.hist[0] + of_v.at, of_v.n);
    if (of_p.n) atomicAdd(SH.u.hist[0] + of_p.at, of_p.n);
}

// The histogram of a list that missed, summed over the CTAs: threshold bin, keys at or below it, eligible entries.
template <bool PF>
__device__ __noinline__ void list_threshold(const GridArgs &ga, uint32_t l)
{
    constexpr uint32_t PER = CS_HIST_BINS / SG_THREADS;
    const uint32_t tid = threadIdx.x, k = ga.k[l];
    uint32_t loc[PER], sum = 0;
#pragma unroll
    for (uint32_t q = 0; q < PER / 4; ++q) {
        const uint4 v = cs_ld_cg_pinned((const uint4 *)ga.ws[l].hist + tid * (PER / 4) + q);
        loc[4 * q] = v.x; loc[4 * q + 1] = v.y; loc[4 * q + 2] = v.z; loc[4 * q + 3] = v.w;
        sum += v.x + v.y + v.z + v.w;
    }
    uint32_t n_elig;
    const uint32_t before = sel_block_scan(sum, SH.part, n_elig);
    if (k && n_elig >= k && before < k && k <= before + sum) {
        uint32_t run = before;
#pragma unroll
        for (uint32_t q = 0; q < PER; ++q) {
            run += loc[q];
            if (run >= k) { SH.words[0] = tid * PER + q; SH.words[1] = run; break; }
        }
    }
    __syncthreads();
    if (tid == 0) {
        ListShared &L = SH.list[l];
        const Bins bins = {ga.bin_lo[l], ga.bin_shift[l]};
        const bool enough = n_elig >= k;
        L.b0 = enough && k ? SH.words[0] : CS_HIST_BINS - 1u;
        L.c = k == 0u ? 0u : (enough ? SH.words[1] : n_elig);
        L.n_elig = n_elig;
        L.n_out = enough ? k : n_elig;
        L.spec = 0u;
        L.bound = k ? (primary_limit<PF>(bins, L.b0) << 32) - 1ull : 0ull;
        L.nb = 0u;                                             // (its boundaries lie under the histograms)
    }
    __syncthreads();
}

// A remembered key when the clock has gone on by `passed` (or back).  The ends of the range stay what they are.
__device__ __forceinline__ u64 moved_key(u64 km, uint32_t passed, bool pf)
{
    if (km >= ~0ull - 1ull) return km;
    const long long la = (long long)(pf ? ~(uint32_t)km : (uint32_t)km) + (int)passed;
    const uint32_t at = la < 0ll ? 0u : (la > 0xFFFFFFFFll ? 0xFFFFFFFFu : (uint32_t)la);
    return (km & 0xFFFFFFFF00000000ull) | (pf ? ~at : at);
}
// The key that the next call of the kind gets.
__device__ __forceinline__ u64 list_next_bound(const ListShared &L, uint32_t k, u64 ahead, u64 kth)
{
    cs_sel_state st;
    st.c = L.c;
    st.n_elig = L.n_elig;
    st.bound = L.bound;
    st.ahead = ahead;
    st.spec = L.spec;
    return next_bound(st, k, kth, sg_ahead(k));
}
__device__ __forceinline__ void remember_bound(const GridArgs &ga, cs_grid_state *g, const ListShared &L, uint32_t l, u64 bound)
{
    ga.ws[0].sc->sel_T[l] = bound;
    g->rem_T[l] = bound;
    g->rem_now[l] = L.now;
}
// Where the boundaries for the next call lie in this one's order: every step-th key up to `end`, more than a list beyond its own end, because
// a list's entries may be gone by then.
struct NextBuckets { uint32_t step, nb, end; };
__device__ __forceinline__ NextBuckets next_buckets(uint32_t n_out, uint32_t ranked)        // ranked: keys whose places are known
{
    NextBuckets N;
    N.end = min(2u * n_out + n_out / 4u + 256u, ranked);
    N.step = max(SG_STEP, (N.end + CS_BUCKETS - 1u) / CS_BUCKETS);
    N.nb = (N.end + N.step - 1u) / N.step;
    return N;
}

// ---- 2 finish: buckets filled by the scan ---------------------------------------------------------------------------------------------------
// Whether a bucket is wanted: for the list, or for the next call's boundaries.
__device__ __forceinline__ bool bucket_wanted(const ListShared &L, uint32_t off) { return off < L.ranked && (off < L.n_out || off <= L.end); }
// One key at its place in the order.
__device__ __forceinline__ void key_out(const GridArgs &ga, cs_grid_state *g, uint32_t l, uint32_t pos, u64 km, uint32_t id, bool sampled)
{
    const ListShared &L = SH.list[l];
    if (pos < L.n_out) ga.ids[l][pos] = id;
    if (!ga.speculate) return;
    if (pos == L.n_out - 1u && (sampled || L.c <= sg_ahead(ga.k[l]) / 4u * 5u))
        remember_bound(ga, g, L, l, list_next_bound(L, ga.k[l], sampled ? cs_ld_cg_pinned(&g->list[L.epoch][l].ahead) : ~0ull, km));
    if (sampled || L.refresh) return;                          // (the next boundaries are the sample's)
    const uint32_t j = pos / L.step;
    if (pos && pos < L.end && j * L.step == pos) { g->rem_km[l][j] = km; g->rem_id[l][j] = id; }
    if (pos == L.end && L.end < L.ranked) { g->rem_km[l][L.next_nb] = km; g->rem_id[l][L.next_nb] = id; }
    if (pos + 1u == L.end && L.end == L.ranked) {              // the last one known: the end lies right behind it, or nowhere
        g->rem_km[l][L.next_nb] = L.end == L.c ? ~0ull : km;
        g->rem_id[l][L.next_nb] = L.end == L.c ? 0xFFFFFFFFu : id + 1u;
    }
}

// Exclusive prefix sums of four values per thread over the CTA, and their totals.
__device__ __forceinline__ void block_scan4(uint32_t (&v)[4], uint32_t (&total)[4])
{
    uint32_t *const s_part = SH.part;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    uint32_t incl[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl[l], d);
            if (lane >= d) incl[l] += t;
        }
    if (lane == 31)
#pragma unroll
        for (int l = 0; l < 4; ++l) s_part[64 * l + warp] = incl[l];
    __syncthreads();
    if (warp < 4u) {
        uint32_t w = lane < n_warps ? s_part[64u * warp + lane] : 0u;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, w, d);
            if (lane >= d) w += t;
        }
        s_part[64u * warp + 32u + lane] = w;
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        total[l] = s_part[64 * l + 63];
        v[l] = (warp ? s_part[64 * l + 32 + warp - 1] : 0u) + incl[l] - v[l];
    }
}

// The keys [8 sub, 8 sub + 8) of a bucket of m keys, ranked within it by the calling warp, four lanes to a key.  The bucket comes through
// shared memory, SG_KEYS at a time: one trip, where eight keys per lane and round took one per round.
#define SG_PART 8u
__device__ __noinline__ void rank_in_bucket(const GridArgs &ga, cs_grid_state *g, uint32_t l, uint32_t b, uint32_t sub, uint32_t m, uint32_t off,
                                            bool sampled)
{
    const ListShared &L = SH.list[l];
    uint4 *const key = SH.step.finish.key[threadIdx.x >> 5];
    const uint32_t lane = threadIdx.x & 31, own = SG_PART * sub + lane / 4u;
    const u64 *km = ga.ws[l].sort_km + (size_t)b * L.cap;
    const uint32_t *id = ga.ws[l].sort_id + (size_t)b * L.cap;
    const u64 my = cs_ld_cg_pinned(km + min(own, m - 1u));
    const uint32_t mine = cs_ld_cg_pinned(id + min(own, m - 1u));
    uint32_t rank = 0;
    u64 o_km[SG_KEYS / 32u];
    uint32_t o_id[SG_KEYS / 32u];
    auto ask = [&](uint32_t k0) {
#pragma unroll
        for (uint32_t h = 0; h < SG_KEYS / 32u; ++h) {
            const uint32_t o = k0 + 32u * h + lane;
            if (k0 + 32u * h < m) { o_km[h] = cs_ld_cg_pinned(km + min(o, m - 1u)); o_id[h] = cs_ld_cg_pinned(id + min(o, m - 1u)); }
        }
    };
    ask(0u);
    for (uint32_t k0 = 0; k0 < m; k0 += SG_KEYS) {
        const uint32_t n = min(SG_KEYS, m - k0);
        __syncwarp();
#pragma unroll
        for (uint32_t h = 0; h < SG_KEYS / 32u; ++h)
            if (32u * h < n) key[32u * h + lane] = make_uint4(o_id[h], (uint32_t)o_km[h], (uint32_t)(o_km[h] >> 32), 0u);
        __syncwarp();
        if (k0 + SG_KEYS < m) ask(k0 + SG_KEYS);               // (the next ones travel while these are counted)
#pragma unroll 4
        for (uint32_t q = lane & 3u; q < n; q += 4u) {
            const uint4 v = key[q];
            count_less(rank, (u64)v.z << 32 | v.y, v.x, my, mine);
        }
    }
    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 1);
    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 2);
    if (own < m && (lane & 3u) == 0u) key_out(ga, g, l, off + rank, my, mine, sampled);
    __syncwarp();
}

// The lists whose candidates lie in buckets -- by the scan, or (sampled) by the sample's boundaries -- put in order, as far as share `cta` goes;
// returns those whose buckets can be, the same ones for every share.
__device__ __noinline__ uint32_t order_by_buckets(const GridArgs &ga, cs_grid_state *g, uint32_t epoch, uint32_t cta, uint32_t lists, bool sampled)
{
    ListShared *const list = SH.list;
    FinishShared &F = SH.step.finish;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = gridDim.x;
    // ---- one trip: the counts, and the keys of the bucket that is this warp's (bucket x belongs to share x % G) -------------------------------
    const uint32_t my_x = cta + G * warp, my_l = my_x / CS_BUCKETS, my_b = my_x % CS_BUCKETS;
    const bool my_any = my_l < 3u && (lists >> my_l) & 1u && my_b < list[my_l < 3u ? my_l : 0u].nb;
    uint32_t n[3], c_scan = 0, eligible = 0, id[3] = {};
    u64 km[3] = {};
    if (tid < 3u && !sampled) {
        c_scan = cs_ld_cg_pinned(&g->list[epoch][tid].c_scan);
        eligible = cs_ld_cg_pinned(&g->list[epoch][tid].eligible);
    }
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l) {
        n[l] = 0;
        if ((lists >> l) & 1u && tid < list[l].nb) n[l] = cs_ld_cg_pinned(sampled ? &CS_BCOUNT(ga.ws[l], tid) : &g->count[epoch][l][tid * CS_BCOUNT_STRIDE]);
    }
    if (my_any) {
        const uint32_t cap = list[my_l].cap;
        const size_t at = (size_t)my_b * cap;
#pragma unroll
        for (uint32_t h = 0; h < 3u; ++h)
            if (lane + 32u * h < cap) {
                km[h] = cs_ld_cg_pinned(ga.ws[my_l].sort_km + at + lane + 32u * h);
                id[h] = cs_ld_cg_pinned(ga.ws[my_l].sort_id + at + lane + 32u * h);
            }
    }
    if (tid < 3u && (lists >> tid) & 1u) {
        ListShared &L = list[tid];
        if (!sampled) {
            const uint32_t k = ga.k[tid];
            // complete when the k winners lie at or below the key, when fewer than k entries are eligible and all of them do, or when k = 0
            L.spec = k == 0 || c_scan >= k || c_scan == eligible ? 1u : 0u;
            L.c = k ? c_scan : 0u;
            L.n_elig = eligible;
            L.n_out = min(eligible, k);
        }
        L.bad_at = 0xFFFFFFFFu;
    }
    uint32_t at[4] = {n[0], n[1], n[2], 0u}, sum[4], parts[3];
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l) {                        // buckets for more than one warp, and those that no warp of a small grid has
        const bool shared = n[l] > SG_BUCKET_WARP || l * CS_BUCKETS + tid >= G * SG_WARPS;
        parts[l] = shared && n[l] <= SG_BUCKET_MAX ? (n[l] + SG_PART - 1u) / SG_PART : 0u;
        at[3] += parts[l];
    }
    block_scan4(at, sum);                              // (orders the words above as well)
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l) {
        F.off[l][tid] = at[l];
        F.cnt[l][tid] = n[l];
        if (n[l] > min(list[l].cap, SG_BUCKET_MAX)) atomicMin(&list[l].bad_at, at[l]);
        // part x of the whole grid's belongs to share x % G
        for (uint32_t x = at[3] + (cta + G - at[3] % G) % G; x < at[3] + parts[l]; x += G)
            if (x / G < SG_MAP) F.map[x / G] = l << 30 | tid << 16 | (x - at[3]);
        at[3] += parts[l];
    }
    __syncthreads();
    if (tid < 3u && (lists >> tid) & 1u) {
        ListShared &L = list[tid];
        L.ranked = min(tid == 0u ? sum[0] : (tid == 1u ? sum[1] : sum[2]), L.bad_at);
        L.refresh = L.ranked < min(L.c, L.n_out + L.n_out / 2u + 128u) ? 1u : 0u;
        const NextBuckets N = next_buckets(L.n_out, sampled || L.refresh ? L.c : L.ranked);
        L.step = N.step;
        L.next_nb = N.nb;
        L.end = N.end;
    }
    __syncthreads();
    uint32_t done = 0;
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l) {
        const ListShared &L = list[l];
        if ((lists >> l) & 1u && L.spec | sampled && L.n_out && L.nb && L.ranked >= L.n_out && sum[3] <= SG_MAP * G) done |= 1u << l;
    }
    if (!done) return 0u;
    // ---- the keys of a bucket are counted within it ---------------------------------------------------------------------------------------------
    uint4 *key = F.key[warp];
    if (my_any && (done >> my_l) & 1u) {
        const ListShared &L = list[my_l];
        const uint32_t m = F.cnt[my_l][my_b], off = F.off[my_l][my_b];
        if (m && m <= SG_BUCKET_WARP && bucket_wanted(L, off)) {
#pragma unroll
            for (uint32_t h = 0; h < 3u; ++h) key[lane + 32u * h] = make_uint4(id[h], (uint32_t)km[h], (uint32_t)(km[h] >> 32), 0u);
            __syncwarp();
            uint32_t r[3] = {};
            auto count = [&](auto keys) {                      // (keys per lane, as a constant)
#pragma unroll 4
                for (uint32_t q = 0; q < m; ++q) {
                    const uint4 v = key[q];
#pragma unroll
                    for (uint32_t h = 0; h < decltype(keys)::value; ++h) count_less(r[h], (u64)v.z << 32 | v.y, v.x, km[h], id[h]);
                }
            };
            if (m <= 32u) count(std::integral_constant<uint32_t, 1>());
            else if (m <= 64u) count(std::integral_constant<uint32_t, 2>());
            else count(std::integral_constant<uint32_t, 3>());
#pragma unroll
            for (uint32_t h = 0; h < 3u; ++h)
                if (lane + 32u * h < m) key_out(ga, g, my_l, off + r[h], km[h], id[h], sampled);
            __syncwarp();
        }
    }
    const uint32_t n_parts = sum[3] > cta ? (sum[3] - cta + G - 1u) / G : 0u;
    for (uint32_t i = SG_WARPS - 1u - warp; i < n_parts; i += SG_WARPS) {         // (the last warps have no bucket of their own)
        const uint32_t it = F.map[i], l = it >> 30, b = (it >> 16) & 0x3FFFu;
        const ListShared &L = list[l];
        if ((done >> l) & 1u && bucket_wanted(L, F.off[l][b])) rank_in_bucket(ga, g, l, b, it & 0xFFFFu, F.cnt[l][b], F.off[l][b], sampled);
    }
    if (cta == 0 && tid < 3u && (done >> tid) & 1u) {
        if (ga.speculate) g->rem_n[tid] = list[tid].next_nb;
        atomicAdd((unsigned long long *)&ga.ws[0].cnt->region_selects[tid], 1ull);
    }
    return done;
}

// A sample of a list's candidates, ranked by all CTAs, for the next call: where its buckets begin (boundaries; too few keys were ranked), and a
// lower key (bound; too many candidates lay below this one).
__device__ __noinline__ void sample_for_next(const GridArgs &ga, cs_grid_state *g, uint32_t share, uint32_t l, bool boundaries, bool bound)
{
    const ListShared &L = SH.list[l];
    SampleShared &M = SH.step.sample;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, S = min(L.c, CS_SAMPLE);
    __syncthreads();
    for (uint32_t i = tid; i < CS_SAMPLE; i += SG_THREADS) {
        const uint32_t at = (uint32_t)((u64)i * L.c / S);
        M.km[i] = i < S ? __ldcg(ga.ws[l].cand_km + at) : ~0ull;
        M.id[i] = i < S ? __ldcg(ga.ws[l].cand_id + at) : 0xFFFFFFFFu;
    }
    __syncthreads();
    const uint32_t want = (uint32_t)((u64)sg_ahead(ga.k[l]) * S / L.c);
    for (uint32_t i = share * SG_WARPS + warp; i < S; i += gridDim.x * SG_WARPS) {
        uint32_t r = 0;
#pragma unroll 8
        for (uint32_t q = lane; q < CS_SAMPLE; q += 32u) count_less(r, M.km[q], M.id[q], M.km[i], M.id[i]);
        r = __reduce_add_sync(0xFFFFFFFFu, r);
        if (bound && lane == 0 && r == want) remember_bound(ga, g, L, l, M.km[i] < ~0ull - 1ull ? M.km[i] : ~0ull - 1ull);
        if (!boundaries) continue;
        // the boundaries whose places come to this sample's rank (a boundary between two samples is the upper one)
        const uint32_t lo = max(1u, (uint32_t)(((u64)r * L.c + (u64)S * L.step - 1u) / ((u64)S * L.step)));
        for (uint32_t j = lo + lane; j < L.next_nb && (u64)j * L.step * S / L.c == r; j += 32u) { g->rem_km[l][j] = M.km[i]; g->rem_id[l][j] = M.id[i]; }
        if (lane == 0 && L.end < L.c && (uint32_t)((u64)L.end * S / L.c) == r) { g->rem_km[l][L.next_nb] = M.km[i]; g->rem_id[l][L.next_nb] = M.id[i]; }
    }
    if (boundaries && share == 0 && tid == 0 && L.end == L.c) { g->rem_km[l][L.next_nb] = ~0ull; g->rem_id[l][L.next_nb] = 0xFFFFFFFFu; }
}

// Lists whose buckets do not hold: a ranked sample, buckets between the samples, keys counted within them.  Two more grid barriers.  The lists
// share the CTAs up to there: one after the other, every list would take the trips of all its steps.  false: a wait ran out.
__device__ __noinline__ bool order_by_sample(const GridArgs &ga, cs_grid_state *g, uint32_t number, uint32_t lists)
{
    StepShared &S = SH.step;
    const uint32_t tid = threadIdx.x, G = gridDim.x, n_lists = __popc(lists), epoch = number & 1u;
    uint32_t many = 0;
    for (uint32_t x = 0; x < 3u; ++x)
        if ((lists >> x) & 1u && SH.list[x].c > FEW_MAX) many |= 1u << x;
    for (uint32_t o = 0; o < SH.n_own; ++o) {
        const uint32_t share = SH.own[o], turn = share % n_lists, l = __fns(lists, 0u, turn + 1u);      // the share's list
        const uint32_t my_cta = share / n_lists, my_G = (G - turn + n_lists - 1u) / n_lists;
        const ListShared &L = SH.list[l];
        const cs_workspace &ws = ga.ws[l];
        const NextBuckets N = next_buckets(L.n_out, L.c);
        if (my_cta == 0) CS_BCOUNT(ws, tid) = 0;
        __syncthreads();
        rank_sample(ws, L.c, L.n_out, sg_ahead(ga.k[l]), &g->list[epoch][l].ahead, S.sample.km, S.sample.id, my_cta, my_G, ga.ids[l], [&](uint32_t pos, u64 km, uint32_t id) {
            if (!ga.speculate) return;
            if (pos && pos < N.end && pos % N.step == 0u) { g->rem_km[l][pos / N.step] = km; g->rem_id[l][pos / N.step] = id; }
            if (pos == N.end) { g->rem_km[l][N.nb] = km; g->rem_id[l][N.nb] = id; }
            if (pos == L.c - 1u && N.end == L.c) { g->rem_km[l][N.nb] = ~0ull; g->rem_id[l][N.nb] = 0xFFFFFFFFu; }
            if (pos == L.n_out - 1u) remember_bound(ga, g, L, l, list_next_bound(L, ga.k[l], ~0ull, km));
        });
        if (my_cta == 0 && tid == 0 && ga.speculate) g->rem_n[l] = N.nb;
    }
    if (!many) return true;
    if (!all_here(ga, g, number, 3u)) return false;
    for (uint32_t o = 0; o < SH.n_own; ++o) {
        const uint32_t share = SH.own[o], turn = share % n_lists, l = __fns(lists, 0u, turn + 1u);
        const uint32_t my_cta = share / n_lists, my_G = (G - turn + n_lists - 1u) / n_lists;
        if (!((many >> l) & 1u)) continue;
        const ListShared &L = SH.list[l];
        const NextBuckets N = next_buckets(L.n_out, L.c);
        PlaceShared &Q = S.place;
        if (o) __syncthreads();
        place_candidates(ga.ws[l], make_uint4(L.c, L.n_out, L.n_elig, 0u), ga.a.max_blocks, ga.a.region_cap_max, Q.s_km, Q.s_id, Q.b_km, Q.b_id, my_cta, my_G, [] {});
        if (my_cta == my_G - 1u && ga.speculate) {
            // the next call's boundaries out of the sample
            for (uint32_t j = tid + 1u; j <= N.nb; j += SG_THREADS) {
                const u64 at = (u64)(j < N.nb ? j * N.step : N.end) * CS_SAMPLE;
                const uint32_t x = (uint32_t)(at / L.c), f = (uint32_t)(at % L.c);           // between sample x - 1 and sample x
                const bool last = j == N.nb && N.end == L.c;
                const u64 lo = x ? Q.s_km[x - 1u] : 0ull, hi = x < CS_SAMPLE ? Q.s_km[x] : L.bound, gap = hi > lo ? hi - lo : 0ull;
                g->rem_km[l][j] = last ? ~0ull : lo + gap / L.c * f;
                g->rem_id[l][j] = last ? 0xFFFFFFFFu : (x && !(gap / L.c * f) ? Q.s_id[x - 1u] : 0u);
            }
        }
    }
    if (!all_here(ga, g, number, 4u)) return false;
    if (tid < 3u && (many >> tid) & 1u) {
        const OrderPlan P = order_plan(SH.list[tid].c, SH.list[tid].n_out, ga.a.max_blocks, ga.a.region_cap_max);
        SH.list[tid].nb = P.nb;
        SH.list[tid].cap = P.cap;
    }
    uint32_t left = 0;
    for (uint32_t o = 0; o < SH.n_own; ++o) {
        __syncthreads();
        left = many & ~order_by_buckets(ga, g, epoch, SH.own[o], many, true);
    }
    // ---- buckets that outgrew their regions, or have too many keys for a warp: every bucket by a CTA
    for (uint32_t x = 0; x < 3u; ++x) {
        if (!((left >> x) & 1u)) continue;
        const ListShared &X = SH.list[x];
        const cs_workspace &w = ga.ws[x];
        const OrderPlan P = order_plan(X.c, X.n_out, ga.a.max_blocks, ga.a.region_cap_max);
        const uint32_t n_t = cs_ld_cg_pinned(&CS_BCOUNT(w, tid));
        const u64 ahead = cs_ld_cg_pinned(&g->list[epoch][x].ahead);
        for (uint32_t o = 0; o < SH.n_own; ++o)
            for (uint32_t b = SH.own[o]; b < P.nb; b += G) {
                __syncthreads();
                if (tid < 3u) SH.words[tid] = 0;
                __syncthreads();
                finish_bucket(w, X.c, X.n_out, P, b, n_t, cs_ld_cg_pinned(&CS_BCOUNT(w, b)), x, S.sample.km, S.sample.id, SH.words, SH.words + 1, SH.words + 2, ga.ids[x],
                              [&](uint32_t pos, u64 km, uint32_t) {
                                  if (ga.speculate && pos == X.n_out - 1u) remember_bound(ga, g, X, x, list_next_bound(X, ga.k[x], ahead, km));
                              });
            }
    }
    return true;
}

// Lists without the candidates they need: a histogram of the full keys, a threshold, another look at the index.  primed: the first tiles of the CTA's own
// share are on their way.  false: a wait ran out.
template <int TIERS, bool PF>
__device__ __noinline__ bool collect_missed(const GridArgs &ga, Sg s, uint32_t number, uint32_t missed, bool primed, bool first)
{
    ScanOrHist *const u = &SH.u;
    const uint32_t tid = threadIdx.x;
    __syncthreads();                                           // (the tiles' place is the copies' again)
    for (uint32_t i = tid; i < 3u * CS_HIST_BINS; i += SG_THREADS) u->hist[0][i] = 0;
    __syncthreads();
    for (uint32_t o = 0; o < SH.n_own; ++o) {
        s.share = SH.own[o];                                   // (its own is the first)
        if (o || !primed) walk_start(ga, s);
        count_index<TIERS, PF>(ga, s, missed);
    }
    __syncthreads();
    for (uint32_t l = 0; l < 3u; ++l) {
        if (!((missed >> l) & 1u)) continue;
        for (uint32_t i = tid; i < CS_HIST_BINS; i += SG_THREADS) {
            const uint32_t v = u->hist[l][i];
            if (v) atomicAdd(&ga.ws[l].hist[i], v);
        }
    }
    if (!all_here(ga, s.g, number, 1u)) return false;
    uint32_t collect = 0;
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l) {
        if (!((missed >> l) & 1u)) continue;
        if (PF && l == 2u) list_threshold<true>(ga, l);
        else list_threshold<false>(ga, l);
        if (ga.k[l]) collect |= 1u << l;
    }
    for (uint32_t o = 0; collect && o < SH.n_own; ++o) {
        s.share = SH.own[o];
        walk_start(ga, s);
        scan_index<TIERS, PF>(ga, s, collect, 1u);
    }
    if (!all_here(ga, s.g, number, 2u)) return false;
    if (first)                                                 // ready for the next call
        for (uint32_t l = 0; l < 3u; ++l)
            if ((missed >> l) & 1u)
                for (uint32_t i = tid; i < CS_HIST_BINS; i += SG_THREADS) ga.ws[l].hist[i] = 0;
    return true;
}

// Shares that the first barrier has given this CTA besides its own, until there are none left.
template <int TIERS, bool PF>
__device__ __noinline__ uint32_t take_over(const GridArgs &ga, Sg s, uint32_t number, uint32_t scanned, uint32_t share)
{
    const uint32_t tid = threadIdx.x;
    while (share < gridDim.x) {
        s.share = share;
        if (scanned) {
            walk_start(ga, s);
            scan_index<TIERS, PF>(ga, s, scanned, 0u);
            __syncthreads();
            if (tid < 3u && SH.elig[tid]) { atomicAdd(&s.g->list[number & 1u][tid].eligible, SH.elig[tid]); SH.elig[tid] = 0; }
        }
        share = grid_barrier(ga, s.g, number, 0u, 1u, true);
    }
    return share;
}

// ---- the kernel -------------------------------------------------------------------------------------------------------------------------------
// TIERS: tiers whose victims are wanted, PF: the prefetch list.
//
// Shared memory allows one CTA per SM, so registers are free up to what a compaction's CTAs beside it need (two of 64 threads).  Three lists of 20,000 out of
// 4,000,000 entries, static index, and a select of 1,000,000 beside back-to-back compactions, us: 64 registers 37 / 36, 80 35 / 31, 96 34 / 28, 124 33 / 73.
template <int TIERS, bool PF>
__global__ void __maxnreg__(96) cs_select_grid_kernel(const __grid_constant__ GridArgs ga)
{
    const uint32_t tid = threadIdx.x, n_threads = SG_THREADS, cta = blockIdx.x, G = gridDim.x;
    const cs_workspace &ws = ga.ws[0];
    // ---- what depends on the context's constants only, before the predecessor is waited for --------------------------------------------
    const SelArgs &a = ga.a;
    ScanOrHist *const u = &SH.u;
    uint2 *const agent = (uint2 *)(sg_smem + sizeof(CtaShared));
    float *const gtab = (float *)(agent + a.A);
    cs_grid_state *const g = ws.grid;
    if (tid < 3u) SH.elig[tid] = SH.bad[tid] = 0;
    if (tid == 0) { SH.n_own = 1u; SH.own[0] = (uint16_t)cta; }
    const float g_sat = cs_recency(a.lambda, a.delta, a.age_sat);
    for (uint32_t i = tid; i <= a.gtab_len; i += n_threads) gtab[i] = i < a.gtab_len ? ws.gtab[i] : g_sat;
    __syncthreads();
    cs_wait_for_predecessor();
    if (ga.give_up == SG_LATE && cta % 3u) late_start(g);
    // ---- one trip: what is remembered and the tables that change; the first tiles behind it (a small load waits for the megabytes of all SMs
    // when these are asked for first) -------------------------------------------------------------------------------------------------------
    const bool depth = PF && a.anchor;
    u64 b_km[3], bound = ~0ull, end_km = 0, rem_T = 0;
    uint32_t b_id[3], nb = 0, end_id = 0, then = 0;
    uint2 t[2];
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l)
        if ((ga.want >> l) & 1u) { b_km[l] = cs_ld_cg_pinned(&g->rem_km[l][tid]); b_id[l] = cs_ld_cg_pinned(&g->rem_id[l][tid]); }
    // (one thread per word: 2,368 warps asking for one sector each wait for another)
    u64 taken = 0;
    if (tid == 64u) taken = atomicAdd(g->taken + cta, 1ull);
    const uint32_t *word = (tid == 33u ? &ws.sc->a_star : (tid == 34u ? &ws.sc->gate : (tid == 35u ? &ws.sc->last_agent : a.now_dev)));
    uint32_t scalar = a.now;
    if (tid >= 33u && tid < (a.now_dev ? 37u : 36u)) scalar = cs_ld_cg_pinned(word);
#pragma unroll
    for (uint32_t h = 0; h < 2u; ++h) {                        // (at most 1,024 agents, at least 512 threads)
        const uint32_t i = tid + h * n_threads;
        t[h] = make_uint2(0u, 0xFFFFFFFFu);
        if (i < a.A) t[h].x = cs_ld_cg_pinned((const uint32_t *)a.fsurv + i);
        if (depth && i < a.A) t[h].y = cs_ld_cg_pinned(a.anchor + i);
    }
    if (tid < 3u) {
        bound = cs_ld_cg_pinned(&ws.sc->sel_T[ga.speculate ? tid : 3u]);
        nb = cs_ld_cg_pinned(&g->rem_n[tid]);
        then = cs_ld_cg_pinned(&g->rem_now[tid]);
        rem_T = cs_ld_cg_pinned(&g->rem_T[tid]);
        end_km = cs_ld_cg_pinned(&g->rem_km[tid][CS_BUCKETS]);
        end_id = cs_ld_cg_pinned(&g->rem_id[tid][CS_BUCKETS]);
    }
    if (tid >= 33u && tid < 37u) SH.scalar[tid - 32u] = scalar;
    // (the share's word comes back last: it is put down further below)
#pragma unroll
    for (uint32_t h = 0; h < 2u; ++h)
        if (tid + h * n_threads < a.A) agent[tid + h * n_threads] = t[h];
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l)
        if ((ga.want >> l) & 1u) u->s.b_id[l][tid] = b_id[l];
    if (tid < 3u) {
        ListShared &L = SH.list[tid];
        u->s.b_km[tid][CS_BUCKETS] = end_km;
        u->s.b_id[tid][CS_BUCKETS] = end_id;
        L.bound = bound;
        L.known = bound != ~0ull;
        L.nb = L.known && nb <= CS_BUCKETS ? nb : 0u;
        L.then = then;
        L.moves = bound == rem_T;
        L.cap = L.nb ? a.max_blocks / L.nb : 0u;
        if (a.region_cap_max && L.cap > a.region_cap_max) L.cap = a.region_cap_max;
        L.c = L.n_elig = L.n_out = 0;
        L.spec = 1u;
        L.ranked = 0;
    }
    Sg s = {g, 0u, 0u, 0u, cta, (uint32_t)__cvta_generic_to_shared(agent), (uint32_t)__cvta_generic_to_shared(gtab), a.gtab_len == a.age_sat, depth};
    walk_start(ga, s);
    __syncthreads();
    s.a_star = SH.scalar[1];
    s.now = SH.scalar[4];
    // Blocks age as the clock goes on, and those that leave the index are replaced by those that reach their age: what is remembered stands for
    // scores and ages, so its last_access moves on with the clock.
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l)
        if ((ga.want >> l) & 1u) u->s.b_km[l][tid] = moved_key(b_km[l], s.now - SH.list[l].then, l == 2u);
    if (tid < 3u) {
        ListShared &L = SH.list[tid];
        L.now = s.now;
        u->s.b_km[tid][CS_BUCKETS] = moved_key(u->s.b_km[tid][CS_BUCKETS], s.now - L.then, tid == 2u);
        if (L.moves) L.bound = moved_key(L.bound, s.now - L.then, tid == 2u);
    }
    __syncthreads();
    const uint32_t open = ga.want & (PF && SH.scalar[2] && SH.scalar[3] < a.A ? 7u : 3u);       // (the prefetch list is empty while the gate is closed)
    uint32_t scanned = 0;
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l)
        if ((open >> l) & 1u && SH.list[l].known) scanned |= 1u << l;
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l)                          // (boundaries that are not in order are none)
        if ((scanned >> l) & 1u && tid && tid < SH.list[l].nb && less96(u->s.b_km[l][tid + 1], u->s.b_id[l][tid + 1], u->s.b_km[l][tid], u->s.b_id[l][tid]))
            SH.bad[l] = 1u;
    __syncthreads();
    if (tid < 3u && SH.bad[tid]) SH.list[tid].nb = 0;
    if (tid == 64u) {
        SH.scalar[0] = (uint32_t)taken;
        SH.lost = share_is_free(taken, (uint32_t)taken) ? 0u : 1u;
    }
    __syncthreads();
    const uint32_t number = SH.scalar[0], epoch = number & 1u;
    s.epoch = epoch;
    if (tid < 3u) SH.list[tid].epoch = epoch;
    if (SH.lost) return walk_drain();                          // (what it has read besides may be what the others have made of it since)
    const bool primed = !scanned;                              // the first tiles of a walk that nobody has begun are on their way
    if (scanned) {
        scan_index<TIERS, PF>(ga, s, scanned, 0u);
        __syncthreads();
        if (tid < 3u && SH.elig[tid]) { atomicAdd(&g->list[epoch][tid].eligible, SH.elig[tid]); SH.elig[tid] = 0; }
    }
    uint32_t at_barrier = grid_barrier(ga, g, number, 0u, 1u, true);
    if (at_barrier < G) at_barrier = take_over<TIERS, PF>(ga, s, number, scanned, at_barrier);
    const uint32_t n_own = SH.n_own;
    bool first = cta == 0;                                     // share 0 is this CTA's
    for (uint32_t o = 1; o < n_own; ++o) first |= SH.own[o] == 0;
    if (first) prepare_next_launch(g, epoch);
    if (at_barrier == SG_FAILED) {
        walk_drain();
        return give_up(ga, g);
    }
    cs_release_successor();
    uint32_t quick = scanned ? order_by_buckets(ga, g, epoch, cta, scanned, false) : 0u, missed = open & ~scanned;
    for (uint32_t o = 1; scanned && o < n_own; ++o) {
        __syncthreads();
        quick = order_by_buckets(ga, g, epoch, SH.own[o], scanned, false);
    }
#pragma unroll
    for (uint32_t l = 0; l < 3u; ++l)
        if ((scanned >> l) & 1u && !SH.list[l].spec) missed |= 1u << l;
    if (missed) {
        if (!collect_missed<TIERS, PF>(ga, s, number, missed, primed, first)) return give_up(ga, g);
    } else if (primed) {
        walk_drain();                                          // (no list is open)
    }
    // ---- the ends of the lists, and the work counters -----------------------------------------------------------------------------------
    uint32_t rest = 0;
    for (uint32_t l = 0; l < 3u; ++l) {
        if (!((ga.want >> l) & 1u)) continue;
        const ListShared &L = SH.list[l];
        for (uint32_t o = 0; L.n_out < ga.k[l] && o < n_own; ++o)
            for (uint32_t i = L.n_out + SH.own[o] * n_threads + tid; i < ga.k[l]; i += G * n_threads) ga.ids[l][i] = CS_ID_NONE;
        if (first && tid == 0) {
            *ga.n_out[l] = L.n_out;
            count_select(ws, l, L.n_elig, L.n_out);
            count_candidates(ws, l, L.c, L.spec != 0u);
        }
        if (L.n_out && !((quick >> l) & 1u)) rest |= 1u << l;
        if ((quick >> l) & 1u && ga.speculate) {
            const bool bound = L.c > sg_ahead(ga.k[l]) / 4u * 5u;
            for (uint32_t o = 0; (bound || L.refresh) && o < n_own; ++o) sample_for_next(ga, g, SH.own[o], l, L.refresh != 0u, bound);
        }
    }
    if (rest && !order_by_sample(ga, g, number, rest)) give_up(ga, g);
}

// ---- host -----------------------------------------------------------------------------------------------------------------------------------

// Asked once per process and device: shares of a launch, one per SM; 0 when the kernels' shared memory is not to be had.
struct GridDevice { int ready, ctas; };
static std::mutex g_grid_mu;
static GridDevice g_grid_dev[64];

static int grid_ctas(int device, int sm_count)
{
    if (device < 0 || device >= 64) return 0;
    std::lock_guard<std::mutex> lock(g_grid_mu);
    GridDevice &d = g_grid_dev[device];
    if (!d.ready) {
        const int most = (int)sg_smem_bytes(CS_MAX_AGENTS, CS_GTAB_MAX);
        cudaError_t e = cudaSuccess;
        for (const auto kernel : {cs_select_grid_kernel<0, true>, cs_select_grid_kernel<1, false>, cs_select_grid_kernel<1, true>,
                                  cs_select_grid_kernel<2, false>, cs_select_grid_kernel<2, true>})
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        d.ctas = e == cudaSuccess ? std::min<int>(sm_count, CS_GRID_MAX_CTAS) : 0;
        (void)cudaGetLastError();
        d.ready = 1;
    }
    return d.ctas;
}

// The lists with a count pointer, over one index.  CS_ENOTIMPL: not by this route (nothing has been enqueued).
int cs_launch_select_grid(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, const uint32_t k[3], uint32_t *const ids[3],
                          uint32_t *const n_out[3], cudaStream_t s)
{
    if (!ctx->ws.grid || ctx->grid_refused || idx->n_blocks == 0) return CS_ENOTIMPL;
    const int most = grid_ctas(ctx->device, ctx->sm_count);
    if (most < 8) return CS_ENOTIMPL;                          // (a CTA for every list at least)
    GridArgs ga;
    cs_fill_sel_args(ctx, idx, now, ctx->fsurv_override ? ctx->fsurv_override : ctx->ws.fsurv, ga.a);
    ga.want = 0;
    int job = 0;
    for (uint32_t l = 0; l < 3u; ++l) {
        ga.ws[l] = ctx->ws;
        ga.k[l] = k[l];
        ga.ids[l] = ids[l];
        ga.n_out[l] = n_out[l];
        cs_fill_sel_bins(ctx, ga.a, l == 2u);
        ga.bin_lo[l] = ga.a.bin_lo;
        ga.bin_shift[l] = ga.a.bin_shift;
        if (!n_out[l]) continue;
        if (job) {
            ga.ws[l] = ctx->ws_job[job - 1];
            if (!ctx->concurrent_selects) ga.a.max_blocks = CS_SELECT_CLUSTER_MAX_BLOCKS;      // (as the workspace is laid out)
        }
        ++job;
        ga.want |= 1u << l;
    }
    ga.speculate = ctx->no_speculation ? 0u : 1u;
    ga.give_up = ctx->grid_give_up;
    const bool pf = (ga.want & 4u) != 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = CS_USE_PDL;
    cfg.gridDim = dim3(most);                                  // (the same for every launch of a context: cs_grid_state.taken)
    cfg.blockDim = dim3(SG_THREADS);
    cfg.dynamicSmemBytes = sg_smem_bytes(ga.a.A, ga.a.gtab_len);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int tiers = (ga.want & 1u) + ((ga.want >> 1) & 1u);
    const auto kernel = tiers == 2 ? (pf ? cs_select_grid_kernel<2, true> : cs_select_grid_kernel<2, false>)
                                   : (tiers == 1 ? (pf ? cs_select_grid_kernel<1, true> : cs_select_grid_kernel<1, false>) : cs_select_grid_kernel<0, true>);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, ga);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();                              // (nothing has been enqueued)
        ctx->grid_refused = 1;
        return CS_ENOTIMPL;
    }
    ctx->n_launches++;
    return CS_OK;
}
