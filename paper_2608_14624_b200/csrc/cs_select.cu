// Block scoring (Eq. 9 / ScoreBlock of Algorithm 1) and exact, ordered top-k selection of
// eviction victims (Evict of Algorithm 1) and prefetch candidates (BetweenStep, Eq. 10-11).
//
// Every kernel that walks the block index reads the SoA metadata in 512-entry warp tiles
// (contiguous 128-, 64- and 32-bit loads; 16 entries per thread and iteration) and the select
// path never materialises the score.
// A positive fp32 score orders like its bit pattern, so each eligible entry has a 96-bit
// integer key (primary, secondary, id) and "the k best in order" is "the k smallest keys in
// ascending order":
//   victims : primary = score bits,                      secondary = last_access
//   prefetch: primary = (not a*)<<31 | ~score bits[30:0], secondary = ~last_access
//
// This file holds the choice of the way (select_route()) and the multi-launch path, used above 262,144 entries for a list's first call, for
// the largest indexes and the longest lists (others take the single launch of cs_select_cluster.cu or cs_select_grid.cu).  Six launches, none of which waits
// on another CTA outside its own cluster:
//   0 fast pass : one scan against a key remembered from the last call of this kind; when the k
//                 winners lie at or below it (the usual case) the candidates are complete and launches 1 and 2
//                 return at once.
//   1 histogram : 4096-bin histogram of the primary keys; the last CTA to finish finds
//                 the threshold bin b0 (first bin whose running count reaches k).
//   2 collect   : every eligible entry whose bin <= b0 is appended to the candidate buffer
//                 (c >= min(k, eligible) keys).
//   3 sample    : 1,024 of the candidates, ranked.
//   4 place     : what lies beyond the output's share of the sample is dropped; the rest goes to up to 512 buckets of
//                 consecutive samples, each with a fixed region of the sort arrays.
//   5 finish    : every bucket's keys are ranked by one CTA, which stores their ids.  Chooses the key that the next call of
//                 this kind gets.
// Keys are unique (the id is part of the key), so the order is total and the output does not
// depend on the order in which atomics were served.
#include "cs_common.cuh"

#include <algorithm>
#include <initializer_list>
#include <tuple>

#include "cs_select_buckets.cuh"

// ---------------------------------------------------------------------------------------------
// ScoreBlock for every entry (cs_score_blocks).
//
// Large indexes: bound by HBM; warp tiles of 512 entries, the recency table in shared memory.
// Small ones (at most SCORE_SMALL_MAX entries): bound by latency, so the index is spread over the whole GPU in units of 128
// entries, four per lane, and the recency table is read where an entry needs it (from L2, then L1): copying it takes longer
// than the work.  Per call, back to back in a CUDA graph (spread / tiles): 20,000 entries 2.2 / 4.8 us, 80,000 2.9 / 4.9 us,
// 300,000 5.7 / 4.9 us, 1,000,000 14.7 / 4.9 us (gathers from L1 are slower than from shared memory); the line lies between.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(SEL_THREADS) cs_score_kernel(SelArgs a, cs_workspace ws, float *__restrict__ out)
{
    extern __shared__ float smem[];
    Tables T;
    load_tables_static(a, ws, smem, T);
    cs_wait_for_predecessor();
    cs_release_successor();
    resolve_now(a);
    load_tables_dynamic(a, ws, T, false);
    __syncthreads();
    const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const uint32_t lane = threadIdx.x & 31, n_tiles = a.n / TILE;
    for (uint32_t t = gtid >> 5; t < n_tiles; t += nth >> 5) {
        Group G;
        load_group<false, false>(a, t, lane, G);            // the score needs agent, last_access and size only
        float s[GRP];
#pragma unroll
        for (int j = 0; j < GRP; ++j) {
            const uint32_t ag = grp_u16(G.ag0, G.ag1, j);
            const uint32_t tok = a.ntok ? grp_u8(G.tk, j) : a.block_tokens;
            if (ag < a.A) s[j] = score_of(a, T, ag, grp_u32(G, j), tok);
            else { s[j] = 0.0f; atomicOr(&ws.sc->status, CS_ST_BAD_AGENT); }
        }
        float4 *o = (float4 *)out + t * 128u + lane;         // quad q of this lane: coalesced 512 B per warp store
#pragma unroll
        for (int q = 0; q < 4; ++q) __stcs(o + 32 * q, make_float4(s[4 * q], s[4 * q + 1], s[4 * q + 2], s[4 * q + 3]));
    }
    const uint32_t t0 = n_tiles * TILE;
    if (gtid < a.n - t0) {
        const uint32_t i = t0 + gtid;
        const uint32_t ag = a.agent[i];
        const uint32_t tok = a.ntok ? a.ntok[i] : a.block_tokens;
        if (ag < a.A) out[i] = score_of(a, T, ag, a.la[i], tok);
        else { out[i] = 0.0f; atomicOr(&ws.sc->status, CS_ST_BAD_AGENT); }
    }
}

#define SCORE_SMALL_THREADS 256u
#define SCORE_SMALL_MAX (1u << 17)
// SEARCH (at most 32 agents): the search of Eq. 7 / 8 from the sources as well, by every warp for itself -- lane v holds agent v's
// predecessors and in the end its survival factor -- so that it needs no launch of its own.  80,000 entries, 12 agents, three sources:
// 9.6 us per call in two launches, which is what the host takes to issue them, 7.2 in one.  (More agents: the search wants a CTA.)
struct ScoreSources {
    const uint16_t *list;
    uint32_t n, e_max;
};
template <bool SEARCH>
__global__ void __launch_bounds__(SCORE_SMALL_THREADS)
cs_score_small_kernel(SelArgs a, cs_workspace ws, float *__restrict__ out, ScoreSources src)
{
    Tables T;
    T.gtab = ws.gtab;
    T.g_sat = cs_recency(a.lambda, a.delta, a.age_sat);
    T.fsurv = const_cast<float *>(a.fsurv);
    cs_wait_for_predecessor();
    cs_release_successor();
    float f_mine = 0.0f;
    if (SEARCH) {
        const uint32_t v = threadIdx.x & 31u, row = v < a.A ? cs_ld_cg_pinned(ws.adjT + v) : 0u;
        uint32_t mine = 0;
        for (uint32_t i = v; i < src.n; i += 32u) {
            const uint32_t ag = src.list[i];
            if (ag < a.A) mine |= 1u << ag;
            else atomicOr(&ws.sc->status, CS_ST_BAD_SOURCE);
        }
        uint32_t front = __reduce_or_sync(0xFFFFFFFFu, mine), seen = front, hops = (front >> v) & 1u ? 0u : CS_HOP_NONE;
        for (uint32_t level = 1; front; ++level) {            // (every level adds an agent to `seen`, or is the last)
            const bool fresh = (row & front) != 0u && !((seen >> v) & 1u);
            front = __ballot_sync(0xFFFFFFFFu, fresh);
            seen |= front;
            if (fresh) hops = level;
        }
        f_mine = cs_survival_of(hops, src.e_max, a.delta);
    }
    const uint32_t lane = threadIdx.x & 31, gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_warps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t n_quads = (a.n + 3u) / 4u;                 // (the arrays' last quad may be short)
    resolve_now(a);
    for (uint32_t q0 = gw * 32u; q0 < n_quads; q0 += n_warps * 32u) {       // (whole warps: the factors come by shuffle)
        const bool any = q0 + lane < n_quads;
        const uint32_t q = any ? q0 + lane : n_quads - 1u, i0 = 4u * q;
        const bool whole = i0 + 4u <= a.n;
        uint32_t la[4], ag[4], tk[4];
        if (whole) {
            const uint4 l = __ldg((const uint4 *)a.la + q);
            const uint2 g = __ldg((const uint2 *)a.agent + q);
            const uint32_t t = a.ntok ? __ldg((const uint32_t *)a.ntok + q) : 0u;
            la[0] = l.x; la[1] = l.y; la[2] = l.z; la[3] = l.w;
            ag[0] = g.x & 0xFFFFu; ag[1] = g.x >> 16; ag[2] = g.y & 0xFFFFu; ag[3] = g.y >> 16;
#pragma unroll
            for (int r = 0; r < 4; ++r) tk[r] = a.ntok ? (t >> (8 * r)) & 0xFFu : a.block_tokens;
        } else {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint32_t i = i0 + r < a.n ? i0 + r : i0;
                la[r] = __ldg(a.la + i);
                ag[r] = __ldg(a.agent + i);
                tk[r] = a.ntok ? __ldg(a.ntok + i) : a.block_tokens;
            }
        }
        float f[4], g[4], s[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {                         // the eight look-ups travel together
            const uint32_t age = max(a.now, la[r]) - la[r];
            if (SEARCH) f[r] = __shfl_sync(0xFFFFFFFFu, f_mine, (int)(ag[r] & 31u));
            else f[r] = __ldcg(T.fsurv + (ag[r] < a.A ? ag[r] : 0u));
            g[r] = __ldg(T.gtab + (age < a.gtab_len ? age : 0u));
            if (age >= a.gtab_len) g[r] = age >= a.age_sat ? T.g_sat : cs_recency(a.lambda, a.delta, age);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            s[r] = __fmul_rn(__fmul_rn(f[r], g[r]), (float)tk[r]);
            if (ag[r] >= a.A) { s[r] = 0.0f; atomicOr(&ws.sc->status, CS_ST_BAD_AGENT); }
        }
        if (whole) {
            if (any) __stcs((float4 *)out + q, make_float4(s[0], s[1], s[2], s[3]));
        } else if (any) {
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (i0 + r < a.n) out[i0 + r] = s[r];
        }
    }
}

// ---------------------------------------------------------------------------------------------
// 0 fast pass (remembered key)
//
// The k-th smallest key moves little from one call to the next, so each kind of call (GPU victims, host
// victims, prefetch) remembers a key T somewhat above the one it ended with (cs_ahead()).  With T known, almost
// every eligible entry is dismissed by ONE compare of its last_access:
//   a  for a fixed agent and the common block size the key never decreases with last_access (victims: younger blocks score
//      higher, equal scores order by last_access; IEEE products are monotone, and g never increases with age) or never
//      increases (prefetch), so "key <= T" is a half-line of last_access.  Its end is found once per agent and CTA by
//      binary search over ages -- exactly, the part of a tie in score that lies below T's last_access included.  (A cut
//      by score alone let every entry tied with T through: 70,000 of 1,000,000 for k = 10,000, 990,000 of 9,400,000 for
//      k = 203, where a fifth of the ages are past the point at which the recency factor saturates.)
//   b  what is left (the candidates, and blocks of another size) is queued per warp as entry ids and worked off with all 32
//      lanes busy: the key is built and compared with T; candidates are appended to the buffer.
// Dismissed entries are only counted.  If at least k candidates were found, or nothing eligible lies above T, the
// candidates are complete and the index has been read ONCE.  Otherwise (the threshold rose above T, or nothing is
// remembered yet) the pass reports a miss and the full histogram and collect passes below run.  The result never depends
// on T.
// ---------------------------------------------------------------------------------------------
#define FQ_CAP 544u                 // per-warp queue: at most 31 left over + the 512 entries of one warp tile

// Largest value of every 16-bit half over eight packed words.
__device__ __forceinline__ uint32_t max_halves(const uint4 &a, const uint4 &b)
{
    const uint32_t m0 = __vmaxu2(__vmaxu2(a.x, a.y), __vmaxu2(a.z, a.w)), m1 = __vmaxu2(__vmaxu2(b.x, b.y), __vmaxu2(b.z, b.w));
    const uint32_t m = __vmaxu2(m0, m1);
    return max(m & 0xFFFFu, m >> 16);
}

// End of the half-line of last_access that an agent's blocks of the common size need for a key at or below T: victims
// la <= cut, prefetch la >= cut.  (Entries on the line's side of it that fail after all are sorted out by the exact test.)
template <bool PF>
__device__ __forceinline__ uint32_t la_cut(const SelArgs &a, const Tables &T, uint32_t agent, u64 bound)
{
    const uint32_t Tp = (uint32_t)(bound >> 32), Ts = (uint32_t)bound;
    const uint32_t flip = (PF && agent != T.a_star) ? 0x80000000u : 0u;
    const float f = T.fsurv[agent], tb = (float)a.block_tokens;
    // smallest possible primary key at an age (a copy on the other tier would make it that; the exact test tells).  The
    // table covers every age before saturation (gtab_len = age_sat) and ends with the saturated factor.
    auto primary = [&](uint32_t age) {
        const uint32_t bits = __float_as_uint(__fmul_rn(__fmul_rn(f, T.gtab[age]), tb));
        return PF ? (flip | (~bits & 0x7FFFFFFFu)) : (a.prefer_copy ? bits << 1 : bits);
    };
    // victims: primary falls with age: n_le = first age with primary <= Tp, n_lt = first with primary < Tp (age_sat + 1: none);
    // prefetch: it rises: n_le = first age with primary > Tp, n_lt = first with primary >= Tp.  Both found in step, without a
    // branch: the binary search over 2,263 ages is the longest chain between the scan's first load and its first compare.
    uint32_t n_le = 0, n_lt = 0;
    for (uint32_t step = CS_GTAB_MAX; step > 0; step >>= 1) {
        const uint32_t a0 = n_le + step - 1u, a1 = n_lt + step - 1u;
        const uint32_t p0 = primary(min(a0, a.age_sat)), p1 = primary(min(a1, a.age_sat));
        n_le += (a0 <= a.age_sat && (PF ? p0 <= Tp : p0 > Tp)) ? step : 0u;
        n_lt += (a1 <= a.age_sat && (PF ? p1 < Tp : p1 >= Tp)) ? step : 0u;
    }
    if (!PF) {
        if (n_le > a.age_sat) return 0u;                                   // no age qualifies
        // la <= now - n_lt for the ages below T's score; at T's score (n_le <= age < n_lt) also la <= Ts.  Age 0 stands for
        // every last_access from now on.
        const uint32_t by_score = n_lt > a.age_sat ? 0u : (n_lt == 0 ? 0xFFFFFFFFu : (a.now >= n_lt ? a.now - n_lt : 0u));
        const uint32_t at_score = min(n_le == 0 ? 0xFFFFFFFFu : (a.now >= n_le ? a.now - n_le : 0u), Ts);
        return max(by_score, at_score);
    } else {
        if (n_le == 0) return 0xFFFFFFFFu;                                 // not even age 0
        // la > now - n_lt for the ages above T's score; at T's score (n_lt <= age < n_le) also ~la <= Ts
        const uint32_t by_score = n_lt > a.age_sat ? 0u : (n_lt == 0 ? 0xFFFFFFFFu : (a.now >= n_lt ? a.now - n_lt + 1u : 0u));
        const uint32_t at_score = max(n_le > a.age_sat ? 0u : (a.now >= n_le ? a.now - n_le + 1u : 0u), ~Ts);
        return min(by_score, at_score);
    }
}

template <bool PF>
__global__ void __launch_bounds__(SEL_THREADS, 2) cs_sel_fast_kernel(SelArgs a, cs_workspace ws)
{
    extern __shared__ float smem[];                 // tables, per-warp queues, per-warp candidate staging, cuts
    __shared__ uint32_t s_above;
    __shared__ bool s_flag;
    constexpr int PS = PF ? 8 : 0;                  // phase-stamp slots of this kind of scan (profiling builds)
    (void)PS;
    CS_STAMP(ws, CS_PS_SCAN_ENTRY + PS, blockIdx.x == 0 && threadIdx.x == 0);
    // Before waiting for the predecessor grid: what depends only on the context's constants.
    Tables T;
    const size_t table_words = ((size_t)(a.A + a.gtab_len + 1) * 4 + (size_t)a.A * 2 + 15) / 16 * 4;
    uint32_t *queues = (uint32_t *)smem + table_words;
    uint32_t *s_cut = queues + (size_t)(SEL_THREADS / 32) * (FQ_CAP + STAGE_CAP * 3) + 4;     // after queues and staging
    load_tables_static(a, ws, smem, T);
    T.anchor += 2;                                  // (one entry more than the table: the saturated factor, for the cuts)
    if (threadIdx.x == 0) { s_above = 0; T.gtab[a.gtab_len] = T.g_sat; }
    CS_STAMP(ws, CS_PS_SCAN_SETUP + PS, blockIdx.x == 0 && threadIdx.x == 0);
    cs_wait_for_predecessor();
    CS_STAMP(ws, CS_PS_SCAN_WAITED + PS, blockIdx.x == 0 && threadIdx.x == 0);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const uint32_t n_tiles = a.n / TILE, n_warps = nth >> 5;
    // the first tile travels with the tables
    const u64 bound = cs_ld_cg_pinned(&ws.sc->sel_T[a.hint_slot]);      // ~0: nothing remembered
    const uint32_t monotone = cs_ld_cg_pinned(&ws.sc->gtab_monotone);
    const bool enabled = !PF || prefetch_enabled(ws, a.A);
    Group G;
    if ((gtid >> 5) < n_tiles) load_group<PF>(a, gtid >> 5, lane, G);
    resolve_now(a);
    // (Not earlier: the chain behind would fill the SMs while the refresh and the other lists' scans still come and go.
    // observe + select_step on 1,000,000 entries, replayed from a graph: 50.2 us with the release on entry, 42.5 here.)
    cs_release_successor();
    load_tables_dynamic(a, ws, T, PF && a.anchor);
    if (bound == ~0ull) {                                     // every CTA sees the same word
        if (blockIdx.x == 0 && threadIdx.x == 0) ws.sel->spec = 0;
        return;
    }
    __syncthreads();
    CS_STAMP(ws, CS_PS_SCAN_TABLES + PS / 2, blockIdx.x == 0 && threadIdx.x == 0);
    // the cuts rely on g never increasing with age (checked when the table was built) and on the table covering every
    // unsaturated age; otherwise nothing is dismissed and every eligible entry takes the exact test
    const bool usable = monotone && a.gtab_len == a.age_sat;
    for (uint32_t e = threadIdx.x; e < a.A; e += blockDim.x) {
        s_cut[PF ? 2u * e : e] = usable ? la_cut<PF>(a, T, e, bound) : (PF ? 0u : 0xFFFFFFFFu);
        if (PF && a.anchor) s_cut[2u * e + 1u] = T.anchor[e];         // (read together with the cut)
    }
    __syncthreads();
    CS_STAMP(ws, CS_PS_SCAN_CUTS + PS / 2, blockIdx.x == 0 && threadIdx.x == 0);
    const uint32_t Tb = a.block_tokens;
    uint32_t *q = queues + warp * FQ_CAP;
    uint32_t qn = 0;                                           // queued ids of this warp (same value in every lane)
    WarpStage st;
    {
        unsigned long long *stage_km = (unsigned long long *)(((uintptr_t)(queues + (SEL_THREADS / 32) * FQ_CAP) + 7) & ~(uintptr_t)7);
        stage_init(st, stage_km, (uint32_t *)(stage_km + (SEL_THREADS / 32) * STAGE_CAP));
    }
    uint32_t n_above = 0;

    // Works off whole rounds of 32 queued entries (all of them when `all`), every lane busy.
    auto drain = [&](bool all) {
        const uint32_t rounds = all ? (qn + 31u) / 32u : qn / 32u;
        for (uint32_t r = 0; r < rounds; ++r) {
            const uint32_t i = r * 32u + lane;
            bool cand = false;
            uint32_t id = 0, pr = 0, se = 0;
            if (i < qn) {
                id = q[i];
                const uint32_t ag = __ldg(a.agent + id), la = __ldg(a.la + id), fl = __ldg(a.flags + id);
                const uint32_t tok = a.ntok ? __ldg(a.ntok + id) : Tb, dp = (PF && a.anchor) ? __ldg(a.depth + id) : 0u;
                if (entry_key_rest<PF>(a, T, &ws.sc->status, ag, dp, fl, la, tok, pr, se)) {
                    cand = (((u64)pr << 32) | se) <= bound;
                    if (!cand) ++n_above;
                }
            }
            // candidates gather in the warp's slice of shared memory and leave it 32 or more at a time
            stage_push(st, cand, pr, se, id, &ws.sel->c_spec, ws.cand_km, ws.cand_id);
        }
        if (!all) {
            const uint32_t done = rounds * 32u, left = qn - done;        // < 32
            __syncwarp();
            const uint32_t v = lane < left ? q[done + lane] : 0u;
            __syncwarp();
            if (lane < left) q[lane] = v;
            __syncwarp();
            qn = left;
        } else {
            qn = 0;
        }
    };

    if (enabled) {
        const uint32_t n_iter = (n_tiles + n_warps - 1) / n_warps;     // whole warps stay in the shuffles
        for (uint32_t it = 0; it < n_iter; ++it) {
            const uint32_t t = it * n_warps + (gtid >> 5);
            uint32_t rem = 0;                                          // entries that need the exact test
            if (t < n_tiles) {
                if (it) load_group<PF>(a, t, lane, G);
                const uint32_t em = group_elig<PF>(a, G);
                uint32_t near = 0;                                     // on the cut's side of last_access, or of another size
                uint32_t el = em;                                      // eligible as far as can be told here
                if (max_halves(G.ag0, G.ag1) < a.A) {                  // (a bad agent id anywhere: everything takes the exact test)
                    if (!PF) {
#pragma unroll
                        for (int j = 0; j < GRP; ++j) near |= (grp_u32(G, j) <= s_cut[grp_u16(G.ag0, G.ag1, j)] ? 1u : 0u) << j;
                    } else if (!a.anchor) {
#pragma unroll
                        for (int j = 0; j < GRP; ++j) near |= (grp_u32(G, j) >= s_cut[2u * grp_u16(G.ag0, G.ag1, j)] ? 1u : 0u) << j;
                    } else {
                        // no branch per entry, the cut and the anchor in one read: 64,000,000 entries 169.6 us with
                        // branches, 135.5 so (140.8 and 112.8 without anchors)
                        uint32_t ahead = 0;
#pragma unroll
                        for (int j = 0; j < GRP; ++j) {
                            const uint2 ca = *(const uint2 *)&s_cut[2u * grp_u16(G.ag0, G.ag1, j)];
                            near |= (grp_u32(G, j) >= ca.x ? 1u : 0u) << j;
                            ahead |= (grp_u16(G.dp0, G.dp1, j) < ca.y ? 1u : 0u) << j;
                        }
                        el &= ahead;
                    }
                    if (a.ntok) {
#pragma unroll
                        for (int w = 0; w < 4; ++w)
                            near |= (~nibble_of_flags(zero_bytes(u4_word(G.tk, w) ^ (0x01010101u * Tb))) & 0xFu) << (4 * w);
                    }
                } else {
                    near = 0xFFFFu;
                }
                n_above += __popc(el & ~near);
                rem = el & near;
            }
            // queue the remaining entries of the warp (ids only), then work off whole rounds
            if (!__any_sync(0xFFFFFFFFu, rem != 0u)) continue;
            const uint32_t cnt = __popc(rem);
            uint32_t incl = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if (lane >= d) incl += v;
            }
            const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
            uint32_t pos = qn + incl - cnt;
            while (rem) {
                const int j = __ffs(rem) - 1;
                rem &= rem - 1;
                q[pos++] = grp_id(t, lane, j);
            }
            qn += total;
            __syncwarp();
            if (qn >= 32u) drain(false);
        }
        CS_STAMP(ws, CS_PS_SCAN_WALKED + PS / 2, blockIdx.x == 0 && threadIdx.x == 0);
        drain(true);
        stage_flush(st, &ws.sel->c_spec, ws.cand_km, ws.cand_id);
        CS_STAMP(ws, CS_PS_SCAN_READ + PS, blockIdx.x == 0 && threadIdx.x == 0);
        const uint32_t t0 = n_tiles * TILE;
        if (gtid < a.n - t0) {                                // ragged tail, one entry per thread
            const uint32_t i = t0 + gtid;
            uint32_t pr, se;
            const uint32_t tok = a.ntok ? a.ntok[i] : Tb;
            if (entry_key<PF>(a, T, &ws.sc->status, a.agent[i], a.depth[i], a.ref[i], a.flags[i], a.la[i], tok, pr, se)) {
                if ((((u64)pr << 32) | se) <= bound) {
                    const uint32_t pos = atomicAdd(&ws.sel->c_spec, 1u);
                    ws.cand_km[pos] = ((unsigned long long)pr << 32) | se;
                    ws.cand_id[pos] = i;
                } else {
                    ++n_above;
                }
            }
        }
    }
    n_above = __reduce_add_sync(0xFFFFFFFFu, n_above);
    if (lane == 0 && n_above) atomicAdd(&s_above, n_above);
    __syncthreads();
    if (threadIdx.x == 0 && s_above) atomicAdd(&ws.sel->n_above, s_above);
    CS_STAMP(ws, CS_PS_SCAN_FLUSHED + PS, blockIdx.x == 0 && threadIdx.x == 0);
    if (!last_cta_done(&ws.sel->ticket[0], &s_flag)) return;
    CS_STAMP(ws, CS_PS_SCAN_LAST_CTA + PS, threadIdx.x == 0);
    if (threadIdx.x == 0) {
        const uint32_t c = __ldcg(&ws.sel->c_spec), above = __ldcg(&ws.sel->n_above), total = c + above;
        // complete when the k winners lie at or below T, when fewer than k entries are eligible and all of them do, or when k = 0
        const bool hit = a.k == 0 || c >= a.k || above == 0;
        ws.sel->spec = hit ? 1u : 0u;
        if (hit) {
            const uint32_t n_out = total < a.k ? total : a.k;
            ws.sel->c = c;
            ws.sel->n_out = n_out;
            ws.sel->n_elig = total;
            ws.sel->bound = bound;
            count_select(ws, a.kind, total, n_out);
            count_candidates(ws, a.kind, a.k ? c : 0u, true);
        }
        ws.sel->c_spec = 0;
        ws.sel->n_above = 0;
        ws.sel->ticket[0] = 0;
    }
    CS_STAMP(ws, CS_PS_SCAN_TAIL_DONE + PS, threadIdx.x == 0);
}

// ---------------------------------------------------------------------------------------------
// 1 histogram (runs when the fast pass missed or had nothing to go by)
//
// Full keys of all eligible entries into a 4096-bin histogram; the last CTA finds the threshold bin.
// ---------------------------------------------------------------------------------------------
template <bool PF>
__global__ void __launch_bounds__(SEL_THREADS) cs_sel_hist_kernel(SelArgs a, cs_workspace ws)
{
    extern __shared__ float smem[];
    __shared__ __align__(16) uint32_t s_hist[CS_HIST_BINS];
    __shared__ uint32_t s_part[SEL_THREADS];
    __shared__ uint32_t s_b0;
    __shared__ bool s_flag;
    cs_wait_for_predecessor();
    cs_release_successor();
    if (ws.sel->spec) return;          // the fast pass already has the candidates
    resolve_now(a);
    Tables T;
    load_tables(a, ws, smem, T, PF && a.anchor);
    for (uint32_t i = threadIdx.x; i < CS_HIST_BINS; i += blockDim.x) s_hist[i] = 0;
    __syncthreads();
    if (!PF || prefetch_enabled(ws, a.A)) {
        uint32_t run_bin = 0xFFFFFFFFu, run_cnt = 0;                    // adjacent entries often share a bin
        for_each_eligible<PF>(a, T, &ws.sc->status, [&](uint32_t, uint32_t pr, uint32_t) {
            const uint32_t bin = bin_of<PF>(a, pr);
            if (bin == run_bin) { ++run_cnt; return; }
            if (run_cnt) atomicAdd(&s_hist[run_bin], run_cnt);
            run_bin = bin;
            run_cnt = 1;
        });
        if (run_cnt) atomicAdd(&s_hist[run_bin], run_cnt);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < CS_HIST_BINS; i += blockDim.x) {
        const uint32_t v = s_hist[i];
        if (v) atomicAdd(&ws.hist[i], v);
    }
    if (!last_cta_done(&ws.sel->ticket[1], &s_flag)) return;

    // ---- last CTA: threshold bin = first bin whose inclusive running count reaches k ------------
    constexpr uint32_t PER = CS_HIST_BINS / SEL_THREADS;
    uint32_t loc[PER], sum = 0;
#pragma unroll
    for (uint32_t q = 0; q < PER; ++q) {
        loc[q] = __ldcg(&ws.hist[threadIdx.x * PER + q]);
        ws.hist[threadIdx.x * PER + q] = 0;                 // ready for the next call
        sum += loc[q];
    }
    s_part[threadIdx.x] = sum;
    if (threadIdx.x == 0) s_b0 = (a.k == 0) ? 0xFFFFFFFFu : CS_HIST_BINS - 1;   // k = 0: nothing; k > eligible: everything
    __syncthreads();
    for (uint32_t d = 1; d < SEL_THREADS; d <<= 1) {         // inclusive scan
        const uint32_t v = threadIdx.x >= d ? s_part[threadIdx.x - d] : 0;
        __syncthreads();
        s_part[threadIdx.x] += v;
        __syncthreads();
    }
    const uint32_t total = s_part[SEL_THREADS - 1];
    const uint32_t before = s_part[threadIdx.x] - sum;
    if (a.k && total >= a.k && before < a.k && a.k <= before + sum) {
        uint32_t run = before;
#pragma unroll
        for (uint32_t q = 0; q < PER; ++q) {
            run += loc[q];
            if (run >= a.k) { s_b0 = threadIdx.x * PER + q; break; }
        }
    }
    __syncthreads();
    const uint32_t b0 = s_b0;
    if (threadIdx.x == 0) {
        ws.sel->b0 = b0;
        ws.sel->n_elig = total;
        ws.sel->n_out = total < a.k ? total : a.k;
        ws.sel->bound = b0 == 0xFFFFFFFFu ? 0ull : (primary_limit<PF>(a, b0) << 32) - 1ull;
        count_select(ws, a.kind, total, total < a.k ? total : a.k);
        ws.sel->c = 0;
        ws.sel->ticket[1] = 0;
    }
}

// ---------------------------------------------------------------------------------------------
// 2 collect
// ---------------------------------------------------------------------------------------------
// Age limits.  For a fixed agent and block size the score never increases with age (the recency
// table is checked to be monotone, IEEE multiplication is), so "first digit <= b0" is an interval
// of ages: victims  age >= lim (low scores are old blocks), prefetch  age + 1 <= lim (high scores
// are young blocks).  One limit per (agent, size) found by binary search lets the scan of a large
// index decide with one table look-up per entry; the full key is computed for candidates only.
#define AGE_LIM_MAX 8192u
#define AGE_CLAMP 0xFFFFFFFEu

template <bool PF>
__device__ __forceinline__ uint32_t age_limit_of(const SelArgs &a, const Tables &T, uint32_t agent, uint32_t tok,
                                                 uint32_t b0)
{
    const uint32_t n_age = a.age_sat;                        // ages >= age_sat all score like age_sat
    const u64 limit = primary_limit<PF>(a, b0);              // candidate <=> primary key < limit
    const uint32_t flip = (PF && agent != T.a_star) ? 0x80000000u : 0u;
    uint32_t lo = 0, hi = n_age + 1;                          // victims: first age that qualifies; prefetch: first that does not
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        const uint32_t bits = __float_as_uint(score_from_age(a, T, agent, mid, tok));
        const uint32_t pr = PF ? (flip | (~bits & 0x7FFFFFFFu)) : (a.prefer_copy ? bits << 1 : bits);
        if ((pr < limit) != PF) hi = mid;
        else lo = mid + 1;
    }
    return lo > n_age ? 0xFFFFFFFFu : lo;                     // victims: 0xFFFFFFFF: no age qualifies (ages are clamped below it);
                                                              // prefetch: candidate <=> age + 1 <= lo  (0: none, 0xFFFFFFFF: all)
}

template <bool PF>
__global__ void __launch_bounds__(SEL_THREADS) cs_sel_collect_kernel(SelArgs a, cs_workspace ws)
{
    extern __shared__ float smem[];
    __shared__ bool s_flag;
    cs_wait_for_predecessor();
    cs_release_successor();
    if (ws.sel->spec) return;          // the fast pass already collected the candidates
    resolve_now(a);
    Tables T;
    load_tables(a, ws, smem, T, PF && a.anchor);
    __syncthreads();
    const uint32_t b0 = ws.sel->b0;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t n_cls = a.ntok ? a.block_tokens : 1u;     // size classes: tok = 1 .. block_tokens (or the constant)
    const bool limits = a.use_age_limits && ws.sc->gtab_monotone && b0 != 0xFFFFFFFFu;
    uint32_t *s_lim = (uint32_t *)(smem + a.A + a.gtab_len) + (a.A + 1) / 2;      // after the tables (and the anchor table)
    if (limits) {
        for (uint32_t e = threadIdx.x; e < a.A * n_cls; e += blockDim.x) {
            const uint32_t agent = e / n_cls, tok = a.ntok ? (e - agent * n_cls) + 1u : a.block_tokens;
            s_lim[e] = age_limit_of<PF>(a, T, agent, tok, b0);
        }
        __syncthreads();
    }
    if (b0 != 0xFFFFFFFFu && (!PF || prefetch_enabled(ws, a.A))) {
        // Whole groups: count this thread's candidates, reserve a range with one atomic per warp,
        // then write.  The loop bound is rounded up so that whole warps stay in the shuffles.
        const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
        const uint32_t n_tiles = a.n / TILE, n_warps = nth >> 5;
        const uint32_t n_iter = (n_tiles + n_warps - 1) / n_warps;
        for (uint32_t it = 0; it < n_iter; ++it) {
            const uint32_t t = it * n_warps + (gtid >> 5);
            uint32_t mask = 0;               // keys are recomputed for the (few) candidates instead of kept in registers
            Group G;
            if (t < n_tiles) {
                load_group<PF>(a, t, lane, G);
                const uint32_t em = group_elig<PF>(a, G);
#pragma unroll
                for (int j = 0; j < GRP; ++j) {
                    if (!((em >> j) & 1u)) continue;
                    uint32_t se;
                    const uint32_t tok = a.ntok ? grp_u8(G.tk, j) : a.block_tokens;
                    const uint32_t dp = (PF && a.anchor) ? grp_u16(G.dp0, G.dp1, j) : 0u;
                    const uint32_t ag = grp_u16(G.ag0, G.ag1, j);
                    if (limits && ag < a.A && tok - 1u < n_cls) {
                        // prefilter: one look-up; exact, so the key is only needed when the entry is written
                        const uint32_t la = grp_u32(G, j);
                        uint32_t age = la <= a.now ? a.now - la : 0u;
                        age = age < AGE_CLAMP ? age : AGE_CLAMP;
                        const uint32_t lim = s_lim[ag * n_cls + (a.ntok ? tok - 1u : 0u)];
                        const bool in = PF ? (age + 1u <= lim) : (age >= lim);
                        if (in && !(PF && a.anchor && !(dp < T.anchor[ag]))) mask |= 1u << j;
                        continue;
                    }
                    uint32_t prj;
                    if (entry_key_rest<PF>(a, T, &ws.sc->status, ag, dp, grp_u8(G.fl, j), grp_u32(G, j), tok, prj, se) &&
                        bin_of<PF>(a, prj) <= b0)
                        mask |= 1u << j;
                }
            }
            if (!__any_sync(0xFFFFFFFFu, mask != 0)) continue;      // most warps hold no candidate at all
            const uint32_t cnt = __popc(mask);
            uint32_t incl = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if (lane >= d) incl += v;
            }
            uint32_t base = 0;
            if (lane == 31 && incl) base = atomicAdd(&ws.sel->c, incl);
            base = __shfl_sync(0xFFFFFFFFu, base, 31);
            uint32_t pos = base + incl - cnt;
#pragma unroll
            for (int j = 0; j < GRP; ++j) {
                if (mask & (1u << j)) {
                    uint32_t prj, se;
                    const uint32_t tok = a.ntok ? grp_u8(G.tk, j) : a.block_tokens;
                    const uint32_t dp = (PF && a.anchor) ? grp_u16(G.dp0, G.dp1, j) : 0u;
                    const bool ok = entry_key_rest<PF>(a, T, &ws.sc->status, grp_u16(G.ag0, G.ag1, j), dp, grp_u8(G.fl, j),
                                                       grp_u32(G, j), tok, prj, se) && bin_of<PF>(a, prj) <= b0;
                    // (a slot was reserved from the prefilter's verdict; should the exact key ever disagree,
                    //  the slot gets a key that sorts behind every real candidate and is never emitted)
                    ws.cand_km[pos] = ok ? (((unsigned long long)prj << 32) | se) : ~0ull;
                    ws.cand_id[pos] = ok ? grp_id(t, lane, j) : CS_ID_NONE;
                    ++pos;
                }
            }
        }
        const uint32_t t0 = n_tiles * TILE;
        if (gtid < a.n - t0) {
            const uint32_t i = t0 + gtid;
            uint32_t p, se;
            const uint32_t tok = a.ntok ? a.ntok[i] : a.block_tokens;
            if (entry_key<PF>(a, T, &ws.sc->status, a.agent[i], a.depth[i], a.ref[i], a.flags[i], a.la[i], tok, p, se) &&
                bin_of<PF>(a, p) <= b0) {
                const uint32_t pos = atomicAdd(&ws.sel->c, 1u);
                ws.cand_km[pos] = ((unsigned long long)p << 32) | se;
                ws.cand_id[pos] = i;
            }
        }
    }
    if (!last_cta_done(&ws.sel->ticket[2], &s_flag)) return;

    if (threadIdx.x == 0) { ws.sel->ticket[2] = 0; count_candidates(ws, a.kind, __ldcg(&ws.sel->c), false); }
}

// ---------------------------------------------------------------------------------------------
// 3 - 5 ordering the candidates (cs_select_buckets.cuh), a launch per step
// ---------------------------------------------------------------------------------------------
#define SAMPLE_CTAS 64u
// The key the next call of this kind gets, from whoever places the list's last id.
__device__ __forceinline__ void remember_key(const cs_workspace &ws, const cs_sel_state &st, uint32_t k, uint32_t hint_slot, uint32_t pos, u64 km)
{
    if (pos == st.n_out - 1u && hint_slot < 3u) ws.sc->sel_T[hint_slot] = next_bound(st, k, km, cs_ahead(k));
}

__global__ void __launch_bounds__(512) cs_sel_sample_kernel(SelArgs a, cs_workspace ws, uint32_t *__restrict__ ids_out,
                                                            uint32_t *__restrict__ n_out_dev)
{
    __shared__ u64 s_km[FEW_MAX];
    __shared__ uint32_t s_id[FEW_MAX];
    const uint32_t tid = threadIdx.x;
    cs_wait_for_predecessor();
    CS_STAMP(ws, CS_PS_SAMPLE_WAITED + (a.kind == 2 ? 8 : 0), blockIdx.x == 0 && tid == 0);
    cs_release_successor();
    const uint4 st = cs_ld_cg_pinned((const uint4 *)&ws.sel->c);      // c, n_out, n_elig, b0
    const uint32_t c = st.x, n_out = st.y;
    for (uint32_t i = n_out + blockIdx.x * blockDim.x + tid; i < a.k; i += gridDim.x * blockDim.x) ids_out[i] = CS_ID_NONE;
    if (blockIdx.x == 0) {
        CS_BCOUNT(ws, tid) = 0;
        if (tid == 0) *n_out_dev = n_out;
    }
    if (n_out == 0) return;
    rank_sample(ws, c, n_out, cs_ahead(a.k), &ws.sel->ahead, s_km, s_id, blockIdx.x, gridDim.x, ids_out, [&](uint32_t pos, u64 km, uint32_t) {
        if (pos != n_out - 1u) return;
        cs_sel_state now = *ws.sel;
        now.ahead = ~0ull;                                    // (another CTA may not have stored it yet)
        remember_key(ws, now, a.k, a.hint_slot, pos, km);
    });
    CS_STAMP(ws, CS_PS_SAMPLE_DONE + (a.kind == 2 ? 8 : 0), blockIdx.x == 0 && tid == 0);
}

__global__ void __launch_bounds__(256) cs_sel_place_kernel(cs_workspace ws, uint32_t max_blocks, uint32_t region_max, uint32_t kind)
{
    __shared__ u64 s_km[CS_SAMPLE], b_km[CS_BUCKETS];         // the sample, and where the buckets start
    __shared__ uint32_t s_id[CS_SAMPLE], b_id[CS_BUCKETS];
    cs_wait_for_predecessor();
    CS_STAMP(ws, CS_PS_PLACE_WAITED + (kind == 2 ? 8 : 0), blockIdx.x == 0 && threadIdx.x == 0);
    (void)kind;
    const uint4 st = cs_ld_cg_pinned((const uint4 *)&ws.sel->c);          // c, n_out, n_elig, b0
    // (the ranking CTAs, four per SM, not before these keys are here)
    place_candidates(ws, st, max_blocks, region_max, s_km, s_id, b_km, b_id, blockIdx.x, gridDim.x, [] { cs_release_successor(); });
    CS_STAMP(ws, CS_PS_PLACE_DONE + (kind == 2 ? 8 : 0), blockIdx.x == 0 && threadIdx.x == 0);
}

__global__ void __launch_bounds__(FINISH_THREADS, 3)
cs_sel_finish_kernel(cs_workspace ws, uint32_t k, uint32_t max_blocks, uint32_t region_max, uint32_t kind, uint32_t hint_slot,
                     uint32_t *__restrict__ ids_out)
{
    __shared__ u64 t_km[RANK_TILE];
    __shared__ uint32_t t_id[RANK_TILE];
    __shared__ uint32_t s_off, s_max, s_n;
    const uint32_t tid = threadIdx.x, b = blockIdx.x;
    if (tid == 0) { s_off = 0; s_max = 0; s_n = 0; }
    __syncthreads();
    cs_wait_for_predecessor();
    CS_STAMP(ws, CS_PS_FINISH_WAITED + (kind == 2 ? 8 : 0), b == 0 && tid == 0);
    cs_release_successor();
    const uint4 st = cs_ld_cg_pinned((const uint4 *)&ws.sel->c);          // c, n_out, n_elig, b0
    const uint32_t n_t = cs_ld_cg_pinned(&CS_BCOUNT(ws, tid)), m = cs_ld_cg_pinned(&CS_BCOUNT(ws, b)), c = st.x, n_out = st.y;
    if (n_out == 0 || c <= FEW_MAX) return;
    const OrderPlan P = order_plan(c, n_out, max_blocks, region_max);
    if (b >= P.nb) return;
    finish_bucket(ws, c, n_out, P, b, n_t, m, kind, t_km, t_id, &s_off, &s_max, &s_n, ids_out,
                  [&](uint32_t pos, u64 km, uint32_t) { if (pos == n_out - 1u) remember_key(ws, *ws.sel, k, hint_slot, pos, km); });
    CS_STAMP(ws, CS_PS_FINISH_DONE + (kind == 2 ? 8 : 0), b == 0 && tid == 0);
}

// ---------------------------------------------------------------------------------------------
void cs_fill_sel_args(const cs_ctx *ctx, const cs_block_index *idx, uint32_t now, const float *fsurv, SelArgs &a)
{
    a.agent = idx->agent;
    a.depth = idx->depth;
    a.ref = idx->ref_count;
    a.flags = idx->flags;
    a.la = idx->last_access;
    a.ntok = idx->n_tokens;
    a.anchor = idx->anchor_blocks;
    a.fsurv = fsurv;
    a.n = idx->n_blocks;
    a.now = now;
    a.A = ctx->p.n_agents;
    a.block_tokens = ctx->p.block_tokens;
    a.gtab_len = ctx->gtab_len;
    a.age_sat = ctx->age_sat;
    a.lambda = ctx->p.lambda;
    a.delta = ctx->p.delta;
    a.tier = 0;
    a.k = 0;
    a.prefer_copy = ctx->p.prefer_other_copy ? 1u : 0u;
    a.use_age_limits = 0;
    a.hint_slot = 0;
    a.kind = 0;
    a.now_dev = ctx->step_now_dev ? ctx->step_now_dev : ctx->clock_dev;
    a.region_cap_max = ctx->region_cap_max;
    a.max_blocks = ctx->p.max_blocks;
    a.bin_lo = 0;
    a.bin_shift = 20;
}

// The scores of Eq. 9 lie between delta^2 (one token) and (1 + delta)^2 |b|: the bins of the cluster select divide that range.
// A survival table of the caller's own, or a block with more tokens, may leave it; the bins clamp.
void cs_fill_sel_bins(const cs_ctx *ctx, SelArgs &a, int prefetch)
{
    const float d = ctx->p.delta, lo_f = 0.99f * d * d, hi_f = 1.01f * (1.0f + d) * (1.0f + d) * (float)ctx->p.block_tokens;
    uint32_t lo, hi;
    memcpy(&lo, &lo_f, 4);
    memcpy(&hi, &hi_f, 4);
    if (!(lo_f > 0.0f) || lo >= 0x7F800000u) lo = 0;                // delta^2 underflows
    if (hi > 0x7F800000u || hi <= lo) hi = 0x7F800000u;
    if (prefetch) {                                                 // primary = ~bits without the sign: high scores first
        const uint32_t t = 0x7FFFFFFFu - hi;
        hi = 0x7FFFFFFFu - lo;
        lo = t;
    } else if (a.prefer_copy) {                                     // one bit more below the score
        lo <<= 1;
        hi = (hi << 1) | 1u;
    }
    const uint32_t bins = (prefetch ? CS_HIST_BINS / 2 : CS_HIST_BINS) - 1u;
    uint32_t shift = 0;
    while (((hi - lo) >> shift) >= bins) ++shift;
    a.bin_lo = lo;
    a.bin_shift = shift;
}

uint32_t cs_scan_grid(const cs_ctx *ctx, uint32_t n, uint32_t per_cta, uint32_t ctas_per_sm)
{
    uint32_t g = (n + per_cta - 1) / per_cta;
    const uint32_t cap = ctas_per_sm * (uint32_t)ctx->sm_count;
    if (g > cap) g = cap;
    return g ? g : 1u;
}

size_t cs_table_smem(const cs_ctx *ctx)
{
    return (size_t)(ctx->p.n_agents + ctx->gtab_len) * sizeof(float) + (size_t)ctx->p.n_agents * sizeof(uint16_t) + 16;
}

bool cs_score_searches(const cs_ctx *ctx, uint32_t n_blocks) { return ctx->p.n_agents <= 32u && n_blocks && n_blocks <= SCORE_SMALL_MAX; }

int cs_launch_score(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, const float *fsurv, const uint16_t *sources, uint32_t n_sources,
                    float *scores_out, cudaStream_t s)
{
    const uint32_t grid_small = cs_scan_grid(ctx, idx->n_blocks, SCORE_SMALL_THREADS * 4u, 8u);
    const ScoreSources src = {sources, n_sources, ctx->p.e_max};
    SelArgs a;
    cs_fill_sel_args(ctx, idx, now, fsurv, a);
    a.anchor = nullptr;
    if (sources)
        cs_launch_chained(cs_score_small_kernel<true>, grid_small, SCORE_SMALL_THREADS, 0, s, a, ctx->ws, scores_out, src);
    else if (idx->n_blocks <= SCORE_SMALL_MAX)
        cs_launch_chained(cs_score_small_kernel<false>, grid_small, SCORE_SMALL_THREADS, 0, s, a, ctx->ws, scores_out, src);
    else
        cs_launch_chained(cs_score_kernel, cs_scan_grid(ctx, idx->n_blocks, SEL_THREADS * GRP), SEL_THREADS, cs_table_smem(ctx), s, a,
                          ctx->ws, scores_out);
    return cs_check_launch(ctx);
}

// Shared-memory opt-in of the scan kernels that keep age limits in shared memory: an attribute of the
// function on a device, set once per process and device to one fixed size.
#include <mutex>
#define SCAN_SMEM_OPT_IN (96 * 1024)
static std::mutex g_scan_mu;
static bool g_scan_opted[64];
static int scan_opt_in(cs_ctx *ctx)
{
    if (ctx->device < 0 || ctx->device >= 64) return CS_EINVAL;
    std::lock_guard<std::mutex> lock(g_scan_mu);
    if (g_scan_opted[ctx->device]) return CS_OK;
    cudaError_t e = cudaFuncSetAttribute(cs_sel_collect_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCAN_SMEM_OPT_IN);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(cs_sel_collect_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCAN_SMEM_OPT_IN);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(cs_sel_fast_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCAN_SMEM_OPT_IN);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(cs_sel_fast_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCAN_SMEM_OPT_IN);
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
    g_scan_opted[ctx->device] = true;
    return CS_OK;
}

// One select through the grid-wide kernels, on the scratch of one job: the arguments, and its six launches one by one, so
// that the launches of several selects can be issued in turn or become the nodes of a graph.
#define SELECT_STAGES CS_SELECT_STAGES
struct SelectChain {
    SelArgs a;
    const cs_workspace *ws;
    uint32_t prefetch, *ids_out, *n_out;
    cudaStream_t s;
};

// Where a stage goes: launched on the chain's stream, or the node of (job, stage) in a graph of selects side by side --
// added behind the node of the stage before it, or given new arguments.
struct StageSink {
    cs_select_graph *g;            // NULL: launched
    int job, stage;
    template <class... KArgs, class... Args>
    cudaError_t put(cudaStream_t s, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args) const
    {
        if (!g) {
            cs_launch_chained(kernel, grid, block, smem, s, args...);
            return cudaGetLastError();
        }
        std::tuple<KArgs...> held((KArgs)args...);
        return std::apply([&](auto &...arg) { return put_node((void *)kernel, grid, block, smem, {(void *)&arg...}); }, held);
    }
    cudaError_t put_node(void *kernel, dim3 grid, dim3 block, size_t smem, std::initializer_list<void *> args) const
    {
        void *params[16];
        std::copy(args.begin(), args.end(), params);
        cudaGraphNodeParams np = {};
        np.type = cudaGraphNodeTypeKernel;
        np.kernel.func = kernel;
        np.kernel.gridDim = grid;
        np.kernel.blockDim = block;
        np.kernel.sharedMemBytes = (unsigned)smem;
        np.kernel.kernelParams = params;
        if (g->exec) return cudaGraphExecNodeSetParams(g->exec, g->node[job][stage], &np);
        cudaGraphEdgeData edge = {};
        edge.type = cudaGraphDependencyTypeProgrammatic;
        edge.from_port = cudaGraphKernelNodePortProgrammatic;
        return cudaGraphAddNode_v2(&g->node[job][stage], g->graph, stage ? &g->node[job][stage - 1] : nullptr, stage ? &edge : nullptr,
                                   stage ? 1 : 0, &np);
    }
};

static void prepare_chain(const cs_ctx *ctx, int job, const cs_block_index *idx, uint32_t now, int prefetch, uint32_t tier, uint32_t k,
                          uint32_t *ids_out, uint32_t *n_out, cudaStream_t s, SelectChain &c)
{
    c.ws = job == 0 ? &ctx->ws : &ctx->ws_job[job - 1];
    c.prefetch = prefetch ? 1u : 0u;
    c.ids_out = ids_out;
    c.n_out = n_out;
    c.s = s;
    cs_fill_sel_args(ctx, idx, now, ctx->fsurv_override ? ctx->fsurv_override : ctx->ws.fsurv, c.a);
    c.a.tier = tier;
    c.a.k = k;
    c.a.hint_slot = ctx->no_speculation ? 3u : (prefetch ? 2u : tier);
    c.a.kind = prefetch ? 2u : tier;
    cs_fill_sel_bins(ctx, c.a, prefetch);
}

static int launch_stage(cs_ctx *ctx, SelectChain &c, int stage, cs_select_graph *graph = nullptr, int job = 0)
{
    const uint32_t grid = cs_scan_grid(ctx, c.a.n, SEL_THREADS * GRP), grid_c = cs_scan_grid(ctx, c.a.n, 1024), A = ctx->p.n_agents;
    const size_t sm = cs_table_smem(ctx);
    const cs_workspace &ws = *c.ws;
    const StageSink to = {graph, job, stage};
    cudaError_t e = cudaSuccess;
    if (stage == 0) {
        // tables, per-warp queues, per-warp candidate staging, cuts
        const size_t sm_fast = (sm + 4 + 15) / 16 * 16 + (size_t)(SEL_THREADS / 32) * (FQ_CAP * sizeof(uint32_t) + STAGE_CAP * 12) + 32 +
                               (size_t)A * (c.prefetch ? 2u : 1u) * sizeof(uint32_t);
        if (c.prefetch) e = to.put(c.s, cs_sel_fast_kernel<true>, grid, SEL_THREADS, sm_fast, c.a, ws);
        else e = to.put(c.s, cs_sel_fast_kernel<false>, grid, SEL_THREADS, sm_fast, c.a, ws);
    } else if (stage == 1) {
        if (c.prefetch) e = to.put(c.s, cs_sel_hist_kernel<true>, grid, SEL_THREADS, sm, c.a, ws);
        else e = to.put(c.s, cs_sel_hist_kernel<false>, grid, SEL_THREADS, sm, c.a, ws);
    } else if (stage == 2) {
        // large indexes: the collect pass prefilters by age limits (one look-up per entry instead of the full key)
        const uint32_t n_cls = c.a.ntok ? ctx->p.block_tokens : 1u;
        size_t sm_collect = sm;
        if (c.a.n >= CS_AGE_LIMIT_MIN_BLOCKS && (size_t)A * n_cls <= AGE_LIM_MAX) {
            c.a.use_age_limits = 1;
            sm_collect += (size_t)A * n_cls * sizeof(uint32_t);
        }
        if (c.prefetch) e = to.put(c.s, cs_sel_collect_kernel<true>, grid, SEL_THREADS, sm_collect, c.a, ws);
        else e = to.put(c.s, cs_sel_collect_kernel<false>, grid, SEL_THREADS, sm_collect, c.a, ws);
    } else if (stage == 3) {
        e = to.put(c.s, cs_sel_sample_kernel, SAMPLE_CTAS, 512, 0, c.a, ws, c.ids_out, c.n_out);
    } else if (stage == 4) {
        e = to.put(c.s, cs_sel_place_kernel, grid_c, 256, 0, ws, c.a.max_blocks, c.a.region_cap_max, c.a.kind);
    } else {
        e = to.put(c.s, cs_sel_finish_kernel, CS_BUCKETS, FINISH_THREADS, 0, ws, c.a.k, c.a.max_blocks, c.a.region_cap_max, c.a.kind,
                          c.a.hint_slot, c.ids_out);
    }
    ctx->n_launches++;
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
    return CS_OK;
}

// The route of selects over n entries, the longest list k: a cluster per list, one launch on the whole GPU for all of them, or a launch chain
// per list.  Both sides of the lines, mean us per call replayed from a graph, an index that does not change but for the clock (static) / one whose victims
// are used again and whose prefetched entries are gone for eight calls (moving); v: one list of k, vhp: three.
//   cluster / whole GPU   80,000, k = 256, vhp 19.0 / 18.2 (and the refresh) and 27.6 / 37.0, 140,000 30.7 / 18.5 and 31.0 / 29.7; 80,000, k = 4,000, vhp 39.1 / 22.4 and 39.8 / 42.7,
//                         131,072, k = 4,000 43.3 / 20.6 and 42.5 / 35.2, 262,144, k = 16,000 73.5 / 25.8 and 76.2 / 51.0
//   chain / whole GPU     300,000, k = 256, vhp 33.2 / 21.4 and 40.2 / 30.2; 1,000,000, k = 10,000, v 33.3 / 22 and 34.3 / 35.9; 4,000,000, k = 20,000, vhp 66.5 / 34.3
//                         and 108 / 87; 16,000,000, k = 10,000, v 55.9 / 45 and 70 / 75.5; 32,000,000 73.7 / 70.4, 64,000,000 114.3 / 119.5 (static).
//                         Long lists, v: 1,000,000, k = 30,000 moving 46.1 / 50.3, k = 100,000 70.0 / 47.1 and 78 / 106; 300,000, k = 75,000 67.6 / 60.6 and 71.7 / 91
// Where victims leave by the thousand, entries of one call are tied but for their ids and swell single buckets, and the list goes on to the ranked
// sample; the lines lie where the two kinds of index together are no longer faster.
// A list's first call finds nothing remembered and has four passes more: it takes the route that the list would have without this one
// (1,000,000 entries, two lists: 114 us, 123 in one launch).
enum { ROUTE_CLUSTER, ROUTE_GRID, ROUTE_CHAIN };
static int select_route(cs_ctx *ctx, uint32_t n, uint32_t k, uint32_t lists, cudaStream_t s)
{
    if (ctx->select_path == CS_SELECT_MULTI) return ROUTE_CHAIN;
    const bool fits = n <= CS_SELECT_CLUSTER_MAX_BLOCKS, asked = (ctx->lists_asked & lists) == lists;
    if (ctx->select_path == CS_SELECT_CLUSTER) return fits ? ROUTE_CLUSTER : ROUTE_CHAIN;
    const bool grid = fits ? n > CS_SELECT_GRID_MIN_BLOCKS || (n > CS_SELECT_GRID_LONG_BLOCKS && k >= CS_SELECT_GRID_LONG_LIST)
                           : n <= CS_SELECT_GRID_MAX_BLOCKS && k <= CS_SELECT_GRID_MAX_LIST;
    if (grid) ctx->lists_asked |= lists;
    if (grid && !asked) {
        // (what is captured runs again: its later runs are not first calls)
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) (void)cudaGetLastError();
        if (capture == cudaStreamCaptureStatusActive) return ROUTE_GRID;
    }
    if (grid && asked) return ROUTE_GRID;
    return fits ? ROUTE_CLUSTER : ROUTE_CHAIN;
}

// One select.
static int launch_select_job(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, int prefetch, uint32_t tier,
                             uint32_t k, uint32_t *ids_out, uint32_t *n_out, cudaStream_t s)
{
    const uint32_t l = prefetch ? 2u : tier, ks[3] = {k, k, k};
    int route = select_route(ctx, idx->n_blocks, k, 1u << l, s), rc = CS_ENOTIMPL;
    if (route == ROUTE_GRID) {
        uint32_t *ids[3] = {}, *cnt[3] = {};
        ids[l] = ids_out;
        cnt[l] = n_out;
        rc = cs_launch_select_grid(ctx, idx, now, ks, ids, cnt, s);
        if (rc != CS_ENOTIMPL) return rc;
        if (idx->n_blocks <= CS_SELECT_CLUSTER_MAX_BLOCKS) route = ROUTE_CLUSTER;
    }
    SelectChain c;
    prepare_chain(ctx, 0, idx, now, prefetch, tier, k, ids_out, n_out, s, c);
    if (route == ROUTE_CLUSTER) {
        rc = cs_launch_select_cluster(ctx, &c.a, c.ws, prefetch, ids_out, n_out, s);
        if (rc != CS_ENOTIMPL) return rc;            // no usable cluster on this device: fall through
    }
    rc = scan_opt_in(ctx);
    for (int stage = 0; stage < SELECT_STAGES && rc == CS_OK; ++stage) rc = launch_stage(ctx, c, stage);
    return rc;
}

int cs_launch_select(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, int prefetch, uint32_t tier, uint32_t k,
                     uint32_t *ids_out, uint32_t *n_out, cudaStream_t s)
{
    return launch_select_job(ctx, idx, now, prefetch, tier, k, ids_out, n_out, s);
}

// The chains of selects side by side as one graph launch: true when it was launched, false when it has to be done launch by launch.
// A launch costs the host 2.5 us, so that the 12 or 18 of a step (33 and 50 us) took longer than
// their kernels (34 us for two lists of 1,000,000 entries); a node's new arguments take 0.2 us and the graph's launch 2 us.
// A single select stays six launches: its kernels take longer than issuing them (29 and 16 us), and its first launch
// overlaps the work before it on the stream, which a graph's does not.  Every argument is set anew on every call.
//
// The graph of a mix of lists is built (150 to 220 us) when a context is asked for that mix a second time: one that is asked
// once, or never has large indexes, does not pay for it.  The driver keeps a graph's nodes in device memory, so on a GPU that its
// user has filled any of these calls may be refused.  None of them has then enqueued anything: the launches stay single, in that call
// and from then on, and the call reports no error of its own.
static void drop_select_graph(cs_select_graph &g)
{
    if (g.exec) (void)cudaGraphExecDestroy(g.exec);
    if (g.graph) (void)cudaGraphDestroy(g.graph);
    g.exec = nullptr;
    g.graph = nullptr;
}

void cs_drop_select_graphs(cs_ctx *ctx)
{
    for (cs_select_graph &g : ctx->sel_graph) drop_select_graph(g);
}

static bool build_select_graph(cs_ctx *ctx, cs_select_graph &g, int n_jobs, SelectChain *chain)
{
    // (another thread may be capturing a stream of its own, which is nothing that these calls disturb)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return false;
    bool ok = cudaGraphCreate(&g.graph, 0) == cudaSuccess;
    if (!ok) g.graph = nullptr;
    for (int i = 0; i < n_jobs; ++i)
        for (int stage = 0; stage < SELECT_STAGES && ok; ++stage) ok = launch_stage(ctx, chain[i], stage, &g, i) == CS_OK;
    if (ok && cudaGraphInstantiate(&g.exec, g.graph, 0) != cudaSuccess) { ok = false; g.exec = nullptr; }
    (void)cudaThreadExchangeStreamCaptureMode(&mode);
    if (!ok) drop_select_graph(g);
    return ok;
}

static bool graph_of_selects(cs_ctx *ctx, uint32_t mask, int n_jobs, SelectChain *chain, cudaStream_t s)
{
    cs_select_graph &g = ctx->sel_graph[mask];
    if (g.refused) return false;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    if (st != cudaStreamCaptureStatusNone) return false;
    if (!g.exec && ++g.asked < 2) return false;
    const uint64_t launches = ctx->n_launches;
    const int last_error = ctx->last_cuda_error;
    bool ok = g.exec || build_select_graph(ctx, g, n_jobs, chain);
    ctx->n_launches = launches;                      // (adding the nodes launched nothing)
    for (int i = 0; i < n_jobs; ++i)
        for (int stage = 0; stage < SELECT_STAGES && ok; ++stage) ok = launch_stage(ctx, chain[i], stage, &g, i) == CS_OK;
    if (ok && cudaGraphLaunch(g.exec, s) == cudaSuccess) return true;
    // (a graph that has run stays until the context goes: earlier launches of it may still be running)
    g.refused = 1;
    ctx->n_launches = launches;
    ctx->last_cuda_error = last_error;
    (void)cudaGetLastError();
    return false;
}

// The selects of a step side by side.  Select q (0 GPU-tier victims, 1 host-tier victims, 2 prefetch candidates)
// is skipped when its count pointer is NULL.  Where the single-launch select applies they are the clusters of ONE
// launch; otherwise every select is a chain of grid-wide kernels (each has its own select state, histogram and candidate /
// sort regions), the chains side by side in one graph or, on the first call and while the caller's stream is being captured, the first on that
// stream and the others on the context's two extra streams, forked from and joined back into it with events.  Indexes beyond CS_CONCURRENT_MAX_BLOCKS entries
// have no private regions of that size: their selects run one after the other.
int cs_launch_select_step(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, uint32_t k_victims, uint32_t k_prefetch,
                          uint32_t *gpu_victims, uint32_t *n_gpu, uint32_t *host_victims, uint32_t *n_host,
                          uint32_t *prefetch_ids, uint32_t *n_prefetch, cudaStream_t s)
{
    uint32_t *const ids[3] = {gpu_victims, host_victims, prefetch_ids};
    uint32_t *const cnt[3] = {n_gpu, n_host, n_prefetch};
    const uint32_t ks[3] = {k_victims, k_victims, k_prefetch};
    int jobs[3], n_jobs = 0;
    for (int q = 0; q < 3; ++q)
        if (cnt[q]) jobs[n_jobs++] = q;
    if (n_jobs == 0) return CS_OK;
    uint32_t k_most = 0, lists = 0;
    for (int i = 0; i < n_jobs; ++i) {
        k_most = std::max(k_most, ks[jobs[i]]);
        lists |= 1u << jobs[i];
    }
    const bool together = ctx->concurrent_selects || idx->n_blocks <= CS_SELECT_CLUSTER_MAX_BLOCKS;           // every list has scratch of its own
    int route = together ? select_route(ctx, idx->n_blocks, k_most, lists, s) : ROUTE_CHAIN, rc = CS_OK;
    if (route == ROUTE_GRID) {
        rc = cs_launch_select_grid(ctx, idx, now, ks, ids, cnt, s);
        if (rc != CS_ENOTIMPL) return rc;
        route = idx->n_blocks <= CS_SELECT_CLUSTER_MAX_BLOCKS ? ROUTE_CLUSTER : ROUTE_CHAIN;
    }
    if (route == ROUTE_CLUSTER) {
        SelArgs a[3];
        uint32_t *j_ids[3], *j_cnt[3];
        uint32_t pf[3];
        for (int i = 0; i < n_jobs; ++i) {
            const int q = jobs[i];
            cs_fill_sel_args(ctx, idx, now, ctx->fsurv_override ? ctx->fsurv_override : ctx->ws.fsurv, a[i]);
            a[i].tier = q == 0 ? 0u : 1u;
            a[i].k = ks[q];
            a[i].hint_slot = ctx->no_speculation ? 3u : (uint32_t)q;
            a[i].kind = (uint32_t)q;
            cs_fill_sel_bins(ctx, a[i], q == 2);
            j_ids[i] = ids[q];
            j_cnt[i] = cnt[q];
            pf[i] = q == 2 ? 1u : 0u;
        }
        rc = cs_launch_select_clusters(ctx, n_jobs, a, pf, j_ids, j_cnt, s);
        if (rc != CS_ENOTIMPL) return rc;
    }
    rc = CS_OK;
    if (!ctx->concurrent_selects || n_jobs == 1) {
        for (int i = 0; i < n_jobs && rc == CS_OK; ++i) {
            const int q = jobs[i];
            rc = launch_select_job(ctx, idx, now, q == 2, q == 0 ? 0u : 1u, ks[q], ids[q], cnt[q], s);
        }
        return rc;
    }
    if ((rc = scan_opt_in(ctx)) != CS_OK) return rc;
    SelectChain chain[3];
    for (int i = 0; i < n_jobs; ++i) {
        const int q = jobs[i];
        prepare_chain(ctx, i, idx, now, q == 2, q == 0 ? 0u : 1u, ks[q], ids[q], cnt[q], i ? ctx->sel_stream[i - 1] : s, chain[i]);
    }
    uint32_t mask = 0;
    for (int i = 0; i < n_jobs; ++i) mask |= 1u << jobs[i];
    if (graph_of_selects(ctx, mask, n_jobs, chain, s)) return CS_OK;
    // Launched one by one: in turn, because issued one chain after the other the second one started 20 us (six launches) after
    // the first and both ended that much later.
    cudaError_t e = cudaEventRecord(ctx->ev_sel_fork, s);
    for (int i = 1; i < n_jobs && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(ctx->sel_stream[i - 1], ctx->ev_sel_fork, 0);
    for (int stage = 0; stage < SELECT_STAGES && e == cudaSuccess; ++stage)
        for (int i = 0; i < n_jobs && rc == CS_OK; ++i) rc = launch_stage(ctx, chain[i], stage);
    for (int i = 1; i < n_jobs && e == cudaSuccess; ++i) {
        e = cudaEventRecord(ctx->ev_sel_join[i - 1], ctx->sel_stream[i - 1]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ctx->ev_sel_join[i - 1], 0);
    }
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
    return rc;
}

// =============================================================================================
// Victim selection for callers that cannot allocate device memory.
//
// Some embedders of this library never get to call cudaMalloc: a serving engine that has handed
// the whole GPU to its own KV pool at start-up, a plug-in hook that runs while allocation is
// forbidden (inside a region where the host application has frozen its memory map), or a
// process whose memory budget is fixed by its launcher.  They can pass inputs and outputs they
// already own, but not a workspace.  For them the scratch of the select kernels (recency table,
// histogram, candidate keys, buckets, counters) lives in the file-scope array below, which
// every GPU that loads the library holds until the process exits.
//
// The array's name is only a host-side handle: the device address is obtained once per device
// with cudaGetSymbolAddress() and that pointer is what the kernels get.
// =============================================================================================
#define CS_STATIC_MAX_DEVICES 64
#define CS_STATIC_ALIGN(x) (((x) + 255u) / 256u * 256u)
// layout of the static scratch, byte offsets (every region 256-byte aligned)
#define CS_SO_SC 0u
#define CS_SO_SEL (CS_SO_SC + CS_STATIC_ALIGN(sizeof(cs_scalars)))
#define CS_SO_GTAB (CS_SO_SEL + CS_STATIC_ALIGN(sizeof(cs_sel_state)))
#define CS_SO_HIST (CS_SO_GTAB + CS_GTAB_MAX * 4u)
#define CS_SO_SPLKM (CS_SO_HIST + CS_HIST_BINS * 4u)
#define CS_SO_SPLID (CS_SO_SPLKM + CS_STATIC_ALIGN(CS_SAMPLE * 8u))
#define CS_SO_BCOUNT (CS_SO_SPLID + CS_STATIC_ALIGN(CS_SAMPLE * 4u))
#define CS_SO_CANDKM (CS_SO_BCOUNT + CS_STATIC_ALIGN(CS_BUCKETS * CS_BCOUNT_STRIDE * 4u))
#define CS_SO_SORTKM (CS_SO_CANDKM + CS_STATIC_MAX_BLOCKS * 8u)
#define CS_SO_CANDID (CS_SO_SORTKM + CS_STATIC_MAX_BLOCKS * 8u)
#define CS_SO_CANDBKT (CS_SO_CANDID + CS_STATIC_MAX_BLOCKS * 4u)
#define CS_SO_CANDSLOT (CS_SO_CANDBKT + CS_STATIC_MAX_BLOCKS * 4u)
#define CS_SO_SORTID (CS_SO_CANDSLOT + CS_STATIC_MAX_BLOCKS * 4u)
#define CS_SO_CNT (CS_SO_SORTID + CS_STATIC_MAX_BLOCKS * 4u)
#define CS_STATIC_BYTES (CS_SO_CNT + CS_STATIC_ALIGN(sizeof(cs_counters)))

static __device__ __align__(256) unsigned char cs_static_scratch[CS_STATIC_BYTES];   // 2 MiB + 60 KiB

static std::mutex g_static_mu;
static unsigned char *g_static_ptr[CS_STATIC_MAX_DEVICES];     // device address of the array, per device
static int g_static_sms[CS_STATIC_MAX_DEVICES];

// Everything the select kernels expect to find zeroed, and the recency table for this call's
// lambda / delta.  The array keeps the previous call's contents, so this runs on every call.
__global__ void cs_static_prepare_kernel(cs_workspace ws, uint32_t gtab_len, float lambda, float delta)
{
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    for (uint32_t i = tid; i < CS_HIST_BINS; i += nth) ws.hist[i] = 0;
    for (uint32_t i = tid; i < gtab_len; i += nth) ws.gtab[i] = cs_recency(lambda, delta, i);
    if (tid == 0) {
        cs_scalars z;
        memset(&z, 0, sizeof(z));
        z.last_agent = CS_AGENT_NONE;
        z.a_star = 0xFFFFFFFFu;
        z.sel_T[0] = z.sel_T[1] = z.sel_T[2] = z.sel_T[3] = ~0ull;
        *ws.sc = z;
        cs_sel_state zs;
        memset(&zs, 0, sizeof(zs));
        *ws.sel = zs;
    }
}

extern "C" int cs_select_victims_static(const cs_params *p, const float *fsurv, const cs_block_index *idx,
                                        uint32_t now, uint32_t tier, uint32_t k, uint32_t *ids_out, uint32_t *n_out,
                                        cs_stream_t stream)
{
    int rc = cs_validate_params(p);
    if (rc != CS_OK) return rc;
    if (!idx || !fsurv || (((uintptr_t)fsurv) & 3u) || tier > 1) return CS_EINVAL;
    if (idx->n_blocks > CS_STATIC_MAX_BLOCKS || k > CS_STATIC_MAX_BLOCKS) return CS_ECAPACITY;
    if (!n_out || (((uintptr_t)n_out) & 3u)) return CS_EINVAL;
    if (k && (!ids_out || (((uintptr_t)ids_out) & 15u))) return CS_EINVAL;
    if (idx->n_blocks) {
        if (!idx->agent || !idx->depth || !idx->ref_count || !idx->flags || !idx->last_access) return CS_EINVAL;
        const uintptr_t any = (uintptr_t)idx->agent | (uintptr_t)idx->depth | (uintptr_t)idx->ref_count |
                              (uintptr_t)idx->flags | (uintptr_t)idx->last_access | (uintptr_t)idx->n_tokens;
        if (any & 15u) return CS_EINVAL;
    }
    // Memory the SMs cannot address (a pageable host array) would fault the GPU: every pointer the kernels
    // dereference is looked up first (a host-side query that allocates nothing); nothing is launched on failure.
    {
        const void *ptrs[10] = {fsurv, n_out, k ? ids_out : nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
        if (idx->n_blocks) {
            ptrs[3] = idx->agent; ptrs[4] = idx->depth; ptrs[5] = idx->ref_count; ptrs[6] = idx->flags;
            ptrs[7] = idx->last_access; ptrs[8] = idx->n_tokens;
        }
        for (int i = 0; i < 10; ++i)
            if (ptrs[i] && !cs_device_can_address(ptrs[i])) return CS_EINVAL;
    }
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= CS_STATIC_MAX_DEVICES) return CS_ECUDA;
    int stream_dev = dev;        // the array of the CURRENT device is used: a stream of another device is refused
    if (stream && cudaStreamGetDevice((cudaStream_t)stream, &stream_dev) == cudaSuccess && stream_dev != dev) return CS_EINVAL;
    (void)cudaGetLastError();
    {
        // first call on this device: resolve the device address of the array (once, with the device current)
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (!g_static_ptr[dev]) {
            void *ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, cs_static_scratch) != cudaSuccess || !ptr) return CS_ECUDA;
            int sms = 0;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return CS_ECUDA;
            g_static_sms[dev] = sms;
            g_static_ptr[dev] = (unsigned char *)ptr;
        }
    }
    unsigned char *base;
    int sms;
    {
        std::lock_guard<std::mutex> lock(g_static_mu);
        base = g_static_ptr[dev];
        sms = g_static_sms[dev];
    }
    cs_ctx ctx;                                        // host-side descriptor only; nothing is allocated
    memset(&ctx, 0, sizeof(ctx));
    ctx.p = *p;
    ctx.p.max_blocks = CS_STATIC_MAX_BLOCKS;
    cs_recency_table_shape(p, &ctx.gtab_len, &ctx.age_sat);
    ctx.device = dev;
    ctx.sm_count = sms;
    cs_workspace &ws = ctx.ws;
    ws.sc = (cs_scalars *)(base + CS_SO_SC);
    ws.sel = (cs_sel_state *)(base + CS_SO_SEL);
    ws.gtab = (float *)(base + CS_SO_GTAB);
    ws.hist = (uint32_t *)(base + CS_SO_HIST);
    ws.spl_km = (unsigned long long *)(base + CS_SO_SPLKM);
    ws.spl_id = (uint32_t *)(base + CS_SO_SPLID);
    ws.bcount = (uint32_t *)(base + CS_SO_BCOUNT);
    ws.cand_km = (unsigned long long *)(base + CS_SO_CANDKM);
    ws.sort_km = (unsigned long long *)(base + CS_SO_SORTKM);
    ws.cand_id = (uint32_t *)(base + CS_SO_CANDID);
    ws.cand_bkt = (uint32_t *)(base + CS_SO_CANDBKT);
    ws.cand_slot = (uint32_t *)(base + CS_SO_CANDSLOT);
    ws.sort_id = (uint32_t *)(base + CS_SO_SORTID);
    ws.cnt = (cs_counters *)(base + CS_SO_CNT);
    ws.fsurv = const_cast<float *>(fsurv);             // input table, read only
    cudaStream_t s = (cudaStream_t)stream;
    cs_static_prepare_kernel<<<16, 256, 0, s>>>(ws, ctx.gtab_len, p->lambda, p->delta);
    if ((rc = cs_check_launch(&ctx)) != CS_OK) return rc;
    return cs_launch_select(&ctx, idx, now, 0, tier, k, ids_out, n_out, s);
}
