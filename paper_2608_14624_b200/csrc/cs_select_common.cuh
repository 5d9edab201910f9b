// Device helpers shared by the select kernels: the per-entry eligibility rules and 96-bit key
// (Algorithm 1, Evict / BetweenStep; Eq. 9), 128-bit loads of the SoA block index, small tables.
#pragma once
#include "cs_common.cuh"

typedef unsigned long long u64;

#define SEL_THREADS 512
#define GRP 16                    // index entries per thread and iteration

struct SelArgs {
    const uint16_t *agent;
    const uint16_t *depth;
    const uint8_t *ref;
    const uint8_t *flags;
    const uint32_t *la;
    const uint8_t *ntok;
    const uint16_t *anchor;
    const float *fsurv;
    uint32_t n, now, A, block_tokens, gtab_len, age_sat;
    float lambda, delta;
    uint32_t tier, k, prefer_copy;
    uint32_t use_age_limits;      // collect pass may prefilter by per-(agent, size) age limits (large indexes)
    uint32_t hint_slot;           // which remembered key (cs_scalars.sel_T) this call may speculate on
    uint32_t kind;                // 0 GPU-tier victims, 1 host-tier victims, 2 prefetch candidates (work counters)
    const uint32_t *now_dev;      // when set, the clock is read from device memory at execution time (graph replay)
    uint32_t region_cap_max;      // cap on the keys of a bucket (0: none)
    uint32_t max_blocks;          // keys the candidate and sort buffers hold
    uint32_t bin_lo, bin_shift;   // histogram bins: (primary - bin_lo) >> bin_shift, set per list kind
};

// host helpers defined in cs_select.cu
void cs_fill_sel_args(const cs_ctx *ctx, const cs_block_index *idx, uint32_t now, const float *fsurv, SelArgs &a);
void cs_fill_sel_bins(const cs_ctx *ctx, SelArgs &a, int prefetch);
uint32_t cs_scan_grid(const cs_ctx *ctx, uint32_t n, uint32_t per_cta, uint32_t ctas_per_sm = 2);
size_t cs_table_smem(const cs_ctx *ctx);

// How many candidates the next large select of a kind should find at or below the key it is given: enough that an index
// which loses its k best entries between calls, or whose survival table shifts, still has k of them; few enough that
// collecting and ordering them costs little.
__host__ __device__ __forceinline__ uint32_t cs_ahead(uint32_t k) { return k < 0x10000000u ? 3u * k + 4096u : 0x40000000u; }

// Work counters of one finished select (called by one thread).
__device__ __forceinline__ void count_select(const cs_workspace &ws, uint32_t kind, uint32_t n_elig, uint32_t n_out)
{
    if (kind > 2) return;
    atomicAdd((unsigned long long *)&ws.cnt->selects[kind], 1ull);
    atomicAdd((unsigned long long *)&ws.cnt->selected[kind], (unsigned long long)n_out);
    ws.cnt->eligible[kind] = n_elig;
}

__device__ __forceinline__ void count_candidates(const cs_workspace &ws, uint32_t kind, uint32_t c, bool fast_hit)
{
    if (kind > 2) return;
    ws.cnt->candidates[kind] = c;
    if (fast_hit) atomicAdd((unsigned long long *)&ws.cnt->fast_hits[kind], 1ull);
}

// The clock of a call: by value, or from device memory when the caller asked for that.
__device__ __forceinline__ void resolve_now(SelArgs &a)
{
    if (a.now_dev) a.now = __ldg(a.now_dev);
}

// Per-CTA copies of the small tables every entry looks up.
struct Tables {
    float *fsurv;       // [A]
    float *gtab;        // [gtab_len]
    uint16_t *anchor;   // [A] or unused
    float g_sat;
    uint32_t a_star;
};

// The recency table depends only on the context's constants (written when the context was created), so a kernel
// launched with programmatic dependent launch may copy it before it waits for its predecessor ...
__device__ __forceinline__ void load_tables_static(const SelArgs &a, const cs_workspace &ws, float *smem, Tables &T)
{
    T.fsurv = smem;
    T.gtab = smem + a.A;
    T.anchor = (uint16_t *)(smem + a.A + a.gtab_len);
    for (uint32_t i = threadIdx.x; i < a.gtab_len; i += blockDim.x) T.gtab[i] = ws.gtab[i];
    T.g_sat = cs_recency(a.lambda, a.delta, a.age_sat);
}
// ... while the survival table, the anchor lengths and a* may have been written by that predecessor.
__device__ __forceinline__ void load_tables_dynamic(const SelArgs &a, const cs_workspace &ws, Tables &T, bool want_anchor)
{
    for (uint32_t i = threadIdx.x; i < a.A; i += blockDim.x) T.fsurv[i] = a.fsurv[i];
    if (want_anchor)
        for (uint32_t i = threadIdx.x; i < a.A; i += blockDim.x) T.anchor[i] = a.anchor[i];
    T.a_star = ws.sc->a_star;           // arg-max successor of the current agent, kept by the learner refresh
}

__device__ __forceinline__ void load_tables(const SelArgs &a, const cs_workspace &ws, float *smem, Tables &T,
                                            bool want_anchor)
{
    load_tables_static(a, ws, smem, T);
    load_tables_dynamic(a, ws, T, want_anchor);
}

// Recency factor of Eq. 9 for an age: from the table, the saturated constant, or (a decay so slow that the
// table does not reach saturation) computed directly.
__device__ __forceinline__ float recency_of_age(const SelArgs &a, const Tables &T, uint32_t age)
{
    if (age < a.gtab_len) return T.gtab[age];
    if (age >= a.age_sat) return T.g_sat;
    return cs_recency(a.lambda, a.delta, age);
}

__device__ __forceinline__ float score_from_age(const SelArgs &a, const Tables &T, uint32_t agent, uint32_t age,
                                                uint32_t tok)
{
    return __fmul_rn(__fmul_rn(T.fsurv[agent], recency_of_age(a, T, age)), (float)tok);      // two roundings, never an FMA
}

__device__ __forceinline__ float score_of(const SelArgs &a, const Tables &T, uint32_t agent, uint32_t la,
                                          uint32_t tok)
{
    const uint32_t age = la <= a.now ? a.now - la : 0u;
    float g;
    if (age < a.gtab_len) g = T.gtab[age];
    else if (age >= a.age_sat) g = T.g_sat;
    else g = cs_recency(a.lambda, a.delta, age);
    return __fmul_rn(__fmul_rn(T.fsurv[agent], g), (float)tok);      // two roundings, never an FMA
}

// Histogram bin of a primary key: the range of possible scores divided evenly over the bins (of both classes of a prefetch
// list), clamped at its ends, which keeps the order whatever the survival table holds.
template <bool PF, class Bins>
__device__ __forceinline__ uint32_t bin_of(const Bins &a, uint32_t pr)
{
    const uint32_t v = PF ? pr & 0x7FFFFFFFu : pr;
    const uint32_t x = (v > a.bin_lo ? v - a.bin_lo : 0u) >> a.bin_shift;
    constexpr uint32_t PER_CLASS = PF ? CS_HIST_BINS / 2 : CS_HIST_BINS;
    const uint32_t b = x < PER_CLASS - 1u ? x : PER_CLASS - 1u;
    return PF ? b + ((pr >> 31) ? PER_CLASS : 0u) : b;
}

// "bin <= b0" as a limit on the primary key: candidate <=> primary < limit.
template <bool PF, class Bins>
__device__ __forceinline__ u64 primary_limit(const Bins &a, uint32_t b0)
{
    constexpr uint32_t PER_CLASS = PF ? CS_HIST_BINS / 2 : CS_HIST_BINS;
    const uint32_t b = b0 % PER_CLASS;
    const u64 cls = PF && b0 >= PER_CLASS ? 0x80000000ull : 0ull, end = PF ? 0x80000000ull : 0x100000000ull;
    const u64 lim = (u64)a.bin_lo + ((u64)(b + 1u) << a.bin_shift);
    return cls + (b == PER_CLASS - 1u || lim > end ? end : lim);     // (a class's last bin holds the rest of it)
}

// Key of an entry already known to pass the flag / ref_count rules: the agent range check, the
// anchor-depth rule of the prefetch list, and the 96-bit key.
template <bool PF>
__device__ __forceinline__ bool entry_key_rest(const SelArgs &a, const Tables &T, uint32_t *status, uint32_t agent,
                                               uint32_t depth, uint32_t flags, uint32_t la, uint32_t tok,
                                               uint32_t &primary, uint32_t &secondary)
{
    if (agent >= a.A) { atomicOr(status, CS_ST_BAD_AGENT); return false; }
    if (PF && a.anchor && !(depth < T.anchor[agent])) return false;
    const uint32_t bits = __float_as_uint(score_of(a, T, agent, la, tok));
    if (PF) {
        primary = ((agent == T.a_star) ? 0u : 0x80000000u) | (~bits & 0x7FFFFFFFu);
        secondary = ~la;
    } else {
        // Optional preference (Sec. 4) for victims whose contents already exist on the other tier:
        // one extra key bit right below the score (a positive float leaves bit 31 free).
        primary = a.prefer_copy ? ((bits << 1) | ((flags & CS_FLAG_OTHER_COPY) ? 0u : 1u)) : bits;
        secondary = la;
    }
    return true;
}

// Eligibility and key of one entry.  PF = prefetch-candidate rules, else eviction-victim rules.
template <bool PF>
__device__ __forceinline__ bool entry_key(const SelArgs &a, const Tables &T, uint32_t *status, uint32_t agent,
                                          uint32_t depth, uint32_t ref, uint32_t flags, uint32_t la, uint32_t tok,
                                          uint32_t &primary, uint32_t &secondary)
{
    if (!(flags & CS_FLAG_VALID) || (flags & CS_FLAG_PINNED) || ref != 0) return false;
    if (PF) {
        if (!(flags & CS_FLAG_TIER_HOST) || (flags & CS_FLAG_OTHER_COPY)) return false;
    } else {
        if (((flags >> 2) & 1u) != a.tier) return false;
    }
    return entry_key_rest<PF>(a, T, status, agent, depth, flags, la, tok, primary, secondary);
}

// The index is walked in warp tiles of 512 entries.  In step q (0..3) lane L owns the four
// consecutive entries tile*512 + q*128 + 4L .. +3, so every load instruction of a warp covers one
// contiguous, fully used span: 512 B of last_access (128-bit loads), 256 B of agent / depth
// (64-bit), 128 B of flags / ref_count / n_tokens (32-bit).  A thread's 16 entries are numbered
// j = 4q + r locally; Group keeps them in the order the accessors below expect.
#define TILE 512u
struct Group {
    uint4 ag0, ag1, dp0, dp1, rf, fl, la0, la1, la2, la3, tk;
};

__device__ __forceinline__ uint32_t grp_id(uint32_t tile, uint32_t lane, int j)
{
    return tile * TILE + (uint32_t)(j >> 2) * 128u + 4u * lane + (uint32_t)(j & 3);
}

template <bool PF, bool FLAGS = true>
__device__ __forceinline__ void load_group(const SelArgs &a, uint32_t tile, uint32_t lane, Group &G)
{
    const uint32_t q0 = tile * 128u + lane;            // index of this lane's first quad, in units of 4 entries
    const uint4 *la = (const uint4 *)a.la + q0;
    G.la0 = __ldg(la);
    G.la1 = __ldg(la + 32);
    G.la2 = __ldg(la + 64);
    G.la3 = __ldg(la + 96);
    const uint2 *ag = (const uint2 *)a.agent + q0;
    const uint2 g0 = __ldg(ag), g1 = __ldg(ag + 32), g2 = __ldg(ag + 64), g3 = __ldg(ag + 96);
    G.ag0 = make_uint4(g0.x, g0.y, g1.x, g1.y);
    G.ag1 = make_uint4(g2.x, g2.y, g3.x, g3.y);
    if (FLAGS) {
        const uint32_t *rf = (const uint32_t *)a.ref + q0, *fl = (const uint32_t *)a.flags + q0;
        G.rf = make_uint4(__ldg(rf), __ldg(rf + 32), __ldg(rf + 64), __ldg(rf + 96));
        G.fl = make_uint4(__ldg(fl), __ldg(fl + 32), __ldg(fl + 64), __ldg(fl + 96));
    }
    if (a.ntok) {
        const uint32_t *tk = (const uint32_t *)a.ntok + q0;
        G.tk = make_uint4(__ldg(tk), __ldg(tk + 32), __ldg(tk + 64), __ldg(tk + 96));
    }
    if (PF && a.anchor) {
        const uint2 *dp = (const uint2 *)a.depth + q0;
        const uint2 d0 = __ldg(dp), d1 = __ldg(dp + 32), d2 = __ldg(dp + 64), d3 = __ldg(dp + 96);
        G.dp0 = make_uint4(d0.x, d0.y, d1.x, d1.y);
        G.dp1 = make_uint4(d2.x, d2.y, d3.x, d3.y);
    }
}

__device__ __forceinline__ uint32_t u4_word(const uint4 &v, int w)
{
    return w == 0 ? v.x : (w == 1 ? v.y : (w == 2 ? v.z : v.w));
}
__device__ __forceinline__ uint32_t grp_u16(const uint4 &lo, const uint4 &hi, int j)   // j in [0,16)
{
    const uint32_t w = u4_word(j < 8 ? lo : hi, (j & 7) >> 1);
    return (w >> ((j & 1) * 16)) & 0xFFFFu;
}
__device__ __forceinline__ uint32_t grp_u8(const uint4 &v, int j)
{
    return (u4_word(v, j >> 2) >> ((j & 3) * 8)) & 0xFFu;
}
__device__ __forceinline__ uint32_t grp_u32(const Group &G, int j)
{
    const uint4 &v = j < 4 ? G.la0 : (j < 8 ? G.la1 : (j < 12 ? G.la2 : G.la3));
    return u4_word(v, j & 3);
}

// Flag / ref_count rules for the 16 entries of a group at once, four entries per 32-bit word
// (byte-wise SIMD compares): bit j of the result is set when entry j is VALID, not PINNED, on the
// requested tier (prefetch: on the host tier without a GPU copy) and unreferenced.
// 0x80 in every byte of x that is zero (exact for all four bytes at once, plain integer operations).
__device__ __forceinline__ uint32_t zero_bytes(uint32_t x)
{
    return ~(((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x | 0x7F7F7F7Fu);
}
// The four 0x80 flags of a word gathered into a nibble (bit i = byte i).
__device__ __forceinline__ uint32_t nibble_of_flags(uint32_t t)
{
    return (((t >> 7) * 0x01020408u) >> 24) & 0xFu;
}

template <bool PF>
__device__ __forceinline__ uint32_t group_elig(const SelArgs &a, const Group &G)
{
    const uint32_t fmask = PF ? 0x0F0F0F0Fu : 0x07070707u;
    const uint32_t fpat = PF ? 0x05050505u : (0x01010101u * (CS_FLAG_VALID | (a.tier << 2)));
    uint32_t out = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        // a byte of x is zero exactly when the entry's flags match the pattern and its ref_count is 0
        const uint32_t x = ((u4_word(G.fl, w) & fmask) ^ fpat) | u4_word(G.rf, w);
        out |= nibble_of_flags(zero_bytes(x)) << (4 * w);
    }
    return out;
}

// Calls f(id, primary, secondary) for every eligible entry this thread owns: whole warp tiles
// grid-strided, then the ragged tail (n % 512 entries) one entry per thread.
template <bool PF, typename F>
__device__ __forceinline__ void for_each_eligible(const SelArgs &a, const Tables &T, uint32_t *status, F f)
{
    const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const uint32_t lane = threadIdx.x & 31, n_tiles = a.n / TILE;
    for (uint32_t t = gtid >> 5; t < n_tiles; t += nth >> 5) {
        Group G;
        load_group<PF>(a, t, lane, G);
        const uint32_t em = group_elig<PF>(a, G);
#pragma unroll
        for (int j = 0; j < GRP; ++j) {
            if (!((em >> j) & 1u)) continue;
            uint32_t pr, se;
            const uint32_t tok = a.ntok ? grp_u8(G.tk, j) : a.block_tokens;
            const uint32_t dp = (PF && a.anchor) ? grp_u16(G.dp0, G.dp1, j) : 0u;
            if (entry_key_rest<PF>(a, T, status, grp_u16(G.ag0, G.ag1, j), dp, grp_u8(G.fl, j), grp_u32(G, j), tok, pr, se))
                f(grp_id(t, lane, j), pr, se);
        }
    }
    const uint32_t t0 = n_tiles * TILE;
    if (gtid < a.n - t0) {
        const uint32_t i = t0 + gtid;
        uint32_t pr, se;
        const uint32_t tok = a.ntok ? a.ntok[i] : a.block_tokens;
        if (entry_key<PF>(a, T, status, a.agent[i], a.depth[i], a.ref[i], a.flags[i], a.la[i], tok, pr, se))
            f(i, pr, se);
    }
}

// Warp-private staging of candidates.  Inside the 16-entry loop of a scan every lane holds at most one
// candidate per step; a ballot gives each its slot in the warp's shared-memory slice, with no atomic and no
// second pass over the group.  A slice that is more than half full is appended to the global candidate
// buffer: one atomic per flush, coalesced writes.  Every call below is made by all 32 lanes of the warp.
#define STAGE_CAP 64u
struct WarpStage {
    unsigned long long *km;      // [STAGE_CAP]
    uint32_t *id;                // [STAGE_CAP]
    uint32_t n;                  // staged entries (same value in every lane)
};

__device__ __forceinline__ void stage_init(WarpStage &st, unsigned long long *km_all, uint32_t *id_all)
{
    const uint32_t warp = threadIdx.x >> 5;
    st.km = km_all + warp * STAGE_CAP;
    st.id = id_all + warp * STAGE_CAP;
    st.n = 0;
}

__device__ __forceinline__ void stage_flush(WarpStage &st, uint32_t *counter, unsigned long long *out_km, uint32_t *out_id)
{
    if (st.n == 0) return;
    const uint32_t lane = threadIdx.x & 31;
    __syncwarp();
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(counter, st.n);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    for (uint32_t i = lane; i < st.n; i += 32) {
        out_km[base + i] = st.km[i];
        out_id[base + i] = st.id[i];
    }
    __syncwarp();
    st.n = 0;
}

__device__ __forceinline__ void stage_push(WarpStage &st, bool cand, uint32_t pr, uint32_t se, uint32_t id,
                                           uint32_t *counter, unsigned long long *out_km, uint32_t *out_id)
{
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, cand);
    if (b == 0) return;
    if (cand) {
        const uint32_t pos = st.n + __popc(b & ((1u << (threadIdx.x & 31)) - 1u));
        st.km[pos] = ((unsigned long long)pr << 32) | se;
        st.id[pos] = id;
    }
    st.n += __popc(b);
    if (st.n > STAGE_CAP - 32u) stage_flush(st, counter, out_km, out_id);
}

// The prefetch list is empty unless the gate of Eq. 11 is open and a current agent exists.
__device__ __forceinline__ bool prefetch_enabled(const cs_workspace &ws, uint32_t A)
{
    return ws.sc->gate != 0 && ws.sc->last_agent < A;
}

__device__ __forceinline__ bool last_cta_done(uint32_t *ticket, bool *s_flag)
{
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) *s_flag = (atomicAdd(ticket, 1u) == gridDim.x - 1);
    __syncthreads();
    const bool last = *s_flag;
    if (last) __threadfence();
    return last;
}

// Exclusive prefix sum of one value per thread over the CTA (warp shuffles, three barriers); also returns the total.
// s_part: at least 64 words.
__device__ __forceinline__ uint32_t sel_block_scan(uint32_t v, uint32_t *s_part, uint32_t &total)
{
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += t;
    }
    __syncthreads();
    if (lane == 31) s_part[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < n_warps ? s_part[lane] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, w, d);
            if (lane >= d) w += t;
        }
        s_part[32 + lane] = w;                         // inclusive warp totals
    }
    __syncthreads();
    total = s_part[32 + n_warps - 1];
    const uint32_t before = warp ? s_part[32 + warp - 1] : 0;
    return before + incl - v;
}

// Adds 1 to `count` where (ka, ia) < (kb, ib): the borrow of a 96-bit subtraction.
__device__ __forceinline__ void count_less(uint32_t &count, u64 ka, uint32_t ia, u64 kb, uint32_t ib)
{
    uint32_t r;
    asm("{\n\t.reg .u32 x;\n\tsub.cc.u32 x, %1, %2;\n\tsubc.cc.u32 x, %3, %4;\n\tsubc.cc.u32 x, %5, %6;\n\tsubc.u32 %0, 0, 0;\n\t}"
        : "=r"(r)
        : "r"(ia), "r"(ib), "r"((uint32_t)ka), "r"((uint32_t)kb), "r"((uint32_t)(ka >> 32)), "r"((uint32_t)(kb >> 32)));
    count -= r;
}
__device__ __forceinline__ bool less96(u64 ka, uint32_t ia, u64 kb, uint32_t ib)
{
    uint32_t n = 0;
    count_less(n, ka, ia, kb, ib);
    return n != 0;
}

// Ranks m keys against c keys, both in shared memory: emit(rank, km, id) for each.  Whole CTA; up to 32 neighbouring
// lanes share a key.
template <class Emit>
__device__ __forceinline__ void rank_keys(const u64 *km, const uint32_t *id, uint32_t m, const u64 *all_km, const uint32_t *all_id,
                                          uint32_t c, Emit emit)
{
    uint32_t parts = 1;
    while (parts < 32u && 2u * parts * m <= blockDim.x) parts <<= 1;
    const uint32_t sub = threadIdx.x & (parts - 1u), step = blockDim.x / parts;
    for (uint32_t k0 = 0; k0 < m; k0 += step) {                     // (uniform: whole warps stay in the shuffles)
        const uint32_t k = k0 + threadIdx.x / parts;
        const bool have = k < m;
        const u64 my = have ? km[k] : 0ull;
        const uint32_t mine = have ? id[k] : 0u;
        uint32_t r = 0;
#pragma unroll 4
        for (uint32_t q = sub; q < c; q += parts) count_less(r, all_km[q], all_id[q], my, mine);
        for (uint32_t d = parts >> 1; d > 0; d >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, d);
        if (have && sub == 0) emit(r, my, mine);
    }
}

// Sorts a list of places of keys, ascending by the keys.  Whole CTA.  Bitonic, with the first step of every merge between mirror images,
// so that every comparator moves the smaller key to the lower place: places past the end then never take part, and any length will do.
static __device__ __noinline__ void sort_places(uint32_t *list, uint32_t m, const u64 *__restrict__ km, const uint32_t *__restrict__ id)
{
    constexpr int ITEMS = 4;                                  // comparators per thread whose loads travel together
    uint32_t P = 2;
    while (P < m) P <<= 1;                                    // (at most 2^31: a list is no longer than an index)
    for (uint32_t half = 1; half < m; half <<= 1)
        for (uint32_t step = half, mirror = 1; step > 0; step >>= 1, mirror = 0) {
            for (uint32_t t0 = threadIdx.x; t0 < P / 2; t0 += ITEMS * blockDim.x) {
                uint32_t lo[ITEMS], hi[ITEMS], a[ITEMS], b[ITEMS], ia[ITEMS], ib[ITEMS];
                u64 ka[ITEMS], kb[ITEMS];
                bool in[ITEMS];
#pragma unroll
                for (int u = 0; u < ITEMS; ++u) {
                    const uint32_t t = t0 + u * blockDim.x, x = t & (step - 1u);
                    lo[u] = 2u * t - x;
                    hi[u] = mirror ? lo[u] + 2u * (step - x) - 1u : lo[u] + step;
                    in[u] = t < P / 2 && hi[u] < m;
                    a[u] = in[u] ? __ldcg(list + lo[u]) : 0u;
                    b[u] = in[u] ? __ldcg(list + hi[u]) : 0u;
                }
#pragma unroll
                for (int u = 0; u < ITEMS; ++u) {
                    ka[u] = __ldcg(km + a[u]);
                    kb[u] = __ldcg(km + b[u]);
                    ia[u] = __ldcg(id + a[u]);
                    ib[u] = __ldcg(id + b[u]);
                }
#pragma unroll
                for (int u = 0; u < ITEMS; ++u)
                    if (in[u] && less96(kb[u], ib[u], ka[u], ia[u])) { list[lo[u]] = b[u]; list[hi[u]] = a[u]; }
            }
            __syncthreads();
        }
}

__device__ __forceinline__ bool key_less(unsigned long long km_a, uint32_t id_a, unsigned long long km_b,
                                         uint32_t id_b)
{
    return km_a < km_b || (km_a == km_b && id_a < id_b);
}



// ---------------------------------------------------------------------------------------------
// Bitonic sort of P keys (power of two, 64 <= P <= 2 * threads of the CTA) held in shared memory,
// ascending by (km, id).  Each thread keeps two neighbouring elements in registers; compare-
// exchange steps whose partner lies in the same warp (element distance <= 32) use shuffles and
// no barrier, only the longer distances go through shared memory.  Called by every thread.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void cx_keep(unsigned long long &k, uint32_t &i, unsigned long long pk, uint32_t pi,
                                        bool keep_min)
{
    const bool partner_less = key_less(pk, pi, k, i);
    if (partner_less == keep_min) { k = pk; i = pi; }
}

__device__ __forceinline__ void bitonic_sort_fast(unsigned long long *km, uint32_t *id, uint32_t P)
{
    const uint32_t t = threadIdx.x;
    const bool act = t < P / 2;                           // whole warps, because P >= 64
    unsigned long long k0 = 0, k1 = 0;
    uint32_t i0 = 0, i1 = 0;
    if (act) { k0 = km[2 * t]; k1 = km[2 * t + 1]; i0 = id[2 * t]; i1 = id[2 * t + 1]; }
    for (uint32_t size = 2; size <= P; size <<= 1) {
        const bool up = ((2 * t) & size) == 0;            // both of this thread's elements share the direction
        uint32_t stride = size >> 1;
        if (stride >= 64) {                               // partners in other warps: through shared memory
            if (act) { km[2 * t] = k0; km[2 * t + 1] = k1; id[2 * t] = i0; id[2 * t + 1] = i1; }
            __syncthreads();
            for (; stride >= 64; stride >>= 1) {
                if (act) {
                    const uint32_t lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                    const bool up2 = (lo & size) == 0;
                    const unsigned long long ka = km[lo], kb = km[hi];
                    const uint32_t ia = id[lo], ib = id[hi];
                    if (key_less(kb, ib, ka, ia) == up2) { km[lo] = kb; id[lo] = ib; km[hi] = ka; id[hi] = ia; }
                }
                __syncthreads();
            }
            if (act) { k0 = km[2 * t]; k1 = km[2 * t + 1]; i0 = id[2 * t]; i1 = id[2 * t + 1]; }
        }
        if (act) {
            for (; stride >= 2; stride >>= 1) {           // partner thread t ^ (stride / 2), same warp
                const uint32_t d = stride >> 1;
                const unsigned long long pk0 = __shfl_xor_sync(0xFFFFFFFFu, k0, d), pk1 = __shfl_xor_sync(0xFFFFFFFFu, k1, d);
                const uint32_t pi0 = __shfl_xor_sync(0xFFFFFFFFu, i0, d), pi1 = __shfl_xor_sync(0xFFFFFFFFu, i1, d);
                const bool keep_min = ((t & d) == 0) == up;
                cx_keep(k0, i0, pk0, pi0, keep_min);
                cx_keep(k1, i1, pk1, pi1, keep_min);
            }
            if (key_less(k1, i1, k0, i0) == up) {         // distance 1: this thread's own pair
                const unsigned long long tk = k0; k0 = k1; k1 = tk;
                const uint32_t ti = i0; i0 = i1; i1 = ti;
            }
        }
    }
    __syncthreads();
    if (act) { km[2 * t] = k0; km[2 * t + 1] = k1; id[2 * t] = i0; id[2 * t + 1] = i1; }
    __syncthreads();
}

// ---------------------------------------------------------------------------------------------
// Sorts the first m keys of a shared-memory tile ascending (bitonic; m is padded to a power of two, which the tile has to hold,
// with keys that sort last).  Whole CTA.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void sort_tile(unsigned long long *t_km, uint32_t *t_id, uint32_t m)
{
    uint32_t P = 64;
    while (P < m) P <<= 1;
    for (uint32_t i = m + threadIdx.x; i < P; i += blockDim.x) { t_km[i] = ~0ull; t_id[i] = 0xFFFFFFFFu; }
    __syncthreads();
    if (P <= 2 * blockDim.x) {
        bitonic_sort_fast(t_km, t_id, P);
        return;
    }
    for (uint32_t size = 2; size <= P; size <<= 1) {
        for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
            for (uint32_t t = threadIdx.x; t < P / 2; t += blockDim.x) {
                const uint32_t lo = 2 * t - (t & (stride - 1));
                const uint32_t hi = lo + stride;
                const bool up = (lo & size) == 0;
                const unsigned long long ka = t_km[lo], kb = t_km[hi];
                const uint32_t ia = t_id[lo], ib = t_id[hi];
                if (key_less(kb, ib, ka, ia) == up) {
                    t_km[lo] = kb; t_id[lo] = ib;
                    t_km[hi] = ka; t_id[hi] = ia;
                }
            }
            __syncthreads();
        }
    }
}
