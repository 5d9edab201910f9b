// Ordering the candidates of a large select on the whole GPU: ranks of a sample, buckets between the samples, keys counted within their
// bucket.  Device functions over (CTA, number of CTAs), used by the launch chain of cs_select.cu, a launch per step, and by the one
// launch of cs_select_grid.cu, with grid barriers between the steps.
#pragma once
#include "cs_select_common.cuh"

// ---------------------------------------------------------------------------------------------
// Ordering the candidates.
//
// The n_out smallest of c candidates, in order, by ranks of a sample: 1,024 candidates at even distances are ranked against
// each other (counting smaller ones: 96-bit compares spread over 64 CTAs), and J of them cover the output with four
// standard deviations to spare.  Everything beyond the J-th is dropped; the rest is split at the samples into nb buckets of a few dozen
// keys, which are small enough to be ranked by counting as well.  Whole-GPU launches, because the work is comparisons:
// one cluster of 16 SMs took 36 us for 35,000 candidates, k = 10,000 (8 us the sample, 14 us the buckets, 8 us the ranks).
// A bucket has a fixed region of the sort arrays; one that outgrows it is gathered again from the candidates by its CTA.
//
// At most FEW_MAX candidates (short lists: the remembered key follows a list of a few hundred down to about a thousand) all go into the
// sample: their ranks are their places, and the other two launches return at once.  Per select of 741,250 entries, k = 300: 22.1 us
// with buckets, 18.7 so; three lists side by side 33.2 and 26.2.  The line: with 1,024 the three lists of k = 800 stay at 32.6 (30.5
// with 2,048); 3,072 gives a list of 2,500 candidates nothing or costs it 2 us.  (Ranges of a sample in each of the 64 CTAs, as in a cluster,
// for up to 8,192: as fast up to about 1,400 candidates, 1 to 2 us slower than the buckets beyond.)
// ---------------------------------------------------------------------------------------------
#define FEW_MAX 2048u             // a multiple of 1,024
#define RANK_TILE 2048u           // keys of the shared-memory tile a bucket is sorted in
struct OrderPlan {
    uint32_t S, J;            // samples; of those, how many cover the output
    uint32_t gaps;            // gap g lies between samples g - 1 and g (the first from the smallest key, the last to the largest
                              // key when no sample lies beyond the output)
    uint32_t sub, join;       // buckets per gap, gaps per bucket; one of them is 1
    uint32_t nb, cap;         // buckets, and keys a bucket's region holds
};
__device__ __forceinline__ OrderPlan order_plan(uint32_t c, uint32_t n_out, uint32_t max_blocks, uint32_t region_max)
{
    OrderPlan P;
    P.S = c < CS_SAMPLE ? c : CS_SAMPLE;
    const float e = (float)n_out * (float)P.S / (float)c;
    const uint32_t want = (uint32_t)(e + 4.0f * sqrtf(e)) + 3u;
    P.J = want < P.S ? want : P.S;
    P.gaps = P.J + (P.J == P.S ? 1u : 0u);
    P.sub = P.gaps <= CS_BUCKETS ? CS_BUCKETS / P.gaps : 1u;
    P.join = (P.gaps + CS_BUCKETS - 1u) / CS_BUCKETS;
    P.nb = P.join > 1u ? (P.gaps + P.join - 1u) / P.join : P.gaps * P.sub;
    P.cap = max_blocks / P.nb;
    if (region_max && P.cap > region_max) P.cap = region_max;
    return P;
}
// Smallest key of bucket j.  A gap that is several buckets is divided evenly: locally the keys of a tie in score are spread
// evenly over last_access, and the largest of a few hundred gaps is six times the mean one.
__device__ __forceinline__ void bucket_start(const OrderPlan &P, const u64 *s_km, const uint32_t *s_id, uint32_t j, u64 &km, uint32_t &id)
{
    const uint32_t g = P.join > 1u ? j * P.join : j / P.sub, f = P.join > 1u ? 0u : j - g * P.sub;
    km = g ? s_km[g - 1] : 0ull;
    id = g ? s_id[g - 1] : 0u;
    if (j >= P.nb) {
        km = ~0ull;
        id = 0xFFFFFFFFu;
    } else if (f) {
        const u64 step = ((g < P.J ? s_km[g] : ~0ull) - km) / P.sub;
        if (step) id = 0u;                                    // (a gap inside a tie down to the id is not divided)
        km += step * f;
    }
}

// The key the next call of this kind gets: the one it had while the candidates it gave were enough and not too many; where
// they were too many, the key below which `ahead` of them lay; where they were few, as much beyond it as the
// candidates above the list's last entry say that so many would need.
__device__ __forceinline__ u64 next_bound(const cs_sel_state &st, uint32_t k, u64 kth, uint32_t ahead)
{
    const u64 none = ~0ull, all = ~0ull - 1ull;
    if (st.n_elig <= k) return all;                           // everything eligible is wanted
    if (st.ahead != none && (!st.spec || st.c > ahead + ahead / 4u)) return st.ahead < all ? st.ahead : all;
    if (st.c >= 2ull * k + 1024ull || st.c >= st.n_elig || st.bound >= all || st.bound < kth) return st.bound < all ? st.bound : all;
    const u64 gap = st.bound - kth, per = (ahead - st.c) / (st.c - k + 1u);
    const u64 more = (gap < (1ull << 40) ? gap : (1ull << 40)) * (per < 8ull ? per : 8ull) + 64ull;
    return more < all - st.bound ? st.bound + more : all;
}

// The sample, ranked by all CTAs (a warp per key); the ids themselves when all candidates are in it.  s_km / s_id: FEW_MAX keys.
// next(kth key) is called by whoever places the list's last id.
template <class Next>
__device__ __forceinline__ void rank_sample(const cs_workspace &ws, uint32_t c, uint32_t n_out, uint32_t ahead, unsigned long long *ahead_out,
                                            u64 *s_km, uint32_t *s_id, uint32_t cta, uint32_t n_ctas, uint32_t *__restrict__ ids_out, Next next)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_threads = blockDim.x, n_warps = n_threads >> 5;
    const bool few = c <= FEW_MAX;
    const uint32_t S = few ? c : CS_SAMPLE, padded = (S + 255u) & ~255u;
    for (uint32_t s0 = 0; s0 < S; s0 += 2u * n_threads) {
        u64 km[2];
        uint32_t id[2];
#pragma unroll
        for (uint32_t u = 0; u < 2; ++u) {
            const uint32_t s = s0 + tid + u * n_threads, at = s < S ? (uint32_t)((u64)s * c / S) : 0u;
            km[u] = cs_ld_cg_pinned(ws.cand_km + at);
            id[u] = cs_ld_cg_pinned(ws.cand_id + at);
        }
#pragma unroll
        for (uint32_t u = 0; u < 2; ++u) {
            const uint32_t s = s0 + tid + u * n_threads;
            s_km[s] = s < S ? km[u] : ~0ull;
            s_id[s] = s < S ? id[u] : 0xFFFFFFFFu;
        }
    }
    if (cta == 0 && tid == 0 && c <= ahead) *ahead_out = ~0ull;
    __syncthreads();
    for (uint32_t s = cta * n_warps + warp; s < S; s += n_ctas * n_warps) {
        const u64 my = s_km[s];
        const uint32_t mine = s_id[s];
        uint32_t r = 0;
#pragma unroll 8
        for (uint32_t q = lane; q < padded; q += 32u) count_less(r, s_km[q], s_id[q], my, mine);
        r = __reduce_add_sync(0xFFFFFFFFu, r);
        if (few) {
            if (lane == 0 && r < n_out) ids_out[r] = mine;
            if (lane == 0) next(r, my, mine);
        } else if (lane == 0) {
            ws.spl_km[r] = my;
            ws.spl_id[r] = mine;
            if (c > ahead && r == (uint32_t)((u64)ahead * S / c)) *ahead_out = my;
        }
    }
}

// The candidates below the cut go to their buckets.  st: c and n_out of the select, asked for by the caller; s_km / s_id: CS_SAMPLE
// keys, b_km / b_id: CS_BUCKETS.  ready() is called once this thread's first keys and the tables are there.
template <class Ready>
__device__ __forceinline__ void place_candidates(const cs_workspace &ws, uint4 st, uint32_t max_blocks, uint32_t region_max, u64 *s_km, uint32_t *s_id,
                                                 u64 *b_km, uint32_t *b_id, uint32_t cta, uint32_t n_ctas, Ready ready)
{
    constexpr int ITEMS = 4;                                  // candidates per thread and round
    constexpr int PER = 4;                                    // (at least 256 threads)
    const uint32_t tid = threadIdx.x, NT = blockDim.x;
    // Everything the first round needs is asked for at once -- the select's state, the ranked sample and the round's keys
    // (addresses bounded by the capacity of the buffers; what lies beyond the live counts is ignored below).  Item u of a
    // round lies a grid-wide sweep after item u - 1, so that few candidates spread over all CTAs.
    const uint32_t sweep = n_ctas * NT, lane0 = cta * NT + tid;
    u64 km[ITEMS], sk[PER];
    uint32_t id[ITEMS], si[PER];
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        const uint32_t i = u * sweep + lane0, ii = i < max_blocks ? i : 0u;
        km[u] = cs_ld_cg_pinned(ws.cand_km + ii);
        id[u] = cs_ld_cg_pinned(ws.cand_id + ii);
    }
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (tid + NT * u < CS_SAMPLE) { sk[u] = cs_ld_cg_pinned(ws.spl_km + tid + NT * u); si[u] = cs_ld_cg_pinned(ws.spl_id + tid + NT * u); }
    const uint32_t c = st.x, n_out = st.y;
    if (n_out == 0 || c <= FEW_MAX) return;
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (tid + NT * u < CS_SAMPLE) { s_km[tid + NT * u] = sk[u]; s_id[tid + NT * u] = si[u]; }
    const OrderPlan P = order_plan(c, n_out, max_blocks, region_max);
    __syncthreads();
    const u64 cut_km = s_km[P.J - 1];
    const uint32_t cut_id = s_id[P.J - 1];
    for (uint32_t j = tid; j < CS_BUCKETS; j += NT) bucket_start(P, s_km, s_id, j, b_km[j], b_id[j]);
    __syncthreads();
    ready();
    for (uint32_t base = 0; base < c; base += sweep * ITEMS) {
        if (base != 0) {
#pragma unroll
            for (int u = 0; u < ITEMS; ++u) {
                const uint32_t i = base + u * sweep + lane0, ii = i < c ? i : 0u;
                km[u] = cs_ld_cg_pinned(ws.cand_km + ii);
                id[u] = cs_ld_cg_pinned(ws.cand_id + ii);
            }
        }
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            const uint32_t i = base + u * sweep + lane0;
            // keys from the cut up are dropped when there are samples beyond it
            if (i >= c || (P.J < P.S && !less96(km[u], id[u], cut_km, cut_id))) continue;
            uint32_t b = 0;                                   // the last bucket that starts at or below the key
#pragma unroll
            for (uint32_t step = CS_BUCKETS / 2; step > 0; step >>= 1)
                b += less96(km[u], id[u], b_km[b + step], b_id[b + step]) ? 0u : step;
            const uint32_t slot = atomicAdd(&CS_BCOUNT(ws, b), 1u);
            if (slot < P.cap) {
                ws.sort_km[(size_t)b * P.cap + slot] = km[u];
                ws.sort_id[(size_t)b * P.cap + slot] = id[u];
            }
        }
    }
}

// Bucket b of CTA b: ranked by counting while it is small, sorted in the tile (bitonic, O(m log^2 m)) when it is larger, and through a
// list of its keys' places, sorted in global memory, when the tile does not hold it.  The list lies where the bucket's ids lie in the
// whole order -- [off, off + m) of an array of one word per entry -- so that no two buckets share a word.  Long lists come here as a
// matter of course: the keys between two samples are exponentially spread, so the largest of several hundred buckets is four to six times
// the mean one (432,000 candidates, k = 150,000: one or two buckets of 2,300 keys; 1,730,000, k = 600,000: 9,000).
#define FINISH_THREADS 512u
#define FINISH_COUNT_MAX 512u
// Whole CTA.  t_km / t_id: RANK_TILE keys; s_off, s_max, s_n: a word each, zero before; next(place, key) as in rank_sample().
template <class Next>
__device__ __forceinline__ void finish_bucket(const cs_workspace &ws, uint32_t c, uint32_t n_out, const OrderPlan &P, uint32_t b, uint32_t n_t,
                                              uint32_t m, uint32_t kind, u64 *t_km, uint32_t *t_id, uint32_t *s_off, uint32_t *s_max,
                                              uint32_t *s_n, uint32_t *__restrict__ ids_out, Next next)
{
    const uint32_t tid = threadIdx.x;
    const uint32_t before = __reduce_add_sync(0xFFFFFFFFu, tid < b ? n_t : 0u);
    if ((tid & 31) == 0 && before) atomicAdd(s_off, before);
    if (b == 0) {                                             // work counters, and whether any bucket outgrew its region
        const uint32_t most = __reduce_max_sync(0xFFFFFFFFu, n_t);
        if ((tid & 31) == 0) atomicMax(s_max, most);
    }
    __syncthreads();
    const uint32_t off = *s_off;
    if (b == 0 && tid == 0 && kind < 3) {
        atomicAdd((unsigned long long *)&ws.cnt->region_selects[kind], 1ull);
        if (*s_max > P.cap) atomicAdd((unsigned long long *)&ws.cnt->region_overflows[kind], 1ull);
    }
    // (should the sample have misled, the last bucket takes everything from its start on)
    const bool rest = b == P.nb - 1u && P.J < P.S && off + m < n_out;
    if (rest) m = c - off;
    if (off >= n_out || m == 0) return;
    const u64 *src_km = ws.sort_km + (size_t)b * P.cap;
    const uint32_t *src_id = ws.sort_id + (size_t)b * P.cap;
    auto emit = [&](uint32_t r, u64 km, uint32_t id) {       // one id of the list
        const uint32_t pos = off + r;
        if (pos >= n_out) return;
        ids_out[pos] = id;
        next(pos, km, id);
    };
    const bool outgrown = m > P.cap || rest, fits = m <= RANK_TILE;
    uint32_t *const list = ws.cand_bkt + off;                 // [m] places of the keys when the tile does not hold them
    if (outgrown) {
        // the region was too small: the bucket's keys once more, out of all candidates
        u64 lo_km, hi_km;
        uint32_t lo_id, hi_id;
        bucket_start(P, ws.spl_km, ws.spl_id, b, lo_km, lo_id);
        bucket_start(P, ws.spl_km, ws.spl_id, b + 1u, hi_km, hi_id);
        if (b == P.nb - 1u && P.J < P.S && !rest) { hi_km = ws.spl_km[P.J - 1]; hi_id = ws.spl_id[P.J - 1]; }
        for (uint32_t i0 = tid; i0 < c; i0 += 4u * blockDim.x) {
            u64 km[4];
            uint32_t id[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * blockDim.x;
                km[u] = __ldcg(ws.cand_km + (i < c ? i : 0u));
                id[u] = __ldcg(ws.cand_id + (i < c ? i : 0u));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * blockDim.x;
                if (i >= c || less96(km[u], id[u], lo_km, lo_id) || !less96(km[u], id[u], hi_km, hi_id)) continue;
                const uint32_t at = atomicAdd(s_n, 1u);      // (m of them: the bucket's counter has counted the same keys)
                if (at >= m) continue;
                if (fits) { t_km[at] = km[u]; t_id[at] = id[u]; }
                else list[at] = i;
            }
        }
        __syncthreads();
        m = min(m, *s_n);
    } else if (fits) {
        for (uint32_t i = tid; i < m; i += blockDim.x) {
            t_km[i] = __ldcg(src_km + i);
            t_id[i] = __ldcg(src_id + i);
        }
        __syncthreads();
    } else {
        for (uint32_t i = tid; i < m; i += blockDim.x) list[i] = i;
        __syncthreads();
    }
    if (!fits) {
        const u64 *k_km = outgrown ? ws.cand_km : src_km;
        const uint32_t *k_id = outgrown ? ws.cand_id : src_id;
        sort_places(list, m, k_km, k_id);
        for (uint32_t i = tid; i < m && off + i < n_out; i += blockDim.x) {
            const uint32_t at = __ldcg(list + i);
            emit(i, __ldcg(k_km + at), __ldcg(k_id + at));
        }
        return;
    }
    if (m <= FINISH_COUNT_MAX) {
        rank_keys(t_km, t_id, m, t_km, t_id, m, emit);
    } else {
        sort_tile(t_km, t_id, m);
        for (uint32_t i = tid; i < m; i += blockDim.x) emit(i, t_km[i], t_id[i]);
    }
}
