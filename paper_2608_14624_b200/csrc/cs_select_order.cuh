// Ordering the candidates of a select inside one thread-block cluster.
//
// A select ends with c candidates of which the n_out smallest, in ascending order, are the answer.  Sorting them in one SM
// is bound by that SM's shared memory and shuffles (measured: 1,024 keys of 96 bits take 13,600 cycles as a bitonic sort,
// 10,000 as warp sorts merged by binary search, twice that for 2,048).  Two facts make it cheap on a cluster: a key's place in
// the output is the number of smaller keys, so keys can be placed without being moved; and keys that fall into ranges of
// their own never have to be compared with each other.  So every CTA (few candidates) or every warp (many) takes ranges
// chosen from the ranks of a sample, and counts.  Four instructions per comparison: a 96-bit subtraction whose borrow is
// added up.
//
//   c <= 4,096  every CTA reads all candidates, keeps the range that is its share of the output, splits it at the samples
//               inside it and counts within the parts;
//   more        the whole cluster ranks a sample of 512 or 1,024.  Where the output is a small part of the candidates, what
//               lies beyond it is dropped and the rest is looked at afresh; else the keys go to up to 256 buckets, one
//               range each, whose keys are counted by the warps of one CTA, 32 at a time;
//   long lists  (more than 30,720 ids) are not ordered here: a bucket of m keys takes m^2 comparisons, and 256 buckets are all there
//               are.  The caller's sample sort does them (OR_LONG).
//
// What CTAs hand each other goes through L2, in runs: distributed shared memory moves scattered 8-byte words at about one
// per four cycles and SM (handing the ranked sample of 1,024 to 16 CTAs that way took 8.6 us with the ranking, 6.4 us through L2;
// 2,000 candidates pulled out of 16 CTAs' lists 2.6 us, 0.75 us); it carries counters only.
//
// Keys are unique (the id is part of the key): the output does not depend on the order in which atomics were served, nor on
// the sample.
#pragma once
#include <cooperative_groups.h>

#include "cs_select_common.cuh"

namespace cg = cooperative_groups;

#define OR_THREADS 512u
#define OR_WARPS (OR_THREADS / 32u)
#define OR_ALL 4096u              // candidates a CTA holds at once
#define OR_BUCKETS 256u
// Longest list whose buckets are counted: 120 keys per bucket on average.  Per select of 262,144 entries, counted / sorted (us):
// k = 28,672 80 - 93 / 89, 32,768 103 - 108 / 94, 65,536 878 - 1,095 / 143 - 160, all 112,700 415 - 432 / 221 - 228 (the lower figures with
// every entry of one age).
#define OR_LONG (120u * OR_BUCKETS)
#define OR_SAMPLE CS_SAMPLE       // largest sample
#define OR_SMALL_SAMPLE 128u
#define OR_PART 256u              // keys of a part of a CTA's range (few candidates)
#define OR_PARTS 8u               // parts: samples a CTA's range spans, at most, + the start
static_assert(OR_PARTS * OR_PART <= 2 * OR_SAMPLE, "parts lie in the sample's memory");

struct OrderSmem {
    u64 *all_km;                  // [cap] candidates: everybody's (few), this CTA's buckets (many)
    u64 *s_km;                    // [2 * OR_SAMPLE] the sample, as drawn and in ascending order; the parts of a range
    uint32_t *all_id, *s_id;
    uint32_t *cnt, *off;          // [OR_BUCKETS + 4] sizes and output positions of the buckets
    uint32_t *part;               // [64] scan scratch
    uint32_t *misc;               // [OM_WORDS]
    uint32_t cap;
};
// OM_BELOW and OM_FILL (one word per part) are order_few()'s own: it clears them on entry with no barrier before that, while slower
// warps may still be reading any other word (OM_TOTAL in particular, on the way from a cut of the candidates).
enum { OM_B0 = 0, OM_CTOT, OM_LIST, OM_GLOBAL, OM_GLOBAL2, OM_OVERFLOW, OM_BELOW, OM_IN, OM_TOTAL, OM_FILL = 16, OM_WORDS = OM_FILL + (int)OR_PARTS };
static_assert(OM_TOTAL != OM_BELOW && (OM_TOTAL < OM_FILL || OM_TOTAL >= OM_FILL + (int)OR_PARTS), "read while order_few() clears its words");

// Where the candidates are and where they may be moved to; all of it private to the select.
struct OrderBufs {
    u64 *src_km, *dst_km, *spl_km;
    uint32_t *src_id, *dst_id, *spl_id;
    uint32_t *bcount;
    uint32_t dst_cap;             // keys dst holds
};
__device__ __forceinline__ OrderBufs order_bufs(const cs_workspace &ws, uint32_t cap)
{
    return OrderBufs{ws.cand_km, ws.sort_km, ws.spl_km, ws.cand_id, ws.sort_id, ws.spl_id, ws.bcount, cap};
}

__host__ __device__ inline size_t order_smem_bytes(uint32_t cap)
{
    return (size_t)(cap + 2 * OR_SAMPLE) * 12 + (2 * (OR_BUCKETS + 4) + 64 + OM_WORDS) * 4;
}

__device__ __forceinline__ void order_carve(unsigned char *base, uint32_t cap, OrderSmem &O)
{
    O.cap = cap;
    O.all_km = (u64 *)base;
    O.s_km = O.all_km + cap;
    O.all_id = (uint32_t *)(O.s_km + 2 * OR_SAMPLE);
    O.s_id = O.all_id + cap;
    O.cnt = O.s_id + 2 * OR_SAMPLE;
    O.off = O.cnt + OR_BUCKETS + 4;
    O.part = O.off + OR_BUCKETS + 4;
    O.misc = O.part + 64;
}

// One warp ranks the keys [k0, k0 + 32) of a part of m keys in shared memory.
__device__ __forceinline__ void rank_item(const u64 *km, const uint32_t *id, uint32_t m, uint32_t k0, uint32_t base, uint32_t n_out,
                                          uint32_t *__restrict__ ids_out)
{
    const uint32_t k = k0 + (threadIdx.x & 31);
    const u64 my = k < m ? km[k] : 0ull;
    const uint32_t mine = k < m ? id[k] : 0u;
    uint32_t r = 0;
#pragma unroll 8
    for (uint32_t q = 0; q < m; ++q) count_less(r, km[q], id[q], my, mine);
    if (k < m && base + r < n_out) ids_out[base + r] = mine;
}

// Sorts c keys in shared memory, ascending.  Whole CTA.  Bitonic with mirrored merges, as sort_places().
__device__ __noinline__ void sort_keys(u64 *km, uint32_t *id, uint32_t c)
{
    uint32_t P = 2;
    while (P < c) P <<= 1;
    for (uint32_t half = 1; half < c; half <<= 1)
        for (uint32_t step = half, mirror = 1; step > 0; step >>= 1, mirror = 0) {
            for (uint32_t t = threadIdx.x; t < P / 2; t += OR_THREADS) {
                const uint32_t x = t & (step - 1u), lo = 2u * t - x, hi = mirror ? lo + 2u * (step - x) - 1u : lo + step;
                if (hi >= c) continue;
                const u64 ka = km[lo], kb = km[hi];
                const uint32_t ia = id[lo], ib = id[hi];
                if (less96(kb, ib, ka, ia)) { km[lo] = kb; id[lo] = ib; km[hi] = ka; id[hi] = ia; }
            }
            __syncthreads();
        }
}

// Appends one key per participating lane to a list with a counter in shared memory; returns the lane's place.
__device__ __forceinline__ uint32_t warp_append(bool in, uint32_t *counter)
{
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, in), lane = threadIdx.x & 31;
    uint32_t at = 0;
    if (b && lane == 0) at = atomicAdd(counter, __popc(b));
    return __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(b & ((1u << lane) - 1u));
}

// c <= O.cap candidates: in all_km / all_id already (a cluster of one CTA), or to be read from src.  Every CTA of the cluster
// calls; CTAs do not meet.
__device__ __noinline__ void order_few(const OrderSmem &O, const u64 *src_km, const uint32_t *src_id, uint32_t c, uint32_t n_out,
                                       uint32_t *__restrict__ ids_out)
{
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    u64 *const all_km = O.all_km;
    uint32_t *const all_id = O.all_id;
    if (src_km) {
        for (uint32_t i0 = 0; i0 < c; i0 += 4u * OR_THREADS) {      // a round's loads travel together
            u64 km[4];
            uint32_t id[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * OR_THREADS + tid;
                if (i < c) { km[u] = cs_ld_cg_pinned(src_km + i); id[u] = cs_ld_cg_pinned(src_id + i); }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * OR_THREADS + tid;
                if (i < c) { all_km[i] = km[u]; all_id[i] = id[u]; }
            }
        }
    }
    if (tid <= OR_PARTS) O.misc[tid < OR_PARTS ? OM_FILL + tid : OM_BELOW] = 0;
    __syncthreads();
    if ((unsigned long long)c * c <= 32768ull * CL) {
        // few: every CTA places an equal share of the keys, each counted against all of them
        const uint32_t k0 = rank * c / CL, k1 = (rank + 1u) * c / CL;
        rank_keys(all_km + k0, all_id + k0, k1 - k0, all_km, all_id, c, [&](uint32_t r, u64, uint32_t id) {
            if (r < n_out) ids_out[r] = id;
        });
        return;
    }
    // ---- a sample of 128, ranked by everybody, splits the output among the CTAs -------------------------------------------------
    constexpr uint32_t S = OR_SMALL_SAMPLE;
    u64 *s_km = O.s_km, *t_km = O.s_km + S;
    uint32_t *s_id = O.s_id, *t_id = O.s_id + S;
    if (tid < S) {
        const uint32_t at = (uint32_t)((unsigned long long)tid * c / S);
        s_km[tid] = all_km[at];
        s_id[tid] = all_id[at];
    }
    __syncthreads();
    {
        const u64 my = s_km[tid >> 2];
        const uint32_t mine = s_id[tid >> 2];
        uint32_t r = 0;
#pragma unroll 8
        for (uint32_t q = tid & 3u; q < S; q += 4u) count_less(r, s_km[q], s_id[q], my, mine);
        r += __shfl_xor_sync(0xFFFFFFFFu, r, 1);
        r += __shfl_xor_sync(0xFFFFFFFFu, r, 2);
        if ((tid & 3u) == 0) { t_km[r] = my; t_id[r] = mine; }
    }
    __syncthreads();
    // sample ranks that cover the output with four standard deviations to spare; should they fall short, the last CTA
    // takes everything above
    const float e = (float)n_out * (float)S / (float)c;
    const uint32_t want = (uint32_t)(e + 4.0f * sqrtf(e)) + 3u, J = want < S ? want : S;
    const uint32_t l0 = rank * J / CL, l1 = (rank + 1u) * J / CL;      // this CTA: from sample l0 - 1 (0: the start) up to sample l1 - 1
    if (l0 == l1 && rank != CL - 1) return;
    // the samples inside the range split it into parts
    const uint32_t per = (l1 - l0 + OR_PARTS - 1u) / OR_PARTS, n_parts = per ? (l1 - l0 + per - 1u) / per : 1u;
    u64 b_km[OR_PARTS + 1];
    uint32_t b_id[OR_PARTS + 1];
#pragma unroll
    for (uint32_t p = 0; p <= OR_PARTS; ++p) {
        const uint32_t l = l0 + p * per < l1 ? l0 + p * per : l1;
        const bool end = l == l1 && l1 == S;                           // beyond the last sample: no limit
        b_km[p] = l == 0 ? 0ull : (end ? ~0ull : t_km[l - 1]);
        b_id[p] = l == 0 ? 0u : (end ? 0xFFFFFFFFu : t_id[l - 1]);
    }
    __syncthreads();                                                   // (the parts overwrite the samples)
    u64 hi_km = b_km[OR_PARTS];
    uint32_t hi_id = b_id[OR_PARTS];
    for (int pass = 0; pass < 2; ++pass) {
        uint32_t below = 0;
        for (uint32_t i0 = 0; i0 < c; i0 += OR_THREADS) {
            const uint32_t i = i0 + tid;
            const u64 km = i < c ? all_km[i] : ~0ull;
            const uint32_t id = i < c ? all_id[i] : 0xFFFFFFFFu;
            const bool lt = i < c && less96(km, id, b_km[0], b_id[0]);
            const bool in = i < c && !lt && less96(km, id, hi_km, hi_id);
            below += lt ? 1u : 0u;
            if (in) {
                uint32_t p = 0;
#pragma unroll
                for (uint32_t x = 1; x < OR_PARTS; ++x)
                    if (x < n_parts && !less96(km, id, b_km[x], b_id[x])) p = x;
                const uint32_t at = atomicAdd(&O.misc[OM_FILL + p], 1u);
                if (at < OR_PART) { O.s_km[p * OR_PART + at] = km; O.s_id[p * OR_PART + at] = id; }
            }
        }
        below = __reduce_add_sync(0xFFFFFFFFu, below);
        if (lane == 0 && below) atomicAdd(&O.misc[OM_BELOW], below);
        __syncthreads();
        uint32_t m = 0, largest = 0;
#pragma unroll
        for (uint32_t p = 0; p < OR_PARTS; ++p) {
            const uint32_t f = O.misc[OM_FILL + p];
            m += f;
            largest = largest > f ? largest : f;
        }
        const uint32_t base = O.misc[OM_BELOW];
        if (rank == CL - 1 && base + m < n_out && (hi_km != ~0ull || hi_id != 0xFFFFFFFFu)) {
            __syncthreads();                                           // the sample misjudged: take the rest as well
            hi_km = ~0ull;
            hi_id = 0xFFFFFFFFu;
            if (tid <= OR_PARTS) O.misc[tid < OR_PARTS ? OM_FILL + tid : OM_BELOW] = 0;
            __syncthreads();
            continue;
        }
        if (base >= n_out || m == 0) return;
        if (largest <= OR_PART) {
            uint32_t item = 0, at = base;
            for (uint32_t p = 0; p < n_parts; ++p) {
                const uint32_t f = O.misc[OM_FILL + p];
                for (uint32_t k0 = 0; k0 < f; k0 += 32u, ++item)
                    if ((item & (OR_WARPS - 1u)) == warp)
                        rank_item(O.s_km + p * OR_PART, O.s_id + p * OR_PART, f, k0, at, n_out, ids_out);
                at += f;
            }
        } else {
            // A part too long for its place: gaps between samples are exponentially spread, so of 4,000 candidates one list in thirty has
            // a gap of 256 keys or more, and a sample that misleads has nearly all of them in one.  All candidates are here: sorted,
            // every key is at its place in the list.  (Counting each of the range's keys against all of them took 800 us, this 55.)
            sort_keys(all_km, all_id, c);
            for (uint32_t i = base + tid; i < base + m && i < n_out; i += OR_THREADS) ids_out[i] = all_id[i];
        }
        return;
    }
}

// c > 0 candidates in B.src, n_out > 0.  Every CTA of the cluster calls, after a cluster barrier; the candidates' writes are
// visible.  False: the list is too long, the buckets overflowed or a sample misled; nothing was stored, the candidates are in B.src.
__device__ __noinline__ bool order_candidates(const OrderSmem &O, OrderBufs &B, uint32_t &c, uint32_t n_out,
                                                     uint32_t *__restrict__ ids_out)
{
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    u64 *s_km = O.s_km, *t_km = O.s_km + OR_SAMPLE;                 // the sample, and the same in ascending order
    uint32_t *s_id = O.s_id, *t_id = O.s_id + OR_SAMPLE;
    uint32_t *lead = cluster.map_shared_rank(O.misc, 0);
    for (uint32_t round = 0;; ++round) {
        if (c <= OR_ALL && c <= O.cap) {
            order_few(O, B.src_km, B.src_id, c, n_out, ids_out);
            return true;
        }
        if (n_out > OR_LONG || round == 6) return false;        // (every round drops most of the candidates)
        // ---- a sample, ranked by the cluster; CL lanes share a key ------------------------------------------------------
        const uint32_t S = c <= 12288u ? OR_SAMPLE / 2 : OR_SAMPLE;
        for (uint32_t s = tid; s < S; s += OR_THREADS) {
            const uint32_t at = (uint32_t)((unsigned long long)s * c / S);
            s_km[s] = __ldcg(B.src_km + at);
            s_id[s] = __ldcg(B.src_id + at);
        }
        uint32_t *total_word = lead + (round & 1u ? OM_GLOBAL2 : OM_GLOBAL);
        if (rank == 0) {
            for (uint32_t b = tid; b < OR_BUCKETS; b += OR_THREADS) B.bcount[(size_t)b * CS_BCOUNT_STRIDE] = 0;
            if (tid == 0) { O.misc[round & 1u ? OM_GLOBAL2 : OM_GLOBAL] = 0; O.misc[OM_OVERFLOW] = 0; }
        }
        __syncthreads();
        for (uint32_t s0 = rank * (S / CL); s0 < (rank + 1u) * (S / CL); s0 += OR_THREADS / CL) {
            const uint32_t s = s0 + tid / CL, sub = tid & (CL - 1u);
            const u64 my = s_km[s];
            const uint32_t mine = s_id[s];
            uint32_t r = 0;
#pragma unroll 8
            for (uint32_t q = sub; q < S; q += CL) count_less(r, s_km[q], s_id[q], my, mine);
            for (uint32_t d = CL >> 1; d > 0; d >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, d);
            if (sub == 0) { B.spl_km[r] = my; B.spl_id[r] = mine; }
        }
        __threadfence();
        cluster.sync();
        for (uint32_t s = tid; s < S; s += OR_THREADS) { t_km[s] = cs_ld_cg_pinned(B.spl_km + s); t_id[s] = cs_ld_cg_pinned(B.spl_id + s); }
        const float e = (float)n_out * (float)S / (float)c;
        const uint32_t want = (uint32_t)(e + 4.0f * sqrtf(e)) + 3u, J = want < S ? want : S;      // sample ranks that cover the output
        __syncthreads();
        const u64 cut_km = J < S ? t_km[J - 1] : ~0ull;
        const uint32_t cut_id = J < S ? t_id[J - 1] : 0xFFFFFFFFu;
        const uint32_t beg = (uint32_t)((unsigned long long)rank * c / CL), end = (uint32_t)((unsigned long long)(rank + 1u) * c / CL);
        const bool fill = J >= 96u;                                 // enough samples below the cut to split the output evenly
        const uint32_t nb = J < OR_BUCKETS ? J : OR_BUCKETS;
        // (no more than a CTA holds: the workspace may have been made for a far larger index than this one, and a sample that misleads
        // may put nearly all candidates into one bucket)
        const uint32_t cap = min(B.dst_cap / nb, O.cap);
        // ---- what lies below the cut: into buckets, or into dst for another round ----------------------------------------
        for (uint32_t i0 = beg; i0 < end; i0 += 4u * OR_THREADS) {
            u64 km[4];
            uint32_t id[4], b[4], slot[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * OR_THREADS + tid, ii = i < end ? i : beg;
                km[u] = cs_ld_cg_pinned(B.src_km + ii);
                id[u] = cs_ld_cg_pinned(B.src_id + ii);
            }
            if (!fill) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t i = i0 + u * OR_THREADS + tid;
                    const bool in = i < end && less96(km[u], id[u], cut_km, cut_id);
                    if (!__any_sync(0xFFFFFFFFu, in)) continue;
                    const uint32_t at = warp_append(in, total_word);
                    if (in) { B.dst_km[at] = km[u]; B.dst_id[at] = id[u]; }       // (dst holds as many keys as src)
                }
                continue;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) b[u] = 0;
#pragma unroll 1
            for (uint32_t step = OR_BUCKETS / 2; step > 0; step >>= 1) {
                // splitters at or below the key; splitter j (from 1) = sample rank j J / nb
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t j = b[u] + step, at = (j < nb ? j : 0u) * J / nb;
                    if (j < nb && !less96(km[u], id[u], t_km[at], t_id[at])) b[u] = j;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {                           // the round's atomics are in flight together
                const uint32_t i = i0 + u * OR_THREADS + tid;
                if (i >= end || !(J == S || less96(km[u], id[u], cut_km, cut_id))) b[u] = 0xFFFFFFFFu;
                else slot[u] = atomicAdd(B.bcount + (size_t)b[u] * CS_BCOUNT_STRIDE, 1u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (b[u] == 0xFFFFFFFFu) continue;
                if (slot[u] < cap) {
                    B.dst_km[(size_t)b[u] * cap + slot[u]] = km[u];
                    B.dst_id[(size_t)b[u] * cap + slot[u]] = id[u];
                } else {
                    lead[OM_OVERFLOW] = 1u;
                }
            }
        }
        __threadfence();
        cluster.sync();
        if (!fill) {
            if (tid == 0) O.misc[OM_TOTAL] = *total_word;
            cluster.barrier_arrive();
            __syncthreads();
            const uint32_t total = O.misc[OM_TOTAL];
            cluster.barrier_wait();                                 // (the leader may go on, or leave)
            if (total < n_out || total >= c) return false;      // the sample misjudged
            u64 *a_km = B.src_km; B.src_km = B.dst_km; B.dst_km = a_km;
            uint32_t *a_id = B.src_id; B.src_id = B.dst_id; B.dst_id = a_id;
            c = total;
            continue;
        }
        // ---- the buckets: b belongs to CTA b % CL ----------------------------------------------------------------------
        const uint32_t mine = tid < nb ? cs_ld_cg_pinned(B.bcount + (size_t)tid * CS_BCOUNT_STRIDE) : 0u;
        if (tid == 0) O.misc[OM_TOTAL] = lead[OM_OVERFLOW];
        uint32_t total;
        const uint32_t excl = sel_block_scan(mine, O.part, total);
        if (tid < nb) { O.off[tid] = excl; O.cnt[tid] = mine; }
        cluster.barrier_arrive();                                   // (the leader's flag has been read; waited for at the end)
        __syncthreads();
        const uint32_t per = nb > rank ? (nb - rank + CL - 1u) / CL : 0u;      // this CTA's buckets
        const bool ok = !O.misc[OM_TOTAL] && total >= n_out;
        // as many buckets at a time as shared memory holds (one always fits), up to the end of the output (offsets grow with the bucket)
        for (uint32_t first = 0; ok && first < per && O.off[first * CL + rank] < n_out;) {
            uint32_t need = 0, last = first;
            for (; last < per; ++last) {                            // keys into shared memory, a warp per bucket in turn
                const uint32_t g = last * CL + rank, m = O.cnt[g];
                if (O.off[g] >= n_out || need + m > O.cap) break;
                if ((last & (OR_WARPS - 1u)) == warp)
                    for (uint32_t i = lane; i < m; i += 32u) {
                        O.all_km[need + i] = __ldcg(B.dst_km + (size_t)g * cap + i);
                        O.all_id[need + i] = __ldcg(B.dst_id + (size_t)g * cap + i);
                    }
                need += m;
            }
            __syncthreads();
            uint32_t item = 0, at = 0;
            for (uint32_t lb = first; lb < last; ++lb) {
                const uint32_t g = lb * CL + rank, m = O.cnt[g];
                for (uint32_t k0 = 0; k0 < m; k0 += 32u, ++item)    // items of 32 keys, dealt to the warps in turn
                    if ((item & (OR_WARPS - 1u)) == warp)
                        rank_item(O.all_km + at, O.all_id + at, m, k0, O.off[g], n_out, ids_out);
                at += m;
            }
            first = last;
            __syncthreads();                                        // (before the next buckets take their place)
        }
        cluster.barrier_wait();
        return ok;
    }
}

// Moves the candidates back to where the general routes expect them (after order_candidates gave up).
__device__ __forceinline__ void order_restore(const OrderBufs &B, u64 *want_km, uint32_t *want_id, uint32_t c)
{
    cg::cluster_group cluster = cg::this_cluster();
    if (B.src_km != want_km)
        for (uint32_t i = cluster.block_rank() * OR_THREADS + threadIdx.x; i < c; i += cluster.num_blocks() * OR_THREADS) {
            want_km[i] = __ldcg(B.src_km + i);
            want_id[i] = __ldcg(B.src_id + i);
        }
    __threadfence();
    cluster.sync();
}
