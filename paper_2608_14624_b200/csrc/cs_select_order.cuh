// Ordering the candidates of a select inside one thread-block cluster.
//
// A select ends with c candidates of which the n_out smallest, in ascending order, are the answer.  Sorting them in one SM
// is bound by that SM's shared memory and shuffles (measured: 1,024 keys of 96 bits take 13,600 cycles as a bitonic sort,
// 10,000 as warp sorts merged by binary search, twice that for 2,048).  Two facts make it cheap on a cluster: a key's place in
// the output is the number of smaller keys, so keys can be placed without being moved; and keys that fall into ranges of
// their own never have to be compared with each other.  So every CTA (few candidates) or every warp (many) takes one range,
// chosen from the ranks of a sample, and counts.  Four instructions per comparison: a 96-bit subtraction whose borrow is
// added up.
//
//   order_small   c <= OR_LIST: every CTA reads all candidates out of the cluster's shared memory, keeps the range that is
//                 its share of the output, counts.
//   order_global  more: the candidates are in global memory.  A sample of 512 or 1,024 is ranked by the whole cluster; what
//                 lies beyond the output's share of it is dropped; the rest goes to up to 256 buckets kept in the cluster's
//                 shared memory, one range each, whose keys are counted by the warps of the bucket's CTA, 32 at a time.
//
// Keys are unique (the id is part of the key): the output does not depend on the order in which atomics were served, nor on
// the sample.
#pragma once
#include <cooperative_groups.h>

#include "cs_select_common.cuh"

namespace cg = cooperative_groups;

#define OR_THREADS 512u
#define OR_WARPS (OR_THREADS / 32u)
#define OR_MAX_CLUSTER 16u
#define OR_LIST 4096u             // keys a CTA keeps for the others to read; candidates order_small takes
#define OR_REGION 6144u           // keys of a CTA's buckets
#define OR_BUCKETS 256u
#define OR_SAMPLE 1024u           // largest sample of order_global
#define OR_GATHER 2048u           // keys of a range that order_small gathers
#define OR_SMALL_SAMPLE 128u

typedef unsigned long long u64_key;

struct OrderSmem {
    u64_key *list_km;             // [list_cap] this CTA's candidates; the count is misc[OM_LIST]
    u64_key *reg_km;              // [reg_cap] everybody's candidates (order_small), this CTA's buckets (order_global)
    u64_key *g_km;                // [OR_GATHER] the sample, unsorted and sorted; the keys of a range
    uint32_t *list_id, *reg_id, *g_id;
    uint32_t *cnt;                // [OR_BUCKETS] fill of this CTA's buckets
    uint32_t *off;                // [OR_BUCKETS + 1]
    uint32_t *part;               // [64] scan scratch
    uint32_t *misc;               // [OM_WORDS]
    uint32_t list_cap, reg_cap;
};
enum { OM_B0 = 0, OM_LIST, OM_GLOBAL, OM_BELOW, OM_IN, OM_CTOT, OM_OVERFLOW, OM_BASE = 8, OM_WORDS = 32 };

__host__ __device__ inline size_t order_smem_bytes(uint32_t list_cap, uint32_t reg_cap)
{
    return (size_t)(list_cap + reg_cap + OR_GATHER) * 12 + (OR_BUCKETS + OR_BUCKETS + 4 + 64 + OM_WORDS) * 4;
}

__device__ __forceinline__ void order_carve(unsigned char *base, uint32_t list_cap, uint32_t reg_cap, OrderSmem &O)
{
    O.list_cap = list_cap;
    O.reg_cap = reg_cap;
    O.list_km = (u64_key *)base;
    O.reg_km = O.list_km + list_cap;
    O.g_km = O.reg_km + reg_cap;
    O.list_id = (uint32_t *)(O.g_km + OR_GATHER);
    O.reg_id = O.list_id + list_cap;
    O.g_id = O.reg_id + reg_cap;
    O.cnt = O.g_id + OR_GATHER;
    O.off = O.cnt + OR_BUCKETS;
    O.part = O.off + OR_BUCKETS + 4;
    O.misc = O.part + 64;
}

// -1 where (ka, ia) < (kb, ib), else 0, added to `count` negated: the borrow of a 96-bit subtraction.
__device__ __forceinline__ void count_less(uint32_t &count, u64_key ka, uint32_t ia, u64_key kb, uint32_t ib)
{
    uint32_t r;
    asm("{\n\t.reg .u32 x;\n\tsub.cc.u32 x, %1, %2;\n\tsubc.cc.u32 x, %3, %4;\n\tsubc.cc.u32 x, %5, %6;\n\tsubc.u32 %0, 0, 0;\n\t}"
        : "=r"(r)
        : "r"(ia), "r"(ib), "r"((uint32_t)ka), "r"((uint32_t)kb), "r"((uint32_t)(ka >> 32)), "r"((uint32_t)(kb >> 32)));
    count -= r;
}
__device__ __forceinline__ bool less96(u64_key ka, uint32_t ia, u64_key kb, uint32_t ib)
{
    uint32_t n = 0;
    count_less(n, ka, ia, kb, ib);
    return n != 0;
}

// Ranks m keys against c keys, both in shared memory, and stores the ids at base + rank (below n_out).  Whole CTA; up to
// 32 neighbouring lanes share a key.  The thread that places the last id of the list reports its key.
__device__ __forceinline__ void rank_and_store(const u64_key *km, const uint32_t *id, uint32_t m, const u64_key *all_km,
                                               const uint32_t *all_id, uint32_t c, uint32_t base, uint32_t n_out,
                                               uint32_t *__restrict__ ids_out, u64_key *last_km)
{
    uint32_t parts = 1;
    while (parts < 32u && 2u * parts * m <= OR_THREADS) parts <<= 1;
    const uint32_t sub = threadIdx.x & (parts - 1u), step = OR_THREADS / parts;
    for (uint32_t k0 = 0; k0 < m; k0 += step) {                     // (uniform: whole warps stay in the shuffles)
        const uint32_t k = k0 + threadIdx.x / parts;
        const bool have = k < m;
        const u64_key my = have ? km[k] : 0ull;
        const uint32_t mine = have ? id[k] : 0u;
        uint32_t r = 0;
#pragma unroll 4
        for (uint32_t q = sub; q < c; q += parts) count_less(r, all_km[q], all_id[q], my, mine);
        for (uint32_t d = parts >> 1; d > 0; d >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, d);
        if (have && sub == 0 && base + r < n_out) {
            ids_out[base + r] = mine;
            if (last_km && base + r == n_out - 1) *last_km = my;
        }
    }
}

// The candidates are in the cluster's lists (counts in misc[OM_LIST], at most OR_LIST and reg_cap in all); every CTA of the
// cluster calls, after a cluster barrier, and the cluster meets once more before it returns (the lists may then go).
__device__ __noinline__ void order_small(const OrderSmem &O, uint32_t n_out, uint32_t *__restrict__ ids_out, u64_key *last_km)
{
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (warp == 0) {
        const uint32_t mine = lane < CL ? cluster.map_shared_rank(O.misc, lane)[OM_LIST] : 0u;
        uint32_t incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= d) incl += t;
        }
        if (lane < CL) O.misc[OM_BASE + lane] = incl;              // end of CTA `lane`'s keys in the common order
        if (lane == 0) { O.misc[OM_BELOW] = 0; O.misc[OM_IN] = 0; }
    }
    __syncthreads();
    const uint32_t c = O.misc[OM_BASE + CL - 1];
    const u64_key *all_km = O.reg_km;
    const uint32_t *all_id = O.reg_id;
    if (CL == 1) {
        all_km = O.list_km;
        all_id = O.list_id;
    } else {
        const uint32_t r = warp & (CL - 1u), split = OR_WARPS / CL;
        const uint32_t end = O.misc[OM_BASE + r], beg = r ? O.misc[OM_BASE + r - 1] : 0u;
        const u64_key *src_km = cluster.map_shared_rank(O.list_km, r);
        const uint32_t *src_id = cluster.map_shared_rank(O.list_id, r);
#pragma unroll 4
        for (uint32_t i = (warp / CL) * 32u + lane; i < end - beg; i += 32u * split) {
            O.reg_km[beg + i] = src_km[i];
            O.reg_id[beg + i] = src_id[i];
        }
        __syncthreads();
        cluster.barrier_arrive();                                   // this CTA reads no list any more; waited for at the end
    }
    if ((unsigned long long)c * c <= 32768ull * CL) {
        // few: every CTA places an equal share of the keys, each counted against all of them
        const uint32_t k0 = rank * c / CL, k1 = (rank + 1u) * c / CL;
        rank_and_store(all_km + k0, all_id + k0, k1 - k0, all_km, all_id, c, 0u, n_out, ids_out, last_km);
    } else {
        // a sample of 128, ranked by everybody, splits the output among the CTAs
        u64_key *s_km = O.g_km;
        uint32_t *s_id = O.g_id;
        if (tid < OR_SMALL_SAMPLE) {
            const uint32_t at = (uint32_t)((unsigned long long)tid * c / OR_SMALL_SAMPLE);
            s_km[tid] = all_km[at];
            s_id[tid] = all_id[at];
        }
        __syncthreads();
        {
            const uint32_t s = tid >> 2;
            const u64_key my = s_km[s];
            const uint32_t mine = s_id[s];
            uint32_t r = 0;
#pragma unroll 8
            for (uint32_t q = tid & 3u; q < OR_SMALL_SAMPLE; q += 4u) count_less(r, s_km[q], s_id[q], my, mine);
            r += __shfl_xor_sync(0xFFFFFFFFu, r, 1);
            r += __shfl_xor_sync(0xFFFFFFFFu, r, 2);
            if ((tid & 3u) == 0) { s_km[OR_SMALL_SAMPLE + r] = my; s_id[OR_SMALL_SAMPLE + r] = mine; }
        }
        __syncthreads();
        const u64_key *t_km = s_km + OR_SMALL_SAMPLE;
        const uint32_t *t_id = s_id + OR_SMALL_SAMPLE;
        // sample ranks that cover the output with four standard deviations to spare; should they fall short, the last CTA
        // takes everything above
        const float e = (float)n_out * (float)OR_SMALL_SAMPLE / (float)c;
        const uint32_t want = (uint32_t)(e + 4.0f * sqrtf(e)) + 3u;
        const uint32_t J = want < OR_SMALL_SAMPLE ? want : OR_SMALL_SAMPLE;
        const uint32_t l0 = rank * J / CL, l1 = (rank + 1u) * J / CL;
        const u64_key lo_km = l0 ? t_km[l0 - 1] : 0ull;
        const uint32_t lo_id = l0 ? t_id[l0 - 1] : 0u;
        u64_key hi_km = l1 < OR_SMALL_SAMPLE ? t_km[l1 ? l1 - 1 : 0] : ~0ull;
        uint32_t hi_id = l1 < OR_SMALL_SAMPLE ? t_id[l1 ? l1 - 1 : 0] : 0xFFFFFFFFu;
        const bool empty = l0 == l1 && rank != CL - 1;
        __syncthreads();                                            // (the gather below overwrites the samples)
        u64_key *in_km = O.g_km;
        uint32_t *in_id = O.g_id;
        for (int pass = 0; pass < 2 && !empty; ++pass) {
            uint32_t below = 0;
            for (uint32_t i0 = 0; i0 < c; i0 += OR_THREADS) {
                const uint32_t i = i0 + tid;
                const u64_key km = i < c ? all_km[i] : ~0ull;
                const uint32_t id = i < c ? all_id[i] : 0xFFFFFFFFu;
                const bool lt = i < c && less96(km, id, lo_km, lo_id);
                const bool in = i < c && !lt && less96(km, id, hi_km, hi_id);
                below += lt ? 1u : 0u;
                const uint32_t b = __ballot_sync(0xFFFFFFFFu, in);
                if (b) {
                    uint32_t at = 0;
                    if (lane == 0) at = atomicAdd(&O.misc[OM_IN], __popc(b));
                    at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(b & ((1u << lane) - 1u));
                    if (in && at < OR_GATHER) { in_km[at] = km; in_id[at] = id; }
                }
            }
            below = __reduce_add_sync(0xFFFFFFFFu, below);
            if (lane == 0 && below) atomicAdd(&O.misc[OM_BELOW], below);
            __syncthreads();
            const uint32_t m = O.misc[OM_IN], base = O.misc[OM_BELOW];
            const bool again = rank == CL - 1 && base + m < n_out && (hi_km != ~0ull || hi_id != 0xFFFFFFFFu);
            __syncthreads();
            if (again) {                                            // the sample misjudged: take the rest as well
                hi_km = ~0ull;
                hi_id = 0xFFFFFFFFu;
                if (tid == 0) { O.misc[OM_IN] = 0; O.misc[OM_BELOW] = 0; }
                __syncthreads();
                continue;
            }
            if (base < n_out) {
                if (m <= OR_GATHER) {
                    rank_and_store(in_km, in_id, m, in_km, in_id, m, base, n_out, ids_out, last_km);
                } else {
                    for (uint32_t i = tid; i < c; i += OR_THREADS) {
                        const u64_key km = all_km[i];
                        const uint32_t id = all_id[i];
                        if (less96(km, id, lo_km, lo_id) || !less96(km, id, hi_km, hi_id)) continue;
                        uint32_t r = 0;
                        for (uint32_t q = 0; q < c; ++q) count_less(r, all_km[q], all_id[q], km, id);
                        if (r < n_out) {
                            ids_out[r] = id;
                            if (last_km && r == n_out - 1) *last_km = km;
                        }
                    }
                }
            }
            break;
        }
    }
    if (CL > 1) cluster.barrier_wait();
}

// What order_global reports to its caller.
struct OrderResult {
    bool done;                // false: too many keys for the cluster's buckets (nothing was stored)
    uint32_t kept;            // candidates that were left after the cut
};

// Key at position i of the candidates: in global memory (lists == false), else in the cluster's lists (ends in misc[OM_BASE..]).
__device__ __forceinline__ void order_fetch(const OrderSmem &O, cg::cluster_group &cluster, uint32_t CL, bool lists,
                                            const u64_key *__restrict__ g_km, const uint32_t *__restrict__ g_id, uint32_t i, u64_key &km,
                                            uint32_t &id)
{
    if (!lists) { km = __ldcg(g_km + i); id = __ldcg(g_id + i); return; }
    uint32_t r = 0;
    while (r + 1 < CL && i >= O.misc[OM_BASE + r]) ++r;
    const uint32_t at = i - (r ? O.misc[OM_BASE + r - 1] : 0u);
    km = cluster.map_shared_rank(O.list_km, r)[at];
    id = cluster.map_shared_rank(O.list_id, r)[at];
}

// c > 0 candidates in global memory, n_out > 0.  Every CTA of the cluster calls; the writes of the candidates are visible.
// sel_T (may be null): receives the key up to which about `ahead` candidates lie, ~0 when that is all of them.
__device__ __noinline__ OrderResult order_global(const OrderSmem &O, const u64_key *__restrict__ g_km, const uint32_t *__restrict__ g_id,
                                                 uint32_t c, uint32_t n_out, uint32_t *__restrict__ ids_out, u64_key *last_km,
                                                 uint32_t ahead, u64_key *sel_T, uint32_t region_max)
{
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    bool lists = false;                                             // where the candidates are
    uint32_t n_list = 0;
    u64_key cut_km = ~0ull;
    uint32_t cut_id = 0xFFFFFFFFu;
    u64_key *s_km = O.g_km, *t_km = O.g_km + OR_SAMPLE;             // the sample, and the same in ascending order
    uint32_t *s_id = O.g_id, *t_id = O.g_id + OR_SAMPLE;
    if (sel_T && rank == 0 && tid == 0 && c <= ahead) *sel_T = ~0ull;
    bool first = true;
    for (;;) {
        uint32_t S = 0, J = 0;
        const bool sampled = c > OR_LIST || c > O.reg_cap;
        if (sampled) {
            // ---- a sample, ranked by the cluster: CL lanes share a key and each hands it to one CTA -----------------------
            S = c <= 12288u ? OR_SAMPLE / 2 : OR_SAMPLE;
            for (uint32_t s = tid; s < S; s += OR_THREADS)
                order_fetch(O, cluster, CL, lists, g_km, g_id, (uint32_t)((unsigned long long)s * c / S), s_km[s], s_id[s]);
            __syncthreads();
            for (uint32_t s0 = rank * (S / CL); s0 < (rank + 1u) * (S / CL); s0 += OR_THREADS / CL) {
                const uint32_t s = s0 + tid / CL, sub = tid & (CL - 1u);
                const u64_key my = s_km[s];
                const uint32_t mine = s_id[s];
                uint32_t r = 0;
#pragma unroll 8
                for (uint32_t q = sub; q < S; q += CL) count_less(r, s_km[q], s_id[q], my, mine);
                for (uint32_t d = CL >> 1; d > 0; d >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, d);
                cluster.map_shared_rank(t_km, sub)[r] = my;
                cluster.map_shared_rank(t_id, sub)[r] = mine;
            }
            if (tid < OR_BUCKETS) O.cnt[tid] = 0;
            if (tid == 0) O.misc[OM_OVERFLOW] = 0;
            cluster.sync();
            const float e = (float)n_out * (float)S / (float)c;
            const uint32_t want = (uint32_t)(e + 4.0f * sqrtf(e)) + 3u;
            J = want < S ? want : S;                                // sample ranks that cover the output
            if (first && sel_T && rank == 0 && tid == 0 && c > ahead) {
                const uint32_t at = (uint32_t)((unsigned long long)ahead * S / c);
                *sel_T = t_km[at < S ? at : S - 1u];
            }
            cut_km = J < S ? t_km[J - 1] : ~0ull;
            cut_id = J < S ? t_id[J - 1] : 0xFFFFFFFFu;
        }
        const bool drop = !sampled || J < 3u * S / 4u || J < 96u;
        // ---- into the lists: everything when it is little, what lies below the cut when that is well below c -------------
        if (!lists || drop) {
            u64_key *keep_km = lists ? O.reg_km : O.list_km;        // (a second round keeps a copy, the others read the lists)
            uint32_t *keep_id = lists ? O.reg_id : O.list_id;
            const uint32_t keep_cap = lists ? O.reg_cap : O.list_cap;
            if (tid == 0) { O.misc[OM_IN] = 0; }
            __syncthreads();
            const uint32_t beg = lists ? 0u : (uint32_t)((unsigned long long)rank * c / CL);
            const uint32_t end = lists ? n_list : (uint32_t)((unsigned long long)(rank + 1u) * c / CL);
            for (uint32_t i0 = beg; i0 < end; i0 += 4u * OR_THREADS) {
                u64_key km[4];
                uint32_t id[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t i = i0 + u * OR_THREADS + tid;
                    km[u] = ~0ull;
                    id[u] = 0xFFFFFFFFu;
                    if (i < end) {
                        km[u] = lists ? O.list_km[i] : __ldcg(g_km + i);
                        id[u] = lists ? O.list_id[i] : __ldcg(g_id + i);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t i = i0 + u * OR_THREADS + tid;
                    const bool in = i < end && (!sampled || J == S || less96(km[u], id[u], cut_km, cut_id));
                    const uint32_t b = __ballot_sync(0xFFFFFFFFu, in);
                    if (!b) continue;
                    uint32_t at = 0;
                    if (lane == 0) at = atomicAdd(&O.misc[OM_IN], __popc(b));
                    at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(b & ((1u << lane) - 1u));
                    if (in && at < keep_cap) { keep_km[at] = km[u]; keep_id[at] = id[u]; }
                }
            }
            __syncthreads();
            n_list = O.misc[OM_IN];
            if (lists) {
                cluster.sync();                                     // nobody reads the old list any more
                for (uint32_t i = tid; i < n_list; i += OR_THREADS) { O.list_km[i] = O.reg_km[i]; O.list_id[i] = O.reg_id[i]; }
            }
            if (tid == 0) O.misc[OM_LIST] = n_list;
            cluster.sync();
            uint32_t total = 0;
            bool fits = true;
            for (uint32_t r = 0; r < CL; ++r) {
                const uint32_t n_r = cluster.map_shared_rank(O.misc, r)[OM_LIST];
                total += n_r;
                fits = fits && n_r <= O.list_cap;
                if (tid == 0) O.misc[OM_BASE + r] = total;
            }
            __syncthreads();
            cluster.sync();                                         // (misc[] is read by everybody before it changes again)
            if (!fits || (total < n_out && sampled)) return OrderResult{false, total};   // (or the sample misjudged: very rare)
            lists = true;
            c = total;
        }
        first = false;
        if (c <= OR_LIST && c <= O.reg_cap) {
            order_small(O, n_out, ids_out, last_km);
            return OrderResult{true, c};
        }
        if (sampled && J >= 96u) {
            // ---- buckets: one range of the sample each, bucket b in the shared memory of CTA b % CL --------------------------
            const uint32_t nb = J < OR_BUCKETS ? J : OR_BUCKETS, per = (nb + CL - 1u) / CL;
            uint32_t cap = O.reg_cap / per;
            if (region_max && cap > region_max) cap = region_max;
            for (uint32_t i = tid; i < n_list; i += OR_THREADS) {
                const u64_key km = O.list_km[i];
                const uint32_t id = O.list_id[i];
                if (J < S && !less96(km, id, cut_km, cut_id)) continue;
                uint32_t b = 0;                                     // splitters at or below the key; splitter j = sample rank (j + 1) J / nb
#pragma unroll 1
                for (uint32_t step = OR_BUCKETS / 2; step > 0; step >>= 1) {
                    const uint32_t j = b + step;                    // 1-based
                    if (j < nb) {
                        const uint32_t at = j * J / nb;
                        if (!less96(km, id, t_km[at], t_id[at])) b = j;
                    }
                }
                const uint32_t slot = atomicAdd(cluster.map_shared_rank(O.cnt, b & (CL - 1u)) + b / CL, 1u);
                if (slot < cap) {
                    cluster.map_shared_rank(O.reg_km, b & (CL - 1u))[(b / CL) * cap + slot] = km;
                    cluster.map_shared_rank(O.reg_id, b & (CL - 1u))[(b / CL) * cap + slot] = id;
                } else {
                    cluster.map_shared_rank(O.misc, 0)[OM_OVERFLOW] = 1u;
                }
            }
            cluster.sync();
            const uint32_t over = cluster.map_shared_rank(O.misc, 0)[OM_OVERFLOW];
            const uint32_t mine = tid < nb ? cluster.map_shared_rank(O.cnt, tid & (CL - 1u))[tid / CL] : 0u;
            uint32_t total;
            const uint32_t excl = sel_block_scan(mine, O.part, total, whole_cta());
            if (tid < nb) O.off[tid] = excl;
            cluster.barrier_arrive();                               // remote reads done; waited for at the end
            __syncthreads();
            const bool ok = !over && total >= n_out;
            if (ok) {
                // work items of 32 keys of a bucket, dealt to the warps in turn
                uint32_t item = 0;
                for (uint32_t lb = 0; lb < per; ++lb) {
                    const uint32_t b = lb * CL + rank;
                    if (b >= nb || O.off[b] >= n_out) break;        // (offsets grow with b)
                    const uint32_t m = O.cnt[lb], base = O.off[b];
                    const u64_key *b_km = O.reg_km + (size_t)lb * cap;
                    const uint32_t *b_id = O.reg_id + (size_t)lb * cap;
                    for (uint32_t k0 = 0; k0 < m; k0 += 32u, ++item) {
                        if ((item & (OR_WARPS - 1u)) != warp) continue;
                        const uint32_t k = k0 + lane;
                        const u64_key my = k < m ? b_km[k] : 0ull;
                        const uint32_t my_id = k < m ? b_id[k] : 0u;
                        uint32_t r = 0;
#pragma unroll 4
                        for (uint32_t q = 0; q < m; ++q) count_less(r, b_km[q], b_id[q], my, my_id);
                        if (k < m && base + r < n_out) {
                            ids_out[base + r] = my_id;
                            if (last_km && base + r == n_out - 1) *last_km = my;
                        }
                    }
                }
            }
            cluster.barrier_wait();
            return OrderResult{ok, total};
        }
        // few of the sample below the cut: the lists are far shorter than the candidates were, sample them again
    }
}
