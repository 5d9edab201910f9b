// Single-launch select: the whole top-k (histogram -> threshold -> collect -> order) inside ONE
// thread-block cluster, for index sizes where a handful of SMs can stream the metadata in a few
// microseconds (every configuration of this library's workloads).  It occupies at most 16 SMs per select, which
// leaves the rest of the GPU to the serving kernels.  Same key, same eligibility rules, same exact ordered output as
// the grid-wide kernels of cs_select.cu.
//
// Phases, between hardware cluster barriers (no spin-waits of our own; a cluster of one CTA has none):
//   1 every CTA computes the keys of its slice of the index -- up to 16 per thread, which stay in registers when the slice
//     is no larger -- and counts them in a 4096-bin histogram of the primary key in its shared memory.  The bins divide the
//     range that scores can have, not the 32 bits of the key: a bin is 1/128 of an octave instead of 1/8;
//   2 CTA r sums bins [r*B/CL, (r+1)*B/CL) over all CTAs through DSMEM and writes the sums into
//     every CTA's copy of the total histogram; each CTA then finds the threshold bin b0;
//   3 the entries with bin <= b0 (c >= min(k, eligible) keys) go to the candidate buffer (a single CTA keeps them in shared
//     memory);
//   4 they are put in order (cs_select_order.cuh); where buckets overflow there, by a sample sort through global memory.
//
// Bound by latency: trips to L2, barriers, and the instructions of one warp's entries.  The three selects of
// a step, back to back in a CUDA graph: 2,560 entries, k = 32 / 64: 26.8 us when the index was scanned twice, bins were an
// eighth of an octave and one CTA sorted the candidates, 6.6 us like this; 80,000 entries, k = 256 / 384: 32.2 -> 12.3 us.
#include "cs_select_order.cuh"

#define CSEL_THREADS OR_THREADS
#define CSEL_MAX_CLUSTER 16
#define CSEL_UNIT 128u            // entries of a warp's step: four per lane
#define CSEL_UNITS 4              // units a warp holds in registers
static_assert(2 * CS_HIST_BINS * 4 <= 48 * 1024, "histograms");

__host__ __device__ inline size_t csel_table_bytes(uint32_t A, uint32_t gtab_len)
{
    return (((size_t)(A + gtab_len + 1) * 4 + (size_t)A * 2) + 15) / 16 * 16;
}
// Candidates a CTA holds at once: no more than the index has entries.
static uint32_t csel_cap(uint32_t n)
{
    return n < 256u ? 256u : (n < OR_ALL ? (n + 255u) / 256u * 256u : OR_ALL);
}
static size_t csel_smem_bytes(uint32_t A, uint32_t gtab_len, uint32_t n)
{
    return csel_table_bytes(A, gtab_len) + 2 * CS_HIST_BINS * 4 + order_smem_bytes(csel_cap(n));
}

// Four consecutive entries per lane, as they come from memory.
struct Quad {
    uint4 la;
    uint2 ag, dp;
    uint32_t rf, fl, tk;
};
template <bool PF>
__device__ __forceinline__ void load_quad(const SelArgs &a, uint32_t q, Quad &Q)
{
    Q.la = __ldg((const uint4 *)a.la + q);
    Q.ag = __ldg((const uint2 *)a.agent + q);
    Q.rf = __ldg((const uint32_t *)a.ref + q);
    Q.fl = __ldg((const uint32_t *)a.flags + q);
    Q.tk = a.ntok ? __ldg((const uint32_t *)a.ntok + q) : 0u;
    Q.dp = make_uint2(0u, 0u);
    if (PF && a.anchor) Q.dp = __ldg((const uint2 *)a.depth + q);
}

// Ordering through global memory, for candidates the cluster's buckets cannot hold: a 1,024-key sample is sorted, every
// candidate finds its bucket, the needed buckets are grouped and each is sorted in shared memory (a padded bucket has room there: more
// candidates than O.cap come here, and O.cap is then OR_ALL, a power of two).
__device__ __noinline__ void csel_order_general(const cs_workspace &ws, const OrderSmem &O, uint32_t c, uint32_t n_out,
                                                uint32_t *__restrict__ ids_out)
{
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank(), tid = threadIdx.x;
    const uint32_t cthreads = CL * CSEL_THREADS, ctid = rank * CSEL_THREADS + tid;
    u64 *km_s = O.s_km;
    uint32_t *id_s = O.s_id;
    uint32_t *s_off = O.off;
    cluster.sync();
    if (rank == 0) {
        for (uint32_t i = tid; i < CS_SAMPLE; i += CSEL_THREADS) {
            const uint32_t pos = (uint32_t)(((unsigned long long)i * c) / CS_SAMPLE);
            km_s[i] = __ldcg(&ws.cand_km[pos]);
            id_s[i] = __ldcg(&ws.cand_id[pos]);
        }
        __syncthreads();
        bitonic_sort_fast(km_s, id_s, CS_SAMPLE);
        // buckets of about 384 keys, which a CTA sorts in little more time than 128, but a bucket for every CTA at least
        const uint32_t n_spl = min(CS_MAX_SPLITTERS, max(c / 384u, CL));
        for (uint32_t j = tid; j <= CS_MAX_SPLITTERS; j += CSEL_THREADS) {
            if (j < CS_MAX_SPLITTERS) {
                const uint32_t q = (j + 1u) * CS_SAMPLE / (n_spl + 1u);
                ws.spl_km[j] = j < n_spl ? km_s[q] : ~0ull;      // (behind every key: the buckets beyond stay empty)
                ws.spl_id[j] = j < n_spl ? id_s[q] : 0xFFFFFFFFu;
            }
            CS_BCOUNT(ws, j) = 0;
        }
    }
    __threadfence();
    cluster.sync();
    for (uint32_t j = tid; j < CS_MAX_SPLITTERS; j += CSEL_THREADS) { km_s[j] = __ldcg(&ws.spl_km[j]); id_s[j] = __ldcg(&ws.spl_id[j]); }
    if (tid == 0) O.misc[OM_IN] = 0;
    __syncthreads();
    for (uint32_t i = ctid; i < c; i += cthreads) {
        const u64 km = __ldcg(&ws.cand_km[i]);
        const uint32_t id = __ldcg(&ws.cand_id[i]);
        uint32_t lo = 0, hi = CS_MAX_SPLITTERS;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (key_less(km, id, km_s[mid], id_s[mid])) hi = mid;
            else lo = mid + 1;
        }
        ws.cand_bkt[i] = lo;
        ws.cand_slot[i] = atomicAdd(&CS_BCOUNT(ws, lo), 1u);
    }
    __threadfence();
    cluster.sync();
    // offsets (every CTA computes the same prefix sum), then scatter the needed buckets into bucket order
    const uint32_t mine = tid <= CS_MAX_SPLITTERS ? __ldcg(&CS_BCOUNT(ws, tid)) : 0u;
    uint32_t total;
    const uint32_t excl = sel_block_scan(mine, O.part, total);
    if (tid <= CS_MAX_SPLITTERS) s_off[tid] = excl;
    if (tid == CS_MAX_SPLITTERS) s_off[CS_MAX_SPLITTERS + 1] = excl + mine;
    if (mine && excl <= n_out - 1 && n_out - 1 < excl + mine) O.misc[OM_IN] = tid;     // last needed bucket (n_out > 0 here)
    __syncthreads();
    const uint32_t b_last = O.misc[OM_IN];
    for (uint32_t i = ctid; i < c; i += cthreads) {
        const uint32_t b = __ldcg(&ws.cand_bkt[i]);
        if (b > b_last) continue;
        const uint32_t pos = s_off[b] + __ldcg(&ws.cand_slot[i]);
        ws.sort_km[pos] = __ldcg(&ws.cand_km[i]);
        ws.sort_id[pos] = __ldcg(&ws.cand_id[i]);
    }
    __threadfence();
    cluster.sync();
    for (uint32_t b = rank; b <= b_last; b += CL) {
        const uint32_t beg = s_off[b], m = s_off[b + 1] - beg;
        __syncthreads();
        if (m <= O.cap) {
            uint32_t P = 64;
            while (P < m) P <<= 1;
            for (uint32_t i = tid; i < P; i += CSEL_THREADS) {
                O.all_km[i] = i < m ? __ldcg(&ws.sort_km[beg + i]) : ~0ull;
                O.all_id[i] = i < m ? __ldcg(&ws.sort_id[beg + i]) : 0xFFFFFFFFu;
            }
            __syncthreads();
            if (P <= 2u * CSEL_THREADS) bitonic_sort_fast(O.all_km, O.all_id, P);
            else sort_tile(O.all_km, O.all_id, P);
            for (uint32_t i = tid; i < m; i += CSEL_THREADS)
                if (beg + i < n_out) ids_out[beg + i] = O.all_id[i];
        } else {                                     // more than shared memory holds
            uint32_t *list = ws.cand_bkt + beg;      // (the candidates' buckets are no longer wanted; nobody else's part of the array)
            for (uint32_t i = tid; i < m; i += CSEL_THREADS) list[i] = i;
            __syncthreads();
            sort_places(list, m, ws.sort_km + beg, ws.sort_id + beg);
            for (uint32_t i = tid; i < m && beg + i < n_out; i += CSEL_THREADS) ids_out[beg + i] = __ldcg(&ws.sort_id[beg + __ldcg(list + i)]);
        }
    }
}

// One whole select by the calling cluster.  `ws` carries this select's private candidate / sort regions, so several
// clusters of one launch can run different selects at once.
template <bool PF>
__device__ __forceinline__ void csel_body(SelArgs a, const cs_workspace &ws, uint32_t *__restrict__ ids_out,
                                          uint32_t *__restrict__ n_out_dev, unsigned char *dsm, uint32_t cap)
{
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t CL = cluster.num_blocks(), rank = cluster.block_rank();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int PS = PF ? 8 : 0;                                // phase-stamp slots (profiling builds)
    const bool stamp = rank == 0 && tid == 0;
    (void)PS;
    (void)stamp;
    CS_STAMP(ws, CS_PS_SCAN_ENTRY + PS, stamp);
    OrderSmem O;
    uint32_t *hist = (uint32_t *)(dsm + csel_table_bytes(a.A, a.gtab_len));       // [4096] this CTA's histogram
    uint32_t *tot = hist + CS_HIST_BINS;                                          // [4096] the cluster's (same in every CTA)
    order_carve((unsigned char *)(tot + CS_HIST_BINS), cap, O);
    Tables T;
    load_tables_static(a, ws, (float *)dsm, T);
    // the table covers every age before saturation: one entry more stands for all the others
    T.anchor += 2;
    const bool whole_table = a.gtab_len == a.age_sat;
    if (tid == 0) T.gtab[a.gtab_len] = T.g_sat;
    for (uint32_t i = tid; i < CS_HIST_BINS / 4; i += CSEL_THREADS) ((uint4 *)hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < OM_WORDS) O.misc[tid] = 0;
    CS_STAMP(ws, CS_PS_SCAN_SETUP + PS, stamp);
    cs_wait_for_predecessor();
    cs_release_successor();
    CS_STAMP(ws, CS_PS_SCAN_WAITED + PS, stamp);
    resolve_now(a);
    // the first pass's loads travel with the tables'
    const uint32_t n_units = a.n / CSEL_UNIT, n_warps = CL * OR_WARPS, gw = rank * OR_WARPS + warp;
    const uint32_t pass_units = n_warps * CSEL_UNITS;
    const bool one_pass = n_units <= pass_units;                  // the keys stay in registers between the two scans
    Quad Q[CSEL_UNITS];
    auto load_pass = [&](uint32_t u0) {
#pragma unroll
        for (int q = 0; q < CSEL_UNITS; ++q) {
            const uint32_t u = u0 + q * n_warps + gw;
            if (u < n_units) load_quad<PF>(a, u * 32u + lane, Q[q]);
        }
    };
    load_pass(0u);
    const uint32_t t0 = n_units * CSEL_UNIT, ctid = rank * CSEL_THREADS + tid;     // the ragged tail: one entry per thread
    bool tail = ctid < a.n - t0;
    const uint32_t tail_id = t0 + ctid;
    uint32_t tail_pr = 0, tail_se = 0, tl_ag = 0, tl_dp = 0, tl_rf = 0, tl_fl = 0, tl_la = 0, tl_tk = a.block_tokens;
    if (tail) {
        tl_ag = __ldg(a.agent + tail_id);
        if (PF && a.anchor) tl_dp = __ldg(a.depth + tail_id);    // (a caller without workspace vouches for no depth array)
        tl_rf = __ldg(a.ref + tail_id);
        tl_fl = __ldg(a.flags + tail_id);
        tl_la = __ldg(a.la + tail_id);
        if (a.ntok) tl_tk = __ldg(a.ntok + tail_id);
    }
    load_tables_dynamic(a, ws, T, PF && a.anchor);
    const bool enabled = !PF || prefetch_enabled(ws, a.A);
    __syncthreads();
    tail = tail && enabled && entry_key<PF>(a, T, &ws.sc->status, tl_ag, tl_dp, tl_rf, tl_fl, tl_la, tl_tk, tail_pr, tail_se);
    uint32_t pr[4 * CSEL_UNITS], em = 0;                          // primary keys; bit 4 q + r: entry r of unit q is eligible
    uint32_t b0 = 0xFFFFFFFFu, n_out = 0, c = 0;
    // candidates: in shared memory when one CTA is all there is and they fit, else in L2, numbered by the first CTA
    uint32_t *counter = cluster.map_shared_rank(O.misc, 0) + OM_LIST;
    u64 *to_km = ws.cand_km;
    uint32_t *to_id = ws.cand_id;
    bool here = false;
#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase) {
        // phase 0 counts the keys, phase 1 puts those at or below the threshold bin away
#pragma unroll 1
        for (uint32_t u0 = 0; u0 < n_units && enabled; u0 += pass_units) {
            if (phase == 0 || !one_pass) {
                if (phase || u0) load_pass(u0);
                em = 0;
#pragma unroll
                for (int q = 0; q < CSEL_UNITS; ++q) {
                    if (u0 + q * n_warps + gw >= n_units) break;
                    const uint32_t fmask = PF ? 0x0F0F0F0Fu : 0x07070707u;
                    const uint32_t fpat = PF ? 0x05050505u : (0x01010101u * (CS_FLAG_VALID | (a.tier << 2)));
                    uint32_t ok = nibble_of_flags(zero_bytes(((Q[q].fl & fmask) ^ fpat) | Q[q].rf));
                    if (!__any_sync(0xFFFFFFFFu, ok != 0u)) continue;
                    // the four keys side by side, without a branch: an entry that is not eligible gets one nobody looks at
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const uint32_t ag = ((r < 2 ? Q[q].ag.x : Q[q].ag.y) >> ((r & 1) * 16)) & 0xFFFFu;
                        const uint32_t agc = ag < a.A ? ag : 0u;
                        if (ag >= a.A && ((ok >> r) & 1u)) {
                            atomicOr(&ws.sc->status, CS_ST_BAD_AGENT);
                            ok &= ~(1u << r);
                        }
                        if (PF && a.anchor) {
                            const uint32_t dp = ((r < 2 ? Q[q].dp.x : Q[q].dp.y) >> ((r & 1) * 16)) & 0xFFFFu;
                            ok &= ~((dp < T.anchor[agc] ? 0u : 1u) << r);
                        }
                        const uint32_t tok = a.ntok ? (Q[q].tk >> (8 * r)) & 0xFFu : a.block_tokens, la = u4_word(Q[q].la, r);
                        const uint32_t age = max(a.now, la) - la;
                        float g;
                        if (whole_table) g = T.gtab[min(age, a.gtab_len)];             // (its last entry is the saturated factor)
                        else g = recency_of_age(a, T, age);
                        const uint32_t bits = __float_as_uint(__fmul_rn(__fmul_rn(T.fsurv[agc], g), (float)tok));
                        if (PF) pr[4 * q + r] = (agc == T.a_star ? 0u : 0x80000000u) | (~bits & 0x7FFFFFFFu);
                        else pr[4 * q + r] = a.prefer_copy ? ((bits << 1) | ((Q[q].fl >> (8 * r + 3)) & 1u ^ 1u)) : bits;
                    }
                    em |= ok << (4 * q);
                    if (phase == 0) {
#pragma unroll
                        for (int r = 0; r < 4; ++r)
                            if ((ok >> r) & 1u) atomicAdd(&hist[bin_of<PF>(a, pr[4 * q + r])], 1u);
                    }
                }
            }
            if (phase == 0) continue;
            uint32_t mask = 0;
#pragma unroll
            for (int e = 0; e < 4 * CSEL_UNITS; ++e)
                if (((em >> e) & 1u) && bin_of<PF>(a, pr[e]) <= b0) mask |= 1u << e;
            const uint32_t cnt = __popc(mask);
            uint32_t incl = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if (lane >= d) incl += v;
            }
            uint32_t base = 0;
            if (lane == 31 && incl) base = atomicAdd(counter, incl);
            uint32_t pos = __shfl_sync(0xFFFFFFFFu, base, 31) + incl - cnt;
#pragma unroll
            for (int e = 0; e < 4 * CSEL_UNITS; ++e) {
                if (!((mask >> e) & 1u)) continue;
                const uint32_t la = u4_word(Q[e >> 2].la, e & 3);
                to_km[pos] = ((u64)pr[e] << 32) | (PF ? ~la : la);
                to_id[pos] = (u0 + (uint32_t)(e >> 2) * n_warps + gw) * CSEL_UNIT + 4u * lane + (uint32_t)(e & 3);
                ++pos;
            }
        }
        if (phase) break;
        if (tail) atomicAdd(&hist[bin_of<PF>(a, tail_pr)], 1u);
        CS_STAMP(ws, CS_PS_SCAN_READ + PS, stamp);
        // ---- reduce the histograms through DSMEM, broadcast, find the threshold bin ---------------------------------------
        const uint32_t *sums = hist;
        if (CL > 1) {
            cluster.sync();
            const uint32_t per = CS_HIST_BINS / CL;                 // CL is a power of two <= 16
            for (uint32_t b = tid; b < per; b += CSEL_THREADS) {
                const uint32_t bin = rank * per + b;
                uint32_t sum = 0;
#pragma unroll 8
                for (uint32_t q = 0; q < CL; ++q) sum += cluster.map_shared_rank(hist, q)[bin];
#pragma unroll 8
                for (uint32_t q = 0; q < CL; ++q) cluster.map_shared_rank(tot, q)[bin] = sum;
            }
            cluster.sync();
            sums = tot;
        } else {
            __syncthreads();
        }
        CS_STAMP(ws, CS_PS_SCAN_FLUSHED + PS, stamp);
        constexpr uint32_t PER = CS_HIST_BINS / CSEL_THREADS;
        uint32_t loc[PER], sum = 0;
#pragma unroll
        for (uint32_t q = 0; q < PER / 4; ++q) {
            const uint4 v = ((const uint4 *)sums)[tid * (PER / 4) + q];
            loc[4 * q] = v.x; loc[4 * q + 1] = v.y; loc[4 * q + 2] = v.z; loc[4 * q + 3] = v.w;
            sum += v.x + v.y + v.z + v.w;
        }
        uint32_t n_elig;
        const uint32_t before = sel_block_scan(sum, O.part, n_elig);
        n_out = n_elig < a.k ? n_elig : a.k;
        if (a.k && n_elig >= a.k && before < a.k && a.k <= before + sum) {
            uint32_t run = before;
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                run += loc[q];
                if (run >= a.k) { O.misc[OM_B0] = tid * PER + q; O.misc[OM_CTOT] = run; break; }
            }
        }
        __syncthreads();
        if (n_elig >= a.k) { b0 = O.misc[OM_B0]; c = O.misc[OM_CTOT]; }
        else { b0 = CS_HIST_BINS - 1u; c = n_elig; }                // fewer than k: everything
        // the tail of the list is known now: pad it while the candidates are being collected
        for (uint32_t i = n_out + ctid; i < a.k; i += CL * CSEL_THREADS) ids_out[i] = CS_ID_NONE;
        if (ctid == 0) {
            *n_out_dev = n_out;
            count_select(ws, a.kind, n_elig, n_out);
            count_candidates(ws, a.kind, n_out ? c : 0u, false);
        }
        if (n_out == 0) return;                                     // nothing eligible or nothing asked for (same in every CTA)
        here = CL == 1 && c <= cap;
        if (here) { to_km = O.all_km; to_id = O.all_id; }
    }
    if (tail && bin_of<PF>(a, tail_pr) <= b0) {
        const uint32_t pos = atomicAdd(counter, 1u);
        to_km[pos] = ((u64)tail_pr << 32) | tail_se;
        to_id[pos] = tail_id;
    }
    CS_STAMP(ws, CS_PS_SCAN_LAST_CTA + PS, stamp);
    if (here) {
        __syncthreads();
        order_few(O, nullptr, nullptr, c, n_out, ids_out);
    } else {
        __threadfence();
        cluster.sync();
        OrderBufs B = order_bufs(ws, a.max_blocks);
        if (!order_candidates(O, B, c, n_out, ids_out)) {
            order_restore(B, ws.cand_km, ws.cand_id, c);
            csel_order_general(ws, O, c, n_out, ids_out);
        }
    }
    CS_STAMP(ws, CS_PS_SCAN_TAIL_DONE + PS, stamp);
}

template <bool PF>
__global__ void __launch_bounds__(CSEL_THREADS, 1)
cs_select_cluster_kernel(SelArgs a, cs_workspace ws, uint32_t *__restrict__ ids_out, uint32_t *__restrict__ n_out_dev, uint32_t cap)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    csel_body<PF>(a, ws, ids_out, n_out_dev, dsm, cap);
}

// The three selects of a step in one launch: cluster q of the grid runs select q (GPU-tier victims,
// host-tier victims, prefetch candidates).  The selects share the index and the tables and nothing else.
struct SelJob {
    SelArgs a;
    cs_workspace ws;
    uint32_t *ids_out, *n_out;
    uint32_t prefetch;
};
struct SelJobs { SelJob j[3]; uint32_t cap; };     // the grid holds one cluster per job in use

__global__ void __launch_bounds__(CSEL_THREADS, 1) cs_select_step_kernel(const __grid_constant__ SelJobs jobs)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    const uint32_t q = blockIdx.x / cg::this_cluster().num_blocks();
    const SelJob &J = jobs.j[q];
    if (J.prefetch) csel_body<true>(J.a, J.ws, J.ids_out, J.n_out, dsm, jobs.cap);
    else csel_body<false>(J.a, J.ws, J.ids_out, J.n_out, dsm, jobs.cap);
}

// ---------------------------------------------------------------------------------------------
// Per-device set-up of the cluster kernels, done once per process and device.  The dynamic shared-memory
// opt-in is an attribute of the FUNCTION (on a device), not of a context, so it is raised once to the fixed
// maximum any parameter set can ask for (CS_MAX_AGENTS agents, the longest recency table) and never lowered:
// contexts of different shape and the static-scratch entry point can then share the kernels.  The largest
// usable cluster is probed with that same maximum, which makes the answer independent of the caller's sizes.
#include <mutex>

#define CSEL_MAX_DEVICES 64
struct CselDevice {
    int ready;                       // 0 = not set up yet
    int max_v, max_pf, max_step;     // largest usable cluster per kernel (-1 = none)
};
static std::mutex g_csel_mu;
static CselDevice g_csel_dev[CSEL_MAX_DEVICES];

// Returns the device's entry (set up on first use, with `device` current), or nullptr for a device index out of range.
static const CselDevice *csel_device(int device)
{
    if (device < 0 || device >= CSEL_MAX_DEVICES) return nullptr;
    std::lock_guard<std::mutex> lock(g_csel_mu);
    CselDevice &d = g_csel_dev[device];
    if (!d.ready) {
        const size_t smem_max = csel_smem_bytes(CS_MAX_AGENTS, CS_GTAB_MAX, CS_SELECT_CLUSTER_MAX_BLOCKS);
        d.max_v = cs_probe_cluster(cs_select_cluster_kernel<false>, CSEL_MAX_CLUSTER, CSEL_THREADS, smem_max, 1);
        d.max_pf = cs_probe_cluster(cs_select_cluster_kernel<true>, CSEL_MAX_CLUSTER, CSEL_THREADS, smem_max, 1);
        d.max_step = cs_probe_cluster(cs_select_step_kernel, CSEL_MAX_CLUSTER, CSEL_THREADS, smem_max, 3);
        d.ready = 1;
    }
    return &d;
}

// smallest power-of-two cluster whose warps have at most two units of the index each and whose CTAs place at most 64 ids
// of the list, at most max_cl
static int csel_cluster_size(uint32_t n, uint32_t k, int max_cl)
{
    int cl = 1;
    while (cl < max_cl && ((uint32_t)cl * OR_WARPS * 2u * CSEL_UNIT < n || (uint32_t)cl * 64u < k)) cl <<= 1;
    return cl;
}

// A cluster launch; chained to the kernel before it (programmatic dependent launch) unless that kernel writes the recency
// table, which the kernels read ahead of the dependency wait (the static-scratch entry point, the only one with no workspace).
static void csel_config(cs_ctx *ctx, cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int cl, int n_jobs, size_t smem,
                               cudaStream_t s)
{
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = CS_USE_PDL;
    cfg.gridDim = dim3(n_jobs * cl);
    cfg.blockDim = dim3(CSEL_THREADS);
    cfg.dynamicSmemBytes = smem;                                 // <= the opted-in maximum by construction
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->ws_bytes ? 2 : 1;
}

template <bool PF>
static int launch_cluster(cs_ctx *ctx, const SelArgs &a, const cs_workspace &ws, uint32_t *ids_out, uint32_t *n_out,
                          cudaStream_t s)
{
    const CselDevice *d = csel_device(ctx->device);
    const int max_cl = d ? (PF ? d->max_pf : d->max_v) : -1;
    if (max_cl < 1) return CS_ENOTIMPL;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    csel_config(ctx, cfg, attr, csel_cluster_size(a.n, a.k, max_cl), 1, csel_smem_bytes(a.A, a.gtab_len, a.n), s);
    cudaError_t e = cudaLaunchKernelEx(&cfg, cs_select_cluster_kernel<PF>, a, ws, ids_out, n_out, csel_cap(a.n));
    ctx->n_launches++;
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
    return CS_OK;
}

int cs_launch_select_clusters(cs_ctx *ctx, int n_jobs, const void *sel_args, const uint32_t *prefetch,
                              uint32_t *const *ids_out, uint32_t *const *n_out, cudaStream_t s)
{
    const SelArgs *aj = (const SelArgs *)sel_args;
    const CselDevice *d = csel_device(ctx->device);
    const int max_cl = d ? d->max_step : -1;
    if (max_cl < 1) return CS_ENOTIMPL;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    uint32_t k = 0;
    for (int q = 0; q < n_jobs; ++q) k = aj[q].k > k ? aj[q].k : k;
    SelJobs jobs;
    jobs.cap = csel_cap(aj[0].n);
    csel_config(ctx, cfg, attr, csel_cluster_size(aj[0].n, k, max_cl), n_jobs, csel_smem_bytes(aj[0].A, aj[0].gtab_len, aj[0].n), s);
    for (int q = 0; q < n_jobs; ++q) {
        jobs.j[q].a = aj[q];
        jobs.j[q].ws = q == 0 ? ctx->ws : ctx->ws_job[q - 1];
        if (q && !ctx->concurrent_selects) jobs.j[q].a.max_blocks = CS_SELECT_CLUSTER_MAX_BLOCKS;      // (as the workspace is laid out)
        jobs.j[q].ids_out = ids_out[q];
        jobs.j[q].n_out = n_out[q];
        jobs.j[q].prefetch = prefetch[q];
    }
    for (int q = n_jobs; q < 3; ++q) jobs.j[q] = jobs.j[0];          // unused slots: defined contents
    cudaError_t e = cudaLaunchKernelEx(&cfg, cs_select_step_kernel, jobs);
    ctx->n_launches++;
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
    return CS_OK;
}

int cs_launch_select_cluster(cs_ctx *ctx, const void *sel_args, const cs_workspace *ws, int prefetch, uint32_t *ids_out,
                             uint32_t *n_out, cudaStream_t s)
{
    const SelArgs &a = *(const SelArgs *)sel_args;
    return prefetch ? launch_cluster<true>(ctx, a, *ws, ids_out, n_out, s) : launch_cluster<false>(ctx, a, *ws, ids_out, n_out, s);
}
