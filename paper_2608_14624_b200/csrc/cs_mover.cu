// Paged-KV block mover: gathers / scatters whole multi-layer KV blocks between two pools that
// may differ in location (HBM or pinned host memory), slot count and layout.  The paper reuses
// its serving engine's offload path unchanged (Sec. 4); this file is that path for B200.
//
// Unit of work: one "piece" of one chunk (one layer, one plane, one block).  Consecutive work
// items are consecutive pieces, so neighbouring CTAs stream neighbouring addresses.  The slot
// lists and the optional device-resident count come straight from the select kernels' output,
// so no host round trip sits between a decision and its transfer.  Pinned host memory is
// addressed directly by the SMs (unified addressing), which lets both slot lists stay scattered.
//
// Two data paths:
//  * bulk path (default): every warp of a CTA runs its own software pipeline of 1-D bulk
//    asynchronous copies (TMA): global -> shared memory ring (mbarrier completion), shared ->
//    global (bulk groups).  One lane per warp issues; the copy engines of the SM move the
//    bytes, so a handful of CTAs keep hundreds of KiB in flight without occupying the
//    load/store pipelines that co-resident kernels need.
//  * load/store path: 4 x 128-bit loads per thread in flight, streaming cache hints.  Used when
//    asked for (cs_set_mover_path) and as the comparison point in the profiles.
// No copy is multicast and no kernel waits on another CTA; every mbarrier wait is bounded.
#include <mutex>
#include <type_traits>

#include "cs_common.cuh"

#define MV_THREADS 256
#define MV_UNROLL 4
#define MV_PIECE (MV_THREADS * MV_UNROLL * 16)      // bytes per work item of the load/store path

// A pipeline owns a ring of 48 KiB in shared memory, divided into slots of the size of its pieces: with slots of 16 KiB
// only, a chunk of 2 KiB used an eighth of the ring and the transfer waited for memory (64 MB out of a layer-major pool of
// 1 KiB chunks into the host tier 12 -> 50 GB/s, in from it 24 -> 51, both ways 26 -> 79; of 2 KiB chunks 24 -> 52, 44 -> 51,
// 49 -> 79; inside the device 400 blocks of 4 KiB chunks 67 -> 38 us).  Where both pools keep a block together it is one run of bytes whatever
// its chunks.
#define TM_RING 49152u                               // bytes of ring per pipeline
#define TM_WARPS 2                                   // most pipelines per CTA
#define TM_PIECE 16384u                              // largest piece
#define TM_SMEM (TM_WARPS * TM_RING)                 // 96 KiB
#define CS_EXCHANGE_PIPES 32u                         // default width of the two-way transfer, in warp pipelines
#define TM_SPIN_LIMIT (1u << 20)                     // bounded mbarrier wait (polls with back-off: >= 0.1 s)

struct MoverArgs {
    const char *src;
    char *dst;
    uint32_t src_total, dst_total, src_layout, dst_layout, pieces, src_first, dst_first, piece_bytes, n_pipes;
    uint32_t n_chunks;                // runs of bytes of a block: layers x planes, or 1 when both pools keep a block together
    unsigned long long chunk;
    const uint32_t *src_slots, *dst_slots, *n_dev;
    uint32_t n_max;
    uint32_t *status;
    cs_counters *cnt;                 // work counters: blocks and bytes per direction, skipped entries
    uint32_t kind;                    // CS_MOVE_*
    unsigned long long block_bytes;
};

__device__ __forceinline__ unsigned long long chunk_offset(uint32_t layout, uint32_t n_chunks, uint32_t n_slots, uint32_t lp,
                                                           uint32_t s, unsigned long long chunk)
{
    if (layout == CS_LAYER_MAJOR) return ((unsigned long long)lp * n_slots + s) * chunk;
    return ((unsigned long long)s * n_chunks + lp) * chunk;
}

// List entries of work item w: source and destination block id.
__device__ __forceinline__ uint2 fetch_slots(const MoverArgs &a, unsigned long long w, uint32_t per_block)
{
    const uint32_t i = (uint32_t)(w / per_block);
    // a missing list means "packed": entry i is slot i (the staging ring of the copy-engine path)
    return make_uint2(a.src_slots ? __ldg(a.src_slots + i) : i, a.dst_slots ? __ldg(a.dst_slots + i) : i);
}

// Resolves work item w to a source / destination address and a byte count; false = skip.  One piece per block does the block's
// bookkeeping: book = 1 adds it to the work counters, -1 takes it back (a bad slot stays reported: the list does hold it), 0 leaves them.
__device__ __forceinline__ bool resolve_piece(const MoverArgs &a, unsigned long long w, uint32_t per_block, uint2 slots,
                                              const char *&sp, char *&dp, uint32_t &bytes, int book)
{
    const uint32_t i = (uint32_t)(w / per_block);
    const uint32_t r = (uint32_t)(w - (unsigned long long)i * per_block);
    const uint32_t lp = r / a.pieces, piece = r - lp * a.pieces;
    uint32_t s = slots.x, d = slots.y;
    const bool first = book != 0 && r == 0;
    const unsigned long long one = (unsigned long long)(long long)book;
    if (s == CS_ID_NONE || d == CS_ID_NONE) {
        if (first) atomicAdd((unsigned long long *)&a.cnt->blocks_skipped, one);
        return false;
    }
    s -= a.src_first;                                   // ids below first_id wrap and fail the range check
    d -= a.dst_first;
    if (s >= a.src_total || d >= a.dst_total) {
        if (first) { atomicOr(a.status, CS_ST_BAD_SLOT); atomicAdd((unsigned long long *)&a.cnt->blocks_skipped, one); }
        return false;
    }
    if (first) {
        atomicAdd((unsigned long long *)&a.cnt->blocks_moved[a.kind], one);
        atomicAdd((unsigned long long *)&a.cnt->bytes_moved[a.kind], one * a.block_bytes);
    }
    const unsigned long long in_chunk = (unsigned long long)piece * a.piece_bytes;
    sp = a.src + chunk_offset(a.src_layout, a.n_chunks, a.src_total, lp, s, a.chunk) + in_chunk;
    dp = a.dst + chunk_offset(a.dst_layout, a.n_chunks, a.dst_total, lp, d, a.chunk) + in_chunk;
    const unsigned long long left = a.chunk - in_chunk;
    bytes = (uint32_t)(left < a.piece_bytes ? left : a.piece_bytes);
    return true;
}

__device__ __forceinline__ uint32_t mover_count(const MoverArgs &a)
{
    uint32_t n = a.n_max;
    if (a.n_dev) { const uint32_t nd = *a.n_dev; n = nd < n ? nd : n; }
    return n;
}

// ---------------------------------------------------------------------------------------------
// load/store path
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(MV_THREADS) cs_mover_kernel(MoverArgs a)
{
    const uint32_t n = mover_count(a);
    const uint32_t per_block = a.n_chunks * a.pieces;
    const unsigned long long total = (unsigned long long)n * per_block;
    for (unsigned long long w = blockIdx.x; w < total; w += gridDim.x) {
        const char *sp0;
        char *dp0;
        uint32_t bytes;
        if (!resolve_piece(a, w, per_block, fetch_slots(a, w, per_block), sp0, dp0, bytes, threadIdx.x == 0 ? 1 : 0)) continue;
        const uint4 *sp = (const uint4 *)sp0;
        uint4 *dp = (uint4 *)dp0;
        const uint32_t nvec = bytes >> 4;
        uint4 v[MV_UNROLL];
#pragma unroll
        for (int u = 0; u < MV_UNROLL; ++u) {
            const uint32_t x = threadIdx.x + u * MV_THREADS;
            if (x < nvec) v[u] = __ldcs(sp + x);
        }
#pragma unroll
        for (int u = 0; u < MV_UNROLL; ++u) {
            const uint32_t x = threadIdx.x + u * MV_THREADS;
            if (x < nvec) __stcs(dp + x, v[u]);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// bulk (TMA) path
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after TM_SPIN_LIMIT polls (each poll may itself block for a short,
// hardware-bounded time) and reports failure instead of spinning forever.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint32_t limit = TM_SPIN_LIMIT)
{
    for (uint32_t spin = 0; spin < limit; ++spin) {
        if (mbar_test(bar, parity)) return true;
        if (spin > 64) __nanosleep(128);
    }
    return false;
}
// KV blocks stream through once: both directions of every copy carry an evict-first L2 policy, so the
// gigabytes a step moves do not push the (L2-resident) block index and tables of the select kernels out.
#ifndef TM_EVICT_FIRST
#define TM_EVICT_FIRST 1
#endif
__device__ __forceinline__ unsigned long long l2_stream_policy()
{
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void *src, uint32_t bytes, uint32_t bar,
                                          unsigned long long pol)
{
#if TM_EVICT_FIRST
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst_smem),
                 "l"(src), "r"(bytes), "r"(bar), "l"(pol)
                 : "memory");
#else
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_smem),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
#endif
}
__device__ __forceinline__ void bulk_store(void *dst, uint32_t src_smem, uint32_t bytes, unsigned long long pol)
{
#if TM_EVICT_FIRST
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(dst), "r"(src_smem),
                 "r"(bytes), "l"(pol)
                 : "memory");
#else
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src_smem), "r"(bytes)
                 : "memory");
#endif
}

// One pipeline per warp.  The lanes resolve the pipeline's next 32 items side by side (the slot list look-ups of a piece
// cost as much time as moving 2 KiB); lane 0 issues the copies.  Iteration `it` first stores item it - LAG, whose load was
// issued LAG iterations ago, and then issues the load of item `it` into the ring slot whose previous store has finished
// reading shared memory.  `fetch(it)` looks an item's list entries up, a batch of 32 ahead of
// `item(it, slots, sp, dp, bytes, book)`, which resolves it; false = nothing to copy.  The work counters are booked with the batch; when a
// wait runs out, what the batch holds from the item on whose load was never issued is taken back.
template <int STAGES> struct PipeShared {
    unsigned long long bar[STAGES];
    char *dst[STAGES];                // destination of the item loaded into each ring slot
    uint32_t bytes[STAGES];           // 0: nothing in flight there
};
template <int STAGES, class Fetch, class Item>
__device__ __forceinline__ void bulk_pipeline(unsigned char *my_ring, PipeShared<STAGES> &ps, unsigned long long n_items, uint32_t *status,
                                              Fetch fetch, Item item)
{
    constexpr uint32_t PIECE = TM_RING / STAGES;
    constexpr int LAG = STAGES - (STAGES + 2) / 3;    // two thirds of the slots load, one third store
    constexpr uint32_t ALL = 0xFFFFFFFFu;
    const uint32_t lane = threadIdx.x & 31;
    const unsigned long long pol = l2_stream_policy();
    uint32_t phase_bits = 0;          // parity to wait for, one bit per ring slot
    bool failed = false;
    char *sp = nullptr, *dp = nullptr;
    uint32_t bytes = 0;
    uint2 next = make_uint2(CS_ID_NONE, CS_ID_NONE);
    if (lane < n_items) next = fetch(lane);
    int st_load = 0, st_store = 0;    // ring slots of items it and it - LAG
    unsigned long long it = 0;
    for (; it < n_items + LAG; ++it) {
        if ((it & 31u) == 0 && it < n_items) {                // resolve the next 32 items
            const char *s = nullptr;
            bytes = 0;
            if (it + lane < n_items && !item(it + lane, next, s, dp, bytes, 1)) bytes = 0;
            sp = const_cast<char *>(s);
            if (it + 32u + lane < n_items) next = fetch(it + 32u + lane);
        }
        const int from = (int)(it & 31u);
        const char *src = (const char *)__shfl_sync(ALL, (unsigned long long)sp, from);
        char *dst = (char *)__shfl_sync(ALL, (unsigned long long)dp, from);
        const uint32_t n = it < n_items ? __shfl_sync(ALL, bytes, from) : 0u;
        if (lane == 0 && !failed) {
            if (it >= (unsigned long long)LAG) {                              // store item it - LAG
                const uint32_t m = ps.bytes[st_store];
                if (m) {
                    const uint32_t bar = smem_u32(&ps.bar[st_store]);
                    if (!mbar_wait_bounded(bar, (phase_bits >> st_store) & 1u)) {
                        failed = true;
                        atomicOr(status, CS_ST_TIMEOUT);
                    } else {
                        ps.bytes[st_store] = 0;
                        phase_bits ^= 1u << st_store;
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        bulk_store(ps.dst[st_store], smem_u32(my_ring + (size_t)st_store * PIECE), m, pol);
                    }
                }
                // one group per item, empty for a skipped item, so that group counts match item counts
                if (!failed) asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
            if (n && !failed) {                                               // load item `it`
                // the slot's previous store (item it - STAGES) was committed STAGES - LAG iterations ago: at most the
                // groups since then may still be reading shared memory
                asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(STAGES - LAG) : "memory");
                ps.dst[st_load] = dst;
                ps.bytes[st_load] = n;
                const uint32_t bar = smem_u32(&ps.bar[st_load]);
                mbar_expect_tx(bar, n);
                bulk_load(smem_u32(my_ring + (size_t)st_load * PIECE), src, n, bar, pol);
            }
        }
        st_load = st_load + 1 == STAGES ? 0 : st_load + 1;
        if (it >= (unsigned long long)LAG) st_store = st_store + 1 == STAGES ? 0 : st_store + 1;
        if (__shfl_sync(ALL, failed ? 1 : 0, 0)) break;
    }
    if (it < n_items) {                                       // a wait ran out before the load of item `it` was issued
        const unsigned long long mine = (it & ~31ull) + lane;
        const char *s;
        if (mine >= it && mine < n_items) (void)item(mine, fetch(mine), s, dp, bytes, -1);
    }
    if (lane == 0) {
        if (failed) {
            // give the loads still in flight a bounded chance to land before shared memory is released
            for (int st = 0; st < STAGES; ++st)
                if (ps.bytes[st]) mbar_wait_bounded(smem_u32(&ps.bar[st]), (phase_bits >> st) & 1u);
        }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");             // all stores written
    }
}

// Per-warp set-up shared by the bulk kernels: ring slice and barriers.  Returns false for warps that have nothing to do.
template <int STAGES>
__device__ __forceinline__ bool bulk_setup(unsigned char *ring, PipeShared<STAGES> *pipes, uint32_t n_pipes, unsigned char *&my_ring,
                                           unsigned long long &first)
{
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    my_ring = ring + (size_t)warp * TM_RING;
    if (lane == 0) {
        for (int st = 0; st < STAGES; ++st) {
            mbar_init(smem_u32(&pipes[warp].bar[st]), 1);
            pipes[warp].bytes[st] = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    first = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + warp;
    return first < n_pipes;
}

__device__ __forceinline__ unsigned long long items_of_pipe(unsigned long long total, unsigned long long first,
                                                            unsigned long long n_pipes)
{
    return first < total ? (total - first + n_pipes - 1) / n_pipes : 0;
}

// One transfer: pipeline `first` of n_pipes takes the pieces first, first + n_pipes, ...
template <int STAGES>
__global__ void __launch_bounds__(TM_WARPS * 32, 1) cs_mover_bulk_kernel(MoverArgs a)
{
    extern __shared__ __align__(128) unsigned char ring[];
    __shared__ __align__(8) PipeShared<STAGES> pipes[TM_WARPS];
    unsigned char *my_ring;
    unsigned long long first;
    if (!bulk_setup<STAGES>(ring, pipes, a.n_pipes, my_ring, first)) return;
    const uint32_t per_block = a.n_chunks * a.pieces;
    const unsigned long long total = (unsigned long long)mover_count(a) * per_block;
    const unsigned long long n_pipes = a.n_pipes;
    bulk_pipeline<STAGES>(my_ring, pipes[threadIdx.x >> 5], items_of_pipe(total, first, n_pipes), a.status,
                          [&](unsigned long long it) { return fetch_slots(a, first + it * n_pipes, per_block); },
                          [&](unsigned long long it, uint2 slots, const char *&sp, char *&dp, uint32_t &bytes, int book) {
                              return resolve_piece(a, first + it * n_pipes, per_block, slots, sp, dp, bytes, book);
                          });
}

// Two transfers in opposite directions over the host link in one launch.  Every pipeline takes its
// share of both piece lists and walks them interleaved in proportion to their lengths, so the two
// directions advance in lock step and finish together whatever the link's arbitration between reads
// and writes would otherwise give each of them.
template <int STAGES>
__global__ void __launch_bounds__(TM_WARPS * 32, 1) cs_exchange_bulk_kernel(MoverArgs off, MoverArgs pre)
{
    extern __shared__ __align__(128) unsigned char ring[];
    __shared__ __align__(8) PipeShared<STAGES> pipes[TM_WARPS];
    unsigned char *my_ring;
    unsigned long long first;
    if (!bulk_setup<STAGES>(ring, pipes, off.n_pipes, my_ring, first)) return;
    const uint32_t per_block = off.n_chunks * off.pieces;
    const unsigned long long n_pipes = off.n_pipes;
    const unsigned long long n_o = items_of_pipe((unsigned long long)mover_count(off) * per_block, first, n_pipes);
    const unsigned long long n_p = items_of_pipe((unsigned long long)mover_count(pre) * per_block, first, n_pipes);
    const unsigned long long n_items = n_o + n_p;
    // item `it` as a piece of one of the two lists: offload pieces among the first `it` items: floor(it * n_o / n_items)
    const auto offloads = [&](unsigned long long it, unsigned long long &w) {
        const unsigned long long before = it * n_o / n_items, after = (it + 1) * n_o / n_items;
        w = first + (after != before ? before : it - before) * n_pipes;
        return after != before;
    };
    bulk_pipeline<STAGES>(my_ring, pipes[threadIdx.x >> 5], n_items, off.status,
                          [&](unsigned long long it) {
                              unsigned long long w;
                              return offloads(it, w) ? fetch_slots(off, w, per_block) : fetch_slots(pre, w, per_block);
                          },
                          [&](unsigned long long it, uint2 slots, const char *&sp, char *&dp, uint32_t &bytes, int book) {
                              unsigned long long w;
                              return offloads(it, w) ? resolve_piece(off, w, per_block, slots, sp, dp, bytes, book)
                                                     : resolve_piece(pre, w, per_block, slots, sp, dp, bytes, book);
                          });
}

// ---------------------------------------------------------------------------------------------
// Slot size of a bulk transfer's rings: the smallest that holds a chunk, at most 16 KiB.
static uint32_t bulk_piece(unsigned long long chunk)
{
    uint32_t piece = 2048u;
    while (piece < TM_PIECE && piece < chunk) piece <<= 1;
    return piece;
}

static void fill_mover_args(cs_ctx *ctx, MoverArgs &a, const cs_kv_pool *src, const cs_kv_pool *dst,
                            const uint32_t *src_slots, const uint32_t *dst_slots, uint32_t n_max, const uint32_t *n_dev,
                            uint32_t piece_bytes, int kind)
{
    a.cnt = ctx->ws.cnt;
    a.kind = (uint32_t)kind;
    a.src = (const char *)src->base;
    a.dst = (char *)dst->base;
    a.src_total = src->n_slots;
    a.dst_total = dst->n_slots;
    a.src_first = src->first_id;
    a.dst_first = dst->first_id;
    a.src_layout = src->layout;
    a.dst_layout = dst->layout;
    a.n_chunks = 2u * src->n_layers;
    a.chunk = (unsigned long long)src->block_tokens * src->n_kv_heads * src->head_dim * src->elem_bytes;
    a.block_bytes = a.n_chunks * a.chunk;
    if (src->layout == CS_BLOCK_MAJOR && dst->layout == CS_BLOCK_MAJOR) {      // a block is one run of bytes on both sides
        a.chunk = a.block_bytes;
        a.n_chunks = 1;
    }
    if (!piece_bytes) piece_bytes = bulk_piece(a.chunk);
    a.src_slots = src_slots;
    a.dst_slots = dst_slots;
    a.n_dev = n_dev;
    a.n_max = n_max;
    a.status = &ctx->ws.sc->status;
    a.n_pipes = 0;
    a.piece_bytes = piece_bytes;
    a.pieces = (uint32_t)((a.chunk + piece_bytes - 1) / piece_bytes);
}

// Shape of a bulk launch: pipelines (warps), and how many of them share a CTA.
//  host link: as few pipelines as keep the link full, one per CTA (a ring of 48 KiB fits the SMs' default shared-memory
//    split).  8 out, 24 in, 32 both ways; more for small pieces, whose issue takes longer than their flight (4 KiB pieces out:
//    8 pipelines 51.0 GB/s, 24 52.4; 2 KiB: 8 45.5, 32 52.4; 1 KiB both ways: 32 76.6, 64 79.0).
//  inside the device: much in flight, but no more than the memory takes.  Long moves: 1.7 pipelines per SM, two per CTA
//    (256 blocks of 2 MiB: 148 pipelines 207 us, 200 182, 220 to 268 178, 296 179, 328 197; four per CTA need 280 for the same,
//    and longer to start).  Short ones, where starting and draining decide, and small pieces: four per SM, one per CTA (16 blocks
//    of 2 MiB: 9.5 us against 12.7 with 296 in CTAs of four; 64 blocks: 47.5 against 45.2, so the line lies between; 400 blocks
//    of 64 chunks of 4 KiB: 252 pipelines 42.4 us, 592 37.9).
#define D2D_SHORT_BYTES (48ull << 20)
struct BulkShape { uint32_t pipes, per_cta; };
static BulkShape bulk_shape(const cs_ctx *ctx, int kind, uint32_t piece, unsigned long long chunk, unsigned long long bytes)
{
    const uint32_t sms = (uint32_t)ctx->sm_count;
    if (kind == CS_MOVE_D2D) {
        const bool fine = bytes < D2D_SHORT_BYTES || piece <= 4096u;
        const uint32_t pipes = ctx->d2d_ctas ? ctx->d2d_ctas : (fine ? 4u * sms : sms * 17u / 10u);
        return BulkShape{pipes, fine || pipes <= 64u ? 1u : (uint32_t)TM_WARPS};
    }
    // (a pack / scatter launch of the copy-engine path only has to keep ahead of the host link: 64 pipelines move
    //  about 1.5 TB/s and leave most SMs to the kernels running beside it)
    if (kind == CS_MOVE_STAGE) return BulkShape{64u, 1u};
    uint32_t pipes = ctx->host_link_ctas;
    if (!pipes) {
        if (kind == CS_MOVE_OFFLOAD) pipes = piece >= 8192u ? 8u : (piece >= 4096u ? 24u : 32u);
        else if (kind == CS_MOVE_PREFETCH) pipes = 24u;
        else pipes = chunk >= 2048u ? CS_EXCHANGE_PIPES : 2u * CS_EXCHANGE_PIPES;
    }
    return BulkShape{pipes, pipes <= 64u ? 1u : (uint32_t)TM_WARPS};
}
#define CS_MOVE_EXCHANGE 4         // bulk_shape(): both directions in one launch

// Shared-memory opt-in of the bulk kernels: an attribute of the function on a device, so it is set once per
// process and device (always to the same fixed size).
static std::mutex g_bulk_mu;
static bool g_bulk_opted[64];
template <int STAGES>
static cudaError_t bulk_opt_in_one()
{
    cudaError_t e = cudaFuncSetAttribute(cs_mover_bulk_kernel<STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, TM_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cs_exchange_bulk_kernel<STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, TM_SMEM);
    // The largest split of the SMs' memory: beside it a CTA of the whole-GPU select (up to 131 KiB) still fits, which would wait for the end of the
    // move otherwise (selects beside back-to-back compactions of 256 blocks of 2 MiB: 217 us each, 99 with this).
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cs_mover_bulk_kernel<STAGES>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cs_exchange_bulk_kernel<STAGES>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e;
}
static int bulk_opt_in(cs_ctx *ctx)
{
    if (ctx->device < 0 || ctx->device >= 64) return CS_EINVAL;
    std::lock_guard<std::mutex> lock(g_bulk_mu);
    if (g_bulk_opted[ctx->device]) return CS_OK;
    cudaError_t e = bulk_opt_in_one<3>();
    if (e == cudaSuccess) e = bulk_opt_in_one<6>();
    if (e == cudaSuccess) e = bulk_opt_in_one<12>();
    if (e == cudaSuccess) e = bulk_opt_in_one<24>();
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
    g_bulk_opted[ctx->device] = true;
    return CS_OK;
}

// One launch with rings cut for pieces of piece_bytes.
template <class F>
static void bulk_by_piece(uint32_t piece_bytes, F launch)
{
    if (piece_bytes <= 2048u) launch(std::integral_constant<int, 24>());
    else if (piece_bytes <= 4096u) launch(std::integral_constant<int, 12>());
    else if (piece_bytes <= 8192u) launch(std::integral_constant<int, 6>());
    else launch(std::integral_constant<int, 3>());
}
static_assert(TM_RING / 24 == 2048 && TM_RING / 3 == TM_PIECE, "slots of 2 to 16 KiB");

int cs_launch_mover(cs_ctx *ctx, const cs_kv_pool *src, const cs_kv_pool *dst, const uint32_t *src_slots,
                    const uint32_t *dst_slots, uint32_t n_max, const uint32_t *n_dev, int kind, cudaStream_t s)
{
    return cs_launch_mover_as(ctx, src, dst, src_slots, dst_slots, n_max, n_dev, kind, kind, s);
}

// `kind` decides the width of the launch (which memory the bytes cross), `count_as` the direction the work
// counters book the blocks under (the pack and scatter launches of the copy-engine path move blocks inside the
// device on behalf of an offload or a prefetch).
int cs_launch_mover_as(cs_ctx *ctx, const cs_kv_pool *src, const cs_kv_pool *dst, const uint32_t *src_slots,
                       const uint32_t *dst_slots, uint32_t n_max, const uint32_t *n_dev, int kind, int count_as,
                       cudaStream_t s)
{
    const bool bulk = ctx->mover_path != CS_MOVER_LDST;
    MoverArgs a;
    fill_mover_args(ctx, a, src, dst, src_slots, dst_slots, n_max, n_dev, bulk ? 0u : MV_PIECE, count_as);
    const unsigned long long total = (unsigned long long)n_max * a.n_chunks * a.pieces;
    if (bulk) {
        const BulkShape sh = bulk_shape(ctx, kind, a.piece_bytes, a.chunk, n_max * a.block_bytes);
        a.n_pipes = (uint32_t)(total < sh.pipes ? total : sh.pipes);
        if (a.n_pipes == 0) a.n_pipes = 1;
        const uint32_t wpc = sh.per_cta, grid = (a.n_pipes + wpc - 1) / wpc;
        const int rc = bulk_opt_in(ctx);
        if (rc != CS_OK) return rc;
        bulk_by_piece(a.piece_bytes, [&](auto stages) { cs_mover_bulk_kernel<decltype(stages)::value><<<grid, wpc * 32, (size_t)wpc * TM_RING, s>>>(a); });
    } else {
        const uint32_t dflt = kind == CS_MOVE_D2D ? 8u * (uint32_t)ctx->sm_count
                            : (kind == CS_MOVE_STAGE ? 64u : (kind == CS_MOVE_OFFLOAD ? 8u : 12u));
        const uint32_t asked = kind == CS_MOVE_D2D ? ctx->d2d_ctas : (kind == CS_MOVE_STAGE ? 0u : ctx->host_link_ctas);
        const unsigned long long cap = asked ? asked : dflt;
        const uint32_t grid = (uint32_t)(total < cap ? total : cap);
        cs_mover_kernel<<<grid ? grid : 1u, MV_THREADS, 0, s>>>(a);
    }
    return cs_check_launch(ctx);
}

// Offload and prefetch of one step as a single launch (bulk path only).
int cs_launch_exchange(cs_ctx *ctx, const cs_kv_pool *gpu, const cs_kv_pool *host, const uint32_t *off_gpu_slots,
                       const uint32_t *off_host_slots, uint32_t n_off_max, const uint32_t *n_off_dev,
                       const uint32_t *pre_host_slots, const uint32_t *pre_gpu_slots, uint32_t n_pre_max,
                       const uint32_t *n_pre_dev, cudaStream_t s)
{
    MoverArgs off, pre;
    fill_mover_args(ctx, off, gpu, host, off_gpu_slots, off_host_slots, n_off_max, n_off_dev, 0u, CS_MOVE_OFFLOAD);
    fill_mover_args(ctx, pre, host, gpu, pre_host_slots, pre_gpu_slots, n_pre_max, n_pre_dev, 0u, CS_MOVE_PREFETCH);
    const unsigned long long total = ((unsigned long long)n_off_max + n_pre_max) * off.n_chunks * off.pieces;
    const BulkShape sh = bulk_shape(ctx, CS_MOVE_EXCHANGE, off.piece_bytes, off.chunk, 0);
    uint32_t n_pipes = (uint32_t)(total < sh.pipes ? total : sh.pipes);
    if (n_pipes == 0) n_pipes = 1;
    off.n_pipes = pre.n_pipes = n_pipes;
    const uint32_t wpc = sh.per_cta, grid = (n_pipes + wpc - 1) / wpc;
    const int rc = bulk_opt_in(ctx);
    if (rc != CS_OK) return rc;
    bulk_by_piece(off.piece_bytes, [&](auto stages) {
        cs_exchange_bulk_kernel<decltype(stages)::value><<<grid, wpc * 32, (size_t)wpc * TM_RING, s>>>(off, pre);
    });
    return cs_check_launch(ctx);
}

// ---------------------------------------------------------------------------------------------
// Self-test of the bounded wait: one warp, one barrier, no copy.  The wait cannot succeed, so it runs out
// after `max_polls` polls and the kernel reports exactly as a stalled transfer would.  Nothing is in flight.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(32) cs_bounded_wait_selftest_kernel(uint32_t max_polls, uint32_t *status)
{
    __shared__ __align__(8) unsigned long long bar_mem;
    if (threadIdx.x != 0) return;
    const uint32_t bar = smem_u32(&bar_mem);
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait_bounded(bar, 0, max_polls)) atomicOr(status, CS_ST_TIMEOUT);
}

int cs_launch_bounded_wait_selftest(cs_ctx *ctx, uint32_t max_polls, cudaStream_t s)
{
    cs_bounded_wait_selftest_kernel<<<1, 32, 0, s>>>(max_polls, &ctx->ws.sc->status);
    return cs_check_launch(ctx);
}
