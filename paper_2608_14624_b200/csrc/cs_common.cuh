// Internal declarations shared by the translation units of libcachescout (sm_100a only).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "cachescout.h"

// NVTX ranges around the entry points that enqueue work: a timeline tool shows which library call a kernel belongs
// to.  Header-only (NVTX 3 loads the tool's injection library on first use; without a tool a range costs a few
// nanoseconds).  -DCS_NO_NVTX compiles the ranges out.
#ifndef CS_NO_NVTX
#include <nvtx3/nvToolsExt.h>
struct cs_nvtx_range {
    explicit cs_nvtx_range(const char *name) { nvtxRangePushA(name); }
    ~cs_nvtx_range() { nvtxRangePop(); }
};
#define CS_RANGE(name) cs_nvtx_range cs_range_guard_(name)
#else
#define CS_RANGE(name) do { } while (0)
#endif

#if defined(__CUDA_ARCH__) && (__CUDA_ARCH__ < 1000)
#error "libcachescout is written for sm_100a (B200) only"
#endif

#define CS_SELECT_CLUSTER_MAX_BLOCKS (1u << 18)   // largest index of the single-launch cluster select

// Index sizes and list lengths that take the one-launch select on the whole GPU (cs_select_grid.cu).
#define CS_SELECT_GRID_MIN_BLOCKS (1u << 17)
#define CS_SELECT_GRID_LONG_BLOCKS (1u << 16)      // with a list of CS_SELECT_GRID_LONG_LIST ids or more
#define CS_SELECT_GRID_LONG_LIST 2048u
#define CS_SELECT_GRID_MAX_BLOCKS (1u << 25)
#define CS_SELECT_GRID_MAX_LIST 50000u

#define CS_CONCURRENT_MAX_BLOCKS (1u << 22)        // up to this index size every select of a step has full-size scratch of its own

#define CS_AGE_LIMIT_MIN_BLOCKS (1u << 21)        // index size from which the collect pass builds age limits

#define CS_MOVE_D2D 0
#define CS_MOVE_OFFLOAD 1
#define CS_MOVE_PREFETCH 2
#define CS_MOVE_STAGE 3            // pack / scatter launch of the copy-engine path: inside the device, deliberately narrow

#define CS_HIST_BINS 4096u        // bins of the select's histogram: the range that scores can have, divided evenly
#define CS_MAX_SPLITTERS 255u     // bucket sort of the candidates: up to 256 buckets
#define CS_SAMPLE 1024u           // candidates sampled to choose the splitters
#define CS_BUCKETS 512u           // buckets of the grid-wide ordering
#define CS_GTAB_MAX 4096u          // largest recency table kept in shared memory (ages below saturation)

// Scalars the kernels share, one 256-byte line in the workspace.
#define CS_BCOUNT_STRIDE 8u                                      // words between bucket counters
#define CS_BCOUNT(ws, b) ((ws).bcount[(size_t)(b) * CS_BCOUNT_STRIDE])          // candidates of a bucket
// Phase stamps (builds with -DCS_PHASE_STAMPS only; cs_debug_phase_stamps() reads them).  A call's kernels are chains
// of dependent steps whose cost is latency, not work, so "where does the time go" is answered by the GPU's global
// nanosecond timer read at the boundaries: CS_STAMP(ws, slot, cond) stores it into slot `slot` when `cond` holds
// (one thread of one CTA).  In ordinary builds the macro is empty and the slots do not exist.
#define CS_N_PHASE_STAMPS 64
enum {
    CS_PS_REFRESH_ENTRY = 0, CS_PS_REFRESH_WAITED, CS_PS_REFRESH_ROWS_DONE, CS_PS_REFRESH_LAST_CTA, CS_PS_REFRESH_SUMS_DONE,
    CS_PS_REFRESH_END,
    CS_PS_SCAN_ENTRY = 8,       // + 8 for the prefetch select: entry, set-up done, waited, index read, flushed, last CTA, tail done
    CS_PS_SCAN_SETUP, CS_PS_SCAN_WAITED, CS_PS_SCAN_READ, CS_PS_SCAN_FLUSHED, CS_PS_SCAN_LAST_CTA, CS_PS_SCAN_TAIL_DONE,
    CS_PS_SAMPLE_WAITED = 24,   // + 8 for the prefetch select: sample waited / done, place waited / done, finish waited / done
    CS_PS_SAMPLE_DONE, CS_PS_PLACE_WAITED, CS_PS_PLACE_DONE, CS_PS_FINISH_WAITED, CS_PS_FINISH_DONE,
    CS_PS_SCAN_TABLES = 56,     // + 4 for the prefetch select: per-call tables loaded, cuts built, index tiles walked (CTA 0)
    CS_PS_SCAN_CUTS, CS_PS_SCAN_WALKED
};
#ifdef CS_PHASE_STAMPS
#define CS_STAMP(ws, slot, cond)                                                         \
    do {                                                                                 \
        if (cond) {                                                                      \
            unsigned long long cs_t_;                                                    \
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(cs_t_)::"memory");          \
            (ws).sc->stamps[slot] = cs_t_;                                               \
        }                                                                                \
    } while (0)
#else
#define CS_STAMP(ws, slot, cond) do { } while (0)
#endif

struct cs_scalars {
    uint32_t status;        // CS_ST_* bits
    uint32_t last_agent;    // agent of the last non-warmup event, CS_AGENT_NONE initially
    uint32_t a_star;        // arg-max successor of last_agent (Eq. 10), ~0 while there is no current agent; kept by the refresh
    float R;                // Eq. 2
    uint32_t gate;          // Eq. 11: R >= r_min
    uint32_t n_transitions; // sum of all counts
    uint32_t refresh_ticket;       // CTAs of a refresh of many agents that are done; 0 between calls
    uint32_t gtab_monotone; // the recency table covers every unsaturated age and never increases with age
    uint32_t status_read;   // cs_get_status(): the value swapped out of `status`
    uint32_t val_le, val_elig, val_ticket;   // cs_validate_selection(): keys at or below the last one, eligible entries, ticket
    unsigned long long sel_T[4];   // key (primary, secondary) up to which the next large select of each kind (GPU victims,
                            // host victims, prefetch) collects in its one scan, chosen by the previous call of the kind;
                            // ~0 = none; slot 3 is never written: calls that must not speculate read it
#ifdef CS_PHASE_STAMPS
    unsigned long long stamps[CS_N_PHASE_STAMPS];   // %globaltimer at phase boundaries of the latest call (profiling builds)
#endif
};

// State of one select in flight, rewritten by every call.  The selects of a step that run side by side each
// have their own (with their own histogram, candidate and sort regions).
struct cs_sel_state {
    uint32_t c;             // candidates collected
    uint32_t n_out;         // min(k, eligible)
    uint32_t n_elig;        // eligible entries
    uint32_t b0;            // threshold bin of the histogram (after a miss)
    unsigned long long bound;      // key up to which the candidates were collected
    unsigned long long ahead;      // key up to which about cs_ahead(k) candidates lie, ~0: fewer were collected
    uint32_t ticket[4];     // "last CTA done" counters, one per kernel that has an epilogue
    uint32_t c_spec;        // candidates appended by the fast pass; 0 between calls
    uint32_t n_above;       // eligible entries the fast pass found above the remembered key; 0 between calls
    uint32_t spec;          // 1: the fast pass's candidates cover the k winners, the histogram and collect passes are skipped
};

// State of the one-launch select of large indexes (cs_select_grid.cu), one per context.  What a launch counts in lies twice, used by turns:
// a launch clears the set of the next one.
#define CS_GRID_MAX_CTAS 160u
struct cs_grid_list {
    uint32_t c_scan, c_collect, eligible, pad; // candidates of the scan and of the collect pass; eligible entries that the scan saw
    unsigned long long ahead;                  // key below which about sg_ahead(k) candidates lie, ~0: there are fewer
    uint32_t pad2[2];
};
struct cs_grid_state {
    uint32_t failed, pad[31];                  // shares of a launch whose CTAs have left it because a wait ran out, 0 between launches
    unsigned long long taken[CS_GRID_MAX_CTAS];        // by share: starts of its CTA (the launch's number, its parity the set in use), and, in the upper
                                               // half, the complement of the last launch in which another CTA took the share over
    uint32_t bar[2][8][32];                    // grid barriers, a line each: shares that are done, and whether a wait for the others has run out
    cs_grid_list list[2][4];
    uint32_t count[2][3][CS_BUCKETS * CS_BCOUNT_STRIDE];       // keys per bucket
    uint32_t rem_n[4];                         // by list: buckets of the next call of the kind, and where they start (from 1 on; [rem_n]: the end)
    uint32_t rem_now[4];                       // the clock at which that was so,
    unsigned long long rem_T[4];               // and the key remembered with it (cs_scalars.sel_T, unless another route has chosen one since)
    unsigned long long rem_km[3][CS_BUCKETS + 8];
    uint32_t rem_id[3][CS_BUCKETS + 8];
};

// Device pointers into the caller's workspace.
struct cs_workspace {
    cs_scalars *sc;
    cs_counters *cnt;     // work counters (cs_get_counters)
    cs_sel_state *sel;    // this select's state (one per concurrent select)
    cs_grid_state *grid;  // large indexes in one launch
    uint32_t *C;          // [A*A] transition counts
    uint32_t *rowsum;     // [A]
    uint16_t *cur;        // [n_chains]
    float *P;             // [A*A] Eq. 3
    uint16_t *amax;       // [A]
    uint32_t *adjT;       // [W][A] transpose of the Eq. 7 adjacency, W = ceil(A/32): bit b of word w of column v = an edge from
                          // agent 32 w + b to agent v (word by word, so that one thread per agent reads it coalesced)
    unsigned long long *qsum;      // [A] a refresh of many agents: column sums of Eq. 2 in the making, 0 between calls
    unsigned long long *cta_base;  // and what its CTAs leave for the last one (RfShared::base, hc)
    double *cta_hc;
    uint16_t *hops;       // [A]
    float *fsurv;         // [A] p~ + delta for the cached source
    uint16_t *hops_tmp;   // [A] same, for cs_score_blocks() with explicit sources
    float *fsurv_tmp;     // [A]
    float *gtab;          // [gtab_len] exp(-lambda*age)+delta for age < gtab_len
    uint32_t *hist;       // [CS_HIST_BINS]
    unsigned long long *cand_km;    // [max_blocks] (primary<<32 | secondary) of each candidate
    uint32_t *cand_id;    // [max_blocks]
    uint32_t *cand_bkt;   // [max_blocks] cluster select, ordering through global memory: bucket of each candidate; launch chain: places of
                          // the keys of buckets that outgrow the tile, every bucket at its offset in the order
    uint32_t *cand_slot;  // [max_blocks] cluster select: slot in that bucket
    unsigned long long *sort_km;    // [max_blocks] candidates grouped by bucket
    uint32_t *sort_id;    // [max_blocks]
    unsigned long long *spl_km;     // [CS_SAMPLE] the ranked sample; the splitters of the general route
    uint32_t *spl_id;     // [CS_SAMPLE]
    uint32_t *bcount;     // bucket counters, one per 32-byte sector (CS_BCOUNT): atomics on counters that share a sector
                          // queue up behind one another in L2 (measured: 3.6 us for 16,000 of them on adjacent words,
                          // 0.8 us on separate sectors; separate 128-byte lines are no faster and cost the readers more)
};

// Six-launch selects side by side as one graph: node[job][launch] gets its arguments anew on every call.
#define CS_SELECT_STAGES 6
struct cs_select_graph {
    cudaGraph_t graph;
    cudaGraphExec_t exec;
    cudaGraphNode_t node[3][CS_SELECT_STAGES];
    uint32_t asked, refused;       // calls that wanted it before it was there (up to 2); 1: it could not be built or launched
};

struct cs_ctx {
    cs_params p;
    cs_workspace ws;
    cs_workspace ws_job[2];        // the same workspace with private candidate / sort regions: jobs 1 and 2 of a fused select
    size_t ws_bytes;
    uint32_t W;            // adjacency words per row
    uint32_t gtab_len;     // ages [0, gtab_len) come from the table
    uint32_t age_sat;      // ages >= age_sat all give g_sat
    int device;
    int sm_count;
    uint32_t host_link_ctas, d2d_ctas;
    uint32_t mover_path;   // CS_MOVER_*
    uint32_t select_path;  // CS_SELECT_*
    uint32_t no_speculation;       // 1: the histogram pass never collects ahead of the threshold
    uint32_t region_cap_max;       // cap on the keys of a bucket's own region in the sort arrays (0: none)
    uint32_t source_mode;          // CS_SOURCES_*: where the cached BFS of Eq. 8 starts
    const float *fsurv_override;   // caller's survival table for score / select, NULL = the BFS table of Eq. 8
    const uint32_t *clock_dev;           // cs_set_device_clock(): selects and scores read the clock from here when they run
    const uint32_t *step_now_dev;        // set only while cs_step() issues its calls: device-resident clock / event count
    const uint32_t *step_n_events_dev;
    cudaEvent_t ev_fork, ev_join;        // cs_step(): main -> side and side -> main
    cudaStream_t sel_stream[2];          // the second and third select of a step run here, beside the first
    cudaEvent_t ev_sel_fork, ev_sel_join[2];
    int concurrent_selects;              // the per-select scratch regions are full size
    uint32_t lists_asked;                // lists that a select has been asked for, one bit each
    uint32_t grid_refused;               // 1: the driver would not launch the whole-GPU select; the launch chain does from then on
    uint32_t grid_give_up;               // cs_selftest_select_wait(): the grid barrier (1 ..) at which its waits give up at once, 6: late CTAs, 0: neither
    cs_select_graph sel_graph[8];        // selects side by side, by the lists wanted (bit q: select q)
    // copy-engine path of the mover (cs_set_mover_staging): caller-owned device ring split into four sub-buffers
    // (two per direction, double-buffered), two streams of the context for the two DMA directions, and the events
    // that order packing / copying / scattering
    unsigned char *stage_ring;
    size_t stage_bytes;
    cudaStream_t copy_stream[4];         // 0, 1: device -> host; 2, 3: host -> device
    cudaStream_t scatter_stream;         // scatter launches of staged prefetches
    cudaEvent_t ev_stage_fork, ev_stage_join[2];
    cudaEvent_t ev_packed[2], ev_copied[4], ev_filled[4], ev_scattered[2];   // [ring buffer] or [2 * ring buffer + copy stream]
    uint64_t n_launches;
    int last_cuda_error;
};

// ---- workspace layout (host) -------------------------------------------------------------------
size_t cs_layout_workspace(const cs_params *p, uint32_t gtab_len, void *base, cs_workspace *ws, cs_workspace *ws_job);
int cs_validate_params(const cs_params *p);
void cs_recency_table_shape(const cs_params *p, uint32_t *gtab_len, uint32_t *age_sat);

// ---- launchers implemented in the kernel files ---------------------------------------------------
int cs_launch_init(cs_ctx *ctx, cudaStream_t s);
int cs_launch_observe(cs_ctx *ctx, const uint32_t *chain, const uint16_t *agent, const uint8_t *evflags,
                      uint32_t n_events, cudaStream_t s);
int cs_launch_import(cs_ctx *ctx, const uint32_t *C_in, const uint16_t *cur_in, uint32_t last_agent, cudaStream_t s);
int cs_launch_survival(cs_ctx *ctx, const uint16_t *sources, uint32_t n_sources, cudaStream_t s);
int cs_launch_exact_survival(cs_ctx *ctx, uint32_t a0, uint32_t K, float *psurv_out, float *fsurv_out, cudaStream_t s);
bool cs_score_searches(const cs_ctx *ctx, uint32_t n_blocks);     // a score of so many entries can search from sources itself
int cs_launch_score(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, const float *fsurv, const uint16_t *sources,
                    uint32_t n_sources, float *scores_out, cudaStream_t s);
int cs_launch_select(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, int prefetch, uint32_t tier,
                     uint32_t k, uint32_t *ids_out, uint32_t *n_out, cudaStream_t s);
int cs_launch_select_step(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, uint32_t k_victims, uint32_t k_prefetch,
                          uint32_t *gpu_victims, uint32_t *n_gpu, uint32_t *host_victims, uint32_t *n_host,
                          uint32_t *prefetch_ids, uint32_t *n_prefetch, cudaStream_t s);
int cs_launch_select_grid(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, const uint32_t k[3], uint32_t *const ids[3],
                          uint32_t *const n_out[3], cudaStream_t s);
void cs_drop_select_graphs(cs_ctx *ctx);
int cs_launch_select_clusters(cs_ctx *ctx, int n_jobs, const void *sel_args, const uint32_t *prefetch,
                              uint32_t *const *ids_out, uint32_t *const *n_out, cudaStream_t s);
int cs_launch_select_cluster(cs_ctx *ctx, const void *sel_args, const cs_workspace *ws, int prefetch, uint32_t *ids_out,
                             uint32_t *n_out, cudaStream_t s);
int cs_launch_mover(cs_ctx *ctx, const cs_kv_pool *src, const cs_kv_pool *dst, const uint32_t *src_slots,
                    const uint32_t *dst_slots, uint32_t n_max, const uint32_t *n_dev, int kind,
                    cudaStream_t s);

int cs_launch_mover_as(cs_ctx *ctx, const cs_kv_pool *src, const cs_kv_pool *dst, const uint32_t *src_slots,
                       const uint32_t *dst_slots, uint32_t n_max, const uint32_t *n_dev, int kind, int count_as,
                       cudaStream_t s);
int cs_launch_bounded_wait_selftest(cs_ctx *ctx, uint32_t max_polls, cudaStream_t s);
int cs_launch_validate_selection(cs_ctx *ctx, const cs_block_index *idx, uint32_t now, int prefetch, uint32_t tier,
                                 uint32_t k, const uint32_t *ids, const uint32_t *n_out, cudaStream_t s);
int cs_launch_validate_lists(cs_ctx *ctx, const uint32_t *w_list, const uint32_t *w_partner, uint32_t nw_max,
                             const uint32_t *nw_dev, const uint32_t *x_list, const uint32_t *x_partner, uint32_t nx_max,
                             const uint32_t *nx_dev, int self, cudaStream_t s);
bool cs_device_can_address(const void *ptr);
void cs_release_staging(cs_ctx *ctx);

int cs_launch_exchange(cs_ctx *ctx, const cs_kv_pool *gpu, const cs_kv_pool *host, const uint32_t *off_gpu_slots,
                       const uint32_t *off_host_slots, uint32_t n_off_max, const uint32_t *n_off_dev,
                       const uint32_t *pre_host_slots, const uint32_t *pre_gpu_slots, uint32_t n_pre_max,
                       const uint32_t *n_pre_dev, cudaStream_t s);

static inline int cs_check_launch(cs_ctx *ctx)
{
    cudaError_t e = cudaGetLastError();
    ctx->n_launches++;
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return CS_ECUDA; }
    return CS_OK;
}

#ifdef __CUDACC__
// Eq. 8 with the floor of Eq. 9 added: p~ + delta of an agent so many hops away.
__device__ __forceinline__ float cs_survival_of(uint32_t hops, uint32_t e_max, float delta)
{
    const uint32_t m = hops < e_max ? hops : e_max;                        // CS_HOP_NONE > e_max by construction
    const double ptilde = 1.0 - (double)m / (double)e_max;
    return (float)(ptilde + (double)delta);
}

// Programmatic dependent launch.  The chains of small kernels (observe -> refresh; scan -> histogram ->
// collect -> sample -> place -> finish) are bound by launch latency, so each kernel of a chain is launched with the
// programmatic-serialisation attribute: its launch overlaps the tail of its predecessor, and its first
// instruction waits until the predecessor grid has completed and its writes are visible.  A kernel launched
// without the attribute executes the wait as a no-op.
#ifndef CS_USE_PDL
#define CS_USE_PDL 1
#endif
// Loads that stay where they are written.  The compiler is free to sink an ordinary load to its first use, which
// turns "fetch sixteen words, then work on them" into sixteen round trips to L2, one after the other (measured:
// 950 cycles each).  These can neither be sunk nor reordered against each other or against other memory
// operations, so a run of them is in flight together and costs one round trip.
__device__ __forceinline__ uint32_t cs_ld_cg_pinned(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint2 cs_ld_cg_pinned(const uint2 *p)
{
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint16_t cs_ld_cg_pinned(const uint16_t *p)
{
    uint16_t v;
    asm volatile("ld.global.cg.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long cs_ld_cg_pinned(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.global.cg.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 cs_ld_cg_pinned(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ ulonglong2 cs_ld_cg_pinned(const ulonglong2 *p)
{
    ulonglong2 v;
    asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void cs_wait_for_predecessor()
{
#if CS_USE_PDL
    asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}
// Lets the successor's launch proceed; called once the calling CTA no longer competes for the SM.
__device__ __forceinline__ void cs_release_successor()
{
#if CS_USE_PDL
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}

// A chained launch; cluster > 1 makes every `cluster` consecutive CTAs a thread-block cluster.  The caller reads the
// error with cs_check_launch().
template <class... KArgs, class... Args>
static inline void cs_launch_chained_clusters(void (*kernel)(KArgs...), dim3 grid, uint32_t cluster, dim3 block, size_t smem,
                                              cudaStream_t s, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = CS_USE_PDL;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster ? 2 : 1;
    (void)cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <class... KArgs, class... Args>
static inline void cs_launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args)
{
    cs_launch_chained_clusters(kernel, grid, 0u, block, smem, s, args...);
}

// Largest cluster (a power of two, at most `most`) of which `clusters_needed` fit the current device at once with this
// block size and dynamic shared memory, -1 when not even single CTAs do.  Raises the function's limits for it.
template <class Kernel>
static inline int cs_probe_cluster(Kernel kernel, int most, int threads, size_t smem, int clusters_needed)
{
    if ((smem && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return -1;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    for (int cl = most; cl >= 1; cl >>= 1) {
        cfg.gridDim = dim3(clusters_needed * cl);
        attr[0].val.clusterDim.x = cl;
        int n_clusters = 0;
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&n_clusters, kernel, &cfg);
        if (e == cudaSuccess && n_clusters >= clusters_needed) return cl;
        (void)cudaGetLastError();
    }
    return -1;
}

// Recency factor of Eq. 9 as every kernel computes it: fp64 exp and add, rounded once to fp32.
__device__ __forceinline__ float cs_recency(float lambda, float delta, uint32_t age)
{
    return (float)(exp(-(double)lambda * (double)age) + (double)delta);
}
#endif
