// Internal kernel entry points of libtpg (host-callable launchers).
#pragma once
#include <cuda_runtime.h>

#include <atomic>

#include "common.cuh"
#include "tp_order_dev.cuh"

namespace tpg {

// kernels launched by this library in this process (tpg_kernel_launches)
extern std::atomic<long long> g_kernel_launches;
inline void note_launch(int n = 1) { g_kernel_launches.fetch_add(n, std::memory_order_relaxed); }

// per-chunk level counts of the frontier launch: a level is cut into
// ENUM_UPW chunks per warp of the launch (CPG = ENUM_UPW x warps per block
// chunks per block); 3 rotating slots of {children, PPs} per chunk and per
// block.  enum_agg_words(grid, CPG) int64 values hold them for one launch;
// enum_agg_words_max(num_sms) for any tile shape on that GPU (at most 64
// warps and 8 blocks per SM).
#ifndef TPG_ENUM_UPW
#define TPG_ENUM_UPW 4
#endif
constexpr int ENUM_UPW = TPG_ENUM_UPW;
constexpr long long enum_agg_words(long long grid, long long cpg) { return 3 * (2 * cpg * grid + 2 * grid) + 4; }
constexpr long long enum_agg_words_max(long long num_sms) {
    return 3 * (2 * ENUM_UPW * 64 * num_sms + 2 * 8 * num_sms) + 4;
}
// frontier count word of a path: bits 0-12 are the mask of the successors of
// its last vertex that extend it (successor list position s -> bit s; lists
// of at most CNT_MASK_DEG successors), or, with CNT_WIDE set, the number of
// such successors (at most TPG_MAX_N); CNT_PP flags a prime path
constexpr unsigned CNT_BITS = 0x1fffu;
constexpr unsigned CNT_WIDE = 0x4000u;
constexpr unsigned CNT_PP = 0x8000u;
constexpr int CNT_MASK_DEG = 13;
__host__ __device__ inline int cnt_children(unsigned cw) {
#ifdef __CUDA_ARCH__
    return (cw & CNT_WIDE) ? (int)(cw & CNT_BITS) : __popc(cw & CNT_BITS);
#else
    return (cw & CNT_WIDE) ? (int)(cw & CNT_BITS) : __builtin_popcount(cw & CNT_BITS);
#endif
}
// count word of a path that is evaluated with the vertex bitsets: bits 0-9
// are the number of its children, CNT_ON says that every predecessor of its
// first vertex is on it (it may be clear although they are), CNT_DOOM that it
// has dropped extensions, CNT_ENTRY that its first vertex is a DOOM_ENTRY one
constexpr unsigned CNT_MASK_BITS = 0x3ffu;
constexpr unsigned CNT_ENTRY = 0x800u;
constexpr unsigned CNT_ON = 0x1000u;
constexpr unsigned CNT_DOOM = 0x2000u;
// control block of a launch (err, stop_level, ...); the frontier's grid
// barrier lives at CTL_BAR_OFFSET
constexpr int CTL_BYTES = 1024;
constexpr int CTL_BAR_OFFSET = 256;
constexpr int CTL_HANDOFF_OFFSET = 64;    // level a frontier launch's single-block start hands to the grid

struct EnumArgs {
    GraphDev g;
    DoomDev dm;
    int2 *seg;               // current arena segment (nodes {last, parent})
    long long seg_cap;
    int2 *seg_place;         // the segment's places, node i's at [i] (null: not kept; see place_pps)
    int2 *next_nodes;        // where level start_level+1 starts (null: right after level start_level)
    int *pp_seg;             // current PP-reference segment
    long long pp_seg_cap;
    int2 *tfl[2];            // ping-pong {first, last}
    unsigned *tvis[2];       // ping-pong bitsets, W word-arrays of lvl_cap each
    unsigned short *tcnt[2]; // ping-pong count words (children | PP flag)
    long long lvl_cap;
    LevelRec *levels;        // [max_levels]
    int max_levels;
    int start_level;         // first level processed by this launch
    int seed_level1;         // 1 on a fresh run: level 1 is written first (never on a resume)
    int split;               // work units per chunk in the per-warp levels (1..4; results never depend on it)
    long long *agg;          // per-block level counts (no initialisation needed)
    long long agg_cap;       // int64 values in agg (enum_agg_words(grid, chunks per block) at least)
    int *err;                // error flags (zeroed)
    int *stop_level;         // level whose next level did not fit (written with the flags)
    unsigned *bar;           // grid barrier: bar[0] is its arrival counter (zeroed)
    unsigned long long *root_counts;  // optional [3*N]: per first vertex, simple paths, PPs, PP vertices
    unsigned long long spin_ns;       // limit of every grid-barrier wait (SPIN_LIMIT_NS unless set)
    unsigned long long *trace;        // optional [LEVEL_TRACE_WORDS * max_levels] per-level timing
    int *handoff;            // optional: on a fresh run, block 0 walks the small first levels alone and
                             // leaves here the level the grid starts at (null: the grid does every level)
};
// per-level trace of a frontier launch, 4 words per level: ~(earliest block
// start), latest warp end, summed busy time of the warps with work, number
// of those warps (globaltimer nanoseconds; zeroed before the launch)
constexpr int LEVEL_TRACE_WORDS = 4;

// enumerate.cu
struct EnumShape {
    int block;  // threads per block
    int items;  // paths per thread; a tile is block * items consecutive paths
};
int bitset_words_supported(int maxn);
bool enum_shape_supported(int W, EnumShape shape);
EnumShape default_enum_shape(int W);
// level capacity of the ping-pong frontier: a multiple of 2048 paths (tiles
// and bulk copies stay 16-byte aligned), at least x, below 2^31 - 1
long long round_frontier_cap(long long x);
cudaError_t launch_enumerate(const EnumArgs &args, EnumShape shape, int num_sms, cudaStream_t s, int *grid_out);
// level 1 of a fresh run (one path per vertex)
cudaError_t launch_seed_level1(const EnumArgs &args, cudaStream_t s);
// copy the first `count` frontier records to buffers of another capacity
cudaError_t relayout_frontier(const int2 *fl_old, const unsigned *vis_old, long long cap_old, int2 *fl_new,
                              unsigned *vis_new, long long cap_new, long long count, int W, cudaStream_t s);

// scan.cu: exclusive scan of int64 (in may equal out); tmp must hold
// scan_tmp_elems(n) int64 values.  out[n] receives the total.
size_t scan_tmp_elems(long long n);
cudaError_t scan_i64(const long long *in, long long *out, long long n, long long *tmp, cudaStream_t s);
// scan_i64 in two halves: the total first (at tmp[scan_total_index(n)]),
// the prefix array only when it is needed
cudaError_t scan_i64_sums(const long long *in, long long n, long long *tmp, cudaStream_t s);
long long scan_total_index(long long n);
cudaError_t scan_i64_finish(const long long *in, long long *out, long long n, const long long *tmp, cudaStream_t s);
// exclusive scan of int32 inputs into int64 outputs (out[n] = total)
cudaError_t scan_i32_to_i64(const int *in, long long *out, long long n, long long *tmp, cudaStream_t s);

// doomed.cu
// tables of every graph (cmask, flags, xinfo), from the BFS tables
cudaError_t doom_tables(const GraphDev &g, const DoomDev &dm, cudaStream_t s);
inline long long doom_d_cells(long long tbl, long long N) { return tbl + 2 * N; }
inline long long doom_x_cells(long long tbl, long long G) { return 2 * tbl + 1024 * G; }
// zero before an enumeration: `levels` (level_bytes), `ctl` (CTL_BYTES) and,
// if dm counts, its counters and level[max_levels]
cudaError_t enum_reset(const GraphDev &g, const DoomDev &dm, long long tbl, LevelRec *levels, int max_levels, void *ctl,
                       unsigned long long *level, cudaStream_t s);
// the dropped paths of every length (level[], added to) after a finished
// enumeration; D is used up
cudaError_t doom_count(const GraphDev &g, const DoomDev &dm, const LevelRec *levels, int max_levels,
                       unsigned long long *level, cudaStream_t s);

// thin.cu
// Walks of thin graphs.  thin_count: paths (as differences: their running sums)
// and PPs by number of vertices (zero before), PPs and their vertices by first vertex, or *stop (zero before) is set
// and nothing else is of use; thin_write: the PPs, from the prefixes of the
// latter two.
struct ThinArgs {
    GraphDev g;
    int *stop;
    long long *paths, *pps;              // [max_levels]
    long long *root_pp, *root_ppv;       // [N]
    const long long *pp_at, *ppv_at;     // [N + 1] their prefixes
    long long *off;                      // [PPs + 1]
    int *vert, *pgraph;                  // pgraph may be null
    int2 *ends;                          // (first, last) local vertex of each PP
};
cudaError_t thin_count(const ThinArgs &a, cudaStream_t s);
cudaError_t thin_write(const ThinArgs &a, cudaStream_t s);

// order.cu
// canonical ordering of PP references across levels (ancestor-index merge)
cudaError_t order_init_run(const int *pp_refs_level, int level, long long n, int *keys,
                           long long *refs, cudaStream_t s);
cudaError_t order_ascend(int *keys, long long n, const LevelRec *levels, int from_level, int to_level,
                         cudaStream_t s);
cudaError_t order_merge(const int *ka, const long long *ra, long long na, const int *kb, int level_b,
                        long long nb, int *kc, long long *rc, const LevelRec *levels, int from_level,
                        cudaStream_t s);
cudaError_t pp_lengths(const long long *refs, long long n, long long *len_out, cudaStream_t s);
cudaError_t pp_offsets_single_level(long long *off, long long n, int level, cudaStream_t s);
// out_graph and out_ends (optional) receive each PP's graph id and its
// (first, last) local vertex.
cudaError_t pp_materialize(const long long *refs, const int *single_refs, int single_level, long long n,
                           const long long *offsets, const LevelRec *levels, int max_levels, const GraphDev &g,
                           int *out_vertices, int *out_graph, cudaStream_t s, int2 *out_ends = nullptr);
cudaError_t graph_ptr_from_ids(const int *ids, long long n, int G, long long *ptr, cudaStream_t s);

// canonical PP order: every PP's place from the arena's nodes and places (one
// launch without waiting between blocks; all level sizes are read from the
// device level table)
struct PlaceArgs {
    const LevelRec *levels;
    int max_levels;
    long long *refs;      // [cap]: the sorted PP references (level << 32 | index)
    long long *off;       // [cap + 1]: first vertex of every PP, then the total
    long long cap;
    const int *skip;      // optional: nothing is done when (*skip & skip_mask)
    int skip_mask;
};
cudaError_t place_pps(const PlaceArgs &a, int num_sms, cudaStream_t s);

// graphmode.cu: the device-driven pipeline captured into a CUDA graph
enum : int {
    GM_ENUM_FAILED = 1,  // the frontier launch stopped (capacity) or failed
    GM_OVF_PP = 2,       // more PPs than P_cap
    GM_OVF_PPV = 4,      // more PP vertices than V_cap
    GM_UNREACH = 8,      // a PP cannot be toured
    GM_TIMEOUT = ERR_TIMEOUT,  // a bounded grid barrier ran out (the barrier ORs this bit)
    GM_OVF_TPV0 = 32,    // more TP vertices (before dedup) than TV0_cap
    GM_OVF_TPV = 64,     // more TP vertices (after dedup) than TV_cap
};
static_assert(GM_TIMEOUT == 16, "flag bits must stay distinct");
struct GmCounts {
    long long P, V, TV0, T, TV;
    int flags;
};
struct GmArgs {
    GraphDev g;
    const LevelRec *levels;
    int max_levels;
    const int *enum_err;
    long long P_cap, V_cap, TV0_cap, TV_cap;
    int num_sms, tp_rounds;
    long long *refs;        // [P_cap] the ordered PPs: level << 32 | node
    long long *len;         // [P_cap]
    long long *scan_tmp;    // gm_scan_tmp_elems(P_cap)
    long long *pp_off;      // [P_cap+1]
    int *pp_vert;           // [V_cap]
    int *pp_graph;          // [P_cap] (batches)
    long long *pp_gptr;     // [G+1]
    long long *tp_len;      // [P_cap]
    long long *tp_off0;     // [P_cap+1]
    long long *key_off;     // [P_cap+1] word offsets of the packed TP keys
    unsigned long long *key;  // [K_cap] packed TP keys
    long long K_cap;
    int key_bits;           // 8 (graphs of <= 255 vertices) or 16
    TpOrder order;          // the TPs' order (arrays for P_cap TPs)
    long long slots;        // TP slots of all graphs
    int *keep;              // [P_cap]
    long long *keep_off, *keep_rank;  // [P_cap+1]
    long long *tp_off;      // [P_cap+1]
    int *tp_vert;           // [TV_cap]
    int *tp_graph;          // [P_cap]
    long long *tp_gptr;     // [G+1]
    GmCounts *counts;
};
int gm_tp_rounds(int maxn);
size_t gm_scan_tmp_elems(long long n_cap);
cudaError_t gm_enqueue_pp(const GmArgs &a, cudaStream_t s);
cudaError_t gm_enqueue_tp(const GmArgs &a, cudaStream_t s);

// sizer.cu: the learned sizer's network
struct SizerNet;
struct SzGraph {
    long long N;
    const int *rp, *col, *prp, *pcol;  // successor / predecessor CSR (global ids)
    const float *X;                    // [N][8] features
    const float *T;                    // [N][3] targets (training only)
};
int sz_param_count();
int sz_features_per_vertex();
int sz_targets();
SizerNet *sz_create(unsigned long long seed, cudaStream_t s, int num_sms);
void sz_destroy(SizerNet *n);
cudaError_t sz_set_params(SizerNet *n, const float *host);
cudaError_t sz_get_params(SizerNet *n, float *host);
cudaError_t sz_get_grads(SizerNet *n, float *host);
cudaError_t sz_features(const GraphDev &g, float *X, cudaStream_t s, int num_sms);
cudaError_t sz_labels(const unsigned long long *counts, long long N, float *T, cudaStream_t s, int num_sms);
cudaError_t sz_forward(SizerNet *n, const SzGraph &b);
cudaError_t sz_loss_backward(SizerNet *n, const SzGraph &b, double *loss_host);
cudaError_t sz_adam_step(SizerNet *n, float lr);
cudaError_t sz_predict(SizerNet *n, const SzGraph &b, float *Y_host, double *totals_host);
cudaError_t sz_log_totals(SizerNet *n, const float *Y, long long N, double *totals_host);
// device allocator of the library (api.cu)
void *lib_dev_alloc(size_t bytes, cudaStream_t s);
void lib_dev_free(void *p, cudaStream_t s);

// preprocess.cu
cudaError_t build_union_csr(const int *unused, const long long *rp_base_dev,
                            const long long *arc_base_dev, const int *rp_cat, const int *col_cat,
                            int G, int N, long long M, int *rp, int *col, int *vgraph, int *vbase_out,
                            cudaStream_t s);
cudaError_t validate_csr_device(const int *rp, const int *col, int n, long long m, int entry, int exit,
                                int *err, cudaStream_t s);
cudaError_t build_pred_csr(const GraphDev &g, int *prp, int *pcol, int *indeg_tmp, long long *scan_tmp,
                           long long *scan_buf, cudaStream_t s);
// gate (optional): a device flag; the BFS does nothing when it is nonzero.
cudaError_t bfs_all_pairs(const GraphDev &g, cudaStream_t s, const int *gate);
// One graph of at most PREP_SMALL_N vertices: optional CSR validation (sets
// ERR_INVAL in *err, which must be zero on entry, and skips the rest), the
// predecessor CSR, tbl_base, the BFS tables and the tour tables in three
// launches; g.pre_seq / g.suf_seq must hold N(N+1)/2 entries each.  The TP
// slots (tree_slots_block) as well and, with masks (at most 256 vertices), the
// masks and the tables of dm.
constexpr int PREP_SMALL_N = 1024;
cudaError_t preprocess_small(const GraphDev &g, int *prp, int *pcol, long long *tbl_base, bool validate, int entry,
                             int exit, int *err, cudaStream_t s, int *arc_slot, int *end_slot, unsigned *smask = nullptr,
                             unsigned *pmask = nullptr, const DoomDev &dm = DoomDev{});
// successor / predecessor bitsets of every vertex (GraphDev::smask, pmask),
// W <= MASK_MAX_W; nothing is done while *gate is nonzero (gate optional)
cudaError_t build_vertex_masks(const GraphDev &g, unsigned *smask, unsigned *pmask, const int *gate, cudaStream_t s);
cudaError_t tour_lengths(const GraphDev &g, long long *scan_tmp, cudaStream_t s);
cudaError_t tour_fill(const GraphDev &g, cudaStream_t s);

// testpaths.cu
cudaError_t tp_lengths(const long long *pp_off, const int2 *pp_ends, const int *pp_graph, long long P,
                       const GraphDev &g, long long *tp_len, int *err, unsigned long long *runs, cudaStream_t s);
cudaError_t tp_write(const long long *pp_off, const int *pp_vert, const int *pp_graph, long long P,
                     const GraphDev &g, const long long *tp_off, int *tp_vert, cudaStream_t s);
cudaError_t tp_iota(long long *perm, long long P, cudaStream_t s);
cudaError_t tp_gather(const long long *perm, const int *keep, const long long *keep_rank, long long P,
                      const long long *tp_off, const int *tp_vert, const int *tp_graph,
                      const long long *keep_off, long long *final_off, int *out_vert, int *out_graph,
                      cudaStream_t s);

}  // namespace tpg
