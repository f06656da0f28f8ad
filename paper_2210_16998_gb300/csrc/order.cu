// Canonical order of the prime paths (kernel (e) for PPs) and their
// materialisation as vertex sequences.
//
// Every level of the path arena is in lexicographic order, and the prime
// paths form an antichain of the prefix tree (a PP is never a proper prefix
// of a simple path, Def. 1).  So for two PPs x (k vertices) and y (>= k
// vertices), x < y exactly when x's index in level k is below the index of
// y's level-k ancestor.  The canonical list is built from the deepest level
// upward: the run accumulated so far is keyed by each element's ancestor
// index at the current level (one parent-link step per level), and merged
// with that level's own PPs by key.  Keys of the two inputs never tie.
#include "common.cuh"
#include "kernels.h"
#include "paths_dev.cuh"

namespace tpg {

__global__ void order_init_run_kernel(const int *pp, int level, long long n, int *keys, long long *refs) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int r = pp[i];
        keys[i] = r;
        refs[i] = ((long long)level << 32) | (unsigned)r;
    }
}

cudaError_t order_init_run(const int *pp_refs_level, int level, long long n, int *keys, long long *refs,
                           cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int grid = (int)((n + 255) / 256 < 65535 * 8 ? (n + 255) / 256 : 65535 * 8);
    order_init_run_kernel<<<grid, 256, 0, s>>>(pp_refs_level, level, n, keys, refs);
    note_launch();
    return cudaGetLastError();
}

__global__ void order_ascend_kernel(int *keys, long long n, const LevelRec *levels, int from_level, int to_level) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        int key = keys[i];
        for (int j = from_level; j > to_level; --j) key = levels[j].nodes[key].y;
        keys[i] = key;
    }
}

cudaError_t order_ascend(int *keys, long long n, const LevelRec *levels, int from_level, int to_level,
                         cudaStream_t s) {
    if (n <= 0 || from_level <= to_level) return cudaSuccess;
    const long long blocks = (n + 255) / 256;
    order_ascend_kernel<<<(unsigned)(blocks < 1 << 20 ? blocks : 1 << 20), 256, 0, s>>>(
        keys, n, levels, from_level, to_level);
    note_launch();
    return cudaGetLastError();
}

constexpr int MERGE_ITEMS = 8;

// Merge path: thread t produces outputs [t*ITEMS, t*ITEMS + ITEMS).  The
// keys of run A are stored at level from_level and lifted to level
// to_level (the level of run B) on the fly.  On equal keys A goes first
// (cannot happen between A and B here, but keeps the merge stable).
__global__ void order_merge_kernel(const int *ka, const long long *ra, long long na, const int *kb,
                                   int level_b, long long nb, int *kc, long long *rc, const LevelRec *levels,
                                   int from_level) {
    const long long total = na + nb;
    const long long diag = (blockIdx.x * (long long)blockDim.x + threadIdx.x) * MERGE_ITEMS;
    if (diag >= total) return;
    auto lift = [&](long long i) {
        int key = ka[i];
        for (int j = from_level; j > level_b; --j) key = levels[j].nodes[key].y;
        return key;
    };
    long long lo = diag > nb ? diag - nb : 0;
    long long hi = diag < na ? diag : na;
    while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        if (lift(mid) <= kb[diag - mid - 1]) lo = mid + 1;
        else hi = mid;
    }
    long long i = lo, j = diag - lo;
    int ki = (i < na) ? lift(i) : 0;
    for (int t = 0; t < MERGE_ITEMS && diag + t < total; ++t) {
        if (i < na && (j >= nb || ki <= kb[j])) {
            kc[diag + t] = ki;
            rc[diag + t] = ra[i];
            ++i;
            if (i < na) ki = lift(i);
        } else {
            const int r = kb[j];
            kc[diag + t] = r;
            rc[diag + t] = ((long long)level_b << 32) | (unsigned)r;
            ++j;
        }
    }
}

cudaError_t order_merge(const int *ka, const long long *ra, long long na, const int *kb, int level_b, long long nb,
                        int *kc, long long *rc, const LevelRec *levels, int from_level, cudaStream_t s) {
    const long long total = na + nb;
    if (total <= 0) return cudaSuccess;
    const long long threads = (total + MERGE_ITEMS - 1) / MERGE_ITEMS;
    order_merge_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(ka, ra, na, kb, level_b, nb, kc, rc, levels,
                                                                        from_level);
    note_launch();
    return cudaGetLastError();
}

__global__ void pp_lengths_kernel(const long long *refs, long long n, long long *len) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        len[i] = refs[i] >> 32;
}

cudaError_t pp_lengths(const long long *refs, long long n, long long *len_out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const long long blocks = (n + 255) / 256;
    pp_lengths_kernel<<<(unsigned)(blocks < 1 << 20 ? blocks : 1 << 20), 256, 0, s>>>(refs, n, len_out);
    note_launch();
    return cudaGetLastError();
}

__global__ void pp_offsets_single_kernel(long long *off, long long n, int level) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i <= n;
         i += (long long)gridDim.x * blockDim.x)
        off[i] = i * level;
}

cudaError_t pp_offsets_single_level(long long *off, long long n, int level, cudaStream_t s) {
    const long long blocks = (n + 1 + 255) / 256;
    pp_offsets_single_kernel<<<(unsigned)(blocks < 1 << 20 ? blocks : 1 << 20), 256, 0, s>>>(off, n, level);
    note_launch();
    return cudaGetLastError();
}

constexpr int MAT_WARPS = 8;

template <int CH, typename T>
__global__ void __launch_bounds__(MAT_WARPS * 32, 8)
    pp_materialize_kernel(const long long *refs, const int *single_refs, int single_level, long long n,
                          const long long *offsets, const LevelRec *levels, int max_levels, GraphDev g,
                          int *out, int *out_graph, int2 *out_ends) {
    __shared__ T buf[MAT_WARPS][MAT_BUF * CH];
    __shared__ int2 *s_nodes[MAT_MAX_LV];
    int2 *const *lv = cache_level_nodes(levels, max_levels, s_nodes);
    materialize_warps<MAT_WARPS, CH, T>(refs, single_refs, single_level, n, offsets, levels, g, out, out_graph, buf,
                                        lv, out_ends);
}

cudaError_t pp_materialize(const long long *refs, const int *single_refs, int single_level, long long n,
                           const long long *offsets, const LevelRec *levels, int max_levels, const GraphDev &g,
                           int *out_vertices, int *out_graph, cudaStream_t s, int2 *out_ends) {
    if (n <= 0) return cudaSuccess;
    const bool small = g.maxn <= MAT_SMALL_N;
    const long long warps = (n + (small ? 63 : 31)) / (small ? 64 : 32);
    long long blocks = (warps + MAT_WARPS - 1) / MAT_WARPS;
    if (blocks > 152 * 64) blocks = 152 * 64;
    if (small)
        pp_materialize_kernel<2, unsigned char><<<(unsigned)blocks, MAT_WARPS * 32, 0, s>>>(
            refs, single_refs, single_level, n, offsets, levels, max_levels, g, out_vertices, out_graph, out_ends);
    else
        pp_materialize_kernel<1, unsigned short><<<(unsigned)blocks, MAT_WARPS * 32, 0, s>>>(
            refs, single_refs, single_level, n, offsets, levels, max_levels, g, out_vertices, out_graph, out_ends);
    note_launch();
    return cudaGetLastError();
}

// graph_path_ptr[g] = first path index whose graph id is >= g (ids sorted).
__global__ void graph_ptr_kernel(const int *ids, long long n, int G, long long *ptr) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i <= n;
         i += (long long)gridDim.x * blockDim.x) {
        const int cur = (i < n) ? ids[i] : G;
        const int prev = (i > 0) ? ids[i - 1] : -1;
        for (int gg = prev + 1; gg <= cur; ++gg) ptr[gg] = i;
    }
}

cudaError_t graph_ptr_from_ids(const int *ids, long long n, int G, long long *ptr, cudaStream_t s) {
    const long long blocks = (n + 1 + 255) / 256;
    graph_ptr_kernel<<<(unsigned)(blocks < 1 << 20 ? blocks : 1 << 20), 256, 0, s>>>(ids, n, G, ptr);
    note_launch();
    return cudaGetLastError();
}


// ---------------------------------------------------------------------------
// PP order by place (Def. 1 makes the PPs leaves of the prefix tree)
// ---------------------------------------------------------------------------
// The arena is the prefix tree of all simple paths: level k holds the paths
// of k vertices in lexicographic order, every node points at its parent, and
// the children of a node are consecutive and ordered by their last vertex.
// Lexicographic order with a proper prefix first is the tree's pre-order, and
// a PP has no descendant (it is never a proper prefix of a simple path).  So
// the PPs before PP x = node i of level j are, in level k,
//   k < j: those before x's ancestor of that level,
//   k = j: those before i,
//   k > j: those before the place where i's descendants would be.
// The frontier leaves for every node its `place`: where its children start in
// the next level, and the PPs before it in its own level (both known to the
// warp that expands the node).  A PP's rank is then the sum of one number per
// level, read while its parent links are followed up and its child links
// down, and its first vertex's offset is the same sum with level k's number
// taken k times.  No level waits for another: what bounds it are two dependent
// chains of loads per PP (a quarter of them L2 hits), so a step's three loads
// are issued together and it runs with as many threads as an SM holds (4096
// graphs, 14.4M PPs: 4, 6, 8 blocks per SM 1.89, 1.43, 1.33 ms; with a node's
// place read after its parent link, at 6 blocks and a grid for 8, 2.88 ms).
// Order + materialise, against a bottom-up and a top-down sweep over all nodes
// with a grid barrier per level and sweep: 120-vertex CFG (15.0M nodes, 54
// levels, 1.09M PPs) 1.053 -> 0.259 ms; 333 graphs (10.1M nodes, 0.42M PPs)
// 1.01 -> 0.092 ms; 4096 graphs (196M nodes, 13.5M PPs) 4.40 -> 3.64 ms; the
// frontier writes 8 more bytes per node (k=22 chain, 67M nodes: 1.14 -> 1.23 ms).
struct PlaceLevel {
    const int2 *nodes, *place;
    const int *pp;
    long long pp_before;  // PPs of the levels before this one
    int count, pp_count;
};
constexpr int PLACE_BLOCK = 256, PLACE_BLOCKS_SM = 8;

__global__ void __launch_bounds__(PLACE_BLOCK, PLACE_BLOCKS_SM) place_pps_kernel(PlaceArgs a) {
    extern __shared__ __align__(16) unsigned char place_smem[];
    __shared__ int s_L;
    PlaceLevel *lv = (PlaceLevel *)place_smem;  // [max_levels], level 0 unused
    if (a.skip && (*a.skip & a.skip_mask)) return;
    // the level table, PPs before every level, the deepest level
    if (threadIdx.x == 0) s_L = 0;
    __syncthreads();
    long long carry = 0;
    for (int base = 0; base < a.max_levels; base += PLACE_BLOCK) {
        const int k = base + threadIdx.x;
        LevelRec r = {};
        if (k >= 1 && k < a.max_levels) r = a.levels[k];
        const long long c = r.count > 0 ? r.pp_count : 0;
        long long tot;
        const long long ex = block_excl_scan_i64<PLACE_BLOCK>(c, tot);
        if (k < a.max_levels) {
            lv[k] = PlaceLevel{r.nodes, r.place, r.pp, carry + ex, (int)r.count, (int)c};
            if (r.count > 0) atomicMax(&s_L, k);
        }
        carry += tot;
    }
    __syncthreads();
    const int L = s_L;
    const long long P = carry;
    if (P > a.cap) return;  // (the caller has seen it)
    for (long long t = blockIdx.x * (long long)PLACE_BLOCK + threadIdx.x; t < P;
         t += (long long)gridDim.x * PLACE_BLOCK) {
        int lo = 1, hi = L;  // the last level with pp_before <= t holds PP t
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (lv[mid].pp_before <= t) lo = mid;
            else hi = mid - 1;
        }
        const int j = lo, idx = lv[j].pp[(int)(t - lv[j].pp_before)];
        long long rank = 0, off = 0;
        // ku: the level of `up`, whose place and parent load together; kd: that of `down`
        int up = idx, down = 0, ku = j, kd = L + 1;
        {
            const int2 pl = lv[j].place[up];
            if (j > 1) up = lv[j].nodes[up].y;
            rank = pl.y;
            off = (long long)pl.y * j;
            down = pl.x;
            ku = j - 1;
            kd = j + 1;
        }
        while (ku >= 1 || kd <= L) {
            int parent = 0;
            int2 pu = make_int2(0, 0), pd = pu;
            if (ku >= 1) {
                pu = lv[ku].place[up];
                if (ku > 1) parent = lv[ku].nodes[up].y;
            }
            if (kd <= L) {
                if (down < lv[kd].count) pd = lv[kd].place[down];
                else pd = make_int2(kd < L ? lv[kd + 1].count : 0, lv[kd].pp_count);  // past the level's end
            }
            rank += pu.y + (long long)pd.y;
            off += (long long)pu.y * ku + (long long)pd.y * kd;
            up = parent;
            down = pd.x;
            --ku;
            ++kd;
        }
        a.refs[rank] = ((long long)j << 32) | (unsigned)idx;
        a.off[rank] = off;
        if (rank == P - 1) a.off[P] = off + j;
    }
    if (P == 0 && blockIdx.x == 0 && threadIdx.x == 0) a.off[0] = 0;
}

cudaError_t place_pps(const PlaceArgs &a, int num_sms, cudaStream_t s) {
    const size_t smem = sizeof(PlaceLevel) * (size_t)a.max_levels;
    if (smem > 40 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(place_pps_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const long long need = (a.cap + PLACE_BLOCK - 1) / PLACE_BLOCK;
    const long long fit = (long long)PLACE_BLOCKS_SM * num_sms;
    const long long grid = need < 1 ? 1 : need < fit ? need : fit;
    place_pps_kernel<<<(unsigned)grid, PLACE_BLOCK, smem, s>>>(a);
    note_launch();
    return cudaGetLastError();
}

}  // namespace tpg
