// Tables of the paths that are dropped (DoomDev), one block per graph.
#pragma once
#include "common.cuh"

namespace tpg {

// All BLOCK threads of a block, for graph gid of at most BLOCK vertices and
// MASK_MAX_W mask words, from its BFS tables.  What bounds it is its chain of
// dependent loads: a thread per vertex, and a warp per entry vertex for the
// sizes of their SCCs.
template <int BLOCK>
__device__ __forceinline__ void doom_tables_block(const GraphDev &g, const DoomDev &dm, int gid) {
    __shared__ int s_size[BLOCK], s_ent[BLOCK], s_ents;
    unsigned *const cmask = const_cast<unsigned *>(dm.cmask);
    unsigned char *const flags = const_cast<unsigned char *>(dm.flags);
    int2 *const xinfo = const_cast<int2 *>(dm.xinfo);
    const int W = g.W, v = threadIdx.x, lane = v & 31;
    const int vb = g.vgraph ? g.vbase[gid] : 0, n = (g.vgraph ? g.vbase[gid + 1] : g.N) - vb;
    const int *D = g.dist + g.tbl_base[gid];  // D[u * n + v] >= 0: v is reachable from u
    if (v == 0) s_ents = 0;
    s_size[v] = 0;
    __syncthreads();
    unsigned f = 0u, cm[MASK_MAX_W];
#pragma unroll
    for (int j = 0; j < MASK_MAX_W; ++j) cm[j] = 0u;
    const int gv = vb + v;
    if (v < n) {
        bool entered = false;
        const int e1 = g.rp[gv + 1], p1 = g.prp[gv + 1];
        for (int e = g.rp[gv]; e < e1; ++e) {
            const int w = g.col[e] - vb;
            if (D[w * n + v] >= 0) {
                f |= DOOM_CYCLIC;
            } else {
                f |= DOOM_LEAVES;
#pragma unroll
                for (int j = 0; j < MASK_MAX_W; ++j) cm[j] |= (w >> 5) == j ? 1u << (w & 31) : 0u;
            }
        }
        for (int e = g.prp[gv]; e < p1; ++e) entered |= D[v * n + (g.pcol[e] - vb)] < 0;
        if ((f & DOOM_CYCLIC) && entered) {
            f |= DOOM_ENTRY;
            s_ent[atomicAdd(&s_ents, 1)] = v;
        }
    }
    __syncthreads();
    // sizes of the entry vertices' SCCs
    for (int i = v >> 5; i < s_ents; i += BLOCK / 32) {
        const int x = s_ent[i];
        int size = 0;
        for (int u = lane; u < n; u += 32) size += D[x * n + u] >= 0 && D[u * n + x] >= 0;
        size = __reduce_add_sync(0xffffffffu, size);
        if (lane == 0) s_size[x] = size;
    }
    __syncthreads();
    const long long cells = (f & DOOM_ENTRY) ? (long long)(s_size[v] + 1) * (n + 1) : 0;
    long long used;
    const long long at = block_excl_scan_i64<BLOCK>(cells, used);
    // counters beyond the graph's share: nothing of this graph is dropped
    const bool fits = used <= 2ll * n * n + 1024;
    if (v < n) {
        for (int j = 0; j < W; ++j) {
            unsigned c = 0u;
#pragma unroll
            for (int i = 0; i < MASK_MAX_W; ++i) c = i == j ? cm[i] : c;
            cmask[(long long)gv * W + j] = fits ? c : 0u;
        }
        if (!fits) f &= DOOM_CYCLIC;
        flags[gv] = (unsigned char)f;
        xinfo[gv] = (f & DOOM_ENTRY) ? make_int2((int)at, s_size[v] + 1) : make_int2(-1, 0);
    }
}

}  // namespace tpg
