// Paths that cannot become PPs: their tables, and how many there are.
//
// The frontier drops an extension by w when w lies in another strongly
// connected component (SCC) than the path's last vertex and a predecessor of
// the path's first vertex is off the path: what follows w never comes back to
// the first vertex's SCC, so that predecessor stays off the path and the arc
// that would close a cycle is out of reach; nothing that begins so is prime
// (Def. 1 wants every predecessor of the first vertex on an acyclic PP).
//
// The number of simple paths is still reported exactly.  The paths dropped
// are those that begin with a dropped extension, and how a path goes on once
// it has entered an SCC does not depend on how it came there.  With M(k, y)
// the paths of k vertices that were dropped on entering y, or that continue a
// dropped path and enter y:
//   M(k, y) = D(k, y) + sum over arcs x -> y of M(k-1, x)   for x without a cycle,
// and a cyclic SCC entered at x holds, and is left by, exactly the paths that
// x's own walk of it found (x has a predecessor outside, so all its ways out
// were dropped and counted): I(j) paths of j vertices and X(j, y) ways out to y
// give I(j) M(k, x) paths of k + j - 1 vertices and add X(j, y) M(k, x) to
// M(k + j, y).  D, I and X are counted by the frontier.
//
// What it is worth (enumeration without -> with): 333-graph batch 0.84 -> 0.59
// ms, 4096-graph batch 5.92 -> 3.82, k=22 chain 1.23 -> 0.52; of a graph that
// is one SCC nearly nothing is dropped, and looking for it costs 8% (118 of
// 120 vertices in one: 0.91 -> 0.98 ms).
#include "common.cuh"
#include "doom_dev.cuh"
#include "kernels.h"

namespace tpg {

namespace {

constexpr int DOOM_BLOCK = 256;
constexpr unsigned long long DOOM_MAX = 1ull << 52;  // counts saturate here (a level of 2^31 is refused anyway)

__device__ __forceinline__ unsigned long long doom_mul(unsigned long long a, unsigned long long b) {
    if (__umul64hi(a, b)) return DOOM_MAX;
    const unsigned long long p = a * b;
    return p < DOOM_MAX ? p : DOOM_MAX;
}

__global__ void __launch_bounds__(DOOM_BLOCK) doom_tables_kernel(GraphDev g, DoomDev dm) {
    doom_tables_block<DOOM_BLOCK>(g, dm, blockIdx.x);
}

// what starts at zero, in one launch (16 bytes a thread and step)
struct ZeroArgs {
    void *p[5];
    long long n16[5];  // 16-byte words
};
__global__ void __launch_bounds__(256) zero_kernel(ZeroArgs z) {
    const long long t = blockIdx.x * 256ll + threadIdx.x, T = gridDim.x * 256ll;
#pragma unroll
    for (int i = 0; i < 5; ++i)
        for (long long k = t; k < z.n16[i]; k += T) ((int4 *)z.p[i])[k] = make_int4(0, 0, 0, 0);
}

// Counters of the entry vertices that are not zero.
struct DoomItem {
    unsigned char x, j, target, is_target;  // entry vertex, length - 1, where a dropped extension led (target number)
    unsigned count;
};
constexpr int DOOM_ITEMS = 1024, DOOM_PEND = 2048, DOOM_ROWS = 8;

// One block per graph, thread y (n <= 256 = the block), M(k, .) row by row in
// a ring of shared rows.  What bounds it is the chain of rows (one barrier
// each, two where a cyclic SCC was left), so the rows of D are loaded
// DOOM_ROWS at a time, one batch ahead, and a batch's rows are added up a
// warp per row.  4096 graphs 0.36 ms (0.50 with atomics on the lengths' sums
// and the counters read entry by entry), 333 graphs 0.08 (0.19).
__global__ void __launch_bounds__(DOOM_BLOCK) doom_count_kernel(GraphDev g, DoomDev dm, const LevelRec *levels,
                                                                int max_levels, unsigned long long *level) {
    static_assert(DOOM_BLOCK == 32 * DOOM_ROWS, "a warp per row of a batch");
    __shared__ unsigned long long s_m[DOOM_ROWS][DOOM_BLOCK + 1], s_lvl[DOOM_BLOCK + 4];  // (column DOOM_BLOCK: zero)
    __shared__ unsigned long long s_pend[DOOM_PEND];  // [row of a ring][target]: paths that leave a cyclic SCC
    __shared__ DoomItem s_item[DOOM_ITEMS];
    __shared__ int2 s_entry[DOOM_BLOCK];  // entry vertices: {vertex, offset of its counters}
    __shared__ short s_tnum[DOOM_BLOCK];
    __shared__ unsigned char s_cyc[DOOM_BLOCK];
    __shared__ int s_n, s_ents, s_targets, s_live, s_maxj, s_used;
    const int gid = blockIdx.x, y = threadIdx.x, lane = y & 31, wid = y >> 5;
    const int vb = g.vgraph ? g.vbase[gid] : 0, n = (g.vgraph ? g.vbase[gid + 1] : g.N) - vb;
    const long long tb = g.tbl_base[gid];
    unsigned long long *D = dm.D + doom_d_base(tb, vb);
    const unsigned *X = dm.X + doom_x_base(tb, gid);
    if (y == 0) s_n = s_ents = s_targets = s_live = s_maxj = s_used = 0;
    for (int r = 0; r < DOOM_ROWS; ++r) {
        s_m[r][y] = 0ull;
        if (y == 0) s_m[r][DOOM_BLOCK] = 0ull;
    }
    s_tnum[y] = -1;
    for (int k = y; k < DOOM_BLOCK + 4; k += DOOM_BLOCK) s_lvl[k] = 0ull;
    for (int k = y; k < DOOM_PEND; k += DOOM_BLOCK) s_pend[k] = 0ull;
    const int gy = vb + y;
    const unsigned f = y < n ? dm.flags[gy] : 0u;
    const int2 xi = y < n ? dm.xinfo[gy] : make_int2(-1, 0);
    const int e0 = y < n ? g.prp[gy] : 0, e1 = y < n ? g.prp[gy + 1] : 0;
    const bool cyc = f & DOOM_CYCLIC;
    s_cyc[y] = cyc;
    __syncthreads();
    // rows of D past the deepest level are zero
    for (int k = y; k < max_levels; k += DOOM_BLOCK)
        if (levels[k].count > 0) atomicMax(&s_live, k);
    if (xi.x >= 0) {
        s_entry[atomicAdd(&s_ents, 1)] = make_int2(y, xi.x);
        atomicMax(&s_used, xi.x + xi.y * (n + 1));  // (their counters lie end to end)
    }
    // this thread's acyclic predecessors (the first few in registers)
    int pr[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        pr[i] = e0 + i < e1 ? g.pcol[e0 + i] - vb : DOOM_BLOCK;
        if (pr[i] < DOOM_BLOCK && s_cyc[pr[i]]) pr[i] = DOOM_BLOCK;
    }
    __syncthreads();
    const int ents = s_ents, live = s_live, used = s_used;
#pragma unroll 8
    for (int c = y; c < used; c += DOOM_BLOCK) {
        const unsigned count = __ldcg(X + c);
        if (count == 0u) continue;
        int2 ent = s_entry[0];
        for (int i = 1; i < ents; ++i)
            if (s_entry[i].y <= c && (s_entry[i].y > ent.y || ent.y > c)) ent = s_entry[i];
        const int j = (c - ent.y) / (n + 1), to = c - ent.y - j * (n + 1), at = atomicAdd(&s_n, 1);
        if (at < DOOM_ITEMS)
            s_item[at] = DoomItem{(unsigned char)ent.x, (unsigned char)(j - 1), (unsigned char)to, (unsigned char)(to < n), count};
        if (to < n) s_tnum[to] = 0;
        atomicMax(&s_maxj, j);
    }
    __syncthreads();
    if (s_tnum[y] == 0) s_tnum[y] = (short)atomicAdd(&s_targets, 1);
    __syncthreads();
    const int items = s_n, T = s_targets;
    int ring = 1;  // rows that lie ahead of the current one: up to s_maxj
    while (ring < s_maxj + 1) ring *= 2;
    const bool listed = items <= DOOM_ITEMS && T * ring <= DOOM_PEND;  // else the counters are walked as they lie
    if (listed)
        for (int t = y; t < items; t += DOOM_BLOCK)
            if (s_item[t].is_target) s_item[t].target = (unsigned char)s_tnum[s_item[t].target];
    const int mine = listed ? s_tnum[y] : -1;
    __syncthreads();
    const int last = listed ? min(n + 1, live + 1) : n + 1;  // D's last row that may not be zero
    unsigned long long next[DOOM_ROWS];
#pragma unroll
    for (int r = 0; r < DOOM_ROWS; ++r) next[r] = y < n && 2 + r <= last ? __ldcg(D + (2 + r) * n + y) : 0ull;
    for (int k0 = 2; k0 <= n + 1; k0 += DOOM_ROWS) {
        unsigned long long row[DOOM_ROWS], any = 0ull;
#pragma unroll
        for (int r = 0; r < DOOM_ROWS; ++r) {
            row[r] = next[r];
            const int k = k0 + DOOM_ROWS + r;
            next[r] = y < n && k <= last ? __ldcg(D + k * n + y) : 0ull;
        }
#pragma unroll
        for (int r = 0; r < DOOM_ROWS; ++r) {
            const int k = k0 + r;
            if (k > n + 1) break;
            unsigned long long m = row[r];
            if (!listed && y < n) m = __ldcg(D + k * n + y);  // (earlier rows have added to it)
            if (mine >= 0) {
                unsigned long long *p = s_pend + (k & (ring - 1)) * T + mine;
                m += *p;
                *p = 0ull;
            }
            const unsigned long long *prev = s_m[(k - 1) % DOOM_ROWS];
#pragma unroll
            for (int i = 0; i < 4; ++i) m += prev[pr[i]];
            for (int e = e0 + 4; e < e1; ++e) {
                const int x = g.pcol[e] - vb;
                if (!s_cyc[x]) m += prev[x];
            }
            m = m < DOOM_MAX ? m : DOOM_MAX;
            any |= m;
            s_m[k % DOOM_ROWS][y] = m;
            __syncthreads();
            if (items == 0) continue;
            const unsigned long long *in_row = s_m[k % DOOM_ROWS];
            if (listed) {
                for (int t = y; t < items; t += DOOM_BLOCK) {
                    const DoomItem it = s_item[t];
                    const unsigned long long in = in_row[it.x];
                    if (in == 0ull) continue;
                    const unsigned long long c = doom_mul(in, it.count);
                    if (!it.is_target) {
                        if (k + it.j <= n + 1) atomicAdd(&s_lvl[k + it.j], c);
                    } else {
                        atomicAdd(&s_pend[((k + it.j + 1) & (ring - 1)) * T + it.target], c);
                    }
                }
            } else {
                for (int c0 = y; c0 < used; c0 += DOOM_BLOCK) {
                    const unsigned count = __ldcg(X + c0);
                    if (count == 0u) continue;
                    int2 ent = s_entry[0];
                    for (int i = 1; i < ents; ++i)
                        if (s_entry[i].y <= c0 && (s_entry[i].y > ent.y || ent.y > c0)) ent = s_entry[i];
                    const unsigned long long in = in_row[ent.x];
                    if (in == 0ull) continue;
                    const int j = (c0 - ent.y) / (n + 1), to = c0 - ent.y - j * (n + 1);
                    const unsigned long long c = doom_mul(in, count);
                    if (to == n && k + j - 1 <= n + 1) atomicAdd(&s_lvl[k + j - 1], c);
                    if (to < n && k + j <= n + 1) atomicAdd(D + (long long)(k + j) * n + to, c);
                }
            }
            __syncthreads();
        }
        if (k0 + wid <= n + 1) {  // this batch's acyclic paths, a warp per row
            const int k = k0 + wid;
            unsigned long long sum = 0ull;
#pragma unroll
            for (int i = 0; i < DOOM_BLOCK / 32; ++i) sum += s_cyc[lane + 32 * i] ? 0ull : s_m[k % DOOM_ROWS][lane + 32 * i];
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0 && sum) s_lvl[k] += sum;
        }
        // nothing in this batch, nothing more in D and nothing on its way
        bool more = any != 0ull || k0 + DOOM_ROWS <= last;
        if (!more && mine >= 0)
            for (int i = 0; i < ring; ++i) more |= s_pend[i * T + mine] != 0ull;
        if (!__syncthreads_or(more)) break;
    }
    for (int k = y; k <= n + 1; k += DOOM_BLOCK)
        if (s_lvl[k]) atomicAdd(level + k, s_lvl[k]);
}

}  // namespace

cudaError_t doom_tables(const GraphDev &g, const DoomDev &dm, cudaStream_t s) {
    static_assert(MASK_MAX_W * 32 <= DOOM_BLOCK, "a thread per vertex");
    if (g.W > MASK_MAX_W) return cudaErrorInvalidValue;
    doom_tables_kernel<<<g.G, DOOM_BLOCK, 0, s>>>(g, dm);
    note_launch();
    return cudaGetLastError();
}

cudaError_t enum_reset(const GraphDev &g, const DoomDev &dm, long long tbl, LevelRec *levels, int max_levels, void *ctl,
                       unsigned long long *level, cudaStream_t s) {
    ZeroArgs z{};
    z.p[0] = levels;
    z.n16[0] = (long long)sizeof(LevelRec) * max_levels / 16;
    z.p[1] = ctl;
    z.n16[1] = CTL_BYTES / 16;
    long long most = z.n16[0];
    if (dm.D) {
        // (the buffers are whole 16-byte words long)
        z.p[2] = dm.D;
        z.n16[2] = (8 * doom_d_cells(tbl, g.N) + 15) / 16;
        z.p[3] = dm.X;
        z.n16[3] = (4 * doom_x_cells(tbl, g.G) + 15) / 16;
        z.p[4] = level;
        z.n16[4] = (8ll * max_levels + 15) / 16;
        most = z.n16[2];
    }
    const long long blocks = (most + 255) / 256;
    zero_kernel<<<(unsigned)(blocks < 1216 ? blocks : 1216), 256, 0, s>>>(z);
    note_launch();
    return cudaGetLastError();
}

cudaError_t doom_count(const GraphDev &g, const DoomDev &dm, const LevelRec *levels, int max_levels,
                       unsigned long long *level, cudaStream_t s) {
    doom_count_kernel<<<g.G, DOOM_BLOCK, 0, s>>>(g, dm, levels, max_levels, level);
    note_launch();
    return cudaGetLastError();
}

}  // namespace tpg
