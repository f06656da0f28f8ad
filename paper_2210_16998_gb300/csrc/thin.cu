// Prime paths of thin graphs: a depth-first walk per first vertex.
//
// A level of the frontier (enumerate.cu) costs a grid barrier and two dependent
// rounds over its paths, 7 us however few there are, and a wide graph can have
// thousands of levels with about one path per first vertex in each (a long
// function whose loops follow one another).  There every first vertex's paths
// are walked depth-first by a warp of its own: the path, where each of its
// vertices stands among its arcs, and the visited set lie in shared memory, 32
// arcs are looked at together, and successors in ascending order make the walk
// canonical (Alg. 2-4 with the tree's pre-order; a proper prefix comes first).
// The first launch counts (paths and PPs by length, PPs by first vertex), the
// second walks again and writes each PP at its place; nothing else is stored.
//
// What bounds it is the longest walk's chain of dependent reads (0.25 us a
// vertex; an exhausted path goes straight back to its last branch point, and
// paths are counted a descent at a time), so it is for trees that are hardly more than one path: a walk that
// has taken more than THIN_SLACK + 2 x (its deepest path) vertices ends the
// attempt, and the frontier takes over.  That is soon where paths multiply:
// the deepest path comes first, and the frontier needs a level for each of its
// vertices, many times what the walk spent on it.
//
// Enumeration, order and materialisation, frontier -> walks: 1100-vertex chain
// of 110 loops 9.0 -> 0.57 ms, one of 1500 15.2 -> 0.86, a ring of 2000 40.4 ->
// 2.2, a chain of 300 1.76 -> 0.23; an attempt that is given up costs 0.1 ms of
// 5.8 (2^16 PPs of 349 vertices).
#include "common.cuh"
#include "kernels.h"

namespace tpg {

namespace {

constexpr int THIN_SLACK = 24;

size_t thin_smem(int maxn) {
    const size_t n = (size_t)maxn + 2;
    return 4 * (2 * n + n / 2 + 1 + (n + 31) / 32);
}

template <bool WRITE>
__global__ void __launch_bounds__(32) thin_walk_kernel(ThinArgs a) {
    extern __shared__ unsigned thin_shared[];
    const GraphDev &g = a.g;
    const int root = blockIdx.x, lane = threadIdx.x;
    if (!WRITE && *(volatile int *)a.stop) return;
    const int n2 = g.maxn + 2;
    int *next = (int *)thin_shared;                         // [k] branch points: next arc of vertex k
    int *below = next + n2;                                 // [k] and the branch point before
    unsigned short *path = (unsigned short *)(below + n2);  // [k] local ids
    unsigned *vis = thin_shared + 2 * n2 + n2 / 2 + 1;      // visited set
    const int gid = g.vgraph ? g.vgraph[root] : 0;
    const int vb = g.vgraph ? g.vbase[gid] : 0, n = (g.vgraph ? g.vbase[gid + 1] : g.N) - vb;
    const int first = root - vb, p0 = g.prp[root], p1 = g.prp[root + 1];
    for (int w = lane; w < (n + 31) / 32; w += 32) vis[w] = w == first >> 5 ? 1u << (first & 31) : 0u;
    if (lane == 0) path[0] = (unsigned short)first;
    __syncwarp();
    int e = g.rp[root], e1 = g.rp[root + 1];  // arcs left of the last vertex
    bool leaf = true;                         // the path has not been extended
    int k = 1, taken = 1, deepest = 1;        // vertices on the path; in all; on the deepest path
    int run = 1;                              // paths of run .. k vertices are to be counted (0: none)
    int top = -1;                             // last branch point below the last vertex
    long long pps = 0, ppv = 0;
    if (WRITE) {
        pps = a.pp_at[root];
        ppv = a.ppv_at[root];
    }
    // paths of lo .. hi vertices, one each (a.paths holds differences)
    auto count = [&](int lo, int hi) {
        if (lane == 0) {
            atomicAdd((unsigned long long *)a.paths + lo, 1ull);
            atomicAdd((unsigned long long *)a.paths + hi + 1, ~0ull);
        }
    };
    // the path's k vertices (closed: and the first again) are a PP
    auto found = [&](bool closed) {
        const int len = k + (closed ? 1 : 0);
        if (WRITE) {
            if (lane == 0) {
                a.off[pps] = ppv;
                if (a.pgraph) a.pgraph[pps] = gid;
                a.ends[pps] = make_int2(first, closed ? first : path[k - 1]);
                if (closed) a.vert[ppv + k] = first;
            }
#pragma unroll 4
            for (int i = lane; i < k; i += 32) a.vert[ppv + i] = path[i];
        } else {
            if (lane == 0) atomicAdd((unsigned long long *)a.pps + len, 1ull);
            if (closed) count(len, len);
        }
        ++pps;
        ppv += len;
    };
    for (;;) {
        // the first arc left that extends or closes the path
        const int x = e + lane < e1 ? __ldg(g.col + e + lane) - vb : -1;
        const unsigned m = __ballot_sync(0xffffffffu, x >= 0 && (x == first || !(vis[x >> 5] >> (x & 31) & 1u)));
        if (m) {
            const int at = __ffs(m) - 1, w = __shfl_sync(0xffffffffu, x, at);
            e += at + 1;
            leaf = false;
            if (w == first) {
                found(true);
                continue;
            }
            if (lane == 0) {
                path[k] = (unsigned short)w;
                vis[w >> 5] |= 1u << (w & 31);
                if (e < e1) {
                    next[k - 1] = e;
                    below[k - 1] = top;
                }
            }
            if (e < e1) top = k - 1;
            e = __ldg(g.rp + vb + w);
            e1 = __ldg(g.rp + vb + w + 1);
            leaf = true;
            ++k;
            ++taken;
            if (run == 0) run = k;
            deepest = k > deepest ? k : deepest;
            __syncwarp();
            if (!WRITE) {
                bool stop = taken > THIN_SLACK + 2 * deepest;
                if (stop && lane == 0) *(volatile int *)a.stop = 1;
                if ((taken & 63) == 0) stop |= *(volatile int *)a.stop != 0;
                if (__any_sync(0xffffffffu, stop)) return;
            }
            continue;
        }
        if (e + 32 < e1) {
            e += 32;
            continue;
        }
        if (leaf) {  // prime iff every predecessor of the first vertex is on the path
            bool off = false;
            for (int i = p0 + lane; i < p1; i += 32) {
                const int y = __ldg(g.pcol + i) - vb;
                off |= !(vis[y >> 5] >> (y & 31) & 1u);
            }
            if (!__any_sync(0xffffffffu, off)) found(false);
        }
        if (!WRITE && run) count(run, k);
        run = 0;
        if (top < 0) break;
        // back to the last branch point
        for (int i = top + 1 + lane; i < k; i += 32) {
            const int y = path[i];
            atomicAnd(vis + (y >> 5), ~(1u << (y & 31)));
        }
        k = top + 1;
        e = next[top];
        e1 = __ldg(g.rp + vb + path[top] + 1);
        top = below[top];
        leaf = false;
        __syncwarp();
    }
    if (lane == 0) {
        if (!WRITE) {
            a.root_pp[root] = pps;
            a.root_ppv[root] = ppv;
        } else if (root == g.N - 1) {
            a.off[pps] = ppv;
        }
    }
}

}  // namespace

cudaError_t thin_count(const ThinArgs &a, cudaStream_t s) {
    thin_walk_kernel<false><<<a.g.N, 32, thin_smem(a.g.maxn), s>>>(a);
    note_launch();
    return cudaGetLastError();
}

cudaError_t thin_write(const ThinArgs &a, cudaStream_t s) {
    thin_walk_kernel<true><<<a.g.N, 32, thin_smem(a.g.maxn), s>>>(a);
    note_launch();
    return cudaGetLastError();
}

}  // namespace tpg
