// Canonical order of the test paths (TPs): device code shared by the
// host-driven and the graph-captured pipelines.
//
// TP(p) starts with path(entry -> first p), a path of the entry's BFS tree, and
// follows the tree further until it takes an arc that is not in it (or ends).
// That arc is the TP's slot.  Slots are leaves of the tree with the other arcs
// hung on: no slot's vertices are a prefix of another's, so TPs of different
// slots compare as the slots do, and the slots' order is known from the graph
// alone (tree_slots_block).  PPs come in canonical order, so the TPs of one
// first vertex (a run) are sorted and those of one slot in it lie together: the
// list is a few sorted sub-runs, which are put down slot by slot; only slots
// reached from several first vertices are merged, in ceil(log2(sub-runs))
// rounds, by packed keys from the slot's own vertices on.  Half of the TPs of
// a 4096-graph batch need no merge, and the rest 2.6 rounds on average, where
// merging a graph's runs takes up to 8 for all of them.
#pragma once
#include "paths_dev.cuh"

namespace tpg {

// The slots of graph gid, all BLOCK threads of a block, in s[0 .. 3n) of shared
// memory: arc_slot[e] numbers the arcs outside the entry's BFS tree, end_slot
// the end of a TP at the exit, by their place in the tree's pre-order (a TP
// that ends first, then by arc head).  A vertex's number is the sum of what
// lies before it along its tree path: each thread walks up from its vertices,
// n * depth steps in shared memory.
template <int BLOCK>
__device__ __forceinline__ void tree_slots_block(const GraphDev &g, int gid, int *arc_slot, int *end_slot, int *s) {
    const int vb = g.vgraph ? g.vbase[gid] : 0, n = (g.vgraph ? g.vbase[gid + 1] : g.N) - vb;
    const int en = g.entry[gid] - vb;
    const int *prow = g.pred + g.tbl_base[gid] + (long long)en * n;
    const int *drow = g.dist + g.tbl_base[gid] + (long long)en * n;
    int *par = s, *leaves = s + n, *before = s + 2 * n;
    for (int v = threadIdx.x; v < n; v += BLOCK) {
        par[v] = v != en && drow[v] >= 0 ? prow[v] : -1;
        leaves[v] = before[v] = 0;
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += BLOCK) {
        int own = 1;
        for (int e = g.rp[vb + v]; e < g.rp[vb + v + 1]; ++e) own += par[g.col[e] - vb] != v;
        for (int a = v; a >= 0; a = par[a]) atomicAdd(leaves + a, own);
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += BLOCK) {
        int at = 1;
        for (int e = g.rp[vb + v]; e < g.rp[vb + v + 1]; ++e) {
            const int w = g.col[e] - vb;
            if (par[w] == v) {
                before[w] = at;
                at += leaves[w];
            } else {
                ++at;
            }
        }
    }
    __syncthreads();
    for (int v = threadIdx.x; v < n; v += BLOCK) {
        int at = 0;
        for (int a = v; par[a] >= 0; a = par[a]) at += before[a];
        if (vb + v == g.exit[gid]) end_slot[gid] = at;
        ++at;
        for (int e = g.rp[vb + v]; e < g.rp[vb + v + 1]; ++e) {
            const int w = g.col[e] - vb;
            if (par[w] == v) {
                at += leaves[w];
                arc_slot[e] = -1;
            } else {
                arc_slot[e] = at++;
            }
        }
    }
}

// Everything the ordering works on.  `slot` below is global: graph gid's
// slots start at (arcs + vertices of the graphs before it).
struct TpOrder {
    GraphDev g;
    const long long *pp_off;  // the PPs
    const int *pp_vert, *pp_graph;
    const int *arc_slot, *end_slot;
    int *start;               // [P] a sub-run starts here
    long long *sub_rank;      // [P + 1] its exclusive prefix
    long long *sub_start;     // [sub-runs + 1] first TP (in PP order)
    int2 *sub_slot;           // [sub-runs] {slot, key words that all of its TPs share}
    unsigned long long *sub_at;  // [sub-runs] within the slot: sub-runs before << 32 | TPs before
    long long *slot_n, *slot_at; // [slots], [slots + 1]: sub-runs << 32 | TPs, and the prefix
    longlong2 *sub_dst;       // [sub-runs] {first position, number in slot order | merge rounds << 32}
    long long *bounds;        // [sub-runs + 1] first position, in slot order
    int4 *sub_info;           // [sub-runs] in slot order {first of the slot, sub-runs of the slot, shared words, -}
    int *pos_sub;             // [P] sub-run (in slot order) at each position
    int *max_k;               // most sub-runs of a slot (zero before)
    long long *perm[2];       // [P] TPs by position; the order ends up in perm[0]
    const long long *key_off;
    const unsigned long long *key;
    int bits;
};

// ceil(log2(k)): rounds that merge k sub-runs
__host__ __device__ inline int merge_rounds(long long k) {
    int r = 0;
    while ((1ll << r) < k) ++r;
    return r;
}

// slot of TP(PP i); *len = vertices of the TP up to and including the slot's
__device__ __forceinline__ int tp_slot_of(const TpOrder &o, long long i, int *len) {
    const GraphDev &g = o.g;
    const long long o0 = o.pp_off[i], o1 = o.pp_off[i + 1];
    const int gid = o.pp_graph ? o.pp_graph[i] : 0;
    const int vb = g.vgraph ? g.vbase[gid] : 0, n = (g.vgraph ? g.vbase[gid + 1] : g.N) - vb;
    const int *prow = g.pred + g.tbl_base[gid] + (long long)(g.entry[gid] - vb) * n;
    // along seq[p .. end) as long as its arcs are the tree's, four at a time (a
    // step is two dependent loads); y: the vertex that another arc leads to
    int x = o.pp_vert[o0], y = -1;
    auto follow = [&](const int *seq, long long p, long long end) {
        for (; p < end && y < 0; p += 4) {
            int v[4], pr[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = p + j < end ? seq[p + j] : -1;
#pragma unroll
            for (int j = 0; j < 4; ++j) pr[j] = v[j] >= 0 ? prow[v[j]] : -1;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (y >= 0 || v[j] < 0) continue;
                if (pr[j] == x) x = v[j];
                else y = v[j];
            }
        }
    };
    follow(o.pp_vert, o0 + 1, o1);
    if (y < 0) {  // the PP ends on the tree: on along path(last vertex -> exit)
        const int last = x + vb;
        follow(g.suf_seq + g.suf_off[last], 1, g.suf_len[last]);
    }
    *len = g.pre_len[x + vb] + (y >= 0 ? 1 : 0);
    const int base = g.rp[vb] + vb;
    if (y < 0) return base + o.end_slot[gid];
    int e = g.rp[x + vb];
    const int e1 = g.rp[x + vb + 1];
    while (e + 1 < e1 && g.col[e] != y + vb) ++e;
    return base + o.arc_slot[e];
}

// where the sub-runs start: i = this thread's first TP, step = TPs per pass of
// the grid (whole warps of consecutive TPs)
__device__ __forceinline__ void tp_mark_subs(const TpOrder &o, long long P, long long i, long long step) {
    const int lane = threadIdx.x & 31;
    for (; i - lane < P; i += step) {
        int len, slot = -1, first = -1;
        if (i < P) {
            slot = tp_slot_of(o, i, &len);
            first = o.pp_vert[o.pp_off[i]];
        }
        int pslot = __shfl_up_sync(0xffffffffu, slot, 1), pfirst = __shfl_up_sync(0xffffffffu, first, 1);
        if (i >= P) continue;
        if (lane == 0 && i > 0) {
            pslot = tp_slot_of(o, i - 1, &len);
            pfirst = o.pp_vert[o.pp_off[i - 1]];
        }
        o.start[i] = i == 0 || slot != pslot || first != pfirst;
    }
}

__device__ __forceinline__ void tp_list_subs(const TpOrder &o, long long P, long long i, long long step) {
    for (; i < P; i += step) {
        if (i == P - 1) o.sub_start[o.sub_rank[P]] = P;
        if (!o.start[i]) continue;
        const long long q = o.sub_rank[i];
        int len;
        const int slot = tp_slot_of(o, i, &len);
        o.sub_start[q] = i;
        o.sub_slot[q] = make_int2(slot, len * o.bits / 64);
    }
}

// one thread per sub-run: its place in its slot (any order within one will do)
__device__ __forceinline__ void tp_count_subs(const TpOrder &o, long long P, long long q, long long step) {
    const long long R = P > 0 ? o.sub_rank[P] : 0;
    for (; q < R; q += step) {
        const unsigned long long n = (unsigned long long)(o.sub_start[q + 1] - o.sub_start[q]);
        o.sub_at[q] = atomicAdd((unsigned long long *)o.slot_n + o.sub_slot[q].x, n | 1ull << 32);
    }
}

__device__ __forceinline__ void tp_place_subs(const TpOrder &o, long long P, long long q, long long step) {
    const long long R = P > 0 ? o.sub_rank[P] : 0;
    if (q == 0) o.bounds[R] = P;
    for (; q < R; q += step) {
        const int2 sl = o.sub_slot[q];
        const long long at = o.slot_at[sl.x], end = o.slot_at[sl.x + 1];
        const unsigned long long in = o.sub_at[q];
        const int first = (int)(at >> 32), k = (int)(end >> 32) - first, t = first + (int)(in >> 32);
        const long long pos = (at & 0xffffffffll) + (long long)(in & 0xffffffffull);
        o.bounds[t] = pos;
        o.sub_info[t] = make_int4(first, k, sl.y, 0);
        o.sub_dst[q] = make_longlong2(pos, t | (long long)merge_rounds(k) << 32);
        if (k > *(volatile int *)o.max_k) atomicMax(o.max_k, k);
    }
}

// A TP goes to the buffer from which its slot's last round writes perm[0].
__device__ __forceinline__ void tp_place(const TpOrder &o, long long P, long long i, long long step) {
    for (; i < P; i += step) {
        const long long q = o.sub_rank[i + 1] - 1;
        const longlong2 dst = o.sub_dst[q];
        const long long pos = dst.x + (i - o.sub_start[q]);
        o.pos_sub[pos] = (int)dst.y;
        o.perm[(dst.y >> 32) & 1][pos] = i;
    }
}

// Outputs [d0, d0 + ITEMS) of merge round r: in every slot with more than 2^r
// sub-runs, sub-runs [m 2^(r+1), m 2^(r+1) + 2^r) with the next 2^r.  The split
// is found by binary search, then the heads' first unshared words stay in
// registers (A first on ties, so equal TPs stay adjacent).
template <int ITEMS, int BITS>
__device__ __forceinline__ void tp_merge_items(const TpOrder &o, int r, long long P, long long d0) {
    const long long *in = nullptr;
    long long *out = nullptr;
    long long a_hi = 0, b_hi = -1, i = 0, j = 0, ia = 0, ib = 0;
    const unsigned long long *ka = nullptr, *kb = nullptr;
    unsigned long long wa = 0ull, wb = 0ull;
    int skip = 0;
    auto head_a = [&]() {
        if (i >= a_hi) return;
        ia = in[i];
        ka = o.key + o.key_off[ia] + skip;
        wa = *ka;
    };
    auto head_b = [&]() {
        if (j >= b_hi) return;
        ib = in[j];
        kb = o.key + o.key_off[ib] + skip;
        wb = *kb;
    };
    const long long d1 = d0 + ITEMS < P ? d0 + ITEMS : P;
    for (long long d = d0; d < d1; ++d) {
        if (d >= b_hi) {
            const int t = o.pos_sub[d];
            const int4 info = o.sub_info[t];
            const int k = info.y;
            if (k <= 1 << r) {  // sorted already: on to the next slot
                d = o.bounds[info.x + k] - 1;
                continue;
            }
            const int side = (merge_rounds(k) - r) & 1;
            in = o.perm[side];
            out = o.perm[side ^ 1];
            skip = info.z;
            const long long qa = (long long)((t - info.x) >> (r + 1)) << (r + 1), qb = qa + (1ll << r),
                            qe = qa + (2ll << r);
            const long long a_lo = o.bounds[info.x + qa];
            a_hi = o.bounds[info.x + (qb < k ? qb : k)];
            b_hi = o.bounds[info.x + (qe < k ? qe : k)];
            const long long na = a_hi - a_lo, nb = b_hi - a_hi, diag = d - a_lo;
            long long lo = diag > nb ? diag - nb : 0, hi = diag < na ? diag : na;
            while (lo < hi) {
                const long long mid = (lo + hi) >> 1;
                if (key_cmp_words<BITS>(o.key + o.key_off[in[a_lo + mid]] + skip,
                                        o.key + o.key_off[in[a_hi + diag - mid - 1]] + skip) <= 0)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            i = a_lo + lo;
            j = a_hi + (diag - lo);
            head_a();
            head_b();
        }
        bool take_a;
        if (i >= a_hi) take_a = false;
        else if (j >= b_hi) take_a = true;
        else if (wa != wb) take_a = wa < wb;
        else take_a = key_end<BITS>(wa) || key_cmp_words<BITS>(ka + 1, kb + 1) <= 0;
        out[d] = take_a ? ia : ib;
        if (take_a) {
            ++i;
            head_a();
        } else {
            ++j;
            head_b();
        }
    }
}

// the TP at position i differs from the one before it (TPs of different slots,
// and of one sub-run, always do)
template <int BITS>
__device__ __forceinline__ bool tp_differs(const TpOrder &o, long long i) {
    const int4 info = o.sub_info[o.pos_sub[i]];
    if (info.y == 1 || i == o.bounds[info.x]) return true;
    return key_cmp_words<BITS>(o.key + o.key_off[o.perm[0][i - 1]] + info.z,
                               o.key + o.key_off[o.perm[0][i]] + info.z) != 0;
}

// TPs that a warp of the two kernels below takes at a time, of P: their parts
// are gathered by a lane each, then half a warp goes along one TP.
constexpr int TP_WARPS = 9728;  // 64 warps on each of 152 SMs
__host__ __device__ inline int tp_group(long long P) {
    const long long per = (P + TP_WARPS - 1) / TP_WARPS;
    return per < 2 ? 2 : per > 32 ? 32 : (int)((per + 1) & ~1ll);
}

// Packed keys of the TPs [i0, i0 + group) cut off at P, by one warp: each
// vertex is read once from its part (prefix path, PP, suffix path) and stored
// at its place in its word (words hold the first vertex in their high bits).
template <typename T>
__device__ __forceinline__ void tp_write_keys_warp(const TpOrder &o, const long long *tp_off, unsigned long long *key,
                                                   long long i0, int group, long long P) {
    constexpr int VPW = 8 / sizeof(T);
    const GraphDev &g = o.g;
    const int lane = threadIdx.x & 31, sub = lane & 15;
    const long long i = i0 + lane;
    // lane l's TP: where a position p of it lies, per part, and its key
    const int *pre = nullptr, *pp = nullptr, *suf = nullptr;
    int pl = 0, pe = 0, len = 0;
    long long k0 = 0;
    if (lane < group && i < P) {
        const long long o0 = o.pp_off[i], o1 = o.pp_off[i + 1];
        const int vb = g.vgraph ? g.vbase[o.pp_graph ? o.pp_graph[i] : 0] : 0;
        const int f = o.pp_vert[o0] + vb, l = o.pp_vert[o1 - 1] + vb;
        len = (int)(tp_off[i + 1] - tp_off[i]);
        k0 = o.key_off[i];
        pl = g.pre_len[f] - 1;
        pe = pl + (int)(o1 - o0);
        pre = g.pre_seq + g.pre_off[f];
        pp = o.pp_vert + o0 - pl;
        suf = g.suf_seq + g.suf_off[l] + 1 - pe;
    }
    for (int t = 0; t < group; t += 2) {
        const int src = t + (lane >> 4);
        const int *tpre = (const int *)__shfl_sync(0xffffffffu, (unsigned long long)pre, src);
        const int *tpp = (const int *)__shfl_sync(0xffffffffu, (unsigned long long)pp, src);
        const int *tsuf = (const int *)__shfl_sync(0xffffffffu, (unsigned long long)suf, src);
        const int tpl = __shfl_sync(0xffffffffu, pl, src), tpe = __shfl_sync(0xffffffffu, pe, src);
        const int tlen = __shfl_sync(0xffffffffu, len, src);
        T *dst = (T *)(key + __shfl_sync(0xffffffffu, k0, src));
        const int end = tlen > 0 ? (tlen / VPW + 1) * VPW : 0;
#pragma unroll 4
        for (int p = sub; p < end; p += 16) {
            int v = 0;
            if (p < tlen) v = (p < tpl ? tpre : p < tpe ? tpp : tsuf)[p] + 1;
            dst[p ^ (VPW - 1)] = (T)v;
        }
    }
}

// The kept TPs of the sorted positions [i0, i0 + group), unpacked from their
// keys straight into their final places (contiguous ones), by one warp.
template <typename T>
__device__ __forceinline__ void tp_unpack_warp(const TpOrder &o, const long long *keep_off, const long long *keep_rank,
                                               long long *final_off, int *out_vert, int *out_graph, long long i0,
                                               int group, long long P) {
    constexpr int VPW = 8 / sizeof(T);
    const int lane = threadIdx.x & 31, sub = lane & 15;
    const long long i = i0 + lane;
    const T *from = nullptr;
    long long d0 = 0;
    int len = 0;
    if (lane < group && i < P) {
        d0 = keep_off[i];
        len = (int)(keep_off[i + 1] - d0);  // 0: a duplicate
        if (len > 0) {
            const long long x = o.perm[0][i], r = keep_rank[i];
            from = (const T *)(o.key + o.key_off[x]);
            out_graph[r] = o.pp_graph ? o.pp_graph[x] : 0;
            final_off[r] = d0;
        }
    }
    for (int t = 0; t < group; t += 2) {
        const int src = t + (lane >> 4);
        const T *tfrom = (const T *)__shfl_sync(0xffffffffu, (unsigned long long)from, src);
        const int tlen = __shfl_sync(0xffffffffu, len, src);
        int *dst = out_vert + __shfl_sync(0xffffffffu, d0, src);
#pragma unroll 4
        for (int p = sub; p < tlen; p += 16) dst[p] = (int)tfrom[p ^ (VPW - 1)] - 1;
    }
}

}  // namespace tpg
