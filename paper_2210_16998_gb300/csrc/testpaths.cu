// Test-path assembly (kernel (d)) and canonical sort + dedup of the test
// paths (kernel (e) for TPs).
//
// TP(p) = path(entry -> first p), then p, then path(last p -> exit), joined
// at the shared endpoints (Problem 1 output; the touring of Sec. 7.3), with
// path(a -> b) read from the lowest-id BFS predecessor table.  Because the
// PPs arrive in canonical order, TPs of PPs that share a first vertex share
// their prefix and are already in order among themselves.  How the whole list
// is put in order is told in tp_order_dev.cuh; exact duplicates (two PPs of
// different first vertices can yield the same TP) are dropped at the end.
#include "common.cuh"
#include "kernels.h"
#include "paths_dev.cuh"
#include "testpaths.h"

namespace tpg {

static unsigned grid_for(long long n, int block = 256) {
    long long b = (n + block - 1) / block;
    if (b < 1) b = 1;
    if (b > (1 << 20)) b = 1 << 20;
    return (unsigned)b;
}

// TP lengths from each PP's (first, last) local vertex, which the
// materialisation wrote beside the PP list (coalesced reads only); runs[0] +=
// runs of PPs with one first vertex, runs[1] += graphs that own a PP, runs[2] =
// the longest.
__global__ void __launch_bounds__(256) tp_len_kernel(const long long *__restrict__ pp_off,
                                                     const int2 *__restrict__ pp_ends,
                                                     const int *__restrict__ pp_graph, long long P, GraphDev g,
                                                     long long *tp_len, int *err, unsigned long long *runs) {
    int nruns = 0, ngraphs = 0, longest = 0;
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < P; i += gridDim.x * 256ll) {
        const long long o0 = pp_off[i], o1 = pp_off[i + 1];
        const int gid = pp_graph ? pp_graph[i] : 0;
        const int vb = g.vgraph ? g.vbase[gid] : 0;
        const int2 e = pp_ends[i];
        const int f = e.x + vb, l = e.y + vb;
        const int pl = g.pre_len[f], sl = g.suf_len[l];
        long long len = 0;
        if (pl == 0 || sl == 0) atomicOr(err, ERR_UNREACH);
        else len = (long long)(pl - 1) + (o1 - o0) + (sl - 1);
        tp_len[i] = len;
        longest = len > longest ? (int)len : longest;
        const bool new_graph = i == 0 || (pp_graph && pp_graph[i - 1] != gid);
        ngraphs += new_graph;
        nruns += new_graph || pp_ends[i - 1].x != e.x;
    }
    nruns = __reduce_add_sync(0xffffffffu, nruns);
    ngraphs = __reduce_add_sync(0xffffffffu, ngraphs);
    longest = __reduce_max_sync(0xffffffffu, longest);
    if ((threadIdx.x & 31) == 0 && longest) {
        if (nruns) atomicAdd(runs, (unsigned long long)nruns);
        if (ngraphs) atomicAdd(runs + 1, (unsigned long long)ngraphs);
        if ((unsigned long long)longest > *(volatile unsigned long long *)(runs + 2))
            atomicMax(runs + 2, (unsigned long long)longest);
    }
}

cudaError_t tp_lengths(const long long *pp_off, const int2 *pp_ends, const int *pp_graph, long long P,
                       const GraphDev &g, long long *tp_len, int *err, unsigned long long *runs, cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    const unsigned grid = grid_for(P);
    tp_len_kernel<<<grid < 4864 ? grid : 4864, 256, 0, s>>>(pp_off, pp_ends, pp_graph, P, g, tp_len, err, runs);
    note_launch();
    return cudaGetLastError();
}

// One warp per 32 consecutive TPs.  Lane l first gathers the parts of TP
// i0 + l (prefix path entry -> first vertex, the PP, suffix path last vertex
// -> exit) in parallel with the other lanes; the warp then copies the TPs one
// after another with its lanes striding over positions (coalesced).  When
// every TP of the warp is its own PP (empty prefix and suffix), the 32 TPs
// are one contiguous copy of the 32 PPs.
__global__ void tp_write_kernel(const long long *__restrict__ pp_off, const int *__restrict__ pp_vert,
                                const int *__restrict__ pp_graph, long long P, GraphDev g,
                                const long long *__restrict__ tp_off, int *__restrict__ tp_vert) {
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long i0 = (blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; i0 < P;
         i0 += nw * 32) {
        const long long i = i0 + lane;
        const bool valid = i < P;
        long long o0 = 0, plen = 0, d0 = 0, total = 0;
        int pl = 0;
        const int *pre = nullptr, *suf = nullptr;
        if (valid) {
            o0 = pp_off[i];
            plen = pp_off[i + 1] - o0;
            d0 = tp_off[i];
            total = tp_off[i + 1] - d0;
            const int gid = pp_graph ? pp_graph[i] : 0;
            const int vb = g.vgraph ? g.vbase[gid] : 0;
            const int f = pp_vert[o0] + vb, l = pp_vert[o0 + plen - 1] + vb;
            pl = g.pre_len[f] - 1;
            pre = g.pre_seq + g.pre_off[f];
            suf = g.suf_seq + g.suf_off[l] + 1;
        }
        const int last = (int)((P - i0 < 32 ? P - i0 : 32) - 1);
        if (__all_sync(0xffffffffu, !valid || (pl == 0 && total == plen))) {
            // TP == PP for all: one contiguous range
            const long long src0 = __shfl_sync(0xffffffffu, o0, 0), dst0 = __shfl_sync(0xffffffffu, d0, 0);
            const long long len = __shfl_sync(0xffffffffu, d0 + total, last) - dst0;
            const int *src = pp_vert + src0;
            int *dst = tp_vert + dst0;
            long long p = lane;
            for (; p + 96 < len; p += 128) {
                const int a = src[p], b = src[p + 32], c = src[p + 64], d = src[p + 96];
                dst[p] = a;
                dst[p + 32] = b;
                dst[p + 64] = c;
                dst[p + 96] = d;
            }
            for (; p < len; p += 32) dst[p] = src[p];
            continue;
        }
        for (int t = 0; t <= last; ++t) {
            const long long to0 = __shfl_sync(0xffffffffu, o0, t), td0 = __shfl_sync(0xffffffffu, d0, t);
            const long long tplen = __shfl_sync(0xffffffffu, plen, t), ttot = __shfl_sync(0xffffffffu, total, t);
            const int tpl = __shfl_sync(0xffffffffu, pl, t);
            const int *tpre = (const int *)__shfl_sync(0xffffffffu, (unsigned long long)pre, t);
            const int *tsuf = (const int *)__shfl_sync(0xffffffffu, (unsigned long long)suf, t);
            for (long long p = lane; p < ttot; p += 32) {
                int v;
                if (p < tpl) v = tpre[p];
                else if (p < tpl + tplen) v = pp_vert[to0 + (p - tpl)];
                else v = tsuf[p - tpl - tplen];
                tp_vert[td0 + p] = v;
            }
        }
    }
}

cudaError_t tp_write(const long long *pp_off, const int *pp_vert, const int *pp_graph, long long P,
                     const GraphDev &g, const long long *tp_off, int *tp_vert, cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    long long blocks = (P + 255) / 256;  // 8 warps of 32 TPs
    if (blocks > 65535) blocks = 65535;
    tp_write_kernel<<<(unsigned)blocks, 256, 0, s>>>(pp_off, pp_vert, pp_graph, P, g, tp_off, tp_vert);
    note_launch();
    return cudaGetLastError();
}

__global__ void iota_kernel(long long *perm, long long P) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P;
         i += (long long)gridDim.x * blockDim.x)
        perm[i] = i;
}



cudaError_t tp_iota(long long *perm, long long P, cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    iota_kernel<<<grid_for(P), 256, 0, s>>>(perm, P);
    note_launch();
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) tp_mark_kernel(TpOrder o, long long P) {
    tp_mark_subs(o, P, blockIdx.x * 256ll + threadIdx.x, gridDim.x * 256ll);
}
__global__ void __launch_bounds__(256) tp_list_kernel(TpOrder o, long long P) {
    tp_list_subs(o, P, blockIdx.x * 256ll + threadIdx.x, gridDim.x * 256ll);
}
__global__ void __launch_bounds__(256) tp_count_kernel(TpOrder o, long long P) {
    tp_count_subs(o, P, blockIdx.x * 256ll + threadIdx.x, gridDim.x * 256ll);
}
__global__ void __launch_bounds__(256) tp_place_subs_kernel(TpOrder o, long long P) {
    tp_place_subs(o, P, blockIdx.x * 256ll + threadIdx.x, gridDim.x * 256ll);
}
__global__ void __launch_bounds__(256) tp_place_kernel(TpOrder o, long long P) {
    tp_place(o, P, blockIdx.x * 256ll + threadIdx.x, gridDim.x * 256ll);
}

cudaError_t tp_order_mark(const TpOrder &o, long long P, cudaStream_t s) {
    tp_mark_kernel<<<grid_for(P), 256, 0, s>>>(o, P);
    note_launch();
    return cudaGetLastError();
}

cudaError_t tp_order_list(const TpOrder &o, long long P, long long n_subs, cudaStream_t s) {
    tp_list_kernel<<<grid_for(P), 256, 0, s>>>(o, P);
    tp_count_kernel<<<grid_for(n_subs), 256, 0, s>>>(o, P);
    note_launch(2);
    return cudaGetLastError();
}

cudaError_t tp_order_place(const TpOrder &o, long long P, long long n_subs, cudaStream_t s) {
    tp_place_subs_kernel<<<grid_for(n_subs), 256, 0, s>>>(o, P);
    tp_place_kernel<<<grid_for(P), 256, 0, s>>>(o, P);
    note_launch(2);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) tp_plain_kernel(TpOrder o, long long P, const int *start, const long long *rank,
                                                       int runs) {
    long long *perm = o.perm[merge_rounds(runs) & 1];
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < P; i += gridDim.x * 256ll) {
        perm[i] = i;
        o.pos_sub[i] = (int)(rank[i + 1] - 1);
        if (start[i]) {
            o.bounds[rank[i]] = i;
            o.sub_info[rank[i]] = make_int4(0, runs, 0, 0);
        }
        if (i == 0) {
            o.bounds[runs] = P;
            *o.max_k = runs;
        }
    }
}

cudaError_t tp_order_plain(const TpOrder &o, long long P, const int *start, const long long *rank, long long runs,
                           cudaStream_t s) {
    tp_plain_kernel<<<grid_for(P), 256, 0, s>>>(o, P, start, rank, (int)runs);
    note_launch();
    return cudaGetLastError();
}

constexpr int TPM_ITEMS = 4;  // outputs per thread of a merge round
template <int BITS>
__global__ void __launch_bounds__(256) tp_merge_kernel(TpOrder o, int r, long long P) {
    if (*o.max_k <= 1 << r) return;
    const long long d0 = (blockIdx.x * 256ll + threadIdx.x) * TPM_ITEMS;
    if (d0 < P) tp_merge_items<TPM_ITEMS, BITS>(o, r, P, d0);
}

cudaError_t tp_order_merge(const TpOrder &o, long long P, long long max_k, cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    const int rounds = merge_rounds(max_k);
    const unsigned grid = (unsigned)((P + 256ll * TPM_ITEMS - 1) / (256ll * TPM_ITEMS));
    for (int r = 0; r < rounds; ++r) {
        if (o.bits == 8) tp_merge_kernel<8><<<grid, 256, 0, s>>>(o, r, P);
        else tp_merge_kernel<16><<<grid, 256, 0, s>>>(o, r, P);
    }
    note_launch(rounds);
    return cudaGetLastError();
}

template <int BITS>
__global__ void __launch_bounds__(256) tp_flags_kernel(TpOrder o, long long P, const long long *tp_off,
                                                       long long *keep_len, int *keep) {
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < P; i += gridDim.x * 256ll) {
        const int k = tp_differs<BITS>(o, i);
        const long long x = o.perm[0][i];
        keep[i] = k;
        keep_len[i] = k ? tp_off[x + 1] - tp_off[x] : 0;
    }
}

cudaError_t tp_order_flags(const TpOrder &o, long long P, const long long *tp_off, long long *keep_len, int *keep,
                           cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    if (o.bits == 8) tp_flags_kernel<8><<<grid_for(P), 256, 0, s>>>(o, P, tp_off, keep_len, keep);
    else tp_flags_kernel<16><<<grid_for(P), 256, 0, s>>>(o, P, tp_off, keep_len, keep);
    note_launch();
    return cudaGetLastError();
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK) tree_slots_kernel(GraphDev g, int *arc_slot, int *end_slot) {
    extern __shared__ int s_slots[];
    tree_slots_block<BLOCK>(g, blockIdx.x, arc_slot, end_slot, s_slots);
}

cudaError_t tree_slots(const GraphDev &g, int *arc_slot, int *end_slot, cudaStream_t s) {
    static_assert(3 * sizeof(int) * TPG_MAX_N <= 48 * 1024, "one graph's tables fit the default shared memory");
    const size_t smem = 3 * sizeof(int) * (size_t)g.maxn;
    if (g.maxn <= 256) tree_slots_kernel<128><<<g.G, 128, smem, s>>>(g, arc_slot, end_slot);
    else tree_slots_kernel<1024><<<g.G, 1024, smem, s>>>(g, arc_slot, end_slot);
    note_launch();
    return cudaGetLastError();
}

__global__ void key_len_kernel(const long long *tp_off, long long P, int bits, long long *key_len) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P;
         i += (long long)gridDim.x * blockDim.x)
        key_len[i] = key_words(tp_off[i + 1] - tp_off[i], bits);
}

cudaError_t tp_key_lengths(const long long *tp_off, long long P, int bits, long long *key_len, cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    key_len_kernel<<<grid_for(P), 256, 0, s>>>(tp_off, P, bits, key_len);
    note_launch();
    return cudaGetLastError();
}

// 8 lanes per TP, each packing 64 / bits consecutive vertices into a word
constexpr int KEY_LANES = 8;
__global__ void keys_kernel(const long long *tp_off, const int *tp_vert, long long P, int bits,
                            const long long *key_off, unsigned long long *key) {
    const int sub = threadIdx.x & (KEY_LANES - 1), vpw = 64 / bits;
    const long long groups = (long long)gridDim.x * (blockDim.x / KEY_LANES);
    for (long long i = blockIdx.x * (long long)(blockDim.x / KEY_LANES) + threadIdx.x / KEY_LANES; i < P;
         i += groups) {
        const long long t0 = tp_off[i], len = tp_off[i + 1] - t0, k0 = key_off[i], nw = key_off[i + 1] - k0;
        for (long long w = sub; w < nw; w += KEY_LANES) {
            unsigned long long word = 0;
            for (int q = 0; q < vpw; ++q) {
                const long long p = w * vpw + q;
                const unsigned long long v = p < len ? (unsigned long long)(tp_vert[t0 + p] + 1) : 0ull;
                word = (word << bits) | v;
            }
            key[k0 + w] = word;
        }
    }
}

cudaError_t tp_write_keys(const long long *tp_off, const int *tp_vert, long long P, int bits, const long long *key_off,
                          unsigned long long *key, cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    long long blocks = (P + (256 / KEY_LANES) - 1) / (256 / KEY_LANES);
    if (blocks > (1 << 20)) blocks = 1 << 20;
    keys_kernel<<<(unsigned)blocks, 256, 0, s>>>(tp_off, tp_vert, P, bits, key_off, key);
    note_launch();
    return cudaGetLastError();
}

__global__ void index_map_kernel(const long long *perm, const int *keep, const long long *keep_rank, long long P,
                                 int *map) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P;
         i += (long long)gridDim.x * blockDim.x) {
        if (!perm) map[i] = (int)i;
        else map[perm[i]] = (int)(keep[i] ? keep_rank[i] : keep_rank[i] - 1);
    }
}

cudaError_t tp_index_map(const long long *perm, const int *keep, const long long *keep_rank, long long P, int *map,
                         cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    index_map_kernel<<<grid_for(P), 256, 0, s>>>(perm, keep, keep_rank, P, map);
    note_launch();
    return cudaGetLastError();
}

// What bounds the two kernels are memory round trips (a TP's parts lie behind
// three dependent loads), so a lane gathers each TP's; 8 lanes that gathered and
// packed one TP took 2.24 ms for the 14.4M TPs of 4096 graphs (646M vertices).
template <typename T>
__global__ void __launch_bounds__(256) keys_parts_kernel(TpOrder o, const long long *tp_off, unsigned long long *key,
                                                         int group, long long P) {
    const long long step = gridDim.x * 8ll * group;
    for (long long i0 = (blockIdx.x * 8ll + (threadIdx.x >> 5)) * group; i0 < P; i0 += step)
        tp_write_keys_warp<T>(o, tp_off, key, i0, group, P);
}

cudaError_t tp_write_keys_parts(const TpOrder &o, const long long *tp_off, unsigned long long *key, long long P,
                                cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    const int group = tp_group(P);
    const unsigned grid = grid_for((P + group - 1) / group, 8);
    if (o.bits == 8) keys_parts_kernel<unsigned char><<<grid, 256, 0, s>>>(o, tp_off, key, group, P);
    else keys_parts_kernel<unsigned short><<<grid, 256, 0, s>>>(o, tp_off, key, group, P);
    note_launch();
    return cudaGetLastError();
}

template <typename T>
__global__ void __launch_bounds__(256) assemble_kernel(TpOrder o, const long long *keep_off, const long long *keep_rank,
                                                       long long *final_off, int *out_vert, int *out_graph, int group,
                                                       long long P) {
    const long long step = gridDim.x * 8ll * group;
    for (long long i0 = (blockIdx.x * 8ll + (threadIdx.x >> 5)) * group; i0 < P; i0 += step)
        tp_unpack_warp<T>(o, keep_off, keep_rank, final_off, out_vert, out_graph, i0, group, P);
}

cudaError_t tp_assemble(const TpOrder &o, const long long *keep_off, const long long *keep_rank, long long *final_off,
                        int *out_vert, int *out_graph, long long P, cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    const int group = tp_group(P);
    const unsigned grid = grid_for((P + group - 1) / group, 8);
    if (o.bits == 8)
        assemble_kernel<unsigned char><<<grid, 256, 0, s>>>(o, keep_off, keep_rank, final_off, out_vert, out_graph, group, P);
    else
        assemble_kernel<unsigned short><<<grid, 256, 0, s>>>(o, keep_off, keep_rank, final_off, out_vert, out_graph, group, P);
    note_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// few TPs of one graph: lengths, order, keys, merging and lists in one block.
// What bounds the steps above for such a list is that there are 25 launches and
// two read-backs of them (76 TPs: the whole call 205 us); here a step costs a
// block barrier and its own chain of loads (24 us, the whole call 44).
// ---------------------------------------------------------------------------
constexpr int TPS_BLOCK = 1024;

// out[0 .. n] = exclusive prefix of f(0 .. n - 1), the total returned; all threads, a barrier at the end
template <typename F>
__device__ __forceinline__ long long tps_scan(long long n, long long *out, F f) {
    long long carry = 0;
    for (long long base = 0; base < n; base += TPS_BLOCK) {
        const long long i = base + threadIdx.x;
        long long total;
        const long long ex = block_excl_scan_i64<TPS_BLOCK>(i < n ? (long long)f(i) : 0ll, total);
        if (i < n) out[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) out[n] = carry;
    __syncthreads();
    return carry;
}

template <typename T>
__global__ void __launch_bounds__(TPS_BLOCK) tp_small_kernel(TpSmallArgs a) {
    constexpr int BITS = 8 * sizeof(T);
    __shared__ int s_err, s_longest;
    const TpOrder &o = a.o;
    const GraphDev &g = o.g;
    const long long P = a.P, tid = threadIdx.x;
    if (tid == 0) s_err = s_longest = 0;
    __syncthreads();
    const long long TV = tps_scan(P, a.tp_off, [&](long long i) {
        const int2 e = a.ends[i];
        const int pl = g.pre_len[e.x], sl = g.suf_len[e.y];
        if (pl == 0 || sl == 0) s_err = ERR_UNREACH;
        const long long len = pl == 0 || sl == 0 ? 0 : (long long)(pl - 1) + (o.pp_off[i + 1] - o.pp_off[i]) + (sl - 1);
        a.tp_len[i] = len;
        atomicMax(&s_longest, (int)len);
        return len;
    });
    if (tid == 0) a.result[4] = s_longest;
    if (s_err || TV == a.V) {  // (equal: every TP is its PP)
        if (tid == 0) {
            a.result[0] = s_err;
            a.result[1] = TV;
        }
        return;
    }
    for (long long i = tid; i <= a.slots; i += TPS_BLOCK) o.slot_n[i] = 0;  // and max_k
    tps_scan(P, a.key_off, [&](long long i) { return key_words(a.tp_len[i], BITS); });
    tp_mark_subs(o, P, tid, TPS_BLOCK);
    __syncthreads();
    tps_scan(P, o.sub_rank, [&](long long i) { return o.start[i]; });
    tp_list_subs(o, P, tid, TPS_BLOCK);
    __syncthreads();
    tp_count_subs(o, P, tid, TPS_BLOCK);
    __syncthreads();
    tps_scan(a.slots, o.slot_at, [&](long long i) { return o.slot_n[i]; });
    tp_place_subs(o, P, tid, TPS_BLOCK);
    __syncthreads();
    tp_place(o, P, tid, TPS_BLOCK);
    constexpr int WARPS = TPS_BLOCK / 32;
    const long long each = ((P + WARPS - 1) / WARPS + 1) & ~1ll;
    const int group = each < 32 ? (int)each : 32;
    for (long long i0 = (tid >> 5) * group; i0 < P; i0 += WARPS * group)
        tp_write_keys_warp<T>(o, a.tp_off, a.key, i0, group, P);
    __syncthreads();
    const int max_k = *(volatile int *)o.max_k;
    for (int r = 0; 1 << r < max_k; ++r) {
        for (long long d0 = tid; d0 < P; d0 += TPS_BLOCK) tp_merge_items<1, BITS>(o, r, P, d0);
        __syncthreads();
    }
    const long long kept = tps_scan(P, a.keep_rank, [&](long long i) { return a.keep[i] = tp_differs<BITS>(o, i); });
    const long long FTV = tps_scan(P, a.keep_off, [&](long long i) { return a.keep[i] ? a.tp_len[o.perm[0][i]] : 0ll; });
    for (long long i0 = (tid >> 5) * group; i0 < P; i0 += WARPS * group)
        tp_unpack_warp<T>(o, a.keep_off, a.keep_rank, a.final_off, a.out_vert, a.out_graph, i0, group, P);
    if (a.pp_to_tp)
        for (long long i = tid; i < P; i += TPS_BLOCK)
            a.pp_to_tp[o.perm[0][i]] = (int)(a.keep[i] ? a.keep_rank[i] : a.keep_rank[i] - 1);
    if (tid == 0) {
        a.final_off[kept] = FTV;
        a.gptr[0] = 0;
        a.gptr[1] = kept;
        a.result[0] = 0;
        a.result[1] = TV;
        a.result[2] = kept;
        a.result[3] = FTV;
    }
}

cudaError_t tp_small(const TpSmallArgs &a, cudaStream_t s) {
    if (a.o.bits == 8) tp_small_kernel<unsigned char><<<1, TPS_BLOCK, 0, s>>>(a);
    else tp_small_kernel<unsigned short><<<1, TPS_BLOCK, 0, s>>>(a);
    note_launch();
    return cudaGetLastError();
}

// one warp per kept TP: copy into its final slot
__global__ void tp_gather_kernel(const long long *perm, const int *keep, const long long *keep_rank, long long P,
                                 const long long *off, const int *vert, const int *graph,
                                 const long long *keep_off, long long *final_off, int *out_vert,
                                 int *out_graph) {
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long i = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); i < P; i += nw) {
        if (!keep[i]) continue;
        const long long a = perm[i], r = keep_rank[i];
        const long long s0 = off[a], len = off[a + 1] - s0, d0 = keep_off[i];
        for (long long p = lane; p < len; p += 32) out_vert[d0 + p] = vert[s0 + p];
        if (lane == 0) {
            out_graph[r] = graph[a];
            final_off[r] = d0;
        }
    }
}

cudaError_t tp_gather(const long long *perm, const int *keep, const long long *keep_rank, long long P,
                      const long long *tp_off, const int *tp_vert, const int *tp_graph, const long long *keep_off,
                      long long *final_off, int *out_vert, int *out_graph, cudaStream_t s) {
    if (P <= 0) return cudaSuccess;
    long long blocks = (P + 7) / 8;
    if (blocks > 152 * 64) blocks = 152 * 64;
    tp_gather_kernel<<<(unsigned)blocks, 256, 0, s>>>(perm, keep, keep_rank, P, tp_off, tp_vert, tp_graph, keep_off,
                                                     final_off, out_vert, out_graph);
    note_launch();
    return cudaGetLastError();
}

}  // namespace tpg
