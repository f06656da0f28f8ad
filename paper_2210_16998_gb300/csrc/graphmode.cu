// Graph-captured pipeline: everything after the frontier launch, with every
// size read from device memory, so that the whole hot path of a handle (one
// graph or a batch of thousands) is a fixed sequence of launches that can be
// captured once into a CUDA graph and replayed.
//
// Prime-path order (kernel (e) for PPs): place_pps, as in the host-driven path.
//
// Test-path order: the TPs of one graph that share a first vertex form a
// sorted run; runs are merged pairwise inside each graph in
// ceil(log2(max vertices + 1)) fixed rounds, comparing whole sequences.
#include "common.cuh"
#include "kernels.h"
#include "paths_dev.cuh"

namespace tpg {

namespace {

constexpr int GMB = 256;      // threads per block of the streaming kernels
constexpr int GM_SCAN_ITEMS = 8;
constexpr long long GM_SCAN_TILE = (long long)GMB * GM_SCAN_ITEMS;
constexpr long long GM_SCAN_FEW_TILES = 4096;  // above, the tile sums get a scan of their own

__device__ __forceinline__ long long clampc(long long v, long long cap) { return v < 0 ? 0 : (v > cap ? cap : v); }

// ---------------------------------------------------------------------------
// device-count scans
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(GMB) gm_scan_reduce(const T *in, const long long *n_dev, long long n_cap,
                                                      long long *tile_sums) {
    const long long n = clampc(*n_dev, n_cap);
    const long long ntiles = (n + GM_SCAN_TILE - 1) / GM_SCAN_TILE;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
        long long s = 0;
        for (int j = 0; j < GM_SCAN_ITEMS; ++j) {
            const long long i = t * GM_SCAN_TILE + (long long)j * GMB + threadIdx.x;
            if (i < n) s += (long long)in[i];
        }
        long long total;
        block_excl_scan_i64<GMB>(s, total);
        if (threadIdx.x == 0) tile_sums[t] = total;
    }
}

__global__ void __launch_bounds__(GMB) gm_scan_tiles(long long *tile_sums, const long long *n_dev, long long n_cap) {
    const long long n = clampc(*n_dev, n_cap);
    const long long ntiles = (n + GM_SCAN_TILE - 1) / GM_SCAN_TILE;
    long long carry = 0;
    for (long long base = 0; base < ntiles; base += GMB) {
        const long long i = base + threadIdx.x;
        const long long v = (i < ntiles) ? tile_sums[i] : 0;
        long long total;
        const long long ex = block_excl_scan_i64<GMB>(v, total);
        if (i < ntiles) tile_sums[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) tile_sums[ntiles] = carry;
}

// RAW: tile_sums holds the sums themselves (few tiles: each adds up those
// before it), else their prefix
template <typename T, bool RAW>
__global__ void __launch_bounds__(GMB) gm_scan_down(const T *in, long long *out, const long long *n_dev,
                                                    long long n_cap, const long long *tile_sums) {
    const long long n = clampc(*n_dev, n_cap);
    const long long ntiles = (n + GM_SCAN_TILE - 1) / GM_SCAN_TILE;
    if (RAW && ntiles == 0 && blockIdx.x == 0 && threadIdx.x == 0) out[0] = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const long long base = t * GM_SCAN_TILE + (long long)threadIdx.x * GM_SCAN_ITEMS;
        long long before = 0;
        if constexpr (RAW) {
            for (long long i = threadIdx.x; i < t; i += GMB) before += tile_sums[i];
            block_excl_scan_i64<GMB>(before, before);
        } else {
            before = tile_sums[t];
        }
        long long v[GM_SCAN_ITEMS];
        long long s = 0;
#pragma unroll
        for (int j = 0; j < GM_SCAN_ITEMS; ++j) {
            const long long i = base + j;
            v[j] = (i < n) ? (long long)in[i] : 0;
            s += v[j];
        }
        long long total;
        long long run = block_excl_scan_i64<GMB>(s, total) + before;
#pragma unroll
        for (int j = 0; j < GM_SCAN_ITEMS; ++j) {
            const long long i = base + j;
            if (i < n) out[i] = run;
            run += v[j];
        }
        if (RAW && t == ntiles - 1 && threadIdx.x == 0) out[n] = before + total;
    }
    if (!RAW && blockIdx.x == 0 && threadIdx.x == 0) out[n] = tile_sums[ntiles];
}

// ---------------------------------------------------------------------------
// PP ordering
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(GMB) gm_level_summary(GmArgs a) {
    const int ml = a.max_levels;
    const bool ok = (*a.enum_err == 0);
    long long carry = 0, vcarry = 0;
    for (int base = 0; base < ml; base += GMB) {
        const int k = base + threadIdx.x;
        long long v = 0;
        if (ok && k >= 1 && k < ml) v = a.levels[k].count > 0 ? a.levels[k].pp_count : 0;
        long long total, vtotal;
        block_excl_scan_i64<GMB>(v, total);
        block_excl_scan_i64<GMB>(v * k, vtotal);
        carry += total;
        vcarry += vtotal;
    }
    if (threadIdx.x == 0) {
        GmCounts *c = a.counts;
        c->P = carry;
        c->V = vcarry;
        int f = ok ? 0 : GM_ENUM_FAILED;
        if (carry > a.P_cap) f |= GM_OVF_PP;
        if (vcarry > a.V_cap) f |= GM_OVF_PPV;
        c->flags = f;
    }
}

__device__ __forceinline__ long long gm_P(const GmArgs &a) {
    const GmCounts *c = a.counts;
    if (c->flags & (GM_ENUM_FAILED | GM_OVF_PP | GM_OVF_PPV)) return 0;
    return clampc(c->P, a.P_cap);
}

constexpr int GM_MAT_WARPS = 8;

template <int CH, typename T>
__global__ void __launch_bounds__(GM_MAT_WARPS * 32, 8) gm_materialize(GmArgs a) {
    __shared__ T sbuf[GM_MAT_WARPS][MAT_BUF * CH];
    __shared__ int2 *s_nodes[MAT_MAX_LV];
    int2 *const *lv = cache_level_nodes(a.levels, a.max_levels, s_nodes);
    const long long P = gm_P(a);
    materialize_warps<GM_MAT_WARPS, CH, T>(a.refs, nullptr, 0, P, a.pp_off, a.levels, a.g,
                                           a.pp_vert, a.g.G > 1 ? a.pp_graph : nullptr, sbuf, lv);
}

// graph_path_ptr from sorted graph ids (ids == nullptr: one graph)
__global__ void __launch_bounds__(GMB) gm_graph_ptr(const int *ids, const long long *n_dev, long long n_cap, int G,
                                                    long long *ptr, const GmCounts *c, int fail_mask) {
    const long long n = (c->flags & fail_mask) ? 0 : clampc(*n_dev, n_cap);
    for (long long i = blockIdx.x * (long long)GMB + threadIdx.x; i <= n; i += (long long)gridDim.x * GMB) {
        const int cur = (i < n) ? (ids ? ids[i] : 0) : G;
        const int prev = (i > 0) ? (ids ? ids[i - 1] : 0) : -1;
        for (int gg = prev + 1; gg <= cur; ++gg) ptr[gg] = i;
    }
}

// ---------------------------------------------------------------------------
// TP assembly and ordering
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(GMB) gm_tp_len(GmArgs a) {
    const long long P = gm_P(a);
    const GraphDev &g = a.g;
    for (long long i = blockIdx.x * (long long)GMB + threadIdx.x; i < P; i += (long long)gridDim.x * GMB) {
        const long long o0 = a.pp_off[i], o1 = a.pp_off[i + 1];
        const int gid = g.G > 1 ? a.pp_graph[i] : 0;
        const int vb = g.vgraph ? g.vbase[gid] : 0;
        const int f = a.pp_vert[o0] + vb, l = a.pp_vert[o1 - 1] + vb;
        const int pl = g.pre_len[f], sl = g.suf_len[l];
        long long len = 0;
        if (pl == 0 || sl == 0) atomicOr(&a.counts->flags, GM_UNREACH);
        else len = (long long)(pl - 1) + (o1 - o0) + (sl - 1);
        a.tp_len[i] = len;
        a.len[i] = key_words(len, a.key_bits);
    }
}

__device__ __forceinline__ long long gm_P_tp(const GmArgs &a) {
    const GmCounts *c = a.counts;
    if (c->flags & (GM_ENUM_FAILED | GM_OVF_PP | GM_OVF_PPV | GM_UNREACH | GM_OVF_TPV0)) return 0;
    return clampc(c->P, a.P_cap);
}

__global__ void gm_tp_check(GmArgs a) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        GmCounts *c = a.counts;
        c->TV0 = a.tp_off0[clampc(c->P, a.P_cap)];
        if (c->TV0 > a.TV0_cap || a.key_off[clampc(c->P, a.P_cap)] > a.K_cap) atomicOr(&c->flags, GM_OVF_TPV0);
    }
}

__global__ void __launch_bounds__(GMB) gm_order_mark(GmArgs a) {
    tp_mark_subs(a.order, gm_P_tp(a), blockIdx.x * (long long)GMB + threadIdx.x, gridDim.x * (long long)GMB);
}
__global__ void __launch_bounds__(GMB) gm_order_list(GmArgs a) {
    tp_list_subs(a.order, gm_P_tp(a), blockIdx.x * (long long)GMB + threadIdx.x, gridDim.x * (long long)GMB);
}
__global__ void __launch_bounds__(GMB) gm_order_count(GmArgs a) {
    tp_count_subs(a.order, gm_P_tp(a), blockIdx.x * (long long)GMB + threadIdx.x, gridDim.x * (long long)GMB);
}
__global__ void __launch_bounds__(GMB) gm_order_place_subs(GmArgs a) {
    tp_place_subs(a.order, gm_P_tp(a), blockIdx.x * (long long)GMB + threadIdx.x, gridDim.x * (long long)GMB);
}
__global__ void __launch_bounds__(GMB) gm_order_place(GmArgs a) {
    tp_place(a.order, gm_P_tp(a), blockIdx.x * (long long)GMB + threadIdx.x, gridDim.x * (long long)GMB);
}

// The packed comparison keys of every TP, read from its parts (the TPs
// themselves are unpacked from them once, in sorted order, by gm_tp_gather).
template <typename T>
__global__ void __launch_bounds__(GMB) gm_tp_write(GmArgs a) {
    const long long P = gm_P_tp(a);
    const int group = tp_group(P);
    const long long step = gridDim.x * (GMB / 32ll) * group;
    for (long long i0 = (blockIdx.x * (GMB / 32ll) + (threadIdx.x >> 5)) * group; i0 < P; i0 += step)
        tp_write_keys_warp<T>(a.order, a.tp_off0, a.key, i0, group, P);
}

constexpr int GM_MERGE_ITEMS = 4;  // outputs per thread of a merge round
template <int BITS>
__global__ void __launch_bounds__(GMB) gm_tp_merge_round(GmArgs a, int r) {
    const long long P = gm_P_tp(a);
    if (P <= 0 || *a.order.max_k <= 1 << r) return;
    const long long step = (long long)gridDim.x * GMB * GM_MERGE_ITEMS;
    for (long long d0 = (blockIdx.x * (long long)GMB + threadIdx.x) * GM_MERGE_ITEMS; d0 < P; d0 += step)
        tp_merge_items<GM_MERGE_ITEMS, BITS>(a.order, r, P, d0);
}

template <int BITS>
__global__ void __launch_bounds__(GMB) gm_tp_dedup(GmArgs a) {
    const long long P = gm_P_tp(a);
    for (long long i = blockIdx.x * (long long)GMB + threadIdx.x; i < P; i += (long long)gridDim.x * GMB) {
        const long long x = a.order.perm[0][i];
        const int k = tp_differs<BITS>(a.order, i);
        a.keep[i] = k;
        a.tp_len[i] = k ? a.tp_off0[x + 1] - a.tp_off0[x] : 0;
    }
}

__global__ void gm_tp_totals(GmArgs a) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        GmCounts *c = a.counts;
        const long long P = gm_P_tp(a);
        c->T = P ? a.keep_rank[P] : 0;
        c->TV = P ? a.keep_off[P] : 0;
        if (c->TV > a.TV_cap) atomicOr(&c->flags, GM_OVF_TPV);
    }
}

__device__ __forceinline__ long long gm_P_final(const GmArgs &a) {
    if (a.counts->flags & GM_OVF_TPV) return 0;
    return gm_P_tp(a);
}

// The kept TPs in sorted order, each straight into its final place: the TP
// list is never written in PP order.
template <typename T>
__global__ void __launch_bounds__(GMB) gm_tp_gather(GmArgs a) {
    const long long P = gm_P_final(a);
    const int group = tp_group(P);
    const long long step = gridDim.x * (GMB / 32ll) * group;
    for (long long i0 = (blockIdx.x * (GMB / 32ll) + (threadIdx.x >> 5)) * group; i0 < P; i0 += step)
        tp_unpack_warp<T>(a.order, a.keep_off, a.keep_rank, a.tp_off, a.tp_vert, a.tp_graph, i0, group, P);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const GmCounts *c = a.counts;
        a.tp_off[P ? c->T : 0] = P ? c->TV : 0;
    }
}

unsigned stream_grid(int num_sms) { return (unsigned)(num_sms * 8); }

template <typename T>
cudaError_t gm_scan(const T *in, long long *out, const long long *n_dev, long long n_cap, long long *tmp,
                    int num_sms, cudaStream_t s) {
    const unsigned grid = stream_grid(num_sms);
    gm_scan_reduce<T><<<grid, GMB, 0, s>>>(in, n_dev, n_cap, tmp);
    if (n_cap <= GM_SCAN_FEW_TILES * GM_SCAN_TILE) {
        gm_scan_down<T, true><<<grid, GMB, 0, s>>>(in, out, n_dev, n_cap, tmp);
        note_launch(2);
        return cudaGetLastError();
    }
    gm_scan_tiles<<<1, GMB, 0, s>>>(tmp, n_dev, n_cap);
    gm_scan_down<T, false><<<grid, GMB, 0, s>>>(in, out, n_dev, n_cap, tmp);
    note_launch(3);
    return cudaGetLastError();
}

}  // namespace

int gm_tp_rounds(int maxn) {
    int r = 0;
    while ((1 << r) < maxn + 1) ++r;
    return r;
}

size_t gm_scan_tmp_elems(long long n_cap) { return (size_t)((n_cap + GM_SCAN_TILE - 1) / GM_SCAN_TILE) + 2; }

cudaError_t gm_enqueue_pp(const GmArgs &a, cudaStream_t s) {
    const unsigned grid = stream_grid(a.num_sms);
    gm_level_summary<<<1, GMB, 0, s>>>(a);
    note_launch();
    PlaceArgs r{};
    r.levels = a.levels;
    r.max_levels = a.max_levels;
    r.refs = a.refs;
    r.off = a.pp_off;
    r.cap = a.P_cap;
    r.skip = &a.counts->flags;
    r.skip_mask = GM_ENUM_FAILED | GM_OVF_PP | GM_OVF_PPV;
    cudaError_t e = place_pps(r, a.num_sms, s);
    if (e != cudaSuccess) return e;
    if (a.g.maxn <= MAT_SMALL_N) gm_materialize<2, unsigned char><<<grid, GM_MAT_WARPS * 32, 0, s>>>(a);
    else gm_materialize<1, unsigned short><<<grid, GM_MAT_WARPS * 32, 0, s>>>(a);
    gm_graph_ptr<<<grid, GMB, 0, s>>>(a.g.G > 1 ? a.pp_graph : nullptr, &a.counts->P, a.P_cap, a.g.G, a.pp_gptr,
                                      a.counts, GM_ENUM_FAILED | GM_OVF_PP | GM_OVF_PPV);
    note_launch(2);
    return cudaGetLastError();
}

cudaError_t gm_enqueue_tp(const GmArgs &a, cudaStream_t s) {
    const unsigned grid = stream_grid(a.num_sms);
    gm_tp_len<<<grid, GMB, 0, s>>>(a);
    note_launch();
    cudaError_t e;
    if ((e = gm_scan<long long>(a.tp_len, a.tp_off0, &a.counts->P, a.P_cap, a.scan_tmp, a.num_sms, s)))
        return e;
    if ((e = gm_scan<long long>(a.len, a.key_off, &a.counts->P, a.P_cap, a.scan_tmp, a.num_sms, s)))
        return e;
    gm_tp_check<<<1, 32, 0, s>>>(a);
    gm_order_mark<<<grid, GMB, 0, s>>>(a);
    note_launch(2);
    if ((e = gm_scan<int>(a.order.start, a.order.sub_rank, &a.counts->P, a.P_cap, a.scan_tmp, a.num_sms, s)))
        return e;
    if ((e = cudaMemsetAsync(a.order.slot_n, 0, sizeof(long long) * (a.slots + 1), s))) return e;
    gm_order_list<<<grid, GMB, 0, s>>>(a);
    gm_order_count<<<grid, GMB, 0, s>>>(a);
    note_launch(2);
    if ((e = scan_i64(a.order.slot_n, a.order.slot_at, a.slots, a.scan_tmp, s))) return e;
    gm_order_place_subs<<<grid, GMB, 0, s>>>(a);
    gm_order_place<<<grid, GMB, 0, s>>>(a);
    if (a.key_bits == 8) gm_tp_write<unsigned char><<<grid, GMB, 0, s>>>(a);
    else gm_tp_write<unsigned short><<<grid, GMB, 0, s>>>(a);
    note_launch(3);
    for (int r = 0; r < a.tp_rounds; ++r) {
        if (a.key_bits == 8) gm_tp_merge_round<8><<<grid, GMB, 0, s>>>(a, r);
        else gm_tp_merge_round<16><<<grid, GMB, 0, s>>>(a, r);
    }
    if (a.key_bits == 8) gm_tp_dedup<8><<<grid, GMB, 0, s>>>(a);
    else gm_tp_dedup<16><<<grid, GMB, 0, s>>>(a);
    note_launch(a.tp_rounds + 1);
    if ((e = gm_scan<long long>(a.tp_len, a.keep_off, &a.counts->P, a.P_cap, a.scan_tmp, a.num_sms, s)))
        return e;
    if ((e = gm_scan<int>(a.keep, a.keep_rank, &a.counts->P, a.P_cap, a.scan_tmp, a.num_sms, s)))
        return e;
    gm_tp_totals<<<1, 32, 0, s>>>(a);
    if (a.key_bits == 8) gm_tp_gather<unsigned char><<<grid, GMB, 0, s>>>(a);
    else gm_tp_gather<unsigned short><<<grid, GMB, 0, s>>>(a);
    gm_graph_ptr<<<grid, GMB, 0, s>>>(a.tp_graph, &a.counts->T, a.P_cap, a.g.G, a.tp_gptr, a.counts,
                                      GM_ENUM_FAILED | GM_OVF_PP | GM_OVF_PPV | GM_UNREACH | GM_OVF_TPV0 | GM_OVF_TPV);
    note_launch(3);
    return cudaGetLastError();
}

}  // namespace tpg
