// TP ordering and keys of the host-driven path (testpaths.cu).
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "tp_order_dev.cuh"

namespace tpg {

// Order of the TPs (see tp_order_dev.cuh), in this sequence: mark, a scan of
// o.start into o.sub_rank, list, count (slot_n zero before), a scan of slot_n
// into slot_at, place; then the merge rounds and the flags, with the keys.
// n_subs: an upper bound of the number of sub-runs.
cudaError_t tp_order_mark(const TpOrder &o, long long P, cudaStream_t s);
cudaError_t tp_order_list(const TpOrder &o, long long P, long long n_subs, cudaStream_t s);
cudaError_t tp_order_place(const TpOrder &o, long long P, long long n_subs, cudaStream_t s);
// one slot whose sub-runs start where `start` says (runs of them, `rank` its
// exclusive prefix): bounds, sub_info, pos_sub, perm and max_k are set
cudaError_t tp_order_plain(const TpOrder &o, long long P, const int *start, const long long *rank, long long runs,
                           cudaStream_t s);
// rounds 0 .. merge_rounds(max_k) - 1, max_k an upper bound
cudaError_t tp_order_merge(const TpOrder &o, long long P, long long max_k, cudaStream_t s);
// keep[i] = the TP at position i differs from the one before, its length if so
cudaError_t tp_order_flags(const TpOrder &o, long long P, const long long *tp_off, long long *keep_len, int *keep,
                           cudaStream_t s);
// arc_slot[M], end_slot[G] of every graph (tree_slots_block)
cudaError_t tree_slots(const GraphDev &g, int *arc_slot, int *end_slot, cudaStream_t s);

// Packed comparison keys of the TPs (vertex v as v + 1 in `bits` = 8 or 16
// bits, 64 / bits per word, most significant first; see key_words):
// key_len[i] = words of TP i, then (after a scan into key_off) the words.
cudaError_t tp_key_lengths(const long long *tp_off, long long P, int bits, long long *key_len, cudaStream_t s);
cudaError_t tp_write_keys(const long long *tp_off, const int *tp_vert, long long P, int bits, const long long *key_off,
                          unsigned long long *key, cudaStream_t s);
// packed keys (as tp_write_keys) of TP(p) for every PP p, read from the
// TP's parts (prefix path, PP, suffix path) instead of a written TP list;
// tp_off holds the TPs' offsets (for their lengths), o.key_off the keys'
cudaError_t tp_write_keys_parts(const TpOrder &o, const long long *tp_off, unsigned long long *key, long long P,
                                cudaStream_t s);
// the kept TPs in sorted order (o.perm[0], lengths between keep_off[P + 1]),
// unpacked from their keys into their final places
cudaError_t tp_assemble(const TpOrder &o, const long long *keep_off, const long long *keep_rank, long long *final_off,
                        int *out_vert, int *out_graph, long long P, cudaStream_t s);
// map[perm[i]] = the final index of sorted TP i (keep_rank[i] if it is kept,
// else that of the kept TP it duplicates, keep_rank[i] - 1); with perm null
// the identity map[i] = i
cudaError_t tp_index_map(const long long *perm, const int *keep, const long long *keep_rank, long long P, int *map,
                         cudaStream_t s);

// The whole of it for P TPs (P > 0) of one graph, in one block: result = {error
// word, TP vertices before dedup, TPs, their vertices, the longest TP}, the third,
// the fourth and all lists only if the first is 0 and the second is not V (the PPs' vertices).
// o as for the steps above, with room for P sub-runs; final_off[P + 1],
// out_vert for the vertices before dedup, pp_to_tp (tp_index_map) may be null.
struct TpSmallArgs {
    TpOrder o;
    long long P, V, slots;
    const int2 *ends;
    long long *tp_len, *tp_off, *key_off, *keep_off, *keep_rank;
    int *keep;
    unsigned long long *key;
    long long *final_off;
    int *out_vert, *out_graph;
    long long *gptr;
    int *pp_to_tp;
    long long *result;
};
cudaError_t tp_small(const TpSmallArgs &a, cudaStream_t s);

}  // namespace tpg
