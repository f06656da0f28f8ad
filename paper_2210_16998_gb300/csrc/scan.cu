// Device-wide exclusive prefix sums, no inter-block waiting: up to 8192 values in
// one block; else tile sums, and each tile adds up the sums before its own as
// long as there are at most SCAN_FEW_TILES of them (4.2M values), or takes them
// from a scan of their own in between.  A launch less for each of 333 graphs' eight
// scans: the whole call 1.546 -> 1.514 ms.
#include "common.cuh"
#include "kernels.h"

namespace tpg {

constexpr int SCAN_BLOCK = 256;
constexpr int SCAN_ITEMS = 8;
constexpr long long SCAN_TILE = (long long)SCAN_BLOCK * SCAN_ITEMS;
constexpr long long SCAN_FEW_TILES = 2048;
constexpr int SCAN_ONE = 1024;  // threads of the one-block scans

size_t scan_tmp_elems(long long n) { return (size_t)((n + SCAN_TILE - 1) / SCAN_TILE) + 2; }

template <typename T>
__global__ void __launch_bounds__(SCAN_BLOCK) scan_reduce_kernel(const T *in, long long n, long long *tile_sums) {
    const long long base = blockIdx.x * SCAN_TILE;
    long long s = 0;
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        const long long i = base + (long long)j * SCAN_BLOCK + threadIdx.x;
        if (i < n) s += (long long)in[i];
    }
    long long total;
    block_excl_scan_i64<SCAN_BLOCK>(s, total);
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(SCAN_ONE) scan_tile_sums_kernel(long long *tile_sums, long long ntiles) {
    long long carry = 0;
    for (long long base = 0; base < ntiles; base += SCAN_ONE) {
        const long long i = base + threadIdx.x;
        const long long v = (i < ntiles) ? tile_sums[i] : 0;
        long long total;
        const long long ex = block_excl_scan_i64<SCAN_ONE>(v, total);
        if (i < ntiles) tile_sums[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) tile_sums[ntiles] = carry;
}

// RAW: tile_sums holds the sums themselves, else their prefix
template <typename T, bool RAW>
__global__ void __launch_bounds__(SCAN_BLOCK) scan_down_kernel(const T *in, long long *out, long long n,
                                                               const long long *tile_sums, long long ntiles) {
    const long long base = blockIdx.x * SCAN_TILE + (long long)threadIdx.x * SCAN_ITEMS;
    long long v[SCAN_ITEMS];
    long long s = 0, before = 0;
    if constexpr (RAW)
        for (long long i = threadIdx.x; i < blockIdx.x; i += SCAN_BLOCK) before += tile_sums[i];
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        const long long i = base + j;
        v[j] = (i < n) ? (long long)in[i] : 0;
        s += v[j];
    }
    long long total;
    if constexpr (RAW) block_excl_scan_i64<SCAN_BLOCK>(before, before);
    else before = tile_sums[blockIdx.x];
    long long run = block_excl_scan_i64<SCAN_BLOCK>(s, total) + before;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        const long long i = base + j;
        if (i < n) out[i] = run;
        run += v[j];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = RAW ? before + total : tile_sums[ntiles];
}

template <typename T>
__global__ void __launch_bounds__(SCAN_ONE) scan_one_kernel(const T *in, long long *out, int n) {
    const int base = threadIdx.x * SCAN_ITEMS;
    long long v[SCAN_ITEMS];
    long long s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        v[j] = base + j < n ? (long long)in[base + j] : 0;
        s += v[j];
    }
    long long total;
    long long run = block_excl_scan_i64<SCAN_ONE>(s, total);
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        if (base + j < n) out[base + j] = run;
        run += v[j];
    }
    if (threadIdx.x == 0) out[n] = total;
}

__global__ void scan_empty_kernel(long long *out) { out[0] = 0; }

template <typename T>
static cudaError_t scan_impl(const T *in, long long *out, long long n, long long *tmp, cudaStream_t s) {
    if (n <= 0) {
        scan_empty_kernel<<<1, 1, 0, s>>>(out);
        note_launch();
        return cudaGetLastError();
    }
    if (n <= (long long)SCAN_ONE * SCAN_ITEMS) {
        scan_one_kernel<T><<<1, SCAN_ONE, 0, s>>>(in, out, (int)n);
        note_launch();
        return cudaGetLastError();
    }
    const long long ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    scan_reduce_kernel<T><<<(unsigned)ntiles, SCAN_BLOCK, 0, s>>>(in, n, tmp);
    note_launch();
    if (ntiles <= SCAN_FEW_TILES) {
        scan_down_kernel<T, true><<<(unsigned)ntiles, SCAN_BLOCK, 0, s>>>(in, out, n, tmp, ntiles);
        note_launch();
        return cudaGetLastError();
    }
    scan_tile_sums_kernel<<<1, SCAN_ONE, 0, s>>>(tmp, ntiles);
    note_launch();
    scan_down_kernel<T, false><<<(unsigned)ntiles, SCAN_BLOCK, 0, s>>>(in, out, n, tmp, ntiles);
    note_launch();
    return cudaGetLastError();
}

cudaError_t scan_i64(const long long *in, long long *out, long long n, long long *tmp, cudaStream_t s) {
    return scan_impl<long long>(in, out, n, tmp, s);
}

// The two halves of scan_i64: the first leaves the tile prefixes in tmp and
// the total at tmp[scan_total_index(n)]; the second writes out[0..n].
cudaError_t scan_i64_sums(const long long *in, long long n, long long *tmp, cudaStream_t s) {
    if (n <= 0) {
        scan_empty_kernel<<<1, 1, 0, s>>>(tmp);
        note_launch();
        return cudaGetLastError();
    }
    const long long ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    scan_reduce_kernel<long long><<<(unsigned)ntiles, SCAN_BLOCK, 0, s>>>(in, n, tmp);
    scan_tile_sums_kernel<<<1, SCAN_ONE, 0, s>>>(tmp, ntiles);
    note_launch(2);
    return cudaGetLastError();
}
long long scan_total_index(long long n) { return n <= 0 ? 0 : (n + SCAN_TILE - 1) / SCAN_TILE; }
cudaError_t scan_i64_finish(const long long *in, long long *out, long long n, const long long *tmp, cudaStream_t s) {
    if (n <= 0) {
        scan_empty_kernel<<<1, 1, 0, s>>>(out);
        note_launch();
        return cudaGetLastError();
    }
    const long long ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    scan_down_kernel<long long, false><<<(unsigned)ntiles, SCAN_BLOCK, 0, s>>>(in, out, n, tmp, ntiles);
    note_launch();
    return cudaGetLastError();
}

cudaError_t scan_i32_to_i64(const int *in, long long *out, long long n, long long *tmp, cudaStream_t s) {
    return scan_impl<int>(in, out, n, tmp, s);
}

}  // namespace tpg
