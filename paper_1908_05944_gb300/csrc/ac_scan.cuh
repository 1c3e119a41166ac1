// Exclusive scan of up to SC_MAX elements in one launch: one thread-block
// cluster (or, for a few thousand elements, one block), each block with a
// contiguous chunk. Every block sums its chunk, the sums meet in distributed
// shared memory, and every block scans its chunk from the sum of the chunks
// before it. The scans of a build lie on its critical path between kernels of
// a few microseconds: two launches (tile sums, then tiles) took 11 us for
// 100,000 elements and 8 us for 2,000.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ac {

constexpr int SC_CTAS = 8;
constexpr int SC_THREADS = 1024;
constexpr int SC_ITEMS = 4;
constexpr int SC_TILE = SC_THREADS * SC_ITEMS;
constexpr int64_t SC_ONE = 2 * SC_TILE;         // up to here one block
constexpr int64_t SC_MAX = 8 * SC_CTAS * SC_TILE;  // up to here one cluster

// exclusive prefix of v over the block; *total the block's sum (sums: 33 elements of shared memory)
template <class T>
__device__ __forceinline__ T sc_block_scan(T v, T* sums, T* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) sums[w] = inc;
    __syncthreads();
    if (w == 0) {
        const T x = sums[lane];
        T i = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T t = __shfl_up_sync(0xffffffffu, i, o);
            if (lane >= o) i += t;
        }
        sums[lane] = i - x;
        if (lane == 31) sums[32] = i;
    }
    __syncthreads();
    const T r = inc - v + sums[w];
    *total = sums[32];
    __syncthreads();
    return r;
}

// in(i), i < n -> out[0 .. n], out[n] the total. in may read out itself (a
// block reads a position of its own chunk before it writes it).
template <class T, class In, bool CLUSTER>
__device__ __forceinline__ void scan_chunks(In in, T* out, int64_t n) {
    __shared__ T sums[33];
    __shared__ T part;
    int rank = 0;
    int64_t lo = 0, hi = n + 1;
    T before = 0;
    if constexpr (CLUSTER) {
        namespace cg = cooperative_groups;
        cg::cluster_group cl = cg::this_cluster();
        rank = (int)cl.block_rank();
        const int64_t chunk = (n + SC_CTAS) / SC_CTAS;
        lo = min(rank * chunk, n + 1);
        hi = min(lo + chunk, n + 1);
        T s = 0, total;
        for (int64_t i = lo + threadIdx.x; i < hi; i += SC_THREADS) s += i < n ? in(i) : T(0);
        sc_block_scan(s, sums, &total);
        if (threadIdx.x == 0) part = total;
        cl.sync();
        for (int r = 0; r < rank; r++) before += *cl.map_shared_rank(&part, r);
        cl.sync();  // no block leaves while another still reads its part
    }
    for (int64_t b = lo; b < hi; b += SC_TILE) {
        const int64_t i0 = b + (int64_t)threadIdx.x * SC_ITEMS;
        T v[SC_ITEMS], s = 0, total;
#pragma unroll
        for (int k = 0; k < SC_ITEMS; k++) {
            const int64_t i = i0 + k;
            v[k] = i < hi && i < n ? in(i) : T(0);
            s += v[k];
        }
        T pre = sc_block_scan(s, sums, &total) + before;
#pragma unroll
        for (int k = 0; k < SC_ITEMS; k++) {
            if (i0 + k < hi) out[i0 + k] = pre;
            pre += v[k];
        }
        before += total;
    }
}

template <class T, class In>
__global__ void __cluster_dims__(SC_CTAS, 1, 1) __launch_bounds__(SC_THREADS) k_scan_cluster(In in, T* out, int64_t n) {
    scan_chunks<T, In, true>(in, out, n);
}

template <class T, class In>
__global__ void __launch_bounds__(SC_THREADS) k_scan_block(In in, T* out, int64_t n) {
    scan_chunks<T, In, false>(in, out, n);
}

template <class T>
struct ScanArray {
    const T* p;
    __device__ __forceinline__ T operator()(int64_t i) const { return p[i]; }
};

// n <= SC_MAX
template <class T, class In>
static void launch_small_scan(In in, T* out, int64_t n, cudaStream_t s) {
    if (n < SC_ONE) k_scan_block<T, In><<<1, SC_THREADS, 0, s>>>(in, out, n);
    else k_scan_cluster<T, In><<<SC_CTAS, SC_THREADS, 0, s>>>(in, out, n);
}

}  // namespace ac
