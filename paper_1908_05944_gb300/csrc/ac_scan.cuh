// Exclusive scan of up to SC_MAX elements in one launch: one thread-block
// cluster of SC_CTAS blocks (or, for a few thousand elements, one block), ITEMS
// elements per thread. Every thread loads its elements once, every
// block scans its threads' sums, the blocks exchange theirs in distributed shared
// memory. A build's scans lie on its critical path between kernels of a few
// microseconds: two launches (tile sums, then tiles that add the sums before
// them) take 11 us for 100,000 elements and 8 us for 2,000, this one 10 and 4 (and
// one launch fewer).
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ac {

constexpr int SC_CTAS = 8;
constexpr int SC_THREADS = 1024;
constexpr int SC_ITEMS_MAX = 16;
constexpr int64_t SC_MAX = (int64_t)SC_CTAS * SC_THREADS * SC_ITEMS_MAX - 1;  // n + 1 outputs

// in(i), i < n -> out[0 .. n], out[n] the total. A warp takes 32 ITEMS elements in a
// row, 32 per step (coalesced; with ITEMS in a row per thread every access touched
// 32 lines: 21 us for 100,000 elements). in may read out itself: a thread reads
// all its elements before it writes any.
template <class T, class In, int ITEMS, bool CLUSTER>
__device__ __forceinline__ void scan_chunk(In in, T* out, int64_t n) {
    __shared__ T sums[33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i0 = ((int64_t)blockIdx.x * (SC_THREADS / 32) + w) * (32 * ITEMS) + lane;
    T v[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; k++) v[k] = i0 + 32 * k < n ? in(i0 + 32 * k) : T(0);
    T carry = 0;
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {  // v[k]: exclusive within the warp's elements
        T inc = v[k];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        v[k] = carry + inc - v[k];
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) sums[w] = carry;
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
    T pre = 0;
    if constexpr (CLUSTER) {
        namespace cg = cooperative_groups;
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();
        const int rank = (int)cl.block_rank();
#pragma unroll
        for (int r = 0; r < SC_CTAS - 1; r++)
            if (r < rank) pre += *cl.map_shared_rank(&sums[32], r);
        pre += sums[w];
        cl.sync();  // no block leaves while another still reads its sum
    } else {
        __syncthreads();
        pre = sums[w];
    }
#pragma unroll
    for (int k = 0; k < ITEMS; k++)
        if (i0 + 32 * k <= n) out[i0 + 32 * k] = v[k] + pre;
}

template <class T, class In, int ITEMS>
__global__ void __cluster_dims__(SC_CTAS, 1, 1) __launch_bounds__(SC_THREADS) k_scan_cluster(In in, T* out, int64_t n) {
    scan_chunk<T, In, ITEMS, true>(in, out, n);
}

template <class T, class In, int ITEMS>
__global__ void __launch_bounds__(SC_THREADS) k_scan_block(In in, T* out, int64_t n) {
    scan_chunk<T, In, ITEMS, false>(in, out, n);
}

template <class T>
struct ScanArray {
    const T* p;
    __device__ __forceinline__ T operator()(int64_t i) const { return p[i]; }
};

// n <= SC_MAX
template <class T, class In>
static void launch_small_scan(In in, T* out, int64_t n, cudaStream_t s) {
    if (n < 4 * SC_THREADS) k_scan_block<T, In, 4><<<1, SC_THREADS, 0, s>>>(in, out, n);
    else if (n < 4 * SC_CTAS * SC_THREADS) k_scan_cluster<T, In, 4><<<SC_CTAS, SC_THREADS, 0, s>>>(in, out, n);
    else if (n < 8 * SC_CTAS * SC_THREADS) k_scan_cluster<T, In, 8><<<SC_CTAS, SC_THREADS, 0, s>>>(in, out, n);
    else k_scan_cluster<T, In, SC_ITEMS_MAX><<<SC_CTAS, SC_THREADS, 0, s>>>(in, out, n);
}

}  // namespace ac
