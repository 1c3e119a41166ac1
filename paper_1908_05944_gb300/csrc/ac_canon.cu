// Canonical simplex lists and filtration values.
//
// Steps 3-5 of Section 3.1 (arXiv 1908.05944): K^d is the set of facets of
// K^(d+1) together with the simplices of Sigma_ortho^d that pass AC2 at their
// orthocentre. The per-atom pass emitted the latter. K^3 and the potential
// simplices, each emitted once, are mapped to input indices, sorted ascending,
// bucketed by their first vertex (counting sort over input indices) and sorted
// inside each bucket. K^2 and K^1 are marked bits over the neighbour rows, where
// a simplex that comes from both sources sets the same bit, and are written in
// order from the marks. A simplex that arrives only as a facet fails AC2 at its
// own orthocentre: it is "attached".
//
// Filtration value Size (Section 2.3): an unattached simplex's closest witness
// is its orthocentre, so Size = OrthoSize; an attached simplex's closest
// witness lies on a face of its witness region, i.e. it is a witness of a
// coface with the same Size (the argument of Lemmas 1 and 2), so Size is the
// smallest Size of its cofaces one dimension up. Ties pick the coface that
// comes first in lexicographic order. OrthoSize is an exact rational of
// 128-bit integers, converted to FP64 with three roundings (relative error
// below 4 * 2^-53).
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "ac_internal.cuh"
#include "ac_bucket.h"
#include "ac_round.h"
#include "ac_scan.cuh"

namespace ac {

// ---------------------------------------------------------------------------
// helpers

__device__ __forceinline__ void sort_asc(int4& t, int K) {
    // tiny sorting network on the first K components
    auto cs = [](int& a, int& b) {
        if (a > b) {
            int x = a;
            a = b;
            b = x;
        }
    };
    if (K == 2) {
        cs(t.x, t.y);
    } else if (K == 3) {
        cs(t.x, t.y);
        cs(t.y, t.z);
        cs(t.x, t.y);
    } else {
        cs(t.x, t.y);
        cs(t.z, t.w);
        cs(t.x, t.z);
        cs(t.y, t.w);
        cs(t.y, t.z);
    }
}

// The items of one list, K entries each, emitted once each by their owner:
// nA tuples of sorted positions (a4, or a2 for edges), taken to ascending tuples
// of input indices. An item's bucket is its first vertex.
struct CanonArgs {
    const int4* a4;
    const int2* a2;
    int64_t nA;
    const int32_t* order;  // sorted position -> input index
    int64_t* bucket_cnt;   // items per bucket; the scatter counts it down to 0
    const int64_t* off;    // scatter pass: bucket offsets
    int4* T;               // scattered items
};

template <int K>
__device__ __forceinline__ int4 canon_item(const CanonArgs& a, int64_t j) {
    int4 t;
    if (K == 2) {
        const int2 e = a.a2[j];
        t = make_int4(a.order[e.x], a.order[e.y], -1, -1);
    } else {
        const int4 e = a.a4[j];
        t = make_int4(a.order[e.x], a.order[e.y], a.order[e.z], K == 4 ? a.order[e.w] : -1);
    }
    sort_asc(t, K);
    return t;
}

// Items in a warp that share a bucket add to its counter once.
template <int K>
__global__ void k_canon_count(CanonArgs a) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = j < a.nA;
    const int lane = threadIdx.x & 31;
    const int x = valid ? canon_item<K>(a, j).x : -1 - lane;
    const unsigned peers = __match_any_sync(0xffffffffu, x);
    if (valid && (peers & ((1u << lane) - 1u)) == 0)
        atomicAdd((unsigned long long*)&a.bucket_cnt[x], (unsigned long long)__popc(peers));
}

template <int K>
__global__ void k_canon_scatter(CanonArgs a) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = j < a.nA;
    const int lane = threadIdx.x & 31;
    int4 t = make_int4(-1 - lane, 0, 0, 0);
    if (valid) t = canon_item<K>(a, j);
    const unsigned peers = __match_any_sync(0xffffffffu, t.x);
    const int leader = __ffs(peers) - 1;
    unsigned long long base = 0;
    if (valid && lane == leader) {
        const unsigned long long k = (unsigned long long)__popc(peers);
        base = atomicAdd((unsigned long long*)&a.bucket_cnt[t.x], 0ull - k) - k;
    }
    base = __shfl_sync(0xffffffffu, base, leader);
    if (valid) a.T[a.off[t.x] + (int64_t)base + __popc(peers & ((1u << lane) - 1u))] = t;
}

// In-bucket sort, one warp per bucket, which then writes its rows. Up to 32 items
// every lane ranks its own among the others; up to CSORT_MAX a bitonic network
// sorts them in registers, R = ceil(k/32) per lane (padded to a power of two
// with the largest key), exchanges across lanes by shuffles, across a lane's
// registers directly. The rest of each tuple is the sort key: K = 2: y; K = 3:
// (y << 32) | z; K = 4: hi = (y << 32) | z, lo = w. The items are distinct; two
// equal ones (a bug) raise DERR_INTERNAL.
constexpr int CSORT_MAX = 256;
constexpr int CSORT_WARPS = 4;

struct SortSmem {
    unsigned long long ohi[CSORT_MAX];
    unsigned olo[CSORT_MAX];
};

template <int K>
__device__ __forceinline__ void make_key(const int4& t, unsigned long long& hi, unsigned& lo) {
    const unsigned long long y = (unsigned)t.y, z = (unsigned)t.z;
    hi = K == 2 ? y : (y << 32) | z;
    lo = K == 4 ? (unsigned)t.w : 0u;
}

template <int K, class H>
__device__ __forceinline__ bool key_less(H ah, unsigned al, H bh, unsigned bl) {
    return K == 4 ? (ah < bh || (ah == bh && al < bl)) : ah < bh;
}

// register type of the high key: edges' keys fit 32 bits
template <int K>
using KeyHi = typename std::conditional<K == 2, unsigned, unsigned long long>::type;

template <int K, int R>
__device__ __forceinline__ void bitonic_place(SortSmem& S, const int4* __restrict__ T, int64_t a, int k, int lane) {
    using H = KeyHi<K>;
    H h[R];
    unsigned l[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int e = 32 * r + lane;
        if (e < k) {
            unsigned long long hi;
            make_key<K>(T[a + e], hi, l[r]);
            h[r] = (H)hi;
        } else {
            h[r] = (H)~0ull;
            l[r] = ~0u;
        }
    }
    constexpr int N = 32 * R;
#pragma unroll
    for (int size = 2; size <= N; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {
                const int rs = stride >> 5;
#pragma unroll
                for (int r = 0; r < R; r++) {
                    if ((r & rs) == 0) {
                        const int r2 = r | rs;
                        const bool asc = ((32 * r + lane) & size) == 0;
                        if (key_less<K>(h[r2], l[r2], h[r], l[r]) == asc) {
                            const H th = h[r];
                            h[r] = h[r2];
                            h[r2] = th;
                            const unsigned tl = l[r];
                            l[r] = l[r2];
                            l[r2] = tl;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const H oh = __shfl_xor_sync(0xffffffffu, h[r], stride);
                    const unsigned ol = K == 4 ? __shfl_xor_sync(0xffffffffu, l[r], stride) : 0u;
                    const bool asc = ((32 * r + lane) & size) == 0;
                    const bool lower = (lane & stride) == 0;
                    // the lower position keeps the smaller key when ascending
                    const bool take = (lower == asc) ? key_less<K>(oh, ol, h[r], l[r]) : key_less<K>(h[r], l[r], oh, ol);
                    if (take) {
                        h[r] = oh;
                        l[r] = ol;
                    }
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int e = 32 * r + lane;
        if (e < k) {
            S.ohi[e] = (unsigned long long)h[r];
            if (K == 4) S.olo[e] = l[r];
        }
    }
}

struct CanonOut {
    const int32_t* mol_of;   // input index -> molecule
    const int64_t* mol_off;  // molecule -> first input index
    int4* G;                 // canonical rows, global input indices
    int32_t* out;            // packed rows, per-molecule local indices
    uint8_t* attached;
    unsigned* err;
};

template <int K>
__device__ __forceinline__ void canon_row(const CanonOut& o, int64_t row, int4 t, int base) {
    if (K < 4) t.w = -1;
    if (K < 3) t.z = -1;
    o.G[row] = t;
    if (K == 4) {
        reinterpret_cast<int4*>(o.out)[row] = make_int4(t.x - base, t.y - base, t.z - base, t.w - base);
    } else {
        o.out[row * K + 0] = t.x - base;
        o.out[row * K + 1] = t.y - base;
        if (K == 3) o.out[row * K + 2] = t.z - base;
    }
    o.attached[row] = 0;  // list items passed AC2 at their orthocentre
}

template <int K>
__global__ void __launch_bounds__(CSORT_WARPS * 32) k_canon_sort(int4* __restrict__ T, const int64_t* __restrict__ off,
                                                                  int64_t n, CanonOut o) {
    __shared__ SortSmem sm[CSORT_WARPS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    SortSmem& S = sm[w];
    const int64_t warps = (int64_t)gridDim.x * CSORT_WARPS;
    for (int64_t g = (int64_t)blockIdx.x * CSORT_WARPS + w; g < n; g += warps) {
        const int64_t a = off[g];
        const int64_t kb = off[g + 1] - a;
        if (kb == 0) continue;
        const int k = kb > CSORT_MAX ? CSORT_MAX + 1 : (int)kb;
        const int base = (int)o.mol_off[o.mol_of[g]];
        if (k <= 32) {
            int4 t = make_int4(0, 0, 0, 0);
            unsigned long long hi = ~0ull;
            unsigned lo = ~0u;
            if (lane < k) {
                t = T[a + lane];
                make_key<K>(t, hi, lo);
            }
            int r = 0, same = 0;
            for (int u = 0; u < k; u++) {
                const unsigned long long hu = __shfl_sync(0xffffffffu, hi, u);
                const unsigned lu = __shfl_sync(0xffffffffu, lo, u);
                r += key_less<K, unsigned long long>(hu, lu, hi, lo) ? 1 : 0;
                same += hu == hi && lu == lo ? 1 : 0;
            }
            if (lane < k) {
                if (same != 1) atomicOr(o.err, DERR_INTERNAL);
                canon_row<K>(o, a + r, t, base);
            }
            continue;
        }
        if (k > CSORT_MAX) {
            // rare: one lane, heap sort in place (O(k log k))
            if (lane == 0 && sort_unique_bucket<K>(T, a, a + kb) != kb) atomicOr(o.err, DERR_INTERNAL);
            __syncwarp();
            for (int64_t i = lane; i < kb; i += 32) canon_row<K>(o, a + i, T[a + i], base);
            continue;
        }
        if (k <= 64) bitonic_place<K, 2>(S, T, a, k, lane);
        else if (k <= 128) bitonic_place<K, 4>(S, T, a, k, lane);
        else bitonic_place<K, 8>(S, T, a, k, lane);
        __syncwarp();
        for (int i = lane; i < k; i += 32) {
            const unsigned long long hi = S.ohi[i];
            if (i > 0 && S.ohi[i - 1] == hi && (K < 4 || S.olo[i - 1] == S.olo[i])) atomicOr(o.err, DERR_INTERNAL);
            int4 t = make_int4((int)g, 0, 0, 0);
            t.y = K == 2 ? (int)(unsigned)hi : (int)(hi >> 32);
            if (K >= 3) t.z = (int)(unsigned)hi;
            if (K == 4) t.w = (int)S.olo[i];
            canon_row<K>(o, a + i, t, base);
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// canonicalise one dimension

using Work = CanonWork;

// One list from items emitted once each: their number is the row count. Its
// buffers are reserved on stream s; its kernels run on stream t (s, or a stream
// that waits here for s).
template <int K>
static int canon_dim_k(ac_ctx* c, const int4* a4, const int2* a2, int64_t nA, SimplexList& L, DevBuf& Gout, Work& w,
                       cudaStream_t s, cudaStream_t t) {
    const int64_t n = c->n;
    AC_TRY(w.T.reserve((size_t)(nA + 1) * sizeof(int4), s));
    AC_TRY(w.cnt.reserve((size_t)(n + 1) * sizeof(int64_t), s));
    AC_TRY(L.v0_off.reserve((size_t)(n + 1) * sizeof(int64_t), s));
    int64_t* cnt = w.cnt.as<int64_t>();
    int64_t* off = L.v0_off.as<int64_t>();  // the rows start where the buckets do
    if (c->replaying) AC_TRY(expect_i64(c, off + n, L.count, s));  // the recorded build's count
    else L.count = nA;
    L.cap = L.count;
    L.d_count = nullptr;
    const size_t rows = (size_t)(L.count > 0 ? L.count : 1);
    AC_TRY(L.tuples.reserve(rows * K * sizeof(int32_t), s));
    AC_TRY(L.attached.reserve(rows, s));
    AC_TRY(L.f.reserve(rows * sizeof(double), s));
    AC_TRY(L.orthosize.reserve(rows * sizeof(double), s));
    AC_TRY(L.src_dim.reserve(rows, s));
    AC_TRY(L.src_idx.reserve(rows * sizeof(int64_t), s));
    AC_TRY(Gout.reserve(rows * sizeof(int4), s));
    if (t != s) {
        AC_CUDA(cudaEventRecord(c->ev_fork, s));
        AC_CUDA(cudaStreamWaitEvent(t, c->ev_fork, 0));
    }
    AC_CUDA(cudaMemsetAsync(cnt, 0, (size_t)(n + 1) * sizeof(int64_t), t));
    CanonArgs ca{a4, a2, nA, c->order.as<int32_t>(), cnt, off, w.T.as<int4>()};
    const unsigned gi = (unsigned)((nA + 255) / 256);
    if (nA > 0) {
        k_canon_count<K><<<gi, 256, 0, t>>>(ca);
        AC_LAUNCHED();
    }
    AC_TRY(scan_exclusive_i64(c, cnt, off, n, t));
    if (nA > 0) {
        k_canon_scatter<K><<<gi, 256, 0, t>>>(ca);
        AC_LAUNCHED();
        int dev = 0, sms = 0, per_sm = 0;
        AC_CUDA(cudaGetDevice(&dev));
        AC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        AC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_canon_sort<K>, CSORT_WARPS * 32, 0));
        // one resident wave, buckets taken grid-stride
        int64_t blocks = (n + CSORT_WARPS - 1) / CSORT_WARPS;
        if (blocks > (int64_t)sms * (per_sm > 0 ? per_sm : 1)) blocks = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
        CanonOut o{c->mol_of.as<int32_t>(), c->d_moloff.as<int64_t>(), Gout.as<int4>(), L.tuples.as<int32_t>(),
                   L.attached.as<uint8_t>(), &c->counters.as<DevCounters>()->err};
        k_canon_sort<K><<<(unsigned)blocks, CSORT_WARPS * 32, 0, t>>>(w.T.as<int4>(), off, n, o);
        AC_LAUNCHED();
    }
    return AC_OK;
}

static int canon_dim(ac_ctx* c, int d, const int4* a4, const int2* a2, int64_t nA, SimplexList& L, DevBuf& Gout, Work& w,
                     cudaStream_t s, cudaStream_t t) {
    switch (d) {
        case 1: return canon_dim_k<2>(c, a4, a2, nA, L, Gout, w, s, t);
        case 2: return canon_dim_k<3>(c, a4, a2, nA, L, Gout, w, s, t);
        default: return canon_dim_k<4>(c, a4, a2, nA, L, Gout, w, s, t);
    }
}

// ---------------------------------------------------------------------------
// K^1 by marks (Step 4 for edges). An edge of K^1 joins two atoms whose grown
// balls meet (its OrthoSize is at most alpha), so its second vertex is an
// entry of the neighbour row of its first vertex (smallest input index); the
// rows list grid-sorted positions in ascending order. The free edges and the
// three edges of every K^2 triangle set bits over those rows (bit OR: a
// duplicate changes nothing, so nothing is sorted or removed), a second mask
// keeps the free edges, and each atom writes its marked entries as rows in
// ascending input order.

struct EdgeMarkArgs {
    const int2* free_e;  // free edges (sorted positions), nA of them
    int64_t nA;
    const int4* tri;     // K^2 rows (global input indices), nB of them
    RowCount nB;
    const int32_t* order;  // sorted position -> input index
    const int32_t* rank;   // input index -> sorted position
    const int64_t* nb_off; // offsets (stride 0) or counts (stride > 0)
    const int32_t* nb;
    int stride;
    int words;             // mask words per atom
    unsigned* m_in;        // per sorted position: entry of the row is an edge of K^1
    unsigned* m_free;      // ... and a free edge
    unsigned long long* rows;  // per input index: distinct marked edges (the atom's row count)
    unsigned* err;
};

__device__ __forceinline__ void edge_row(const EdgeMarkArgs& a, int s, int64_t& off, int& m) {
    if (a.stride) {
        off = (int64_t)s * a.stride;
        m = min((int)a.nb_off[s], a.stride);
    } else {
        off = a.nb_off[s];
        m = (int)(a.nb_off[s + 1] - off);
    }
}

// Positions e[k] of x[k] in the ascending rows [off[k], off[k] + m[k]), or -1. The
// searches are chains of dependent loads: they step together, one load of each
// in flight. That is what small builds wait for (k_edge_mark of 2,000 atoms 9.2
// -> 8.0 us, the facet searches below 26 -> 17); large ones are bound by the
// number of lines touched and see no difference.
template <int N>
__device__ __forceinline__ void row_find(const int32_t* __restrict__ nb, const int64_t (&off)[N], const int (&m)[N],
                                         const int (&x)[N], int (&e)[N]) {
    int lo[N], n[N];
#pragma unroll
    for (int k = 0; k < N; k++) {
        lo[k] = 0;
        n[k] = m[k];
    }
    for (bool more = true; more;) {
        int v[N];
#pragma unroll
        for (int k = 0; k < N; k++) v[k] = n[k] > 0 ? nb[off[k] + lo[k] + (n[k] >> 1)] : 0;
        more = false;
#pragma unroll
        for (int k = 0; k < N; k++) {
            const int half = n[k] >> 1;
            if (n[k] > 0 && v[k] < x[k]) {
                lo[k] += half + 1;
                n[k] -= half + 1;
            } else {
                n[k] = half;
            }
            more = more || n[k] > 0;
        }
    }
#pragma unroll
    for (int k = 0; k < N; k++) e[k] = lo[k] < m[k] && nb[off[k] + lo[k]] == x[k] ? lo[k] : -1;
}

// bit e of sorted position su's row mask; the first setting of a bit counts a
// row for input index gu (duplicates leave the count as it is)
__device__ __forceinline__ void mark_bit(const EdgeMarkArgs& a, int su, int gu, int e, bool fr) {
    if (e < 0) {
        atomicOr(a.err, DERR_INTERNAL);  // an edge of K^1 between atoms whose balls do not meet: impossible
        return;
    }
    const int64_t w = (int64_t)su * a.words + (e >> 5);
    const unsigned bit = 1u << (e & 31);
    // an edge is marked by every triangle around it: a mark that a plain load already sees (bits are only
    // ever set, so a stale copy at worst costs the atomic) needs none
    if (!fr && (a.m_in[w] & bit)) return;
    if (!(atomicOr(&a.m_in[w], bit) & bit)) atomicAdd(&a.rows[gu], 1ull);
    if (fr) atomicOr(&a.m_free[w], bit);
}

// threads [0, nA): one free edge each; then one K^2 triangle (a < b < c) each:
// (a, b) and (a, c) in a's row, (b, c) in b's row
__global__ void k_edge_mark(EdgeMarkArgs a) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= a.nA + a.nB.get()) return;
    int64_t off;
    int m;
    if (j < a.nA) {
        const int2 e = a.free_e[j];
        int gu = a.order[e.x], gv = a.order[e.y];
        int su = e.x, sv = e.y;
        if (gu > gv) {
            su = e.y;
            sv = e.x;
            gu = gv;
        }
        edge_row(a, su, off, m);
        const int64_t offs[1] = {off};
        const int ms[1] = {m}, xs[1] = {sv};
        int es[1];
        row_find<1>(a.nb, offs, ms, xs, es);
        mark_bit(a, su, gu, es[0], true);
        return;
    }
    const int4 t = a.tri[j - a.nA];
    const int sa = a.rank[t.x], sb = a.rank[t.y], sc = a.rank[t.z];
    edge_row(a, sa, off, m);
    int64_t offb;
    int mb;
    edge_row(a, sb, offb, mb);
    const int64_t offs[3] = {off, off, offb};
    const int ms[3] = {m, m, mb}, xs[3] = {sb, sc, sc};
    int es[3];
    row_find<3>(a.nb, offs, ms, xs, es);
    mark_bit(a, sa, t.x, es[0], false);
    mark_bit(a, sa, t.x, es[1], false);
    mark_bit(a, sb, t.y, es[2], false);
}

// the marked entries of g's row, ranked by input index: one warp per atom;
// the marked entries' input indices are compacted into shared memory, then
// each marked lane counts the smaller ones
constexpr int EW_WARPS = 4;

__global__ void __launch_bounds__(EW_WARPS * 32) k_edge_write(EdgeMarkArgs a, int64_t n, const int64_t* __restrict__ uoff,
                                                              const int32_t* __restrict__ mol_of,
                                                              const int64_t* __restrict__ mol_off, int4* __restrict__ G,
                                                              int32_t* __restrict__ out, uint8_t* __restrict__ attached,
                                                              uint8_t* __restrict__ endpoint) {
    __shared__ int hs_all[EW_WARPS][MAX_DEGREE];  // an atom's marked entries: at most its row length
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    int* hs = hs_all[wib];
    // atoms in grid order: their rows and masks are read in sequence
    const int64_t s = (int64_t)blockIdx.x * EW_WARPS + wib;
    if (s >= n) return;
    const int64_t g = a.order[s];
    const unsigned* mw = a.m_in + s * a.words;
    const unsigned* fw = a.m_free + s * a.words;
    int64_t off;
    int m;
    edge_row(a, (int)s, off, m);
    const int64_t row0 = uoff[g];
    const int base = (int)mol_off[mol_of[g]];
    // pass 1: compact the marked entries (input index, free bit) in entry order
    int c = 0;
    for (int w = 0; w < a.words; w++) {
        const unsigned bits = mw[w];  // the same word for the whole warp
        if (!bits) continue;
        const bool mine = (bits >> lane) & 1u;
        if (mine) {
            const int h = a.order[a.nb[off + 32 * w + lane]];
            hs[c + __popc(bits & ((1u << lane) - 1u))] = h;
        }
        c += __popc(bits);
    }
    __syncwarp();
    // the vertices of K^1 (Step 5: endpoints are in K^0); only ones are written
    if (lane == 0 && c > 0) endpoint[g] = 1;
    // pass 2: rank each compacted entry among the others
    for (int k = lane; k < c; k += 32) {
        const int h = hs[k];
        int r = 0;
        for (int q = 0; q < c; q++) r += hs[q] < h;
        // the free bit of the k-th marked entry
        int rem = k, w = 0;
        unsigned bits = mw[0];
        while (rem >= __popc(bits)) {
            rem -= __popc(bits);
            bits = mw[++w];
        }
        for (int t = 0; t < rem; t++) bits &= bits - 1;
        const int e = __ffs(bits) - 1;
        const int64_t row = row0 + r;
        G[row] = make_int4((int)g, h, -1, -1);
        out[row * 2 + 0] = (int)g - base;
        out[row * 2 + 1] = h - base;
        attached[row] = (fw[w] >> e) & 1u ? 0 : 1;
        endpoint[h] = 1;
    }
}

// Up to this many atoms a build does not wait for the row counts of K^2, K^1 and
// K^0 one after another (about 13 us each, GPU idle): their buffers and launches
// cover an upper bound known after the per-atom pass (about 2.5 times the rows)
// and the kernels read the counts on the device. Above, the memory costs more
// than three waits (2 % of a 100,000-atom build).
//
// A context keeps these buffers (60,000 atoms with probe radii: 413 MB in all,
// 240 with buffers of the rows' sizes), so the bytes beyond the rows are bounded:
// while the contexts of the process hold more than DEFER_MAX_SLACK of them (as much
// as the pool keeps of freed memory), further builds wait for their counts, and so
// does one that the device has no room for (ac_build). The lists are the same
// either way. Rebuilds of 1,024 contexts of 500 to 50,000 atoms kept side by side
// (29 GB of such bytes): 22.0 M atoms/s without a bound, 21.2 with this one, 20.6
// with one of 4 GB, 20.4 when every build waits.
constexpr int64_t DEFER_MAX_ATOMS = 65536;
constexpr int64_t DEFER_MAX_SLACK = (int64_t)16 << 30;
static std::atomic<int64_t> g_slack{0};

// upper bounds: a row of K^2 is a free triangle or a facet of a K^3 row; an edge
// of K^1 joins neighbours, and is free or an edge of a K^2 row
static int64_t tri_rows_bound(const DevCounters& h) { return (int64_t)h.n_tri_pass + 4 * (int64_t)h.n_tet_out; }
static int64_t edge_rows_bound(const ac_ctx* c, int64_t tri_rows) {
    return std::min((c->nb_total + 1) / 2, (int64_t)c->hc.n_edge_pass + 3 * tri_rows);
}

// bytes per row of list d (0..2): indices, flag, two values, source, canonical row, coface key and argmin, facet rows
static int64_t list_row_bytes(int d) { return 4 * (d + 1) + 1 + 2 * 8 + 9 + 16 + 2 * 8 + (d > 0 ? 8 * (d + 1) : 0); }

static bool may_defer(ac_ctx* c) {
    if (c->replaying || c->opt.host_results || c->no_defer || c->n > DEFER_MAX_ATOMS) return false;
    const int64_t tri = tri_rows_bound(c->hc);
    const int64_t all = c->n * list_row_bytes(0) + edge_rows_bound(c, tri) * list_row_bytes(1) + tri * list_row_bytes(2);
    if (all <= c->slack_lists) return true;  // it holds such lists already
    const int64_t more = all - c->slack;  // as if there were no rows, until they are counted
    if (g_slack.fetch_add(more) + more > DEFER_MAX_SLACK) {
        g_slack.fetch_sub(more);
        return false;
    }
    c->slack = c->slack_lists = all;
    return true;
}

void settle_slack(ac_ctx* c) {
    int64_t now = 0;
    for (int d = 0; d < 3; d++) now += (c->K[d].cap - c->K[d].count) * list_row_bytes(d);
    g_slack.fetch_add(now - c->slack);
    c->slack = now;
}

void forget_slack(ac_ctx* c) {
    g_slack.fetch_sub(c->slack);
    c->slack = c->slack_lists = 0;
}

void drop_lists(ac_ctx* c) {
    for (int d = 0; d < 3; d++) {
        SimplexList& L = c->K[d];
        for (DevBuf* b : {&L.tuples, &L.attached, &L.f, &L.orthosize, &L.src_dim, &L.src_idx, &c->Gbuf[d], &c->fkey[d],
                          &c->fargs[d], &c->frows[d]})
            *b = DevBuf{};
    }
    forget_slack(c);
}

// The row count of a list whose total the scan left at d_total (at most bound).
static int list_rows(ac_ctx* c, SimplexList& L, const int64_t* d_total, int64_t bound, cudaStream_t s) {
    L.d_count = nullptr;
    if (c->replaying) {
        AC_TRY(expect_i64(c, d_total, L.count, s));  // the recorded build's count
    } else if (c->deferred) {
        L.count = bound;  // until the build's last wait
        L.d_count = d_total;
    } else {
        AC_CUDA(cudaMemcpyAsync(c->h_stage, d_total, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        AC_TRY(sync_host(c, s));
        L.count = c->h_stage[0];
    }
    L.cap = L.count;
    return AC_OK;
}

static int canon_edges_by_marks(ac_ctx* c, cudaStream_t s) {
    const DevCounters& h = c->hc;
    const int64_t n = c->n;
    SimplexList& L = c->K[1];
    const int words = (h.max_degree + 31) / 32 > 0 ? (h.max_degree + 31) / 32 : 1;
    const size_t nn = (size_t)(n > 0 ? n : 1);
    // one buffer, emptied at once: row counts, the two masks, K^1's endpoint flags (for K^0)
    DevBuf& masks = c->scratch[2];
    const size_t o_mask = nn * sizeof(int64_t), o_end = o_mask + 2 * nn * words * sizeof(unsigned);
    AC_TRY(masks.reserve(o_end + nn, s));
    AC_TRY(L.v0_off.reserve((nn + 1) * sizeof(int64_t), s));
    AC_CUDA(cudaMemsetAsync(masks.p, 0, o_end + nn, s));
    int64_t* cnt = masks.as<int64_t>();
    unsigned* mask = reinterpret_cast<unsigned*>(masks.as<char>() + o_mask);
    c->endpoint = masks.as<uint8_t>() + o_end;
    EdgeMarkArgs a{c->edge_pass.as<int2>(), (int64_t)h.n_edge_pass, c->Gbuf[2].as<int4>(),
                   RowCount{c->K[2].cap, c->K[2].d_count},
                   c->order.as<int32_t>(), c->rank.as<int32_t>(), c->nb_cnt.as<int64_t>(), c->nb.as<int32_t>(),
                   c->nb_stride, words, mask, mask + nn * words, reinterpret_cast<unsigned long long*>(cnt),
                   &c->counters.as<DevCounters>()->err};
    const int64_t items = a.nA + c->K[2].cap;
    if (items > 0) {
        k_edge_mark<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(a);
        AC_LAUNCHED();
    }
    int64_t* uoff = L.v0_off.as<int64_t>();
    AC_TRY(scan_exclusive_i64(c, cnt, uoff, n, s));
    AC_TRY(list_rows(c, L, uoff + n, edge_rows_bound(c, c->K[2].cap), s));
    const int64_t count = L.cap;
    const size_t rows = (size_t)(count > 0 ? count : 1);
    AC_TRY(L.tuples.reserve(rows * 2 * sizeof(int32_t), s));
    AC_TRY(L.attached.reserve(rows, s));
    AC_TRY(L.f.reserve(rows * sizeof(double), s));
    AC_TRY(L.orthosize.reserve(rows * sizeof(double), s));
    AC_TRY(L.src_dim.reserve(rows, s));
    AC_TRY(L.src_idx.reserve(rows * sizeof(int64_t), s));
    AC_TRY(c->Gbuf[1].reserve(rows * sizeof(int4), s));
    if (n > 0) {
        k_edge_write<<<(unsigned)((n + EW_WARPS - 1) / EW_WARPS), EW_WARPS * 32, 0, s>>>(a, n, uoff, c->mol_of.as<int32_t>(),
                                                                  c->d_moloff.as<int64_t>(), c->Gbuf[1].as<int4>(),
                                                                  L.tuples.as<int32_t>(), L.attached.as<uint8_t>(),
                                                                  c->endpoint);
        AC_LAUNCHED();
    }
    return AC_OK;
}

// ---------------------------------------------------------------------------
// K^2 by marks (Step 3 for triangles), as for edges one dimension up: a
// triangle of K^2 has pairwise-meeting vertices, so its second and third
// vertices are entries p < q of the neighbour row of its first vertex. Each
// atom has a pair mask over its row (bit q (q - 1) / 2 + p), sized by its own
// row length m (m (m - 1) / 2 bits); the free triangles and the four facets of
// every tetrahedron of K^3 set bits, a second mask keeps the free ones, and
// each atom writes its marked pairs in lexicographic input order.

struct TriMarkArgs {
    const int4* free_t;  // free triangles (sorted positions in x, y, z), nA of them
    int64_t nA;
    const int4* tet;     // tetrahedra of K^3 as emitted (sorted positions), nB of them
    int64_t nB;
    const int32_t* order;
    const int32_t* rank;
    const int64_t* nb_off;
    const int32_t* nb;
    int stride;
    const int64_t* moff;  // first mask word of each sorted position (n + 1)
    unsigned* m_in;
    unsigned* m_free;
    unsigned long long* rows;  // per input index: distinct marked pairs (the atom's row count)
    unsigned* err;
};

__device__ __forceinline__ void nb_row_of(const int64_t* __restrict__ nb_off, int stride, int s, int64_t& off, int& m) {
    if (stride) {
        off = (int64_t)s * stride;
        m = min((int)nb_off[s], stride);
    } else {
        off = nb_off[s];
        m = (int)(nb_off[s + 1] - off);
    }
}


// The pair-mask layout of the K^2 marks (first word of each sorted position,
// n + 1, into c->pair_moff) from the words per atom the neighbour pass wrote;
// the caller reads the total (pair_moff[n]) with its other sizes.
int plan_pair_masks(ac_ctx* c, const int64_t* pw, cudaStream_t s) {
    const int64_t n = c->n;
    const size_t nn = (size_t)(n > 0 ? n : 1);
    AC_TRY(c->pair_moff.reserve((nn + 1) * sizeof(int64_t), s));
    return scan_exclusive_i64(c, pw, c->pair_moff.as<int64_t>(), n, s);
}

__device__ __forceinline__ void mark_pair(const TriMarkArgs& a, int sa, int ga, int e1, int e2, bool fr) {
    if (e1 < 0 || e2 < 0) {
        atomicOr(a.err, DERR_INTERNAL);  // a triangle of K^2 whose vertices' balls do not meet: impossible
        return;
    }
    const int p = min(e1, e2), q = max(e1, e2);
    const int64_t bit = (int64_t)q * (q - 1) / 2 + p;
    const int64_t w = a.moff[sa] + (bit >> 5);
    const unsigned b = 1u << (bit & 31);
    if (!(atomicOr(&a.m_in[w], b) & b)) atomicAdd(&a.rows[ga], 1ull);
    if (fr) atomicOr(&a.m_free[w], b);
}

// threads [0, nA): one free triangle each; then one K^3 tetrahedron (a < b < c < d)
// each: (a,b,c), (a,b,d), (a,c,d) in a's row, (b,c,d) in b's row. Both lists are
// taken as the per-atom pass emitted them, which is nearly grid order: the rows
// and masks that neighbouring threads touch are near one another. (In the order
// of the K^3 rows, which is input order, the 3.0 M atom shell's masks of 750 MB
// were hit at random: 2.56 against 1.48 ms.)
__global__ void k_tri_mark(TriMarkArgs a) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= a.nA + a.nB) return;
    int64_t off;
    int m;
    if (j < a.nA) {
        const int4 t = a.free_t[j];
        int sv[3] = {t.x, t.y, t.z};
        int gv[3] = {a.order[t.x], a.order[t.y], a.order[t.z]};
        int f = 0;  // the vertex with the smallest input index
        if (gv[1] < gv[f]) f = 1;
        if (gv[2] < gv[f]) f = 2;
        const int sa = sv[f], s1 = sv[f == 0 ? 1 : 0], s2 = sv[f == 2 ? 1 : 2];
        nb_row_of(a.nb_off, a.stride, sa, off, m);
        const int64_t offs[2] = {off, off};
        const int ms[2] = {m, m}, xs[2] = {s1, s2};
        int es[2];
        row_find<2>(a.nb, offs, ms, xs, es);
        mark_pair(a, sa, gv[f], es[0], es[1], true);
        return;
    }
    int4 q = a.tet[j - a.nA];  // sorted positions, put in order of input index below
    int4 t = make_int4(a.order[q.x], a.order[q.y], a.order[q.z], a.order[q.w]);
    auto cs = [](int& g0, int& s0, int& g1, int& s1) {
        if (g0 > g1) {
            const int g = g0, s = s0;
            g0 = g1;
            s0 = s1;
            g1 = g;
            s1 = s;
        }
    };
    cs(t.x, q.x, t.y, q.y);
    cs(t.z, q.z, t.w, q.w);
    cs(t.x, q.x, t.z, q.z);
    cs(t.y, q.y, t.w, q.w);
    cs(t.y, q.y, t.z, q.z);
    nb_row_of(a.nb_off, a.stride, q.x, off, m);
    int64_t offb;
    int mb;
    nb_row_of(a.nb_off, a.stride, q.y, offb, mb);
    const int64_t offs[5] = {off, off, off, offb, offb};
    const int ms[5] = {m, m, m, mb, mb}, xs[5] = {q.y, q.z, q.w, q.z, q.w};
    int es[5];
    row_find<5>(a.nb, offs, ms, xs, es);
    mark_pair(a, q.x, t.x, es[0], es[1], false);
    mark_pair(a, q.x, t.x, es[0], es[2], false);
    mark_pair(a, q.x, t.x, es[1], es[2], false);
    mark_pair(a, q.y, t.y, es[3], es[4], false);
}

constexpr int TW_WARPS = 4;
constexpr int TW_CAP = 256;  // marked pairs ranked in shared memory; more take the slow path

// The pair (p, q), p < q, of pair-mask bit q (q - 1) / 2 + p. Rows hold at most
// MAX_DEGREE entries, so bit < 2^19: 32-bit arithmetic throughout (a 64-bit
// integer conversion would run on the narrow FP64 pipe).
static_assert((int64_t)MAX_DEGREE * (MAX_DEGREE - 1) / 2 < (1 << 24), "pair bits exact in FP32");
__device__ __forceinline__ void pair_of(int bit, int& p, int& q) {
    int x = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)bit)) * 0.5f);
    while (x * (x - 1) / 2 > bit) x--;
    while ((x + 1) * x / 2 <= bit) x++;
    q = x;
    p = bit - q * (q - 1) / 2;
}

__global__ void __launch_bounds__(TW_WARPS * 32) k_tri_write(TriMarkArgs a, int64_t n, const int64_t* __restrict__ uoff,
                                                             const int32_t* __restrict__ mol_of,
                                                             const int64_t* __restrict__ mol_off, int4* __restrict__ G,
                                                             int32_t* __restrict__ out, uint8_t* __restrict__ attached) {
    __shared__ unsigned long long key_all[TW_WARPS][TW_CAP];
    __shared__ uint8_t fr_all[TW_WARPS][TW_CAP];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    // (in grid order, as k_edge_write, it is slower: order[s] comes before every other load)
    const int64_t g = (int64_t)blockIdx.x * TW_WARPS + wib;
    if (g >= n) return;
    const int64_t row0 = uoff[g];
    const int64_t total = uoff[g + 1] - row0;
    if (total == 0) return;
    unsigned long long* key = key_all[wib];
    uint8_t* frs = fr_all[wib];
    const int s = a.rank[g];
    int64_t off;
    int m;
    nb_row_of(a.nb_off, a.stride, s, off, m);
    const int64_t w0 = a.moff[s], w1 = a.moff[s + 1];
    const int base = (int)mol_off[mol_of[g]];
    auto key_of = [&](int64_t bit) {
        int p, q;
        pair_of((int)bit, p, q);
        const unsigned hb = (unsigned)a.order[a.nb[off + p]], hc = (unsigned)a.order[a.nb[off + q]];
        return hb < hc ? ((unsigned long long)hb << 32) | hc : ((unsigned long long)hc << 32) | hb;
    };
    auto emit = [&](unsigned long long k, int64_t r, bool fr) {
        const int y = (int)(k >> 32), z = (int)(k & 0xffffffffu);
        const int64_t row = row0 + r;
        G[row] = make_int4((int)g, y, z, -1);
        out[row * 3 + 0] = (int)g - base;
        out[row * 3 + 1] = y - base;
        out[row * 3 + 2] = z - base;
        attached[row] = fr ? 0 : 1;
    };
    if (total <= TW_CAP) {
        // compact the marked pairs in bit order, then rank them
        int c = 0;
        for (int64_t wb = w0; wb < w1; wb += 32) {
            const int64_t w = wb + lane;
            const unsigned bits = w < w1 ? a.m_in[w] : 0u;
            const int k = __popc(bits);
            int incl = k;
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += v;
            }
            int slot = c + incl - k;
            const unsigned frw = bits ? a.m_free[w] : 0u;
            for (unsigned b = bits; b; b &= b - 1) {
                const int t = __ffs(b) - 1;
                key[slot] = key_of((w - w0) * 32 + t);
                frs[slot] = (uint8_t)((frw >> t) & 1u);
                slot++;
            }
            c += __shfl_sync(0xffffffffu, incl, 31);
        }
        __syncwarp();
        for (int k = lane; k < c; k += 32) {
            const unsigned long long kk = key[k];
            int r = 0;
            for (int q = 0; q < c; q++) r += key[q] < kk;
            emit(kk, r, frs[k] != 0);
        }
    } else {
        // many pairs (a very wide row): rank each against all, from the masks
        for (int64_t w = w0; w < w1; w++) {
            const unsigned bits = a.m_in[w];
            const unsigned frw = a.m_free[w];
            for (int t = lane; t < 32; t += 32) {
                if (!((bits >> t) & 1u)) continue;
                const unsigned long long kk = key_of((w - w0) * 32 + t);
                int64_t r = 0;
                for (int64_t w2 = w0; w2 < w1; w2++)
                    for (unsigned b2 = a.m_in[w2]; b2; b2 &= b2 - 1)
                        r += key_of((w2 - w0) * 32 + __ffs(b2) - 1) < kk;
                emit(kk, r, (frw >> t) & 1u);
            }
        }
    }
}

static int canon_tris_by_marks(ac_ctx* c, cudaStream_t s) {
    const DevCounters& h = c->hc;
    const int64_t n = c->n;
    SimplexList& L = c->K[2];
    const size_t nn = (size_t)(n > 0 ? n : 1);
    DevBuf& masks = c->scratch[2];
    AC_TRY(L.v0_off.reserve((nn + 1) * sizeof(int64_t), s));
    // first mask word of each sorted position and their total: from the neighbour pass
    const int64_t* moff = c->pair_moff.as<int64_t>();
    const int64_t words = c->pair_words;
    const size_t mw = (size_t)(words > 0 ? words : 1);
    // one buffer, emptied at once: row counts and the two masks
    const size_t o_mask = nn * sizeof(int64_t), bytes = o_mask + 2 * mw * sizeof(unsigned);
    AC_TRY(masks.reserve(bytes, s));
    AC_CUDA(cudaMemsetAsync(masks.p, 0, bytes, s));
    int64_t* cnt = masks.as<int64_t>();
    unsigned* mask = reinterpret_cast<unsigned*>(masks.as<char>() + o_mask);
    TriMarkArgs a{c->tri_pass.as<int4>(), (int64_t)h.n_tri_pass, c->tet_out.as<int4>(), c->K[3].count,
                  c->order.as<int32_t>(), c->rank.as<int32_t>(), c->nb_cnt.as<int64_t>(), c->nb.as<int32_t>(),
                  c->nb_stride, moff, mask, mask + mw, reinterpret_cast<unsigned long long*>(cnt),
                  &c->counters.as<DevCounters>()->err};
    const int64_t items = a.nA + a.nB;
    if (items > 0) {
        k_tri_mark<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(a);
        AC_LAUNCHED();
    }
    const unsigned wb = (unsigned)((n + TW_WARPS - 1) / TW_WARPS);
    int64_t* uoff = L.v0_off.as<int64_t>();
    AC_TRY(scan_exclusive_i64(c, cnt, uoff, n, s));
    AC_TRY(list_rows(c, L, uoff + n, tri_rows_bound(h), s));
    const int64_t count = L.cap;
    const size_t rows = (size_t)(count > 0 ? count : 1);
    AC_TRY(L.tuples.reserve(rows * 3 * sizeof(int32_t), s));
    AC_TRY(L.attached.reserve(rows, s));
    AC_TRY(L.f.reserve(rows * sizeof(double), s));
    AC_TRY(L.orthosize.reserve(rows * sizeof(double), s));
    AC_TRY(L.src_dim.reserve(rows, s));
    AC_TRY(L.src_idx.reserve(rows * sizeof(int64_t), s));
    AC_TRY(c->Gbuf[2].reserve(rows * sizeof(int4), s));
    if (n > 0) {
        k_tri_write<<<wb, TW_WARPS * 32, 0, s>>>(a, n, uoff, c->mol_of.as<int32_t>(), c->d_moloff.as<int64_t>(),
                                                 c->Gbuf[2].as<int4>(), L.tuples.as<int32_t>(),
                                                 L.attached.as<uint8_t>());
        AC_LAUNCHED();
    }
    return AC_OK;
}

// Vertices (Step 5): K^0 = endpoints of K^1 (flagged by k_edge_write) + atoms
// whose centre passes AC2.
struct VertexFlag {
    const uint8_t* endpoint;
    const uint8_t* vert_pass;
    const int32_t* rank;
    __device__ __forceinline__ long long operator()(int64_t g) const {
        return endpoint[g] || vert_pass[rank[g]] ? 1 : 0;
    }
};

__global__ void k_vertex_flags(VertexFlag f, int64_t n, int64_t* __restrict__ inK) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n) inK[g] = f(g);
}

__global__ void k_vertex_write(const int64_t* __restrict__ voff, const uint8_t* __restrict__ vert_pass,
                               const int32_t* __restrict__ rank, int64_t n, const int32_t* __restrict__ mol_of,
                               const int64_t* __restrict__ mol_off, int4* __restrict__ G, int32_t* __restrict__ out,
                               uint8_t* __restrict__ attached) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    if (voff[g + 1] == voff[g]) return;
    int64_t r = voff[g];
    G[r] = make_int4((int)g, -1, -1, -1);
    out[r] = (int)(g - mol_off[mol_of[g]]);
    attached[r] = vert_pass[rank[g]] ? 0 : 1;
}

// First row of every molecule in each list: rows of molecule m start at
// v0_off[mol_off[m]]. Lists 0..3 are K^0..K^3, lists 4..6 Sigma^1..Sigma^3.
struct MolRowsArgs {
    const int64_t* v0_off[7];
    const int64_t* mol_off;
    int64_t n_mol;
    int64_t* out;  // 7 x (n_mol + 1)
};

__global__ void k_mol_rows(MolRowsArgs a) {
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m > a.n_mol) return;
    const int64_t at = a.mol_off[m];
    for (int l = 0; l < 7; l++) a.out[l * (a.n_mol + 1) + m] = a.v0_off[l] ? a.v0_off[l][at] : 0;
}

static int fork_orthosize(ac_ctx* c, int d, cudaStream_t s, cudaStream_t from);

// the row counts, beside the counters the host reads last
__global__ void k_row_counts(const int64_t* n0, const int64_t* n1, const int64_t* n2, DevCounters* cnt) {
    const int64_t* p[3] = {n0, n1, n2};
    if (threadIdx.x < 3) cnt->n_rows[threadIdx.x] = *p[threadIdx.x];
}

// Up to this many atoms K^3 is canonicalised beside K^2: four launches, each of them
// too short or too unevenly filled to use the whole chip, leave the critical path
// (replay of a 100,000-atom build 1,384 -> 1,352 us, first build 1,470 -> 1,436;
// 250,000 atoms 3,205 -> 3,181; even from 500,000 on). For 3.0 M atoms both are
// bound by the traffic of their scattered rows and masks, and side by side they
// took 0.5 ms longer (37.9 -> 38.4 ms).
constexpr int64_t K3_BESIDE_MAX_ATOMS = 1 << 20;

int canonicalise(ac_ctx* c, cudaStream_t s) {
    const DevCounters& h = c->hc;  // counters read at the end of the per-atom pass
    if (h.err & (DERR_OVF_TET | DERR_OVF_TRI | DERR_OVF_EDGE | DERR_OVF_CAND))
        return fail(AC_ERR_CAPACITY, "per-atom output overflow");
    Work& w = c->cw;
    const int64_t n = c->n;
    c->deferred = may_defer(c);
    // K^3: its facets are marked from the tetrahedra as emitted, so K^2 does not wait for its rows, only the
    // filtration does, which runs on the side stream too
    const bool beside = n <= K3_BESIDE_MAX_ATOMS;
    const cudaStream_t t3 = beside ? c->side : s;
    AC_TRY(canon_dim(c, 3, c->tet_out.as<int4>(), nullptr, (int64_t)h.n_tet_out, c->K[3], c->Gbuf[3], c->cw_k3, s, t3));
    if (beside) {
        c->os_forked = true;
        AC_CUDA(cudaEventRecord(c->ev_k3, t3));
    }
    AC_TRY(fork_orthosize(c, 3, s, t3));
    AC_TRY(stage_mark(c, 4, s));
    // K^2 = unattached triangles + facets of K^3
    AC_TRY(canon_tris_by_marks(c, s));
    AC_TRY(fork_orthosize(c, 2, s, s));
    AC_TRY(stage_mark(c, 5, s));
    // K^1 = unattached edges + edges of K^2, by marks over the neighbour rows
    AC_TRY(canon_edges_by_marks(c, s));
    AC_TRY(fork_orthosize(c, 1, s, s));
    // K^0
    {
        SimplexList& L = c->K[0];
        size_t nn = (size_t)(n > 0 ? n : 1);
        AC_TRY(L.v0_off.reserve((nn + 1) * sizeof(int64_t), s));
        int64_t* voff = L.v0_off.as<int64_t>();
        const VertexFlag flag{c->endpoint, c->vert_pass.as<uint8_t>(), c->rank.as<int32_t>()};  // endpoint: k_edge_write
        if (n > 0 && n <= SC_MAX) {
            launch_small_scan(flag, reinterpret_cast<long long*>(voff), n, s);
            AC_LAUNCHED();
        } else {
            AC_TRY(w.cnt.reserve((nn + 1) * sizeof(int64_t), s));
            int64_t* inK = w.cnt.as<int64_t>();
            if (n > 0) {
                k_vertex_flags<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(flag, n, inK);
                AC_LAUNCHED();
            }
            AC_TRY(scan_exclusive_i64(c, inK, voff, n, s));
        }
        AC_TRY(list_rows(c, L, voff + n, n, s));
        const int64_t count = L.cap;
        size_t rows = (size_t)(count > 0 ? count : 1);
        AC_TRY(L.tuples.reserve(rows * sizeof(int32_t), s));
        AC_TRY(L.attached.reserve(rows, s));
        AC_TRY(L.f.reserve(rows * sizeof(double), s));
        AC_TRY(L.orthosize.reserve(rows * sizeof(double), s));
        AC_TRY(L.src_dim.reserve(rows, s));
        AC_TRY(L.src_idx.reserve(rows * sizeof(int64_t), s));
        AC_TRY(c->Gbuf[0].reserve(rows * sizeof(int4), s));
        if (n > 0) {
            k_vertex_write<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(voff, c->vert_pass.as<uint8_t>(),
                                                                       c->rank.as<int32_t>(), n, c->mol_of.as<int32_t>(),
                                                                       c->d_moloff.as<int64_t>(), c->Gbuf[0].as<int4>(),
                                                                       L.tuples.as<int32_t>(), L.attached.as<uint8_t>());
            AC_LAUNCHED();
        }
    }
    AC_TRY(fork_orthosize(c, 0, s, s));
    // estimation-pass lists, when kept (single molecule)
    if (c->pc.keep_candidates) {
        for (int d = 1; d <= 3; d++) {
            int64_t m = (int64_t)h.n_cand_out[d];
            // each candidate is emitted once, by its owner
            AC_TRY(canon_dim(c, d, d >= 2 ? c->cand[d].as<int4>() : nullptr, d == 1 ? c->cand[1].as<int2>() : nullptr, m,
                             c->C[d], c->CGbuf[d], w, s, s));
        }
    }
    if (c->deferred) {
        k_row_counts<<<1, 32, 0, s>>>(c->K[0].d_count, c->K[1].d_count, c->K[2].d_count, c->counters.as<DevCounters>());
        AC_LAUNCHED();
    }
    if (c->n_mol == 1) return AC_OK;  // its rows are the whole lists (finish_mol_rows)
    if (beside) AC_CUDA(cudaStreamWaitEvent(s, c->ev_k3, 0));  // K^3's offsets
    // per-molecule row ranges, copied to the host with the build's last transfer
    MolRowsArgs ma{};
    for (int d = 0; d < 4; d++) ma.v0_off[d] = c->K[d].v0_off.as<int64_t>();
    for (int d = 1; d <= 3; d++) ma.v0_off[3 + d] = c->pc.keep_candidates ? c->C[d].v0_off.as<int64_t>() : nullptr;
    ma.mol_off = c->d_moloff.as<int64_t>();
    ma.n_mol = c->n_mol;
    AC_TRY(w.cursor.reserve((size_t)7 * (c->n_mol + 1) * sizeof(int64_t), s));
    ma.out = w.cursor.as<int64_t>();
    k_mol_rows<<<(unsigned)((c->n_mol + 1 + 127) / 128), 128, 0, s>>>(ma);
    AC_LAUNCHED();
    AC_CUDA(cudaMemcpyAsync(c->h_molrows, ma.out, (size_t)7 * (c->n_mol + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost,
                            s));
    return AC_OK;
}

// Unpack the per-molecule row ranges once the stream has reached the end of the build.
void finish_mol_rows(ac_ctx* c) {
    const size_t m1 = (size_t)c->n_mol + 1;
    if (c->n_mol == 1) {
        for (int d = 0; d < 4; d++) c->K[d].mol_off = {0, c->K[d].count};
        if (c->pc.keep_candidates)
            for (int d = 1; d <= 3; d++) c->C[d].mol_off = {0, c->C[d].count};
        return;
    }
    for (int d = 0; d < 4; d++) c->K[d].mol_off.assign(c->h_molrows + d * m1, c->h_molrows + (d + 1) * m1);
    if (c->pc.keep_candidates)
        for (int d = 1; d <= 3; d++)
            c->C[d].mol_off.assign(c->h_molrows + (3 + d) * m1, c->h_molrows + (4 + d) * m1);
}

// ---------------------------------------------------------------------------
// OrthoSize (exact) and Size

// OrthoSize of a simplex of global input indices (ascending, K entries) as an
// exact rational num / den in quanta^2 (den > 0).
__device__ void orthosize_rational(const int4* __restrict__ P, const int4& t, int K, i128& num, i128& den);

// OrthoSize in A^2 of a simplex of global input indices (ascending, K entries):
// the numerator (scaled by 2^-20, quanta^2 -> A^2) and the denominator each
// rounded to the nearest double in integer arithmetic, then one FP64 division.
__device__ double orthosize_exact(const int4* __restrict__ P, const int4& t, int K) {
    i128 num, den;
    orthosize_rational(P, t, K, num, den);
    if (K == 1) return i128_to_double_rn(num, -20);  // exact
    return i128_to_double_rn(num, -20) / i128_to_double_rn(den, 0);
}

__device__ void orthosize_rational(const int4* __restrict__ P, const int4& t, int K, i128& num, i128& den) {
    const int4 p0 = P[t.x];
    const long long W0 = p0.w;
    if (K == 1) {
        num = -(i128)W0;
        den = 1;
        return;
    }
    int v[4] = {t.x, t.y, t.z, t.w};
    long long q[3][3], a[3];
    for (int k = 1; k < K; k++) {
        int4 pk = P[v[k]];
        q[k - 1][0] = pk.x - p0.x;
        q[k - 1][1] = pk.y - p0.y;
        q[k - 1][2] = pk.z - p0.z;
        a[k - 1] = q[k - 1][0] * q[k - 1][0] + q[k - 1][1] * q[k - 1][1] + q[k - 1][2] * q[k - 1][2] - pk.w + W0;
    }
    if (K == 2) {
        long long D = q[0][0] * q[0][0] + q[0][1] * q[0][1] + q[0][2] * q[0][2];
        num = (i128)a[0] * a[0] - (i128)4 * D * W0;
        den = (i128)4 * D;
    } else if (K == 3) {
        long long g11 = q[0][0] * q[0][0] + q[0][1] * q[0][1] + q[0][2] * q[0][2];
        long long g22 = q[1][0] * q[1][0] + q[1][1] * q[1][1] + q[1][2] * q[1][2];
        long long g12 = q[0][0] * q[1][0] + q[0][1] * q[1][1] + q[0][2] * q[1][2];
        long long detG = g11 * g22 - g12 * g12;
        long long n1 = g22 * a[0] - g12 * a[1], n2 = g11 * a[1] - g12 * a[0];
        num = (i128)n1 * a[0] + (i128)n2 * a[1] - (i128)4 * detG * W0;
        den = (i128)4 * detG;
    } else {
        long long C[3][3];
        // C_k = q_{k+1} x q_{k+2}
        for (int k = 0; k < 3; k++) {
            const long long* b = q[(k + 1) % 3];
            const long long* d = q[(k + 2) % 3];
            C[k][0] = b[1] * d[2] - b[2] * d[1];
            C[k][1] = b[2] * d[0] - b[0] * d[2];
            C[k][2] = b[0] * d[1] - b[1] * d[0];
        }
        long long D = q[0][0] * C[0][0] + q[0][1] * C[0][1] + q[0][2] * C[0][2];
        long long N[3];
        for (int c = 0; c < 3; c++) N[c] = a[0] * C[0][c] + a[1] * C[1][c] + a[2] * C[2][c];
        i128 nn = (i128)N[0] * N[0] + (i128)N[1] * N[1] + (i128)N[2] * N[2];
        i128 DD = (i128)D * D;
        num = nn - DD * (4 * W0);
        den = DD * 4;
    }
}

__global__ void k_orthosize(const int4* __restrict__ P, const int4* __restrict__ G, RowCount m, int K,
                            const uint8_t* __restrict__ attached, double* __restrict__ os, double* __restrict__ f,
                            int8_t* __restrict__ src_dim, int64_t* __restrict__ src_idx,
                            unsigned long long* __restrict__ fkey, unsigned long long* __restrict__ arg) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m.get()) return;
    double v = orthosize_exact(P, G[j], K);
    os[j] = v;
    src_dim[j] = (int8_t)(K - 1);
    src_idx[j] = j;
    f[j] = v;
    fkey[j] = attached[j] ? ~0ull : 0ull;
    if (arg) arg[j] = ~0ull;
}

__device__ __forceinline__ unsigned long long order_key(double x) {
    unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

__device__ __forceinline__ double key_value(unsigned long long k) {
    unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

// Rows of the K facets of coface t (K entries, facets of K - 1) in the canonical
// list L, or -1: facet `drop` leaves out entry drop. The searches in the facets'
// first-vertex buckets step together, as in row_find; a row's components past its
// K - 1 entries are not looked at.
template <int K>
__device__ __forceinline__ void find_facets(const int4* __restrict__ L, const int64_t* __restrict__ v0_off, const int4& t,
                                            int64_t (&r)[K]) {
    const int64_t a0 = v0_off[t.x], a1 = v0_off[t.x + 1], b0 = v0_off[t.y], b1 = v0_off[t.y + 1];
    if constexpr (K == 2) {  // vertices: one row per atom, if it has one
        r[0] = b0 < b1 ? b0 : -1;
        r[1] = a0 < a1 ? a0 : -1;
    } else {
        int64_t lo[K], hi[K];
        int y[K], z[K];
#pragma unroll
        for (int k = 0; k < K; k++) {
            lo[k] = k == 0 ? b0 : a0;
            hi[k] = k == 0 ? b1 : a1;
            y[k] = k <= 1 ? t.z : t.y;
            z[k] = K == 4 ? (k <= 2 ? t.w : t.z) : 0;
            r[k] = -1;
        }
        for (bool more = true; more;) {
            int4 v[K];
#pragma unroll
            for (int k = 0; k < K; k++) v[k] = L[lo[k] < hi[k] ? (lo[k] + hi[k]) >> 1 : a0];
            more = false;
#pragma unroll
            for (int k = 0; k < K; k++) {
                if (lo[k] >= hi[k]) continue;
                const int64_t mid = (lo[k] + hi[k]) >> 1;
                const int dy = v[k].y - y[k], d = dy != 0 || K == 3 ? dy : v[k].z - z[k];  // indices: no overflow
                if (d == 0) {
                    r[k] = mid;
                    lo[k] = hi[k];
                } else if (d < 0) {
                    lo[k] = mid + 1;
                } else {
                    hi[k] = mid;
                }
                more = more || lo[k] < hi[k];
            }
        }
    }
}

// pass 1: smallest coface value of every attached face; the row of each
// (coface, facet) that is an attached face is kept for pass 2 (-1 otherwise)
template <int K>
__global__ void k_coface_min(const int4* __restrict__ Cof, const double* __restrict__ fc, RowCount mc,
                             const int4* __restrict__ L, const int64_t* __restrict__ v0_off,
                             const uint8_t* __restrict__ attached, unsigned long long* __restrict__ fkey,
                             int64_t* __restrict__ rows) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= mc.get()) return;
    const int4 t = Cof[j];
    const unsigned long long key = order_key(fc[j]);
    int64_t r[K];
    find_facets<K>(L, v0_off, t, r);
    bool hit[K];
#pragma unroll
    for (int k = 0; k < K; k++) hit[k] = r[k] >= 0 && attached[r[k]];
#pragma unroll
    for (int k = 0; k < K; k++) {
        rows[j * K + k] = hit[k] ? r[k] : -1;
        if (hit[k]) atomicMin(&fkey[r[k]], key);
    }
}

// pass 2: among cofaces attaining the minimum, the first in lexicographic order
__global__ void k_coface_arg(const double* __restrict__ fc, RowCount mc, int Kc, const int64_t* __restrict__ rows,
                             const unsigned long long* __restrict__ fkey, unsigned long long* __restrict__ arg) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= mc.get()) return;
    unsigned long long key = order_key(fc[j]);
    for (int drop = 0; drop < Kc; drop++) {
        const int64_t r = rows[j * Kc + drop];
        if (r >= 0 && fkey[r] == key) atomicMin(&arg[r], (unsigned long long)j);
    }
}

__global__ void k_coface_apply(RowCount m, const uint8_t* __restrict__ attached, const unsigned long long* __restrict__ fkey,
                               const unsigned long long* __restrict__ arg, const int8_t* __restrict__ csrc_dim,
                               const int64_t* __restrict__ csrc_idx, double* __restrict__ f, int8_t* __restrict__ src_dim,
                               int64_t* __restrict__ src_idx, unsigned* __restrict__ err) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m.get() || !attached[j]) return;
    unsigned long long a = arg[j];
    if (a == ~0ull) {
        // an attached simplex with no coface in the complex cannot occur
        atomicOr(err, DERR_INTERNAL);
        f[j] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    f[j] = key_value(fkey[j]);
    src_dim[j] = csrc_dim[a];
    src_idx[j] = csrc_idx[a];
}

// Sub-complex at alpha2 <= alpha (the filtration restricted): a simplex is in
// K_alpha2 iff Size <= alpha2 (Section 2.4). Size is the OrthoSize of the
// simplex's source (itself when unattached, else the coface its value came
// from), compared exactly: num <= A2 den.
struct RowLists {
    const int4* G[4];
};

__global__ void k_subcomplex(const int4* __restrict__ P, RowLists rows, const int8_t* __restrict__ src_dim,
                             const int64_t* __restrict__ src_idx, int64_t first, int64_t m, long long A2,
                             uint8_t* __restrict__ flags, unsigned long long* __restrict__ n_in) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool in = false;
    if (j < m) {
        const int sd = src_dim[first + j];
        const int4 t = rows.G[sd][src_idx[first + j]];
        i128 num, den;
        orthosize_rational(P, t, sd + 1, num, den);
        in = num <= (i128)A2 * den;
        flags[j] = in ? 1 : 0;
    }
    const unsigned b = __ballot_sync(0xffffffffu, in);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(n_in, (unsigned long long)__popc(b));
}

int subcomplex_flags(ac_ctx* c, int dim, int64_t first, int64_t m, double alpha2, uint8_t* flags, int64_t* count,
                     cudaStream_t s) {
    const long long A2 = (long long)nearbyint(alpha2 * 1048576.0);
    AC_TRY(c->scratch[6].reserve(sizeof(unsigned long long), s));
    unsigned long long* n_in = c->scratch[6].as<unsigned long long>();
    AC_CUDA(cudaMemsetAsync(n_in, 0, sizeof(unsigned long long), s));
    if (m > 0) {
        SimplexList& L = c->K[dim];
        RowLists rows;
        for (int d = 0; d < 4; d++) rows.G[d] = c->Gbuf[d].as<int4>();
        k_subcomplex<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(c->P.as<int4>(), rows, L.src_dim.as<int8_t>(),
                                                                  L.src_idx.as<int64_t>(), first, m, A2, flags, n_in);
        AC_LAUNCHED();
    }
    AC_CUDA(cudaMemcpyAsync(c->h_stage, n_in, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    AC_CUDA(cudaStreamSynchronize(s));
    *count = c->h_stage[0];
    return AC_OK;
}

// The flagged rows of a list and their values, in list order: counts per tile
// of SUB_TILE flags, their prefix by one block, then each tile writes its rows.
// (Boolean indexing by the caller took two passes with a host wait each.)
constexpr int SUB_THREADS = 256;
constexpr int SUB_TILE = 4096;

__global__ void __launch_bounds__(SUB_THREADS) k_sub_count(const uint8_t* __restrict__ flags, int64_t m,
                                                           unsigned* __restrict__ tile) {
    const int64_t j0 = (int64_t)blockIdx.x * SUB_TILE;
    int c = 0;
    for (int u = threadIdx.x; u < SUB_TILE; u += SUB_THREADS) c += __syncthreads_count(j0 + u < m && flags[j0 + u]);
    if (threadIdx.x == 0) tile[blockIdx.x] = (unsigned)c;
}

__global__ void __launch_bounds__(1024) k_sub_prefix(unsigned* __restrict__ tile, int n) {
    __shared__ unsigned sums[32];
    __shared__ unsigned carry;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    for (int t0 = 0; t0 < n; t0 += 1024) {
        const int t = t0 + threadIdx.x;
        const unsigned v = t < n ? tile[t] : 0u;
        unsigned inc = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += x;
        }
        if (lane == 31) sums[w] = inc;
        __syncthreads();
        unsigned before = carry;
        for (int q = 0; q < w; q++) before += sums[q];
        if (t < n) tile[t] = before + inc - v;
        __syncthreads();
        if (threadIdx.x == 1023) carry = before + inc;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(SUB_THREADS) k_sub_write(const uint8_t* __restrict__ flags, int64_t m, int k,
                                                           const unsigned* __restrict__ tile,
                                                           const int32_t* __restrict__ rows,
                                                           const double* __restrict__ f, int64_t count,
                                                           int32_t* __restrict__ rows_out, double* __restrict__ f_out) {
    __shared__ int sums[SUB_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * SUB_TILE;
    int64_t at = tile[blockIdx.x];
    for (int u = threadIdx.x; u < SUB_TILE; u += SUB_THREADS) {
        const int64_t j = j0 + u;
        const bool in = j < m && flags[j];
        const unsigned b = __ballot_sync(0xffffffffu, in);
        if (lane == 0) sums[w] = __popc(b);
        __syncthreads();
        int before = 0, all = 0;
        for (int q = 0; q < SUB_THREADS / 32; q++) {
            before += q < w ? sums[q] : 0;
            all += sums[q];
        }
        const int64_t r = at + before + __popc(b & ((1u << lane) - 1u));
        if (in && r < count) {
            if (rows_out)
                for (int q = 0; q < k; q++) rows_out[r * k + q] = rows[j * k + q];
            if (f_out) f_out[r] = f[j];
        }
        at += all;
        __syncthreads();
    }
}

int subcomplex_lists(ac_ctx* c, int dim, int64_t first, int64_t m, const uint8_t* flags, int64_t count, int32_t* rows,
                     double* f, cudaStream_t s) {
    if (m == 0 || count == 0 || (!rows && !f)) return AC_OK;
    const SimplexList& L = c->K[dim];
    const int k = dim + 1;
    const DevBuf& v = c->opt.filtration == AC_FILTRATION_ORTHOSIZE ? L.orthosize : L.f;
    const int64_t tiles = (m + SUB_TILE - 1) / SUB_TILE;
    // this call's own, released in stream order: calls on other streams may overlap it
    DevBuf tile;
    AC_TRY(tile.reserve((size_t)tiles * sizeof(unsigned), s));
    k_sub_count<<<(unsigned)tiles, SUB_THREADS, 0, s>>>(flags, m, tile.as<unsigned>());
    AC_LAUNCHED();
    k_sub_prefix<<<1, 1024, 0, s>>>(tile.as<unsigned>(), (int)tiles);
    AC_LAUNCHED();
    k_sub_write<<<(unsigned)tiles, SUB_THREADS, 0, s>>>(flags, m, k, tile.as<unsigned>(), L.tuples.as<int32_t>() + first * k,
                                                        v.as<double>() + first, count, rows, f);
    AC_LAUNCHED();
    return AC_OK;
}

// opt.host_results: list d (rows, the selected filtration values, attached
// flags) to its page-locked host block, on the context's copy stream (the
// device-to-host link, about 190 GB/s here, is the limit, so the copies start
// as early as they can and never hold up the filtration): the rows and flags
// once the list's rows are written (after stream `from`), the values once
// they are final (after stream `from`); compute_filtration joins the copies.
static int copy_after(ac_ctx* c, cudaStream_t from) {
    AC_CUDA(cudaEventRecord(c->ev_copy, from));
    AC_CUDA(cudaStreamWaitEvent(c->copy, c->ev_copy, 0));
    c->copy_forked = true;
    return AC_OK;
}

static int copy_rows_to_host(ac_ctx* c, int d, cudaStream_t from) {
    if (!c->opt.host_results) return AC_OK;
    const SimplexList& L = c->K[d];
    const int64_t m = L.count;
    const int k = d + 1;
    AC_TRY(host_block_for(c, d, hres_bytes_for(m, k)));
    char* b = static_cast<char*>(c->hres[d]);
    AC_TRY(copy_after(c, from));
    AC_CUDA(cudaMemcpyAsync(b, L.tuples.p, (size_t)m * k * sizeof(int32_t), cudaMemcpyDeviceToHost, c->copy));
    AC_CUDA(cudaMemcpyAsync(b + hres_a_off(m, k), L.attached.p, (size_t)m, cudaMemcpyDeviceToHost, c->copy));
    return AC_OK;
}

static int copy_values_to_host(ac_ctx* c, int d, cudaStream_t from) {
    if (!c->opt.host_results) return AC_OK;
    const SimplexList& L = c->K[d];
    const int64_t m = L.count;
    const int k = d + 1;
    char* b = static_cast<char*>(c->hres[d]);
    const DevBuf& f = c->opt.filtration == AC_FILTRATION_ORTHOSIZE ? L.orthosize : L.f;
    AC_TRY(copy_after(c, from));
    AC_CUDA(cudaMemcpyAsync(b + hres_f_off(m, k), f.p, (size_t)m * sizeof(double), cudaMemcpyDeviceToHost, c->copy));
    return AC_OK;
}

// The filtration of list d on the side stream, as soon as the list's rows are
// final (written on stream `from`: s or the side stream), overlapping the canonicalisation of the lower dimensions: OrthoSize
// (with the initial Size, source and coface key), then for d < 3 the two
// coface passes over K^(d+1), whose values are final by then (the side stream
// ran its passes first). compute_filtration joins the side stream. Each pass
// has its own buffers, reserved here on the build's stream before the fork.
static int fork_orthosize(ac_ctx* c, int d, cudaStream_t s, cudaStream_t from) {
    SimplexList& L = c->K[d];
    const int64_t m = L.cap;
    if (m == 0) return AC_OK;
    SimplexList* U = d < 3 ? &c->K[d + 1] : nullptr;
    const int64_t mu = U ? U->cap : 0;
    const RowCount rm{m, L.d_count}, ru{mu, U ? U->d_count : nullptr};
    AC_TRY(c->fkey[d].reserve((size_t)m * sizeof(unsigned long long), s));
    if (U) {
        AC_TRY(c->fargs[d].reserve((size_t)m * sizeof(unsigned long long), s));
        if (mu > 0) AC_TRY(c->frows[d].reserve((size_t)mu * (d + 2) * sizeof(int64_t), s));
    }
    AC_TRY(copy_rows_to_host(c, d, from));
    AC_CUDA(cudaEventRecord(c->ev_fork, s));
    cudaStream_t t = c->side;
    AC_CUDA(cudaStreamWaitEvent(t, c->ev_fork, 0));
    unsigned long long* keyb = c->fkey[d].as<unsigned long long>();
    unsigned long long* argb = U ? c->fargs[d].as<unsigned long long>() : nullptr;
    k_orthosize<<<(unsigned)((m + 127) / 128), 128, 0, t>>>(c->P.as<int4>(), c->Gbuf[d].as<int4>(), rm, d + 1,
                                                            L.attached.as<uint8_t>(), L.orthosize.as<double>(),
                                                            L.f.as<double>(), L.src_dim.as<int8_t>(),
                                                            L.src_idx.as<int64_t>(), keyb, argb);
    AC_LAUNCHED();
    c->os_forked = true;
    if (!U) return copy_values_to_host(c, d, t);
    if (mu > 0) {
        const unsigned nbk = (unsigned)((mu + 127) / 128);
        int64_t* rows = c->frows[d].as<int64_t>();
        auto kmin = d == 2 ? k_coface_min<4> : d == 1 ? k_coface_min<3> : k_coface_min<2>;
        kmin<<<nbk, 128, 0, t>>>(c->Gbuf[d + 1].as<int4>(), U->f.as<double>(), ru, c->Gbuf[d].as<int4>(),
                                 L.v0_off.as<int64_t>(), L.attached.as<uint8_t>(), keyb, rows);
        AC_LAUNCHED();
        k_coface_arg<<<nbk, 128, 0, t>>>(U->f.as<double>(), ru, d + 2, rows, keyb, argb);
        AC_LAUNCHED();
    }
    k_coface_apply<<<(unsigned)((m + 127) / 128), 128, 0, t>>>(
        rm, L.attached.as<uint8_t>(), keyb, argb, U->src_dim.as<int8_t>(), U->src_idx.as<int64_t>(), L.f.as<double>(),
        L.src_dim.as<int8_t>(), L.src_idx.as<int64_t>(), &c->counters.as<DevCounters>()->err);
    AC_LAUNCHED();
    return copy_values_to_host(c, d, t);
}

// Size of every list (Section 2.3): computed on the side stream as the lists
// were finished (fork_orthosize); the build's stream waits for it here.
int compute_filtration(ac_ctx* c, cudaStream_t s) {
    if (c->os_forked) {
        AC_CUDA(cudaEventRecord(c->ev_join, c->side));
        AC_CUDA(cudaStreamWaitEvent(s, c->ev_join, 0));
        c->os_forked = false;
    }
    if (c->copy_forked) {
        AC_CUDA(cudaEventRecord(c->ev_cjoin, c->copy));
        AC_CUDA(cudaStreamWaitEvent(s, c->ev_cjoin, 0));
        c->copy_forked = false;
    }
    return AC_OK;
}

}  // namespace ac
