// Differentiation of the filtration values with the combinatorics held fixed.
//
// Every simplex sigma of the complex takes its value from a source simplex s:
// itself when its orthocentre is its closest witness, else the coface whose
// orthocentre is (Section 2.3; the attached case of the proofs of Lemmas 1-2).
// f(sigma) = OrthoSize(s) = min pi(x, b_v0) over the affine set where all
// vertices of s have equal power. With multipliers mu on the equal-power
// constraints the stationarity condition puts the minimiser at
// c = sum_k lambda_k p_k (lambda_0 = 1 - sum mu, lambda_k = mu_k: barycentric
// coordinates of c in aff(s)), and the Lagrangian is sum_k lambda_k pi(c, b_k).
// The envelope theorem then gives
//   dOrthoSize/dp_k = 2 lambda_k (p_k - c),  dOrthoSize/dr_k = -2 r_k lambda_k.
// The gradient is FP64 on the caller's continuous inputs; re-evaluated values
// (for finite-difference checks) use double-double arithmetic.
#include <string.h>

#include <mutex>

#include "ac_internal.cuh"

namespace ac {

struct Ortho {
    double lam[4];
    double c[3];
};

// Orthocentre and barycentric coordinates of K vertices (global input indices,
// ascending) from FP64 centres (n x 3) and radii. A tetrahedron's come from the
// cross products of its edge vectors (y = N / 2D, lambda_k = C_k . y / D): about
// 80 FP64 operations, and a condition number the Gram matrix would square.
template <int K>
__device__ __forceinline__ Ortho ortho_fp64(const double* __restrict__ X, const double* __restrict__ R, const int4& t) {
    Ortho o;
    const int v[4] = {t.x, t.y, t.z, t.w};
    const double p0[3] = {X[3 * v[0]], X[3 * v[0] + 1], X[3 * v[0] + 2]};
    const double w0 = R[v[0]] * R[v[0]];
    double q[3][3], a[3], mu[3] = {0.0, 0.0, 0.0}, y[3] = {0.0, 0.0, 0.0}, g[3];
#pragma unroll
    for (int k = 1; k < K; k++) {
        const double rk = R[v[k]];
        for (int c = 0; c < 3; c++) q[k - 1][c] = X[3 * v[k] + c] - p0[c];
        g[k - 1] = q[k - 1][0] * q[k - 1][0] + q[k - 1][1] * q[k - 1][1] + q[k - 1][2] * q[k - 1][2];
        a[k - 1] = g[k - 1] - rk * rk + w0;
    }
    if constexpr (K == 2) {
        mu[0] = a[0] / (2.0 * g[0]);
        for (int c = 0; c < 3; c++) y[c] = mu[0] * q[0][c];
    } else if constexpr (K == 3) {
        const double g12 = q[0][0] * q[1][0] + q[0][1] * q[1][1] + q[0][2] * q[1][2];
        const double r = 0.5 / (g[0] * g[1] - g12 * g12);
        mu[0] = (g[1] * a[0] - g12 * a[1]) * r;
        mu[1] = (g[0] * a[1] - g12 * a[0]) * r;
        for (int c = 0; c < 3; c++) y[c] = mu[0] * q[0][c] + mu[1] * q[1][c];
    } else if constexpr (K == 4) {
        double C[3][3], N[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const double* b = q[(k + 1) % 3];
            const double* e = q[(k + 2) % 3];
            C[k][0] = b[1] * e[2] - b[2] * e[1];
            C[k][1] = b[2] * e[0] - b[0] * e[2];
            C[k][2] = b[0] * e[1] - b[1] * e[0];
        }
        const double r = 1.0 / (q[0][0] * C[0][0] + q[0][1] * C[0][1] + q[0][2] * C[0][2]);
        for (int c = 0; c < 3; c++) N[c] = a[0] * C[0][c] + a[1] * C[1][c] + a[2] * C[2][c];
        for (int c = 0; c < 3; c++) y[c] = 0.5 * r * N[c];
        for (int k = 0; k < 3; k++) mu[k] = (C[k][0] * y[0] + C[k][1] * y[1] + C[k][2] * y[2]) * r;
    }
    double s = 1.0;
    for (int k = 0; k < K - 1; k++) {
        o.lam[k + 1] = mu[k];
        s -= mu[k];
    }
    o.lam[0] = s;
    for (int c = 0; c < 3; c++) o.c[c] = p0[c] + y[c];
    return o;
}

// Double-double arithmetic (an unevaluated sum hi + lo of two doubles) from the
// error-free transformations TwoSum (Knuth) and TwoProduct via FMA: about 106
// bits, so re-evaluated values of ill-conditioned (flat) simplices stay accurate
// to a few FP64 ulps and central differences with a 1e-6 A step are meaningful.
struct dd {
    double hi, lo;
};

__device__ __forceinline__ dd dd_from(double a) { return {a, 0.0}; }

__device__ __forceinline__ dd two_sum(double a, double b) {
    double s = a + b;
    double bb = s - a;
    double e = (a - (s - bb)) + (b - bb);
    return {s, e};
}

// the same for |a| >= |b| (Dekker's FastTwoSum)
__device__ __forceinline__ dd fast_two_sum(double a, double b) {
    double s = a + b;
    return {s, b - (s - a)};
}

__device__ __forceinline__ dd dd_add(dd a, dd b) {
    dd s = two_sum(a.hi, b.hi);
    dd t = two_sum(a.lo, b.lo);
    s = fast_two_sum(s.hi, s.lo + t.hi);
    return fast_two_sum(s.hi, s.lo + t.lo);
}

__device__ __forceinline__ dd dd_neg(dd a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ dd dd_sub(dd a, dd b) { return dd_add(a, dd_neg(b)); }

__device__ __forceinline__ dd dd_mul(dd a, dd b) {
    const double p = a.hi * b.hi;
    return fast_two_sum(p, fma(a.lo, b.hi, fma(a.hi, b.lo, fma(a.hi, b.hi, -p))));
}

__device__ __forceinline__ dd dd_sqr(dd a) {
    const double p = a.hi * a.hi;
    return fast_two_sum(p, fma(2.0 * a.hi, a.lo, fma(a.hi, a.hi, -p)));
}

// a (a double) times b
__device__ __forceinline__ dd dd_scale(double a, dd b) {
    const double p = a * b.hi;
    return fast_two_sum(p, fma(a, b.lo, fma(a, b.hi, -p)));
}

// three quotient digits, each from the remainder of the ones before (one reciprocal)
__device__ __forceinline__ dd dd_div(dd a, dd b) {
    const double r = 1.0 / b.hi;
    const double q1 = a.hi * r;
    dd e = dd_sub(a, dd_scale(q1, b));
    const double q2 = e.hi * r;
    e = dd_sub(e, dd_scale(q2, b));
    return dd_add(fast_two_sum(q1, q2), dd_from(e.hi * r));
}

// OrthoSize of K vertices from FP64 centres/radii, evaluated in double-double:
// about 1,100 FP64 operations for a tetrahedron, 530 for a triangle, 210 for an edge.
template <int K>
__device__ __forceinline__ double orthosize_dd(const double* __restrict__ X, const double* __restrict__ R, const int4& t) {
    const int v[4] = {t.x, t.y, t.z, t.w};
    const dd w0 = dd_sqr(dd_from(R[v[0]]));
    if constexpr (K == 1) return -w0.hi;
    dd q[3][3], g[3], a[3];
    const double p0[3] = {X[3 * v[0]], X[3 * v[0] + 1], X[3 * v[0] + 2]};
    auto dot = [](const dd* x, const dd* y) {
        return dd_add(dd_add(dd_mul(x[0], y[0]), dd_mul(x[1], y[1])), dd_mul(x[2], y[2]));
    };
#pragma unroll
    for (int k = 1; k < K; k++) {
        for (int c = 0; c < 3; c++) q[k - 1][c] = two_sum(X[3 * v[k] + c], -p0[c]);
        g[k - 1] = dd_add(dd_add(dd_sqr(q[k - 1][0]), dd_sqr(q[k - 1][1])), dd_sqr(q[k - 1][2]));
        a[k - 1] = dd_add(dd_sub(g[k - 1], dd_sqr(dd_from(R[v[k]]))), w0);
    }
    dd num = dd_from(0.0), den = dd_from(1.0);
    if constexpr (K == 2) {
        num = dd_sqr(a[0]);
        den = g[0];
    } else if constexpr (K == 3) {
        const dd g12 = dot(q[0], q[1]);
        const dd n1 = dd_sub(dd_mul(g[1], a[0]), dd_mul(g12, a[1]));
        const dd n2 = dd_sub(dd_mul(g[0], a[1]), dd_mul(g12, a[0]));
        num = dd_add(dd_mul(n1, a[0]), dd_mul(n2, a[1]));
        den = dd_sub(dd_mul(g[0], g[1]), dd_sqr(g12));
    } else if constexpr (K == 4) {
        dd C[3][3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const dd* b = q[(k + 1) % 3];
            const dd* e = q[(k + 2) % 3];
            C[k][0] = dd_sub(dd_mul(b[1], e[2]), dd_mul(b[2], e[1]));
            C[k][1] = dd_sub(dd_mul(b[2], e[0]), dd_mul(b[0], e[2]));
            C[k][2] = dd_sub(dd_mul(b[0], e[1]), dd_mul(b[1], e[0]));
        }
        den = dd_sqr(dot(q[0], C[0]));
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const dd N = dd_add(dd_add(dd_mul(a[0], C[0][c]), dd_mul(a[1], C[1][c])), dd_mul(a[2], C[2][c]));
            num = c == 0 ? dd_sqr(N) : dd_add(num, dd_sqr(N));
        }
    }
    const dd y2 = dd_div(num, den);  // 4 |y|^2: scaling by 1/4 is exact
    const dd f = dd_sub(dd{0.25 * y2.hi, 0.25 * y2.lo}, w0);
    return f.hi + f.lo;
}

// OrthoSize of K vertices in single precision throughout: offsets q_k =
// p_k - p_0 and squared radii from the quantised atoms (exact in FP32), then
// a_k, the Gram matrix, its solve and |y|^2 - w_0 rounded to FP32 at every
// operation. Not used by the build: it measures what FP32 arithmetic would
// do to the filtration values.
__device__ float orthosize_f32(const int4* __restrict__ P, const int4& t, int K) {
    const int v[4] = {t.x, t.y, t.z, t.w};
    const int4 p0 = P[v[0]];
    const float s = 1.0f / 1024.0f, s2 = 1.0f / 1048576.0f;
    const float w0 = (float)p0.w * s2;
    if (K == 1) return -w0;
    float q[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}}, a[3] = {0.f, 0.f, 0.f};
    for (int k = 1; k < K; k++) {
        const int4 pk = P[v[k]];
        q[k - 1][0] = (float)(pk.x - p0.x) * s;
        q[k - 1][1] = (float)(pk.y - p0.y) * s;
        q[k - 1][2] = (float)(pk.z - p0.z) * s;
        a[k - 1] = q[k - 1][0] * q[k - 1][0] + q[k - 1][1] * q[k - 1][1] + q[k - 1][2] * q[k - 1][2] -
                   (float)pk.w * s2 + w0;
    }
    const int d = K - 1;
    float G[3][3];
    for (int i = 0; i < d; i++)
        for (int j = 0; j < d; j++) G[i][j] = q[i][0] * q[j][0] + q[i][1] * q[j][1] + q[i][2] * q[j][2];
    float mu[3] = {0.f, 0.f, 0.f};
    if (d == 1) {
        mu[0] = a[0] / (2.0f * G[0][0]);
    } else if (d == 2) {
        const float det = G[0][0] * G[1][1] - G[0][1] * G[1][0];
        mu[0] = (G[1][1] * a[0] - G[0][1] * a[1]) / (2.0f * det);
        mu[1] = (G[0][0] * a[1] - G[1][0] * a[0]) / (2.0f * det);
    } else {
        float adj[3][3];
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) {
                const int r0 = (i + 1) % 3, r1 = (i + 2) % 3, c0 = (j + 1) % 3, c1 = (j + 2) % 3;
                adj[j][i] = G[r0][c0] * G[r1][c1] - G[r0][c1] * G[r1][c0];
            }
        const float det = G[0][0] * adj[0][0] + G[0][1] * adj[1][0] + G[0][2] * adj[2][0];
        for (int i = 0; i < 3; i++) mu[i] = (adj[i][0] * a[0] + adj[i][1] * a[1] + adj[i][2] * a[2]) / (2.0f * det);
    }
    float y[3] = {0.f, 0.f, 0.f};
    for (int k = 0; k < d; k++)
        for (int c = 0; c < 3; c++) y[c] += mu[k] * q[k][c];
    return y[0] * y[0] + y[1] * y[1] + y[2] * y[2] - w0;
}

struct Rows4 {
    const int4* G[4];
};

__global__ void k_eval_f32(const int4* __restrict__ P, const int8_t* __restrict__ sdim, const int64_t* __restrict__ sidx,
                           int64_t m, Rows4 rows, float* __restrict__ out) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    const int d = sdim[j];
    out[j] = orthosize_f32(P, rows.G[d][sidx[j]], d + 1);
}

int eval_filtration_f32(ac_ctx* c, float* const f_out[4], cudaStream_t s) {
    Rows4 rows;
    for (int d = 0; d < 4; d++) rows.G[d] = c->Gbuf[d].as<int4>();
    for (int d = 0; d < 4; d++) {
        const int64_t m = c->K[d].count;
        if (!f_out[d] || m == 0) continue;
        k_eval_f32<<<(unsigned)((m + 127) / 128), 128, 0, s>>>(c->P.as<int4>(), c->K[d].src_dim.as<int8_t>(),
                                                               c->K[d].src_idx.as<int64_t>(), m, rows, f_out[d]);
        AC_LAUNCHED();
    }
    AC_CUDA(cudaStreamSynchronize(s));
    return AC_OK;
}

// The values at moved atoms, each source evaluated once: a row that is its own
// source (unattached) by its double-double OrthoSize, then every attached row a
// copy of its source's value (100,000-atom probe globule: 2.4 ms; 9.9 ms when
// every row evaluated its source, the four sizes mixed in a warp). The FP64 pipe (2 lanes per clock and SM) bounds
// it, and takes as long for a warp with one active lane as for a full one:
// a block gathers the unattached rows of a tile and evaluates those. A tile of 512
// rows fills its last warp best; short lists take tiles of 128, one evaluation per
// thread, or their few blocks run four long FP64 chains one after another (values
// at moved atoms of a 2,000-atom globule: 330 us, now 157).
constexpr int EVAL_THREADS = 128;
constexpr int EVAL_TILE = 512, EVAL_TILE_SHORT = 128;
constexpr int64_t EVAL_SHORT_ROWS = 2 * 152 * EVAL_TILE;  // two blocks of EVAL_TILE rows for each of 152 SMs

// indices (from first) of the rows of a tile with !skip(row), in no particular order
template <int TILE, class F>
__device__ __forceinline__ int gather_rows(int64_t first, int64_t m, int* list, int* n_list, F&& skip) {
    if (threadIdx.x == 0) *n_list = 0;
    __syncthreads();
    for (int u = threadIdx.x; u < TILE; u += EVAL_THREADS) {
        const bool take = first + u < m && !skip(first + u);
        const unsigned b = __ballot_sync(0xffffffffu, take);
        int base = 0;
        if ((threadIdx.x & 31) == 0 && b) base = atomicAdd(n_list, __popc(b));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (take) list[base + __popc(b & ((1u << (threadIdx.x & 31)) - 1u))] = u;
    }
    __syncthreads();
    return *n_list;
}

template <int K, int TILE>
__global__ void __launch_bounds__(EVAL_THREADS) k_eval_own(const double* __restrict__ X, const double* __restrict__ R,
                                                           const int4* __restrict__ G,
                                                           const uint8_t* __restrict__ attached, int64_t m,
                                                           double* __restrict__ out) {
    __shared__ int list[TILE];
    __shared__ int n_list;
    const int64_t first = (int64_t)blockIdx.x * TILE;
    const int n = gather_rows<TILE>(first, m, list, &n_list, [&](int64_t j) { return attached[j] != 0; });
    for (int u = threadIdx.x; u < n; u += EVAL_THREADS) {
        const int64_t j = first + list[u];
        out[j] = orthosize_dd<K>(X, R, G[j]);
    }
}

struct Vals4 {
    const double* v[4];  // null: a list the caller did not ask for
};

__global__ void k_eval_attached(const uint8_t* __restrict__ attached, const int8_t* __restrict__ sdim,
                                const int64_t* __restrict__ sidx, int64_t m, Vals4 vals, double* __restrict__ out) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m || !attached[j]) return;
    const double* v = vals.v[sdim[j]];
    if (v) out[j] = v[sidx[j]];
}

// The attached rows whose source is in a list the caller did not ask for (K
// vertices, rows Gs): each evaluates its source itself. To evaluate that whole
// list into scratch instead costs its length, however few rows take values from
// it, and memory that calls on several streams would share. 100,000-atom probe
// globule: K^1 alone 898 us against 2,433, K^1 and K^2 2,717 against 2,445.
template <int K, int TILE>
__global__ void __launch_bounds__(EVAL_THREADS) k_eval_source(const double* __restrict__ X, const double* __restrict__ R,
                                                              const int4* __restrict__ Gs,
                                                              const uint8_t* __restrict__ attached,
                                                              const int8_t* __restrict__ sdim,
                                                              const int64_t* __restrict__ sidx, int64_t m,
                                                              double* __restrict__ out) {
    __shared__ int list[TILE];
    __shared__ int n_list;
    const int64_t first = (int64_t)blockIdx.x * TILE;
    const int n = gather_rows<TILE>(first, m, list, &n_list, [&](int64_t j) { return !attached[j] || sdim[j] != K - 1; });
    for (int u = threadIdx.x; u < n; u += EVAL_THREADS) {
        const int64_t j = first + list[u];
        out[j] = orthosize_dd<K>(X, R, Gs[sidx[j]]);
    }
}

template <int K>
__device__ __forceinline__ void add_gradient(const double* __restrict__ X, const double* __restrict__ R, const int4& t,
                                             double w, double* __restrict__ dX, double* __restrict__ dR) {
    const Ortho o = ortho_fp64<K>(X, R, t);
    const int v[4] = {t.x, t.y, t.z, t.w};
    for (int k = 0; k < K; k++) {
        const int a = v[k];
        const double l2 = 2.0 * w * o.lam[k];
        for (int c = 0; c < 3; c++) atomicAdd(&dX[3 * a + c], l2 * (X[3 * a + c] - o.c[c]));
        atomicAdd(&dR[a], -l2 * R[a]);
    }
}

__global__ void k_backward(const double* __restrict__ X, const double* __restrict__ R, const int8_t* __restrict__ sdim,
                           const int64_t* __restrict__ sidx, int64_t m, const int4* const* __restrict__ G,
                           const double* __restrict__ w, double* __restrict__ dX, double* __restrict__ dR) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    const double wj = w[j];
    if (wj == 0.0) return;
    const int d = sdim[j];
    const int4 t = G[d][sidx[j]];
    if (d == 0) add_gradient<1>(X, R, t, wj, dX, dR);
    else if (d == 1) add_gradient<2>(X, R, t, wj, dX, dR);
    else if (d == 2) add_gradient<3>(X, R, t, wj, dX, dR);
    else add_gradient<4>(X, R, t, wj, dX, dR);
}

// The vertices without all of the lists above them, in one launch: hardly any is
// attached, so the sizes of the sources do not mix much, and a small call waits
// for its launches (K^0 alone, 100,000 and 2,000 atoms: 22 and 13 us; by the
// kernels above 40 and 29).
__global__ void k_eval_vertices(const double* __restrict__ X, const double* __restrict__ R,
                                const int8_t* __restrict__ sdim, const int64_t* __restrict__ sidx, int64_t m, Rows4 rows,
                                double* __restrict__ out) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    const int d = sdim[j];
    const int4 t = rows.G[d][sidx[j]];
    out[j] = d == 0   ? orthosize_dd<1>(X, R, t)
             : d == 1 ? orthosize_dd<2>(X, R, t)
             : d == 2 ? orthosize_dd<3>(X, R, t)
                      : orthosize_dd<4>(X, R, t);
}

int eval_filtration(ac_ctx* c, const double* centres, const double* radii, double* const f_out[4], cudaStream_t s) {
    constexpr int T = EVAL_TILE, TS = EVAL_TILE_SHORT;
    Vals4 vals{};
    Rows4 rows;
    bool left_out = false;
    for (int d = 0; d < 4; d++) {
        vals.v[d] = f_out[d];
        rows.G[d] = c->Gbuf[d].as<int4>();
        left_out = left_out || (d > 0 && !f_out[d] && c->K[d].count > 0);
    }
    if (left_out && f_out[0] && c->K[0].count > 0) {
        const int64_t m = c->K[0].count;
        k_eval_vertices<<<(unsigned)((m + 127) / 128), 128, 0, s>>>(centres, radii, c->K[0].src_dim.as<int8_t>(),
                                                                    c->K[0].src_idx.as<int64_t>(), m, rows, f_out[0]);
        AC_LAUNCHED();
    }
    const int lo = left_out ? 1 : 0;
    for (int d = 3; d >= lo; d--) {
        const int64_t m = c->K[d].count;
        if (!f_out[d] || m == 0) continue;
        const bool shrt = m < EVAL_SHORT_ROWS;
        void (*k)(const double*, const double*, const int4*, const uint8_t*, int64_t, double*) =
            d == 3   ? (shrt ? k_eval_own<4, TS> : k_eval_own<4, T>)
            : d == 2 ? (shrt ? k_eval_own<3, TS> : k_eval_own<3, T>)
            : d == 1 ? (shrt ? k_eval_own<2, TS> : k_eval_own<2, T>)
                     : (shrt ? k_eval_own<1, TS> : k_eval_own<1, T>);
        const int tile = shrt ? TS : T;
        k<<<(unsigned)((m + tile - 1) / tile), EVAL_THREADS, 0, s>>>(
            centres, radii, c->Gbuf[d].as<int4>(), c->K[d].attached.as<uint8_t>(), m, f_out[d]);
        AC_LAUNCHED();
    }
    for (int d = lo; d < 3; d++) {  // a tetrahedron is never attached
        const int64_t m = c->K[d].count;
        if (!f_out[d] || m == 0) continue;
        const uint8_t* att = c->K[d].attached.as<uint8_t>();
        const int8_t* sdim = c->K[d].src_dim.as<int8_t>();
        const int64_t* sidx = c->K[d].src_idx.as<int64_t>();
        k_eval_attached<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(att, sdim, sidx, m, vals, f_out[d]);
        AC_LAUNCHED();
        const bool shrt = m < EVAL_SHORT_ROWS;
        const int tile = shrt ? TS : T;
        for (int e = d + 1; e < 4; e++) {
            if (f_out[e] || c->K[e].count == 0) continue;
            void (*k)(const double*, const double*, const int4*, const uint8_t*, const int8_t*, const int64_t*, int64_t,
                      double*) = e == 3 ? (shrt ? k_eval_source<4, TS> : k_eval_source<4, T>)
                                        : (shrt ? k_eval_source<3, TS> : k_eval_source<3, T>);
            k<<<(unsigned)((m + tile - 1) / tile), EVAL_THREADS, 0, s>>>(centres, radii, c->Gbuf[e].as<int4>(), att, sdim,
                                                                         sidx, m, f_out[d]);
            AC_LAUNCHED();
        }
    }
    AC_CUDA(cudaStreamSynchronize(s));
    return AC_OK;
}

// ---------------------------------------------------------------------------
// ac_backward: the same gradient, with every sum taken in a fixed order, so
// that repeated calls give bit-identical results (no floating-point atomics).
//
// Sum over the simplices sigma of w_sigma * dOrthoSize(src(sigma)): grouped by
// source, each source s contributes W_s * dOrthoSize(s), W_s the sum of the
// weights of the simplices whose source it is. An attached simplex takes its
// source from its parent, the coface its value came from (the build's
// coface passes keep, for every coface, the rows of its attached facets, and
// for every attached row its parent), and an unattached one is its own
// source. So:
//   1. k_weights_up, dimension 0 to 3, one thread per row: W'(sigma) =
//      w(sigma) + the W' of the attached facets whose parent sigma is, in
//      facet order. An unattached row's W' is its W_s; an attached row hands
//      its W' up and is no source.
//   2. k_contrib, the unattached rows: the orthocentre and barycentric
//      coordinates of s, and for each vertex k of s the contribution
//      (2 W_s lambda_k (p_k - c), -2 W_s lambda_k r_k).
//   3. k_edge_sums, eight lanes per atom b (a block for one with many rows): of the rows with first vertex b, the
//      contributions to b itself, and to each other vertex x. Such an x is the
//      second vertex of a K^1 row with first vertex b, and its sum is written
//      there (lane by lane in row order, so the order is fixed).
//   4. k_gather_atoms, eight lanes per atom a: its own sum and those of the K^1
//      rows (b, a), b the neighbours of a with a smaller input index (their grown
//      balls meet), each found by a binary search among b's rows; summed per lane
//      and then over the lanes by a fixed tree.
// Without 3. every atom read all the rows of those neighbours (600 rows for the
// 27 that hold it): 1.65 ms for the 100,000-atom probe globule; 3. and 4. take
// 0.19 and 0.07. FP64 additions go
// out at 16 clocks a warp however few lanes take part, so four atoms share a
// warp and a lane of k_edge_sums steps through its own rows only.

struct BackArgs {
    const double* X;         // centres (n x 3), input order
    const double* R;         // radii
    const int4* G[4];        // rows per dimension, global input indices
    const int64_t* v0[4];    // rows with first vertex g start at v0[d][g] (n + 1)
    const uint8_t* att[4];   // attached flags
    const double* w[4];      // dL/df per row (NULL: zero)
    double* Wp[4];           // W' per row (pass 1)
    const int64_t* frows[3]; // frows[d]: rows of the attached facets (dim d) of each coface (dim d + 1), or -1
    const unsigned long long* parent[3];  // parent[d][r]: the coface (row of dim d + 1) of attached row r of dim d
    // per row, per vertex: (dL/dp, dL/dr) contributions of the unattached rows (pass 2). Pass 3 keeps its sums in
    // them: for the second vertex of K^1 row e in C[1][2e + 1], for the rows that start with an atom in C[0] at the
    // atom's row (an atom without a row is in no simplex); only the lane that writes such a place has read it.
    double4* C[4];
    int64_t rows[4];
    const int32_t* rank;     // input index -> sorted position
    const int32_t* order;    // sorted position -> input index
    const int64_t* nb_off;   // neighbour rows (as in the per-atom pass)
    const int32_t* nb;
    int nb_stride;
    int64_t n;
};

__global__ void k_weights_up(BackArgs A, int d) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= A.rows[d]) return;
    double W = A.w[d] ? A.w[d][j] : 0.0;
    if (d >= 1 && A.frows[d - 1]) {
        const int64_t* fr = A.frows[d - 1] + j * (d + 1);
        for (int drop = 0; drop <= d; drop++) {
            const int64_t r = fr[drop];
            if (r >= 0 && A.parent[d - 1][r] == (unsigned long long)j) W += A.Wp[d - 1][r];
        }
    }
    A.Wp[d][j] = W;
}

template <int K, int TILE>
__global__ void __launch_bounds__(EVAL_THREADS) k_contrib(BackArgs A) {
    __shared__ int list[TILE];
    __shared__ int n_list;
    constexpr int d = K - 1;
    const int64_t first = (int64_t)blockIdx.x * TILE;
    const int n = gather_rows<TILE>(first, A.rows[d], list, &n_list, [&](int64_t j) { return A.att[d][j] != 0; });
    for (int u = threadIdx.x; u < n; u += EVAL_THREADS) {
        const int64_t j = first + list[u];
        double4* out = A.C[d] + j * K;
        const double W = A.Wp[d][j];
        if (W == 0.0) {
            for (int k = 0; k < K; k++) out[k] = make_double4(0.0, 0.0, 0.0, 0.0);
            continue;
        }
        const int4 g = A.G[d][j];
        const int v[4] = {g.x, g.y, g.z, g.w};
        const Ortho o = ortho_fp64<K>(A.X, A.R, g);
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int64_t a = v[k];
            const double l2 = 2.0 * W * o.lam[k];
            out[k] = make_double4(l2 * (A.X[3 * a] - o.c[0]), l2 * (A.X[3 * a + 1] - o.c[1]),
                                  l2 * (A.X[3 * a + 2] - o.c[2]), -l2 * A.R[a]);
        }
    }
}

constexpr int SUM_LANES = 8;
constexpr int SUM_THREADS = 128;

__device__ __forceinline__ void add4(double4& s, const double4& q) {
    s.x += q.x;
    s.y += q.y;
    s.z += q.z;
    s.w += q.w;
}

// sum over the SUM_LANES lanes of a group: a fixed tree, the same additions in the same order every call
__device__ __forceinline__ double4 sum_lanes(double4 s) {
#pragma unroll
    for (int o = SUM_LANES / 2; o >= 1; o >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        s.z += __shfl_xor_sync(0xffffffffu, s.z, o);
        s.w += __shfl_xor_sync(0xffffffffu, s.w, o);
    }
    return s;
}

// the sum of K^1 row e = (b, x): the edge's own contribution to x and those of b's triangles and tetrahedra
__device__ __forceinline__ void edge_sum(const BackArgs& A, int64_t b, int64_t e) {
    const int x = A.G[1][e].y;
    double4 s = make_double4(0.0, 0.0, 0.0, 0.0);
    if (!A.att[1][e]) s = A.C[1][e * 2 + 1];  // the edge itself
    for (int d = 2; d < 4; d++) {
        const int64_t r1 = A.v0[d][b + 1];
        for (int64_t r0 = A.v0[d][b]; r0 < r1; r0 += 32) {
            const int cnt = (int)(r1 - r0 < 32 ? r1 - r0 : 32);
            unsigned mask = 0u;  // of these rows, the unattached ones with vertex x
            for (int t = 0; t < cnt; t++) {
                const int4 g = A.G[d][r0 + t];
                if ((g.y == x || g.z == x || g.w == x) && !A.att[d][r0 + t]) mask |= 1u << t;
            }
            for (; mask; mask &= mask - 1) {
                const int64_t r = r0 + __ffs(mask) - 1;
                const int4 g = A.G[d][r];
                add4(s, A.C[d][r * (d + 1) + (g.y == x ? 1 : g.z == x ? 2 : 3)]);
            }
        }
    }
    A.C[1][e * 2 + 1] = s;
}

// Every edge of b goes over all of b's rows, so the work is their product: about
// 150 for an atom of a probe globule, but 900 edges times 6,000 rows for a large
// ball among small ones that comes before them in the input. Such atoms take the
// whole block (each edge is still summed by one lane in row order: the same
// numbers). Eight such balls of 900 neighbours, a whole backward: 2.6 ms; eight
// lanes each: 21.6 ms. The line, backward in us at 2,048 / 4,096 / 8,192 / 16,384:
// 256 balls of 300 neighbours 195 / 200 / 247 / 281, spread radii (20,000 balls)
// 232 / 221 / 241 / 250, globules of 2,000 atoms 197 / 187 / 187 / 174 and 100,000
// 734 / 709 / 706 / 697 (below the line no block waits for a wide atom).
constexpr int64_t SUM_BLOCK_WORK = 4096;

__global__ void __launch_bounds__(SUM_THREADS) k_edge_sums(BackArgs A) {
    __shared__ int64_t wide[SUM_THREADS / SUM_LANES];  // this block's atoms above the line
    __shared__ int n_wide;
    const int sub = threadIdx.x % SUM_LANES;
    const int64_t b = ((int64_t)blockIdx.x * SUM_THREADS + threadIdx.x) / SUM_LANES;
    if (threadIdx.x == 0) n_wide = 0;
    double4 own = make_double4(0.0, 0.0, 0.0, 0.0);
    if (b < A.n) {
        for (int d = 0; d < 4; d++)
            for (int64_t r = A.v0[d][b] + sub; r < A.v0[d][b + 1]; r += SUM_LANES)
                if (!A.att[d][r]) add4(own, A.C[d][r * (d + 1)]);
    }
    own = sum_lanes(own);
    __syncthreads();
    if (b < A.n) {
        if (sub == 0 && A.v0[0][b] < A.v0[0][b + 1]) A.C[0][A.v0[0][b]] = own;
        const int64_t e0 = A.v0[1][b], e1 = A.v0[1][b + 1];
        const int64_t rows = A.v0[2][b + 1] - A.v0[2][b] + A.v0[3][b + 1] - A.v0[3][b];
        if ((e1 - e0) * rows > SUM_BLOCK_WORK) {
            if (sub == 0) wide[atomicAdd(&n_wide, 1)] = b;
        } else {
            for (int64_t e = e0 + sub; e < e1; e += SUM_LANES) edge_sum(A, b, e);
        }
    }
    __syncthreads();
    for (int k = 0; k < n_wide; k++)
        for (int64_t e = A.v0[1][wide[k]] + threadIdx.x; e < A.v0[1][wide[k] + 1]; e += SUM_THREADS) edge_sum(A, wide[k], e);
}

__global__ void __launch_bounds__(SUM_THREADS) k_gather_atoms(BackArgs A, double* __restrict__ dX,
                                                               double* __restrict__ dR) {
    const int sub = threadIdx.x % SUM_LANES;
    const int64_t a = ((int64_t)blockIdx.x * SUM_THREADS + threadIdx.x) / SUM_LANES;
    double4 s = make_double4(0.0, 0.0, 0.0, 0.0);
    if (a < A.n) {
        if (sub == 0 && A.v0[0][a] < A.v0[0][a + 1]) s = A.C[0][A.v0[0][a]];
        const int ia = A.rank[a];
        const int64_t off = A.nb_stride ? (int64_t)ia * A.nb_stride : A.nb_off[ia];
        const int m = A.nb_stride ? (int)A.nb_off[ia] : (int)(A.nb_off[ia + 1] - off);
        for (int t = sub; t < m; t += SUM_LANES) {
            const int64_t b = A.order[A.nb[off + t]];
            if (b >= a) continue;
            int64_t lo = A.v0[1][b], hi = A.v0[1][b + 1];
            const int64_t end = hi;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (A.G[1][mid].y < a) lo = mid + 1;
                else hi = mid;
            }
            if (lo < end && A.G[1][lo].y == a) add4(s, A.C[1][lo * 2 + 1]);
        }
    }
    s = sum_lanes(s);
    if (sub == 0 && a < A.n) {
        dX[3 * a] = s.x;
        dX[3 * a + 1] = s.y;
        dX[3 * a + 2] = s.z;
        dR[a] = s.w;
    }
}

int backward(ac_ctx* c, const double* const dldf[4], double* dc, double* dr, cudaStream_t s) {
    const int64_t n = c->n;
    if (n == 0) return AC_OK;
    BackArgs A;
    memset(&A, 0, sizeof(A));
    A.X = c->centres.as<double>();
    A.R = c->radii.as<double>();
    size_t wrows = 0, crows = 0;
    for (int d = 0; d < 4; d++) {
        wrows += (size_t)c->K[d].count;
        crows += (size_t)c->K[d].count * (d + 1);
    }
    const size_t wbytes = ((wrows > 0 ? wrows : 1) * sizeof(double) + 255) & ~(size_t)255;
    AC_TRY(c->scratch[3].reserve(wbytes + (crows > 0 ? crows : 1) * sizeof(double4), s));
    double* Wbuf = c->scratch[3].as<double>();
    double4* Cbuf = reinterpret_cast<double4*>(static_cast<char*>(c->scratch[3].p) + wbytes);
    for (int d = 0; d < 4; d++) {
        const int64_t m = c->K[d].count;
        A.G[d] = c->Gbuf[d].as<int4>();
        A.v0[d] = c->K[d].v0_off.as<int64_t>();
        A.att[d] = c->K[d].attached.as<uint8_t>();
        A.w[d] = m > 0 ? dldf[d] : nullptr;
        A.Wp[d] = Wbuf;
        A.C[d] = Cbuf;
        A.rows[d] = m;
        Wbuf += m;
        Cbuf += m * (d + 1);
        if (d < 3) {
            const bool cof = c->K[d + 1].count > 0;  // the coface passes ran: frows[d], fargs[d] hold this build's
            A.frows[d] = cof ? c->frows[d].as<int64_t>() : nullptr;
            A.parent[d] = cof ? c->fargs[d].as<unsigned long long>() : nullptr;
        }
    }
    A.rank = c->rank.as<int32_t>();
    A.order = c->order.as<int32_t>();
    A.nb_off = c->nb_cnt.as<int64_t>();
    A.nb = c->nb.as<int32_t>();
    A.nb_stride = c->nb_stride;
    A.n = n;
    for (int d = 0; d < 4; d++) {
        const int64_t m = A.rows[d];
        if (m == 0) continue;
        k_weights_up<<<(unsigned)((m + 127) / 128), 128, 0, s>>>(A, d);
        AC_LAUNCHED();
    }
    for (int d = 0; d < 4; d++) {
        const int64_t m = A.rows[d];
        if (m == 0) continue;
        constexpr int T = EVAL_TILE, TS = EVAL_TILE_SHORT;
        const bool shrt = m < EVAL_SHORT_ROWS;
        void (*k)(BackArgs) = d == 3   ? (shrt ? k_contrib<4, TS> : k_contrib<4, T>)
                              : d == 2 ? (shrt ? k_contrib<3, TS> : k_contrib<3, T>)
                              : d == 1 ? (shrt ? k_contrib<2, TS> : k_contrib<2, T>)
                                       : (shrt ? k_contrib<1, TS> : k_contrib<1, T>);
        const int tile = shrt ? TS : T;
        k<<<(unsigned)((m + tile - 1) / tile), EVAL_THREADS, 0, s>>>(A);
        AC_LAUNCHED();
    }
    const unsigned nb = (unsigned)((n * SUM_LANES + SUM_THREADS - 1) / SUM_THREADS);
    k_edge_sums<<<nb, SUM_THREADS, 0, s>>>(A);
    AC_LAUNCHED();
    k_gather_atoms<<<nb, SUM_THREADS, 0, s>>>(A, dc, dr);
    AC_LAUNCHED();
    AC_CUDA(cudaStreamSynchronize(s));
    return AC_OK;
}

// ---------------------------------------------------------------------------
// ac_backward_noalloc: the gradient without any device allocation.
//
// ac_backward sums in a fixed order with per-simplex scratch it allocates.
// Callers that cannot allocate device memory (for example inside a training
// step whose memory belongs to another allocator, or a service with a fixed
// device memory budget) use this entry point instead: it runs k_backward (one
// thread per simplex, FP64 atomics), whose only scratch is the table of the
// four per-dimension source-list pointers it reads, and that table lives in
// the static array below, which every GPU that loads the library holds until
// the process exits. Maximum: NOALLOC_TABLE_ENTRIES = 4 pointers (one per
// dimension 0..3), 32 bytes in a 256-byte-aligned array. Every call overwrites
// the whole table before its kernels read it, so nothing in it has to start at
// zero; calls that overlap on the GPU (other streams, other host threads)
// share the one table and race. The cached device address of the table does
// not survive a cudaDeviceReset.
constexpr int NOALLOC_TABLE_ENTRIES = 4;
static __device__ __align__(256) const int4* g_noalloc_table[NOALLOC_TABLE_ENTRIES];

// Device addresses of g_noalloc_table, looked up once per device with that
// device current (the host-side name is only a stand-in).
constexpr int NOALLOC_MAX_DEVICES = 64;
static const int4** g_noalloc_addr[NOALLOC_MAX_DEVICES];
static std::mutex g_noalloc_mu;

static int noalloc_table(const int4*** out) {
    int dev = 0;
    AC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return fail(AC_ERR_INVALID_ARG, "device ordinal above 63");
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void* ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_table);
        if (e != cudaSuccess || !ptr) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_table)", __FILE__, __LINE__);
        g_noalloc_addr[dev] = (const int4**)ptr;
    }
    *out = g_noalloc_addr[dev];
    return AC_OK;
}

int backward_noalloc(ac_ctx* c, const double* const dldf[4], double* dc, double* dr, cudaStream_t s) {
    const int lists = 4;
    if (lists > NOALLOC_TABLE_ENTRIES) return fail(AC_ERR_CAPACITY, "more simplex lists than the static table holds");
    const int4** table = nullptr;
    AC_TRY(noalloc_table(&table));
    const int4* h[NOALLOC_TABLE_ENTRIES];
    for (int d = 0; d < lists; d++) h[d] = c->Gbuf[d].as<int4>();
    AC_CUDA(cudaMemcpyAsync(table, h, sizeof(h), cudaMemcpyHostToDevice, s));
    const int64_t n = c->n;
    AC_CUDA(cudaMemsetAsync(dc, 0, (size_t)(n > 0 ? n : 0) * 3 * sizeof(double), s));
    AC_CUDA(cudaMemsetAsync(dr, 0, (size_t)(n > 0 ? n : 0) * sizeof(double), s));
    for (int d = 0; d < lists; d++) {
        const int64_t m = c->K[d].count;
        if (!dldf[d] || m == 0) continue;
        k_backward<<<(unsigned)((m + 127) / 128), 128, 0, s>>>(c->centres.as<double>(), c->radii.as<double>(),
                                                               c->K[d].src_dim.as<int8_t>(), c->K[d].src_idx.as<int64_t>(),
                                                               m, table, dldf[d], dc, dr);
        AC_LAUNCHED();
    }
    AC_CUDA(cudaStreamSynchronize(s));
    return AC_OK;
}

}  // namespace ac
