// gl_vcycle.cu -- the V-cycle that applies R_k = AMG_k(K-hat + 2 D|psi|^2, D .)
// (Eq. prec2): on each level one symmetric Gauss-Seidel step before and after
// the coarse correction (Sec. 4: one pre- and one post-smoothing step), the
// Gauss-Seidel sweeps taken colour by colour (forward: colours ascending,
// backward: descending), and a dense solve on the coarsest level.
//
// All vectors are in the solve ordering, where each colour is a contiguous
// range of positions.  On level 0 the operator is used in its row-scaled form
// K + 2|psi|^2 = D^-1 (K-hat + 2 D|psi|^2): Gauss-Seidel on D^-1 A with right-hand
// side v is Gauss-Seidel on A with right-hand side D v, and the residual handed
// to the restriction is multiplied by D.
#include "gl_internal.cuh"
#include "gl_kernels.cuh"
#include "gl_profile.cuh"

namespace gl {

template <typename T>
struct LevelOps;
template <>
struct LevelOps<double> {
    using C = double2;
    static const Sell<C> &A(const Level &L) { return *L.A; }
    static const double *diag(const Level &L) { return L.diag.get(); }
    static const Sell<C> &P(const Level &L) { return L.P; }
    static const CsrG<C> &PHg(const Level &L) { return L.PHg; }
    static C *b(Level &L) { return L.b.get(); }
    static C *x(Level &L) { return L.x.get(); }
    static C *r(Level &L) { return L.r.get(); }
};
template <>
struct LevelOps<float> {
    using C = float2;
    static const Sell<C> &A(const Level &L) { return *L.A32; }
    static const float *diag(const Level &L) { return L.diag32.get(); }
    static const Sell<C> &P(const Level &L) { return L.P32; }
    static const CsrG<C> &PHg(const Level &L) { return L.PHg32; }
    static C *b(Level &L) { return L.b32.get(); }
    static C *x(Level &L) { return L.x32.get(); }
    static C *r(Level &L) { return L.r32.get(); }
};

// x_i <- (b_i - sum_{k != i} A_ik x_k) / A_ii for the rows of one colour [lo, hi).
// `first`: first forward pass from x = 0, where only positions < lo hold values.
template <typename C, typename R>
__global__ void __launch_bounds__(256) k_gs(int64_t lo, int64_t hi, SellView<C> A, const R *__restrict__ diag,
                                            const C *__restrict__ b, C *__restrict__ x, int first,
                                            const int *__restrict__ stop) {
    if (stop && *stop) return;
    int64_t p = lo + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= hi) return;
    C acc;
    if (first && lo == 0) {  // every neighbour of the first colour still holds zero
        acc.x = 0;
        acc.y = 0;
    } else {
        acc = first ? sell_row_before<C, C>(A, p, x, lo) : sell_row<C, C>(A, p, x);
    }
    C bb = b[p];
    R d = (R)1 / diag[p];
    x[p] = mk((bb.x - acc.x) * d, (bb.y - acc.y) * d);
}

// r = (b - A x) * scale (scale = |V| on level 0, none below)
template <typename C, typename R>
__global__ void __launch_bounds__(256) k_resid(int64_t n, SellView<C> A, const R *__restrict__ diag,
                                               const C *__restrict__ b, const C *__restrict__ x,
                                               const R *__restrict__ scale, C *__restrict__ r,
                                               const int *__restrict__ stop) {
    if (stop && *stop) return;
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    C acc = sell_row<C, C>(A, p, x);
    C xx = x[p], bb = b[p];
    R d = diag[p];
    R sc = scale ? scale[p] : (R)1;
    r[p] = mk((bb.x - acc.x - d * xx.x) * sc, (bb.y - acc.y - d * xx.y) * sc);
}

// the two kernels above on the finest level of an even-N lattice, with the
// tabulated stencil instead of the stored one (FP32).  Each thread takes
// LAT_RPT rows, blockDim.x apart, and issues the neighbour reads of all of them
// before any write: a colour's rows read only the other colour's x.
constexpr int LAT_RPT = 1;

__global__ void __launch_bounds__(256) k_gs_lat(int64_t lo, int64_t hi, LatticeView L, const float *__restrict__ diag,
                                                const float2 *__restrict__ b, float2 *__restrict__ x, int first,
                                                const int *__restrict__ stop) {
    if (stop && *stop) return;
    const int64_t p0 = lo + (int64_t)blockIdx.x * blockDim.x * LAT_RPT + threadIdx.x;
    // from x = 0 the first colour has no nonzero neighbour and the second sees
    // only the first (two colours, each node's neighbours of the other colour)
    const bool none = first && lo == 0;
    float2 acc[LAT_RPT];
#pragma unroll
    for (int u = 0; u < LAT_RPT; ++u) {
        const int64_t p = p0 + (int64_t)u * blockDim.x;
        acc[u] = (p < hi && !none) ? lattice_row(L, p, x) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < LAT_RPT; ++u) {
        const int64_t p = p0 + (int64_t)u * blockDim.x;
        if (p < hi) {
            const float2 bb = b[p];
            const float d = 1.f / diag[p];
            x[p] = make_float2((bb.x - acc[u].x) * d, (bb.y - acc[u].y) * d);
        }
    }
}
// k_gs_lat with two consecutive positions of a colour per thread: for N % 4 == 0
// positions 2t and 2t + 1 of a colour are the nodes v and v + 2 of one x-line,
// so b, diag, |V| and the written x move as 16- and 8-byte vectors, and the
// neighbours of the pair along y and z (and two of the three along x) are
// adjacent positions of the other colour, read as one 16-byte vector each.
// Per row the edges are summed in the order of lattice_row_f.  (Node v of
// colour c sits at position v >> 1; with p even, v = 2p + a, a = 1 when the
// parity of the line start differs from c.)
__global__ void __launch_bounds__(256) k_gs_lat2(int64_t lo, int64_t hi, LatticeView L,
                                                     const float *__restrict__ diag, const float2 *__restrict__ b,
                                                     float2 *__restrict__ x, int first, const int *__restrict__ stop) {
    if (stop && *stop) return;
    const int64_t p = lo + 2 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    if (p >= hi) return;
    const bool none = first && lo == 0;
    const uint32_t c = p >= L.nred ? 1u : 0u;
    const int64_t base = c ? L.nred : 0;
    const int64_t other = c ? 0 : L.nred;
    const uint32_t N = (uint32_t)L.N;
    const uint32_t r = (uint32_t)(p - base);  // even
    const uint32_t v0 = 2u * r;
    const uint32_t row = L.dN.div(v0), k = L.dN.div(row);
    const uint32_t i0 = v0 - row * N, j = row - k * N;
    const uint32_t a = ((i0 + j + k) & 1u) != c ? 1u : 0u;
    const uint32_t i = i0 + a;
    float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
    if (!none) {
        const float2 *xo = x + other;
        auto e = [](float2 &acc, float2 t, float2 xv, bool plus) {
            const float ty = plus ? t.y : -t.y;
            acc.x += t.x * xv.x - ty * xv.y;
            acc.y += t.x * xv.y + ty * xv.x;
        };
        // x-direction: positions r - 1 + a .. r + 1 + a of the other colour
        const float4 xm = *reinterpret_cast<const float4 *>(xo + r);  // r, r + 1
        const float2 xlo = make_float2(xm.x, xm.y), xhi = make_float2(xm.z, xm.w);
        float2 xe = make_float2(0.f, 0.f);
        if (a == 0u) {
            if (i > 0) xe = xo[r - 1];
        } else {
            if (i + 3 < N) xe = xo[r + 2];
        }
        // node 1 (v0 + a): x+ -> (v + 1) >> 1, x- -> (v - 1) >> 1
        // a = 0: x+ = r, x- = r - 1; a = 1: x+ = r + 1, x- = r
        // node 2 (v + 2): a = 0: x+ = r + 1, x- = r; a = 1: x+ = r + 2, x- = r + 1
        const float2 t = __ldg(L.tx + (j + N * k));
        if (a == 0u) {
            e(acc0, t, xlo, true);
            if (i > 0) e(acc0, t, xe, false);
            if (i + 3 < N) e(acc1, t, xhi, true);
            e(acc1, t, xlo, false);
        } else {
            e(acc0, t, xhi, true);
            e(acc0, t, xlo, false);
            if (i + 3 < N) e(acc1, t, xe, true);
            e(acc1, t, xhi, false);
        }
        const uint32_t hN = N / 2;
        {
            const float2 t0 = __ldg(L.ty + (i + N * k)), t1 = __ldg(L.ty + (i + 2 + N * k));
            if (j + 1 < N) {
                const float4 q = *reinterpret_cast<const float4 *>(xo + r + hN);
                e(acc0, t0, make_float2(q.x, q.y), true);
                e(acc1, t1, make_float2(q.z, q.w), true);
            }
            if (j > 0) {
                const float4 q = *reinterpret_cast<const float4 *>(xo + r - hN);
                e(acc0, t0, make_float2(q.x, q.y), false);
                e(acc1, t1, make_float2(q.z, q.w), false);
            }
        }
        if (L.dim == 3) {
            const uint32_t hP = N * N / 2;
            const float2 t0 = __ldg(L.tz + (i + N * j)), t1 = __ldg(L.tz + (i + 2 + N * j));
            if (k + 1 < N) {
                const float4 q = *reinterpret_cast<const float4 *>(xo + r + hP);
                e(acc0, t0, make_float2(q.x, q.y), true);
                e(acc1, t1, make_float2(q.z, q.w), true);
            }
            if (k > 0) {
                const float4 q = *reinterpret_cast<const float4 *>(xo + (int64_t)r - hP);
                e(acc0, t0, make_float2(q.x, q.y), false);
                e(acc1, t1, make_float2(q.z, q.w), false);
            }
        }
        const float2 vv = *reinterpret_cast<const float2 *>(L.vol + p);
        const float iv0 = 1.f / vv.x, iv1 = 1.f / vv.y;
        acc0 = make_float2(acc0.x * iv0, acc0.y * iv0);
        acc1 = make_float2(acc1.x * iv1, acc1.y * iv1);
    }
    const float4 bb = *reinterpret_cast<const float4 *>(b + p);
    const float2 dd = *reinterpret_cast<const float2 *>(diag + p);
    const float d0 = 1.f / dd.x, d1 = 1.f / dd.y;
    *reinterpret_cast<float4 *>(x + p) =
        make_float4((bb.x - acc0.x) * d0, (bb.y - acc0.y) * d0, (bb.z - acc1.x) * d1, (bb.w - acc1.y) * d1);
}
// the first two half-sweeps from x = 0 in one launch: red rows x = b / diag,
// black rows relaxed against their red neighbours' b / diag (the values those
// rows get in the same launch)
__global__ void __launch_bounds__(256) k_gs_lat_first2(int64_t n, LatticeView L, const float *__restrict__ diag,
                                                       const float2 *__restrict__ b, float2 *__restrict__ x,
                                                       const int *__restrict__ stop) {
    if (stop && *stop) return;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    float2 acc = make_float2(0.f, 0.f);
    if (p >= L.nred)
        acc = lattice_row_f(L, p, [&](int64_t q) {
            const float2 bq = b[q];
            const float dq = 1.f / diag[q];
            return make_float2(bq.x * dq, bq.y * dq);
        });
    const float2 bb = b[p];
    const float d = 1.f / diag[p];
    x[p] = make_float2((bb.x - acc.x) * d, (bb.y - acc.y) * d);
}

// the residual of the rows [lo, n) (the rows below lo are not written)
__global__ void __launch_bounds__(256) k_resid_lat(int64_t lo, int64_t n, LatticeView L,
                                                   const float *__restrict__ diag, const float2 *__restrict__ b,
                                                   const float2 *__restrict__ x, const float *__restrict__ scale,
                                                   float2 *__restrict__ r, const int *__restrict__ stop) {
    if (stop && *stop) return;
    const int64_t p0 = lo + (int64_t)blockIdx.x * blockDim.x * LAT_RPT + threadIdx.x;
    float2 acc[LAT_RPT];
#pragma unroll
    for (int u = 0; u < LAT_RPT; ++u) {
        const int64_t p = p0 + (int64_t)u * blockDim.x;
        acc[u] = p < n ? lattice_row(L, p, x) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < LAT_RPT; ++u) {
        const int64_t p = p0 + (int64_t)u * blockDim.x;
        if (p < n) {
            const float2 xx = x[p], bb = b[p];
            const float d = diag[p];
            const float sc = scale ? scale[p] : 1.f;
            r[p] = make_float2((bb.x - acc[u].x - d * xx.x) * sc, (bb.y - acc[u].y - d * xx.y) * sc);
        }
    }
}

// y = S x (add = 0) or y += S x (add = 1) for the rows [lo, n) of a rectangular
// sliced-ELL S
template <typename C>
__global__ void __launch_bounds__(256) k_spmv(int64_t lo, int64_t n, SellView<C> S, const C *__restrict__ x,
                                              C *__restrict__ y, int add, const int *__restrict__ stop) {
    if (stop && *stop) return;
    int64_t p = lo + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    C acc = sell_row<C, C>(S, p, x);
    if (add) acc = cadd(acc, y[p]);
    y[p] = acc;
}

// ---------------------------------------------------------------- grouped-CSR rows
// sum over the stored entries of row `row` (columns below `lim` only) by the G
// lanes of a group; every lane of the warp must call this (shuffles), rows past
// the end pass row < 0.  The result is complete in the group's first lane.
template <int G, typename C>
__device__ __forceinline__ C group_row(const CsrGView<C> &A, int64_t row, int lane, const C *__restrict__ x,
                                       int64_t lim) {
    C acc;
    acc.x = 0;
    acc.y = 0;
    if (row >= 0) {
        const int64_t q1 = A.rp[row + 1];
        int64_t q = A.rp[row] + lane;
        // four entries per step with all their loads issued first (long rows, such
        // as a restriction to a small coarse level, would otherwise wait for one
        // column and one gather per entry in turn); the sum runs in the same order
        for (; q + 3 * G < q1; q += 4 * G) {
            int32_t c[4];
            C v[4], xv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) c[u] = __ldg(A.col + q + u * G);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                v[u] = A.val[q + u * G];
                if (c[u] < lim) xv[u] = x[c[u]];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (c[u] < lim) cfma(acc, v[u], xv[u]);
        }
        for (; q < q1; q += G) {
            int32_t c = __ldg(A.col + q);
            if (c < lim) cfma(acc, A.val[q], x[c]);
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        acc.x += __shfl_down_sync(0xffffffffu, acc.x, o, G);
        acc.y += __shfl_down_sync(0xffffffffu, acc.y, o, G);
    }
    return acc;
}

// y = S x (add = 0) or y += S x (add = 1), grouped CSR
template <int G, typename C>
__global__ void __launch_bounds__(256) k_spmv_g(CsrGView<C> S, const C *__restrict__ x, C *__restrict__ y, int add,
                                                const int *__restrict__ stop) {
    if (stop && *stop) return;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t row = t / G;
    int lane = (int)(t % G);
    bool ok = row < S.nrows;
    C acc = group_row<G, C>(S, ok ? row : -1, lane, x, INT64_MAX);
    if (ok && lane == 0) y[row] = add ? cadd(acc, y[row]) : acc;
}

// dispatch on the group width
#define GL_DISPATCH_G(G_, CALL)                       \
    switch (G_) {                                     \
        case 1: { constexpr int GG = 1; CALL; break; }   \
        case 2: { constexpr int GG = 2; CALL; break; }   \
        case 4: { constexpr int GG = 4; CALL; break; }   \
        case 8: { constexpr int GG = 8; CALL; break; }   \
        case 16: { constexpr int GG = 16; CALL; break; } \
        default: { constexpr int GG = 32; CALL; break; } \
    }

template <typename C>
static void spmv_g(const CsrG<C> &S, const C *x, C *y, int add, const int *stop, cudaStream_t s) {
    GL_DISPATCH_G(S.G, (k_spmv_g<GG, C><<<grid_for(S.nrows * GG, 256), 256, 0, s>>>(S.view(), x, y, add, stop)));
}

// Autotuner: times the grouped-CSR SpMV of one operator for every group width
// (lanes per row) on this GPU and keeps the fastest.  x must hold the
// operator's column count, y its row count (contents irrelevant).
template <typename C>
static void tune_groups(CsrG<C> &S, const C *x, C *y, cudaStream_t s) {
    if (S.nrows <= 0 || S.nnz <= 0) return;
    cudaEvent_t e0, e1;
    GL_CUDA(cudaEventCreate(&e0));
    GL_CUDA(cudaEventCreate(&e1));
    int best = S.G;
    float best_ms = 1e30f;
    for (int g = 1; g <= 32; g *= 2) {
        S.G = g;
        spmv_g<C>(S, x, y, 0, nullptr, s);  // warm
        GL_CUDA(cudaEventRecord(e0, s));
        for (int r = 0; r < 5; ++r) spmv_g<C>(S, x, y, 0, nullptr, s);
        GL_CUDA(cudaEventRecord(e1, s));
        GL_CUDA(cudaEventSynchronize(e1));
        float ms = 0;
        GL_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        if (ms < best_ms) {
            best_ms = ms;
            best = g;
        }
    }
    S.G = best;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
}

void autotune_levels(gl_prec_s *p, bool fp32, cudaStream_t s) {
    for (int l = 0; l + 1 < p->nlev; ++l) {
        Level &L = p->L[l], &Lc = p->L[l + 1];
        if (fp32) {
            tune_groups<float2>(L.PHg32, L.r32.get(), Lc.b32.get(), s);
        } else {
            tune_groups<double2>(L.PHg, L.r.get(), Lc.b.get(), s);
        }
    }
    GL_LAUNCH_CHECK();
}

// x = M b for the dense coarsest inverse (FP64).  The product is bound by the
// FP64 pipe (four FMAs per complex entry), so one warp takes one row and every
// lane keeps four independent accumulators to keep FMAs in flight; b comes
// through L1 (the same 16 n bytes for every row).
constexpr int DMV_WARPS = 8;
__global__ void __launch_bounds__(32 * DMV_WARPS) k_dense_mv(int64_t n, const double2 *__restrict__ M,
                                                             const double2 *__restrict__ b, double2 *__restrict__ x,
                                                             const int *__restrict__ stop) {
    if (stop && *stop) return;
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * DMV_WARPS + (threadIdx.x >> 5);
    if (row >= n) return;
    const double2 *mr = M + row * n;
    double2 a0 = make_double2(0, 0), a1 = a0, a2 = a0, a3 = a0;
    int64_t j = lane;
    for (; j + 96 < n; j += 128) {
        cfma(a0, mr[j], __ldg(b + j));
        cfma(a1, mr[j + 32], __ldg(b + j + 32));
        cfma(a2, mr[j + 64], __ldg(b + j + 64));
        cfma(a3, mr[j + 96], __ldg(b + j + 96));
    }
    for (; j < n; j += 32) cfma(a0, mr[j], __ldg(b + j));
    double sx = (a0.x + a1.x) + (a2.x + a3.x), sy = (a0.y + a1.y) + (a2.y + a3.y);
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_down_sync(0xffffffffu, sx, o);
        sy += __shfl_down_sync(0xffffffffu, sy, o);
    }
    if (lane == 0) x[row] = make_double2(sx, sy);
}

// x = M b for the FP32 V-cycle: b is an FP32 vector (exact), M the dense
// coarsest inverse as double-FP32 pairs, every product error-free and every sum
// compensated (Dot2), so the value carries about 48 significant bits before it
// is rounded to FP32 - the FP64 product's value, at the FP32 pipe's rate (the
// FP64 form of this product is bound by the FP64 pipe).  The product is a
// stream of the matrix (16 B per entry): one warp takes a row, so every row of a
// coarsest level of a few thousand nodes is resident at once (one wave; wider
// blocks left a second, mostly idle wave: 31 us against 25 us at 2720 nodes),
// and every lane keeps U entries in flight; partial (sum, compensation) pairs
// are combined by shuffles.
constexpr int DMV_DF_THREADS = 32;  // one warp
__global__ void __launch_bounds__(DMV_DF_THREADS) k_dense_mv_df(int64_t n, const float4 *__restrict__ M,
                                                                const float2 *__restrict__ b,
                                                                float2 *__restrict__ x, const int *__restrict__ stop) {
    if (stop && *stop) return;
    const int64_t row = blockIdx.x;
    const float4 *mr = M + row * n;
    float rs[2] = {0.f, 0.f}, rc[2] = {0.f, 0.f}, is[2] = {0.f, 0.f}, ic[2] = {0.f, 0.f};
    int64_t j = threadIdx.x;
    constexpr int U = 8;
    for (; j + (U - 1) * DMV_DF_THREADS < n; j += U * DMV_DF_THREADS) {
        float4 m[U];
        float2 bb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            m[u] = mr[j + u * DMV_DF_THREADS];
            bb[u] = __ldg(b + j + u * DMV_DF_THREADS);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int a = u & 1;
            dot2_df(rs[a], rc[a], make_float2(m[u].x, m[u].y), bb[u].x);
            dot2_df(rs[a], rc[a], make_float2(-m[u].z, -m[u].w), bb[u].y);
            dot2_df(is[a], ic[a], make_float2(m[u].x, m[u].y), bb[u].y);
            dot2_df(is[a], ic[a], make_float2(m[u].z, m[u].w), bb[u].x);
        }
    }
    for (; j < n; j += DMV_DF_THREADS) {
        const float4 m = mr[j];
        const float2 bb = __ldg(b + j);
        dot2_df(rs[0], rc[0], make_float2(m.x, m.y), bb.x);
        dot2_df(rs[0], rc[0], make_float2(-m.z, -m.w), bb.y);
        dot2_df(is[0], ic[0], make_float2(m.x, m.y), bb.y);
        dot2_df(is[0], ic[0], make_float2(m.z, m.w), bb.x);
    }
    dot2_add(rs[0], rc[0], rs[1]);
    rc[0] = __fadd_rn(rc[0], rc[1]);
    dot2_add(is[0], ic[0], is[1]);
    ic[0] = __fadd_rn(ic[0], ic[1]);
    for (int o = 16; o > 0; o >>= 1) {
        const float a = __shfl_down_sync(0xffffffffu, rs[0], o), ac = __shfl_down_sync(0xffffffffu, rc[0], o);
        const float c = __shfl_down_sync(0xffffffffu, is[0], o), cc = __shfl_down_sync(0xffffffffu, ic[0], o);
        dot2_add(rs[0], rc[0], a);
        rc[0] = __fadd_rn(rc[0], ac);
        dot2_add(is[0], ic[0], c);
        ic[0] = __fadd_rn(ic[0], cc);
    }
    if (threadIdx.x == 0) x[row] = make_float2(__fadd_rn(rs[0], rc[0]), __fadd_rn(is[0], ic[0]));
}

__global__ void k_split_dense_df(int64_t nn, const double2 *__restrict__ a, float4 *__restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= nn) return;
    const float2 re = split_df(a[i].x), im = split_df(a[i].y);
    out[i] = make_float4(re.x, re.y, im.x, im.y);
}

void coarse_inverse_df(Level &L, cudaStream_t s) {
    const int64_t nn = L.n * L.n;
    // an existing buffer of the right size is kept (captured solve graphs hold its address)
    if (L.Ainv_df.n != (size_t)nn) L.Ainv_df.alloc(nn);
    k_split_dense_df<<<grid_for(nn, 256), 256, 0, s>>>(nn, L.Ainv.get(), L.Ainv_df.get());
    GL_LAUNCH_CHECK();
}

template <typename C>
__global__ void k_axpy_t(int64_t n, const C *__restrict__ e, C *__restrict__ z, const int *__restrict__ stop) {
    if (stop && *stop) return;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) z[i] = cadd(z[i], e[i]);
}

__global__ void k_f2d(int64_t n, const float2 *a, double2 *b, const int *stop) {
    if (stop && *stop) return;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = to64(a[i]);
}
__global__ void k_d2f2(int64_t n, const double2 *a, float2 *b, const int *stop) {
    if (stop && *stop) return;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = to32(a[i]);
}

template <typename T>
static void coarse_solve(gl_prec_s *p, Level &L, const typename LevelOps<T>::C *b, typename LevelOps<T>::C *x,
                         const int *stop, cudaStream_t s);
template <>
void coarse_solve<double>(gl_prec_s *, Level &L, const double2 *b, double2 *x, const int *stop, cudaStream_t s) {
    ProfScope ps("coarse", (double)L.n * L.n * sizeof(double2), s);
    k_dense_mv<<<grid_for(L.n, DMV_WARPS), 32 * DMV_WARPS, 0, s>>>(L.n, L.Ainv.get(), b, x, stop);
}
template <>
void coarse_solve<float>(gl_prec_s *p, Level &L, const float2 *b, float2 *x, const int *stop, cudaStream_t s) {
    if (L.Ainv_df.get()) {
        // double-FP32 product of the FP32 right-hand side
        ProfScope ps("coarse", (double)L.n * L.n * sizeof(float4), s);
        k_dense_mv_df<<<(unsigned)L.n, DMV_DF_THREADS, 0, s>>>(L.n, L.Ainv_df.get(), b, x, stop);
        return;
    }
    // the FP32 right-hand side widened once, the FP64 solve, the result narrowed
    note_launch(2);
    k_f2d<<<grid_for(L.n, 256), 256, 0, s>>>(L.n, b, p->coarse_b64.get(), stop);
    {
        ProfScope ps("coarse", (double)L.n * L.n * sizeof(double2), s);
        k_dense_mv<<<grid_for(L.n, DMV_WARPS), 32 * DMV_WARPS, 0, s>>>(L.n, L.Ainv.get(), p->coarse_b64.get(),
                                                                       p->coarse_x64.get(), stop);
    }
    k_d2f2<<<grid_for(L.n, 256), 256, 0, s>>>(L.n, p->coarse_x64.get(), x, stop);
}

template <typename T>
static void gs_sweep(Level &L, int level, const typename LevelOps<T>::C *b, typename LevelOps<T>::C *x, int c,
                     bool first, const int *stop, cudaStream_t s, const LatticeView *lat = nullptr) {
    using O = LevelOps<T>;
    using C = typename O::C;
    int64_t lo = L.cstart[c], hi = L.cstart[c + 1];
    if (hi <= lo) return;
    if constexpr (sizeof(T) == 4) {
        if (lat) {
            // diagonal, b and the written x per row; the other colour's x once and
            // the phase tables, unless the colour is relaxed from a zero guess
            double bytes = (double)(hi - lo) * (sizeof(T) + 2 * sizeof(C));
            if (!(first && lo == 0))
                bytes += (double)(L.n - (hi - lo)) * sizeof(C) + (double)lat->N * lat->N * lat->dim * 8.0;
            ProfScope ps("gs0", bytes, s);
            if (lat->N % 4 == 0)  // colour ranges of even length, pairs within one x-line
                k_gs_lat2<<<grid_for((hi - lo) / 2, 256), 256, 0, s>>>(lo, hi, *lat, O::diag(L), b, x, first ? 1 : 0,
                                                                       stop);
            else
                k_gs_lat<<<grid_for(hi - lo, 256 * LAT_RPT), 256, 0, s>>>(lo, hi, *lat, O::diag(L), b, x,
                                                                         first ? 1 : 0, stop);
            return;
        }
    }
    // algorithmic bytes: diagonal, b and the written x for each row; the stored
    // off-diagonals (value + column) and each neighbour value once, unless the
    // colour is relaxed from an all-zero guess
    double rows = (double)(hi - lo);
    double bytes = rows * (sizeof(T) + 2 * sizeof(C));
    if (!(first && lo == 0))
        bytes += (double)L.cnnz[c] * (sizeof(C) + 4) + (double)(first ? lo : L.n - (hi - lo)) * sizeof(C);
    // a complex FMA (8 flops) per entry read, (b - acc) / diag per row (6)
    const double flops = (first && lo == 0 ? 0.0 : 8.0 * (double)L.cnnz[c]) + 6.0 * rows;
    ProfScope ps(level == 0 ? "gs0" : "gs", bytes, s, flops);
    k_gs<C, T><<<grid_for(hi - lo, 256), 256, 0, s>>>(lo, hi, O::A(L).view(), O::diag(L), b, x, first ? 1 : 0, stop);
}

// symmetric Gauss-Seidel: forward over colours, then backward; the backward pass
// starts one colour early because re-relaxing the last forward colour with
// unchanged neighbours reproduces the same values
template <typename T>
static void sgs(Level &L, int level, const typename LevelOps<T>::C *b, typename LevelOps<T>::C *x, bool zero_start,
                const int *stop, cudaStream_t s, const LatticeView *lat = nullptr) {
    int nc = L.ncolors;
    if constexpr (sizeof(T) == 4) {
        if (lat && zero_start && nc == 2) {
            // both forward colours in one launch; per row b, diagonal and the written
            // x, the red rows' b and diagonal once more for the black rows, the tables
            double bytes = (double)L.n * (sizeof(T) + 2 * sizeof(typename LevelOps<T>::C)) +
                           (double)L.cstart[1] * (sizeof(T) + sizeof(typename LevelOps<T>::C)) +
                           (double)lat->N * lat->N * lat->dim * 8.0;
            {
                ProfScope ps("gs0", bytes, s);
                k_gs_lat_first2<<<grid_for(L.n, 256), 256, 0, s>>>(L.n, *lat, LevelOps<T>::diag(L), b, x, stop);
            }
            gs_sweep<T>(L, level, b, x, 0, false, stop, s, lat);
            return;
        }
    }
    for (int c = 0; c < nc; ++c) gs_sweep<T>(L, level, b, x, c, zero_start, stop, s, lat);
    for (int c = nc - 2; c >= 0; --c) gs_sweep<T>(L, level, b, x, c, false, stop, s, lat);
}

// closed-form finest-level stencil for the FP32 V-cycle, when the mesh has one
template <typename T>
static bool lattice_for(const gl_prec_s *p, LatticeView &v) {
    if constexpr (sizeof(T) == 4) {
        if (p->lattice && p->mesh->lat_ok && p->L[0].ncolors == 2) {
            v = lattice_view(p->mesh);
            return true;
        }
    }
    return false;
}

// pre- or post-smoothing on the finest level: per-colour launches (two colours on a
// lattice, more on a general mesh beyond the sizes of sweep_finest)
template <typename T>
static void smooth_finest(gl_prec_s *p, const typename LevelOps<T>::C *b, typename LevelOps<T>::C *x, bool zero_start,
                          const int *stop, cudaStream_t s) {
    LatticeView lv;
    const bool lat = lattice_for<T>(p, lv);
    sgs<T>(p->L[0], 0, b, x, zero_start, stop, s, lat ? &lv : nullptr);
}

template <typename T>
static void vcycle(gl_prec_s *p, int l, const typename LevelOps<T>::C *b, typename LevelOps<T>::C *x,
                   const int *stop, cudaStream_t s) {
    using O = LevelOps<T>;
    using C = typename O::C;
    Level &L = p->L[l];
    if (l == p->nlev - 1) {
        coarse_solve<T>(p, L, b, x, stop, s);
        return;
    }
    Level &Lc = p->L[l + 1];
    C *r = O::r(L);
    bool restrict_black = false;
    const T *scale;  // of the residual handed to the restriction
    if constexpr (sizeof(T) == 8)
        scale = l == 0 ? p->mesh->volp.get() : nullptr;
    else
        scale = l == 0 ? p->mesh->volp32.get() : nullptr;
    if (p->swept(l, sizeof(T) == 4)) {
        sweep_step<T>(p, l, b, x, true, r, scale, stop, s);  // and the residual
    } else {
        smooth_finest<T>(p, b, x, true, stop, s);
        ProfScope ps("resid0", 0, s);
        LatticeView lv;
        bool lat = lattice_for<T>(p, lv);
        if constexpr (sizeof(T) == 4) {
            if (lat) {
                // the pre-smoothing ended by relaxing the red rows against black
                // neighbours it left unchanged, so their residual is zero (up to the
                // rounding of that relaxation): only the black rows are formed, and
                // the restriction below reads only black columns
                const int64_t lo = L.PHg32b.nrows > 0 ? L.cstart[1] : 0;
                k_resid_lat<<<grid_for(L.n - lo, 256 * LAT_RPT), 256, 0, s>>>(lo, L.n, lv, O::diag(L), b, x, scale,
                                                                              r, stop);
            }
        }
        if (!lat)
            k_resid<C, T><<<grid_for(L.n, 256), 256, 0, s>>>(L.n, O::A(L).view(), O::diag(L), b, x, scale, r, stop);
        restrict_black = lat && sizeof(T) == 4 && L.PHg32b.nrows > 0;
    }
    {
        ProfScope ps("restrict", 0, s);
        if constexpr (sizeof(T) == 4) {
            if (restrict_black) {
                spmv_g<C>(L.PHg32b, r, O::b(Lc), 0, stop, s);
            } else {
                spmv_g<C>(O::PHg(L), r, O::b(Lc), 0, stop, s);
            }
        } else {
            spmv_g<C>(O::PHg(L), r, O::b(Lc), 0, stop, s);
        }
    }
    vcycle<T>(p, l + 1, O::b(Lc), O::x(Lc), stop, s);
    {
        // x += P e_c.  The post-smoothing that follows relaxes colour 0 first, and a
        // Gauss-Seidel relaxation of a row does not read the row's own old value,
        // so the correction of colour-0 rows would be overwritten unread: only the
        // rows of the other colours are corrected (the same values, bit for bit)
        const int64_t lo = L.ncolors > 1 ? L.cstart[1] : 0;
        ProfScope ps("prolong", 0, s);
        k_spmv<C><<<grid_for(L.n - lo, 256), 256, 0, s>>>(lo, L.n, O::P(L).view(), O::x(Lc), x, 1, stop);
    }
    if (p->swept(l, sizeof(T) == 4))
        sweep_step<T>(p, l, b, x, false, nullptr, nullptr, stop, s);
    else
        smooth_finest<T>(p, b, x, false, stop, s);
    GL_LAUNCH_CHECK();
}

// ------------------------------------------------------------------ R_inf
// partial sums of ||x||_D^2 = sum_i |V_i| |x_i|^2 (fixed grid RED_BLOCKS x RED_THREADS)
__global__ void __launch_bounds__(RED_THREADS) k_dnorm2_part(int64_t n, const double2 *__restrict__ x,
                                                             const double *__restrict__ vol,
                                                             double *__restrict__ part, const int *stop) {
    if (stop && *stop) return;
    __shared__ double sh[RED_THREADS];
    double acc = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double2 a = x[i];
        acc += vol[i] * (a.x * a.x + a.y * a.y);
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int w = RED_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// sum of the RED_BLOCKS partial sums by one block of RED_THREADS (every thread gets it)
__device__ double sum_parts(const double *__restrict__ part) {
    __shared__ double sh[RED_THREADS];
    double acc = 0;
    for (int i = threadIdx.x; i < RED_BLOCKS; i += RED_THREADS) acc += part[i];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int w = RED_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    return sh[0];
}

__global__ void __launch_bounds__(RED_THREADS) k_rinf_begin(RinfDev *R, const double *__restrict__ part,
                                                            const int *stop) {
    if (stop && *stop) return;
    double v2 = sum_parts(part);
    if (threadIdx.x == 0) {
        R->v2 = v2;
        R->k = 0;
    }
}

// after a cycle: continue while ||r||_D^2 > tol^2 ||v||_D^2 and fewer than kmax
// cycles ran (a NaN stops the loop; MINRES reports it).  Always sets the
// condition, so the loop ends whatever the state.
__global__ void __launch_bounds__(RED_THREADS) k_rinf_decide(cudaGraphConditionalHandle h, RinfDev *R,
                                                             const double *__restrict__ part, const int *stop,
                                                             double tol2, int kmax) {
    const bool halted = stop && *stop;
    double r2 = 0;
    if (!halted) r2 = sum_parts(part);
    if (threadIdx.x == 0) {
        unsigned go = 0;
        if (!halted) {
            int k = R->k + 1;
            R->k = k;
            bool above = r2 > tol2 * R->v2;
            go = (above && k < kmax) ? 1u : 0u;
            if (!go) {
                R->cycles += (unsigned long long)k;
                R->applies += 1ull;
                if (above) R->hit_max = 1;
            }
        }
        cudaGraphSetConditional(h, go);
    }
}

// z = R_inf v on a capturing stream: the first cycle from z = 0, its residual
// and the decision, then a WHILE node whose body runs one more cycle, the
// correction, the residual and the decision.
static void rinf_enqueue(gl_prec_s *p, const double2 *v, double2 *z, const int *stop, cudaStream_t s) {
    using O = LevelOps<double>;
    Level &L = p->L[0];
    const int64_t n = L.n;
    double2 *r = p->cyc_r.get(), *e = p->cyc_e.get();
    RinfDev *R = p->rinf_dev.get();
    double *part = p->rinf_part.get();
    const double *vol = p->mesh->volp.get();
    const double tol2 = RINF_TOL * RINF_TOL;
    note_launch(5);
    k_dnorm2_part<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, v, vol, part, stop);
    k_rinf_begin<<<1, RED_THREADS, 0, s>>>(R, part, stop);
    vcycle<double>(p, 0, v, z, stop, s);
    k_resid<double2, double><<<grid_for(n, 256), 256, 0, s>>>(n, O::A(L).view(), O::diag(L), v, z, nullptr, r, stop);
    k_dnorm2_part<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, r, vol, part, stop);
    GL_LAUNCH_CHECK();
    cudaStreamCaptureStatus cst;
    cudaGraph_t cg = nullptr;
    const cudaGraphNode_t *deps = nullptr;
    size_t ndeps = 0;
    GL_CUDA(cudaStreamGetCaptureInfo(s, &cst, nullptr, &cg, &deps, nullptr, &ndeps));
    cudaGraphConditionalHandle h;
    GL_CUDA(cudaGraphConditionalHandleCreate(&h, cg, 0, cudaGraphCondAssignDefault));
    k_rinf_decide<<<1, RED_THREADS, 0, s>>>(h, R, part, stop, tol2, RINF_MAXCYC);
    GL_LAUNCH_CHECK();
    GL_CUDA(cudaStreamGetCaptureInfo(s, &cst, nullptr, &cg, &deps, nullptr, &ndeps));
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t wnode;
    GL_CUDA(cudaGraphAddNode(&wnode, cg, deps, nullptr, ndeps, &cp));
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    GL_CUDA(cudaStreamUpdateCaptureDependencies(s, &wnode, nullptr, 1, cudaStreamSetCaptureDependencies));
    cudaStream_t sb = p->rinf_body;
    GL_CUDA(cudaStreamBeginCaptureToGraph(sb, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    try {
        vcycle<double>(p, 0, r, e, stop, sb);
        note_launch(4);
        k_axpy_t<double2><<<grid_for(n, 256), 256, 0, sb>>>(n, e, z, stop);
        k_resid<double2, double><<<grid_for(n, 256), 256, 0, sb>>>(n, O::A(L).view(), O::diag(L), v, z, nullptr,
                                                                    r, stop);
        k_dnorm2_part<<<RED_BLOCKS, RED_THREADS, 0, sb>>>(n, r, vol, part, stop);
        k_rinf_decide<<<1, RED_THREADS, 0, sb>>>(h, R, part, stop, tol2, RINF_MAXCYC);
        GL_LAUNCH_CHECK();
    } catch (...) {
        cudaStreamEndCapture(sb, &body);
        throw;
    }
    GL_CUDA(cudaStreamEndCapture(sb, &body));
}

// R_inf on any stream: inserted into the graph being captured, or (outside
// capture) captured into a graph of its own and launched once.  No event nodes
// of the profiler go into the loop body.
static void rinf_apply(gl_prec_s *p, const double2 *v, double2 *z, const int *stop, cudaStream_t s) {
    Profiler &pr = profiler();
    const bool was_active = pr.active;
    pr.active = false;
    struct Restore {
        Profiler &pr;
        bool a;
        ~Restore() { pr.active = a; }
    } restore{pr, was_active};
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    GL_CUDA(cudaStreamIsCapturing(s, &st));
    if (st == cudaStreamCaptureStatusActive) {
        rinf_enqueue(p, v, z, stop, s);
        return;
    }
    cudaStream_t se = p->rinf_eager;
    GL_CUDA(cudaEventRecord(p->rinf_ev[0], s));
    GL_CUDA(cudaStreamWaitEvent(se, p->rinf_ev[0], 0));
    cudaGraph_t g = nullptr;
    GL_CUDA(cudaStreamBeginCapture(se, cudaStreamCaptureModeThreadLocal));
    try {
        rinf_enqueue(p, v, z, stop, se);
    } catch (...) {
        cudaStreamEndCapture(se, &g);
        if (g) cudaGraphDestroy(g);
        throw;
    }
    GL_CUDA(cudaStreamEndCapture(se, &g));
    cudaGraphExec_t ex = nullptr;
    cudaError_t ie = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    GL_CUDA(ie);
    cudaError_t le = cudaGraphLaunch(ex, se);
    cudaGraphExecDestroy(ex);  // released when the launch completes
    GL_CUDA(le);
    GL_CUDA(cudaEventRecord(p->rinf_ev[1], se));
    GL_CUDA(cudaStreamWaitEvent(s, p->rinf_ev[1], 0));
}

template <typename T>
static void precond_apply_t(gl_prec_s *p, const typename LevelOps<T>::C *v, typename LevelOps<T>::C *z,
                            const int *stop, cudaStream_t s) {
    using O = LevelOps<T>;
    using C = typename O::C;
    if (p->rinf) {
        if constexpr (sizeof(T) == 8) {
            rinf_apply(p, v, z, stop, s);
            return;
        } else {
            GL_REQUIRE(false, GL_ERR_ARG, "R_inf runs in FP64 only");
        }
    }
    if (p->cycles <= 1) {
        vcycle<T>(p, 0, v, z, stop, s);
    } else {
        // R_k: k steps of z <- z + V(v - (K + 2|psi|^2) z) from z = 0
        Level &L = p->L[0];
        C *r, *e;
        if constexpr (sizeof(T) == 8) {
            r = p->cyc_r.get();
            e = p->cyc_e.get();
        } else {
            r = p->cyc_r32.get();
            e = p->cyc_e32.get();
        }
        for (int k = 0; k < p->cycles; ++k) {
            if (k == 0) {
                vcycle<T>(p, 0, v, z, stop, s);
                continue;
            }
            note_launch(2);
            k_resid<C, T><<<grid_for(L.n, 256), 256, 0, s>>>(L.n, O::A(L).view(), O::diag(L), v, z, nullptr, r, stop);
            vcycle<T>(p, 0, r, e, stop, s);
            k_axpy_t<C><<<grid_for(L.n, 256), 256, 0, s>>>(L.n, e, z, stop);
        }
    }
    GL_LAUNCH_CHECK();
}

void precond_apply_p(gl_prec_s *p, const double2 *v, double2 *z, const int *stop, cudaStream_t s) {
    precond_apply_t<double>(p, v, z, stop, s);
}
void precond_apply_p32(gl_prec_s *p, const float2 *v, float2 *z, const int *stop, cudaStream_t s) {
    precond_apply_t<float>(p, v, z, stop, s);
}
void precond_apply_p64_via32(gl_prec_s *p, const double2 *v, double2 *z, const int *stop, cudaStream_t s) {
    int64_t n = p->mesh->n;
    note_launch(2);
    k_d2f2<<<grid_for(n, 256), 256, 0, s>>>(n, v, p->mp_in.get(), stop);
    precond_apply_t<float>(p, p->mp_in.get(), p->mp_out.get(), stop, s);
    k_f2d<<<grid_for(n, 256), 256, 0, s>>>(n, p->mp_out.get(), z, stop);
    GL_LAUNCH_CHECK();
}

}  // namespace gl
