// gl_solve.cu -- preconditioned MINRES (Paige & Saunders 1975) for the Newton
// system J(psi) x = b (Eq. Newton system) in the real inner product
// <x, y>_R = Re sum_i |V_i| conj(x_i) y_i (Eq. disc inner2), in which J is
// self-adjoint (Sec. 3) and R_k (Eq. prec2) is self-adjoint positive definite.
//
// The Lanczos/Givens scalars live on the device; every reduction writes one
// partial per block of a fixed grid and is summed in index order, so results do
// not depend on scheduling.  A device status word stops all kernels once the
// solve has converged or failed.  A solve is one CUDA graph that loops on the
// device (a WHILE conditional node over one iteration), so the host waits once;
// options.device_loop = 0 replays a body of six iterations from the host instead,
// reading the status word between replays.
//
// GL_MIXED: FP64 defect correction x <- x + e around inner MINRES solves of
// J e = r whose vectors, Jacobian applies and V-cycles are FP32 (dots and
// scalars FP64, coarsest solve FP64); the FP64 true residual decides.
#include <chrono>
#include <memory>

#include "gl_internal.cuh"
#include "gl_kernels.cuh"
#include "gl_profile.cuh"

namespace gl {

struct MinresDev {
    double gamma, eta, eta0, c, c_old, s, s_old, delta;
    double bnorm, tol, est, true_rel;
    double rho0;      // ||b - J x0||_D / ||b||_D: scales the recurrence's estimate to be relative to b
    // factors of the vector kernels, formed once by the scalar steps (an FP64 division a
    // thread kept the FP64 pipe for longer than a small vector's own work)
    double ig, dg, go;        // v_new = ig q - dg v - go v_old; ig = 1 / gamma
    double k2, k3;            // w_new = ig z - k3 w_old - k2 w; the direction is sig w
    double sig, sig_old;
    double tau;               // x += tau w_new
    double est_scale;         // rho0 / eta0
    double go_next, ig_next;  // go and ig of the next iteration
    int it, maxit, check_true, status, lucky, use_true, replays;
    unsigned done;    // blocks of the current reduction that have written their partials
    double stall;     // > 0: stop with ST_STALL once the estimate is below stall * tol while the true
                      // residual is still above tol (0: never)
};
enum { ST_RUN = 0, ST_CONV = 1, ST_BREAK = 2, ST_NAN = 3, ST_MAXIT = 4, ST_STALL = 5, ST_TIMEOUT = 6 };
static_assert(ST_TIMEOUT == STATUS_TIMEOUT, "the sweeps write STATUS_TIMEOUT into the status word");

template <typename T>
struct SolveOps;
template <>
struct SolveOps<double> {
    using C = double2;
    static SellView<C> K(const gl_mesh_s *m) { return m->K.view(); }
    static const double *kdiag(const gl_mesh_s *m) { return m->kdiag.get(); }
    static const double *vol(const gl_mesh_s *m) { return m->volp.get(); }
};
template <>
struct SolveOps<float> {
    using C = float2;
    static SellView<C> K(const gl_mesh_s *m) { return m->K32.view(); }
    static const float *kdiag(const gl_mesh_s *m) { return m->kdiag32.get(); }
    static const float *vol(const gl_mesh_s *m) { return m->volp32.get(); }
};

template <typename C>
__device__ __forceinline__ double redot(C a, C b) {  // Re(conj(a) b)
    return (double)a.x * (double)b.x + (double)a.y * (double)b.y;
}

// ------------------------------------------------------------------ scalar steps
// A reduction writes one partial per block of its fixed grid; the block that finishes
// last sums the partials in index order and takes the scalar step that follows, so a
// reduction and its scalars are one launch (a one-block kernel behind each reduction
// took 4 to 6 us, as long as a small system's vector kernels).
__device__ double sum_parts(const double *part, double *sh) {
    double a = 0;
    for (int i = threadIdx.x; i < RED_BLOCKS; i += blockDim.x) a += __ldcg(part + i);
    return block_sum(a, sh);
}
// true in every thread of the last block to get here (its partials are written)
__device__ bool last_block(MinresDev *S) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&S->done, 1u) == gridDim.x - 1;
        if (last) S->done = 0;
        __threadfence();
    }
    __syncthreads();
    return last;
}

// The WHILE node of a device-side MINRES loop; its condition is written by the last
// kernel of a loop body (use != 0).
struct LoopGate {
    cudaGraphConditionalHandle h;
    int use;
};
// end of a loop body: another one while the solve runs, at most maxit + 2 (then
// ST_MAXIT), so the loop ends whatever the state
__device__ void loop_next(MinresDev *S, const LoopGate &g) {
    if (!g.use) return;
    S->replays += 1;
    bool run = S->status == ST_RUN;
    if (run && S->replays >= S->maxit + 2) {
        S->status = ST_MAXIT;
        run = false;
    }
    cudaGraphSetConditional(g.h, run ? 1u : 0u);
}

// bb = <b, b>_R, vv = ||b - J x0||_D^2
__device__ void scal_init(MinresDev *S, double bb, double vv) {
    double tol = S->tol;
    int use_true = S->use_true;
    S->it = 0;
    S->replays = 0;
    S->status = ST_RUN;
    S->check_true = 0;
    S->lucky = 0;
    S->bnorm = sqrt(bb);
    S->true_rel = S->bnorm == 0 ? 0.0 : sqrt(vv) / S->bnorm;
    // the tolerance is relative to b, the recurrence's estimate to r0 = b - J x0:
    // scaled by ||r0||_D / ||b||_D (exactly 1 from x0 = 0)
    S->rho0 = S->true_rel;
    S->est = 1.0;
    if (isnan(bb)) {  // (before b = 0: a comparison with NaN is false)
        S->status = ST_NAN;
    } else if (S->bnorm == 0) {
        S->status = ST_CONV;
        S->est = 0;
    } else if (use_true && S->true_rel <= tol) {
        S->status = ST_CONV;
    } else if (!isfinite(S->true_rel)) {
        S->status = ST_NAN;
    } else if (S->maxit <= 0) {
        S->status = ST_MAXIT;
    }
}
// g2 = <v_1, z_1>_R
__device__ void scal_gamma0(MinresDev *S, double g2) {
    if (!isfinite(g2)) {
        S->status = ST_NAN;
        return;
    }
    if (g2 < 0) {
        S->status = ST_BREAK;
        return;
    }
    double g = sqrt(g2);
    S->gamma = g;
    S->ig_next = 1.0 / g;
    S->go_next = g;  // v_0 = 0, with gamma_0 = 1
    S->sig = S->sig_old = 1.0;
    S->eta = S->eta0 = g;
    S->est_scale = S->rho0 / g;
    S->c = S->c_old = 1.0;
    S->s = S->s_old = 0.0;
    if (g == 0) S->status = ST_CONV;
}
// d = <J z, z>_R
__device__ void scal_delta(MinresDev *S, double d) {
    const double ig = S->ig_next, g = S->gamma;
    S->ig = ig;
    S->go = S->go_next;
    d = d * ig * ig;
    S->delta = d;
    S->dg = d * ig;
    S->k3 = S->s_old * g * S->sig_old;
    S->k2 = (S->s * d + S->c_old * S->c * g) * S->sig;
}
// g2 = <v_new, z_new>_R.  One thread takes the step, so its dependent FP64 divisions and
// square roots are what it costs: two roots and two reciprocals, one of them in another
// warp (`other`), where a division per scalar took 3 us more.
__device__ void scal_givens(MinresDev *S, double g2, bool other) {
    const double gn = sqrt(g2);
    if (other) {  // the next iteration's own factors (unused unless it runs)
        S->go_next = gn * S->ig;
        S->ig_next = 1.0 / gn;
        return;
    }
    if (!isfinite(g2) || !isfinite(S->delta)) {
        S->status = ST_NAN;
        return;
    }
    if (g2 < 0) {
        S->status = ST_BREAK;
        return;
    }
    const double a0 = S->c * S->delta - S->c_old * S->s * S->gamma;
    const double a1 = sqrt(a0 * a0 + gn * gn);
    const double ia1 = 1.0 / a1, cn = a0 * ia1, sn = gn * ia1;
    S->sig_old = S->sig;
    S->sig = ia1;
    S->tau = cn * S->eta * ia1;
    S->eta = -sn * S->eta;
    S->gamma = gn;
    S->c_old = S->c;
    S->c = cn;
    S->s_old = S->s;
    S->s = sn;
    S->it += 1;
    S->est = S->est_scale * fabs(S->eta);
    S->lucky = (gn == 0);
    S->check_true = (S->est <= S->tol) || S->lucky;
}
// the end of an iteration; r2 = ||b - J x||_D^2 when a check was asked for
__device__ void scal_true(MinresDev *S, double r2) {
    if (S->check_true) {
        if (S->use_true) {
            S->true_rel = sqrt(r2) / S->bnorm;
            if (!isfinite(S->true_rel))
                S->status = ST_NAN;
            else if (S->true_rel <= S->tol)
                S->status = ST_CONV;
            else if (S->stall > 0 && S->est <= S->stall * S->tol)
                S->status = ST_STALL;  // the recurrence has run far past what the true residual shows
        } else {
            S->status = ST_CONV;  // inner solves stop on the estimate alone
        }
        if (!S->status && S->lucky) S->status = ST_MAXIT;  // Krylov space exhausted above tol
    }
    if (!S->status && S->it >= S->maxit) S->status = ST_MAXIT;
}

// ------------------------------------------------------------------ vector kernels
// v = b - J x ; <b, b>_R and <v, v>_R
template <typename C, typename R>
__global__ void __launch_bounds__(RED_THREADS) k_init_resid(int64_t n, SellView<C> K, const R *kd, const R *vol,
                                                            const C *psi, const C *b, const C *x, C *v,
                                                            double *part, MinresDev *S) {
    __shared__ double sh[32];
    double ab = 0, av = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        C acc = sell_row<C, C>(K, p, x);
        C jx = jacobian_epilogue(acc, kd[p], psi[p], x[p]);
        C bb = b[p];
        C vv = csub(bb, jx);
        v[p] = vv;
        ab += (double)vol[p] * redot(bb, bb);
        av += (double)vol[p] * redot(vv, vv);
    }
    double t = block_sum(ab, sh);
    double u = block_sum(av, sh);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = t;
        part[RED_BLOCKS + blockIdx.x] = u;
    }
    if (!last_block(S)) return;
    const double bb = sum_parts(part, sh), vv = sum_parts(part + RED_BLOCKS, sh);
    if (threadIdx.x == 0) scal_init(S, bb, vv);
}

// <v, z>_R and the scalar step behind it: gamma_1 with v = v0, or (givens) Givens with
// the vector that k_step wrote, v1 and v0 in turn.  z may be the FP32 vector of a
// mixed-precision solve, whose FP64 image it stands for.
template <typename C, typename R, typename Y>
__global__ void __launch_bounds__(RED_THREADS) k_dot(int64_t n, const R *vol, const C *v0, const C *v1, const Y *y,
                                                     double *part, MinresDev *S, int givens) {
    __shared__ double sh[32];
    if (S->status) return;
    const C *x = givens && !(S->it & 1) ? v1 : v0;
    double a = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    auto term = [](R w, C u, Y v) { return (double)w * ((double)u.x * (double)v.x + (double)u.y * (double)v.y); };
    // four rows per step, every load issued before the first use
    for (; p + 3 * stride < n; p += 4 * stride) {
        C u[4];
        Y v[4];
        R w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            u[k] = x[p + k * stride];
            v[k] = y[p + k * stride];
            w[k] = vol[p + k * stride];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) a += term(w[k], u[k], v[k]);
    }
    for (; p < n; p += stride) a += term(vol[p], x[p], y[p]);
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
    if (!last_block(S)) return;
    double g2 = sum_parts(part, sh);
    if (threadIdx.x == 0) sh[0] = g2;
    __syncthreads();
    g2 = sh[0];
    if (threadIdx.x != 0 && threadIdx.x != 32) return;
    if (givens)
        scal_givens(S, g2, threadIdx.x == 32);
    else if (threadIdx.x == 0)
        scal_gamma0(S, g2);
}

// q = J z (z not yet normalised) ; <J z, z>_R and delta.  Z: float2 when z is the FP32
// V-cycle's output in a mixed-precision solve.
template <typename C, typename R, typename Z>
__global__ void __launch_bounds__(RED_THREADS) k_jz(int64_t n, SellView<C> K, const R *kd, const R *vol, const C *psi,
                                                    const Z *z, C *q, double *part, MinresDev *S) {
    __shared__ double sh[32];
    if (S->status) return;
    double a = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        C acc = sell_row<C, Z>(K, p, z);
        const Z zp = z[p];
        C zz = mk((R)zp.x, (R)zp.y);
        C jz = jacobian_epilogue(acc, kd[p], psi[p], zz);
        q[p] = jz;
        a += (double)vol[p] * redot(jz, zz);
    }
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
    if (!last_block(S)) return;
    const double d = sum_parts(part, sh);
    if (threadIdx.x == 0) scal_delta(S, d);
}

// the same from the FP64 lattice tables (the matrix-free stencil of a lattice mesh)
template <typename Z>
__global__ void __launch_bounds__(RED_THREADS) k_jz_lat64(int64_t n, LatticeView64 L, const double *kd,
                                                          const double2 *psi, const Z *z, double2 *q,
                                                          double *part, MinresDev *S) {
    __shared__ double sh[32];
    if (S->status) return;
    double a = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const double2 acc = lattice_row64(L, p, z);
        const Z zp = z[p];
        const double2 zz = make_double2(zp.x, zp.y);
        const double2 jz = jacobian_epilogue(acc, kd[p], psi[p], zz);
        q[p] = jz;
        a += L.vol[p] * redot(jz, zz);
    }
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
    if (!last_block(S)) return;
    const double d = sum_parts(part, sh);
    if (threadIdx.x == 0) scal_delta(S, d);
}

// ------------------------------------------------------------------ double-float Jacobian apply
// In the mixed-precision solve (FP64 MINRES, FP32 V-cycle) every z that meets
// the Jacobian is the FP64 image of the V-cycle's FP32 output, so its FP32 copy
// is exact.  On even-N lattices J z is then formed with FP32 arithmetic only
// (far faster than FP64 on this GPU) from double-float data (hi + lo):
//   (J z)_i = 2^b_i sum_k a_ik (z_i - u_ik z_k) + (r_i - 1 + 2|psi_i|^2) z_i + psi_i^2 conj(z_i)
// with a = |K-hat| / h^d and the unit phase u = exp(-i theta) tabulated per axis
// (gl_lattice.cu), K_ik = -2^b_i a_ik u_ik (|V_i| = h^d 2^-b_i, b_i boundary
// coordinates: an exact power-of-2 factor) and r_i = K_ii - sum_k |K_ik|.  The
// differences z_i - u z_k are formed with Knuth's error-free TwoSum after an
// FMA-based TwoProd, so a smooth z cancels without error, and products and sums
// accumulate in the compensated form of Ogita, Rump and Oishi's Dot2 (an FP32
// running sum and an FP32 compensation collecting the exact rounding errors):
// about 48 significant bits, against 53 in FP64.  The solve watches for the
// consequence (see scal_true) and finishes with the FP64 apply if it stalls.
// per-solve coefficients of the local part: d = r - 1 + 2|psi|^2 and psi^2
__global__ void k_jz_coef(int64_t n, const double *__restrict__ rem, const double2 *__restrict__ psi,
                          float2 *__restrict__ d, float4 *__restrict__ p2) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 ps = psi[i];
    d[i] = split_df(rem[i] - 1.0 + 2.0 * (ps.x * ps.x + ps.y * ps.y));
    float2 re = split_df(ps.x * ps.x - ps.y * ps.y), im = split_df(2.0 * ps.x * ps.y);
    p2[i] = make_float4(re.x, re.y, im.x, im.y);
}

// q = J z from the FP32 V-cycle output z; <J z, z>_R and delta (S null: q alone)
__global__ void __launch_bounds__(RED_THREADS) k_jz_latdf(int64_t n, LatticeDfView L, double hd,
                                                          const float2 *__restrict__ d, const float4 *__restrict__ p2,
                                                          const float2 *__restrict__ z, double2 *__restrict__ q,
                                                          double *part, MinresDev *S) {
    __shared__ double sh[32];
    if (S && S->status) return;
    float as = 0.f, ac = 0.f;
    const uint32_t N = (uint32_t)L.N;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = p >= L.nred ? 1u : 0u;
        uint32_t v = 2u * (uint32_t)(p - (c ? L.nred : 0));
        const uint32_t r = L.dN.div(v), k = L.dN.div(r);
        uint32_t i = v - r * N;
        const uint32_t j = r - k * N;
        if (((i + j + k) & 1u) != c) {
            ++v;
            ++i;
        }
        const int64_t other = c ? 0 : L.nred;
        const int b = (i == 0 || i == N - 1) + (j == 0 || j == N - 1) + (L.dim == 3 && (k == 0 || k == N - 1));
        const float2 zp = z[p];
        float rs = 0.f, rc = 0.f, is = 0.f, ic = 0.f;
        // + a (z_p - u z_u) for the edge to node u; conj: the -e edge
        auto edge = [&](int64_t idx, uint32_t u, bool conj) {
            const float2 a = L.a[idx];
            const float4 t = L.u[idx];
            const float2 ur = make_float2(t.x, t.y);
            const float2 ui = conj ? make_float2(-t.z, -t.w) : make_float2(t.z, t.w);
            const float2 zu = z[(int64_t)(u >> 1) + other];
            float ws = 0.f, wc = 0.f, vs = 0.f, vc = 0.f;
            dot2_df(ws, wc, ur, zu.x);
            dot2_df(ws, wc, ui, -zu.y);
            dot2_df(vs, vc, ur, zu.y);
            dot2_df(vs, vc, ui, zu.x);
            float tr = zp.x, er = 0.f, ti = zp.y, ei = 0.f;
            dot2_add(tr, er, -ws);
            er = __fadd_rn(er, -wc);
            dot2_add(ti, ei, -vs);
            ei = __fadd_rn(ei, -vc);
            dot2_df(rs, rc, a, tr);
            rc = __fmaf_rn(a.x, er, rc);
            dot2_df(is, ic, a, ti);
            ic = __fmaf_rn(a.x, ei, ic);
        };
        {
            const int64_t idx = j + (int64_t)N * k;
            if (i + 1 < N) edge(idx, v + 1, false);
            if (i > 0) edge(idx, v - 1, true);
        }
        {
            const int64_t idx = L.per_axis + i + (int64_t)N * k;
            if (j + 1 < N) edge(idx, v + N, false);
            if (j > 0) edge(idx, v - N, true);
        }
        if (L.dim == 3) {
            const int64_t idx = 2 * L.per_axis + i + (int64_t)N * j;
            if (k + 1 < N) edge(idx, v + N * N, false);
            if (k > 0) edge(idx, v - N * N, true);
        }
        // row scale 2^b (exact), then + d z + psi^2 conj(z)
        const float sb = (float)(1 << b);
        rs *= sb;
        rc *= sb;
        is *= sb;
        ic *= sb;
        const float2 dd = d[p];
        const float4 pp = p2[p];
        const float2 pr = make_float2(pp.x, pp.y), pi = make_float2(pp.z, pp.w);
        dot2_df(rs, rc, dd, zp.x);
        dot2_df(rs, rc, pr, zp.x);
        dot2_df(rs, rc, pi, zp.y);
        dot2_df(is, ic, dd, zp.y);
        dot2_df(is, ic, pi, zp.x);
        dot2_df(is, ic, pr, -zp.y);
        q[p] = make_double2((double)rs + (double)rc, (double)is + (double)ic);
        // |V_p| Re(conj(q_p) z_p) / h^d = 2^-b Re(conj(q_p) z_p)
        float ts = 0.f, tc = 0.f;
        dot2_df(ts, tc, make_float2(rs, rc), zp.x);
        dot2_df(ts, tc, make_float2(is, ic), zp.y);
        const float isb = 1.f / sb;
        dot2_add(as, ac, ts * isb);
        ac = __fadd_rn(ac, tc * isb);
    }
    if (!S) return;  // an apply outside a solve
    double t = block_sum(((double)as + (double)ac) * hd, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
    if (!last_block(S)) return;
    const double delta = sum_parts(part, sh);
    if (threadIdx.x == 0) scal_delta(S, delta);
}

__global__ void k_round32(int64_t n, const double2 *a, float2 *b) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) b[p] = to32(a[p]);
}

// y = J(psi) phi by the double-float lattice kernel the GL_MIXED_PRECOND solve
// runs, for phi rounded to FP32 (in the solve that rounding is exact); solve
// ordering, synchronises s
void jacobian_apply_pdf(gl_mesh_s *m, const double2 *psi, const double2 *phi, double2 *y, cudaStream_t s) {
    mesh_ensure_fp32(m, s);
    GL_REQUIRE(m->lat_ok, GL_ERR_ARG,
               "the double-FP32 Jacobian needs a mesh with an even number of nodes per side (checked lattice stencil)");
    const int64_t n = m->n;
    DBuf<float2> d(n), z(n);
    DBuf<float4> p2(n);
    const int G = grid_for(n, 256);
    note_launch(3);
    k_jz_coef<<<G, 256, 0, s>>>(n, m->lat_krem.get(), psi, d.get(), p2.get());
    k_round32<<<G, 256, 0, s>>>(n, phi, z.get());
    k_jz_latdf<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, lattice_df_view(m), m->lat_hd, d.get(), p2.get(), z.get(), y,
                                                  nullptr, nullptr);
    GL_LAUNCH_CHECK();
    GL_CUDA(cudaStreamSynchronize(s));
}

// The two recurrences that follow the Jacobian:
//   v_new = q / gamma - (delta / gamma) v - (gamma / gamma_old) v_old
//   w_new = z / gamma - a3 w_old - a2 w
// (w_new without its factor 1 / a1, which the next scalar step knows and hands on as
// sig), each written over its oldest vector; the two vectors of a pair change roles
// with the iteration's parity, so one captured iteration serves all.  in: the V-cycle's
// input, v_new as it is or (float2) rounded; Z: float2 when z is the FP32 V-cycle's
// output.  Four rows per step with every load issued first.
template <typename C, typename R, typename Z>
__global__ void __launch_bounds__(RED_THREADS) k_step(int64_t n, const MinresDev *S, const C *q, C *v0, C *v1, C *w0,
                                                      C *w1, const Z *z, Z *in) {
    if (S->status) return;
    const R ig = (R)S->ig, dg = (R)S->dg, go = (R)S->go, k2 = (R)S->k2, k3 = (R)S->k3;
    const bool odd = S->it & 1;
    C *v = odd ? v1 : v0, *vo = odd ? v0 : v1, *w = odd ? w1 : w0, *wo = odd ? w0 : w1;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    auto put = [&](int64_t i, C a, C b, C c, Z zz, C ww, C wv) {
        const C r = mk(a.x * ig - dg * b.x - go * c.x, a.y * ig - dg * b.y - go * c.y);
        vo[i] = r;
        Z o;
        o.x = r.x;
        o.y = r.y;
        in[i] = o;
        wo[i] = mk((R)zz.x * ig - k3 * wv.x - k2 * ww.x, (R)zz.y * ig - k3 * wv.y - k2 * ww.y);
    };
    for (; p + stride < n; p += 2 * stride) {
        C a[2], b[2], c[2], d[2], e[2];
        Z f[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            a[u] = q[p + u * stride];
            b[u] = v[p + u * stride];
            c[u] = vo[p + u * stride];
            f[u] = z[p + u * stride];
            d[u] = w[p + u * stride];
            e[u] = wo[p + u * stride];
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) put(p + u * stride, a[u], b[u], c[u], f[u], d[u], e[u]);
    }
    if (p < n) put(p, q[p], v[p], vo[p], z[p], w[p], wo[p]);
}

// x += tau w_new (the vector that k_step wrote; the Givens step has counted the iteration)
template <typename C, typename R>
__global__ void __launch_bounds__(RED_THREADS) k_update(int64_t n, const MinresDev *S, const C *w0, const C *w1, C *x) {
    if (S->status) return;
    const R tau = (R)S->tau;
    const C *w = S->it & 1 ? w1 : w0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (; p + 3 * stride < n; p += 4 * stride) {
        C ww[4], xx[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            ww[u] = w[p + u * stride];
            xx[u] = x[p + u * stride];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) x[p + u * stride] = mk(xx[u].x + tau * ww[u].x, xx[u].y + tau * ww[u].y);
    }
    for (; p < n; p += stride) x[p] = mk(x[p].x + tau * w[p].x, x[p].y + tau * w[p].y);
}

// ||b - J x||_D^2 when the Givens step asked for a check, and the end of the iteration;
// with `final` the true residual of the solve's result, whatever the status
template <typename C, typename R>
__global__ void __launch_bounds__(RED_THREADS) k_true_resid(int64_t n, SellView<C> K, const R *kd, const R *vol,
                                                            const C *psi, const C *b, const C *x, double *part,
                                                            MinresDev *S, LoopGate g, int final) {
    __shared__ double sh[32];
    if (!final && (S->status || !S->check_true)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            if (!S->status) scal_true(S, 0.0);
            loop_next(S, g);
        }
        return;
    }
    double a = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        C acc = sell_row<C, C>(K, p, x);
        C jx = jacobian_epilogue(acc, kd[p], psi[p], x[p]);
        C r = csub(b[p], jx);
        a += (double)vol[p] * redot(r, r);
    }
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
    if (!last_block(S)) return;
    const double r2 = sum_parts(part, sh);
    if (threadIdx.x) return;
    if (final) {
        if (S->bnorm != 0) S->true_rel = sqrt(r2) / S->bnorm;
        return;
    }
    scal_true(S, r2);
    loop_next(S, g);
}

// solve parameters, written before the captured init phase reads them
__global__ void k_set_params(MinresDev *S, double tol, int maxit, int use_true, double stall) {
    S->tol = tol;
    S->maxit = maxit;
    S->use_true = use_true;
    S->stall = stall;
    S->done = 0;
}

__global__ void k_loop_begin(cudaGraphConditionalHandle h, const MinresDev *S) {
    cudaGraphSetConditional(h, S->status == ST_RUN ? 1u : 0u);
}

// ------------------------------------------------------------------ MINRES driver
// A solve is the initial phase and a WHILE node over one iteration, captured once per
// (state, right-hand side, solution, preconditioner): the vectors of the recurrences
// change roles by the iteration's parity on the device, so the body is one iteration
// and the loop stops where the solve does.  (Six iterations in IF nodes, which the
// rotation of the buffers needed before, took 0.29 ms more to capture and instantiate
// for every new state.)  For profilers the host replays a body of ITER_UNROLL
// iterations instead; kernels behind the end of the solve return at once.
constexpr int ITER_UNROLL = 6;

struct Graph {
    cudaGraphExec_t exec = nullptr;
    std::vector<int> slots;  // profiler event slots recorded inside the graph
    int64_t launches = 0;
    void reset() {
        if (exec) cudaGraphExecDestroy(exec);
        exec = nullptr;
        slots.clear();
        launches = 0;
    }
};

struct GraphKey {
    const void *psi = nullptr, *b = nullptr, *x = nullptr;
    int64_t mesh_uid = -1, prec_uid = -1, generation = -1, mesh_version = -1;
    int vc32 = 0, df = 0, loop = 0;
    bool operator==(const GraphKey &o) const {
        return psi == o.psi && b == o.b && x == o.x && mesh_uid == o.mesh_uid && prec_uid == o.prec_uid &&
               generation == o.generation && mesh_version == o.mesh_version && vc32 == o.vc32 && df == o.df &&
               loop == o.loop;
    }
};

template <typename T>
struct MinresWork {
    using C = cplx_t<T>;
    DBuf<C> v[2], w[2], q;
    DBuf<C> z, in;     // the V-cycle's output and input (FP32 V-cycles have the next two)
    DBuf<float2> z32;
    DBuf<float2> jd;      // double-float Jacobian coefficients (mixed-precision solve)
    DBuf<float4> jp2;
    DBuf<double> part;
    DBuf<MinresDev> S;
    int64_t n = 0;
    cudaStream_t cap = nullptr, cap_body = nullptr;
    GraphKey key;
    Graph init, body;
    // the device-side loop: the whole solve in one graph; launches of its initial
    // phase and of one iteration (counted at capture)
    Graph loop;
    int64_t loop_init_launches = 0, loop_iter_launches = 0;
    void ensure(int64_t nn, bool vc32) {
        if (!cap) GL_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
        if (!cap_body) GL_CUDA(cudaStreamCreateWithFlags(&cap_body, cudaStreamNonBlocking));
        if (n != nn) {
            init.reset();
            body.reset();
            loop.reset();
            key = GraphKey{};
            for (auto &b : v) b.alloc(nn);
            z.release();
            in.release();
            z32.release();
            for (auto &b : w) b.alloc(nn);
            q.alloc(nn);
            part.alloc(2 * RED_BLOCKS);
            S.alloc(1);
            jd.release();
            jp2.release();
            n = nn;
        }
        if (vc32) {
            z32.reserve(nn);
        } else {
            z.reserve(nn);
            in.reserve(nn);
        }
    }
    void ensure_df() {
        if (jd.n != (size_t)n) {
            jd.alloc(n);
            jp2.alloc(n);
        }
    }
};

struct MinresResult {
    int status, iters;
    double est, true_rel;
};

template <typename T>
static void precond_apply_any(gl_prec_s *p, const cplx_t<T> *v, cplx_t<T> *z, const int *stop, cudaStream_t s);
template <>
void precond_apply_any<double>(gl_prec_s *p, const double2 *v, double2 *z, const int *stop, cudaStream_t s) {
    precond_apply_p(p, v, z, stop, s);
}
template <>
void precond_apply_any<float>(gl_prec_s *p, const float2 *v, float2 *z, const int *stop, cudaStream_t s) {
    precond_apply_p32(p, v, z, stop, s);
}

// b = 0 has the solution x = 0 whatever the initial guess
template <typename C>
__global__ void k_zero_if_bzero(int64_t n, const MinresDev *S, C *x) {
    if (S->bnorm != 0) return;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) x[i] = mk(decltype(x[0].x)(0), decltype(x[0].x)(0));
}

template <typename C>
__global__ void k_copy_if(int64_t n, const C *a, C *b, const int *stop) {
    if (*stop) return;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = a[i];
}

// captures whatever `enqueue` launches on a private stream into g
template <typename F>
static void capture(Graph &g, cudaStream_t cs, F &&enqueue) {
    g.reset();
    Profiler &pr = profiler();
    int64_t l0 = pr.launches.load();
    pr.capture = &g.slots;
    cudaGraph_t graph = nullptr;
    GL_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    try {
        enqueue(cs);
    } catch (...) {
        cudaStreamEndCapture(cs, &graph);
        if (graph) cudaGraphDestroy(graph);
        pr.capture = nullptr;
        throw;
    }
    GL_CUDA(cudaStreamEndCapture(cs, &graph));
    pr.capture = nullptr;
    g.launches = pr.launches.load() - l0;
    pr.launches.fetch_sub(g.launches);
    GL_CUDA(cudaGraphInstantiate(&g.exec, graph, 0));
    GL_CUDA(cudaGraphDestroy(graph));
}

static void replay(Graph &g, cudaStream_t s) {
    GL_CUDA(cudaGraphLaunch(g.exec, s));
    note_launch((int)g.launches);
}
static void harvest(Graph &g) {
    Profiler &pr = profiler();
    if (pr.active) pr.harvest(g.slots);
    pr.harvest_direct();
}

// Enqueues the initial phase of MINRES (v_1 = b - J x_0, z_1 = R v_1,
// gamma_1) on `cs`; the parameters tol/maxit/use_true are read from S.
template <typename T>
static void enqueue_init(gl_mesh_s *m, gl_prec_s *p, const cplx_t<T> *psi, const cplx_t<T> *b, cplx_t<T> *x,
                         bool vc32, bool df, MinresWork<T> &W, cudaStream_t cs) {
    using O = SolveOps<T>;
    using C = cplx_t<T>;
    int64_t n = m->n;
    MinresDev *S = W.S.get();
    const int *stop = &S->status;
    double *part = W.part.get();
    int G = grid_for(n, 256);
    C *v = W.v[0].get();
    GL_CUDA(cudaMemsetAsync(W.v[1].get(), 0, n * sizeof(C), cs));
    for (auto &w : W.w) GL_CUDA(cudaMemsetAsync(w.get(), 0, n * sizeof(C), cs));
    if constexpr (std::is_same<T, double>::value) {
        if (df) {
            note_launch();
            k_jz_coef<<<G, 256, 0, cs>>>(n, m->lat_krem.get(), psi, W.jd.get(), W.jp2.get());
        }
    }
    note_launch(2);
    k_init_resid<C, T><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, O::K(m), O::kdiag(m), O::vol(m), psi, b, x, v, part, S);
    k_zero_if_bzero<C><<<G, 256, 0, cs>>>(n, S, x);
    GL_LAUNCH_CHECK();
    if constexpr (std::is_same<T, double>::value) {
        if (vc32 && p) {
            note_launch(2);
            k_round32<<<G, 256, 0, cs>>>(n, v, p->mp_in.get());
            precond_apply_p32(p, p->mp_in.get(), W.z32.get(), stop, cs);
            k_dot<C, T, float2><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, O::vol(m), v, v, W.z32.get(), part, S, 0);
            GL_LAUNCH_CHECK();
            return;
        }
    }
    if (p) {
        precond_apply_any<T>(p, v, W.z.get(), stop, cs);
    } else {
        note_launch();
        k_copy_if<C><<<G, 256, 0, cs>>>(n, v, W.z.get(), stop);
    }
    note_launch();
    k_dot<C, T, C><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, O::vol(m), v, v, W.z.get(), part, S, 0);
    GL_LAUNCH_CHECK();
}

// Enqueues one MINRES iteration on `cs`; with `gate` it ends a loop body.
template <typename T>
static void enqueue_iteration(gl_mesh_s *m, gl_prec_s *p, const cplx_t<T> *psi, const cplx_t<T> *b, cplx_t<T> *x,
                              bool vc32, bool df, MinresWork<T> &W, cudaStream_t cs,
                              const LoopGate &gate = LoopGate{{}, 0}) {
    using O = SolveOps<T>;
    using C = cplx_t<T>;
    int64_t n = m->n;
    MinresDev *S = W.S.get();
    const int *stop = &S->status;
    double *part = W.part.get();
    auto K = O::K(m);
    auto kd = O::kdiag(m);
    auto vol = O::vol(m);
    C *v0 = W.v[0].get(), *v1 = W.v[1].get(), *w0 = W.w[0].get(), *w1 = W.w[1].get();
    C *q = W.q.get(), *z = W.z.get();
    float2 *y = W.z32.get();  // z around an FP32 V-cycle
    bool mp = false;          // FP64 vectors around an FP32 V-cycle
    if constexpr (std::is_same<T, double>::value) mp = vc32 && p;
    {
        // algorithmic bytes of the fused Jacobian + dot: off-diagonals, K_ii,
        // |V|, psi, z (own row; neighbours cached) and the written q
        int64_t nnz = (sizeof(T) == 8) ? m->K.nnz_real : m->K32.nnz_real;
        bool done = false;
        if constexpr (std::is_same<T, double>::value) {
            if (df) {
                // z (8 B), d and psi^2 (24 B) and the written q (16 B) per row; the
                // neighbours' z and the tables from cache
                // FP32 operations of the error-free transformations, counted from the
                // kernel: about 84 per stored neighbour and 100 per row, as flop
                // equivalents (2 per operation: each takes an FMA issue slot)
                ProfScope ps("jz", (double)n * (8 + 24 + 16), cs,
                             2.0 * (84.0 * (double)m->K.nnz_real + 100.0 * (double)n));
                k_jz_latdf<<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, lattice_df_view(m), m->lat_hd, W.jd.get(),
                                                               W.jp2.get(), y, q, part, S);
                done = true;
            } else if (m->lat64_ok && p && p->lattice64) {
                // own z, K_ii, |V|, psi and the written q per row (48 + 16 B); the
                // neighbours' z and the tables from cache; per row the six
                // complex FMAs, the 1 / |V| scaling, the local terms and the dot
                ProfScope ps("jz", (double)n * (3 * sizeof(C) + 2 * sizeof(T)), cs,
                             8.0 * (double)nnz + 28.0 * (double)n);
                if (mp)
                    k_jz_lat64<<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, lattice_view64(m), kd, psi, y, q, part, S);
                else
                    k_jz_lat64<<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, lattice_view64(m), kd, psi, z, q, part, S);
                done = true;
            }
        }
        if (!done) {
            double jb = (double)nnz * (sizeof(C) + 4) + (double)n * (2 * sizeof(T) + 3 * sizeof(C));
            // a complex FMA (8 flops) per stored entry; per row the local terms (13)
            // and the dot (5)
            ProfScope ps("jz", jb, cs, 8.0 * (double)nnz + 18.0 * (double)n);
            if constexpr (std::is_same<T, double>::value) {
                if (mp) k_jz<C, T, float2><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, K, kd, vol, psi, y, q, part, S);
            }
            if (!mp) k_jz<C, T, C><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, K, kd, vol, psi, z, q, part, S);
        }
    }
    note_launch(4);
    if constexpr (std::is_same<T, double>::value) {
        if (mp) {
            k_step<C, T, float2><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, S, q, v0, v1, w0, w1, y, p->mp_in.get());
            precond_apply_p32(p, p->mp_in.get(), y, stop, cs);
            k_dot<C, T, float2><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, vol, v0, v1, y, part, S, 1);
        }
    }
    if (!mp) {
        // without a preconditioner z = v
        C *in = p ? W.in.get() : z;
        k_step<C, T, C><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, S, q, v0, v1, w0, w1, z, in);
        if (p) precond_apply_any<T>(p, in, z, stop, cs);
        k_dot<C, T, C><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, vol, v0, v1, z, part, S, 1);
    }
    k_update<C, T><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, S, w0, w1, x);
    k_true_resid<C, T><<<RED_BLOCKS, RED_THREADS, 0, cs>>>(n, K, kd, vol, psi, b, x, part, S, gate, 0);
    GL_LAUNCH_CHECK();
}

// Adds a WHILE node over `body` behind what `cs` has captured; `body` enqueues one
// iteration on the stream it is given, ending with the gate.
template <typename F>
static void enqueue_loop(cudaStream_t cs, cudaStream_t body_stream, MinresDev *S, F &&body) {
    cudaStreamCaptureStatus cst;
    cudaGraph_t cg = nullptr;
    const cudaGraphNode_t *deps = nullptr;
    size_t ndeps = 0;
    GL_CUDA(cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cg, &deps, nullptr, &ndeps));
    LoopGate gate{{}, 1};
    GL_CUDA(cudaGraphConditionalHandleCreate(&gate.h, cg, 0, cudaGraphCondAssignDefault));
    k_loop_begin<<<1, 1, 0, cs>>>(gate.h, S);
    GL_LAUNCH_CHECK();
    GL_CUDA(cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cg, &deps, nullptr, &ndeps));
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = gate.h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t wnode;
    GL_CUDA(cudaGraphAddNode(&wnode, cg, deps, nullptr, ndeps, &cp));
    cudaGraph_t graph = cp.conditional.phGraph_out[0];
    GL_CUDA(cudaStreamUpdateCaptureDependencies(cs, &wnode, nullptr, 1, cudaStreamSetCaptureDependencies));
    GL_CUDA(cudaStreamBeginCaptureToGraph(body_stream, graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    try {
        body(body_stream, gate);
    } catch (...) {
        cudaStreamEndCapture(body_stream, &graph);
        throw;
    }
    GL_CUDA(cudaStreamEndCapture(body_stream, &graph));
}

// Runs MINRES on J x = b with x as the initial guess (overwritten).  use_true:
// stop on the FP64 true residual (FP64 path) or on the estimate alone (inner).
template <typename T>
static MinresResult minres(gl_mesh_s *m, gl_prec_s *p, const cplx_t<T> *psi, const cplx_t<T> *b, cplx_t<T> *x,
                           double tol, int maxit, bool use_true, bool vc32, MinresWork<T> &W, cudaStream_t s,
                           bool df = false, bool device_loop = true) {
    using O = SolveOps<T>;
    using C = cplx_t<T>;
    int64_t n = m->n;
    W.ensure(n, std::is_same<T, double>::value && vc32 && p);
    if (df) W.ensure_df();
    MinresDev *S = W.S.get();
    double *part = W.part.get();
    // The device-side loop (the whole solve in one graph: the initial phase, then a
    // WHILE node over one iteration) whenever no kernel class is being timed (the
    // profiler's event nodes cannot sit in conditional bodies) and R_inf does not nest
    // its own loop.
    const bool timing_class = profiler().active && !profiler().name.empty();
    const bool loop = device_loop && !timing_class && !(p && p->rinf);
    GraphKey key{psi, b, x, m->uid, p ? p->uid : -1, profiler().generation, m->version, vc32 ? 1 : 0, df ? 1 : 0,
                 loop ? 1 : 0};
    if (!(key == W.key) || (loop ? !W.loop.exec : (!W.init.exec || !W.body.exec))) {
        W.key = key;
        if (loop) {
            capture(W.loop, W.cap, [&](cudaStream_t cs) {
                Profiler &pr = profiler();
                const int64_t l0 = pr.launches.load();
                enqueue_init<T>(m, p, psi, b, x, vc32, df, W, cs);
                const int64_t l1 = pr.launches.load();
                enqueue_loop(cs, W.cap_body, S, [&](cudaStream_t bs, const LoopGate &gate) {
                    enqueue_iteration<T>(m, p, psi, b, x, vc32, df, W, bs, gate);
                });
                W.loop_init_launches = l1 - l0 + 1;  // + k_loop_begin
                W.loop_iter_launches = pr.launches.load() - l1;
            });
        } else {
            capture(W.init, W.cap, [&](cudaStream_t cs) { enqueue_init<T>(m, p, psi, b, x, vc32, df, W, cs); });
            capture(W.body, W.cap, [&](cudaStream_t cs) {
                for (int k = 0; k < ITER_UNROLL; ++k) enqueue_iteration<T>(m, p, psi, b, x, vc32, df, W, cs);
            });
        }
    }
    // Stall test: with the double-FP32 Jacobian the ~48-bit apply limits the true
    // residual, so a recurrence three decades past tol hands over to FP64; in
    // FP64 a true residual that stays above tol while the recurrence runs nine
    // decades past it has reached the attainable accuracy (the rounding floor of
    // J applied to the iterate), and further iterations only repeat the test.
    k_set_params<<<1, 1, 0, s>>>(S, tol, maxit, use_true ? 1 : 0, !use_true ? 0.0 : (df ? 1e-3 : 1e-9));
    GL_LAUNCH_CHECK();
    MinresDev h;
    if (loop) {
        GL_CUDA(cudaGraphLaunch(W.loop.exec, s));
        GL_CUDA(cudaMemcpyAsync(&h, S, sizeof(MinresDev), cudaMemcpyDeviceToHost, s));
        GL_CUDA(cudaStreamSynchronize(s));
        // the kernels that ran: the initial phase and one iteration's launches per iteration
        note_launch((int)(W.loop_init_launches + (int64_t)h.it * W.loop_iter_launches));
        GL_REQUIRE(h.status != ST_RUN, GL_ERR_TIMEOUT, "MINRES status word was not updated");
    } else {
    replay(W.init, s);
    int64_t polls = 0, max_polls = (int64_t)maxit / ITER_UNROLL + 3;
    bool init_timed = false;  // the initial phase's profiler events are summed once per solve
    for (;;) {
        GL_CUDA(cudaMemcpyAsync(&h, S, sizeof(MinresDev), cudaMemcpyDeviceToHost, s));
        GL_CUDA(cudaStreamSynchronize(s));
        if (!init_timed) {
            harvest(W.init);
            init_timed = true;
        }
        if (h.status != ST_RUN) break;
        GL_REQUIRE(polls++ <= max_polls, GL_ERR_TIMEOUT, "MINRES status word was not updated");
        replay(W.body, s);
        GL_CUDA(cudaMemcpyAsync(&h, S, sizeof(MinresDev), cudaMemcpyDeviceToHost, s));
        GL_CUDA(cudaStreamSynchronize(s));
        harvest(W.body);
        if (h.status != ST_RUN) break;
    }
    }
    if (use_true) {
        note_launch();
        k_true_resid<C, T><<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, O::K(m), O::kdiag(m), O::vol(m), psi, b, x, part, S,
                                                              LoopGate{{}, 0}, 1);
        GL_LAUNCH_CHECK();
        GL_CUDA(cudaMemcpyAsync(&h, S, sizeof(MinresDev), cudaMemcpyDeviceToHost, s));
        GL_CUDA(cudaStreamSynchronize(s));
    }
    return MinresResult{h.status, h.it, h.est, h.true_rel};
}

static gl_status status_of(int st) {
    switch (st) {
        case ST_CONV: return GL_OK;
        case ST_BREAK: return GL_ERR_BREAKDOWN;
        case ST_NAN: return GL_ERR_NAN;
        case ST_TIMEOUT: return GL_ERR_TIMEOUT;
        default: return GL_ERR_NOT_CONVERGED;
    }
}

// ------------------------------------------------------------------ mixed precision
__global__ void k_resid64_scaled(int64_t n, SellView<double2> K, const double *kd, const double *vol,
                                 const double2 *psi, const double2 *b, const double2 *x, double2 *r, double *part) {
    __shared__ double sh[32];
    double a = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        double2 acc = sell_row<double2, double2>(K, p, x);
        double2 jx = jacobian_epilogue(acc, kd[p], psi[p], x[p]);
        double2 rr = csub(b[p], jx);
        r[p] = rr;
        a += vol[p] * (rr.x * rr.x + rr.y * rr.y);
    }
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}
__global__ void k_sumsq_vol(int64_t n, const double *vol, const double2 *b, double *part) {
    __shared__ double sh[32];
    double a = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
        a += vol[p] * (b[p].x * b[p].x + b[p].y * b[p].y);
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}
__global__ void k_sum_to(const double *part, double *out) {
    __shared__ double sh[32];
    double a = 0;
    for (int i = threadIdx.x; i < RED_BLOCKS; i += blockDim.x) a += part[i];
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) *out = t;
}
// r32 = r / scale
__global__ void k_down(int64_t n, const double2 *r, double scale, float2 *r32, float2 *e32) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) {
        r32[p] = make_float2((float)(r[p].x / scale), (float)(r[p].y / scale));
        e32[p] = make_float2(0.f, 0.f);
    }
}
// x += scale * e32
__global__ void k_up(int64_t n, const float2 *e32, double scale, double2 *x) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) {
        x[p].x += scale * (double)e32[p].x;
        x[p].y += scale * (double)e32[p].y;
    }
}
__global__ void k_psi32(int64_t n, const double2 *a, float2 *b) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) b[p] = to32(a[p]);
}

struct SolveWork {
    MinresWork<double> w64;
    MinresWork<float> w32;
    DBuf<double2> r;
    DBuf<float2> r32, e32, psi32;
    DBuf<double> part, sc;
};
static SolveWork &solve_work() {
    static thread_local SolveWork w;
    return w;
}

// ------------------------------------------------------------------ batched solves
// Many independent systems J(psi_s) x_s = b_s in ONE CUDA-graph launch: each
// instance is a branch of the graph (its own buffers and preconditioner), and
// its MINRES iterations run inside a WHILE conditional node whose condition the
// iteration's last kernel sets from the instance's status word, so the whole batch runs
// on the device without host round trips.
struct BatchInst {
    gl_mesh_s *m = nullptr;
    gl_prec_s *p = nullptr;
    MinresWork<double> W;
    DBuf<double2> b, x;  // solve ordering
    bool df = false;     // double-float Jacobian (FP32 V-cycle on a lattice mesh)
};

}  // namespace gl

struct gl_batch_s {
    std::vector<std::unique_ptr<gl::BatchInst>> inst;
    gl_options o{};
    bool vc32 = false;
    cudaGraphExec_t exec = nullptr;
    std::vector<const void *> b_ptr, x_ptr;  // user pointers the graph was built for
    cudaStream_t s0 = nullptr, sb = nullptr;
    std::vector<cudaStream_t> br;
    std::vector<cudaEvent_t> ev;
    int64_t launches = 0;
    ~gl_batch_s() {
        cudaDeviceSynchronize();
        if (exec) cudaGraphExecDestroy(exec);
        for (auto e : ev) cudaEventDestroy(e);
        for (auto t : br) cudaStreamDestroy(t);
        if (s0) cudaStreamDestroy(s0);
        if (sb) cudaStreamDestroy(sb);
        for (auto &i : inst) delete i->p;
    }
};

namespace gl {

gl_batch_s *batch_new() { return new gl_batch_s(); }
void batch_delete(gl_batch_s *B) { delete B; }
size_t batch_size(const gl_batch_s *B) { return B->inst.size(); }

void batch_create(gl_batch_s *B, int count, gl_mesh_s *const *meshes, const double2 *const *psi, const gl_options &o,
                  cudaStream_t s) {
    B->o = o;
    B->vc32 = (o.precision != GL_FP64);
    gl_options so = o;
    so.precision = B->vc32 ? GL_MIXED_PRECOND : GL_FP64;
    for (int i = 0; i < count; ++i) {
        auto I = std::make_unique<BatchInst>();
        I->m = meshes[i];
        I->p = new gl_prec_s();
        precond_setup(I->p, I->m, psi[i], so, s);
        I->W.ensure(I->m->n, B->vc32);
        // as in a single mixed solve: the double-float Jacobian wherever the mesh
        // has the checked lattice stencil
        I->df = B->vc32 && I->p->lattice && I->m->lat_ok;
        if (I->df) I->W.ensure_df();
        I->b.alloc(I->m->n);
        I->x.alloc(I->m->n);
        B->inst.push_back(std::move(I));
    }
    GL_CUDA(cudaStreamCreateWithFlags(&B->s0, cudaStreamNonBlocking));
    GL_CUDA(cudaStreamCreateWithFlags(&B->sb, cudaStreamNonBlocking));
    B->br.resize(count);
    for (auto &t : B->br) GL_CUDA(cudaStreamCreateWithFlags(&t, cudaStreamNonBlocking));
    B->ev.resize(count + 1);
    for (auto &e : B->ev) GL_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
}

static void batch_build(gl_batch_s *B, const double2 *const *b, double2 *const *x) {
    if (B->exec) cudaGraphExecDestroy(B->exec);
    B->exec = nullptr;
    Profiler &pr = profiler();
    bool was_active = pr.active;
    pr.active = false;  // no event nodes inside conditional bodies
    int64_t l0 = pr.launches.load();
    cudaStream_t s0 = B->s0;
    cudaGraph_t graph = nullptr;
    GL_CUDA(cudaStreamBeginCapture(s0, cudaStreamCaptureModeThreadLocal));
    try {
        GL_CUDA(cudaEventRecord(B->ev[0], s0));
        for (size_t i = 0; i < B->inst.size(); ++i) {
            BatchInst &I = *B->inst[i];
            cudaStream_t si = B->br[i];
            int64_t n = I.m->n;
            MinresDev *S = I.W.S.get();
            GL_CUDA(cudaStreamWaitEvent(si, B->ev[0], 0));
            permute_in(n, I.m->perm.get(), b[i], I.b.get(), si);
            permute_in(n, I.m->perm.get(), x[i], I.x.get(), si);
            // the double-float Jacobian's stall test, as in a single solve
            k_set_params<<<1, 1, 0, si>>>(S, B->o.tol, B->o.maxit, 1, I.df ? 1e-3 : 0.0);
            enqueue_init<double>(I.m, I.p, I.p->psi_p.get(), I.b.get(), I.x.get(), B->vc32, I.df, I.W, si);
            enqueue_loop(si, B->sb, S, [&](cudaStream_t bs, const LoopGate &gate) {
                enqueue_iteration<double>(I.m, I.p, I.p->psi_p.get(), I.b.get(), I.x.get(), B->vc32, I.df, I.W, bs,
                                          gate);
            });
            // final FP64 true residual, back to node order
            k_true_resid<double2, double><<<RED_BLOCKS, RED_THREADS, 0, si>>>(
                n, I.m->K.view(), I.m->kdiag.get(), I.m->volp.get(), I.p->psi_p.get(), I.b.get(), I.x.get(),
                I.W.part.get(), S, LoopGate{{}, 0}, 1);
            GL_LAUNCH_CHECK();
            permute_out(n, I.m->perm.get(), I.x.get(), x[i], si);
            GL_CUDA(cudaEventRecord(B->ev[i + 1], si));
            GL_CUDA(cudaStreamWaitEvent(s0, B->ev[i + 1], 0));
        }
    } catch (...) {
        cudaStreamEndCapture(s0, &graph);
        if (graph) cudaGraphDestroy(graph);
        pr.active = was_active;
        throw;
    }
    GL_CUDA(cudaStreamEndCapture(s0, &graph));
    pr.active = was_active;
    B->launches = pr.launches.load() - l0;
    pr.launches.fetch_sub(B->launches);
    GL_CUDA(cudaGraphInstantiate(&B->exec, graph, 0));
    GL_CUDA(cudaGraphDestroy(graph));
    B->b_ptr.assign(b, b + B->inst.size());
    B->x_ptr.assign(x, x + B->inst.size());
}

gl_status batch_run(gl_batch_s *B, const double2 *const *b, double2 *const *x, gl_solve_info *infos, cudaStream_t s) {
    size_t k = B->inst.size();
    for (auto &I : B->inst)
        GL_REQUIRE(I->p->mesh_version == I->m->version, GL_ERR_ARG, "a batch mesh's mu changed after gl_batch_create");
    bool same = B->exec && B->b_ptr.size() == k;
    for (size_t i = 0; same && i < k; ++i) same = (B->b_ptr[i] == b[i] && B->x_ptr[i] == x[i]);
    if (!same) batch_build(B, b, x);
    auto t0 = std::chrono::steady_clock::now();
    GL_CUDA(cudaGraphLaunch(B->exec, s));
    note_launch((int)B->launches);  // captured launches; loop bodies replay on the device
    GL_CUDA(cudaStreamSynchronize(s));
    double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    gl_status first = GL_OK;
    for (size_t i = 0; i < k; ++i) {
        BatchInst &I = *B->inst[i];
        MinresDev h;
        GL_CUDA(cudaMemcpy(&h, I.W.S.get(), sizeof(MinresDev), cudaMemcpyDeviceToHost));
        int restarts = 0, its = h.it;
        if (h.status == ST_STALL) {
            // the double-float Jacobian's ~48-bit apply held the true residual above
            // tol: this instance continues from its x with the FP64 Jacobian, as a
            // single solve does
            const auto t1 = std::chrono::steady_clock::now();
            MinresResult r = minres<double>(I.m, I.p, I.p->psi_p.get(), I.b.get(), I.x.get(), B->o.tol,
                                            std::max(B->o.maxit - its, 1), true, B->vc32, I.W, s, false, true);
            permute_out(I.m->n, I.m->perm.get(), I.x.get(), x[i], s);
            GL_CUDA(cudaStreamSynchronize(s));
            ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t1).count();
            h.status = r.status;
            h.true_rel = r.true_rel;
            h.est = r.est;
            its += r.iters;
            restarts = 1;
        }
        if (infos) {
            gl_solve_info inf{};
            inf.iters = its;
            inf.outer_iters = 1;
            inf.converged = (h.status == ST_CONV && h.true_rel <= B->o.tol);
            inf.true_relres = h.true_rel;
            inf.est_relres = h.est;
            inf.solve_ms = ms;
            inf.df_jacobian = I.df ? 1 : 0;
            inf.stall_restarts = restarts;
            infos[i] = inf;
        }
        gl_status st = (h.status == ST_CONV) ? (h.true_rel <= B->o.tol ? GL_OK : GL_ERR_NOT_CONVERGED)
                                             : status_of(h.status);
        if (st == GL_ERR_TIMEOUT) {
            sweeps_reset(B->inst[i]->p, s);
            GL_CUDA(cudaStreamSynchronize(s));
            st = GL_ERR_TIMEOUT;
            if (infos) infos[i].converged = 0;
        }
        if (st != GL_OK && first == GL_OK) first = st;
    }
    return first;
}

gl_status jacobian_solve_p(gl_mesh_s *m, gl_prec_s *p, const double2 *psi_p, const double2 *b_p, double2 *x_p,
                           const gl_options &o, gl_solve_info *info, cudaStream_t s) {
    SolveWork &W = solve_work();
    auto t0 = std::chrono::steady_clock::now();
    gl_status st;
    gl_solve_info inf{};
    GL_REQUIRE(!(p && p->rinf) || o.precision == GL_FP64, GL_ERR_ARG, "R_inf needs precision GL_FP64");
    rinf_reset(p, s);
    if (o.warmstart)
        warmstart_apply_p(o.warmstart, m, psi_p, b_p, x_p, s, (const double2 *)o.warmstart_hint);
    else if (o.warmstart_hint)
        hint_guess_p(m, psi_p, b_p, (const double2 *)o.warmstart_hint, x_p, s);
    bool mixed = (o.precision == GL_MIXED) && p;
    if (!mixed) {
        bool vc32 = (o.precision == GL_MIXED_PRECOND) && p;
        if (vc32) precond_ensure_fp32(p, s);
        // the double-float Jacobian on lattices; if its ~48-bit arithmetic stalls
        // the FP64 true residual above tol, MINRES restarts from the current x
        // with the FP64 Jacobian
        const bool df = vc32 && p->lattice && m->lat_ok;
        const bool dl = o.device_loop != 0;
        MinresResult r = minres<double>(m, p, psi_p, b_p, x_p, o.tol, o.maxit, true, vc32, W.w64, s, df, dl);
        inf.df_jacobian = df ? 1 : 0;
        if (df && r.status == ST_STALL) {
            int used = r.iters;
            r = minres<double>(m, p, psi_p, b_p, x_p, o.tol, std::max(o.maxit - used, 1), true, vc32, W.w64, s, false,
                               dl);
            r.iters += used;
            inf.stall_restarts = 1;
        }
        inf.iters = r.iters;
        inf.outer_iters = 1;
        inf.true_relres = r.true_rel;
        inf.est_relres = r.est;
        inf.converged = (r.status == ST_CONV);
        st = status_of(r.status);
    } else {
        precond_ensure_fp32(p, s);
        int64_t n = m->n;
        if (W.r.n != (size_t)n) {
            W.r.alloc(n);
            W.r32.alloc(n);
            W.e32.alloc(n);
            W.psi32.alloc(n);
        }
        W.part.alloc(RED_BLOCKS);
        W.sc.alloc(2);
        int G = grid_for(n, 256);
        k_psi32<<<G, 256, 0, s>>>(n, psi_p, W.psi32.get());
        k_sumsq_vol<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, m->volp.get(), b_p, W.part.get());
        k_sum_to<<<1, 1024, 0, s>>>(W.part.get(), W.sc.get());
        double bb = 0;
        GL_CUDA(cudaMemcpyAsync(&bb, W.sc.get(), sizeof(double), cudaMemcpyDeviceToHost, s));
        GL_CUDA(cudaStreamSynchronize(s));
        double bnorm = std::sqrt(bb);
        st = GL_ERR_NOT_CONVERGED;
        int max_outer = o.max_outer > 0 ? o.max_outer : 20;
        double inner_tol = o.inner_tol > 0 ? o.inner_tol : 1e-5;
        double rel = 0;
        int total = 0, outer = 0;
        double est = 0;
        if (bnorm == 0) {
            GL_CUDA(cudaMemsetAsync(x_p, 0, n * sizeof(double2), s));
            st = GL_OK;
        }
        for (; st != GL_OK && outer <= max_outer; ++outer) {
            k_resid64_scaled<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, m->K.view(), m->kdiag.get(), m->volp.get(), psi_p,
                                                                b_p, x_p, W.r.get(), W.part.get());
            k_sum_to<<<1, 1024, 0, s>>>(W.part.get(), W.sc.get());
            double rr = 0;
            GL_CUDA(cudaMemcpyAsync(&rr, W.sc.get(), sizeof(double), cudaMemcpyDeviceToHost, s));
            GL_CUDA(cudaStreamSynchronize(s));
            rel = std::sqrt(rr) / bnorm;
            if (!std::isfinite(rel)) {
                st = GL_ERR_NAN;
                break;
            }
            if (rel <= o.tol) {
                st = GL_OK;
                break;
            }
            if (outer == max_outer || total >= o.maxit) break;
            double scale = std::sqrt(rr);
            k_down<<<G, 256, 0, s>>>(n, W.r.get(), scale, W.r32.get(), W.e32.get());
            GL_LAUNCH_CHECK();
            MinresResult r = minres<float>(m, p, W.psi32.get(), W.r32.get(), W.e32.get(), inner_tol,
                                           o.maxit - total, false, false, W.w32, s, false, o.device_loop != 0);
            total += r.iters;
            est = r.est;
            if (r.status == ST_BREAK || r.status == ST_NAN || r.status == ST_TIMEOUT) {
                st = status_of(r.status);
                break;
            }
            k_up<<<G, 256, 0, s>>>(n, W.e32.get(), scale, x_p);
            GL_LAUNCH_CHECK();
        }
        inf.iters = total;
        inf.outer_iters = outer;
        inf.true_relres = rel;
        inf.est_relres = est;
        inf.converged = (st == GL_OK);
    }
    GL_CUDA(cudaStreamSynchronize(s));
    auto t1 = std::chrono::steady_clock::now();
    // a coarse-sweep wait that ran out (it wrote the status word) left the
    // sweeps' counters out of step
    if (p && st == GL_ERR_TIMEOUT) {
        sweeps_reset(p, s);
        GL_CUDA(cudaStreamSynchronize(s));
        st = GL_ERR_TIMEOUT;
        inf.converged = 0;
    }
    inf.solve_ms = std::chrono::duration<double, std::milli>(t1 - t0).count();
    inf.warmstart_used = o.warmstart ? warmstart_used(o.warmstart, s) : (o.warmstart_hint ? 1 : 0);
    inf.lattice_stencil = (p && p->has32 && o.precision != GL_FP64 && p->lattice && m->lat_ok) ? 1 : 0;
    // MINRES's FP64 Jacobian (FP64 solves; mixed-preconditioner solves without the
    // double-float apply or after its stall) read the FP64 tables
    const bool fp64_j = o.precision == GL_FP64 ||
                        (o.precision == GL_MIXED_PRECOND && (!inf.df_jacobian || inf.stall_restarts));
    inf.jacobian_tables = (fp64_j && m->lat64_ok && p && p->lattice64) ? 1 : 0;
    if (p && p->rinf) {
        // measured: every application ran its own number of cycles, each followed by a residual
        const RinfDev R = rinf_read(p, s);
        const double per = p->cost_fine > 0 ? (p->cost_vcycle + p->cost_fine) / p->cost_fine : 0.0;
        inf.matvec_equiv = (double)(inf.iters + inf.outer_iters) + (double)R.cycles * per;
        inf.cycles_per_apply = R.applies ? (double)R.cycles / (double)R.applies : 0.0;
    } else {
        inf.matvec_equiv = (double)(inf.iters + inf.outer_iters) * (1.0 + (p ? precond_cost(p, p->cycles) : 0.0));
        inf.cycles_per_apply = p ? (double)p->cycles : 0.0;
    }
    if (info) {
        double setup = info->setup_ms;
        *info = inf;
        info->setup_ms = setup;
    }
    return st;
}

}  // namespace gl
