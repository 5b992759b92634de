// gl_ops.cu -- the fused sliced-ELL operators of the discrete GL problem, on vectors
// in the solve ordering (red nodes first, then black) and in node order:
//   Jacobian (Sec. 3): y_i = (K phi)_i + (-1 + 2|psi_i|^2) phi_i + psi_i^2 conj(phi_i)
//   residual (Eq. discr ginla): r_i = (K psi)_i - psi_i (1 - |psi_i|^2)
// with K = D^-1 K-hat (Remark rmk:dk) stored as off-diagonals + diagonal.
#include "gl_internal.cuh"
#include "gl_kernels.cuh"

namespace gl {

__global__ void k_gather(int64_t n, const int32_t *__restrict__ perm, const double2 *__restrict__ nat,
                         double2 *__restrict__ sol) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) sol[p] = nat[perm[p]];
}
__global__ void k_scatter(int64_t n, const int32_t *__restrict__ perm, const double2 *__restrict__ sol,
                          double2 *__restrict__ nat) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) nat[perm[p]] = sol[p];
}

void permute_in(int64_t n, const int32_t *perm, const double2 *nat, double2 *sol, cudaStream_t s) {
    k_gather<<<grid_for(n, 256), 256, 0, s>>>(n, perm, nat, sol);
    GL_LAUNCH_CHECK();
}
void permute_out(int64_t n, const int32_t *perm, const double2 *sol, double2 *nat, cudaStream_t s) {
    k_scatter<<<grid_for(n, 256), 256, 0, s>>>(n, perm, sol, nat);
    GL_LAUNCH_CHECK();
}

// y = J(psi) phi, FP64
__global__ void k_jacobian64(int64_t n, SellView<double2> K, const double *__restrict__ kdiag,
                             const double2 *__restrict__ psi, const double2 *__restrict__ phi,
                             double2 *__restrict__ y) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    double2 acc = sell_row<double2, double2>(K, p, phi);
    y[p] = jacobian_epilogue(acc, kdiag[p], psi[p], phi[p]);
}

// the same from the FP64 lattice tables (meshes whose stored K matches them)
__global__ void k_jacobian_lat64(int64_t n, LatticeView64 L, const double *__restrict__ kdiag,
                                 const double2 *__restrict__ psi, const double2 *__restrict__ phi,
                                 double2 *__restrict__ y) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    double2 acc = lattice_row64(L, p, phi);
    y[p] = jacobian_epilogue(acc, kdiag[p], psi[p], phi[p]);
}

// y = J(psi) phi with the FP32 operator and FP32 arithmetic (FP64 in/out)
__global__ void k_jacobian32(int64_t n, SellView<float2> K, const float *__restrict__ kdiag,
                             const double2 *__restrict__ psi, const double2 *__restrict__ phi,
                             double2 *__restrict__ y) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    int64_t s = p >> 5;
    int lane = (int)(p & 31);
    int64_t beg = K.sptr[s];
    int w = (int)((K.sptr[s + 1] - beg) >> 5);
    float2 acc = make_float2(0.f, 0.f);
    for (int k = 0; k < w; ++k) {
        int64_t q = beg + (int64_t)k * SELL_C + lane;
        cfma(acc, K.val[q], to32(phi[K.col[q]]));
    }
    float2 r = jacobian_epilogue(acc, kdiag[p], to32(psi[p]), to32(phi[p]));
    y[p] = to64(r);
}

// The FP64 operators on vectors in node order, for the public calls: one thread per
// node v reads the row of its solve position iperm[v] with the columns as node
// numbers.  Consecutive nodes alternate between the two colours of a lattice, so a
// warp reads its matrix entries as two runs of 16 and its vectors as one of 32, and
// nothing is gathered and scattered around the apply.  Bound by the FP64 pipe (35
// operations a row in 3D, 117 us for 128^3 rows at 1.25 TFLOP/s; the bytes would take 55
// us).  Whole calls, before (two gathers, the apply on reordered vectors, a scatter) and
// now: Jacobian on 128^3 nodes 193 and
// 129 us, on 64^2 22.8 and 15.0 us; residual on 1023^2 63 and 45 us.
__device__ __forceinline__ double2 row_nodes(const SellView<double2> &K, const int32_t *__restrict__ coln, int64_t p,
                                             const double2 *__restrict__ x) {
    const int64_t beg = __ldg(K.sptr + (p >> 5));
    const int w = (int)((__ldg(K.sptr + (p >> 5) + 1) - beg) >> 5);
    const int32_t *cp = coln + beg + (p & 31);
    const double2 *vp = K.val + beg + (p & 31);
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int k = 0; k < w; ++k) cfma(acc, vp[(int64_t)k * SELL_C], __ldg(x + __ldg(cp + (int64_t)k * SELL_C)));
    return acc;
}
__global__ void __launch_bounds__(256) k_jacobian_nodes(int64_t n, SellView<double2> K,
                                                        const int32_t *__restrict__ coln,
                                                        const int32_t *__restrict__ iperm,
                                                        const double *__restrict__ kdiag,
                                                        const double2 *__restrict__ psi,
                                                        const double2 *__restrict__ phi, double2 *__restrict__ y) {
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v >= n) return;
    const int64_t p = iperm[v];
    const double2 ps = psi[v], ph = phi[v];
    y[v] = jacobian_epilogue(row_nodes(K, coln, p, phi), kdiag[p], ps, ph);
}
// r = GL(psi): (K psi)_i - psi_i (1 - |psi_i|^2) = offdiag + (K_ii - 1 + |psi_i|^2) psi_i
__global__ void __launch_bounds__(256) k_residual_nodes(int64_t n, SellView<double2> K,
                                                        const int32_t *__restrict__ coln,
                                                        const int32_t *__restrict__ iperm,
                                                        const double *__restrict__ kdiag,
                                                        const double2 *__restrict__ psi, double2 *__restrict__ r) {
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v >= n) return;
    const int64_t p = iperm[v];
    const double2 ps = psi[v];
    const double2 acc = row_nodes(K, coln, p, psi);
    const double a2 = ps.x * ps.x + ps.y * ps.y;
    const double d = kdiag[p] - 1.0 + a2;
    r[v] = mk(acc.x + d * ps.x, acc.y + d * ps.y);
}
// Newton right-hand side (Eq. Newton system): r <- -r in place, with per-block
// partials of ||r||_R^2 = sum |V_i| |r_i|^2
__global__ void k_negate_norm(int64_t n, const double *__restrict__ vol, double2 *__restrict__ r, double *part) {
    __shared__ double sh[32];
    double a = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double2 v = r[i];
        a += vol[i] * (v.x * v.x + v.y * v.y);
        r[i] = make_double2(-v.x, -v.y);
    }
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}
__global__ void k_sum_parts_sqrt(const double *part, int np, double *out) {
    __shared__ double sh[32];
    double a = 0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) a += part[i];
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) *out = sqrt(t);
}
// psi <- psi + d
__global__ void k_axpy64(int64_t n, const double2 *__restrict__ d, double2 *__restrict__ psi) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) psi[i] = cadd(psi[i], d[i]);
}

double newton_rhs(const gl_mesh_s *m, double2 *r, double *part, double *scal, cudaStream_t s) {
    k_negate_norm<<<RED_BLOCKS, RED_THREADS, 0, s>>>(m->n, m->vol.get(), r, part);
    k_sum_parts_sqrt<<<1, 1024, 0, s>>>(part, RED_BLOCKS, scal);
    GL_LAUNCH_CHECK();
    double g = 0;
    GL_CUDA(cudaMemcpyAsync(&g, scal, sizeof(double), cudaMemcpyDeviceToHost, s));
    GL_CUDA(cudaStreamSynchronize(s));
    return g;
}
void newton_update(int64_t n, const double2 *d, double2 *psi, cudaStream_t s) {
    k_axpy64<<<grid_for(n, 256), 256, 0, s>>>(n, d, psi);
    GL_LAUNCH_CHECK();
}

void jacobian_apply_p(const gl_mesh_s *m, const double2 *psi, const double2 *phi, double2 *y, cudaStream_t s) {
    k_jacobian64<<<grid_for(m->n, 256), 256, 0, s>>>(m->n, m->K.view(), m->kdiag.get(), psi, phi, y);
    GL_LAUNCH_CHECK();
}
// the same matrix-free from the lattice stencil's FP64 tables (meshes whose stored
// K matches them to 16 ulp of its largest entry: the same operator up to rounding)
void jacobian_apply_lat64_p(const gl_mesh_s *m, const double2 *psi, const double2 *phi, double2 *y, cudaStream_t s) {
    GL_REQUIRE(m->lat64_ok, GL_ERR_ARG, "the mesh has no FP64 lattice stencil (odd N, or K does not match it)");
    k_jacobian_lat64<<<grid_for(m->n, 256), 256, 0, s>>>(m->n, lattice_view64(m), m->kdiag.get(), psi, phi, y);
    GL_LAUNCH_CHECK();
}
void jacobian_apply_p32(const gl_mesh_s *m, const double2 *psi, const double2 *phi, double2 *y, cudaStream_t s) {
    k_jacobian32<<<grid_for(m->n, 256), 256, 0, s>>>(m->n, m->K32.view(), m->kdiag32.get(), psi, phi, y);
    GL_LAUNCH_CHECK();
}
void jacobian_apply_nodes(const gl_mesh_s *m, const double2 *psi, const double2 *phi, double2 *y, cudaStream_t s) {
    k_jacobian_nodes<<<grid_for(m->n, 256), 256, 0, s>>>(m->n, m->K.view(), m->K.node_col(), m->iperm.get(),
                                                         m->kdiag.get(), psi, phi, y);
    GL_LAUNCH_CHECK();
}
void residual_nodes(const gl_mesh_s *m, const double2 *psi, double2 *r, cudaStream_t s) {
    k_residual_nodes<<<grid_for(m->n, 256), 256, 0, s>>>(m->n, m->K.view(), m->K.node_col(), m->iperm.get(),
                                                         m->kdiag.get(), psi, r);
    GL_LAUNCH_CHECK();
}

}  // namespace gl
