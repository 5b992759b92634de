// gl_warmstart.cu -- learned initial guess for the Jacobian solve J(psi) x = b
// (Sec. 3, Eq. (16)); the paper has no learned part, the network is defined here.
//
//   x0 = ||b||_D * y(psi, b / ||b||_D) / K_ii,      ||b||_D^2 = sum_i |V_i| |b_i|^2
//
// y is a 4-layer, 64-channel graph network on the mesh.  Channels come in 32
// complex pairs; channel 63 is the constant 1 (it carries the biases).
//   h^0_i   = [Re b^_i, Im b^_i, Re psi_i, Im psi_i, |psi_i|^2, 0 ... 0, 1]
//   a^l_i   = [h^l_i ; (S h^l)_i],  (S u)_i = sum_k (-K-hat_ik / K-hat_ii) u_k  (per pair)
//   h^{l+1} = relu(W^l a^l), channel 63 reset to 1            (W^l: 64 x 128)
//   y_i     = U h^4_i                                          (U: 2 x 64)
// S = I - diag(K)^-1 K is the magnetic Jacobi operator: the edge weights and
// phases of Eq. (10) normalised per row.  Training minimises the squared relative
// true-Jacobian residual L = ||b^ - J x^||_D^2 of the guess (x^ = y / K_ii).
//
// GPU layout and precision:
//   * every vector is in the solve ordering of the mesh (red nodes first); the
//     aggregation reads the FP32 copy of K (sliced ELL) and K_ii;
//   * activations h^l are n x 64 BF16, node-major (128 B per node);
//   * the dense layers are tcgen05 MMAs (kind::f16, BF16 operands, FP32
//     accumulators in tensor memory), one 128-node tile per MMA group.  Operands
//     are staged in shared memory: activations and dz as rows of 128 bytes a node with
//     swizzled chunks (SWIZZLE_128B), W as K-major tiles of 8-row x 16-byte core matrices
//     without swizzle: leading-dimension offset 128 B (next core matrix along K),
//     stride-dimension offset 16 K bytes (next 8-row group);
//   * forward: one persistent kernel per layer builds [h, S h] for its tile
//     (gathering the neighbours' BF16 rows), issues 8 MMAs (K = 16 each) into a
//     128 x 64 FP32 accumulator, and applies relu (and the head on the last layer)
//     in the epilogue;
//   * backward: one persistent kernel per layer issues dA = dz W (M = 128 nodes,
//     N = 128, K = 64) and accumulates dW^T += a^T dz (M = 128 inputs, N = 64,
//     K = 128 nodes of the tile) in tensor memory across all of its tiles, both from the
//     same swizzled rows of [h, S h] and dz; the adjoint aggregation S^T and the relu mask
//     follow in a gather kernel;
//   * parameters are FP32 masters with Adam moments; BF16 images of each W in
//     the two shared-memory operand layouts are rebuilt after every update.
// Every reduction (loss, dW, dU, ||b||) sums per-block partials in a fixed order,
// so results are deterministic for a given launch configuration.
#include <cuda_bf16.h>

#include <cstring>

#include "gl_internal.cuh"
#include "gl_profile.cuh"

namespace gl {
namespace ws {

constexpr int CH = 64;               // channels
constexpr int CIN = 2 * CH;          // [h, S h]
constexpr int NL = 4;                // layers
constexpr int WSZ = CH * CIN;        // one W^l
constexpr int NPARAM = NL * WSZ + 2 * CH;
constexpr int TILE = 128;            // nodes per MMA tile (= M)
constexpr int DU_BLOCKS = 2 * NUM_SMS_HINT;
constexpr long long WAIT_CYCLES = 4000000000LL;   // about 2 s at the maximum SM clock

static_assert(NPARAM == GL_WS_NPARAM, "parameter count must match the header");

// ------------------------------------------------------------------ tcgen05 helpers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// element offset (in 2-byte units) of (row r, column k) in an R x K K-major tile
// of 8 x 8 core matrices, K fastest between core matrices
__device__ __forceinline__ int cm_off(int r, int k, int K) {
    return (((r >> 3) * (K >> 3) + (k >> 3)) << 6) + ((r & 7) << 3) + (k & 7);
}

// shared-memory matrix descriptor: no swizzle, version 1
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// the same for rows of 64 BF16 (128 bytes) whose 16-byte chunks are XOR-swizzled by the
// row within groups of eight rows (SWIZZLE_128B): 1024 bytes from group to group.  Rows
// may be M or N (K-major) or K (MN-major; lbo: bytes to the next 64 columns of M or N)
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr, uint32_t lbo = 16) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// instruction descriptor of kind::f16: BF16 A and B, FP32 D, both K-major
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint64_t *mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar)));
}

// wait on an mbarrier phase for at most WAIT_CYCLES; returns false if that ran out
__device__ __forceinline__ bool mbar_try(uint64_t *mbar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(smem_u32(mbar)), "r"(parity)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity) {
    if (mbar_try(mbar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(mbar, parity))
        if (clock64() - t0 > WAIT_CYCLES) return false;
    return true;
}

// 16 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols));
}

__device__ __forceinline__ void mbar_init_n(uint64_t *mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t *mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(mbar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t *mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes) : "memory");
}
// global -> shared, both 16-byte aligned, a multiple of 16 bytes
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(mbar))
                 : "memory");
}

// ------------------------------------------------------------------ BF16 row helpers
// 8 BF16 <-> 8 floats in one 16-byte word
__device__ __forceinline__ void unpack8(uint4 u, float *f) {
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 t = __bfloat1622float2(h[i]);
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
    }
}
__device__ __forceinline__ uint4 pack8(const float *f) {
    uint4 u;
    __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    return u;
}

// accumulate K_pq h_q over one 16-byte chunk (four complex pairs) of h_q, two pairs at a
// time in packed FP32 arithmetic: acc + fma(v.x, re, -(v.y im)), acc + fma(v.x, im, v.y re);
// re/im of pairs (0, 1) and (2, 3).  Twelve instructions where scalar ones are 24.
struct Acc4 {
    float2 re[2], im[2];
};
__device__ __forceinline__ void cacc4_packed(Acc4 &acc, float2 v, uint4 r) {
    const float2 vx = make_float2(v.x, v.x), vy = make_float2(v.y, v.y), ny = make_float2(-v.y, -v.y);
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const float2 re = make_float2(__uint_as_float(w[2 * t] << 16), __uint_as_float(w[2 * t + 1] << 16));
        const float2 im = make_float2(__uint_as_float(w[2 * t] & 0xffff0000u), __uint_as_float(w[2 * t + 1] & 0xffff0000u));
        acc.re[t] = __fadd2_rn(acc.re[t], __ffma2_rn(vx, re, __fmul2_rn(ny, im)));
        acc.im[t] = __fadd2_rn(acc.im[t], __ffma2_rn(vx, im, __fmul2_rn(vy, re)));
    }
}

// ------------------------------------------------------------------ small kernels
// partials of sum |V_i| |b_i|^2
__global__ void k_bnorm_part(int64_t n, const double *__restrict__ vol, const double2 *__restrict__ b,
                             double *part) {
    __shared__ double sh[32];
    double a = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double2 v = b[i];
        a += vol[i] * (v.x * v.x + v.y * v.y);
    }
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}
// bn[0] = ||b||_D, bn[1] = 1 / ||b||_D (0 if b = 0)
__global__ void k_bnorm_final(const double *part, int np, double *bn) {
    __shared__ double sh[32];
    double a = 0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) a += part[i];
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) {
        double r = sqrt(t);
        bn[0] = r;
        bn[1] = r > 0 ? 1.0 / r : 0.0;
    }
}

// ---- the hint: alpha = <J a, b>_R / <J a, J a>_R, r = b - alpha J a
// partials of <q, b>_R, <q, q>_R and ||a||_D^2 (q = J a)
__global__ void k_hint_part(int64_t n, const double *__restrict__ vol, const double2 *__restrict__ q,
                            const double2 *__restrict__ b, const double2 *__restrict__ a, double *part) {
    __shared__ double sh[32];
    double qb = 0, qq = 0, aa = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 qv = q[i], bv = b[i], av = a[i];
        const double w = vol[i];
        qb += w * (qv.x * bv.x + qv.y * bv.y);
        qq += w * (qv.x * qv.x + qv.y * qv.y);
        aa += w * (av.x * av.x + av.y * av.y);
    }
    const double t0 = block_sum(qb, sh);
    const double t1 = block_sum(qq, sh);
    const double t2 = block_sum(aa, sh);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = t0;
        part[RED_BLOCKS + blockIdx.x] = t1;
        part[2 * RED_BLOCKS + blockIdx.x] = t2;
    }
}
// hs[0] = alpha (0 when J a = 0), hs[1] = 1 / ||a||_D (0 when a = 0)
__global__ void k_hint_final(const double *part, double *hs) {
    __shared__ double sh[32];
    double s0 = 0, s1 = 0, s2 = 0;
    for (int i = threadIdx.x; i < RED_BLOCKS; i += blockDim.x) {
        s0 += part[i];
        s1 += part[RED_BLOCKS + i];
        s2 += part[2 * RED_BLOCKS + i];
    }
    const double qb = block_sum(s0, sh);
    const double qq = block_sum(s1, sh);
    const double aa = block_sum(s2, sh);
    if (threadIdx.x == 0) {
        hs[0] = (aa > 0 && qq > 0) ? qb / qq : 0.0;
        hs[1] = aa > 0 ? 1.0 / sqrt(aa) : 0.0;
    }
}
// r = b - alpha q
__global__ void k_hint_resid(int64_t n, const double *__restrict__ hs, const double2 *__restrict__ b,
                             const double2 *__restrict__ q, double2 *__restrict__ r) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double al = hs[0];
    r[i] = make_double2(b[i].x - al * q[i].x, b[i].y - al * q[i].y);
}
// x0 = alpha a
__global__ void k_hint_set(int64_t n, const double *__restrict__ hs, const double2 *__restrict__ a,
                           double2 *__restrict__ x0) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double al = hs[0];
    x0[i] = make_double2(al * a[i].x, al * a[i].y);
}
// x0 += alpha a
__global__ void k_hint_add(int64_t n, const double *__restrict__ hs, const double2 *__restrict__ a,
                           double2 *__restrict__ x0) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double al = hs[0];
    x0[i] = make_double2(x0[i].x + al * a[i].x, x0[i].y + al * a[i].y);
}

// h^0 rows: [Re r^, Im r^, Re psi, Im psi, |psi|^2, 0, Re a^, Im a^, 0 ..., 1]
// (the hint a^ = a / ||a||_D as the complex channel pair (6, 7), zero without one)
__global__ void k_features(int64_t n, const double2 *__restrict__ b, const double2 *__restrict__ psi,
                           const double *__restrict__ bn, const double2 *__restrict__ hint,
                           const double *__restrict__ hs, uint4 *__restrict__ H0, int compact) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    double inv = bn[1];
    double2 bv = b[p], ps = psi[p];
    float f[8] = {(float)(bv.x * inv), (float)(bv.y * inv), (float)ps.x, (float)ps.y,
                  (float)(ps.x * ps.x + ps.y * ps.y), 0.f, 0.f, 0.f};
    if (hint) {
        const double ia = hs[1];
        f[6] = (float)(hint[p].x * ia);
        f[7] = (float)(hint[p].y * ia);
    }
    float z[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float last[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 1.f};
    if (compact) {  // only the chunks that hold anything
        H0[2 * p] = pack8(f);
        H0[2 * p + 1] = pack8(last);
        return;
    }
    uint4 *row = H0 + p * 8;
    row[0] = pack8(f);
#pragma unroll
    for (int j = 1; j < 7; ++j) row[j] = pack8(z);
    row[7] = pack8(last);
}

// ------------------------------------------------------------------ forward layer
enum { FWD_HIDDEN = 0, FWD_LAST_TRAIN = 1, FWD_LAST_PREDICT = 2 };

// the aggregated features of one layer
struct TileArgs {
    int64_t n;
    int64_t ntiles;
    SellView<float2> K;
    const float *kdiag;
    const uint4 *Hin;        // n x 8 uint4 (compact: n x 2, the first and the last chunk)
};

struct FwdArgs {
    TileArgs t;
    uint4 *Hout;             // n x 8 uint4 (hidden layers, and h^4 when training)
    const uint4 *Wimg;       // 64 x 128 BF16 operand image (1024 uint4)
    const float *U;          // 2 x 64 head (last layer)
    float2 *xhat;            // training: x^ (FP32)
    double2 *x0;             // prediction: ||b|| x^ (FP64)
    const double *bn;
    int *err;
};

// One layer.  Bound by the gathers: six neighbour rows of 128 bytes a node through L1 (1.6 GB
// at 128^3 nodes, half of it from L2) around 0.7 GB of HBM traffic; the MMAs take a few
// percent of the time.  Eight threads a node read one 16-byte chunk of every row each, so
// the registers decide how many rows are in flight: one CTA per SM holds as many gathering
// warps as its registers allow with two nodes a thread requested ahead, and nothing else
// runs in those warps:
//   * three warps bring the K entries, slice widths and -1 / K_pp of the tiles to come into
//     shared memory (bulk copies; the offsets and diagonals they need are requested three
//     tiles earlier, or their latency alone is 3 us a tile);
//   * the gathering warps build operand tiles: their own rows by cp.async, S h from the
//     neighbours' chunks, two channel pairs at a time in packed FP32.  Rows of 64 channels
//     are 128 bytes with XOR-swizzled chunks (SWIZZLE_128B operands), so that a node's
//     eight threads write different banks (eight-way conflicts without);
//   * four warps take the finished tiles: one thread issues the MMAs of the next one into the
//     other of two accumulators, then all take the current accumulator through relu (and
//     head) to global memory.
// Two operand tiles leave more L1 to the gathers than three (365 us against 377, before the
// registers were split as below).  The first layer's rows hold two chunks that are not
// zero; only these are stored and gathered (COMPACT), and there the third operand tile pays:
// 160 us against 190.
// Every wait is bounded; a warp whose wait runs out leaves, the others follow.
// 128^3 nodes: 291 us a layer, 160 the first, 313 the last (588 each with three CTAs an SM
// going through staging, gathers, MMA and epilogue in turn); 63^3 nodes: 37 us (70).
constexpr int FWD_KSTAGES = 3;                         // tiles whose K entries are in shared memory (at most 4)
constexpr int FWD_K = 6;                               // staged K entries a row (further ones are read where used)
constexpr int FWD_TILE_BYTES = TILE * CIN * 2;
// gathering warps; + four epilogue warps + four of which FWD_KSTAGES bring K entries
__host__ __device__ constexpr int fwd_gw(bool compact) { return compact ? 8 : 16; }
__host__ __device__ constexpr int fwd_stages(bool compact) { return compact ? 3 : 2; }
__host__ __device__ constexpr int fwd_smem(bool compact) {  // operand tiles, W image, output rows, K entries
    return fwd_stages(compact) * FWD_TILE_BYTES + CH * CIN * 2 + TILE * CH * 2 + FWD_KSTAGES * FWD_K * TILE * 12;
}
__host__ __device__ constexpr int fwd_threads(bool compact) { return 32 * (fwd_gw(compact) + 8); }
// Of the 80 registers a thread of 24 warps can have, 16 warps' gathers want more and the
// others need fewer: 16 x 96 + 4 x 64 + 4 x 32 = 24 x 80 (291 us a layer; 365 with 80 for all,
// where the gathers' buffers spill)
template <int N>
__device__ __forceinline__ void regs_raise() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void regs_lower() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

// 16 bytes global -> shared behind the thread's back (zeros if !ok); not through L1
__device__ __forceinline__ void copy16(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// shared memory of the tile-building warps
struct TileBufs {
    unsigned char *tiles;          // operand tiles: h, S h (and dz) of 128 nodes, 128 bytes a row, swizzled
    float2 *val;                   // FWD_KSTAGES x 4 slices x FWD_K x 32 K entries
    int32_t *col;
    float (*sc)[TILE];             // -1 / K_pp
    int (*wid)[TILE / SELL_C];     // entries a row of each slice
    uint64_t *full, *empty, *kfull, *kempty;
};

// the warps that build operand tiles (true: a wait ran out)
template <bool COMPACT, int GW, int STAGES, int BYTES, bool WITH_DZ>
__device__ __forceinline__ bool build_tiles(const TileArgs &a, const TileBufs &b, const uint4 *__restrict__ dZ, int warp,
                                            int lane) {
    constexpr int NI = COMPACT ? 1 : 2;     // nodes of a tile for each thread
    constexpr int RS = COMPACT ? 2 : 8;     // chunks of a stored row
    const int jc = COMPACT ? (lane & 1) : (lane & 7), j = COMPACT ? 7 * jc : jc;
    const int r0 = COMPACT ? warp * 16 + (lane >> 1) : warp * 4 + (lane >> 3);
    const uint4 *__restrict__ Hj = a.Hin + jc;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    bool failed = false;
    int st = 0, ks = 0;
    uint32_t ph = 1, kph = 0;  // (the first round of the operand tiles is empty already)
    // request a chunk of a node's own row (into the operand tile) and of its neighbours'
    auto request = [&](uint4 (&nb)[FWD_K], int64_t t, int kst, int r, int stage) {
        const int64_t p = t * TILE + r;
        const bool ok = p < a.n;
        copy16(b.tiles + stage * BYTES + r * 128 + ((j ^ (r & 7)) << 4), ok ? Hj + p * RS : Hj, ok);
        if (WITH_DZ)
            copy16(b.tiles + stage * BYTES + (2 * TILE + r) * 128 + ((j ^ (r & 7)) << 4), ok ? dZ + p * 8 + j : dZ, ok);
        if (!ok) return;
        const int w = b.wid[kst][r >> 5];
        const int32_t *c = b.col + (kst * (TILE / SELL_C) + (r >> 5)) * (FWD_K * SELL_C) + (r & 31);
#pragma unroll
        for (int e = 0; e < FWD_K; ++e)
            if (e < w) nb[e] = __ldg(Hj + (int64_t)c[e * SELL_C] * RS);
    };
    // the chunk of S h
    auto finish = [&](const uint4 (&nb)[FWD_K], int64_t t, int kst, int r, int stage) {
        const int64_t p = t * TILE + r;
        uint4 out = zero;
        if (p < a.n) {
            Acc4 acc;
            acc.re[0] = acc.re[1] = acc.im[0] = acc.im[1] = make_float2(0.f, 0.f);
            const int w = b.wid[kst][r >> 5];
            const float2 *v = b.val + (kst * (TILE / SELL_C) + (r >> 5)) * (FWD_K * SELL_C) + (r & 31);
#pragma unroll
            for (int e = 0; e < FWD_K; ++e)
                if (e < w) cacc4_packed(acc, v[e * SELL_C], nb[e]);
            // rows wider than FWD_K (not produced by the lattice meshes)
            for (int e = FWD_K; e < w; ++e) {
                const int64_t q = a.K.sptr[p >> 5] + (int64_t)e * SELL_C + (p & 31);
                cacc4_packed(acc, a.K.val[q], __ldg(Hj + (int64_t)a.K.col[q] * RS));
            }
            const float sc = b.sc[kst][r];
            const float f[8] = {acc.re[0].x * sc, acc.im[0].x * sc, acc.re[0].y * sc, acc.im[0].y * sc,
                                acc.re[1].x * sc, acc.im[1].x * sc, acc.re[1].y * sc, acc.im[1].y * sc};
            out = pack8(f);
        }
        *reinterpret_cast<uint4 *>(b.tiles + stage * BYTES + (TILE + r) * 128 + ((j ^ (r & 7)) << 4)) = out;
    };
    uint4 A[FWD_K], B[FWD_K];
    bool more = blockIdx.x < a.ntiles;
    if (more) {
        failed = !__all_sync(0xffffffffu, mbar_wait(&b.kfull[0], 0));
        if (!failed) request(A, blockIdx.x, 0, r0, 0);
        if (NI == 1) copy_commit();
    }
    for (int64_t t = blockIdx.x; more && !failed; t += gridDim.x) {
        more = t + gridDim.x < a.ntiles;
        const int kn = ks + 1 == FWD_KSTAGES ? 0 : ks + 1, sn = st + 1 == STAGES ? 0 : st + 1;
        const uint32_t kpn = kn ? kph : kph ^ 1, pn = sn ? ph : ph ^ 1;
        if (NI == 2) {
            request(B, t, ks, r0 + TILE / 2, st);
            copy_commit();
            finish(A, t, ks, r0, st);
        }
        if (more && !__all_sync(0xffffffffu, mbar_wait(&b.kfull[kn], kpn) && mbar_wait(&b.empty[sn], pn))) {
            failed = true;
            break;
        }
        if (NI == 2) {
            if (more) request(A, t + gridDim.x, kn, r0, sn);
            finish(B, t, ks, r0 + TILE / 2, st);
            copy_wait<0>();
        } else {
            if (more) request(B, t + gridDim.x, kn, r0, sn);
            copy_commit();
            finish(A, t, ks, r0, st);
            copy_wait<1>();
#pragma unroll
            for (int e = 0; e < FWD_K; ++e) A[e] = B[e];
        }
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(&b.full[st]);
            mbar_arrive(&b.kempty[ks]);
        }
        st = sn;
        ph = pn;
        ks = kn;
        kph = kpn;
    }
    copy_wait<0>();
    return failed;
}

// the warps that bring K entries for them, one for each stage of the ring; slice offsets and
// diagonals are requested one round ahead
__device__ __forceinline__ bool stage_entries(const TileArgs &a, const TileBufs &b, int ks, int lane) {
    constexpr int NS = TILE / SELL_C;
    const int64_t step = (int64_t)FWD_KSTAGES * gridDim.x;
    int64_t s0;
    int w;
    float kd[NS];
    auto fetch = [&](int64_t t) {
        const int64_t sl = t * NS + lane;
        s0 = 0;
        w = 0;
        if (lane < NS && sl * SELL_C < a.n) {
            s0 = __ldg(a.K.sptr + sl);
            w = (int)((__ldg(a.K.sptr + sl + 1) - s0) / SELL_C);
        }
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            const int64_t p = t * TILE + SELL_C * q + lane;
            kd[q] = p < a.n ? __ldg(a.kdiag + p) : 1.f;
        }
    };
    uint32_t ph = 1;
    int64_t t = blockIdx.x + (int64_t)ks * gridDim.x;
    fetch(t);
    for (; t < a.ntiles; t += step) {
        if (!__all_sync(0xffffffffu, mbar_wait(&b.kempty[ks], ph))) {
            mbar_wait(&b.kfull[ks], ph);  // (the round before's)
            return true;
        }
#pragma unroll
        for (int q = 0; q < NS; ++q) b.sc[ks][SELL_C * q + lane] = -1.f / kd[q];
        if (lane < NS) {
            const uint32_t ne = (uint32_t)min(w, FWD_K) * SELL_C;
            const int dst = (ks * NS + lane) * (FWD_K * SELL_C);
            b.wid[ks][lane] = w;
            mbar_arrive_tx(&b.kfull[ks], ne * 12);
            if (ne) {
                bulk_load(b.col + dst, a.K.col + s0, ne * 4, &b.kfull[ks]);
                bulk_load(b.val + dst, a.K.val + s0, ne * 8, &b.kfull[ks]);
            }
        } else {
            mbar_arrive(&b.kfull[ks]);
        }
        fetch(t + step);
        ph ^= 1;
        // no copy may be in flight when the block ends
        if (t + step >= a.ntiles) mbar_wait(&b.kfull[ks], ph);
    }
    return false;
}

template <int MODE, bool COMPACT>
__global__ void __launch_bounds__(fwd_threads(COMPACT), 1) k_fwd(FwdArgs a) {
    constexpr int GW = fwd_gw(COMPACT), NTHREADS = fwd_threads(COMPACT), STAGES = fwd_stages(COMPACT);
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sA = smem;                                                        // STAGES x [h, S h] x 128 x 64
    uint4 *sW = reinterpret_cast<uint4 *>(smem + STAGES * FWD_TILE_BYTES);           // 64 x 128 image
    uint4 *sOut = sW + CH * CIN / 8;                                                 // 128 rows of 8 chunks
    float2 *sVal = reinterpret_cast<float2 *>(sOut + TILE * CH / 8);                 // FWD_KSTAGES x 4 slices x FWD_K x 32
    int32_t *sCol = reinterpret_cast<int32_t *>(sVal + FWD_KSTAGES * FWD_K * TILE);
    __shared__ float sSc[FWD_KSTAGES][TILE];             // -1 / K_pp
    __shared__ int sWid[FWD_KSTAGES][TILE / SELL_C];     // entries a row of each slice
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2], kfull[FWD_KSTAGES],
        kempty[FWD_KSTAGES];
    __shared__ uint32_t tslot;
    __shared__ float sU[2 * CH];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < CH * CIN / 8; i += NTHREADS) sW[i] = a.Wimg[i];
    if (COMPACT)  // the chunks that are not stored are zero in every tile
        for (int i = tid; i < STAGES * FWD_TILE_BYTES / 16; i += NTHREADS) reinterpret_cast<uint4 *>(sA)[i] = zero;
    if (MODE != FWD_HIDDEN && tid < 2 * CH) sU[tid] = a.U[tid];
    if (warp == GW) tmem_alloc(&tslot, 2 * CH);
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init_n(&full[i], GW);
            mbar_init_n(&empty[i], 1);
        }
        for (int i = 0; i < FWD_KSTAGES; ++i) {
            mbar_init_n(&kfull[i], 32);
            mbar_init_n(&kempty[i], GW);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init_n(&tfull[i], 1);
            mbar_init_n(&tempty[i], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    proxy_fence();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    const TileBufs bufs{sA, sVal, sCol, sSc, sWid, full, empty, kfull, kempty};
    bool failed = false;
    if (warp < GW) {
        if (!COMPACT) regs_raise<96>();
        failed = build_tiles<COMPACT, GW, STAGES, FWD_TILE_BYTES, false>(a.t, bufs, nullptr, warp, lane);
    } else if (warp >= GW + 4) {
        if (!COMPACT) regs_lower<32>();
        if (warp < GW + 4 + FWD_KSTAGES) failed = stage_entries(a.t, bufs, warp - GW - 4, lane);
    } else {
        if (!COMPACT) regs_lower<64>();
        // ---- MMAs (one thread) and epilogue: warp quarter's 32 rows of the 128 x 64
        // accumulator, one a thread
        const int quarter = warp - GW;
        const int r = quarter * 32 + lane;
        const uint32_t idesc = idesc_bf16(TILE, CH);
        uint4 *stage = sOut + quarter * 32 * 8;
        int st = 0;
        uint32_t ph = 0;
        // the MMAs of the CTA's i-th tile, once it is built and its accumulator read out
        auto issue = [&](int i) {
            const int buf = i & 1;
            if (!mbar_wait(&full[st], ph) || !mbar_wait(&tempty[buf], ((i >> 1) & 1) ^ 1)) return false;
            // the tile's generic writes, ordered before this thread by the barrier, before the
            // MMA's reads (a fence in the gathering warps would wait for their rows in flight)
            proxy_fence();
            tc_fence_after();
            const uint32_t a0 = smem_u32(sA + st * FWD_TILE_BYTES), b0 = smem_u32(sW);
#pragma unroll
            for (int ks = 0; ks < CIN / 16; ++ks)
                mma_bf16(tmem + buf * CH, sdesc_sw128(a0 + (ks >> 2) * (TILE * 128) + (ks & 3) * 32),
                         sdesc(b0 + ks * 256, 128, CIN * 16), idesc, ks > 0);
            mma_commit(&empty[st]);
            mma_commit(&tfull[buf]);
            if (++st == STAGES) st = 0, ph ^= 1;
            return true;
        };
        const bool issuer = quarter == 0 && lane == 0;
        if (issuer && blockIdx.x < a.t.ntiles) failed = !issue(0);
        int it = 0;
        for (int64_t t = blockIdx.x; t < a.t.ntiles; t += gridDim.x, ++it) {
            const int buf = it & 1;
            if (issuer && !failed && t + gridDim.x < a.t.ntiles) failed = !issue(it + 1);
            __syncwarp();
            if (!__all_sync(0xffffffffu, !failed && mbar_wait(&tfull[buf], (it >> 1) & 1))) {
                failed = true;
                break;
            }
            tc_fence_after();
            const uint32_t lane_base = tmem + buf * CH + ((uint32_t)(quarter * 32) << 16);
            const int64_t p = t * TILE + r;
            float y0 = 0.f, y1 = 0.f;
#pragma unroll
            for (int c = 0; c < CH; c += 16) {
                float h[16];
                tmem_ld16(lane_base + c, h);
                if (c == CH - 16) {  // the accumulator has been read
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[buf]);
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) h[i] = fmaxf(h[i], 0.f);
                if (c == CH - 16) h[15] = 1.f;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int ch = (c >> 3) + u;
                    const uint4 packed = pack8(h + 8 * u);
                    // the warp's rows through shared memory (chunks XOR-swizzled by row), so
                    // that its stores are whole lines
                    if (MODE != FWD_LAST_PREDICT) stage[lane * 8 + (ch ^ (lane & 7))] = packed;
                    if (MODE != FWD_HIDDEN) {
                        // head on the stored (BF16-rounded) h^4
                        float f[8];
                        unpack8(packed, f);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            y0 = fmaf(sU[8 * ch + i], f[i], y0);
                            y1 = fmaf(sU[CH + 8 * ch + i], f[i], y1);
                        }
                    }
                }
            }
            if (MODE != FWD_HIDDEN && p < a.t.n) {
                float inv = 1.f / a.t.kdiag[p];
                if (MODE == FWD_LAST_TRAIN) {
                    a.xhat[p] = make_float2(y0 * inv, y1 * inv);
                } else {
                    double s = a.bn[0];
                    a.x0[p] = make_double2(s * (double)(y0 * inv), s * (double)(y1 * inv));
                }
            }
            if (MODE != FWD_LAST_PREDICT) {
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int idx = i * 32 + lane, rr = idx >> 3, c = idx & 7;
                    const int64_t node = t * TILE + quarter * 32 + rr;
                    if (node < a.t.n) a.Hout[node * 8 + c] = stage[rr * 8 + (c ^ (rr & 7))];
                }
                __syncwarp();
            }
        }
    }
    if (failed) atomicExch(a.err, 1);
    __syncthreads();
    if (warp == GW) tmem_free(tmem, 2 * CH);
}

// ------------------------------------------------------------------ loss and its gradient in x^
// r^ = b^ - J x^ (FP32 arithmetic), loss partials sum |V| |r^|^2
__global__ void k_resid(int64_t n, SellView<float2> K, const float *__restrict__ kdiag,
                        const float *__restrict__ volp, const double2 *__restrict__ psi,
                        const double2 *__restrict__ b, const double *__restrict__ bn,
                        const float2 *__restrict__ xh, float2 *__restrict__ r, double *part) {
    __shared__ double sh[32];
    double a = 0;
    float inv = (float)bn[1];
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        int64_t s = p >> 5;
        int lane = (int)(p & 31);
        int64_t beg = K.sptr[s];
        int w = (int)((K.sptr[s + 1] - beg) >> 5);
        float2 acc = make_float2(0.f, 0.f);
        for (int k = 0; k < w; ++k) {
            int64_t q = beg + (int64_t)k * SELL_C + lane;
            cfma(acc, K.val[q], xh[K.col[q]]);
        }
        float2 ps = to32(psi[p]);
        float2 x = xh[p];
        float a2 = ps.x * ps.x + ps.y * ps.y;
        float d = kdiag[p] - 1.f + 2.f * a2;
        // J x = offdiag + (K_ii - 1 + 2|psi|^2) x + psi^2 conj(x)
        float2 p2 = make_float2(ps.x * ps.x - ps.y * ps.y, 2.f * ps.x * ps.y);
        float jx = acc.x + d * x.x + (p2.x * x.x + p2.y * x.y);
        float jy = acc.y + d * x.y + (p2.y * x.x - p2.x * x.y);
        double2 bv = b[p];
        float2 rr = make_float2((float)(bv.x * inv) - jx, (float)(bv.y * inv) - jy);
        r[p] = rr;
        a += (double)volp[p] * ((double)rr.x * rr.x + (double)rr.y * rr.y);
    }
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// loss[slot] += scale * sum(part)
__global__ void k_loss_acc(const double *part, int np, double scale, double *loss, int slot) {
    __shared__ double sh[32];
    double a = 0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) a += part[i];
    double t = block_sum(a, sh);
    if (threadIdx.x == 0) loss[slot] += scale * t;
}

// dy = scale * (-2 |V| (J r^)) / K_ii   (Euclidean gradient of L in y)
__global__ void k_gout(int64_t n, SellView<float2> K, const float *__restrict__ kdiag, const float *__restrict__ volp,
                       const double2 *__restrict__ psi, const float2 *__restrict__ r, float scale,
                       float2 *__restrict__ dy) {
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    int64_t s = p >> 5;
    int lane = (int)(p & 31);
    int64_t beg = K.sptr[s];
    int w = (int)((K.sptr[s + 1] - beg) >> 5);
    float2 acc = make_float2(0.f, 0.f);
    for (int k = 0; k < w; ++k) {
        int64_t q = beg + (int64_t)k * SELL_C + lane;
        cfma(acc, K.val[q], r[K.col[q]]);
    }
    float2 ps = to32(psi[p]);
    float2 x = r[p];
    float a2 = ps.x * ps.x + ps.y * ps.y;
    float d = kdiag[p] - 1.f + 2.f * a2;
    float2 p2 = make_float2(ps.x * ps.x - ps.y * ps.y, 2.f * ps.x * ps.y);
    float jx = acc.x + d * x.x + (p2.x * x.x + p2.y * x.y);
    float jy = acc.y + d * x.y + (p2.y * x.x - p2.x * x.y);
    float f = -2.f * scale * volp[p] / kdiag[p];
    dy[p] = make_float2(f * jx, f * jy);
}

// dz^3 = (U^T dy) masked by h^4 > 0 (channel 63 -> 0), rounded to BF16, and the partials of
// dU = sum_i dy_i h4_i^T: eight threads a node, one 16-byte chunk of h^4 each, so that a
// warp reads whole lines.  63^3 nodes: 18 us (107 for dU alone when a block summed one node
// after the other).
__global__ void __launch_bounds__(256) k_head(int64_t n, const float2 *__restrict__ dy, const uint4 *__restrict__ H4,
                                              const float *__restrict__ U, uint4 *__restrict__ dZ,
                                              float *__restrict__ part) {
    __shared__ float sh[8][2 * CH];
    const int j = threadIdx.x & 7, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float u0[8], u1[8], d0[8], d1[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        u0[i] = U[8 * j + i];
        u1[i] = U[CH + 8 * j + i];
        d0[i] = d1[i] = 0.f;
    }
#pragma unroll 2
    for (int64_t p = blockIdx.x * 32 + (threadIdx.x >> 3); p < n; p += (int64_t)gridDim.x * 32) {
        const float2 g = dy[p];
        float f[8], dz[8];
        unpack8(__ldg(H4 + p * 8 + j), f);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            d0[i] = fmaf(g.x, f[i], d0[i]);
            d1[i] = fmaf(g.y, f[i], d1[i]);
            const float v = u0[i] * g.x + u1[i] * g.y;
            dz[i] = f[i] > 0.f ? v : 0.f;
        }
        if (j == 7) dz[7] = 0.f;
        dZ[p * 8 + j] = pack8(dz);
    }
    // the four nodes of a warp, then its block's warps, in a fixed order
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
        for (int m = 8; m < 32; m <<= 1) {
            d0[i] += __shfl_xor_sync(0xffffffffu, d0[i], m);
            d1[i] += __shfl_xor_sync(0xffffffffu, d1[i], m);
        }
        if (lane < 8) {
            sh[warp][8 * j + i] = d0[i];
            sh[warp][CH + 8 * j + i] = d1[i];
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 * CH) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += sh[w][threadIdx.x];
        part[(int64_t)blockIdx.x * 2 * CH + threadIdx.x] = t;
    }
}

// g += the sum of np partials of a gradient.  A warp takes 32 neighbouring parameters, its
// block's eight warps every eighth partial each (whole lines; one thread a parameter with
// the partials strided took 40 us for a W, this one 5).  W: partials are dW^T (128 in x
// 64 out), g is W's layout (64 out x 128 in).
template <bool W>
__global__ void __launch_bounds__(256) k_sum_parts(const float *__restrict__ part, int np, int width, float *g) {
    __shared__ float sh[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;  // (width is a multiple of 32)
    float t = 0.f;
#pragma unroll 4
    for (int b = warp; b < np; b += 8) t += __ldg(part + (int64_t)b * width + e);
    sh[warp][lane] = t;
    __syncthreads();
    if (warp == 0) {
        t = sh[0][lane];
#pragma unroll
        for (int w = 1; w < 8; ++w) t += sh[w][lane];
        g[W ? (e % CH) * CIN + e / CH : e] += t;
    }
}

// ------------------------------------------------------------------ backward layer
struct BwdArgs {
    TileArgs t;              // h^l (the operand a^l is rebuilt)
    const float *volp;
    const uint4 *dZ;         // dz^l rows (BF16, masked)
    const uint4 *Wbimg;      // 128 x 64 BF16 operand image of W^l (rows = inputs)
    float *dA;               // n x 128: [dA_self, dA_nbr / (K_ii |V_i|)]
    float *dWpart;           // grid x 128 x 64 (rows = inputs)
    int *err;
};

// One layer: dA = dz W and dW^T += a^T dz.  The same warps as in the forward layer build
// [h, S h] and dz tiles, one row of 128 swizzled bytes a node; the MMA of dA reads dz with
// the channels as K, that of dW reads both with the nodes as K (MN-major operands), so
// nothing is transposed on the way.  Bound by the gathers, as the forward layer, and the
// FP32 rows of dA (512 bytes a node), written through shared memory as whole lines.
// 63^3 nodes: 59 us, 43 for the first layer, which needs no dA (163 to 203 and 158 with one
// thread a node, whose rows and transposed two-byte stores met in the same banks).
constexpr int BWD_TILE_BYTES = 3 * TILE * 128;
constexpr int BWD_STAGES = 2;
constexpr int BWD_GW = fwd_gw(false), BWD_THREADS = fwd_threads(false);
constexpr int BWD_SMEM =
    BWD_STAGES * BWD_TILE_BYTES + CIN * CH * 2 + TILE * 128 + FWD_KSTAGES * FWD_K * TILE * 12;

template <bool NEED_DA>
__global__ void __launch_bounds__(BWD_THREADS, 1) k_bwd(BwdArgs a) {
    constexpr int GW = BWD_GW, STAGES = BWD_STAGES;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sA = smem;                                                     // STAGES x [h, S h, dz] x 128 x 64
    uint4 *sW = reinterpret_cast<uint4 *>(smem + STAGES * BWD_TILE_BYTES);        // 128 in x 64 out
    float4 *sOut = reinterpret_cast<float4 *>(sW + CIN * CH / 8);                 // 128 rows of 32 FP32
    float2 *sVal = reinterpret_cast<float2 *>(sOut + TILE * 8);
    int32_t *sCol = reinterpret_cast<int32_t *>(sVal + FWD_KSTAGES * FWD_K * TILE);
    __shared__ float sSc[FWD_KSTAGES][TILE];
    __shared__ int sWid[FWD_KSTAGES][TILE / SELL_C];
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2], kfull[FWD_KSTAGES],
        kempty[FWD_KSTAGES];
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (NEED_DA)
        for (int i = tid; i < CIN * CH / 8; i += BWD_THREADS) sW[i] = a.Wbimg[i];
    if (warp == GW) tmem_alloc(&tslot, 512);
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init_n(&full[i], GW);
            mbar_init_n(&empty[i], 1);
        }
        for (int i = 0; i < FWD_KSTAGES; ++i) {
            mbar_init_n(&kfull[i], 32);
            mbar_init_n(&kempty[i], GW);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init_n(&tfull[i], 1);
            mbar_init_n(&tempty[i], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    proxy_fence();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;  // two accumulators of dA (128 columns each), then dW^T (64)
    const uint32_t tm_dW = tmem + 2 * CIN;
    const TileBufs bufs{sA, sVal, sCol, sSc, sWid, full, empty, kfull, kempty};
    bool failed = false;
    if (warp < GW) {
        regs_raise<96>();
        failed = build_tiles<false, GW, STAGES, BWD_TILE_BYTES, true>(a.t, bufs, a.dZ, warp, lane);
    } else if (warp >= GW + 4) {
        regs_lower<32>();
        if (warp < GW + 4 + FWD_KSTAGES) failed = stage_entries(a.t, bufs, warp - GW - 4, lane);
    } else {
        regs_lower<64>();
        const int quarter = warp - GW;
        const uint32_t id_dA = idesc_bf16(TILE, CIN);                               // 128 nodes x 128 inputs
        const uint32_t id_dW = idesc_bf16(CIN, CH) | (1u << 15) | (1u << 16);       // 128 inputs x 64 outputs, MN-major
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        int st = 0;
        uint32_t ph = 0;
        auto issue = [&](int i) {
            const int buf = i & 1;
            if (!mbar_wait(&full[st], ph) || !mbar_wait(&tempty[buf], ((i >> 1) & 1) ^ 1)) return false;
            proxy_fence();
            tc_fence_after();
            const uint32_t a0 = smem_u32(sA + st * BWD_TILE_BYTES), dz0 = a0 + 2 * TILE * 128, b0 = smem_u32(sW);
            if (NEED_DA) {
#pragma unroll
                for (int ks = 0; ks < CH / 16; ++ks)
                    mma_bf16(tmem + buf * CIN, sdesc_sw128(dz0 + ks * 32), sdesc(b0 + ks * 256, 128, CH * 16), id_dA,
                             ks > 0);
            }
#pragma unroll
            for (int ks = 0; ks < TILE / 16; ++ks)
                mma_bf16(tm_dW, sdesc_sw128(a0 + ks * 16 * 128, TILE * 128), sdesc_sw128(dz0 + ks * 16 * 128, TILE * 128),
                         id_dW, (ks > 0 || i > 0) ? 1u : 0u);
            mma_commit(&empty[st]);
            mma_commit(&tfull[buf]);
            if (++st == STAGES) st = 0, ph ^= 1;
            return true;
        };
        const bool issuer = quarter == 0 && lane == 0;
        if (issuer && blockIdx.x < a.t.ntiles) failed = !issue(0);
        int it = 0;
        for (int64_t t = blockIdx.x; t < a.t.ntiles; t += gridDim.x, ++it) {
            const int buf = it & 1;
            if (issuer && !failed && t + gridDim.x < a.t.ntiles) failed = !issue(it + 1);
            __syncwarp();
            if (!__all_sync(0xffffffffu, !failed && mbar_wait(&tfull[buf], (it >> 1) & 1))) {
                failed = true;
                break;
            }
            tc_fence_after();
            if (!NEED_DA) {
                // nothing to read, but the issuer must not get two tiles ahead of this warp:
                // tfull's parity would have turned twice and the wait above would miss both
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[buf]);
                continue;
            }
            const int64_t p = t * TILE + quarter * 32 + lane;
            const float sn = p < a.t.n ? 1.f / (a.t.kdiag[p] * a.volp[p]) : 0.f;
            float4 *stage = sOut + quarter * 32 * 8;
#pragma unroll
            for (int c = 0; c < CIN; c += 32) {
                // 32 columns of the warp's rows through shared memory (chunks XOR-swizzled
                // by row): stores of whole 128-byte lines
                const float f = c < CH ? 1.f : sn;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float v[16];
                    tmem_ld16(lane_base + buf * CIN + c + 16 * u, v);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        stage[lane * 8 + ((4 * u + i) ^ (lane & 7))] =
                            make_float4(v[4 * i] * f, v[4 * i + 1] * f, v[4 * i + 2] * f, v[4 * i + 3] * f);
                }
                if (c == CIN - 32) {  // the accumulator has been read
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[buf]);
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = i * 4 + (lane >> 3), ch = lane & 7;
                    const int64_t node = t * TILE + quarter * 32 + rr;
                    if (node < a.t.n)
                        *reinterpret_cast<float4 *>(a.dA + node * CIN + c + 4 * ch) = stage[rr * 8 + (ch ^ (rr & 7))];
                }
                __syncwarp();
            }
        }
        // dW^T partial of this CTA: lane = input feature, 64 output columns
        const bool ok = it > 0 && !failed;
        float *dst = a.dWpart + ((int64_t)blockIdx.x * CIN + quarter * 32 + lane) * CH;
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < CH; c += 16) {
            float v[16];
            tmem_ld16(tm_dW + ((uint32_t)(quarter * 32) << 16) + c, v);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                *reinterpret_cast<float4 *>(dst + c + 4 * i) =
                    ok ? make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        tc_fence_before();
    }
    if (failed) atomicExch(a.err, 1);
    __syncthreads();
    if (warp == GW) tmem_free(tmem, 512);
}

// dz^{l-1}_k = (dA_self_k - |V_k| sum_i K_ki dA~_i) masked by h^l_k > 0 (channel 63 -> 0).
// Bound by the latency of its gathers of 256-byte rows (0.44 GB from L2 at 63^3 nodes):
// sixteen threads a node, one 16-byte chunk each, all of a batch's rows requested at once.
// 82 us, 124 with one thread a node.  Fewer registers for more warps spill (104), several
// slices a block one after the other share rows in L1 but wait longer (137).
constexpr int DH_BATCH = 6;
__global__ void __launch_bounds__(256, 4) k_dh(int64_t n, SellView<float2> K, const float *__restrict__ volp,
                                            const float *__restrict__ dA, const uint2 *__restrict__ Hl,
                                            uint2 *__restrict__ dZ) {
    const int64_t p = blockIdx.x * (int64_t)16 + (threadIdx.x >> 4);
    const int j = threadIdx.x & 15;
    if (p >= n) return;
    const int64_t s = p >> 5, beg = K.sptr[s] + (p & 31);
    const int w = (int)((K.sptr[s + 1] - K.sptr[s]) >> 5);
    const float4 *rows = reinterpret_cast<const float4 *>(dA) + j;
    const float4 self = __ldg(rows + p * (CIN / 4));
    const uint2 h = __ldg(Hl + p * 16 + j);
    const float vk = -volp[p];
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k0 = 0; k0 < w; k0 += DH_BATCH) {
        float2 kv[DH_BATCH];
        float4 u[DH_BATCH];
#pragma unroll
        for (int k = 0; k < DH_BATCH; ++k)
            if (k0 + k < w) {
                const int64_t q = beg + (int64_t)(k0 + k) * SELL_C;
                kv[k] = __ldg(K.val + q);
                u[k] = __ldg(rows + (int64_t)__ldg(K.col + q) * (CIN / 4) + CH / 4);
            }
#pragma unroll
        for (int k = 0; k < DH_BATCH; ++k)
            if (k0 + k < w && (kv[k].x != 0.f || kv[k].y != 0.f)) {
                acc[0] += kv[k].x * u[k].x - kv[k].y * u[k].y;
                acc[1] += kv[k].x * u[k].y + kv[k].y * u[k].x;
                acc[2] += kv[k].x * u[k].z - kv[k].y * u[k].w;
                acc[3] += kv[k].x * u[k].w + kv[k].y * u[k].z;
            }
    }
    const float sv[4] = {self.x, self.y, self.z, self.w};
    const uint32_t hw[2] = {h.x, h.y};
    float o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float hf = __uint_as_float((i & 1) ? (hw[i >> 1] & 0xffff0000u) : (hw[i >> 1] << 16));
        const float g = sv[i] + vk * acc[i];
        o[i] = hf > 0.f ? g : 0.f;
    }
    if (j == 15) o[3] = 0.f;
    const __nv_bfloat162 lo = __floats2bfloat162_rn(o[0], o[1]), hi = __floats2bfloat162_rn(o[2], o[3]);
    dZ[p * 16 + j] = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
}

// ------------------------------------------------------------------ zero-guess fallback
// per-block partials of sum |V| |b - J x|^2 and sum |V| |b|^2 (FP64 J)
__global__ void k_fallback_part(int64_t n, SellView<double2> K, const double *__restrict__ kdiag,
                                const double *__restrict__ volp, const double2 *__restrict__ psi,
                                const double2 *__restrict__ b, const double2 *__restrict__ x, double *part) {
    __shared__ double sh[32];
    double rr = 0, bb = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        int64_t s = p >> 5;
        int lane = (int)(p & 31);
        int64_t beg = K.sptr[s];
        int w = (int)((K.sptr[s + 1] - beg) >> 5);
        double2 acc = make_double2(0.0, 0.0);
        for (int k = 0; k < w; ++k) {
            int64_t q = beg + (int64_t)k * SELL_C + lane;
            cfma(acc, K.val[q], x[K.col[q]]);
        }
        double2 ps = psi[p], xv = x[p], bv = b[p];
        double d = kdiag[p] - 1.0 + 2.0 * (ps.x * ps.x + ps.y * ps.y);
        double p2r = ps.x * ps.x - ps.y * ps.y, p2i = 2.0 * ps.x * ps.y;
        double jx = acc.x + d * xv.x + (p2r * xv.x + p2i * xv.y);
        double jy = acc.y + d * xv.y + (p2i * xv.x - p2r * xv.y);
        double rx = bv.x - jx, ry = bv.y - jy;
        rr += volp[p] * (rx * rx + ry * ry);
        bb += volp[p] * (bv.x * bv.x + bv.y * bv.y);
    }
    double t1 = block_sum(rr, sh);
    double t2 = block_sum(bb, sh);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = t1;
        part[2 * blockIdx.x + 1] = t2;
    }
}
// flag = 1 if the guess lowers the residual below ||b||_D (and is finite)
__global__ void k_fallback_decide(const double *part, int np, int *flag) {
    __shared__ double sh[32];
    double a = 0, c = 0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) {
        a += part[2 * i];
        c += part[2 * i + 1];
    }
    double rr = block_sum(a, sh);
    double bb = block_sum(c, sh);
    if (threadIdx.x == 0) *flag = (rr < bb) ? 1 : 0;   // false for NaN
}
__global__ void k_fallback_apply(int64_t n, const int *flag, double2 *x) {
    if (*flag) return;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
        x[p] = make_double2(0.0, 0.0);
}

// ------------------------------------------------------------------ parameters
__global__ void k_adam(int np, float *th, const float *g, float *m, float *v, float lr, float b1, float b2, float c1,
                       float c2, float eps) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    float gi = g[i];
    float mi = b1 * m[i] + (1.f - b1) * gi;
    float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    th[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// BF16 operand images of every W^l: forward (rows = 64 outputs, K = 128 inputs)
// and backward (rows = 128 inputs, K = 64 outputs)
__global__ void k_pack(const float *th, __nv_bfloat16 *Wf, __nv_bfloat16 *Wb) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= NL * WSZ) return;
    int l = idx / WSZ, r = idx % WSZ;
    int o = r / CIN, i = r % CIN;
    __nv_bfloat16 v = __float2bfloat16_rn(th[idx]);
    Wf[(int64_t)l * WSZ + cm_off(o, i, CIN)] = v;
    Wb[(int64_t)l * WSZ + cm_off(i, o, CH)] = v;
}

}  // namespace ws
}  // namespace gl

using namespace gl;
using namespace gl::ws;

struct gl_warmstart_s {
    DBuf<float> theta, grad, m, v;
    DBuf<__nv_bfloat16> Wf, Wb;
    int64_t t = 0;           // Adam step count
    int64_t cap = 0;         // nodes the work buffers hold
    DBuf<__nv_bfloat16> H;   // 5 x cap x 64
    DBuf<__nv_bfloat16> dZ;  // cap x 64
    DBuf<float> dA;          // cap x 128
    DBuf<float2> xh, r, dy;
    DBuf<double> bn, part, loss;
    DBuf<float> dWpart, dUpart;
    DBuf<int> err;
    DBuf<int> used;          // zero-guess fallback decision of the last solve
    DBuf<double> fpart;      // its partials
    // the hint: J a, the residual r = b - alpha J a, the hint in the solve ordering,
    // partials and (alpha, 1 / ||a||_D)
    DBuf<double2> qa, rb, hp;
    DBuf<double> hpart, hsc;
    int grid = 0;   // blocks of a layer's kernel
};

namespace {

template <typename F>
gl_status ws_guard(F &&f) {
    try {
        set_error("");
        return f();
    } catch (const Error &e) {
        set_error(e.msg);
        return e.code;
    } catch (const std::bad_alloc &) {
        set_error("host allocation failed");
        return GL_ERR_OOM;
    }
}

cudaStream_t as_stream(void *s) { return reinterpret_cast<cudaStream_t>(s); }

void ws_pack(gl_warmstart_s *w, cudaStream_t s) {
    k_pack<<<grid_for(NL * WSZ, 256), 256, 0, s>>>(w->theta.get(), w->Wf.get(), w->Wb.get());
    GL_LAUNCH_CHECK();
}

void ws_reserve(gl_warmstart_s *w, int64_t n) {
    if (n <= w->cap) return;
    w->H.alloc((size_t)5 * n * CH);
    w->dZ.alloc((size_t)n * CH);
    w->dA.alloc((size_t)n * CIN);
    w->xh.alloc(n);
    w->r.alloc(n);
    w->dy.alloc(n);
    w->qa.alloc(n);
    w->rb.alloc(n);
    w->hp.alloc(n);
    w->cap = n;
}

void ws_setup_kernels(gl_warmstart_s *w) {
    if (w->grid) return;
    GL_CUDA(cudaFuncSetAttribute(k_fwd<FWD_HIDDEN, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd_smem(true)));
    for (const void *fn : {(const void *)k_fwd<FWD_HIDDEN, false>, (const void *)k_fwd<FWD_LAST_TRAIN, false>,
                           (const void *)k_fwd<FWD_LAST_PREDICT, false>})
        GL_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd_smem(false)));
    GL_CUDA(cudaFuncSetAttribute(k_bwd<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, BWD_SMEM));
    GL_CUDA(cudaFuncSetAttribute(k_bwd<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, BWD_SMEM));
    int dev = 0, nsm = 0;
    GL_CUDA(cudaGetDevice(&dev));
    GL_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    w->grid = nsm;  // one CTA per SM
    w->part.alloc(RED_BLOCKS);
    w->bn.alloc(2);
    w->dWpart.alloc((size_t)w->grid * CIN * CH);
    w->dUpart.alloc((size_t)DU_BLOCKS * 128);
    w->err.alloc(1);
    GL_CUDA(cudaMemset(w->err.get(), 0, sizeof(int)));
    w->used.alloc(1);
    w->fpart.alloc(2 * RED_BLOCKS);
    w->hpart.alloc(3 * RED_BLOCKS);
    w->hsc.alloc(2);
}

// with a hint (solve ordering): alpha and 1 / ||a||_D into hsc, and the residual
// b - alpha J a the network works on; returns the right-hand side to use
const double2 *ws_hint(gl_warmstart_s *w, gl_mesh_s *m, const double2 *psi_p, const double2 *b_p,
                       const double2 *hint_p, cudaStream_t s) {
    if (!hint_p) return b_p;
    const int64_t n = m->n;
    jacobian_apply_p(m, psi_p, hint_p, w->qa.get(), s);
    note_launch(3);
    k_hint_part<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, m->volp.get(), w->qa.get(), b_p, hint_p, w->hpart.get());
    k_hint_final<<<1, 1024, 0, s>>>(w->hpart.get(), w->hsc.get());
    k_hint_resid<<<grid_for(n, 256), 256, 0, s>>>(n, w->hsc.get(), b_p, w->qa.get(), w->rb.get());
    GL_LAUNCH_CHECK();
    return w->rb.get();
}

__nv_bfloat16 *Hbuf(gl_warmstart_s *w, int l) { return w->H.get() + (size_t)l * w->cap * CH; }

// forward pass in the solve ordering; train: keep h^1..h^4 and x^, else write x0.
// b_p is the network's right-hand side (the residual the hint leaves, when there
// is one: see ws_hint); hint_p (nullable) fills the hint channels
void ws_forward(gl_warmstart_s *w, gl_mesh_s *m, const double2 *psi_p, const double2 *b_p, bool train, double2 *x0_p,
                cudaStream_t s, const double2 *hint_p = nullptr) {
    const int64_t n = m->n;
    k_bnorm_part<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, m->volp.get(), b_p, w->part.get());
    k_bnorm_final<<<1, 1024, 0, s>>>(w->part.get(), RED_BLOCKS, w->bn.get());
    k_features<<<grid_for(n, 256), 256, 0, s>>>(n, b_p, psi_p, w->bn.get(), hint_p, w->hsc.get(),
                                                reinterpret_cast<uint4 *>(Hbuf(w, 0)), train ? 0 : 1);
    GL_LAUNCH_CHECK();
    note_launch(3);
    const int64_t ntiles = (n + TILE - 1) / TILE;
    const int grid = (int)std::min<int64_t>(ntiles, w->grid);
    // algorithmic bytes of one layer: each node's h row read once (neighbour rows
    // are re-reads of the same array), its K row (value + column) and K_ii, and
    // the written h row (the last layer of a prediction writes x0 instead)
    const double k_bytes = (double)m->K32.nnz_stored * (sizeof(float2) + 4) + (double)n * 4;
    for (int l = 0; l < NL; ++l) {
        const bool last_pred = (l == NL - 1) && !train;
        ProfScope ps("wsf", (double)n * (CH * 2 + (last_pred ? 16 : CH * 2)) + k_bytes, s);
        FwdArgs a{};
        a.t.n = n;
        a.t.ntiles = ntiles;
        a.t.K = m->K32.view();
        a.t.kdiag = m->kdiag32.get();
        // prediction ping-pongs between buffers 0 and 1
        int in = train ? l : (l & 1), out = train ? l + 1 : ((l + 1) & 1);
        a.t.Hin = reinterpret_cast<const uint4 *>(Hbuf(w, in));
        a.Hout = reinterpret_cast<uint4 *>(Hbuf(w, out));
        a.Wimg = reinterpret_cast<const uint4 *>(w->Wf.get() + (size_t)l * WSZ);
        a.U = w->theta.get() + NL * WSZ;
        a.xhat = w->xh.get();
        a.x0 = x0_p;
        a.bn = w->bn.get();
        a.err = w->err.get();
        if (l == 0 && !train)
            k_fwd<FWD_HIDDEN, true><<<grid, fwd_threads(true), fwd_smem(true), s>>>(a);
        else if (l < NL - 1)
            k_fwd<FWD_HIDDEN, false><<<grid, fwd_threads(false), fwd_smem(false), s>>>(a);
        else if (train)
            k_fwd<FWD_LAST_TRAIN, false><<<grid, fwd_threads(false), fwd_smem(false), s>>>(a);
        else
            k_fwd<FWD_LAST_PREDICT, false><<<grid, fwd_threads(false), fwd_smem(false), s>>>(a);
        GL_LAUNCH_CHECK();
    }
}

// loss (added to loss[slot] with weight `scale`) and gradient (added to grad with
// weight `scale`) of one sample; requires ws_forward(train = true) just before
void ws_backward(gl_warmstart_s *w, gl_mesh_s *m, const double2 *psi_p, const double2 *b_p, double scale,
                 double *loss, int slot, cudaStream_t s) {
    const int64_t n = m->n;
    note_launch(5);
    k_resid<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, m->K32.view(), m->kdiag32.get(), m->volp32.get(), psi_p, b_p,
                                               w->bn.get(), w->xh.get(), w->r.get(), w->part.get());
    k_loss_acc<<<1, 1024, 0, s>>>(w->part.get(), RED_BLOCKS, scale, loss, slot);
    k_gout<<<grid_for(n, 256), 256, 0, s>>>(n, m->K32.view(), m->kdiag32.get(), m->volp32.get(), psi_p, w->r.get(),
                                            (float)scale, w->dy.get());
    float *gU = w->grad.get() + NL * WSZ;
    k_head<<<DU_BLOCKS, 256, 0, s>>>(n, w->dy.get(), reinterpret_cast<const uint4 *>(Hbuf(w, NL)),
                                     w->theta.get() + NL * WSZ, reinterpret_cast<uint4 *>(w->dZ.get()),
                                     w->dUpart.get());
    k_sum_parts<false><<<2 * CH / 32, 256, 0, s>>>(w->dUpart.get(), DU_BLOCKS, 2 * CH, gU);
    GL_LAUNCH_CHECK();
    const int64_t ntiles = (n + TILE - 1) / TILE;
    const int grid = (int)std::min<int64_t>(ntiles, w->grid);
    const double k_bytes = (double)m->K32.nnz_stored * (sizeof(float2) + 4) + (double)n * 8;
    for (int l = NL - 1; l >= 0; --l) {
        // algorithmic bytes: h^l and dz rows read, K row, dA rows written
        note_launch(l > 0 ? 2 : 1);
        BwdArgs a{};
        a.t.n = n;
        a.t.ntiles = ntiles;
        a.t.K = m->K32.view();
        a.t.kdiag = m->kdiag32.get();
        a.t.Hin = reinterpret_cast<const uint4 *>(Hbuf(w, l));
        a.volp = m->volp32.get();
        a.dZ = reinterpret_cast<const uint4 *>(w->dZ.get());
        a.Wbimg = reinterpret_cast<const uint4 *>(w->Wb.get() + (size_t)l * WSZ);
        a.dA = w->dA.get();
        a.dWpart = w->dWpart.get();
        a.err = w->err.get();
        {
            // algorithmic bytes: h^l and dz rows read, K row, dA rows written
            ProfScope ps("wsb", (double)n * (CH * 2 + CH * 2 + (l > 0 ? CIN * 4 : 0)) + k_bytes, s);
            if (l > 0)
                k_bwd<true><<<grid, BWD_THREADS, BWD_SMEM, s>>>(a);
            else
                k_bwd<false><<<grid, BWD_THREADS, BWD_SMEM, s>>>(a);
        }
        GL_LAUNCH_CHECK();
        k_sum_parts<true><<<WSZ / 32, 256, 0, s>>>(w->dWpart.get(), grid, WSZ, w->grad.get() + (size_t)l * WSZ);
        GL_LAUNCH_CHECK();
        if (l > 0) {
            k_dh<<<(unsigned)((n + 15) / 16), 256, 0, s>>>(n, m->K32.view(), m->volp32.get(), w->dA.get(),
                                                  reinterpret_cast<const uint2 *>(Hbuf(w, l)),
                                                  reinterpret_cast<uint2 *>(w->dZ.get()));
            GL_LAUNCH_CHECK();
        }
    }
}

void check_err(gl_warmstart_s *w, cudaStream_t s) {
    int e = 0;
    GL_CUDA(cudaMemcpyAsync(&e, w->err.get(), sizeof(int), cudaMemcpyDeviceToHost, s));
    GL_CUDA(cudaStreamSynchronize(s));
    if (e) {
        GL_CUDA(cudaMemsetAsync(w->err.get(), 0, sizeof(int), s));
        throw Error{GL_ERR_TIMEOUT, "warm-start network: a tensor-core completion wait ran out"};
    }
}

void ensure_mesh_scratch(gl_mesh_s *m) {
    if (m->t0.n != (size_t)m->n) {
        m->t0.alloc(m->n);
        m->t1.alloc(m->n);
        m->t2.alloc(m->n);
    }
}

}  // namespace

namespace gl {

// x0_p = network guess for b_p (solve ordering; hint_p nullable, solve ordering)
void warmstart_predict_p(gl_warmstart_s *w, gl_mesh_s *m, const double2 *psi_p, const double2 *b_p, double2 *x0_p,
                         cudaStream_t s, const double2 *hint_p) {
    mesh_ensure_fp32(m, s);
    ws_setup_kernels(w);
    ws_reserve(w, m->n);
    const double2 *r_p = ws_hint(w, m, psi_p, b_p, hint_p, s);
    ws_forward(w, m, psi_p, r_p, false, x0_p, s, hint_p);
    if (hint_p) {
        note_launch();
        k_hint_add<<<grid_for(m->n, 256), 256, 0, s>>>(m->n, w->hsc.get(), hint_p, x0_p);
        GL_LAUNCH_CHECK();
    }
}

void warmstart_apply_p(gl_warmstart_s *w, gl_mesh_s *m, const double2 *psi_p, const double2 *b_p, double2 *x_p,
                       cudaStream_t s, const double2 *hint_nat) {
    const double2 *hint_p = nullptr;
    if (hint_nat) {
        ws_reserve(w, m->n);
        permute_in(m->n, m->perm.get(), hint_nat, w->hp.get(), s);
        hint_p = w->hp.get();
    }
    warmstart_predict_p(w, m, psi_p, b_p, x_p, s, hint_p);
    note_launch(3);
    k_fallback_part<<<RED_BLOCKS, RED_THREADS, 0, s>>>(m->n, m->K.view(), m->kdiag.get(), m->volp.get(), psi_p, b_p,
                                                       x_p, w->fpart.get());
    k_fallback_decide<<<1, 1024, 0, s>>>(w->fpart.get(), RED_BLOCKS, w->used.get());
    k_fallback_apply<<<grid_for(m->n, 256, 4 * NUM_SMS_HINT), 256, 0, s>>>(m->n, w->used.get(), x_p);
    GL_LAUNCH_CHECK();
}

// the hint's minimal-residual multiple alone (no network): x_p = alpha a with
// alpha = <J a, b>_R / <J a, J a>_R, which is never a worse guess than zero
void hint_guess_p(gl_mesh_s *m, const double2 *psi_p, const double2 *b_p, const double2 *hint_nat, double2 *x_p,
                  cudaStream_t s) {
    struct HintWork {
        DBuf<double2> a, q;
        DBuf<double> part, hs;
    };
    static thread_local HintWork H;
    const int64_t n = m->n;
    if (H.a.n != (size_t)n) {
        H.a.alloc(n);
        H.q.alloc(n);
    }
    if (!H.part.get()) {
        H.part.alloc(3 * RED_BLOCKS);
        H.hs.alloc(2);
    }
    permute_in(n, m->perm.get(), hint_nat, H.a.get(), s);
    jacobian_apply_p(m, psi_p, H.a.get(), H.q.get(), s);
    note_launch(3);
    k_hint_part<<<RED_BLOCKS, RED_THREADS, 0, s>>>(n, m->volp.get(), H.q.get(), b_p, H.a.get(), H.part.get());
    k_hint_final<<<1, 1024, 0, s>>>(H.part.get(), H.hs.get());
    k_hint_set<<<grid_for(n, 256), 256, 0, s>>>(n, H.hs.get(), H.a.get(), x_p);
    GL_LAUNCH_CHECK();
}

int warmstart_used(gl_warmstart_s *w, cudaStream_t s) {
    check_err(w, s);
    int u = 0;
    GL_CUDA(cudaMemcpyAsync(&u, w->used.get(), sizeof(int), cudaMemcpyDeviceToHost, s));
    GL_CUDA(cudaStreamSynchronize(s));
    return u;
}

}  // namespace gl

extern "C" {

gl_status gl_warmstart_create(const float *params, gl_warmstart *out) {
    return ws_guard([&] {
        GL_REQUIRE(out, GL_ERR_ARG, "out must not be NULL");
        auto *w = new gl_warmstart_s();
        try {
            w->theta.alloc(NPARAM);
            w->grad.alloc(NPARAM);
            w->m.alloc(NPARAM);
            w->v.alloc(NPARAM);
            w->Wf.alloc((size_t)NL * WSZ);
            w->Wb.alloc((size_t)NL * WSZ);
            w->loss.alloc(1);
            if (params)
                GL_CUDA(cudaMemcpy(w->theta.get(), params, NPARAM * sizeof(float), cudaMemcpyHostToDevice));
            else
                GL_CUDA(cudaMemset(w->theta.get(), 0, NPARAM * sizeof(float)));
            GL_CUDA(cudaMemset(w->grad.get(), 0, NPARAM * sizeof(float)));
            GL_CUDA(cudaMemset(w->m.get(), 0, NPARAM * sizeof(float)));
            GL_CUDA(cudaMemset(w->v.get(), 0, NPARAM * sizeof(float)));
            ws_pack(w, 0);
            GL_CUDA(cudaDeviceSynchronize());
        } catch (...) {
            delete w;
            throw;
        }
        *out = w;
        return GL_OK;
    });
}

gl_status gl_warmstart_destroy(gl_warmstart w) {
    return ws_guard([&] {
        if (w) {
            cudaDeviceSynchronize();
            delete w;
        }
        return GL_OK;
    });
}

gl_status gl_warmstart_get_params(gl_warmstart w, float *params) {
    return ws_guard([&] {
        GL_REQUIRE(w && params, GL_ERR_ARG, "NULL argument");
        GL_CUDA(cudaMemcpy(params, w->theta.get(), NPARAM * sizeof(float), cudaMemcpyDeviceToHost));
        return GL_OK;
    });
}

gl_status gl_warmstart_set_params(gl_warmstart w, const float *params) {
    return ws_guard([&] {
        GL_REQUIRE(w && params, GL_ERR_ARG, "NULL argument");
        GL_CUDA(cudaMemcpy(w->theta.get(), params, NPARAM * sizeof(float), cudaMemcpyHostToDevice));
        GL_CUDA(cudaMemset(w->m.get(), 0, NPARAM * sizeof(float)));
        GL_CUDA(cudaMemset(w->v.get(), 0, NPARAM * sizeof(float)));
        w->t = 0;
        ws_pack(w, 0);
        GL_CUDA(cudaDeviceSynchronize());
        return GL_OK;
    });
}

gl_status gl_warmstart_predict(gl_warmstart w, gl_mesh m, const void *psi, const void *b, const void *hint, void *x0,
                               void *stream) {
    return ws_guard([&] {
        GL_REQUIRE(w && m && psi && b && x0, GL_ERR_ARG, "NULL argument");
        cudaStream_t s = as_stream(stream);
        ensure_mesh_scratch(m);
        permute_in(m->n, m->perm.get(), (const double2 *)psi, m->t0.get(), s);
        permute_in(m->n, m->perm.get(), (const double2 *)b, m->t1.get(), s);
        const double2 *hp = nullptr;
        if (hint) {
            ws_setup_kernels(w);
            ws_reserve(w, m->n);
            permute_in(m->n, m->perm.get(), (const double2 *)hint, w->hp.get(), s);
            hp = w->hp.get();
        }
        warmstart_predict_p(w, m, m->t0.get(), m->t1.get(), m->t2.get(), s, hp);
        permute_out(m->n, m->perm.get(), m->t2.get(), (double2 *)x0, s);
        check_err(w, s);
        return GL_OK;
    });
}

gl_status gl_warmstart_grad(gl_warmstart w, gl_mesh m, const void *psi, const void *b, const void *hint,
                            float *grad_host, double *loss_out, void *stream) {
    return ws_guard([&] {
        GL_REQUIRE(w && m && psi && b, GL_ERR_ARG, "NULL argument");
        cudaStream_t s = as_stream(stream);
        ensure_mesh_scratch(m);
        mesh_ensure_fp32(m, s);
        ws_setup_kernels(w);
        ws_reserve(w, m->n);
        permute_in(m->n, m->perm.get(), (const double2 *)psi, m->t0.get(), s);
        permute_in(m->n, m->perm.get(), (const double2 *)b, m->t1.get(), s);
        const double2 *hp = nullptr;
        if (hint) {
            permute_in(m->n, m->perm.get(), (const double2 *)hint, w->hp.get(), s);
            hp = w->hp.get();
        }
        GL_CUDA(cudaMemsetAsync(w->grad.get(), 0, NPARAM * sizeof(float), s));
        GL_CUDA(cudaMemsetAsync(w->loss.get(), 0, sizeof(double), s));
        const double2 *r_p = ws_hint(w, m, m->t0.get(), m->t1.get(), hp, s);
        ws_forward(w, m, m->t0.get(), r_p, true, nullptr, s, hp);
        ws_backward(w, m, m->t0.get(), r_p, 1.0, w->loss.get(), 0, s);
        check_err(w, s);
        if (grad_host) GL_CUDA(cudaMemcpy(grad_host, w->grad.get(), NPARAM * sizeof(float), cudaMemcpyDeviceToHost));
        if (loss_out) GL_CUDA(cudaMemcpy(loss_out, w->loss.get(), sizeof(double), cudaMemcpyDeviceToHost));
        return GL_OK;
    });
}

gl_status gl_warmstart_train(gl_warmstart w, int count, const gl_mesh *meshes, const void *const *psi,
                             const void *const *b, const void *const *hints, int steps, int batch, float lr,
                             double *loss_out, void *stream) {
    return ws_guard([&] {
        GL_REQUIRE(w && meshes && psi && b, GL_ERR_ARG, "NULL argument");
        GL_REQUIRE(count > 0 && steps >= 0 && batch > 0 && lr > 0, GL_ERR_ARG, "bad count, steps, batch or lr");
        cudaStream_t s = as_stream(stream);
        ws_setup_kernels(w);
        for (int j = 0; j < count; ++j) {
            GL_REQUIRE(meshes[j] && psi[j] && b[j], GL_ERR_ARG, "NULL sample");
            ensure_mesh_scratch(meshes[j]);
            mesh_ensure_fp32(meshes[j], s);
            ws_reserve(w, meshes[j]->n);
        }
        DBuf<double> losses(std::max(steps, 1));
        GL_CUDA(cudaMemsetAsync(losses.get(), 0, losses.bytes(), s));
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        for (int st = 0; st < steps; ++st) {
            GL_CUDA(cudaMemsetAsync(w->grad.get(), 0, NPARAM * sizeof(float), s));
            for (int j = 0; j < batch; ++j) {
                int k = (int)(((int64_t)st * batch + j) % count);
                gl_mesh_s *m = meshes[k];
                permute_in(m->n, m->perm.get(), (const double2 *)psi[k], m->t0.get(), s);
                permute_in(m->n, m->perm.get(), (const double2 *)b[k], m->t1.get(), s);
                const double2 *hp = nullptr;
                if (hints && hints[k]) {
                    permute_in(m->n, m->perm.get(), (const double2 *)hints[k], w->hp.get(), s);
                    hp = w->hp.get();
                }
                const double2 *r_p = ws_hint(w, m, m->t0.get(), m->t1.get(), hp, s);
                ws_forward(w, m, m->t0.get(), r_p, true, nullptr, s, hp);
                ws_backward(w, m, m->t0.get(), r_p, 1.0 / batch, losses.get(), st, s);
            }
            w->t += 1;
            float c1 = 1.f - powf(b1, (float)w->t), c2 = 1.f - powf(b2, (float)w->t);
            k_adam<<<grid_for(NPARAM, 256), 256, 0, s>>>(NPARAM, w->theta.get(), w->grad.get(), w->m.get(),
                                                         w->v.get(), lr, b1, b2, c1, c2, eps);
            GL_LAUNCH_CHECK();
            ws_pack(w, s);
            if ((st & 15) == 15) check_err(w, s);
        }
        check_err(w, s);
        if (loss_out && steps > 0)
            GL_CUDA(cudaMemcpy(loss_out, losses.get(), steps * sizeof(double), cudaMemcpyDeviceToHost));
        return GL_OK;
    });
}

gl_status gl_warmstart_adam_step(gl_warmstart w, const float *grad_host, float lr) {
    return ws_guard([&] {
        GL_REQUIRE(w && grad_host && lr > 0, GL_ERR_ARG, "bad argument");
        GL_CUDA(cudaMemcpy(w->grad.get(), grad_host, NPARAM * sizeof(float), cudaMemcpyHostToDevice));
        w->t += 1;
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        float c1 = 1.f - powf(b1, (float)w->t), c2 = 1.f - powf(b2, (float)w->t);
        k_adam<<<grid_for(NPARAM, 256), 256>>>(NPARAM, w->theta.get(), w->grad.get(), w->m.get(), w->v.get(), lr, b1,
                                               b2, c1, c2, eps);
        GL_LAUNCH_CHECK();
        ws_pack(w, 0);
        GL_CUDA(cudaDeviceSynchronize());
        return GL_OK;
    });
}

}  // extern "C"
