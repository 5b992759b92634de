// gl_sweep.cu -- the multicolour symmetric Gauss-Seidel steps of the V-cycle's
// many-coloured levels (Sec. 4: one pre- and one post-step per level), each a
// single launch, with the residual that follows the pre-step: the coarse levels,
// and the finest level of a general simplicial mesh up to the sizes of sweep_finest (on a
// lattice the finest level is red-black: three large launches, gl_vcycle.cu).
//
// A level's operator is stored by rows with the entries of lower colours (solve
// positions below the row's own) first and those of higher colours behind them.
// With the row sums split the same way, one symmetric step is
//   pre-pass (nonzero guess):     t_i = b_i - sum_upper A_ik x_k      (else t_i = b_i)
//   forward, colours ascending:   x_i = (t_i - sum_lower A_ik x_k) / A_ii,
//                                 t_i <- b_i - sum_lower A_ik x_k
//   backward, colours descending: x_i = (t_i - sum_upper A_ik x_k) / A_ii
//   residual:                     r_i = sum_lower A_ik (x_k at the forward visit - x_k final)
// because the lower neighbours of a row do not change between its forward and its
// backward visit, and the backward visit leaves b - (forward lower sum) - (final
// upper sum) - A_ii x_i = 0.  So from a zero guess every stored entry is read once
// (plus the lower half for the residual) where two full sweeps and a residual
// read them three times, and nothing of the row is recomputed.
//
// What bounds a step is latency: 2 C - 1 dependent phases for C colours, each a
// few thousand rows.  Two forms, which give the same bits for the same lanes per
// row (every row sees the same values and sums them in the same order):
//   * dataflow (the default): there is no barrier and no flag.  Beside x the level
//     holds a slot for every row's forward and one for its backward value, empty
//     (a bit pattern no value has) until the row stores it; a row that needs a
//     neighbour's value polls that slot itself.  The critical path of a phase is one store, the
//     load that sees it, and the row's sum: no fence behind the writes, no CTA
//     barrier, no counter to publish and poll, no wait for rows that are not
//     neighbours.  Warps run as far ahead as their own rows allow, and load the
//     matrix entries of their next rows while they poll.
//   * grid barrier (options.sweep_sync = 1): plain x, a grid-wide barrier between
//     colours.
//
// Measured on a GB300, one pre-step with its residual and one post-step, before (two
// full sweeps with neighbour flags, a separate residual) and now:
//   128^3 cube, level 1 (188,428 rows, 6.2 M entries, 16 colours): FP32 240 -> 155 us,
//     FP64 600 -> 323 us;  97^3, level 1 (82,455 rows): FP64 520 -> 190 us
//   1024^2 square, FP32: level 1 (146,813 rows, 9 colours) 122 -> 59 us, level 2 (8,707
//     rows, 10 colours) 123 -> 47 us
//   64^2 square, level 1 (592 rows, 8 colours): FP64 198 -> 43 us, FP32 80 -> 29 us
//   triangulation of 150^2 nodes, finest level (FP64; one launch per colour and a
//     residual before): 101 -> 35 us
// A phase takes 0.75 us on small levels (a store seen by another SM's poll takes 0.5 to
// 0.75 us by itself) and 2.5 us on the 128^3 level, where the slowest of many
// dependencies counts.  Carrying a tag beside every value instead of the empty slots
// (16 and 32 byte slots) measured 170 -> 246 us on the 128^3 level (FP32), and
// computing a warp's rows in the kernel instead of listing them accounted for most
// of that.
#include <type_traits>

#include "gl_internal.cuh"
#include "gl_kernels.cuh"
#include "gl_profile.cuh"

namespace gl {

// ---------------------------------------------------------------- bounded waits
// Every wait is bounded by SWEEP_WAIT_NS of the global timer.  A wait that runs
// out sets the preconditioner's error word and, when the launch belongs to a
// solve, the solve's status word to STATUS_TIMEOUT, so every later kernel of the
// solve returns at once and the host reports GL_ERR_TIMEOUT; every sweep launch
// returns at once while the error word is set, until the host resets the
// synchronisation state (sweeps_reset).
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// spins until *p >= want; false if SWEEP_WAIT_NS passed first
__device__ __forceinline__ bool spin_geq(const unsigned long long *p, unsigned long long want) {
    if (ld_acquire_u64(p) >= want) return true;
    const unsigned long long t0 = globaltimer_ns();
    for (unsigned spins = 1;; ++spins) {
        if (ld_acquire_u64(p) >= want) return true;
        if ((spins & 63u) == 0 && globaltimer_ns() - t0 > (unsigned long long)SWEEP_WAIT_NS) return false;
    }
}
__device__ __forceinline__ void report_timeout(int *err, int *stop) {
    atomicExch(err, 1);
    if (stop) atomicExch(stop, STATUS_TIMEOUT);
}
__device__ __forceinline__ bool sweep_halted(const int *stop, const int *err) {
    return (stop && *(volatile const int *)stop) || *(volatile const int *)err;
}

// Grid barrier: one 64-bit arrival counter per (level, precision) that only
// grows.  Every launch on a counter uses the same number of CTAs nb, so the
// counter is a multiple of nb between launches.  At its first barrier a CTA takes
// a ticket with an atomic add (the ticket rounded down to a multiple of nb is the
// launch's base); at every later barrier it only adds one with a release
// reduction.  Barrier k is passed when the counter reaches base + (k + 1) nb, which
// one thread per CTA observes with acquiring loads.
__device__ __forceinline__ void grid_arrive(unsigned long long *cnt, unsigned k, unsigned long long &base) {
    __syncthreads();
    if (threadIdx.x == 0) {
        if (k == 0) {
            unsigned long long t;
            asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], 1;" : "=l"(t) : "l"(cnt) : "memory");
            base = t - t % gridDim.x;
        } else {
            asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(cnt) : "memory");
        }
    }
}
// waits for barrier k; false if the wait ran out (thread 0 holds base and the
// extra offset of every wait target, nonzero only when a test has asked for
// waits that cannot end)
__device__ __forceinline__ bool grid_wait(const unsigned long long *cnt, unsigned k, unsigned long long base,
                                          unsigned long long extra, int *err, int *stop) {
    __shared__ int ok;
    if (threadIdx.x == 0) {
        const unsigned long long want = base + (unsigned long long)(k + 1) * gridDim.x + extra;
        ok = spin_geq(cnt, want) ? 1 : 0;
        if (!ok) report_timeout(err, stop);
    }
    __syncthreads();
    return ok;
}

// ---------------------------------------------------------------- values in flight
// A slot of the dataflow arrays is written once per launch; until then it holds the
// sentinel (all bits set) in both components.  A component is one relaxed access,
// which the memory model makes single-copy atomic: a reader that sees anything but
// the sentinel has the value.  (A relaxation never stores the sentinel: a NaN of
// that bit pattern becomes another NaN.)
template <typename R>
struct Slot;
template <>
struct Slot<float> {
    float2 v;
    __device__ __forceinline__ void clear() { v = make_float2(0.f, 0.f); }
    __device__ __forceinline__ void load(const float2 *p) {
        unsigned a, b;
        asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "l"(p));
        v = make_float2(__uint_as_float(a), __uint_as_float(b));
    }
    __device__ __forceinline__ bool empty() const {
        return __float_as_uint(v.x) == 0xffffffffu || __float_as_uint(v.y) == 0xffffffffu;
    }
    static __device__ __forceinline__ void store(float *p, float x) {
        unsigned u = __float_as_uint(x);
        if (u == 0xffffffffu) u = 0x7fffffffu;
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(u));
    }
};
template <>
struct Slot<double> {
    double2 v;
    __device__ __forceinline__ void clear() { v = make_double2(0., 0.); }
    __device__ __forceinline__ void load(const double2 *p) {
        unsigned long long a, b;
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
        v = make_double2(__longlong_as_double((long long)a), __longlong_as_double((long long)b));
    }
    __device__ __forceinline__ bool empty() const {
        return __double_as_longlong(v.x) == -1ll || __double_as_longlong(v.y) == -1ll;
    }
    static __device__ __forceinline__ void store(double *p, double x) {
        unsigned long long u = (unsigned long long)__double_as_longlong(x);
        if (u == ~0ull) u = 0x7fffffffffffffffull;
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(u));
    }
};

// ---------------------------------------------------------------- the sweep
// Entries per lane loaded ahead of their row's turn (PF): the part of a row beyond PF
// G entries costs its step a second round of loads, so long rows on few lanes take 8
// (155 against 170 us for the pre- and post-step of the 128^3 cube's level 1 on 4
// lanes), where the registers for 8 cost short rows more than they save (35 against
// 29 us on the 64^2 square's level 1, 10 entries a row, on 4 lanes).
static int sweep_pf(int G, bool fp32, int64_t nnz, int64_t n) {
    return fp32 && (G == 2 || (G == 4 && nnz >= 16 * n)) ? 8 : 4;
}
// resident CTAs per SM the registers are limited for: one row of the largest colour of
// a 128^3 cube's level 1 per group of 8 (FP32) or 4 lanes (FP64 and PF = 8)
template <typename R, int PF>
__host__ __device__ constexpr int sweep_ctas_per_sm() {
    return sizeof(R) == 4 && PF == 4 ? 7 : 4;
}
constexpr int FLOW_THREADS = 128;       // no CTA-wide step: small CTAs spread a level over the SMs
constexpr int GRID_THREADS = 512;

template <typename C, typename R>
struct SweepArgs {
    const RowDesc *desc;         // per warp: its rows in colour order, 32 / G per step
    const int32_t *woff;         // first step of every warp (one more entry behind the last)
    const int32_t *cfirst;       // grid form: first step of every (warp, colour)
    const int32_t *col;
    const C *val;
    const R *idiag;              // 1 / A_ii
    int ncolors;
    int64_t n;
    const C *b;
    C *x;
    int zero_start;              // the forward pass starts from x = 0 (x is not read)
    C *t;                        // work vector (may be r)
    C *r;                        // nullable: the residual b - A x afterwards (zero_start only)
    const R *scale;              // nullable: factor of the residual's rows
    C *xs;                       // dataflow: two sets of (forward, backward) slots
    unsigned *state;             // dataflow: launches, CTAs done; grid: the arrival counter
    const unsigned long long *extra;
    int *err, *stop;
};

enum SweepStage { ST_PRE, ST_FWD, ST_BWD, ST_POST };

// A group of G lanes relaxes one row; a warp takes 32 / G consecutive rows of a
// colour per step, and each warp a proportional share of every colour's rows
// (positions of a colour hold ascending node ids, so a warp's rows of all colours
// lie in about the same part of the level).  What a warp does is listed beforehand
// (RowDesc), so a step computes no index but its addresses: the instructions of a
// step lie on the critical path of every phase.
//
// Why the dataflow form cannot deadlock: every warp walks its rows in phase order,
// a row waits only for values of earlier phases, and all CTAs are resident
// (cooperative launch).  Every slot is written once per launch (a row's forward and
// its backward value have slots of their own), and the launch's set of slots was
// emptied by the launch before it, so nothing is ever overwritten unread.  Plain x
// is read in the pre-pass only, by rows of lower colours, and written by a row's
// last relaxation, which waits for those rows' forward values.  That read and that write
// have no release and acquire between them: the read's value goes into the reader's
// forward value, the writer polls that value, and what it writes is formed from it, so the
// read could only see the write in a circle of dependences (a value out of thin air, which
// the PTX memory model excludes).  It does not order the two otherwise: a pre-pass whose
// result did not go into the polled value would need a copy of x.
template <int G, int PF, typename C, typename R, bool FLOW>
struct Sweep {
    static constexpr int RPW = 32 / G, H = G / 2;
    const SweepArgs<C, R> &a;
    C *xf, *xb;                        // this launch's forward and backward slots
    int lane, grp, gl, comp;           // lane, group in the warp, lane in the group, component it finishes
    bool writer, never;                // never: a test asks for waits that cannot end

    struct Block {
        int32_t col[PF];
        C val[PF];
        uint32_t q;
        int len, row, ne;              // ne: entries per lane of the step's longest row (warp-uniform)
        R in, in2, d;
        bool last;
    };
    __device__ __forceinline__ RowDesc desc_of(int step) const { return a.desc[(size_t)step * RPW + grp]; }
    // the entries j0 + gl, j0 + gl + G, ... of a row's part (value 0 past its end)
    __device__ __forceinline__ void entries(uint32_t q, int left, int32_t (&col)[PF], C (&val)[PF]) const {
        const int32_t *cp = a.col + q + gl;
        const C *vp = a.val + q + gl;
#pragma unroll
        for (int e = 0; e < PF; ++e) {
            val[e].x = 0;
            val[e].y = 0;
            if (gl + e * G < left) {
                col[e] = __ldg(cp + e * G);
                val[e] = vp[e * G];
            }
        }
    }
    // the x-independent data of the group's row
    template <SweepStage S>
    __device__ __forceinline__ void load(const RowDesc &d, Block &B) const {
        constexpr bool UP = S == ST_PRE || S == ST_BWD;
        const int nl = (int)(d.n & 0xffffu), nu = (int)(d.n >> 16);
        B.q = d.q0 + (UP ? nl : 0);
        B.len = UP ? nu : nl;
        B.row = d.row;
        B.last = (d.flags & 1u) != 0;
        B.ne = (int)(UP ? d.flags >> 17 : d.flags >> 1 & 0x7fffu);
        entries(B.q, B.len, B.col, B.val);
        if (writer && d.row >= 0) {
            const size_t o = 2 * (size_t)d.row + comp;
            const R *bp = reinterpret_cast<const R *>(a.b), *tp = reinterpret_cast<const R *>(a.t);
            if (S == ST_PRE) {
                B.in = bp[o];
            } else if (S == ST_FWD) {
                B.in2 = bp[o];
                // (rows of the last colour have no upper entries)
                B.in = a.zero_start || B.last ? B.in2 : tp[o];
                B.d = a.idiag[d.row];
            } else if (S == ST_BWD) {
                B.in = tp[o];
                B.d = a.idiag[d.row];
            } else {
                B.in = bp[o];
                B.in2 = tp[o];
                B.d = a.scale ? a.scale[d.row] : (R)1;
            }
        }
    }
    template <SweepStage S>
    __device__ __forceinline__ void request(const int32_t (&col)[PF], int left, Slot<R> (&raw)[PF]) const {
        const C *src = S == ST_FWD ? xf : xb;
#pragma unroll
        for (int e = 0; e < PF; ++e) {
            raw[e].clear();
            if (gl + e * G < left) {
                if (S == ST_PRE)
                    raw[e].v = a.x[col[e]];
                else if (!FLOW)
                    raw[e].v = __ldca(a.x + col[e]);
                else
                    raw[e].load(src + col[e]);
            }
        }
    }
    // polls the requested slots until all hold their values; false if that took too long
    template <SweepStage S>
    __device__ __forceinline__ bool await(const int32_t (&col)[PF], Slot<R> (&raw)[PF]) const {
        if (S == ST_PRE || !FLOW) return true;
        const C *src = S == ST_FWD ? xf : xb;
        unsigned long long t0 = 0;
        for (unsigned spins = 1;; ++spins) {
            bool pend = never;
#pragma unroll
            for (int e = 0; e < PF; ++e)
                if (raw[e].empty()) {
                    pend = true;
                    raw[e].load(src + col[e]);
                }
            if (!__any_sync(0xffffffffu, pend)) return true;
            if ((spins & 63u) == 0) {
                const unsigned long long now = globaltimer_ns();
                if (t0 == 0) t0 = now;
                const bool out = now - t0 > (unsigned long long)SWEEP_WAIT_NS;
                if (__any_sync(0xffffffffu, out || *(volatile const int *)a.err)) {
                    if (lane == 0) report_timeout(a.err, a.stop);
                    return false;
                }
            }
        }
    }
    // the rows of one step: sums (the first PF entries of every lane already
    // requested), and the rows' new values
    template <SweepStage S>
    __device__ __forceinline__ bool finish(const Block &B, Slot<R> (&raw)[PF]) const {
        C acc;
        acc.x = 0;
        acc.y = 0;
        if (!await<S>(B.col, raw)) return false;
#pragma unroll
        for (int e = 0; e < PF; ++e) {
            if (sizeof(R) == 8 && e >= B.ne) break;  // (FP64 instructions are what a step issues slowest)
            cfma(acc, B.val[e], raw[e].v);
        }
        // rows longer than PF G entries
        for (int e0 = PF; e0 < B.ne; e0 += PF) {
            int32_t col[PF];
            C val[PF];
            const int left = B.len - e0 * G, ne = B.ne - e0;
            entries(B.q + e0 * G, left, col, val);
            request<S>(col, left, raw);
            if (!await<S>(col, raw)) return false;
#pragma unroll
            for (int e = 0; e < PF; ++e) {
                if (sizeof(R) == 8 && e >= ne) break;
                cfma(acc, val[e], raw[e].v);
            }
        }
        // group sum: the lower half of the lanes keeps the real, the upper half the
        // imaginary part, so every step moves and adds one component
        R s = comp ? acc.y : acc.x;
        s += __shfl_xor_sync(0xffffffffu, comp ? acc.x : acc.y, H);
#pragma unroll
        for (int o = H / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (writer && B.row >= 0) {
            const size_t o = 2 * (size_t)B.row + comp;
            R *xp = reinterpret_cast<R *>(a.x), *tp = reinterpret_cast<R *>(a.t);
            if (S == ST_PRE) {
                tp[o] = B.in - s;
            } else if (S == ST_POST) {
                reinterpret_cast<R *>(a.r)[o] = ((B.in - B.in2) - s) * B.d;
            } else {
                const R xv = (B.in - s) * B.d;
                const bool last = S == ST_BWD || B.last;  // the row's last relaxation
                if (FLOW) Slot<R>::store(reinterpret_cast<R *>(last ? xb : xf) + o, xv);
                if (S == ST_FWD) tp[o] = B.in2 - s;
                if (!FLOW || last) xp[o] = xv;
            }
        }
        return true;
    }
    // all steps of a stage in phase order [s0, s1) (backward: from the end), the next
    // step's entries loaded while the current ones are polled, its descriptors two
    // steps ahead.  The backward stage skips the last colour's rows, which it would
    // relax from unchanged neighbours; the residual has no work for the first colour's.
    template <SweepStage S>
    __device__ __forceinline__ bool run(int s0, int s1) const {
        Block B;
        first<S>(s0, s1, B);
        return run<S>(s0, s1, B);
    }
    // the x-independent data of the first step of [s0, s1)
    template <SweepStage S>
    __device__ __forceinline__ void first(int s0, int s1, Block &B) const {
        if (s0 < s1) load<S>(desc_of(S == ST_BWD ? s1 - 1 : s0), B);
    }
    // with that of the first step in B
    template <SweepStage S>
    __device__ __forceinline__ bool run(int s0, int s1, Block &B) const {
        constexpr int dir = S == ST_BWD ? -1 : 1;
        const int cnt = s1 - s0;
        if (cnt <= 0) return true;
        int step = dir > 0 ? s0 : s1 - 1;
        RowDesc dn;
        if (cnt > 1) dn = desc_of(step + dir);
        for (int k = 0; k < cnt; ++k, step += dir) {
            Slot<R> raw[PF];
            request<S>(B.col, B.len, raw);
            Block N;
            if (k + 1 < cnt) load<S>(dn, N);
            if (k + 2 < cnt) dn = desc_of(step + 2 * dir);
            if (!(S == ST_BWD && B.last))
                if (!finish<S>(B, raw)) return false;
            B = N;
        }
        return true;
    }
};

template <int G, int PF, typename C, typename R, bool FLOW>
__global__ void __launch_bounds__(FLOW ? FLOW_THREADS : GRID_THREADS, FLOW ? sweep_ctas_per_sm<R, PF>() : 1)
    k_sweep(SweepArgs<C, R> a) {
    if (sweep_halted(a.stop, a.err)) return;
    const int lane = threadIdx.x & 31, gl = lane % G;
    const int w = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const unsigned parity = FLOW ? *(volatile unsigned *)a.state & 1u : 0u;
    C *set = a.xs + (FLOW ? 2 * (size_t)a.n * parity : 0);
    Sweep<G, PF, C, R, FLOW> S{a,         set,      set + a.n, lane, lane / G, gl, gl >= G / 2 ? 1 : 0, gl % (G / 2) == 0,
                           *a.extra != 0};
    const int s0 = a.woff[w], s1 = a.woff[w + 1];
    const bool resid = a.r != nullptr;
    if (FLOW) {
        // the other set of slots is nobody's now: empty it for the next launch
        {
            unsigned long long *o = reinterpret_cast<unsigned long long *>(a.xs + 2 * (size_t)a.n * (parity ^ 1u));
            const size_t words = 2 * (size_t)a.n * (sizeof(C) / 8), nt = (size_t)gridDim.x * blockDim.x;
            for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += nt) o[i] = ~0ull;
        }
        if (!a.zero_start && !S.template run<ST_PRE>(s0, s1)) return;
        if (!S.template run<ST_FWD>(s0, s1)) return;
        if (!S.template run<ST_BWD>(s0, s1)) return;
        if (resid && !S.template run<ST_POST>(s0, s1)) return;
        // the last CTA to finish counts the launch
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(a.state + 1, 1u) == gridDim.x - 1) {
                a.state[1] = 0;
                a.state[0] += 1;
            }
        }
    } else {
        unsigned long long *cnt = reinterpret_cast<unsigned long long *>(a.state);
        unsigned long long base = 0;
        const unsigned long long extra = threadIdx.x == 0 ? *a.extra : 0ull;
        unsigned k = 0;
        const int32_t *cf = a.cfirst + (size_t)w * (a.ncolors + 1);
        if (!a.zero_start) S.template run<ST_PRE>(s0, s1);
        // the first rows of the next colour are loaded between arriving and waiting
        typename Sweep<G, PF, C, R, FLOW>::Block B;
        S.template first<ST_FWD>(cf[0], cf[1], B);
        for (int c = 0; c < a.ncolors; ++c) {
            S.template run<ST_FWD>(cf[c], cf[c + 1], B);
            grid_arrive(cnt, k, base);
            if (c + 1 < a.ncolors)
                S.template first<ST_FWD>(cf[c + 1], cf[c + 2], B);
            else if (c > 0)
                S.template first<ST_BWD>(cf[c - 1], cf[c], B);
            if (!grid_wait(cnt, k++, base, extra, a.err, a.stop)) return;
        }
        for (int c = a.ncolors - 2; c >= 0; --c) {
            S.template run<ST_BWD>(cf[c], cf[c + 1], B);
            grid_arrive(cnt, k, base);
            if (c > 0) S.template first<ST_BWD>(cf[c - 1], cf[c], B);
            if (!grid_wait(cnt, k++, base, extra, a.err, a.stop)) return;
        }
        if (resid) S.template run<ST_POST>(s0, s1);
    }
}

// ---------------------------------------------------------------- what every warp does
// The W warps form K shifts (K divides W), and colour c belongs to the warps w with w mod K = c mod
// K.  Colour c's rows are cut into S_c steps of 32 / G consecutive rows, and the k-th
// of the W / K warps of its shift takes the steps [floor(S_c k K / W), floor(S_c (k +
// 1) K / W)).
__device__ __forceinline__ int64_t share(int64_t S, int64_t k, int64_t n) { return S * k / n; }
__device__ __forceinline__ int64_t warp_steps(int64_t S, int c, int w, int W, int K) {
    return w % K == c % K ? share(S, w / K + 1, W / K) - share(S, w / K, W / K) : 0;
}

__global__ void k_sweep_count(int W, int K, int nc, int rpw, const int64_t *__restrict__ cstart,
                              int64_t *__restrict__ cnt) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= W) return;
    int64_t o = 0;
    for (int c = 0; c < nc; ++c) o += warp_steps((cstart[c + 1] - cstart[c] + rpw - 1) / rpw, c, w, W, K);
    cnt[w] = o;
}
__global__ void k_sweep_first(int W, int K, int nc, int rpw, const int64_t *__restrict__ cstart,
                              const int64_t *__restrict__ off, int32_t *__restrict__ woff,
                              int32_t *__restrict__ cfirst) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w > W) return;
    int64_t o = off[w];
    woff[w] = (int32_t)o;
    if (w == W) return;
    for (int c = 0; c < nc; ++c) {
        cfirst[(size_t)w * (nc + 1) + c] = (int32_t)o;
        o += warp_steps((cstart[c + 1] - cstart[c] + rpw - 1) / rpw, c, w, W, K);
    }
    cfirst[(size_t)w * (nc + 1) + nc] = (int32_t)o;
}
// one thread per (colour blockIdx.y, step of the colour)
__global__ void k_sweep_desc(int W, int K, int nc, int rpw, const int64_t *__restrict__ cstart,
                             const int32_t *__restrict__ cfirst, const RowSplit *__restrict__ rows,
                             RowDesc *__restrict__ desc) {
    const int c = blockIdx.y;
    const int64_t lo = cstart[c], m = cstart[c + 1] - lo, S = (m + rpw - 1) / rpw, n = W / K;
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= S) return;
    const int64_t k = ((j + 1) * n - 1) / S;  // the largest k with floor(S k / n) <= j
    const int64_t w = k * K + c % K;
    RowDesc *d = desc + (cfirst[(size_t)w * (nc + 1) + c] + (j - share(S, k, n))) * (size_t)rpw;
    const int G = 32 / rpw;
    int ml = 0, mu = 0;  // the longest lower and upper part of the step's rows
    for (int g = 0; g < rpw; ++g) {
        const int64_t i = j * rpw + g;
        if (i < m) {
            ml = max(ml, rows[lo + i].nl);
            mu = max(mu, rows[lo + i].nu);
        }
    }
    const uint32_t flags = (c == nc - 1 ? 1u : 0u) | (uint32_t)((ml + G - 1) / G) << 1 |
                           (uint32_t)((mu + G - 1) / G) << 17;
    for (int g = 0; g < rpw; ++g) {
        const int64_t i = j * rpw + g;
        RowDesc v{0, 0, -1, flags};
        if (i < m) {
            const RowSplit r = rows[lo + i];
            v.q0 = (uint32_t)r.q0;
            v.n = (uint32_t)r.nl | (uint32_t)r.nu << 16;
            v.row = (int32_t)(lo + i);
        }
        d[g] = v;
    }
}

// ---------------------------------------------------------------- operators
__global__ void k_split_len(int64_t nrows, const int32_t *perm, const int32_t *iperm, const int64_t *rp,
                            const int32_t *ci, int64_t *len, RowSplit *rows, int *err) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= nrows) return;
    const int64_t r = perm[p];
    int nl = 0, nu = 0;
    for (int64_t q = rp[r]; q < rp[r + 1]; ++q) {
        const int64_t c = iperm[ci[q]];
        nl += c < p;
        nu += c > p;
    }
    if (nl > 0xfffe || nu > 0xfffe) atomicExch(err, 1);
    len[p] = nl + nu;
    rows[p] = RowSplit{0, nl, nu};
}
template <typename C>
__global__ void k_split_fill(int64_t nrows, const int32_t *perm, const int32_t *iperm, const int64_t *rp,
                             const int32_t *ci, const double2 *v, const double *row_scale, const int64_t *off,
                             RowSplit *rows, int32_t *ocol, C *oval, double *diag_out) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= nrows) return;
    const int64_t r = perm[p];
    int64_t lo = off[p], up = lo + rows[p].nl;
    rows[p].q0 = lo;
    double dg = 0;
    const double sc = row_scale ? 1.0 / row_scale[r] : 1.0;
    for (int64_t q = rp[r]; q < rp[r + 1]; ++q) {
        const int32_t c = iperm[ci[q]];
        const double2 a = make_double2(v[q].x * sc, v[q].y * sc);
        if (c == p) {
            dg = a.x;
            continue;
        }
        const int64_t o = c < p ? lo++ : up++;
        ocol[o] = c;
        C val;
        val.x = a.x;
        val.y = a.y;
        oval[o] = val;
    }
    if (diag_out) diag_out[p] = dg;
}

template <typename C>
void build_split(int64_t n, const int32_t *perm, const int32_t *iperm, const CsrDev &A, const double *row_scale,
                 SplitCsr<C> &out, double *diag_out, cudaStream_t s) {
    out.nrows = n;
    out.nnz = A.nnz - n;  // every row stores its diagonal
    GL_REQUIRE(out.nnz < 0xffffffffll, GL_ERR_CAPACITY, "level operator has too many entries");
    DBuf<int64_t> len(n + 1);
    DBuf<int> err(1);
    GL_CUDA(cudaMemsetAsync(err.get(), 0, sizeof(int), s));
    out.rows.alloc(n);
    k_split_len<<<grid_for(n, 256), 256, 0, s>>>(n, perm, iperm, A.rp.get(), A.ci.get(), len.get(), out.rows.get(),
                                                 err.get());
    GL_LAUNCH_CHECK();
    scan_exclusive(len.get(), len.get(), n, true, s);
    out.col.alloc(out.nnz > 0 ? out.nnz : 1);
    out.val.alloc(out.nnz > 0 ? out.nnz : 1);
    k_split_fill<C><<<grid_for(n, 256), 256, 0, s>>>(n, perm, iperm, A.rp.get(), A.ci.get(), A.v.get(), row_scale,
                                                     len.get(), out.rows.get(), out.col.get(), out.val.get(),
                                                     diag_out);
    GL_LAUNCH_CHECK();
    int herr = 0;
    GL_CUDA(cudaMemcpyAsync(&herr, err.get(), sizeof(int), cudaMemcpyDeviceToHost, s));
    GL_CUDA(cudaStreamSynchronize(s));
    GL_REQUIRE(herr == 0, GL_ERR_CAPACITY, "level operator row too long");
}
template void build_split<double2>(int64_t, const int32_t *, const int32_t *, const CsrDev &, const double *,
                                   SplitCsr<double2> &, double *, cudaStream_t);
template void build_split<float2>(int64_t, const int32_t *, const int32_t *, const CsrDev &, const double *,
                                  SplitCsr<float2> &, double *, cudaStream_t);

template <typename R>
__global__ void k_inverse(int64_t n, const R *__restrict__ d, R *__restrict__ id) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) id[i] = (R)1 / d[i];
}

// ---------------------------------------------------------------- host side
// calls f(std::integral_constant<int, G>, std::integral_constant<int, PF>)
template <typename R, typename F>
static void sweep_dispatch(int G, int PF, F &&f) {
    const std::integral_constant<int, 4> p4;
    if constexpr (sizeof(R) == 4) {
        const std::integral_constant<int, 8> p8;
        if (G == 2) return f(std::integral_constant<int, 2>(), p8);
        if (G == 4 && PF == 8) return f(std::integral_constant<int, 4>(), p8);
    }
    switch (G) {
        case 2: return f(std::integral_constant<int, 2>(), p4);
        case 4: return f(std::integral_constant<int, 4>(), p4);
        case 8: return f(std::integral_constant<int, 8>(), p4);
        case 16: return f(std::integral_constant<int, 16>(), p4);
        default: return f(std::integral_constant<int, 32>(), p4);
    }
}

template <typename T>
struct SweepOps;
template <>
struct SweepOps<double> {
    using C = double2;
    static SweepData<double2, double> &data(Level &L) { return L.sw64; }
    static const double *diag(const Level &L) { return L.diag.get(); }
    static C *b(Level &L) { return L.b.get(); }
    static C *x(Level &L) { return L.x.get(); }
    static C *r(Level &L) { return L.r.get(); }
};
template <>
struct SweepOps<float> {
    using C = float2;
    static SweepData<float2, float> &data(Level &L) { return L.sw32; }
    static const float *diag(const Level &L) { return L.diag32.get(); }
    static C *b(Level &L) { return L.b32.get(); }
    static C *x(Level &L) { return L.x32.get(); }
    static C *r(Level &L) { return L.r32.get(); }
};

// most CTAs of a sweep that can be resident at once (queried once per kernel)
template <int G, int PF, typename C, typename R, bool FLOW>
static int sweep_max_ctas() {
    static const int most = [] {
        int dev = 0, nsm = 0, per_sm = 0;
        GL_CUDA(cudaGetDevice(&dev));
        GL_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        GL_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep<G, PF, C, R, FLOW>,
                                                              FLOW ? FLOW_THREADS : GRID_THREADS, 0));
        GL_REQUIRE(per_sm > 0, GL_ERR_CUDA, "cooperative sweep kernel cannot be resident");
        return per_sm * nsm;
    }();
    return most;
}

template <int G, int PF, typename C, typename R, bool FLOW>
static void launch_sweep(int nb, const SweepArgs<C, R> &a, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nb);
    cfg.blockDim = dim3(FLOW ? FLOW_THREADS : GRID_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    GL_CUDA(cudaLaunchKernelEx(&cfg, k_sweep<G, PF, C, R, FLOW>, a));
}

template <typename T>
static void sweep_launch(gl_prec_s *p, Level &L, const typename SweepOps<T>::C *b, typename SweepOps<T>::C *x,
                         bool zero_start, typename SweepOps<T>::C *r, const T *scale, int *stop, cudaStream_t s) {
    using O = SweepOps<T>;
    using C = typename O::C;
    auto &D = O::data(L);
    SweepArgs<C, T> a;
    a.desc = D.desc.get();
    a.woff = D.woff.get();
    a.cfirst = D.cfirst.get();
    a.col = D.A.col.get();
    a.val = D.A.val.get();
    a.idiag = D.idiag.get();
    a.ncolors = L.ncolors;
    a.n = L.n;
    a.b = b;
    a.x = x;
    a.zero_start = zero_start ? 1 : 0;
    a.t = O::r(L);
    a.r = r;
    a.scale = scale;
    a.xs = D.xs.get();
    a.state = D.state.get();
    a.extra = p->wait_extra.get();
    a.err = p->err.get();
    a.stop = stop;
    sweep_dispatch<T>(D.G, D.PF, [&](auto G, auto PF) {
        if (D.sync == 1)
            launch_sweep<G.value, PF.value, C, T, true>(D.nb, a, s);
        else
            launch_sweep<G.value, PF.value, C, T, false>(D.nb, a, s);
    });
}

// Whether the finest level of a general mesh is swept by k_sweep (on a lattice it has two
// colours and never is).  With a launch per colour the step and its residual read every
// entry 4.5 times, k_sweep reads it 3 times, but writes, empties and polls slots and reads
// lists of rows, 100 to 200 bytes a row more; past the caches that decides.  One
// preconditioner application, a launch per colour against k_sweep, on triangulations (6
// entries a row):
//   nodes            360,000     640,000     1.0 M       1.44 M      2.25 M       16 M
//   FP32 dataflow    339, 252    400, 345    448, 444    538, 568    657, 783     3406, 4962 us
//   FP64 dataflow    500, 387    624, 521    762, 688    961, 893    1270, 1278   6999, 8108
//   FP32 grid        418, 353    481, 445    520, 538    614, 674    727, 889     3515, 5113
//   FP64 grid        637, 569    775, 723    904, 895    1119, 1127  1409, 1487   7255, 8320
// and on a ball's tetrahedra (14 entries a row), 0.6 M and 3.5 M nodes: FP32 768, 480 and
// 2026, 1703 us; FP64 1254, 755 and 4048, 2964; likewise with the grid barrier.  So rows
// of ten entries and more are always swept, shorter ones up to 2^20 (FP32) and 2^21 rows
// (FP64), three quarters of these with the grid barrier.
void sweep_finest(gl_prec_s *p, int sync) {
    const Level &L = p->L[0];
    for (int fp32 = 0; fp32 < 2; ++fp32) {
        const int64_t most = (sync == 1 ? 3 : 4) * (fp32 ? 1ll << 18 : 1ll << 19);
        p->finest_swept[fp32] = L.ncolors > 2 && (L.n <= most || L.A_can.nnz >= 11 * L.n);
    }
}

template <typename T>
void sweep_step(gl_prec_s *p, int l, const typename CT<T>::type *b, typename CT<T>::type *x, bool zero_start,
                typename CT<T>::type *r, const T *scale, const int *stop, cudaStream_t s) {
    using C = typename CT<T>::type;
    Level &L = p->L[l];
    auto &D = SweepOps<T>::data(L);
    // algorithmic bytes: the stored entries (value + column) once, the lower half
    // again for the residual, the upper half again for a nonzero guess; per row the
    // row pointers, b, the diagonal, the work vector written and read, x written (and
    // read from a nonzero guess), and r
    const double rows = (double)L.n, half = 0.5 * (double)D.A.nnz;
    const double ent = 2.0 * half + (r ? half : 0.0) + (zero_start ? 0.0 : half);
    const double bytes = ent * (sizeof(C) + 4) + rows * (sizeof(RowDesc) + sizeof(T) + 4.0 * sizeof(C)) +
                         (r || !zero_start ? 2.0 : 0.0) * rows * sizeof(C);
    ProfScope ps("gs", bytes, s, 8.0 * ent + 6.0 * rows);
    // the status word of the solve this sweep belongs to: a wait that runs out writes it
    sweep_launch<T>(p, L, b, x, zero_start, r, scale, const_cast<int *>(stop), s);
}
template void sweep_step<double>(gl_prec_s *, int, const double2 *, double2 *, bool, double2 *, const double *,
                                 const int *, cudaStream_t);
template void sweep_step<float>(gl_prec_s *, int, const float2 *, float2 *, bool, float2 *, const float *, const int *,
                                cudaStream_t);

template <typename C, typename R>
static void sweep_zero(SweepData<C, R> &D, cudaStream_t s) {
    if (!D.state.get()) return;
    GL_CUDA(cudaMemsetAsync(D.xs.get(), 0xff, D.xs.bytes(), s));
    GL_CUDA(cudaMemsetAsync(D.state.get(), 0, D.state.bytes(), s));
}
// CTAs that give every row of the largest colour a group of its own
static int64_t sweep_ctas_wanted(const Level &L, int G, int K, bool flow) {
    int64_t maxc = 1;
    for (int c = 0; c < L.ncolors; ++c) maxc = std::max(maxc, L.cstart[c + 1] - L.cstart[c]);
    const int64_t per = (flow ? FLOW_THREADS : GRID_THREADS) / G;  // rows per CTA
    return (maxc * K + per - 1) / per;
}
// the sweep's own data of a level in one precision (the operator D.A is built)
template <typename T>
static void sweep_alloc(Level &L, cudaStream_t s) {
    auto &D = SweepOps<T>::data(L);
    D.idiag.alloc(L.n);
    k_inverse<T><<<grid_for(L.n, 256), 256, 0, s>>>(L.n, SweepOps<T>::diag(L), D.idiag.get());
    GL_LAUNCH_CHECK();
    D.xs.alloc(4 * (size_t)L.n);
    D.state.alloc(SWEEP_STATE_WORDS);
    sweep_zero(D, s);
}
// Fixes the form, the lanes per row and the shifts: the CTAs (one row of the largest
// colour per group of its shift, as far as they can be resident; in a batch the
// instances' sweeps run side by side, so a small level never takes the whole GPU),
// and the list of every warp's rows.
template <typename T>
static void sweep_shape(Level &L, int sync, int G, int K, cudaStream_t s) {
    auto &D = SweepOps<T>::data(L);
    D.sync = sync;
    D.G = G;
    D.K = K;
    D.PF = sweep_pf(G, sizeof(T) == 4, D.A.nnz, L.n);
    int most_ctas = 1;
    using C = typename SweepOps<T>::C;
    sweep_dispatch<T>(G, D.PF, [&](auto g, auto pf) {
        most_ctas = sync == 1 ? sweep_max_ctas<g.value, pf.value, C, T, true>()
                              : sweep_max_ctas<g.value, pf.value, C, T, false>();
    });
    D.nb = (int)std::min<int64_t>(sweep_ctas_wanted(L, G, K, sync == 1), most_ctas);
    const int rpw = 32 / G, nc = L.ncolors, W = D.nb * ((sync == 1 ? FLOW_THREADS : GRID_THREADS) / 32);
    GL_REQUIRE(W % K == 0, GL_ERR_ARG, "the warps of a sweep must divide into its shifts");
    int64_t steps = 0, most = 1;
    for (int c = 0; c < nc; ++c) {
        const int64_t S = (L.cstart[c + 1] - L.cstart[c] + rpw - 1) / rpw;
        steps += S;
        most = std::max(most, S);
    }
    D.woff.reserve(W + 1);
    D.cfirst.reserve((size_t)W * (nc + 1));
    D.desc.reserve((size_t)steps * rpw);
    DBuf<int64_t> cnt(W + 1);
    const int GW = grid_for(W + 1, 128);
    k_sweep_count<<<GW, 128, 0, s>>>(W, K, nc, rpw, L.cstart_dev.get(), cnt.get());
    GL_LAUNCH_CHECK();
    scan_exclusive(cnt.get(), cnt.get(), W, true, s);
    k_sweep_first<<<GW, 128, 0, s>>>(W, K, nc, rpw, L.cstart_dev.get(), cnt.get(), D.woff.get(), D.cfirst.get());
    k_sweep_desc<<<dim3((unsigned)((most + 127) / 128), nc), 128, 0, s>>>(W, K, nc, rpw, L.cstart_dev.get(),
                                                                          D.cfirst.get(), D.A.rows.get(),
                                                                          D.desc.get());
    GL_LAUNCH_CHECK();
}

// lanes per row without timing: the power of two nearest a quarter of the mean row length
static int sweep_default_lanes(int64_t nnz, int64_t n) {
    const double avg = n > 0 ? (double)nnz / n : 0;
    int G = 2;
    while (G < 32 && 2 * G * 4 <= avg * 1.5) G *= 2;
    return G;
}

// Chooses how every many-coloured level runs its symmetric Gauss-Seidel steps:
// dataflow unless options.sweep_sync = 1 asks for the grid barrier, the lanes per row
// G, and one or two shifts of warps (two: the warps of a phase have their loads and
// their first polls behind them when the phase before it stores; 48 to 43 us in FP64
// and 33 to 29 us in FP32 for the pre- and post-step of the 64^2 square's level 1,
// slower where the warps of both shifts no longer fit the SMs twice over).  With
// autotuning three numbers of lanes with one shift and, below a quarter of the GPU, two are
// timed (a pre- and a post-step on zero vectors, best of two after a warm-up) and the
// fastest kept: G = 2, 4, 8, or 4, 8, 16 where rows have 48 entries and more (the third
// level of a cube); without it G follows from the mean row length, with one shift.  The
// result depends on G only (the order of a row's sum).  On 2, 4, 8 and 16 lanes, with the
// better number of shifts:
//   97^3, level 2 (1252 rows of 54): FP64 643, 348, 226, 185 us; FP32 222, 136, 132, 123
//   128^3, level 2 (2720 rows): FP64 652, 364, 250, 201; FP32 237, 158, 160, 156
//   97^3, level 1 (82,455 rows of 33 entries): FP64 271, 212, 196, 242; FP32 135, 121, 137, 183
//   1024^2, level 1 (146,813 rows of 10): FP64 104, 124, 164, 294; FP32 60, 70, 94, 140
template <typename T>
static void plan_sweeps_t(gl_prec_s *p, cudaStream_t s) {
    using O = SweepOps<T>;
    using C = typename O::C;
    constexpr bool fp32 = sizeof(T) == 4;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (p->autotune) {
        GL_CUDA(cudaEventCreate(&e0));
        GL_CUDA(cudaEventCreate(&e1));
    }
    for (int l = 0; l < p->nlev - 1; ++l) {
        if (!p->swept(l, sizeof(T) == 4)) continue;
        Level &L = p->L[l];
        auto &D = O::data(L);
        sweep_alloc<T>(L, s);
        const int sync = p->sweep_sync == 1 ? 0 : 1;
        if (!p->autotune) {
            sweep_shape<T>(L, sync, sweep_default_lanes(D.A.nnz, L.n), 1, s);
            continue;
        }
        C *b = O::b(L), *x = O::x(L);
        GL_CUDA(cudaMemsetAsync(b, 0, L.n * sizeof(C), s));
        GL_CUDA(cudaMemsetAsync(x, 0, L.n * sizeof(C), s));
        float best = 1e30f;
        const int least = D.A.nnz >= 48 * L.n ? 4 : 2;
        int bestG = least, bestK = 1;
        for (int cand = 0; cand < 6; ++cand) {
            const int g = least << (cand % 3), K = 1 + cand / 3;
            if (K == 2 && (sync == 0 || sweep_ctas_wanted(L, g, 2, true) > 2 * NUM_SMS_HINT)) continue;
            sweep_shape<T>(L, sync, g, K, s);
            if (sync == 0) sweep_zero(D, s);  // another grid size on the barrier's counter
            float t = 1e30f;
            for (int rep = 0; rep < 3; ++rep) {
                GL_CUDA(cudaEventRecord(e0, s));
                sweep_launch<T>(p, L, b, x, true, O::r(L), nullptr, nullptr, s);
                sweep_launch<T>(p, L, b, x, false, nullptr, nullptr, nullptr, s);
                GL_CUDA(cudaEventRecord(e1, s));
                GL_CUDA(cudaEventSynchronize(e1));
                float ms = 0;
                GL_CUDA(cudaEventElapsedTime(&ms, e0, e1));
                if (rep > 0) t = std::min(t, ms);
            }
            if (verbose())
                fprintf(stderr, "gl: level %d (n %lld, %d colours, %s) sweep G %d, %d shifts, %d CTAs, %s: %.1f us (pre + post)\n", l,
                        (long long)L.n, L.ncolors, fp32 ? "FP32" : "FP64", g, K, D.nb, D.sync ? "dataflow" : "grid",
                        1e3 * t);
            if (t < best) best = t, bestG = g, bestK = K;
        }
        // a wait of a candidate ran out: the launches behind it returned at once, so the
        // times say nothing; the choice is the one made without timing
        if (sweeps_failed(p, s)) bestG = sweep_default_lanes(D.A.nnz, L.n), bestK = 1;
        sweep_shape<T>(L, sync, bestG, bestK, s);
        sweep_zero(D, s);
        GL_CUDA(cudaMemsetAsync(p->err.get(), 0, sizeof(int), s));
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
}

void plan_sweeps(gl_prec_s *p, bool fp32, cudaStream_t s) {
    if (fp32)
        plan_sweeps_t<float>(p, s);
    else
        plan_sweeps_t<double>(p, s);
}

// the choices of a template preconditioner of the same sparsity
template <typename T>
static void adopt_sweeps_t(gl_prec_s *p, const int *lanes, const int *shifts, const int *sync, cudaStream_t s) {
    for (int l = 0; l < p->nlev - 1; ++l) {
        if (!p->swept(l, sizeof(T) == 4)) continue;
        Level &L = p->L[l];
        sweep_alloc<T>(L, s);
        sweep_shape<T>(L, sync[l], lanes[l], shifts[l], s);
    }
}
void adopt_sweeps(gl_prec_s *p, bool fp32, cudaStream_t s) {
    int lanes[MAX_LEVELS], shifts[MAX_LEVELS], sync[MAX_LEVELS];
    for (int l = 0; l < MAX_LEVELS; ++l) {
        lanes[l] = fp32 ? p->tuned[l].sgs32 : p->tuned[l].sgs64;
        shifts[l] = fp32 ? p->tuned[l].shifts32 : p->tuned[l].shifts64;
        sync[l] = fp32 ? p->tuned[l].sync32 : p->tuned[l].sync64;
    }
    if (fp32)
        adopt_sweeps_t<float>(p, lanes, shifts, sync, s);
    else
        adopt_sweeps_t<double>(p, lanes, shifts, sync, s);
}

template <typename T>
static void sweeps_form_t(gl_prec_s *p, int G, int K, cudaStream_t s) {
    for (int l = 0; l < p->nlev - 1; ++l) {
        auto &D = SweepOps<T>::data(p->L[l]);
        if (!D.state.get()) continue;
        sweep_shape<T>(p->L[l], D.sync, G, K, s);
        sweep_zero(D, s);
    }
}
void sweeps_form(gl_prec_s *p, int G, int K, cudaStream_t s) {
    sweeps_form_t<double>(p, G, K, s);
    sweeps_form_t<float>(p, G, K, s);
    p->uid = next_uid();  // captured solves hold the old lists
}

void sweeps_reset(gl_prec_s *p, cudaStream_t s) {
    for (int l = 0; l < p->nlev - 1; ++l) {
        sweep_zero(p->L[l].sw32, s);
        sweep_zero(p->L[l].sw64, s);
    }
    GL_CUDA(cudaMemsetAsync(p->err.get(), 0, sizeof(int), s));
    GL_CUDA(cudaMemsetAsync(p->wait_extra.get(), 0, sizeof(unsigned long long), s));
}

int sweeps_failed(gl_prec_s *p, cudaStream_t s) {
    int h = 0;
    GL_CUDA(cudaMemcpyAsync(&h, p->err.get(), sizeof(int), cudaMemcpyDeviceToHost, s));
    GL_CUDA(cudaStreamSynchronize(s));
    return h;
}

}  // namespace gl
