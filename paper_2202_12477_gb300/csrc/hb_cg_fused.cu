// Fused CG for small meshes: every iteration of Algorithm 1 inside one
// cooperative kernel. On a mesh of a few dozen elements the element kernel
// itself needs a few microseconds of FP64 work, and launching the four
// kernels of an iteration costs more than that; here the phases of an
// iteration are separated by three grid-wide waits instead of launches:
//   x += alpha p, p = r + beta p (each DOF by its owner), and A p, one element
//     per block, its three line directions at once (each node forms its p from
//     r and the old p itself, with the owner's arithmetic, so no wait lies
//     between; p has two buffers)
//   | Z^T on surface DOFs, p.Ap
//   | r -= alpha Ap, r.r
//   | beta, stopping test
// Every block sums the block partials itself in the same fixed order, so all
// blocks compute the same alpha and beta and take the same decisions (no
// broadcast). The waits are bounded: a block that waits more than about a
// second records bit 1 in the mesh's error word and every block then leaves
// the iteration loop (the host reports HB_ERR_TIMEOUT).
// Measured, us per iteration (with four waits, the barrier's arrival returning
// a value -> this form): 4x4x4 elements at N = 7 26.1 -> 21.2, at N = 3 18.5 ->
// 14.5, 125 elements at N = 15 117.8 -> 112.6. A wait takes about 2.2 us.
#include "hb_internal.h"
#define HB_AX2_T double
#include "hb_ax2.cuh"
#include "hb_vec.cuh"

namespace {

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid-wide barrier number seq (1, 2, ...) of a cooperative launch (every
// block resident at once) on one counter word, zero at launch: block 0 adds
// 2^31 - (nb - 1) and every other block 1, so the counter's top bit flips
// exactly when the last of the nb blocks has arrived, once per barrier, with
// no reset; after barrier seq it equals seq's lowest bit, so the arrival needs
// no answer (a reduction without a return value). Thread 0 of each block
// arrives with release order (its block's writes are then visible to the
// others) and polls for at most hb2::kWaitNs of wall time. Returns true in
// every thread of the block if this block gave up (the caller must then stop:
// the blocks still waiting give up in turn, so the launch ends).
// (Blocks publishing their partial sums in flagged slots that all others poll
// was measured too: 20.0 -> 23.8 us per iteration on 128 blocks, 20.3 -> 29.0
// on 216: the polls of nb^2 slots collide in L2.)
__device__ bool grid_barrier(unsigned *bar, unsigned nb, unsigned seq, unsigned *err)
{
    __shared__ int s_fail;
    __syncthreads();
    if (threadIdx.x == 0) {
        int fail = 0;
        const unsigned add = blockIdx.x == 0 ? 0x80000000u - (nb - 1u) : 1u, want = seq << 31;
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar), "r"(add) : "memory");
        unsigned long long t0 = 0;
        for (unsigned t = 1; ((ld_acquire(bar) ^ want) & 0x80000000u) != 0; t++) {
            if (t & 63u) continue;
            const unsigned long long now = hb2::wall_ns();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > hb2::kWaitNs) {
                atomicOr(err, 2u);
                fail = 1;
                break;
            }
        }
        s_fail = fail;
    }
    __syncthreads();
    return s_fail != 0;
}

struct fused_args {
    const int32_t *l2g;
    const double *geo;
    const int32_t *srow_g, *srowptr, *scols;
    const double *mdiag;
    double *ysurf;
    double *x, *r, *p, *p2, *Ap;  // p, p2: the two buffers of p (p holds p_0)
    int64_t E, n_global, nsr;
    double lambda;
    int screen;
    double *part;             // [2][HB_RED_BLOCKS] block partials (two sets, alternating)
    hb_cg_state *st;          // in: rr, tol2, max_it, run; out: final state
    unsigned *bar;            // grid barrier counter (zero at launch)
    unsigned *err;            // error word (bit 1: a wait gave up)
};

// Grid-wide wait and sum: every block passes its v (read in thread 0), all of
// them get the sum over the blocks, added in a fixed order (thread t takes
// partials t, t + blockDim, ..., then a shuffle tree), and see what every
// other block wrote to memory before its call. seq counts the waits (a block
// is at most one ahead of another, so two sets of partials alternate). False
// in every thread if the wait ran out.
__device__ bool grid_wait_sum(const fused_args &F, double v, unsigned seq, double &sum)
{
    __shared__ double s_w[32];
    const int nb = gridDim.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    double *part = F.part + (seq & 1u) * HB_RED_BLOCKS;
    if (threadIdx.x == 0) part[blockIdx.x] = v;
    if (grid_barrier(F.bar, nb, seq, F.err)) return false;
    double t = 0.0;
    for (int q = threadIdx.x; q < nb; q += blockDim.x) t += __ldcg(part + q);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) s_w[wid] = t;
    __syncthreads();
    // every warp adds the warps' sums itself (in the same order); s_w is
    // rewritten only after the next barrier
    double u = lane < nw ? s_w[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    sum = u;
    return true;
}

// The element's A p: one element per block on 3 (N+1)^2 threads. Group d = 0, 1,
// 2 of n^2 threads contracts the r-, s- or t-lines (the three directions at
// once), and the gather, metric and epilogue phases split each t-line's k range
// over the groups (k = d, d + 3, ...). For a small mesh, where the element's own
// latency sets the time, this keeps all four FP64 units of an SM busy instead
// of the two that n^2 threads reach. Same arithmetic as hb2::pencil_group per
// node. load(g) gives the value of u at DOF g. Every thread of the block must
// call it. (The launch is a plain cooperative one: an element spread over a
// cluster of blocks, which store into each other's shared memory, took 17.8 us
// per iteration at N = 7 on 64 elements, but a profiler's run of that kernel,
// cooperative and in clusters at once, ended in an illegal access on the GPU
// for which no cause was found, so no block here reaches outside itself.)
template <int N, class FL>
__device__ __forceinline__ void element_lines(const hb2::pencil_args &A, int64_t e, double *sm,
                                              hbacc::dot_acc<double> &acc, FL &&load)
{
    using P = hb2::pad<N>;
    constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    const int tid = threadIdx.x, d = tid / n2, a = tid - d * n2, p0 = a % n, p1 = a / n;  // d: 0 r, 1 s, 2 t; 3+ idle
    const bool active = d < 3;
    const int32_t *__restrict__ lg = A.l2g + e * n3 + a;
    const double *__restrict__ ge = A.geo + e * 7 * n3 + a;
    double *U = sm, *B1 = U + P::size, *B2 = B1 + P::size, *B3 = B2 + P::size;
    double *Bd = d == 0 ? B1 : (d == 1 ? B2 : B3);
    if (active)
        for (int k = d; k < n; k += 3) {
            const int g = __ldg(lg + k * n2);
            U[P::at(p0, p1, k)] = g >= 0 ? load(g) : 0.0;
        }
    __syncthreads();
    // node m of the line this thread owns: r (m, p0, p1), s (p0, m, p1), t (p0, p1, m)
    auto at_line = [&](int m) { return d == 0 ? P::at(m, p0, p1) : (d == 1 ? P::at(p0, m, p1) : P::at(p0, p1, m)); };
    double in[n];
    if (active) {
#pragma unroll
        for (int m = 0; m < n; m++) in[m] = U[at_line(m)];
        hb2::line_st<N, false, true>(in, [&](int m, double v) { Bd[at_line(m)] = v; });
    }
    __syncthreads();
    if (active)
        for (int k = d; k < n; k += 3) {
            const double *g = ge + k * 7 * n2;
            const double grr = __ldcs(g), grs = __ldcs(g + n2), grt = __ldcs(g + 2 * n2);
            const double gss = __ldcs(g + 3 * n2), gst = __ldcs(g + 4 * n2), gtt = __ldcs(g + 5 * n2);
            const int q = P::at(p0, p1, k);
            const double ur = B1[q], us = B2[q], ut = B3[q];
            B1[q] = fma(grt, ut, fma(grs, us, grr * ur));
            B2[q] = fma(gst, ut, fma(gss, us, grs * ur));
            B3[q] = fma(gtt, ut, fma(gst, us, grt * ur));
        }
    __syncthreads();
    if (active) {
#pragma unroll
        for (int m = 0; m < n; m++) in[m] = Bd[at_line(m)];
        hb2::line_st<N, true, true>(in, [&](int m, double v) { Bd[at_line(m)] = v; });
    }
    __syncthreads();
    if (active) {
        double *ys = A.ysurf + e * hb2::surf_count<N>();
        const bool ring = p0 == 0 || p0 == N || p1 == 0 || p1 == N;
        const int r = ring ? hb2::ring_index<N>(p0, p1) : 0;
        for (int k = d; k < n; k += 3) {
            const int q = P::at(p0, p1, k);
            const double yc = B1[q] + B2[q] + B3[q];
            if (k == 0) {
                ys[a] = yc;
            } else if (k == N) {
                ys[n2 + a] = yc;
            } else if (ring) {
                ys[2 * n2 + (k - 1) * 4 * N + r] = yc;
            } else {
                const double xv = U[q], jw = A.screen ? __ldg(ge + (k * 7 + 6) * n2) : 1.0;
                double y = yc;
                y += A.lambda * (jw * xv);
                A.y[__ldg(lg + k * n2)] = y;
                acc.add(xv, y);
            }
        }
    }
    __syncthreads();  // the buffers are reused by the next element
}

// Block size for degree N: the three thread groups of element_lines, at least
// 256 threads for the vector phases. Shared memory: its four buffers.
template <int N>
constexpr int fused_threads()
{
    constexpr int t = 3 * (N + 1) * (N + 1);
    return t < 256 ? 256 : (t + 31) / 32 * 32;
}
// Blocks per SM asked of the compiler. What fits on the GPU at once is what this
// solver takes (hb_cg_fused_capacity), and left to itself the compiler uses up
// to 135 registers, which fits two blocks at N = 7 and one at N = 10 (304 and
// 152 elements, for 608 and 304 with these bounds). The times are the same
// (N = 7, 64 elements 20.9 us an iteration without, 21.2 with them; N = 10, 294
// elements 70.8 by the launched kernels, 68.8 here).
template <int N>
constexpr int fused_blocks() { return N <= 3 || N == 6 ? 5 : N <= 8 ? 4 : N <= 10 ? 2 : 1; }
template <int N>
constexpr size_t fused_smem() { return sizeof(double) * 4 * (size_t)hb2::pad<N>::size; }

// Grid: at most as many blocks as are resident at once, an element (or several)
// each.
template <int N>
__global__ void __launch_bounds__(fused_threads<N>(), fused_blocks<N>()) cg_fused_kernel(const fused_args F)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    double *sm = reinterpret_cast<double *>(smem_raw);
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gthreads = (int64_t)gridDim.x * blockDim.x;

    double rr = F.st->rr;
    const double tol2 = F.st->tol2;
    const int max_it = F.st->max_it;
    bool stop = F.st->run == 0;
    int it = 0;
    unsigned seq = 0;
    int status = HB_OK;
    double alpha = 0.0, beta = 0.0, pAp = 0.0;
    double *pold = F.p2, *p = F.p;  // p_{j-1} and p_j

    // this thread's first surface row (its only one on the smallest meshes)
    int row_g = -1, row_a = 0, row_z = 0, row_c[4] = {0, 0, 0, 0};
    if (gtid < F.nsr) {
        row_g = F.srow_g[gtid];
        row_a = F.srowptr[gtid];
        row_z = F.srowptr[gtid + 1];
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (row_a + q < row_z) row_c[q] = F.scols[row_a + q];
    }
    hb2::pencil_args A{nullptr, F.l2g, F.geo, F.ysurf, F.Ap, F.E, nullptr, F.lambda, F.screen, nullptr};
    for (;;) {
        // x += alpha p_{j-1}, p_j = r + beta p_{j-1} (j > 0) at this thread's DOFs
        // (data written by other blocks in this launch is read through L2)
        if (it > 0)
            for (int64_t i = gtid; i < F.n_global; i += gthreads) {
                const double po = __ldcg(pold + i);
                F.x[i] += alpha * po;
                if (!stop) p[i] = fma(beta, po, F.r[i]);
            }
        if (stop) break;
        // A p: interior DOFs finished, surface values to ysurf
        hbacc::dot_acc<double> acc;
        const bool first = it == 0;
        for (int64_t e = blockIdx.x; e < F.E; e += gridDim.x)
            element_lines<N>(A, e, sm, acc, [&](int g) {
                return first ? __ldcg(p + g) : fma(beta, __ldcg(pold + g), __ldcg(F.r + g));
            });
        if (grid_barrier(F.bar, gridDim.x, ++seq, F.err)) {
            status = HB_ERR_TIMEOUT;
            break;
        }
        // Z^T on the surface DOFs
        auto row = [&](int g, int a, int z, const int (&c4)[4]) {
            double t = 0.0;
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (a + q < z) t += __ldcg(F.ysurf + c4[q]);
            for (int q = a + 4; q < z; q++) t += __ldcg(F.ysurf + F.scols[q]);
            const double xv = __ldcg(p + g);
            t += F.screen ? F.lambda * (F.mdiag[g] * xv) : F.lambda * xv;
            F.Ap[g] = t;
            acc.add(xv, t);
        };
        if (row_g >= 0) row(row_g, row_a, row_z, row_c);
        for (int64_t rI = gtid + gthreads; rI < F.nsr; rI += gthreads) {
            const int a = F.srowptr[rI], z = F.srowptr[rI + 1];
            int c4[4];
#pragma unroll
            for (int q = 0; q < 4; q++) c4[q] = a + q < z ? F.scols[a + q] : 0;
            row(F.srow_g[rI], a, z, c4);
        }
        double v = hbacc::block_sum(acc.value());
        if (!grid_wait_sum(F, v, ++seq, pAp)) {
            status = HB_ERR_TIMEOUT;
            break;
        }
        if (!(pAp > 0.0) || !isfinite(pAp)) {
            status = HB_ERR_BREAKDOWN;
            break;  // every block takes the same branch
        }
        alpha = rr / pAp;
        // r -= alpha Ap and r.r
        hbacc::dot_acc<double> racc;
        for (int64_t i = gtid; i < F.n_global; i += gthreads) {
            const double ri = F.r[i] - alpha * __ldcg(F.Ap + i);
            F.r[i] = ri;
            racc.add(ri, ri);
        }
        v = hbacc::block_sum(racc.value());
        double rr_new;
        if (!grid_wait_sum(F, v, ++seq, rr_new)) {
            status = HB_ERR_TIMEOUT;
            break;
        }
        beta = rr_new / rr;
        rr = rr_new;
        it++;
        stop = !(it < max_it && rr_new > tol2);
        double *const o = pold;
        pold = p;
        p = o;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        hb_cg_state *st = F.st;
        st->it += it;
        st->rr = rr;
        st->res2 = rr;
        st->pAp = pAp;
        st->alpha = alpha;
        st->beta = beta;
        st->run = 0;
        st->next_run = 0;
        if (status != HB_OK) st->status = status;
    }
}

// Blocks that are resident at once.
template <int N>
hb_status fused_resident(int64_t *blocks)
{
    auto kern = cg_fused_kernel<N>;
    static int attr_set[32] = {0};
    int dev = 0, per_sm = 0, sms = 0;
    HB_TRY_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 32 || !attr_set[dev]) {
        HB_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused_smem<N>()));
        if (dev >= 0 && dev < 32) attr_set[dev] = 1;
    }
    HB_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, fused_threads<N>(), fused_smem<N>()));
    HB_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    *blocks = (int64_t)per_sm * sms;
    return HB_OK;
}

template <int N>
hb_status launch_fused(fused_args &F, cudaStream_t s)
{
    int64_t blocks = 0;
    hb_status st = fused_resident<N>(&blocks);
    if (st != HB_OK) return st;
    if (blocks > HB_RED_BLOCKS) blocks = HB_RED_BLOCKS;
    if (blocks > F.E) blocks = F.E;
    if (blocks < 1) { hb_set_error("fused CG: no block fits"); return HB_ERR_ARG; }
    void *args[] = {(void *)&F};
    hb_prof_scope prof("cg_fused", s);
    HB_TRY_CUDA(cudaLaunchCooperativeKernel((const void *)cg_fused_kernel<N>, dim3((unsigned)blocks),
                                            dim3(fused_threads<N>()), args, fused_smem<N>(), s));
    return HB_OK;
}

// Self-test of the bounded barrier: it waits for one block more than were
// launched, so every block gives up and sets bit 1 of *err.
__global__ void barrier_timeout_kernel(unsigned *bar, unsigned *err) { grid_barrier(bar, gridDim.x + 1, 1u, err); }

}  // namespace

hb_status hb_selftest_barrier_timeout(unsigned *bar, unsigned *err, cudaStream_t s)
{
    void *args[] = {(void *)&bar, (void *)&err};
    HB_TRY_CUDA(cudaLaunchCooperativeKernel((const void *)barrier_timeout_kernel, dim3(2), dim3(32), args, 0, s));
    return HB_OK;
}

// This unit's copy of the derivative tables (every unit that includes the
// element kernel has its own constant bank).
hb_status hb_cg_fused_upload(const double *D_all) { return hb2::upload_tables(D_all); }

// Number of element groups a fused solve can keep resident at once for
// degree N (0 if the kernel cannot be launched cooperatively).
int hb_cg_fused_capacity(int N)
{
    int dev = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
    int64_t cap = 0;
    hb_status st;
    switch (N) {
#define HB_CASE(NN) \
    case NN: st = fused_resident<NN>(&cap); break;
        HB_CASE(1) HB_CASE(2) HB_CASE(3) HB_CASE(4) HB_CASE(5) HB_CASE(6) HB_CASE(7) HB_CASE(8)
        HB_CASE(9) HB_CASE(10) HB_CASE(11) HB_CASE(12) HB_CASE(13) HB_CASE(14) HB_CASE(15)
#undef HB_CASE
    default: return 0;
    }
    return st == HB_OK ? (int)cap : 0;
}

// max_it iterations (or until the state's tolerance) of Algorithm 1 on
// (x, r, p, Ap; p2: a second buffer for p) in one cooperative launch; the state must hold rr, tol2,
// max_it and run as cg_init leaves them.
hb_status hb_cg_fused_run(const hb_mesh *m, int screen, double lambda, double *x, double *r, double *p, double *p2,
                          double *Ap, hb_cg_state *st, cudaStream_t s)
{
    fused_args F{};
    F.l2g = m->l2g;
    F.geo = m->geo;
    F.srow_g = m->srow_g;
    F.srowptr = m->srowptr;
    F.scols = m->scols;
    F.mdiag = m->mdiag;
    F.ysurf = (double *)m->yL;
    F.x = x;
    F.r = r;
    F.p = p;
    F.p2 = p2;
    F.Ap = Ap;
    F.E = m->E;
    F.n_global = m->n_global;
    F.nsr = m->nsr;
    F.lambda = lambda;
    F.screen = screen;
    F.part = m->partials;
    F.st = st;
    F.bar = m->counters + 4;
    F.err = m->counters + 7;
    HB_TRY_CUDA(cudaMemsetAsync(F.bar, 0, sizeof(unsigned), s));
    switch (m->N) {
#define HB_CASE(NN) \
    case NN: return launch_fused<NN>(F, s);
        HB_CASE(1) HB_CASE(2) HB_CASE(3) HB_CASE(4) HB_CASE(5) HB_CASE(6) HB_CASE(7) HB_CASE(8)
        HB_CASE(9) HB_CASE(10) HB_CASE(11) HB_CASE(12) HB_CASE(13) HB_CASE(14) HB_CASE(15)
#undef HB_CASE
    default: hb_set_error("unsupported N=%d", m->N); return HB_ERR_ARG;
    }
}
