// Instantiations of the element-local operator for T = double, N = 1..15.
#include "hb_ax.cuh"
#define HB_AX2_T double
#include "hb_ax2.cuh"

hb_status hb_launch_ax_local_f64(const hb_mesh *m, const double *x, double *yL, const int *run, cudaStream_t s)
{
    const double *Dg = hb_dev_D64(m->N);
    if (!m->geo) { hb_set_error("mesh has no double geometric factors"); return HB_ERR_ARG; }
    switch (m->N) {
#define HB_CASE(NN) \
    case NN: return hb::launch_ax_local<NN, double>(x, m->l2g, m->geo, yL, m->E, Dg, run, s);
        HB_CASE(1) HB_CASE(2) HB_CASE(3) HB_CASE(4) HB_CASE(5) HB_CASE(6) HB_CASE(7) HB_CASE(8)
        HB_CASE(9) HB_CASE(10) HB_CASE(11) HB_CASE(12) HB_CASE(13) HB_CASE(14) HB_CASE(15)
#undef HB_CASE
    default: hb_set_error("unsupported N=%d", m->N); return HB_ERR_ARG;
    }
}

hb_status hb_ax2_upload_f64(const double *D_all) { return hb2::upload_tables(D_all); }

// Pencil variant with the interior/surface split: eo selects the even-odd
// split, eb_mult = 2 doubles the elements per block (N <= 10). Interior DOFs
// are finished here (y, lambda term, partial of x.y); surface values go to
// ysurf for the surface gather.
hb_status hb_launch_ax2_f64(const hb_mesh *m, const double *x, double *ysurf, double *y, double lambda, int screen,
                            double *partials, const int *run, int eo, int eb_mult, cudaStream_t s,
                            int64_t *nblocks)
{
    if (!m->geo) { hb_set_error("mesh has no double geometric factors"); return HB_ERR_ARG; }
    hb2::pencil_args A{x, m->l2g, m->geo, ysurf, y, m->E, run, (double)lambda, screen, partials, nullptr,
                       m->counters + 7, (eb_mult & 8) ? m->spos : nullptr};
    switch (m->N) {
#define HB_CASE(NN) \
    case NN: return eo ? hb2::launch<NN, true>(A, eb_mult, s, nblocks) : hb2::launch<NN, false>(A, eb_mult, s, nblocks);
        HB_CASE(1) HB_CASE(2) HB_CASE(3) HB_CASE(4) HB_CASE(5) HB_CASE(6) HB_CASE(7) HB_CASE(8)
        HB_CASE(9) HB_CASE(10) HB_CASE(11) HB_CASE(12) HB_CASE(13) HB_CASE(14) HB_CASE(15)
#undef HB_CASE
    default: hb_set_error("unsupported N=%d", m->N); return HB_ERR_ARG;
    }
}

// Pencil kernel (even-odd, base block shape) on a contiguous range of E
// elements given by its own arrays (l2g, geo and ysurf start at the range's
// first element); l2g entries <= -2 read halo values. Used by the partitioned
// operator; eo and eb_mult are accepted for symmetry and not used.
hb_status hb_launch_ax2_f64_range(int N, int64_t E, const double *x, const double *halo, const int32_t *l2g,
                                  const double *geo, double *ysurf, double *y, double lambda, int screen,
                                  const int *run, int eo, int eb_mult, cudaStream_t s)
{
    (void)eo;
    (void)eb_mult;
    hb2::pencil_args A{x, l2g, geo, ysurf, y, E, run, lambda, screen, nullptr, halo};
    switch (N) {
#define HB_CASE(NN) \
    case NN: return hb2::launch<NN, true, hb2::GM_HALO>(A, 1, s, nullptr);
        HB_CASE(1) HB_CASE(2) HB_CASE(3) HB_CASE(4) HB_CASE(5) HB_CASE(6) HB_CASE(7) HB_CASE(8)
        HB_CASE(9) HB_CASE(10) HB_CASE(11) HB_CASE(12) HB_CASE(13) HB_CASE(14) HB_CASE(15)
#undef HB_CASE
    default: hb_set_error("unsupported N=%d", N); return HB_ERR_ARG;
    }
}

// Pencil kernel (even-odd, base block shape) on scattered vectors (x_L, y_L
// of length n_local, no l2g): interior nodes of every element get
// y_L = (S_L x_L) + lambda term, surface nodes go to ysurf for the
// gather-scatter; eo and eb_mult are accepted for symmetry and not used.
hb_status hb_launch_ax2_f64_scat(const hb_mesh *m, const double *xL, double *ysurf, double *yL, double lambda,
                                 int screen, const int *run, int eo, int eb_mult, cudaStream_t s)
{
    if (!m->geo) { hb_set_error("mesh has no double geometric factors"); return HB_ERR_ARG; }
    (void)eo;
    (void)eb_mult;
    hb2::pencil_args A{xL, nullptr, m->geo, ysurf, yL, m->E, run, lambda, screen, nullptr, nullptr};
    switch (m->N) {
#define HB_CASE(NN) \
    case NN: return hb2::launch<NN, true, hb2::GM_SCAT>(A, 1, s, nullptr);
        HB_CASE(1) HB_CASE(2) HB_CASE(3) HB_CASE(4) HB_CASE(5) HB_CASE(6) HB_CASE(7) HB_CASE(8)
        HB_CASE(9) HB_CASE(10) HB_CASE(11) HB_CASE(12) HB_CASE(13) HB_CASE(14) HB_CASE(15)
#undef HB_CASE
    default: hb_set_error("unsupported N=%d", m->N); return HB_ERR_ARG;
    }
}

// One element of N = 3 on zeros through the split kernel told that it runs in a
// cluster of two, which the launch makes or (clustered = 0) does not.
extern "C" hb_status hb_selftest_cluster(int clustered, hb_status *status, void *stream)
{
    hb_clear_error();
    if (!status) { hb_set_error("null argument"); return HB_ERR_ARG; }
    if (clustered != 0 && clustered != 1) { hb_set_error("clustered must be 0 or 1"); return HB_ERR_ARG; }
    hb_status st = hb_ensure_device_tables();
    if (st != HB_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    constexpr int N = 3, n3 = 64, NS = hb2::surf_count<N>();
    struct buf {
        double geo[7 * n3], ysurf[NS], x[1], y[1], partials[2];
        int32_t l2g[n3];
        unsigned err;
    } *d = nullptr, h{};
    HB_TRY_CUDA(cudaMalloc((void **)&d, sizeof(buf)));
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof(buf), s);
    if (e == cudaSuccess) {
        const hb2::pencil_args A{d->x, d->l2g, d->geo, d->ysurf, d->y, 1, nullptr, 0.0, 0, d->partials, nullptr, &d->err};
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(2);
        cfg.blockDim = dim3((unsigned)hb2::split<N>::threads(2));
        cfg.dynamicSmemBytes = hb2::split<N>::smem(2);
        cfg.stream = s;
        cfg.attrs = at;
        cfg.numAttrs = clustered;
        hb_count_launch();
        e = cudaLaunchKernelEx(&cfg, hb2::ax_split_kernel<N, true>, A, 2);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(buf), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) {
        hb_set_error("self-test: %s", cudaGetErrorString(e));
        return HB_ERR_CUDA;
    }
    bool nan = std::isnan(h.y[0]) && std::isnan(h.partials[0]) && std::isnan(h.partials[1]);
    bool zero = h.y[0] == 0.0 && h.partials[0] == 0.0 && h.partials[1] == 0.0;
    for (double v : h.ysurf) {
        nan = nan && std::isnan(v);
        zero = zero && v == 0.0;
    }
    *status = hb_dev_err_status(h.err);
    if (*status == HB_OK ? !zero : !nan) { hb_set_error("self-test: unexpected values"); return HB_ERR_CUDA; }
    return HB_OK;
}

int hb_surf_count(int N) { return 2 * (N + 1) * (N + 1) + 4 * N * (N - 1); }

// ---------------------------------------------------------------- serving

#include "hb_serve.h"

namespace hb2 {
namespace {

template <int N, int TH>
__host__ __device__ constexpr int serve_eb() { return TH / ((N + 1) * (N + 1)); }
template <int LO, int HI, int TH>
constexpr size_t serve_smem_range()
{
    constexpr size_t m = sizeof(T) * 4 * serve_eb<LO, TH>() * pad<LO>::size;
    if constexpr (LO == HI) return m;
    else return m > serve_smem_range<LO + 1, HI, TH>() ? m : serve_smem_range<LO + 1, HI, TH>();
}

// Degree dispatch over [NN, HI] (only these degrees are instantiated).
template <int NN, int HI, int TH>
__device__ __forceinline__ void serve_dispatch(int N, const pencil_args &A, T *sm, hbacc::dot_acc<S> &acc)
{
    if (N == NN) {
        constexpr int EB = serve_eb<NN, TH>();
        const int64_t ngroups = (A.E + EB - 1) / EB;
        for (int64_t g = blockIdx.x; g < ngroups; g += gridDim.x) pencil_group<NN, true, EB>(A, g, sm, acc);
    } else if constexpr (NN < HI) {
        serve_dispatch<NN + 1, HI, TH>(N, A, sm, acc);
    }
}

// One slot's FP64 element kernel for the degrees [LO, HI] (the slot's degree is
// read from its descriptor), two blocks of TH threads per SM, each walking
// element groups grid-stride. The degree classes are those of the FP32 kernel:
// one kernel for every degree took 186 registers, so one block per SM, five
// warps of it busy at N = 11 (a burst of 24 requests of 2..16 elements per axis
// 44.3 -> 43.4 ms).
template <int LO, int HI, int TH>
__global__ void __launch_bounds__(TH, 2)
    serve_ax_kernel(const hb_slot_desc *__restrict__ D, const hb_slot_state *__restrict__ St)
{
    const hb_slot_desc &d = *D;
    if (!d.active || St->phase != HB_SLOT_OUTER || d.N < LO || d.N > HI) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    pencil_args A{(const T *)d.x, d.l2g, d.geo, (T *)d.ysurf, (T *)d.Ap, d.E, nullptr, (T)d.lambda,
                  d.screen, nullptr};
    hbacc::dot_acc<S> acc;
    serve_dispatch<LO, HI, TH>(d.N, A, reinterpret_cast<T *>(smem_raw), acc);
}

template <int LO, int HI, int TH>
hb_status serve_class_params(cudaKernelNodeParams *p)
{
    auto kern = serve_ax_kernel<LO, HI, TH>;
    constexpr size_t smem = serve_smem_range<LO, HI, TH>();
    static int attr_set[32] = {0};
    int dev = 0;
    HB_TRY_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 32 || !attr_set[dev]) {
        HB_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        if (dev >= 0 && dev < 32) attr_set[dev] = 1;
    }
    *p = cudaKernelNodeParams{};
    p->func = (void *)kern;
    p->gridDim = dim3(HB_SERVE_GRID);
    p->blockDim = dim3(TH);
    p->sharedMemBytes = (unsigned)smem;
    return HB_OK;
}

}  // namespace
}  // namespace hb2

hb_status hb_serve_ax_f64_params(int cls, cudaKernelNodeParams *p)
{
    return cls == 0   ? hb2::serve_class_params<1, 7, 256>(p)
           : cls == 1 ? hb2::serve_class_params<8, 10, 256>(p)
                      : hb2::serve_class_params<11, 11, 144>(p);
}
