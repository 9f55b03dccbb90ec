// Mesh setup on the device: reference element, node map, Z^T as CSR and the
// geometric factors (hipBone, arXiv 2202.12477, Sec. 2 and Sec. 3.2).
//
// Routes chosen here on purpose differ from the textbook closed forms:
//   - GLL nodes by Newton's method on q(x) = (1-x^2) P_N'(x) written as
//     N (P_{N-1}(x) - x P_N(x)), with q'(x) = -N(N+1) P_N(x);
//   - the derivative matrix from barycentric weights, diagonal by negative sums;
//   - the Jacobian's columns from halved edge differences of the element's eight
//     vertices, bilinear in the other two coordinates (the trilinear map has no
//     other terms), not by applying the derivative matrix to nodal coordinates.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "hb_internal.h"

// ---------------------------------------------------------------- errors

static thread_local char g_err[512];

void hb_set_error(const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
}
void hb_clear_error() { g_err[0] = 0; }

extern "C" const char *hb_last_error(void) { return g_err; }

// ---------------------------------------------------------------- random numbers

__host__ __device__ static inline uint64_t hb_splitmix64(uint64_t state)
{
    uint64_t z = state + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__host__ __device__ static inline double hb_u01_impl(uint64_t seed, uint64_t stream, uint64_t idx)
{
    uint64_t s = (seed ^ (stream * 0x9E3779B97F4A7C15ull)) + idx;
    return (double)(hb_splitmix64(s) >> 11) * 0x1.0p-53;
}

extern "C" double hb_u01(uint64_t seed, uint64_t stream, uint64_t idx)
{
    return hb_u01_impl(seed, stream, idx);
}

// ---------------------------------------------------------------- reference element

static void legendre_pair(int N, double x, double *PN, double *PNm1)
{
    double a = 1.0, b = x;  // P_0, P_1
    if (N == 1) { *PN = b; *PNm1 = a; return; }
    for (int k = 2; k <= N; k++) {
        double c = ((2 * k - 1) * x * b - (k - 1) * a) / k;
        a = b;
        b = c;
    }
    *PN = b;
    *PNm1 = a;
}

void hb_reference_element(int N, double *xi, double *w, double *D)
{
    const int n = N + 1;
    xi[0] = -1.0;
    xi[N] = 1.0;
    for (int i = 1; i < N; i++) {
        double x = -std::cos(M_PI * i / N);
        for (int it = 0; it < 200; it++) {
            double P, Pm;
            legendre_pair(N, x, &P, &Pm);
            // q = N (P_{N-1} - x P_N), q' = -N (N+1) P_N  =>  dx = -q / q'
            double dx = (Pm - x * P) / ((N + 1) * P);
            x += dx;
            if (std::fabs(dx) <= 1e-17) break;
        }
        xi[i] = x;
    }
    for (int i = 0; i < n / 2; i++) {  // symmetric node set
        double a = 0.5 * (xi[N - i] - xi[i]);
        xi[i] = -a;
        xi[N - i] = a;
    }
    if (N % 2 == 0) xi[N / 2] = 0.0;
    for (int i = 0; i < n; i++) {
        double P, Pm;
        legendre_pair(N, xi[i], &P, &Pm);
        w[i] = 2.0 / (N * (N + 1.0) * P * P);
    }
    // barycentric weights lambda_j = 1 / prod_{k != j} (x_j - x_k)
    std::vector<double> lam(n);
    for (int j = 0; j < n; j++) {
        double p = 1.0;
        for (int k = 0; k < n; k++)
            if (k != j) p *= (xi[j] - xi[k]);
        lam[j] = 1.0 / p;
    }
    for (int i = 0; i < n; i++) {
        double diag = 0.0;
        for (int j = 0; j < n; j++) {
            if (i == j) continue;
            double v = (lam[j] / lam[i]) / (xi[i] - xi[j]);
            D[i * n + j] = v;
            diag -= v;
        }
        D[i * n + i] = diag;
    }
    // D is centro-antisymmetric; make the computed matrix exactly so
    for (int i = 0; i < n; i++)
        for (int j = 0; j < n; j++) {
            int ii = N - i, jj = N - j;
            if (i * n + j < ii * n + jj) {
                double a = 0.5 * (D[i * n + j] - D[ii * n + jj]);
                D[i * n + j] = a;
                D[ii * n + jj] = -a;
            } else if (i == ii && j == jj) {
                D[i * n + j] = 0.0;
            }
        }
}

// ---------------------------------------------------------------- device tables

static int d_offset(int N)
{
    int o = 0;
    for (int M = 1; M < N; M++) o += (M + 1) * (M + 1);
    return o;
}
static const int kTableSize = 1496;  // sum_{N=1..15} (N+1)^2 = 1495

__device__ double g_D64[kTableSize];
__device__ float g_D32[kTableSize];
__device__ double g_xi64[16 * 16];   // [N][i]
__device__ double g_w64[16 * 16];

static std::mutex g_table_mu;
static unsigned g_table_done = 0;  // bit per device (devices 0..31)
static double *g_dev_D64[32];
static float *g_dev_D32[32];

hb_status hb_ensure_device_tables()
{
    int dev = 0;
    HB_TRY_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 32) { hb_set_error("device index %d unsupported", dev); return HB_ERR_ARG; }
    std::lock_guard<std::mutex> lk(g_table_mu);
    if (g_table_done & (1u << dev)) return HB_OK;
    std::vector<double> D64(kTableSize, 0.0), xi(256, 0.0), w(256, 0.0);
    std::vector<float> D32(kTableSize, 0.0f);
    for (int N = 1; N <= HB_MAX_N; N++) {
        int n = N + 1;
        std::vector<double> x(n), ww(n), D(n * n);
        hb_reference_element(N, x.data(), ww.data(), D.data());
        for (int q = 0; q < n * n; q++) {
            D64[d_offset(N) + q] = D[q];
            D32[d_offset(N) + q] = (float)D[q];
        }
        for (int i = 0; i < n; i++) { xi[N * 16 + i] = x[i]; w[N * 16 + i] = ww[i]; }
    }
    { hb_status st2 = hb_ax2_upload_f64(D64.data()); if (st2 != HB_OK) return st2; }
    { hb_status st2 = hb_ax2_upload_f32(D64.data()); if (st2 != HB_OK) return st2; }
    { hb_status st2 = hb_ax2_upload_f64x(D64.data()); if (st2 != HB_OK) return st2; }
    { hb_status st2 = hb_cg_fused_upload(D64.data()); if (st2 != HB_OK) return st2; }
    { hb_status st2 = hb_tc_upload(); if (st2 != HB_OK) return st2; }
    HB_TRY_CUDA(cudaMemcpyToSymbol(g_D64, D64.data(), sizeof(double) * kTableSize));
    HB_TRY_CUDA(cudaMemcpyToSymbol(g_D32, D32.data(), sizeof(float) * kTableSize));
    HB_TRY_CUDA(cudaMemcpyToSymbol(g_xi64, xi.data(), sizeof(double) * 256));
    HB_TRY_CUDA(cudaMemcpyToSymbol(g_w64, w.data(), sizeof(double) * 256));
    void *p64 = nullptr, *p32 = nullptr;
    HB_TRY_CUDA(cudaGetSymbolAddress(&p64, g_D64));
    HB_TRY_CUDA(cudaGetSymbolAddress(&p32, g_D32));
    g_dev_D64[dev] = (double *)p64;
    g_dev_D32[dev] = (float *)p32;
    g_table_done |= 1u << dev;
    return HB_OK;
}

const double *hb_dev_D64(int N)
{
    int dev = 0;
    cudaGetDevice(&dev);
    return g_dev_D64[dev] + d_offset(N);
}
const float *hb_dev_D32(int N)
{
    int dev = 0;
    cudaGetDevice(&dev);
    return g_dev_D32[dev] + d_offset(N);
}

// ---------------------------------------------------------------- setup kernels

static int grid_for(int64_t n, int threads)
{
    int64_t g = (n + threads - 1) / threads;
    if (g > 152 * 32) g = 152 * 32;
    return (int)(g < 1 ? 1 : g);
}


struct box_t {
    int Ex, Ey, Ez, N;
    unsigned faces;
};

// One axis of the box's lattice: Ex elements of degree N, points 0 .. N Ex, of
// which x0 at the low end (0 or 1, masked) and possibly the last are no DOFs.
// Point I is held by mult(I) elements along the axis (two on a shared face).
struct axis_t {
    int N, Ex, x0, nu;  // nu: unmasked points
    __host__ __device__ int mult(int I) const { return I % N == 0 && I > 0 && I < N * Ex ? 2 : 1; }
    // sum of mult over the unmasked points before I (a point), and over all
    __host__ __device__ int64_t copies_before(int I) const { return I - x0 + (I > 0 ? (I - 1) / N : 0); }
    __host__ __device__ int64_t copies() const { return nu > 0 ? (int64_t)nu + Ex - 1 : 0; }
    // points strictly inside an element: before I, and all
    __host__ __device__ int64_t inner_before(int I) const { return I - (I + N - 1) / N; }
    __host__ __device__ int64_t inner() const { return (int64_t)Ex * (N - 1); }
};
struct lattice3 {
    axis_t x, y, z;
};
static lattice3 box_lattice(const box_t &b)
{
    auto axis = [&](int E, unsigned lo, unsigned hi) {
        const int x0 = b.faces & lo ? 1 : 0, x1 = b.faces & hi ? 1 : 0;
        return axis_t{b.N, E, x0, b.N * E + 1 - x0 - x1};
    };
    return {axis(b.Ex, 1u, 2u), axis(b.Ey, 4u, 8u), axis(b.Ez, 16u, 32u)};
}

__device__ inline void vertex_pos(const box_t &b, double rho, uint64_t seed, int a, int bb, int c,
                                  double X[3])
{
    X[0] = (double)a / b.Ex;
    X[1] = (double)bb / b.Ey;
    X[2] = (double)c / b.Ez;
    if (a > 0 && a < b.Ex && bb > 0 && bb < b.Ey && c > 0 && c < b.Ez) {
        const double h[3] = {1.0 / b.Ex, 1.0 / b.Ey, 1.0 / b.Ez};
        uint64_t v = ((uint64_t)c * (b.Ey + 1) + bb) * (b.Ex + 1) + a;
        for (int ax = 0; ax < 3; ax++) {
            double u = hb_u01_impl(seed, 1, 3 * v + ax);
            X[ax] += (2.0 * u - 1.0) * rho * h[ax];
        }
    }
}

// Geometric factors, one element per block. The element map is trilinear in
// its 8 vertices, x(r, s, t) = sum_{a,b,c} V_abc phi_a(r) phi_b(s) phi_c(t)
// with phi_0 = (1 - r) / 2, phi_1 = (1 + r) / 2, so its Jacobian column along
// one reference direction is bilinear in the other two coordinates:
//   dx/dr = sum_{b,c} (V_1bc - V_0bc) / 2 phi_b(s) phi_c(t)
// (and likewise for s and t). Each column is formed once per line of nodes
// (3 n^2 lines per element, not n^3 nodes) and shared through shared memory;
// per node, with the adjugate rows a_l (a_r = j_s x j_t, a_s = j_t x j_r,
// a_t = j_r x j_s) and det J = j_r . a_r,
//   G_lm = w_ijk det J (J^-1 J^-T)_lm = (w_ijk / det J) a_l . a_m,
// the six factors of Sec. 2 and the weighted Jacobian w_ijk det J.
// Bound by the FP64 rate (about 60 operations per node, 2 per clock and SM), so
// what can be is integer work: the node map (lexicographic ids over unmasked
// lattice nodes, by closed form) rides along, the smallest det J is found on
// its bits, the FP32 copies are rounded by integer instructions (conversions
// run at the FP64 rate), and w_i w_j comes from a table: 7.0 -> 6.25 ms for
// 32x32x31, N = 11 with FP32 copies (6.12 without), and the node map's own pass
// of 0.40 ms gone.

// Order-preserving unsigned key of a double, and back.
__host__ __device__ inline unsigned long long order_key(double v)
{
    unsigned long long b;
    memcpy(&b, &v, sizeof b);
    return b >> 63 ? ~b : b | (1ull << 63);
}
static double from_order_key(unsigned long long k)
{
    const unsigned long long b = k >> 63 ? k & ~(1ull << 63) : ~k;
    double v;
    memcpy(&v, &b, sizeof v);
    return v;
}

// (float)v, to nearest even: a carry from the 29 dropped bits may step the
// exponent; outside FP32's normal range the conversion instruction.
__device__ __forceinline__ float round_to_float(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned e = (unsigned)(b >> 52) & 0x7FFu;
    if (e - 897u > 1149u - 897u) return (float)v;
    const unsigned long long r = b + ((1ull << 28) - 1ull + ((b >> 29) & 1ull));
    const unsigned m = (unsigned)(r >> 29) - (896u << 23);  // (bits above 31 drop out)
    return __uint_as_float((m & 0x7FFFFFFFu) | ((unsigned)(b >> 32) & 0x80000000u));
}

__global__ void k_geometry(box_t b, lattice3 L, double rho, uint64_t seed, int64_t E, int32_t *l2g, double *geo,
                           float *geo32, unsigned long long *detmin)
{
    extern __shared__ double smem[];
    const int N = b.N, n = N + 1, n2 = n * n, n3 = n2 * n;
    double *col = smem;  // [direction l][axis][line (u + n v)]: column l of J on the line
    __shared__ double V[8][3];
    __shared__ double dV[3][4][3];  // [direction][pair (p + 2 q)][axis]: halved edge differences
    __shared__ double ww[256], wk[16];
    const double *xi = g_xi64 + N * 16, *w = g_w64 + N * 16;
    unsigned long long kmin = ~0ull;
    for (int t = threadIdx.x; t < n2; t += blockDim.x) ww[t] = w[t % n] * w[t / n];
    if (threadIdx.x < n) wk[threadIdx.x] = w[threadIdx.x];
    for (int64_t e = blockIdx.x; e < E; e += gridDim.x) {
        const int ex = (int)(e % b.Ex), ey = (int)((e / b.Ex) % b.Ey), ez = (int)(e / ((int64_t)b.Ex * b.Ey));
        __syncthreads();  // the previous element's columns are consumed
        if (threadIdx.x < 8) {
            const int a = threadIdx.x & 1, bb = (threadIdx.x >> 1) & 1, c = threadIdx.x >> 2;
            vertex_pos(b, rho, seed, ex + a, ey + bb, ez + c, V[threadIdx.x]);
        }
        __syncthreads();
        if (threadIdx.x < 36) {
            // vertex (a, bb, c) at (c * 2 + bb) * 2 + a. Direction l steps a (r),
            // bb (s) or c (t); p and q are the vertex sides of the line's first
            // and second coordinate: (bb, c) for r, (a, c) for s, (a, bb) for t
            const int l = threadIdx.x / 12, pq = (threadIdx.x / 3) % 4, ax = threadIdx.x % 3;
            const int p = pq & 1, q = pq >> 1;
            const int v0 = l == 0 ? (q * 2 + p) * 2 : (l == 1 ? q * 4 + p : q * 2 + p);
            const int step = 1 << l;
            dV[l][pq][ax] = 0.5 * (V[v0 + step][ax] - V[v0][ax]);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < 3 * n2; t += blockDim.x) {
            const int l = t / n2, line = t % n2, u = line % n, v = line / n;
            // the two coordinates of the line: (s, t) for l = r, (r, t) for l = s, (r, s) for l = t
            const double fu0 = 0.5 - 0.5 * xi[u], fu1 = 0.5 + 0.5 * xi[u];
            const double fv0 = 0.5 - 0.5 * xi[v], fv1 = 0.5 + 0.5 * xi[v];
            for (int ax = 0; ax < 3; ax++) {
                // pair (p, q): p the first line coordinate's vertex side, q the second's
                const double c0 = fma(dV[l][1][ax], fu1, dV[l][0][ax] * fu0);
                const double c1 = fma(dV[l][3][ax], fu1, dV[l][2][ax] * fu0);
                col[(l * 3 + ax) * n2 + line] = fma(c1, fv1, c0 * fv0);
            }
        }
        __syncthreads();
        for (int q = threadIdx.x; q < n3; q += blockDim.x) {
            const int i = q % n, j = (q / n) % n, k = q / n2;
            double jr[3], js[3], jt[3];
            for (int ax = 0; ax < 3; ax++) {
                jr[ax] = col[(0 * 3 + ax) * n2 + j + n * k];
                js[ax] = col[(1 * 3 + ax) * n2 + i + n * k];
                jt[ax] = col[(2 * 3 + ax) * n2 + i + n * j];
            }
            double ar[3], as[3], at[3];
            ar[0] = fma(js[1], jt[2], -js[2] * jt[1]);
            ar[1] = fma(js[2], jt[0], -js[0] * jt[2]);
            ar[2] = fma(js[0], jt[1], -js[1] * jt[0]);
            as[0] = fma(jt[1], jr[2], -jt[2] * jr[1]);
            as[1] = fma(jt[2], jr[0], -jt[0] * jr[2]);
            as[2] = fma(jt[0], jr[1], -jt[1] * jr[0]);
            at[0] = fma(jr[1], js[2], -jr[2] * js[1]);
            at[1] = fma(jr[2], js[0], -jr[0] * js[2]);
            at[2] = fma(jr[0], js[1], -jr[1] * js[0]);
            const double det = fma(jr[2], ar[2], fma(jr[1], ar[1], jr[0] * ar[0]));
            const double wq = ww[j * n + i] * wk[k];
            const double sc = wq / det;
            double g[7];
            g[0] = sc * fma(ar[2], ar[2], fma(ar[1], ar[1], ar[0] * ar[0]));
            g[1] = sc * fma(ar[2], as[2], fma(ar[1], as[1], ar[0] * as[0]));
            g[2] = sc * fma(ar[2], at[2], fma(ar[1], at[1], ar[0] * at[0]));
            g[3] = sc * fma(as[2], as[2], fma(as[1], as[1], as[0] * as[0]));
            g[4] = sc * fma(as[2], at[2], fma(as[1], at[1], as[0] * at[0]));
            g[5] = sc * fma(at[2], at[2], fma(at[1], at[1], at[0] * at[0]));
            g[6] = wq * det;
            const int64_t base = ((e * n + k) * 7) * (int64_t)n2 + j * n + i;
            for (int c = 0; c < 7; c++) {
                geo[base + (int64_t)c * n2] = g[c];
                if (geo32) geo32[base + (int64_t)c * n2] = round_to_float(g[c]);
            }
            kmin = min(kmin, order_key(det));
            const int I = N * ex + i - L.x.x0, J = N * ey + j - L.y.x0, K = N * ez + k - L.z.x0;
            const bool dof = (unsigned)I < (unsigned)L.x.nu && (unsigned)J < (unsigned)L.y.nu && (unsigned)K < (unsigned)L.z.nu;
            l2g[e * n3 + q] = dof ? I + L.x.nu * (J + L.y.nu * K) : -1;
        }
    }
    // smallest det J
    for (int o = 16; o > 0; o >>= 1) kmin = min(kmin, __shfl_down_sync(0xffffffffu, kmin, o));
    if ((threadIdx.x & 31) == 0) atomicMin(detmin, kmin);
}

// ---------------------------------------------------------------- rows of Z^T

// Same order as the element kernels: k = 0 face, k = N face, then the ring
// of 4N nodes of each slab k = 1..N-1.
__device__ __forceinline__ int surf_index(int i, int j, int k, int N)
{
    const int n = N + 1, n2 = n * n;
    if (k == 0) return j * n + i;
    if (k == N) return n2 + j * n + i;
    const int r = j == 0 ? i : (j == N ? n + i : 2 * n + 2 * (j - 1) + (i == N ? 1 : 0));
    return 2 * n2 + (k - 1) * 4 * N + r;
}

// Z^T by the box's lattice, both as CSR over all DOFs and restricted to the
// DOFs on element surfaces, with the lumped mass diagonal: row g is lattice
// point (I, J, K), its copies are node (I - N ex, ...) of the elements that hold
// it, and where a row starts is a sum of products of per-axis counts. One pass,
// no counting, scan or sort: one warp per lattice row (J, K), lanes along I. The
// copies of a row ascend by element, as do the columns; the mass is summed in
// that order. 0.62 ms for 32x32x31, N = 11, where counting by atomics, scans,
// filling and sorting the rows took 3.1 ms and five waits of the host.
constexpr int kRowChunk = 1024;
__global__ void __launch_bounds__(256)
    k_rows(lattice3 L, const double *__restrict__ geo, int32_t *__restrict__ rowptr, int32_t *__restrict__ cols,
           double *__restrict__ mdiag, float *__restrict__ mdiag32, int32_t *__restrict__ srow_g,
           int32_t *__restrict__ srowptr, int32_t *__restrict__ scols)
{
    const int N = L.x.N, n = N + 1, n2 = n * n, NS = 2 * n2 + 4 * N * (N - 1);
    const int64_t n3 = (int64_t)n2 * n, TX = L.x.copies(), TY = L.y.copies();
    const int64_t SX = L.x.inner(), SY = L.y.inner();
    const int lane = threadIdx.x & 31;
    const int64_t nrows = (int64_t)L.y.nu * L.z.nu, nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int nch = (L.x.nu + kRowChunk - 1) / kRowChunk;  // (long rows go to several warps)
    for (int64_t unit = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; unit < nrows * nch; unit += nwarps) {
        const int64_t row = unit / nch;
        const int I0 = (int)(unit - row * nch) * kRowChunk, I1 = min(I0 + kRowChunk, L.x.nu);
        const int Ku = (int)(row / L.y.nu), Ju = (int)(row - (int64_t)Ku * L.y.nu);
        const int J = Ju + L.y.x0, K = Ku + L.z.x0;
        const int my = L.y.mult(J), mz = L.z.mult(K);
        const bool in_yz = J % N != 0 && K % N != 0;
        // copies and interior DOFs (one copy each) before this row
        const int64_t c0 = TX * (L.z.copies_before(K) * TY + mz * L.y.copies_before(J));
        const int64_t i0 = SX * (L.z.inner_before(K) * SY + (K % N != 0 ? L.y.inner_before(J) : 0));
        // the first element along y and z, and the local index in it
        const int ey0 = J == 0 ? 0 : (J - 1) / N, ez0 = K == 0 ? 0 : (K - 1) / N, j0 = J - N * ey0, k0 = K - N * ez0;
        for (int Iu = I0 + lane; Iu < I1; Iu += 32) {
            const int I = Iu + L.x.x0, mx = L.x.mult(I), ex0 = I == 0 ? 0 : (I - 1) / N, li = I - N * ex0;
            const int64_t g = row * L.x.nu + Iu, at = c0 + (int64_t)my * mz * L.x.copies_before(I);
            const int64_t before = i0 + (in_yz ? L.x.inner_before(I) : 0);
            const bool surf = !(in_yz && I % N != 0);
            const int64_t sat = at - before;
            rowptr[g] = (int32_t)at;
            if (surf) {
                srow_g[g - before] = (int32_t)g;
                srowptr[g - before] = (int32_t)sat;
            }
            double m = 0.0;
            int q = 0;
            for (int cz = 0; cz < mz; cz++)
                for (int cy = 0; cy < my; cy++)
                    for (int cx = 0; cx < mx; cx++, q++) {
                        // a second element starts at the shared point
                        const int i = cx ? 0 : li, j = cy ? 0 : j0, k = cz ? 0 : k0;
                        const int64_t e = (ex0 + cx) + (int64_t)L.x.Ex * ((ey0 + cy) + (int64_t)L.y.Ex * (ez0 + cz));
                        cols[at + q] = (int32_t)(e * n3 + (k * n + j) * n + i);
                        if (surf) scols[sat + q] = (int32_t)(e * NS + surf_index(i, j, k, N));
                        m += geo[((e * n + k) * 7 + 6) * (int64_t)n2 + j * n + i];
                    }
            mdiag[g] = m;
            if (mdiag32) mdiag32[g] = (float)m;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t ng = nrows * L.x.nu, nnz = TX * TY * L.z.copies(), in = SX * SY * L.z.inner();
        rowptr[ng] = (int32_t)nnz;
        srowptr[ng - in] = (int32_t)(nnz - in);
    }
}

__global__ void k_spos(const int32_t *__restrict__ scols, int64_t nnz, int32_t *__restrict__ spos)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x)
        spos[scols[q]] = (int32_t)q;
}

// CSR position of every surface copy (the inverse of scols), -1 for masked
// surface nodes; built the first time a variant that writes it is chosen.
hb_status hb_mesh_ensure_spos(hb_mesh *m, cudaStream_t s)
{
    if (m->spos) return HB_OK;
    const int64_t total = m->E * (int64_t)hb_surf_count(m->N);
    int32_t *p = nullptr;
    HB_TRY_CUDA(cudaMalloc((void **)&p, sizeof(int32_t) * (total > 0 ? total : 1)));
    cudaError_t e = cudaMemsetAsync(p, 0xFF, sizeof(int32_t) * (total > 0 ? total : 1), s);
    if (e == cudaSuccess && m->nnz_s > 0) {
        hb_count_launch();
        k_spos<<<grid_for(m->nnz_s, 256), 256, 0, s>>>(m->scols, m->nnz_s, p);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        cudaFree(p);
        hb_set_error("surface positions: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? HB_ERR_NOMEM : HB_ERR_CUDA;
    }
    hb_mesh_drop_graphs(m);  // captured runs hold the array pointer of the time
    m->spos = p;
    m->device_bytes += sizeof(int32_t) * (size_t)total;
    return HB_OK;
}

void hb_mesh_drop_graphs(hb_mesh *m)
{
    for (auto &g : m->graphs)
        if (g.exec) {
            cudaGraphExecDestroy(g.exec);
            g.exec = nullptr;
        }
}

// ---------------------------------------------------------------- mesh lifetime


// Frees everything the mesh holds. The arrays allocated while it was built
// are stream-ordered (freed on s); the ones grown later by the solvers and the
// autotuner (cg_vec, spos, inv_diag) are plain allocations.
static void mesh_free(hb_mesh *m, cudaStream_t s)
{
    hb_dev_free(m->l2g, s);
    hb_dev_free(m->geo, s);
    hb_dev_free(m->geo32, s);
    hb_dev_free(m->rowptr, s);
    hb_dev_free(m->cols, s);
    hb_dev_free(m->mdiag, s);
    hb_dev_free(m->mdiag32, s);
    hb_dev_free(m->yL, s);
    hb_dev_free(m->partials, s);
    hb_dev_free(m->counters, s);
    hb_dev_free(m->state, s);
    hb_dev_free(m->srow_g, s);
    hb_dev_free(m->srowptr, s);
    hb_dev_free(m->scols, s);
    hb_dev_free(m->ax_partials, s);
    // (a plain cudaFree may wait for the device: only for arrays that exist)
    if (m->cg_vec) cudaFree(m->cg_vec);
    if (m->spos) cudaFree(m->spos);
    if (m->inv_diag) cudaFree(m->inv_diag);
    if (m->inv_diag32) cudaFree(m->inv_diag32);
    for (auto &g : m->graphs)
        if (g.exec) cudaGraphExecDestroy(g.exec);
    if (m->cg_stream) cudaStreamDestroy(m->cg_stream);
    if (m->cg_ev[0]) cudaEventDestroy(m->cg_ev[0]);
    if (m->cg_ev[1]) cudaEventDestroy(m->cg_ev[1]);
    hb_pinned_put(m->state_host);
    if (m->ev0) cudaEventDestroy(m->ev0);
    if (m->ev1) cudaEventDestroy(m->ev1);
    delete m;
}

extern "C" hb_status hb_mesh_destroy(hb_mesh *m)
{
    if (!m) return HB_OK;
    hb_device_guard dg(m->device);
    // work on any stream may still read the arrays: wait for the device, as a
    // plain cudaFree would
    cudaDeviceSynchronize();
    mesh_free(m, nullptr);
    return HB_OK;
}

void hb_mesh_release(hb_mesh *m, cudaStream_t s)
{
    if (!m) return;
    hb_device_guard dg(m->device);
    mesh_free(m, s);
}

#define HB_TRY_MESH(call)                                                        \
    do {                                                                         \
        cudaError_t e_ = (call);                                                 \
        if (e_ != cudaSuccess) {                                                 \
            hb_set_error("%s:%d %s: %s", __FILE__, __LINE__, #call,              \
                         cudaGetErrorString(e_));                                \
            hb_mesh_destroy(m);                                                  \
            hb_dev_free(tmp_det, s);                                             \
            return e_ == cudaErrorMemoryAllocation ? HB_ERR_NOMEM : HB_ERR_CUDA; \
        }                                                                        \
    } while (0)

extern "C" hb_status hb_mesh_create(const hb_mesh_desc *d, void *stream, hb_mesh **out)
{
    hb_clear_error();
    if (!d || !out) { hb_set_error("null argument"); return HB_ERR_ARG; }
    *out = nullptr;
    if (d->N < 1 || d->N > HB_MAX_N) { hb_set_error("N=%d outside 1..%d", d->N, HB_MAX_N); return HB_ERR_ARG; }
    if (d->ex < 1 || d->ey < 1 || d->ez < 1) { hb_set_error("element counts must be >= 1"); return HB_ERR_ARG; }
    if (!(d->perturb >= 0.0 && d->perturb < 0.5)) { hb_set_error("perturb must be in [0, 0.5)"); return HB_ERR_ARG; }
    if (d->dirichlet_faces > 0x3Fu) { hb_set_error("dirichlet_faces has bits above 0x3F"); return HB_ERR_ARG; }
    const int N = d->N, n = N + 1;
    const int64_t E = (int64_t)d->ex * d->ey * d->ez;
    const int64_t n_local = E * n * n * n;
    if (n_local > 2147483647LL) { hb_set_error("n_local=%lld exceeds 2^31-1", (long long)n_local); return HB_ERR_ARG; }
    hb_status st = hb_ensure_device_tables();
    if (st != HB_OK) return st;

    cudaStream_t s = (cudaStream_t)stream;
    hb_mesh *m = new hb_mesh();
    memset((void *)m, 0, sizeof(hb_mesh));
    unsigned long long *tmp_det = nullptr;
    HB_TRY_MESH(cudaGetDevice(&m->device));
    m->desc = *d;
    m->variant[0] = HB_VAR_PENCIL | HB_VAR_EO;
    m->variant[1] = HB_VAR_PENCIL | HB_VAR_EO;
    m->variant[2] = HB_VAR_PENCIL | HB_VAR_EO;
    m->variant_ax[0] = m->variant_ax[1] = m->variant_ax[2] = -1;
    m->N = N;
    m->n = n;
    m->E = E;
    m->n_local = n_local;
    // counts by closed form
    const box_t b{d->ex, d->ey, d->ez, N, d->dirichlet_faces};
    const lattice3 L = box_lattice(b);
    const bool any = L.x.nu > 0 && L.y.nu > 0 && L.z.nu > 0;
    m->n_global = any ? (int64_t)L.x.nu * L.y.nu * L.z.nu : 0;
    m->nnz = any ? L.x.copies() * L.y.copies() * L.z.copies() : 0;
    const int64_t inner = any ? L.x.inner() * L.y.inner() * L.z.inner() : 0;  // one copy each
    m->nsr = m->n_global - inner;
    m->nnz_s = m->nnz - inner;
    const int64_t ng = m->n_global;

    size_t bytes = 0;
    auto alloc = [&](void **p, size_t b) {
        bytes += b;
        return hb_dev_alloc(p, b, s);
    };
    HB_TRY_MESH(alloc((void **)&m->l2g, sizeof(int32_t) * n_local));
    HB_TRY_MESH(alloc((void **)&m->geo, sizeof(double) * 7 * n_local));
    if (d->keep_fp32_copy) HB_TRY_MESH(alloc((void **)&m->geo32, sizeof(float) * 7 * n_local));
    HB_TRY_MESH(alloc((void **)&m->rowptr, sizeof(int32_t) * (ng + 1)));
    HB_TRY_MESH(alloc((void **)&m->mdiag, sizeof(double) * (ng + 1)));
    if (d->keep_fp32_copy) HB_TRY_MESH(alloc((void **)&m->mdiag32, sizeof(float) * (ng + 1)));
    HB_TRY_MESH(alloc((void **)&m->cols, sizeof(int32_t) * (m->nnz > 0 ? m->nnz : 1)));
    HB_TRY_MESH(alloc((void **)&m->srow_g, sizeof(int32_t) * (m->nsr + 1)));
    HB_TRY_MESH(alloc((void **)&m->srowptr, sizeof(int32_t) * (m->nsr + 1)));
    HB_TRY_MESH(alloc((void **)&m->scols, sizeof(int32_t) * (m->nnz_s > 0 ? m->nnz_s : 1)));
    // one partial per element-kernel block: at most two per element, or HB_SMS (a
    // small mesh split over more, cluster_blocks)
    m->n_ax_partials = 2 * E + HB_SMS;
    HB_TRY_MESH(alloc((void **)&m->ax_partials, sizeof(double) * m->n_ax_partials));
    HB_TRY_MESH(alloc((void **)&m->yL, sizeof(double) * n_local));
    HB_TRY_MESH(alloc((void **)&m->partials, sizeof(double) * HB_RED_MAXV * HB_RED_BLOCKS));
    HB_TRY_MESH(alloc((void **)&m->counters, sizeof(unsigned) * 8));
    HB_TRY_MESH(alloc((void **)&m->state, sizeof(hb_cg_state) * 4));
    HB_TRY_MESH(hb_pinned_get((void **)&m->state_host, sizeof(hb_cg_state)));
    HB_TRY_MESH(cudaEventCreate(&m->ev0));
    HB_TRY_MESH(cudaEventCreate(&m->ev1));
    HB_TRY_MESH(cudaMemsetAsync(m->counters, 0, sizeof(unsigned) * 8, s));
    HB_TRY_MESH(cudaMemsetAsync(m->state, 0, sizeof(hb_cg_state) * 4, s));

    // geometry: one element per block
    // at least 64 threads: 36 of them form the edge differences
    int gthreads = n * n * n < 256 ? std::max(64, ((n * n * n + 31) / 32) * 32) : 256;
    int gblocks = (int)(E < 152 * 64 ? E : 152 * 64);
    // 18.4 KB at N = 15: under the default limit, so no per-call attribute
    // (a per-degree value would race between threads building meshes)
    size_t gsmem = sizeof(double) * 9 * n * n;
    HB_TRY_MESH(hb_dev_alloc((void **)&tmp_det, sizeof *tmp_det, s));
    HB_TRY_MESH(cudaMemsetAsync(tmp_det, 0xFF, sizeof *tmp_det, s));
    hb_count_launch();
    k_geometry<<<gblocks, gthreads, gsmem, s>>>(b, L, d->perturb, d->seed, E, m->l2g, m->geo, m->geo32, tmp_det);
    HB_TRY_MESH(cudaGetLastError());
    if (ng > 0) {
        const int64_t warps = (int64_t)L.y.nu * L.z.nu * ((L.x.nu + kRowChunk - 1) / kRowChunk);
        hb_count_launch();
        k_rows<<<grid_for(warps * 32, 256), 256, 0, s>>>(L, m->geo, m->rowptr, m->cols, m->mdiag, m->mdiag32, m->srow_g,
                                                         m->srowptr, m->scols);
        HB_TRY_MESH(cudaGetLastError());
    } else {
        HB_TRY_MESH(cudaMemsetAsync(m->rowptr, 0, sizeof(int32_t), s));
        HB_TRY_MESH(cudaMemsetAsync(m->srowptr, 0, sizeof(int32_t), s));
    }
    // (into the pinned buffer: a copy to pageable memory would wait here)
    HB_TRY_MESH(cudaMemcpyAsync(m->state_host, tmp_det, sizeof *tmp_det, cudaMemcpyDeviceToHost, s));
    hb_dev_free(tmp_det, s);
    tmp_det = nullptr;
    // every stream-ordered array is ready for any stream once s has drained
    HB_TRY_MESH(cudaStreamSynchronize(s));
    {
        unsigned long long key;
        memcpy(&key, m->state_host, sizeof key);
        m->min_detJ = from_order_key(key);
    }
    m->device_bytes = bytes;
    if (!(m->min_detJ > 0.0)) {
        hb_set_error("non-positive Jacobian determinant (min det J = %g)", m->min_detJ);
        hb_mesh_destroy(m);
        return HB_ERR_GEOMETRY;
    }
    *out = m;
    return HB_OK;
}

extern "C" hb_status hb_mesh_info(const hb_mesh *m, hb_mesh_info_t *o)
{
    if (!m || !o) { hb_set_error("null argument"); return HB_ERR_ARG; }
    o->n_local = m->n_local;
    o->n_global = m->n_global;
    o->n_elem = m->E;
    o->nnz = m->nnz;
    o->N = m->N;
    o->l2g = m->l2g;
    o->geo = m->geo;
    o->geo32 = m->geo32;
    o->csr_rowptr = m->rowptr;
    o->csr_cols = m->cols;
    o->min_detJ = m->min_detJ;
    o->device_bytes = m->device_bytes;
    return HB_OK;
}

extern "C" hb_status hb_mesh_copy_l2g(const hb_mesh *m, int32_t *host)
{
    if (!m || !host) { hb_set_error("null argument"); return HB_ERR_ARG; }
    hb_device_guard dg(m->device);
    HB_TRY_CUDA(cudaMemcpy(host, m->l2g, sizeof(int32_t) * m->n_local, cudaMemcpyDeviceToHost));
    return HB_OK;
}

extern "C" hb_status hb_mesh_copy_geo(const hb_mesh *m, double *host)
{
    if (!m || !host) { hb_set_error("null argument"); return HB_ERR_ARG; }
    hb_device_guard dg(m->device);
    HB_TRY_CUDA(cudaMemcpy(host, m->geo, sizeof(double) * 7 * m->n_local, cudaMemcpyDeviceToHost));
    return HB_OK;
}

// ---------------------------------------------------------------- Jacobi preconditioner

// Diagonal of the element matrix Dbold^T G^e Dbold at every local node:
//   sum_m D[m][i]^2 G_rr(m,j,k) + sum_m D[m][j]^2 G_ss(i,m,k) + sum_m D[m][k]^2 G_tt(i,j,m)
//   + 2 D_ii D_jj G_rs + 2 D_ii D_kk G_rt + 2 D_jj D_kk G_st.
__global__ void k_elem_diag(const double *__restrict__ geo, const double *__restrict__ D, int N, int64_t n_local,
                            double *__restrict__ out)
{
    const int n = N + 1, n2 = n * n;
    const int64_t n3 = (int64_t)n2 * n;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n_local;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = q / n3;
        const int node = (int)(q - e * n3);
        const int i = node % n, j = (node / n) % n, k = node / n2;
        auto G = [&](int c, int ii, int jj, int kk) { return geo[((e * n + kk) * 7 + c) * (int64_t)n2 + jj * n + ii]; };
        double a = 0.0;
        for (int p = 0; p < n; p++) {
            a += D[p * n + i] * D[p * n + i] * G(0, p, j, k);
            a += D[p * n + j] * D[p * n + j] * G(3, i, p, k);
            a += D[p * n + k] * D[p * n + k] * G(5, i, j, p);
        }
        a += 2.0 * D[i * n + i] * D[j * n + j] * G(1, i, j, k);
        a += 2.0 * D[i * n + i] * D[k * n + k] * G(2, i, j, k);
        a += 2.0 * D[j * n + j] * D[k * n + k] * G(4, i, j, k);
        out[q] = a;
    }
}

// diag(A)_g = sum of the copies (CSR order = element order) + screening; stores 1/diag.
__global__ void k_diag_assemble(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ cols,
                                const double *__restrict__ dl, const double *__restrict__ mdiag, int screen,
                                double lambda, int64_t ng, double *__restrict__ inv64, float *__restrict__ inv32)
{
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < ng; g += (int64_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int p = rowptr[g]; p < rowptr[g + 1]; p++) s += dl[cols[p]];
        s += screen ? lambda * mdiag[g] : lambda;
        const double inv = 1.0 / s;
        inv64[g] = inv;
        inv32[g] = (float)inv;
    }
}

hb_status hb_mesh_inv_diag(hb_mesh *m, int screen, double lambda, cudaStream_t s)
{
    if (m->diag_valid && m->diag_screen == screen && m->diag_lambda == lambda) return HB_OK;
    const int64_t ng = m->n_global;
    if (!m->inv_diag) {
        HB_TRY_CUDA(cudaMalloc((void **)&m->inv_diag, sizeof(double) * (ng + 1)));
        HB_TRY_CUDA(cudaMalloc((void **)&m->inv_diag32, sizeof(float) * (ng + 1)));
        m->device_bytes += 12 * (size_t)(ng + 1);
    }
    hb_count_launch();
    k_elem_diag<<<grid_for(m->n_local, 256), 256, 0, s>>>(m->geo, hb_dev_D64(m->N), m->N, m->n_local,
                                                         (double *)m->yL);
    HB_CHECK_LAUNCH();
    hb_count_launch();
    k_diag_assemble<<<grid_for(ng, 256), 256, 0, s>>>(m->rowptr, m->cols, (const double *)m->yL, m->mdiag, screen,
                                                     lambda, ng, m->inv_diag, m->inv_diag32);
    HB_CHECK_LAUNCH();
    m->diag_valid = 1;
    m->diag_screen = screen;
    m->diag_lambda = lambda;
    return HB_OK;
}

extern "C" hb_status hb_diag_A(hb_mesh *m, hb_screen screen, double lambda, double *host_diag, void *stream)
{
    hb_clear_error();
    if (!m || (!host_diag && m->n_global)) { hb_set_error("null argument"); return HB_ERR_ARG; }
    if (screen != HB_SCREEN_IDENTITY && screen != HB_SCREEN_MASS) { hb_set_error("bad screen"); return HB_ERR_ARG; }
    hb_device_guard dg(m->device);
    cudaStream_t s = (cudaStream_t)stream;
    if (m->n_global == 0) return HB_OK;
    hb_status st = hb_mesh_inv_diag(m, screen, lambda, s);
    if (st != HB_OK) return st;
    std::vector<double> inv((size_t)m->n_global);
    HB_TRY_CUDA(cudaMemcpyAsync(inv.data(), m->inv_diag, sizeof(double) * m->n_global, cudaMemcpyDeviceToHost, s));
    HB_TRY_CUDA(cudaStreamSynchronize(s));
    for (int64_t g = 0; g < m->n_global; g++) host_diag[g] = 1.0 / inv[(size_t)g];
    return HB_OK;
}

// ---------------------------------------------------------------- right-hand sides

__global__ void k_rhs_uniform(const int32_t *l2g, box_t b, int64_t n_local, uint64_t seed, double *out)
{
    const int n = b.N + 1;
    const int64_t n3 = (int64_t)n * n * n;
    const int64_t NX = (int64_t)b.N * b.Ex + 1, NY = (int64_t)b.N * b.Ey + 1;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n_local;
         q += (int64_t)gridDim.x * blockDim.x) {
        int32_t g = l2g[q];
        if (g < 0) continue;
        int64_t e = q / n3;
        int node = (int)(q - e * n3);
        int i = node % n, j = (node / n) % n, k = node / (n * n);
        int64_t ex = e % b.Ex, ey = (e / b.Ex) % b.Ey, ez = e / ((int64_t)b.Ex * b.Ey);
        int64_t lat = (b.N * ex + i) + NX * ((b.N * ey + j) + NY * (b.N * ez + k));
        out[g] = 2.0 * hb_u01_impl(seed, 2, (uint64_t)lat) - 1.0;  // same value from every copy
    }
}

// Manufactured load: one thread per global DOF sums Jw f over its copies
// (CSR order), with the physical position recomputed from the element map.
__global__ void k_rhs_manufactured(const int32_t *rowptr, const int32_t *cols, int64_t ng, box_t b,
                                   double rho, uint64_t seed, const double *geo, double lambda, double *out)
{
    const int N = b.N, n = N + 1, n2 = n * n;
    const int64_t n3 = (int64_t)n2 * n;
    const double *xi = g_xi64 + N * 16;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < ng;
         g += (int64_t)gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int p = rowptr[g]; p < rowptr[g + 1]; p++) {
            int64_t lq = cols[p];
            int64_t e = lq / n3;
            int node = (int)(lq - e * n3);
            int i = node % n, j = (node / n) % n, k = node / n2;
            int ex = (int)(e % b.Ex), ey = (int)((e / b.Ex) % b.Ey), ez = (int)(e / ((int64_t)b.Ex * b.Ey));
            double r = xi[i], s = xi[j], t = xi[k];
            double fr[2] = {0.5 * (1 - r), 0.5 * (1 + r)};
            double fs[2] = {0.5 * (1 - s), 0.5 * (1 + s)};
            double ft[2] = {0.5 * (1 - t), 0.5 * (1 + t)};
            double X[3] = {0, 0, 0};
            for (int c = 0; c < 2; c++)
                for (int bb = 0; bb < 2; bb++)
                    for (int a = 0; a < 2; a++) {
                        double V[3];
                        vertex_pos(b, rho, seed, ex + a, ey + bb, ez + c, V);
                        double wgt = fr[a] * fs[bb] * ft[c];
                        for (int ax = 0; ax < 3; ax++) X[ax] += V[ax] * wgt;
                    }
            double f = (3.0 * M_PI * M_PI + lambda) * sin(M_PI * X[0]) * sin(M_PI * X[1]) * sin(M_PI * X[2]);
            acc += geo[((e * n + k) * 7 + 6) * (int64_t)n2 + j * n + i] * f;
        }
        out[g] = acc;
    }
}

extern "C" hb_status hb_fill_rhs(const hb_mesh *m, int kind, uint64_t seed, double lambda, double *bvec,
                                 void *stream)
{
    hb_clear_error();
    if (!m || !bvec) { hb_set_error("null argument"); return HB_ERR_ARG; }
    if (kind != 0 && kind != 1) { hb_set_error("kind must be 0 or 1"); return HB_ERR_ARG; }
    hb_device_guard dg(m->device);
    cudaStream_t s = (cudaStream_t)stream;
    box_t b{m->desc.ex, m->desc.ey, m->desc.ez, m->N, m->desc.dirichlet_faces};
    if (m->n_global == 0) return HB_OK;
    if (kind == 0) {
        hb_count_launch();
        k_rhs_uniform<<<grid_for(m->n_local, 256), 256, 0, s>>>(m->l2g, b, m->n_local, seed, bvec);
    } else {
        hb_count_launch();
        k_rhs_manufactured<<<grid_for(m->n_global, 128), 128, 0, s>>>(
            m->rowptr, m->cols, m->n_global, b, m->desc.perturb, m->desc.seed, m->geo, lambda, bvec);
    }
    HB_CHECK_LAUNCH();
    return HB_OK;
}
