// Tensor-core (tcgen05) pieces of the library: a self-check of the operand
// layouts the tensor-core element kernel relies on.
#include <cuda_fp16.h>

#include <cmath>
#include <cstring>

#include "hb_internal.h"
#include "hb_tc.cuh"
#include "hb_acc.cuh"

namespace {

constexpr unsigned long long kTcWaitNs = 1000000000ull;

__device__ __forceinline__ unsigned long long tc_wall_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait for phase `parity` of an mbarrier: about a second of wall
// time, then bit 0 of *err and return false.
__device__ __forceinline__ bool tc_wait(uint64_t *bar, unsigned parity, unsigned *err)
{
    const unsigned a = hbtc::smem_addr(bar);
    unsigned long long t0 = 0;
    for (unsigned t = 0;; t++) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if ((t & 255u) == 0) {
            const unsigned long long now = tc_wall_ns();
            if (t == 0) t0 = now;
            else if (now - t0 > kTcWaitNs) break;
        }
    }
    atomicOr(err, 1u);
    return false;
}

// Self-check tile: D (128 x 48, FP32) = A (128 x 48) B^T (B: 48 x 48), FP16
// inputs, three K steps of 16. A is staged K-major (mode bit 0 clear) or
// MN-major (set), with the MN core-matrix stride 128 bytes and the K one
// 2048; B is staged K-major (N stride 128, K stride 768). Mode bit 1 swaps
// the leading and stride byte-offset fields of both descriptors (to tell the
// two conventions apart; both stay inside the zeroed staging area).
constexpr int kSelfA = 0, kSelfB = 65536, kSelfBar = 81920, kSelfSmem = 81920 + 64;

__global__ void __launch_bounds__(128) tc_selftest_kernel(const float *__restrict__ A, const float *__restrict__ B,
                                                          float *__restrict__ D, int mode, unsigned *err)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + kSelfBar);
    unsigned *tptr = reinterpret_cast<unsigned *>(sm + kSelfBar + 8);
    const bool a_mn = (mode & 1) != 0, swap = (mode & 2) != 0;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    for (int i = tid; i < kSelfBar / 16; i += 128) reinterpret_cast<uint4 *>(sm)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    for (int idx = tid; idx < 128 * 48; idx += 128) {
        const int mn = idx / 48, k = idx % 48;
        const int off = a_mn ? (mn % 8) * 2 + (k % 8) * 16 + (mn / 8) * 128 + (k / 8) * 2048
                             : (mn % 8) * 16 + (k % 8) * 2 + (mn / 8) * 128 + (k / 8) * 2048;
        *reinterpret_cast<__half *>(sm + kSelfA + off) = __float2half_rn(A[idx]);
    }
    for (int idx = tid; idx < 48 * 48; idx += 128) {
        const int nn = idx / 48, k = idx % 48;
        const int off = (nn % 8) * 16 + (k % 8) * 2 + (nn / 8) * 128 + (k / 8) * 768;
        *reinterpret_cast<__half *>(sm + kSelfB + off) = __float2half_rn(B[idx]);
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(hbtc::smem_addr(bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    hbtc::fence_async_smem();
    __syncthreads();
    if (warp == 0) hbtc::tmem_alloc(tptr, 64);
    hbtc::fence_before_sync();
    __syncthreads();
    hbtc::fence_after_sync();
    const unsigned tmem = *tptr;
    if (tid == 0) {
        unsigned a_lbo = a_mn ? 128u : 2048u, a_sbo = a_mn ? 2048u : 128u;
        unsigned b_lbo = 768u, b_sbo = 128u;
        if (swap) {
            const unsigned t1 = a_lbo; a_lbo = a_sbo; a_sbo = t1;
            const unsigned t2 = b_lbo; b_lbo = b_sbo; b_sbo = t2;
        }
        const unsigned a0 = hbtc::smem_addr(sm + kSelfA), b0 = hbtc::smem_addr(sm + kSelfB);
        const uint32_t idesc = hbtc::idesc_f16(128, 48, a_mn, false);
        for (int ks = 0; ks < 3; ks++)
            hbtc::mma_f16(tmem, hbtc::smem_desc(a0 + ks * 2 * 2048, a_lbo, a_sbo),
                          hbtc::smem_desc(b0 + ks * 2 * 768, b_lbo, b_sbo), idesc, ks > 0);
        hbtc::mma_commit(bar);
    }
    tc_wait(bar, 0, err);
    hbtc::fence_after_sync();
    for (int c = 0; c < 48; c += 16) {
        uint32_t v[16];
        hbtc::tmem_ld16(tmem + ((unsigned)(32 * warp) << 16) + c, v);
        hbtc::tmem_wait_ld(v);
#pragma unroll
        for (int q = 0; q < 16; q++) D[(32 * warp + lane) * 48 + c + q] = __uint_as_float(v[q]);
    }
    hbtc::fence_before_sync();
    __syncthreads();
    if (warp == 0) hbtc::tmem_free(tmem, 64);
}

}  // namespace

extern "C" hb_status hb_tc_selftest(int mode, const float *A_host, const float *B_host, float *D_host,
                                    hb_status *status)
{
    hb_clear_error();
    if (!A_host || !B_host || !D_host || !status || mode < 0 || mode > 3) {
        hb_set_error("hb_tc_selftest: bad argument");
        return HB_ERR_ARG;
    }
    float *dA = nullptr, *dB = nullptr, *dD = nullptr;
    unsigned *derr = nullptr;
    cudaError_t e = cudaMalloc(&dA, sizeof(float) * 128 * 48);
    if (e == cudaSuccess) e = cudaMalloc(&dB, sizeof(float) * 48 * 48);
    if (e == cudaSuccess) e = cudaMalloc(&dD, sizeof(float) * 128 * 48);
    if (e == cudaSuccess) e = cudaMalloc(&derr, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemcpy(dA, A_host, sizeof(float) * 128 * 48, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dB, B_host, sizeof(float) * 48 * 48, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(derr, 0, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(dD, 0xFF, sizeof(float) * 128 * 48);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(tc_selftest_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelfSmem);
    if (e == cudaSuccess) {
        hb_count_launch();
        tc_selftest_kernel<<<1, 128, kSelfSmem>>>(dA, dB, dD, mode, derr);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    unsigned herr = 0;
    if (e == cudaSuccess) e = cudaMemcpy(D_host, dD, sizeof(float) * 128 * 48, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&herr, derr, sizeof(unsigned), cudaMemcpyDeviceToHost);
    cudaFree(dA);
    cudaFree(dB);
    cudaFree(dD);
    cudaFree(derr);
    if (e != cudaSuccess) {
        hb_set_error("hb_tc_selftest: %s", cudaGetErrorString(e));
        return HB_ERR_CUDA;
    }
    *status = herr ? HB_ERR_TIMEOUT : HB_OK;
    return HB_OK;
}

// ---------------------------------------------------------------- tensor-core FP64 element kernel
//
// y_L = S_L Z x (Sec. 2, Eq. stiffness) for N = 3, 7 and 15 with every derivative
// contraction (D along r, s, t and D^T along r, s, t; 12 n^4 of the
// 12 n^4 + 15 n^3 flops of an element) on the tensor cores, exactly, and the
// metric step (the 6 geometric factors, 15 n^3 flops) in FP64 on the CUDA
// cores.
//
// Exact contractions from FP16 products (an Ozaki-style split into slices):
//   - the values u are put on a fixed-point grid, X = round(u / 2^E) with 2^E two
//     bits below the last of the largest value (|X| < 2^55), and written as seven
//     base-256 digits, X = sum_j u_j 256^(6-j), u_0 a signed byte, u_1..u_6
//     unsigned ones. N = 3 and 15: a grid for every line, so a contraction is
//     accurate to its own line, as in floating point, whatever else the element
//     holds, and the directions are added as doubles. N = 7: a grid for the
//     element, on which the directions' sums are added exactly; a line far below
//     the element's largest value loses the bits between;
//   - D is scaled to integers D_int = round(D 2^s) (|D_int| < 2^55) and written
//     as balanced digits b_d in [-128, 128] (seven, and an eighth below the
//     binary point);
//   - digit products are integers below 2^16 and every sum the tensor core
//     forms stays below 2^24, so FP16 inputs with FP32 accumulation add them
//     without rounding. For each diagonal t = j + d <= 7 the MMA forms
//     S_t = sum_{j+d=t} sum_m b_d[i][m] u_j[m] in its own accumulator
//     column; D u = 2^(E-s) sum_t 256^(12-t) S_t up to the dropped diagonals
//     t >= 8, which weigh below 2^-60 of the largest term;
//   - a digit enters the MMA as the FP16 number 256 + u_j (384 + u_0), whose
//     bit pattern is 0x5C00 | (u_j << 2): no conversion instruction. The
//     offsets contribute a constant per accumulator column, replaced inside the
//     same MMA by 1.5 2^23 with an eighth K block: 128 in the A operand times
//     (1.5 2^23 - constant) / 128 (split into FP16-exact parts) in the B operand;
//   - so a column's bits are 0x4B400000 + S_t: the exact integers are combined in
//     two int64 halves and turned into doubles by integer instructions; at N = 7
//     the gradients stay in units of the element's grid (the scale rejoins at
//     the end, in the exponent).
// n = N + 1 is a power of two, so the lines of whole elements fill M-tiles of
// 128 rows. Per M-tile and direction: one MMA chain of n / 2 K = 16 steps, A =
// the lines' digits (128 x 8 n, K-major, K ordered (line position m, digit j)
// so that one node's seven digits and the offset-correction slot j = 7 are one
// 16-byte row piece), B = the digit stack of D (8 n x 8 n: output index i x
// diagonal t by the same K), accumulator 128 x 8 n FP32 in TMEM.
namespace {
namespace tcax {

// Shapes. A tile is MT M-tiles of 128 lines, whole elements; KH = nodes of its
// t-line (and outputs of its r-, s- and t-line rows) a thread owns.
//   N = 3:  16 elements, 256 lines, a thread per line
//   N = 7:  2 elements, 128 lines, two threads per line
//   N = 15: 1 element, 256 lines, four threads per line (1024 threads)
// Every shape puts 32 warps of 64 registers on an SM: four blocks, or the one
// block that N = 15's operands leave room for. Measured at 1.28e8 local nodes,
// ms per launch: N = 3 4.29 with three blocks, 4.13 with four; N = 7 4.52 with
// three blocks of 78 registers and its own t operand, 4.42 with four; N = 15
// 6.43 with 512 threads, 6.16 with 1024. With the accumulators biased, the
// gradients left unscaled and one 64-bit value per sum (fewer integer
// instructions, the busiest pipe beside FP64) 3.94, 4.25 and 5.86. A grid per line
// at N = 3 and 15 (two more fixed-point and two more double conversions a node,
// and the lines' maxima): 4.84 and 6.86, 4.57 and 6.72 with one range check a
// conversion and the element's NaN set at its end. (The FP64 pencil kernel: 8.68,
// 11.8 and 17.4.)
template <int N_>
struct shape {
    static constexpr int N = N_, n = N + 1, n2 = n * n, n3 = n2 * n;
    // The fixed-point grid follows every line, or the element. By element N = 3 and
    // 15 take 3.94 and 5.86 ms for 4.57 and 6.72, but one value of 1e8 among values
    // of 1 left lines that it is not on with 8 digits, where the FP64 pencil kernel
    // keeps 16.
    static constexpr bool LINE = n != 8;
    static_assert(n == 4 || n == 8 || n == 16, "the lines of whole elements fill M-tiles of 128 rows");
    static constexpr int NS = 2 * n2 + 4 * N * (N - 1);  // surface nodes of an element
    static constexpr int MT = n == 8 ? 1 : 2, EPT = MT * 128 / n2;
    static constexpr int KH = 4, TPL = n / KH, THREADS = MT * 128 * TPL;
    static constexpr int BLOCKS = n == 16 ? 1 : 4;  // resident per SM
    // x and node ids of the current and the next tile in registers; else only
    // the next tile's ids, and x and the ids read again (from L1 or L2)
    static constexpr bool HOLD = n == 4;
    // One direction's A operand and M-tile: n K chunks (m) of 128 rows x 8 FP16
    // (16 bytes); rows 16 bytes apart, row chunks of 8 at 128 bytes, K chunks
    // LBO apart: 2048 and what puts the eight threads of a store phase, which
    // differ in (ti, tj), on different banks.
    static constexpr int LBO_R = n == 4 ? 2080 : 2064, LBO_S = n == 4 ? 2112 : 2048, LBO_T = 2048;
    static constexpr int A_R = MT * n * LBO_R, A_S = MT * n * LBO_S, A_T = MT * n * LBO_T;
    // N = 7 and 15 stage t over r, whose MMAs are done by then: room for the
    // fourth block, or for the B images
    static constexpr bool RESTAGE = n != 4;
    static constexpr int OFF_R = 0, OFF_S = A_R, OFF_T = RESTAGE ? 0 : A_R + A_S;
    static constexpr int BIMG = n2 * 128;  // one B operand image (8 n x 8 n FP16)
    static constexpr int OFF_B = RESTAGE ? A_R + A_S : A_R + A_S + A_T;
    static constexpr int OFF_MISC = OFF_B + 2 * BIMG;
    // n = 16: the exponents of the 256 lines of each direction, of u and of v
    static constexpr int OFF_LX = OFF_MISC + 160, LX = n == 16 ? 3 * 256 : 0;
    static constexpr int SMEM = OFF_LX + 2 * LX * 4;
    // The exchange buffers (two doubles or two int64 halves per node of the
    // tile) sit in operands whose MMAs are done by then: r and s, or s alone
    static constexpr int EXS = n == 4 ? 80 : n3;  // node stride of an element
    static constexpr int OFF_EX = RESTAGE ? OFF_S : 0;
    static_assert(2 * EPT * EXS * 8 <= (RESTAGE ? A_S : A_R + A_S), "exchange buffers fit");
    static_assert(A_T <= A_R, "t fits over r");
    // r and s accumulate in DCOLS columns each, then t in r's
    static constexpr int DCOLS = MT * n * 8;
    static constexpr unsigned TMEM_COLS = 2 * DCOLS;

    // node (i, j, k) of element el in the exchange buffers: strides, or at n =
    // 8 and 16 exclusive ors, that keep a half warp's 8-byte accesses apart
    static __device__ __forceinline__ int xq(int el, int i, int j, int k)
    {
        if constexpr (n == 4) return el * EXS + k * 20 + j * 5 + i;
        else if constexpr (n == 8) return el * EXS + k * 64 + ((j * 8 + (i ^ j)) ^ ((k & 1) * 8));
        else return k * 256 + j * 16 + (i ^ j);
    }
};

// B operand images of D (0) and D^T (1) in the shared-memory layout (K-major,
// N chunk stride 128 bytes, K chunk stride 128 n) for n = 4, 8, 16, one after
// the other, and s (D_int = D 2^s) of each.
__host__ __device__ constexpr int img_off(int N) { return N == 3 ? 0 : N == 7 ? 2 * 32 * 32 : 2 * 32 * 32 + 2 * 64 * 64; }
__device__ __align__(16) uint16_t g_tc_bimg[2 * 32 * 32 + 2 * 64 * 64 + 2 * 128 * 128];
__constant__ int c_tc_dshift[3];
__host__ __device__ constexpr int tc_index(int N) { return N == 3 ? 0 : N == 7 ? 1 : N == 15 ? 2 : -1; }

struct tc_args {
    const double *x;
    const int32_t *l2g;
    const double *geo;
    double *ysurf;
    double *y;
    int64_t E;
    const int *run;
    double lambda;
    int screen;
    double *partials;
    unsigned *err;
    const int32_t *spos;  // SP kernels: CSR position of every surface copy (-1 masked)
};

// |v|'s high word: the largest of several carries the largest exponent (>> 20)
__device__ __forceinline__ unsigned abs_hi(double v) { return (unsigned)__double2hiint(v) & 0x7FFFFFFFu; }

// v on the grid of unit 2^(emax - 1077): round(|v| / unit) with the sign of v
// (|result| < 2^55; zero and subnormal v give 0). The two bits below a double's
// last keep the values within two binades of the largest exact and cut the
// rounding of the others to a quarter, at no cost: they fill the leading digit.
// Integer instructions only: 64-bit conversions run at the FP64 rate on this GPU.
constexpr int kUnit = 1077;
__device__ __forceinline__ long long to_fixed(double v, unsigned emax)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned e = (unsigned)(b >> 52) & 0x7FFu;
    // 8m with the implicit bit (m the 53-bit significand), shifted out whole
    // for zero and subnormals
    const long long m8 = (long long)(((b << 3) & 0x7FFFFFFFFFFFF8ull) | (1ull << 55));
    const long long s8 = (b >> 63) ? -m8 : m8;  // (the same for every grid the value enters)
    const unsigned sh = e ? min(emax - e, 62u) : 62u;
    // round(+-4m / 2^sh), halves up: (floor(+-8m / 2^sh) + 1) / 2
    return ((s8 >> sh) + 1) >> 1;
}

// The integer T as a double, rounded to nearest (ties away from zero):
// normalise |T| so its top bit is bit 63, keep 53 bits, round on the 11 below,
// and let a carry out of the mantissa step into the exponent. With OFF, T
// 2^off: results below the normal range flush to zero, above it give infinity.
template <bool OFF>
__device__ __forceinline__ double i64_to_double(long long T, int off)
{
    const unsigned long long sgn = (unsigned long long)T & 0x8000000000000000ull;
    unsigned long long M = T < 0 ? 0ull - (unsigned long long)T : (unsigned long long)T;
    const int lz = __clzll((long long)M);
    M <<= lz;
    const unsigned long long mant = (M >> 11) + ((M >> 10) & 1ull);  // 2^52 .. 2^53
    const int ex = 1023 + 63 - lz + (OFF ? off : 0);
    unsigned long long r = sgn | (((unsigned long long)(ex - 1) << 52) + mant);
    if (T == 0 || (OFF && (unsigned)(ex - 1) >= 2046u)) r = sgn | (T != 0 && ex > 0 ? 0x7FF0000000000000ull : 0ull);
    return __longlong_as_double((long long)r);
}

// floor((2^32 hi + lo) / 2^10) for |hi| < 2^41: what an int64 holds of the sum,
// rounded to nearest where combine has added the half. (Its unit is at most 2^-60
// of the largest product, 1/16 of what the rounding of the values to their grid
// leaves in the sum.)
__device__ __forceinline__ long long halves(long long hi, long long lo)
{
    hi += lo >> 32;
    return (long long)(((unsigned long long)hi << 22) | ((unsigned)lo >> 10));
}

// The A-operand row piece of one node: the FP16 bit patterns of the seven
// digits of X (digit j is byte 6 - j of the little-endian 64-bit word; byte 6
// is the signed leading digit u_0) as the MMA takes them -- digit u as the FP16
// number 256 + u (384 + u_0 for j = 0), pattern 0x5C00 | (u << 2) -- and the
// offset-correction slot, FP16 128.0 (0x5800).
__device__ __forceinline__ uint4 row_piece(long long X)
{
    const unsigned lo = (unsigned)X, hi = (unsigned)((unsigned long long)X >> 32);
    uint4 r;
    // __byte_perm(a, b, s): result byte n is byte (nibble n of s) of b:a; the
    // zero word supplies the empty bytes
    r.x = ((__byte_perm(hi, 0u, 0x4142u) ^ 0x00000080u) << 2) | 0x5C005C00u;           // u_0 + 128, u_1
    r.y = ((__byte_perm(lo, hi, 0x0304u) & 0x00FF00FFu) << 2) | 0x5C005C00u;           // u_2, u_3
    r.z = (__byte_perm(lo, 0u, 0x4142u) << 2) | 0x5C005C00u;                          // u_4, u_5
    r.w = ((lo & 0xFFu) << 2) | 0x58005C00u;                                          // u_6, 128.0
    return r;
}

// Stores the row pieces of the thread's nodes (ti, tj, k0 + q) of element el
// in the A operand of direction DIR:
//   r: line (el, k, j), K chunk m = i;  s: line (el, k, i), m = j;  t: line (el, j, i), m = k.
template <class C, int DIR>
__device__ __forceinline__ void stage(unsigned char *sm, int el, int ti, int tj, int k0, const long long (&X)[C::KH])
{
    constexpr int lbo = DIR == 0 ? C::LBO_R : DIR == 1 ? C::LBO_S : C::LBO_T;
    unsigned char *A = sm + (DIR == 0 ? C::OFF_R : DIR == 1 ? C::OFF_S : C::OFF_T);
#pragma unroll
    for (int q = 0; q < C::KH; q++) {
        const int k = k0 + q;
        const int line = el * C::n2 + (DIR == 0 ? k * C::n + tj : DIR == 1 ? k * C::n + ti : tj * C::n + ti);
        const int m = DIR == 0 ? ti : DIR == 1 ? tj : k;
        *reinterpret_cast<uint4 *>(A + (line >> 7) * C::n * lbo + m * lbo + (line & 127) * 16) = row_piece(X[q]);
    }
}

// The MMA chain of direction DIR into accumulator columns col: K step ks
// covers the K chunks m = 2 ks, 2 ks + 1 of A and B.
template <class C, int DIR>
__device__ __forceinline__ void issue(unsigned tmem, unsigned col, const unsigned char *sm, const unsigned char *Bi)
{
    constexpr uint32_t idesc = hbtc::idesc_f16(128, 8 * C::n, false, false);
    constexpr unsigned lbo = DIR == 0 ? C::LBO_R : DIR == 1 ? C::LBO_S : C::LBO_T;
    const unsigned b0 = hbtc::smem_addr(Bi);
    const unsigned a0 = hbtc::smem_addr(sm + (DIR == 0 ? C::OFF_R : DIR == 1 ? C::OFF_S : C::OFF_T));
#pragma unroll
    for (int mt = 0; mt < C::MT; mt++)
#pragma unroll
        for (int ks = 0; ks < C::n / 2; ks++)
            hbtc::mma_f16(tmem + col + mt * 8 * C::n, hbtc::smem_desc(a0 + mt * C::n * lbo + ks * 2 * lbo, lbo, 128),
                          hbtc::smem_desc(b0 + ks * 2 * 128 * C::n, 128 * C::n, 128), idesc, ks > 0);
}

// Completion of the chain in flight: warp 0 polls the barrier (bounded), the
// block meets at a barrier, which takes no issue slots.
__device__ __forceinline__ void mma_done(uint64_t *bar, unsigned &phase, int warp, unsigned *err, int &gave_up)
{
    if (warp == 0 && !tc_wait(bar, phase, err)) gave_up = 1;
    phase ^= 1u;
    __syncthreads();
    hbtc::fence_after_sync();
}

// The exact diagonal sums of output o of a 16-column chunk (diagonals 0..7)
// as the halves hi = sum_{t<4} S_t 256^(3-t), lo = sum_{t>=4} S_t 256^(7-t):
// the output is 2^72 hi + 2^40 lo in units of the element's grid times 2^-s.
// A column holds S_t + 1.5 2^23 (the bias comes with the offset correction), so
// S_t, an integer below 2^22 in magnitude, is its bits - 0x4B400000.
// HALF: with 2^9 added, so that halves() rounds to nearest.
template <bool HALF>
__device__ __forceinline__ void combine(const uint32_t (&v)[16], int o, long long &hi, long long &lo)
{
    const uint32_t *B = v + o * 8;
    // S_a 256 + S_b fits an int32: form it modulo 2^32 from the raw bits
    constexpr unsigned kBias = 0x4B400000u * 257u;
    const int m0 = (int)(B[0] * 256u + B[1] - kBias);
    const int m1 = (int)(B[2] * 256u + B[3] - kBias);
    const int m2 = (int)(B[4] * 256u + B[5] - kBias);
    const int m3 = (int)(B[6] * 256u + B[7] - kBias + (HALF ? 512u : 0u));
    hi = (long long)m0 * 65536 + m1;
    lo = (long long)m2 * 65536 + m3;
}

// Reads the thread's KH = 4 outputs of one direction out of tensor memory (its
// lane, columns from taddr) and hands each one's two halves to f(q, hi, lo).
template <class C, bool HALF, class F>
__device__ __forceinline__ void read_out(unsigned taddr, F &&f)
{
    static_assert(C::KH == 4, "two loads of 16 columns");
    uint32_t vv[2][16];
    hbtc::tmem_ld16(taddr, vv[0]);
    hbtc::tmem_ld16(taddr + 16, vv[1]);
    hbtc::tmem_wait_ld(vv[0]);
    hbtc::tmem_wait_ld(vv[1]);
#pragma unroll
    for (int c = 0; c < 2; c++)
#pragma unroll
        for (int o = 0; o < 2; o++) {
            long long hi, lo;
            combine<HALF>(vv[c], o, hi, lo);
            f(2 * c + o, hi, lo);
        }
}

// N = 7: largest v over the thread's element (warps 0, 1, 4, 5 hold element 0,
// warps 2, 3, 6, 7 element 1). Every thread calls it; it synchronises the block.
__device__ __forceinline__ unsigned element_max(unsigned v, unsigned *wexp, int el)
{
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) wexp[threadIdx.x >> 5] = v;
    __syncthreads();
    return max(max(wexp[2 * el], wexp[2 * el + 1]), max(wexp[4 + 2 * el], wexp[5 + 2 * el]));
}

// N = 3, 15: the exponents of a thread's four nodes, two 16-bit fields a word
struct exps {
    unsigned w[2];
    __device__ __forceinline__ explicit exps(const double (&v)[4])
    {
        w[0] = (abs_hi(v[0]) >> 20) | (abs_hi(v[1]) >> 20 << 16);
        w[1] = (abs_hi(v[2]) >> 20) | (abs_hi(v[3]) >> 20 << 16);
    }
    __device__ __forceinline__ unsigned at(int q) const { return ((q & 2 ? w[1] : w[0]) >> (q & 1 ? 16 : 0)) & 0xFFFFu; }
    __device__ __forceinline__ unsigned largest() const
    {
        const unsigned m = __vmaxu2(w[0], w[1]);
        return max(m & 0xFFFFu, m >> 16);
    }
    // field by field over the lanes that differ in the bits of the masks lo, 2 lo, ..., hi
    __device__ __forceinline__ void over_lanes(int lo, int hi)
    {
        for (int o = lo; o <= hi; o <<= 1)
            for (int c = 0; c < 2; c++) w[c] = __vmaxu2(w[c], __shfl_xor_sync(0xffffffffu, w[c], o));
    }
};

// The largest exponents along the lines: in er, es (in: of the thread's nodes, by
// what they enter along r and s; out: of their r- and s-lines) and et (out: of its
// t-line); row: of the three lines that are the thread's rows of the r, s and t
// operands; bad: whether any thread of the element passes true. n = 4: an element
// is 16 lanes, all by shuffles. n = 16: r-lines are 16 lanes; s-lines meet in the
// exponents lx in shared memory, as do the t-lines (both zero before the call),
// which synchronises the block.
template <class C>
__device__ __forceinline__ void line_max(exps &er, exps &es, const exps &t, unsigned &et, unsigned (&row)[3],
                                         bool &bad, unsigned *lx, int line, int ti, int tj, int k0)
{
    et = t.largest();
    if constexpr (C::n == 4) {
        er.over_lanes(1, 2);
        es.over_lanes(4, 8);
        // row (k, j) = (tj, ti) of r: held by the lanes of tj = ti; row (k, i) = (tj, ti) of s: here
        exps o = er;
        for (int c = 0; c < 2; c++) o.w[c] = __shfl_sync(0xffffffffu, er.w[c], (threadIdx.x & 16) | (ti * 4));
        row[0] = o.at(tj);
        row[1] = es.at(tj);
        bad = ((__ballot_sync(0xffffffffu, bad) >> (threadIdx.x & 16)) & 0xFFFFu) != 0;
    } else {
        er.over_lanes(1, 8);
        es.over_lanes(16, 16);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (ti == 0) lx[(k0 + q) * 16 + tj] = er.at(q);
            if ((threadIdx.x & 31) < 16) atomicMax(&lx[256 + (k0 + q) * 16 + ti], es.at(q));
        }
        atomicMax(&lx[512 + line], et);
        bad = __syncthreads_or(bad) != 0;
        unsigned v[4];
#pragma unroll
        for (int q = 0; q < 4; q++) v[q] = lx[256 + (k0 + q) * 16 + ti];
        es.w[0] = v[0] | v[1] << 16;
        es.w[1] = v[2] | v[3] << 16;
        row[0] = lx[line];
        row[1] = lx[256 + line];
        et = lx[512 + line];
    }
    row[2] = et;
}

// Thread tid: M-tile mt, TMEM lane tid % 128: line mt 128 + lane of the tile
// (element el; t-line (ti, tj)), and part h of it: nodes k = k0 .. k0 + KH - 1
// of its t-line, the same outputs of its r-, s- and t-line rows. Per tile and
// phase (D, then D^T): stage the operands, run the r and s chains, read r out
// (gradients to the exchange buffers, or the exact sums of D^T), start the t
// chain into r's columns, read s out meanwhile, then t. The six metric factors
// are prefetched into L2 at the tile's start and loaded at the metric step,
// not held in registers. What bounds it (ncu, N = 3 / 7 / 15): the integer pipe 61 /
// 53 / 41 %, the FP64 pipe 59 / 58 / 43 %, issue 52 / 50 / 36 % of the time; DRAM at
// most a quarter of its rate.
template <class C, bool SP>
__global__ void __launch_bounds__(C::THREADS, C::BLOCKS) ax_tc_kernel(const tc_args A)
{
    constexpr int N = C::N, n = C::n, n2 = C::n2, n3 = C::n3, NS = C::NS, KH = C::KH, EPT = C::EPT;
    constexpr bool kHold = C::HOLD;
    if (A.run && *A.run == 0) return;
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int mt = (tid >> 7) % C::MT, h = (tid >> 7) / C::MT, k0 = KH * h;
    const int line = mt * 128 + (tid & 127), el = line / n2, a = line % n2, ti = a % n, tj = a / n;
    unsigned char *Bi = sm + C::OFF_B;
    double *ExR = reinterpret_cast<double *>(sm + C::OFF_EX);
    double *ExS = ExR + EPT * C::EXS;
    long long *Yhi = reinterpret_cast<long long *>(ExR);
    long long *Ylo = reinterpret_cast<long long *>(ExS);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + C::OFF_MISC);
    unsigned *tptr = reinterpret_cast<unsigned *>(sm + C::OFF_MISC + 8);
    unsigned *wexp = reinterpret_cast<unsigned *>(sm + C::OFF_MISC + 16);
    unsigned *lxu = reinterpret_cast<unsigned *>(sm + C::OFF_LX), *lxv = lxu + C::LX;

    for (int q = tid; q < 2 * C::LX; q += C::THREADS) lxu[q] = 0;
    for (int q = tid; q < 2 * C::BIMG / 16; q += C::THREADS)
        reinterpret_cast<uint4 *>(Bi)[q] = reinterpret_cast<const uint4 *>(g_tc_bimg + img_off(N))[q];
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(hbtc::smem_addr(bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) hbtc::tmem_alloc(tptr, C::TMEM_COLS);
    hbtc::fence_async_smem();
    hbtc::fence_before_sync();
    __syncthreads();
    hbtc::fence_after_sync();
    const unsigned tmem = *tptr;
    const int dshift = c_tc_dshift[tc_index(N)];
    const unsigned tl = tmem + ((unsigned)((warp & 3) * 32) << 16) + (unsigned)(8 * (mt * n + k0));

    hbacc::dot_acc<double> acc;
    unsigned phase = 0;
    int gave_up = 0;
    const int64_t ntiles = (A.E + EPT - 1) / EPT;
    int gid_n[KH];
    double u_n[kHold ? KH : 1];
    auto gather = [&](int64_t gg) {
        const int64_t ee = EPT * gg + el;
        const bool act = gg < ntiles && ee < A.E;
        const int32_t *lg = A.l2g + ee * n3 + a;
#pragma unroll
        for (int q = 0; q < KH; q++) gid_n[q] = act ? (kHold ? __ldcs(lg + (k0 + q) * n2) : __ldg(lg + (k0 + q) * n2)) : -1;
        if constexpr (kHold) {
#pragma unroll
            for (int q = 0; q < KH; q++) u_n[q] = gid_n[q] >= 0 ? __ldg(A.x + gid_n[q]) : 0.0;
        }
    };
    gather(blockIdx.x);
    for (int64_t g = blockIdx.x; g < ntiles; g += gridDim.x) {
        const int64_t e = EPT * g + el;
        const bool active = e < A.E;
        int gid[kHold ? KH : 1];
        double u[KH];
#pragma unroll
        for (int q = 0; q < KH; q++) {
            if constexpr (kHold) {
                gid[q] = gid_n[q];
                u[q] = u_n[q];
            } else {
                u[q] = gid_n[q] >= 0 ? __ldg(A.x + gid_n[q]) : 0.0;
            }
        }
        {
            // the tile's six metric factors into L2 now (the first 6 n^2 values
            // of each element's k-slab of 7 n^2; J w only if screening reads
            // it), read at the metric step
            const int64_t e0 = EPT * g;
            const int nel = e0 + EPT <= A.E ? EPT : (int)(A.E - e0);
            constexpr int kLines = 6 * n2 * 8 / 128;
            for (int L = tid; L < nel * n * kLines; L += C::THREADS) {
                const int sl = L / kLines, ln = L - sl * kLines;  // slab sl of the tile
                const double *p = A.geo + e0 * 7 * n3 + (int64_t)sl * 7 * n2 + ln * 16;
                asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
            }
        }
        long long X[KH];
        unsigned eu = 0, row[3];
        bool ubad = false;
        if constexpr (C::LINE) {
            exps er(u), es(u);
            const exps et(u);
            ubad = et.largest() == 0x7FFu;
            line_max<C>(er, es, et, eu, row, ubad, lxu, line, ti, tj, k0);
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = to_fixed(u[q], er.at(q));
            stage<C, 0>(sm, el, ti, tj, k0, X);
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = to_fixed(u[q], es.at(q));
            stage<C, 1>(sm, el, ti, tj, k0, X);
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = to_fixed(u[q], eu);
            // (the s- and t-lines' words for v, read in the tile before)
            for (int q = 256 + tid; q < C::LX; q += C::THREADS) lxv[q] = 0;
        } else {
#pragma unroll
            for (int q = 0; q < KH; q++) eu = max(eu, abs_hi(u[q]));
            eu = element_max(eu, wexp, el) >> 20;
            ubad = eu == 0x7FFu;
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = ubad ? 0 : to_fixed(u[q], eu);
            stage<C, 0>(sm, el, ti, tj, k0, X);
            stage<C, 1>(sm, el, ti, tj, k0, X);
        }
        if constexpr (!C::RESTAGE) stage<C, 2>(sm, el, ti, tj, k0, X);
        hbtc::fence_async_smem();
        hbtc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
            hbtc::fence_after_sync();
            issue<C, 0>(tmem, 0, sm, Bi);
            issue<C, 1>(tmem, C::DCOLS, sm, Bi);
            hbtc::mma_commit(bar);
        }
        mma_done(bar, phase, warp, A.err, gave_up);
        // LINE: gradients by the exponent of their line. Else in units of 2^goff:
        // the element's scale meets only the exponents of the results.
        const int scale = 40 + 10 - kUnit - dshift;
        const int goff = C::LINE ? 0 : (int)eu + scale;
        auto value = [&](int dir, long long hi, long long lo) {
            if constexpr (C::LINE) return i64_to_double<true>(halves(hi, lo), (int)row[dir] + scale);
            return ubad ? __longlong_as_double(0x7FF8000000000000ll) : i64_to_double<false>(halves(hi, lo), 0);
        };
        if constexpr (C::RESTAGE) stage<C, 2>(sm, el, ti, tj, k0, X);
        // ---- gradient along r into its exchange buffer; its columns are free
        // for the t chain once every thread has read them
        read_out<C, true>(tl, [&](int q, long long hi, long long lo) { ExR[C::xq(el, k0 + q, ti, tj)] = value(0, hi, lo); });
        if constexpr (C::RESTAGE) hbtc::fence_async_smem();
        hbtc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
            hbtc::fence_after_sync();
            issue<C, 2>(tmem, 0, sm, Bi);
            hbtc::mma_commit(bar);
        }
        read_out<C, true>(tl + C::DCOLS,
                          [&](int q, long long hi, long long lo) { ExS[C::xq(el, ti, k0 + q, tj)] = value(1, hi, lo); });
        mma_done(bar, phase, warp, A.err, gave_up);
        double gt[KH];
        read_out<C, true>(tl, [&](int q, long long hi, long long lo) { gt[q] = value(2, hi, lo); });
        // ---- metric (FP64): v = G grad at the thread's nodes, factors loaded here
        double vr[KH], vs[KH], vt[KH];
        unsigned evm = 0;
        {
            const double *ge = A.geo + e * 7 * n3 + a;
#pragma unroll
            for (int q = 0; q < KH; q++) {
                double G[6];
#pragma unroll
                for (int c = 0; c < 6; c++) G[c] = active ? __ldcs(ge + (k0 + q) * 7 * n2 + c * n2) : 0.0;
                const int xi = C::xq(el, ti, tj, k0 + q);
                const double ur = ExR[xi], us = ExS[xi], ut = gt[q];
                vr[q] = fma(G[2], ut, fma(G[1], us, G[0] * ur));
                vs[q] = fma(G[4], ut, fma(G[3], us, G[1] * ur));
                vt[q] = fma(G[5], ut, fma(G[4], us, G[2] * ur));
                evm = max(evm, max(abs_hi(vr[q]), max(abs_hi(vs[q]), abs_hi(vt[q]))));
            }
        }
        // A non-finite value makes the whole element NaN. (The block meets here,
        // in every form: every exchange read is done before the operands are
        // staged over the exchange buffers.)
        unsigned ev;
        bool vbad = ubad || evm >> 20 == 0x7FFu;
        if constexpr (C::LINE) {
            exps er(vr), es(vs);
            if constexpr (n == 4) __syncthreads();
            line_max<C>(er, es, exps(vt), ev, row, vbad, lxv, line, ti, tj, k0);
            for (int q = 256 + tid; q < C::LX; q += C::THREADS) lxu[q] = 0;
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = to_fixed(vr[q], er.at(q));
            stage<C, 0>(sm, el, ti, tj, k0, X);
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = to_fixed(vs[q], es.at(q));
            stage<C, 1>(sm, el, ti, tj, k0, X);
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = to_fixed(vt[q], ev);
        } else {
            ev = element_max(evm, wexp, el) >> 20;
            vbad = ev == 0x7FFu;
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = vbad ? 0 : to_fixed(vr[q], ev);
            stage<C, 0>(sm, el, ti, tj, k0, X);
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = vbad ? 0 : to_fixed(vs[q], ev);
            stage<C, 1>(sm, el, ti, tj, k0, X);
#pragma unroll
            for (int q = 0; q < KH; q++) X[q] = vbad ? 0 : to_fixed(vt[q], ev);
        }
        if constexpr (!C::RESTAGE) stage<C, 2>(sm, el, ti, tj, k0, X);
        hbtc::fence_async_smem();
        hbtc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
            hbtc::fence_after_sync();
            issue<C, 0>(tmem, 0, sm, Bi + C::BIMG);
            issue<C, 1>(tmem, C::DCOLS, sm, Bi + C::BIMG);
            hbtc::mma_commit(bar);
        }
        gather(g + gridDim.x);
        mma_done(bar, phase, warp, A.err, gave_up);
        if constexpr (C::RESTAGE) stage<C, 2>(sm, el, ti, tj, k0, X);
        // ---- D^T along r and s summed in the exchange buffers: the directions
        // share a grid and are added exactly, or (LINE) as doubles
        read_out<C, C::LINE>(tl, [&](int q, long long hi, long long lo) {
            const int xi = C::xq(el, k0 + q, ti, tj);
            if constexpr (C::LINE) {
                ExR[xi] = value(0, hi, lo);
            } else {
                Yhi[xi] = hi;
                Ylo[xi] = lo;
            }
        });
        if constexpr (C::RESTAGE) hbtc::fence_async_smem();
        hbtc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
            hbtc::fence_after_sync();
            issue<C, 2>(tmem, 0, sm, Bi + C::BIMG);
            hbtc::mma_commit(bar);
        }
        read_out<C, C::LINE>(tl + C::DCOLS, [&](int q, long long hi, long long lo) {
            const int xi = C::xq(el, ti, k0 + q, tj);
            if constexpr (C::LINE) {
                ExR[xi] += value(1, hi, lo);
            } else {
                Yhi[xi] += hi;
                Ylo[xi] += lo;
            }
        });
        mma_done(bar, phase, warp, A.err, gave_up);
        {
            const int yoff = (int)ev + scale + goff;
            double *ys = A.ysurf + e * NS;
            const bool ring = ti == 0 || ti == N || tj == 0 || tj == N;
            const int r = tj == 0 ? ti : (tj == N ? n + ti : 2 * n + 2 * (tj - 1) + (ti == N ? 1 : 0));
            read_out<C, true>(tl, [&](int q, long long hi, long long lo) {
                const int k = k0 + q, xi = C::xq(el, ti, tj, k);
                double yc;
                if constexpr (C::LINE) {
                    yc = ExR[xi] + i64_to_double<true>(halves(hi, lo), yoff);
                } else {
                    hi += Yhi[xi];
                    lo += Ylo[xi];
                    yc = i64_to_double<true>(halves(hi, lo), yoff);
                }
                if (vbad) yc = __longlong_as_double(0x7FF8000000000000ll);
                if (!active) return;
                if (SP && (k == 0 || k == N || ring)) {
                    const int sidx = k == 0 ? a : (k == N ? n2 + a : 2 * n2 + (k - 1) * 4 * N + r);
                    const int pos = __ldg(A.spos + e * NS + sidx);
                    if (pos >= 0) A.ysurf[pos] = yc;
                } else if (k == 0) {
                    ys[a] = yc;
                } else if (k == N) {
                    ys[n2 + a] = yc;
                } else if (ring) {
                    ys[2 * n2 + (k - 1) * 4 * N + r] = yc;
                } else {
                    int gk;
                    double xv;
                    if constexpr (kHold) {
                        gk = gid[q];
                        xv = u[q];
                    } else {
                        gk = __ldg(A.l2g + e * n3 + k * n2 + a);
                        xv = __ldg(A.x + gk);
                    }
                    const double jw = A.screen ? __ldg(A.geo + (e * n + k) * 7 * n2 + 6 * n2 + a) : 1.0;
                    double yy = yc;
                    yy += A.lambda * (jw * xv);
                    A.y[gk] = yy;
                    acc.add(xv, yy);
                }
            });
        }
        // the next tile stages over the exchange buffers read above
        hbtc::fence_before_sync();
        if (__syncthreads_or(gave_up)) break;
    }
    if (A.partials) {
        const double v = hbacc::block_sum(acc.value());
        if (tid == 0) A.partials[blockIdx.x] = v;
    }
    if (__syncthreads_or(gave_up)) {
        if (tid == 0) tc_wait(bar, phase ^ 1u, A.err);
        __syncthreads();
    }
    hbtc::fence_before_sync();
    __syncthreads();
    hbtc::fence_after_sync();
    if (warp == 0) hbtc::tmem_free(tmem, C::TMEM_COLS);
}

// ---- host: B images and launch

// FP16 bit pattern of an integer that FP16 holds exactly.
static uint16_t fp16_exact(long long v)
{
    if (v == 0) return 0;
    const uint16_t sgn = v < 0 ? 0x8000 : 0;
    unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    int e = 63 - __builtin_clzll(a);
    const unsigned long long f = e >= 10 ? (a >> (e - 10)) : (a << (10 - e));
    return (uint16_t)(sgn | (uint16_t)((e + 15) << 10) | (uint16_t)(f & 0x3FF));
}

// Largest part of c (toward zero) that FP16 holds exactly: its top 11 bits.
static long long fp16_part(long long c)
{
    const unsigned long long a = (unsigned long long)(c < 0 ? -c : c);
    const int e = 63 - __builtin_clzll(a);
    const unsigned long long p = e > 10 ? (a >> (e - 10)) << (e - 10) : a;
    return c < 0 ? -(long long)p : (long long)p;
}

// Double-double host arithmetic (Dekker 1971, Knuth: two-sum, two-product with
// fma), about 106 bits, for the derivative matrix: its digits hold 63 bits,
// more than a double's 53.
struct dd {
    double h, l;
};
static dd dd_norm(double a, double b)
{
    const double s = a + b;
    return {s, b - (s - a)};
}
static dd operator+(dd a, dd b)
{
    const double s = a.h + b.h, v = s - a.h;
    return dd_norm(s, (a.h - (s - v)) + (b.h - v) + (a.l + b.l));
}
static dd operator-(dd a, dd b) { return a + dd{-b.h, -b.l}; }
static dd operator*(dd a, dd b)
{
    const double p = a.h * b.h;
    return dd_norm(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
static dd operator/(dd a, dd b)
{
    const double q = a.h / b.h;
    const dd r = a - b * dd{q, 0.0};
    const double q2 = r.h / b.h;
    return dd_norm(q, q2 + (r - b * dd{q2, 0.0}).h / b.h);
}

// D of degree N in double-double at the GLL nodes that xi approximates: two
// Newton steps on N (P_{N-1} - x P_N), derivative -N (N + 1) P_N; then
// D_ij = P_N(x_i) / (P_N(x_j) (x_i - x_j)), corners -+N (N + 1) / 4.
static void derivative_dd(int N, const double *xi, dd (&D)[16][16])
{
    const int n = N + 1;
    dd x[16], P[16];
    auto legendre = [N](dd z, dd &PN, dd &Pm) {
        dd a{1.0, 0.0}, b = z;
        for (int k = 2; k <= N; k++) {
            const dd c = (dd{2.0 * k - 1.0, 0.0} * z * b - dd{k - 1.0, 0.0} * a) / dd{(double)k, 0.0};
            a = b;
            b = c;
        }
        PN = b;
        Pm = a;
    };
    for (int i = 0; i < n; i++) {
        x[i] = {xi[i], 0.0};
        for (int it = 0; it < 2 && i > 0 && i < N; it++) {
            dd PN, Pm;
            legendre(x[i], PN, Pm);
            x[i] = x[i] + (Pm - x[i] * PN) / (dd{N + 1.0, 0.0} * PN);
        }
    }
    for (int i = 0; i < n; i++) {  // symmetric node set
        dd Pm;
        x[i] = (x[i] - x[N - i]) * dd{0.5, 0.0};
        x[N - i] = {-x[i].h, -x[i].l};
        legendre(x[i], P[i], Pm);
        legendre(x[N - i], P[N - i], Pm);
    }
    for (int i = 0; i < n; i++)
        for (int j = 0; j < n; j++) D[i][j] = i == j ? dd{0.0, 0.0} : P[i] / (P[j] * (x[i] - x[j]));
    D[0][0] = {-N * (N + 1) / 4.0, 0.0};
    D[N][N] = {N * (N + 1) / 4.0, 0.0};
}

}  // namespace tcax
}  // namespace

// Builds the B images of the degrees the kernel takes from their derivative
// matrices and uploads them to the current device (once per device, from
// hb_ensure_device_tables). D (in double-double: a double's rounding of D would
// be most of the kernel's error) is split into eight digits: D_int = D 2^s,
// with |D_int| < 2^55 and eight binary places (the eighth digit meets only the
// leading digit of the values, on the last diagonal). Largest sum of magnitudes
// an accumulator can meet (digits, offsets and the correction with the bias): 0.77,
// 0.81 and 0.87 of the 2^24 that FP32 holds exactly, for N = 3, 7, 15. The sums S_t
// stay below 2^20.8.
hb_status hb_tc_upload()
{
    using namespace tcax;
    static uint16_t img[sizeof(g_tc_bimg) / 2];
    int shift[3];
    std::memset(img, 0, sizeof img);
    for (int N : {3, 7, 15}) {
        const int n = N + 1;
        double xi[16], w[16], D64[256];
        dd D[16][16];
        hb_reference_element(N, xi, w, D64);
        derivative_dd(N, xi, D);
        double mx = 0.0;
        for (int q = 0; q < n * n; q++) mx = std::fmax(mx, std::fabs(D[q / n][q % n].h));
        const int s = 55 - (std::ilogb(mx) + 1);
        shift[tc_index(N)] = s;
        for (int tr = 0; tr < 2; tr++) {
            int b[8][16][16];  // digit d of D_int[i][m] (D^T for tr = 1), weight 256^(6-d)
            for (int i = 0; i < n; i++)
                for (int m = 0; m < n; m++) {
                    const dd v = tr ? D[m][i] : D[i][m];
                    // round(v 2^(s + 8)), |.| < 2^63
                    const double vh = std::ldexp(v.h, s + 8), vr = std::rint(vh);
                    __int128 q = (__int128)(long long)vr + std::llround((vh - vr) + std::ldexp(v.l, s + 8));
                    for (int d = 7; d >= 1; d--) {
                        const int r = (int)((q + 128) & 255) - 128;
                        b[d][i][m] = r;
                        q = (q - r) >> 8;
                    }
                    if (q < -128 || q > 128) {
                        hb_set_error("tensor-core split: leading digit %d out of range", (int)q);
                        return HB_ERR_ARG;
                    }
                    b[0][i][m] = (int)q;
                }
            uint16_t *im = img + img_off(N) + tr * 64 * n * n;
            // element (row (i, t), K (m, digit j)) at i * 128 + t * 16 + m * 128 n + j * 2
            auto put = [&](int i, int t, int j, int m, long long val) {
                im[(i * 128 + t * 16 + m * 128 * n + j * 2) / 2] = fp16_exact(val);
            };
            for (int i = 0; i < n; i++)
                for (int t = 0; t < 8; t++) {
                    long long beta = 0;  // what the digit offsets add to column (i, t)
                    for (int j = 0; j < 7; j++) {
                        const int d = t - j;
                        if (d < 0 || d > 7) continue;
                        long long rs = 0;
                        for (int m = 0; m < n; m++) {
                            put(i, t, j, m, b[d][i][m]);
                            rs += b[d][i][m];
                        }
                        beta += (j == 0 ? 384 : 256) * rs;
                    }
                    // slot j = 7 of each K chunk: 128 (A side) times parts summing to
                    // (1.5 2^23 - beta) / 128
                    long long c = (3 * (1 << 22) - beta) / 128;
                    for (int m = 0; m < n && c != 0; m++) {
                        const long long p = c > 49152 ? 49152 : fp16_part(c);
                        put(i, t, 7, m, p);
                        c -= p;
                    }
                    if (c != 0) {
                        hb_set_error("tensor-core split: offset correction does not fit");
                        return HB_ERR_ARG;
                    }
                }
        }
    }
    HB_TRY_CUDA(cudaMemcpyToSymbol(g_tc_bimg, img, sizeof img));
    HB_TRY_CUDA(cudaMemcpyToSymbol(c_tc_dshift, shift, sizeof shift));
    return HB_OK;
}

namespace {
namespace tcax {

template <int N>
hb_status launch(const tc_args &A, cudaStream_t s, int64_t *nblocks)
{
    using C = shape<N>;
    int dev = 0;
    HB_TRY_CUDA(cudaGetDevice(&dev));
    static int attr_set[64] = {0}, sms[64] = {0};
    if (dev < 0 || dev >= 64) { hb_set_error("device index %d unsupported", dev); return HB_ERR_ARG; }
    if (!attr_set[dev]) {
        HB_TRY_CUDA(cudaFuncSetAttribute(ax_tc_kernel<C, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
        HB_TRY_CUDA(cudaFuncSetAttribute(ax_tc_kernel<C, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
        HB_TRY_CUDA(cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev));
        attr_set[dev] = 1;
    }
    const int64_t ntiles = (A.E + C::EPT - 1) / C::EPT, room = (int64_t)C::BLOCKS * sms[dev];
    const int64_t grid = ntiles < room ? ntiles : room;
    if (nblocks) *nblocks = grid;
    hb_prof_scope prof("ax_local", s);
    if (A.spos) ax_tc_kernel<C, true><<<(unsigned)grid, C::THREADS, C::SMEM, s>>>(A);
    else ax_tc_kernel<C, false><<<(unsigned)grid, C::THREADS, C::SMEM, s>>>(A);
    HB_CHECK_LAUNCH();
    return HB_OK;
}

}  // namespace tcax
}  // namespace

// Tensor-core FP64 element kernel (N = 3, 7, 15): interior DOFs finished here
// (y, lambda term, partial of x.y per block), surface values to ysurf for the
// surface gather. Persistent grid: the blocks that fit on every SM at most.
hb_status hb_launch_ax_tc_f64(const hb_mesh *m, const double *x, double *ysurf, double *y, double lambda,
                              int screen, double *partials, const int *run, bool csr_store, cudaStream_t s,
                              int64_t *nblocks)
{
    using namespace tcax;
    if (!m->geo) { hb_set_error("mesh has no double geometric factors"); return HB_ERR_ARG; }
    if (csr_store && !m->spos) { hb_set_error("surface positions missing"); return HB_ERR_ARG; }
    if (m->E <= 0) return HB_OK;
    const tc_args A{x, m->l2g, m->geo, ysurf, y, m->E, run, lambda, screen, partials, m->counters + 7,
                    csr_store ? m->spos : nullptr};
    switch (m->N) {
    case 3: return launch<3>(A, s, nblocks);
    case 7: return launch<7>(A, s, nblocks);
    case 15: return launch<15>(A, s, nblocks);
    default: hb_set_error("the tensor-core element kernel is built for N = 3, 7 and 15"); return HB_ERR_ARG;
    }
}
