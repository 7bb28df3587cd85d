// Inverse of a Hermitian positive definite complex128 matrix A (eps of Sec. 5.1) by the Newton
// iteration X <- (2I - X A) X on the 16-bit tensor cores, to FP64 accuracy.
//
//  * Start.  X0 = 2 / (1 + u) D^-1, D = diag(A), rs_i = 1 / sqrt(a_ii), u = max_i rs_i sum_j |a_ij| rs_j >=
//    lambda_max(D^-1/2 A D^-1/2).  X0 A is similar to 2 / (1 + u) D^-1/2 A D^-1/2, whose eigenvalues lie
//    in (0, 2), so the error E = I - X A squares each step.  A diagonal entry that is not positive and
//    finite falls back to X0 = 2 / (1 + u) I with the plain row-sum bound.  X0 is diagonal, so the first
//    step, X1 = 2 X0 - X0 A X0, is taken element by element where X1's operand planes are made.
//  * Phase 1.  Newton steps with FP16X3 products (22 significant bits) until max |I - X A| < 2e-4.  A
//    step is two launches: Y = 2I - X A, then X' = Y X.  Each product's epilogue writes the FP16 hi / lo
//    operand planes that the next one reads; no FP64 matrix, slicing pass or slot tile lies between.
//    The planes' power-of-two scales are bounds known before the product: X' <= 2 X in the Loewner order
//    (its eigenvalues grow at most twofold), so max|X'| <= 2 max|X|, and |Y_ij| <= 1 + sqrt(d_max / d_min).
//    FP16 is a floating format, so a bound that is loose by 2^s costs nothing until s is about 10.  The
//    step whose Y met the tolerance is completed (its first product is there): X is then at the floor of
//    the split, which saves a refinement.
//  * Every product has the form C_ij = sum_k P_ik conj(Q_jk) with both operands as rows, k along the row:
//    the planes of A are those of A^H, and X is kept as its rows and as the rows of X^H.  (Computing only
//    one triangle of the Hermitian X and mirroring it would halve a product, but it turns rounding errors of
//    the form delta X, which the next residual sees as delta X A = delta, into X delta^H, which it sees
//    magnified by the condition number: simulated floor 1e-3 against 2e-5 at condition number 2e3.)
//  * Phase 2.  Up to three refinements X <- X + R X with R = I - X A to FP64 accuracy from integer slices
//    (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012): x = sum_t
//    a_t 2^(e - 7 (t + 1)), a_t integers of 7 bits and a sign, exact in FP16; the tensor cores add
//    products of slices exactly as long as a window's sum stays below 2^24.
//      - X is first rounded to 28 bits of its largest entry (it is known to about 22), four slices; A has
//        eight (55 bits).  R takes the 26 slice products t + u <= 7.
//      - A correction dX = R X is rounded to 41 bits of itself (six slices) and added to X in FP64; the
//        next residual is R - dX A, 21 products of a small matrix, where a fresh I - X A with both factors
//        to 54 bits takes 45.
//    FP16X3 is enough for R X because R is small.  A refinement whose residual is <= 1e-9 is the last; a
//    last residual above 1e-8 (or a non-finite one) is GW_E_NUMERIC.
//
// Measured on one GB300 (graph replay, warm), against slot tiles combined and sliced by separate FP64 passes and
// fresh 54-bit residuals: N_g = 691, 980 -> 417 us; 389, 660 -> 289 us; gw_zinv_tc at 1357, 3.62 -> 2.22 ms.
// What bounds it: at N_g = 691 the chain of ~20 dependent launches, each a few microseconds of loads,
// MMAs and a cluster-wide sum; from N_g of about 1400 on the tensor pipe in the residual products.
//
// Operand planes: element (r, k) of plane p sits at 16-bit offset ((kc nb + r/128) NP + p) 2048 +
// ((r%128)/8) 128 + ((k%16)/8) 64 + (r%8) 8 + k%8, kc = k/16, nb = ceil(N/128): the NP planes of one chunk
// of a 128-row block are contiguous.  FP16X3: Im hi, Re hi, Im lo, Re lo.  Slices: Im, Re of slice 0,
// Im, Re of slice 1, ...  From an Im plane of Q the 256 rows are [Im; Re], so with A = Im(P) one N = 256 MMA
// adds Pi Qi into the Re columns of the accumulator and Pi Qr into the Im columns; N = 128 MMAs with
// A = Re(P) add Pr Qr into Re and, by the A-negate bit, -Pr Qi into Im.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "gw_internal.cuh"
#include "ptx.cuh"

namespace gw {

namespace {

constexpr uint32_t PL = 4096;  // bytes of one plane of one block and chunk
constexpr uint32_t LBO = 128, SBO = 256;
constexpr int SCALE_BITS = 15;  // FP16X3 planes hold x 2^(15 - e), |x| < 2^e: below 2^15
constexpr uint64_t DRAIN_NS = 2000000000ull;
constexpr double NS_TOL = 2e-4;     // phase 1 ends with the step from an X with max |I - X A| below this
constexpr double NS_LAST = 1e-9;    // a refinement whose residual is below this is the last one
constexpr double NS_ACCEPT = 1e-8;  // largest residual before the last correction
constexpr int NS_MAX = 16, NS_REFINE = 3;
constexpr int BITS = 7, SL_A = 8, SL_X = 4, SL_D = 6;
constexpr int SL_XD = SL_D;  // slots of the slice planes shared by X and dX

// Scalars of one inverse, zeroed at its start.  Maxima are bits of non-negative floats (they order
// like the values); a maximum taken in FP32 still bounds the FP64 entries through exp_of's margin.
struct Words {
    unsigned a_max, d_max, rs2_max, d_bad, u, uj;
    unsigned dev[NS_MAX + 2];  // [it]: max |I - X_it A|
    unsigned mx[NS_MAX + 2];   // [it]: max |X_it|
    int ex[NS_MAX + 2];        // [it]: exponent of X_it's planes
    int ey, er;                // exponents of Y's, of R's planes
    int done;                  // it + 2 once max |I - X_it A| met the tolerance (X_(it+1) ends phase 1), 0 before
    unsigned mr[NS_REFINE], md[NS_REFINE];  // max |R_j|, max |dX_j|
};

__device__ __forceinline__ float bits_f(unsigned b) { return __uint_as_float(b); }

// e with m < 2^e (0 for a zero or non-finite m; a non-finite residual is caught by the final check)
__device__ __forceinline__ int exp_of(float m)
{
    if (!(m > 0.f) || !isfinite(m))
        return 0;
    int e;
    frexpf(m * (1.0f + 0x1p-20f), &e);
    return e;
}

__device__ __forceinline__ int current_it(const Words *w, int max_steps)
{
    return w->done ? w->done - 1 : max_steps + 1;
}

// Refinement j runs unless an earlier one was the last.
__device__ __forceinline__ bool refine_over(const Words *w, int j)
{
    for (int i = 0; i < j; ++i)
        if (bits_f(w->mr[i]) <= (float)NS_LAST)
            return true;
    return false;
}

__device__ __forceinline__ float finite_or_inf(float d)
{
    return d <= 3.0e38f ? d : __int_as_float(0x7f800000);  // NaN or inf: +inf, which a maximum keeps
}

// Maximum over the block into *w; call with every thread of the block.
__device__ __forceinline__ void block_max(float v, unsigned *w)
{
    __shared__ float red[32];
    v = finite_or_inf(v);
    for (int o = 16; o > 0; o >>= 1)
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i)
            v = fmaxf(v, red[i]);
        atomicMax(w, __float_as_uint(v));
    }
}

// Eight consecutive values as the hi and lo halves of FP16X3 planes.
__device__ __forceinline__ void split8(const float *x, uint4 &hi, uint4 &lo)
{
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2 a = __floats2half2_rn(x[2 * i], x[2 * i + 1]);
        const float2 f = __half22float2(a);
        const __half2 b = __floats2half2_rn(x[2 * i] - f.x, x[2 * i + 1] - f.y);
        h[i] = *reinterpret_cast<const uint32_t *>(&a);
        l[i] = *reinterpret_cast<const uint32_t *>(&b);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// 16-bit offset of (r, k) in a block-chunk of np planes, plane 0
__device__ __forceinline__ size_t plane_at(int kc, int nb, int blk, int np)
{
    return ((size_t)kc * nb + blk) * np * 2048;
}

// FP16X3 planes of eight consecutive k (an octet ko of chunk kc) of row r, scaled values split into hi, lo
__device__ __forceinline__ void store_octet(uint16_t *F, int nb, int kc, int blk, int r, int ko, const float *re,
                                            const float *im)
{
    uint4 h, l;
    uint16_t *p = F + plane_at(kc, nb, blk, 4) + (r >> 3) * 128 + ko * 64 + (r & 7) * 8;
    split8(im, h, l);
    *reinterpret_cast<uint4 *>(p) = h;
    *reinterpret_cast<uint4 *>(p + 2 * 2048) = l;
    split8(re, h, l);
    *reinterpret_cast<uint4 *>(p + 2048) = h;
    *reinterpret_cast<uint4 *>(p + 3 * 2048) = l;
}

// rint(|x| 2^s), with the sign of x, for |x| 2^s < 2^62, on the bits of the double (FP64 arithmetic runs
// at 1/64 of the integer rate here); ties away from zero.
__device__ __forceinline__ long long scaled_int(double x, int s)
{
    const long long b = __double_as_longlong(x);
    const int be = (int)((b >> 52) & 0x7ff);
    if (be == 0)
        return 0;  // zero or denormal
    const long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
    const int sh = be - 1075 + s;
    long long n;
    if (sh >= 0)
        n = sh < 10 ? m << sh : 0;  // 2^53 2^sh; larger only for a non-finite x, whose residual is caught
    else
        n = sh < -54 ? 0 : (m + (1ll << (-sh - 1))) >> -sh;
    return b < 0 ? -n : n;
}

// Balanced base-128 digits of n, most significant first: n = sum_t a_t 128^(ns - 1 - t), |a_t| <= 64 for
// t > 0.  Stores the octets of ns slices (planes 2t: Im, 2t + 1: Re) of row r.
template <int NS>
__device__ __forceinline__ void store_slices(uint16_t *F, int np, int nb, int kc, int blk, int r, int ko,
                                             const long long *nr, const long long *ni)
{
    uint16_t *p = F + plane_at(kc, nb, blk, np) + (r >> 3) * 128 + ko * 64 + (r & 7) * 8;
    long long cr[8], ci[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        cr[i] = nr[i];
        ci[i] = ni[i];
    }
#pragma unroll
    for (int t = NS - 1; t >= 0; --t) {
        uint32_t wr[4], wi[4];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            int a[2], b[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                a[j] = t > 0 ? ((int)(cr[i + j] + 64) & 127) - 64 : (int)cr[i + j];
                b[j] = t > 0 ? ((int)(ci[i + j] + 64) & 127) - 64 : (int)ci[i + j];
                cr[i + j] = (cr[i + j] - a[j]) >> BITS;  // exact
                ci[i + j] = (ci[i + j] - b[j]) >> BITS;
            }
            const __half2 x = __floats2half2_rn((float)a[0], (float)a[1]);  // |a| <= 128: exact
            const __half2 y = __floats2half2_rn((float)b[0], (float)b[1]);
            wr[i / 2] = *reinterpret_cast<const uint32_t *>(&x);
            wi[i / 2] = *reinterpret_cast<const uint32_t *>(&y);
        }
        *reinterpret_cast<uint4 *>(p + (size_t)(2 * t) * 2048) = make_uint4(wi[0], wi[1], wi[2], wi[3]);
        *reinterpret_cast<uint4 *>(p + (size_t)(2 * t + 1) * 2048) = make_uint4(wr[0], wr[1], wr[2], wr[3]);
    }
}

// ------------------------------------------------------------------------------- start

// max(|Re|, |Im|) of A, rs_i = 1 / sqrt(Re a_ii) and the extremes of the diagonal.
__global__ void __launch_bounds__(256) ns_max_kernel(const double2 *__restrict__ A, int N, float *__restrict__ rs,
                                                     Words *w)
{
    float best = 0.f;
    const size_t n = (size_t)N * N;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double2 z = A[i];
        best = fmaxf(best, fmaxf(fabsf((float)z.x), fabsf((float)z.y)));
        if (!(z.x == z.x) || !(z.y == z.y))
            best = __int_as_float(0x7f800000);
    }
    block_max(best, &w->a_max);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const double d = A[(size_t)i * N + i].x;
        const float r = (d > 0.0 && d < 1e30) ? rsqrtf((float)d) : 0.f;
        rs[i] = r;
        if (r > 0.f && isfinite(r)) {
            atomicMax(&w->d_max, __float_as_uint((float)d));
            atomicMax(&w->rs2_max, __float_as_uint(r * r));
        } else {
            rs[i] = 0.f;
            atomicOr(&w->d_bad, 1u);
        }
    }
}

constexpr float SUM_MARGIN = 1.001f;  // the row sums are FP32: the bound stays above the exact sum

// Blocks below nslice: FP16X3 planes and slices of A^H (element (r, k) = conj(A[k][r])) of one 128-row
// block and chunk.  The others: the row-sum bounds, a warp per row.
__global__ void __launch_bounds__(256) ns_prep_kernel(const double2 *__restrict__ A, int N, int nb, int nkc,
                                                      const float *__restrict__ rs, uint16_t *__restrict__ A16,
                                                      uint16_t *__restrict__ ASL, Words *w)
{
    __shared__ double2 tile[16][129];
    const int nslice = nb * nkc;
    if ((int)blockIdx.x >= nslice) {
        const int lane = threadIdx.x & 31;
        const int wid = (blockIdx.x - nslice) * 8 + (threadIdx.x >> 5), nw = (gridDim.x - nslice) * 8;
        float bu = 0.f, bj = 0.f;
        for (int i = wid; i < N; i += nw) {
            float s = 0.f, sj = 0.f;
            for (int j = lane; j < N; j += 32) {
                const double2 a = A[(size_t)i * N + j];
                const float m = fabsf((float)a.x) + fabsf((float)a.y);
                s += m;
                sj = fmaf(m, rs[j], sj);
            }
            for (int o = 16; o > 0; o >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, o);
                sj += __shfl_xor_sync(0xffffffffu, sj, o);
            }
            bu = fmaxf(bu, s);
            bj = fmaxf(bj, sj * rs[i]);
        }
        block_max(bu * SUM_MARGIN, &w->u);
        block_max(bj * SUM_MARGIN, &w->uj);
        return;
    }
    const int kc = blockIdx.x / nb, blk = blockIdx.x - kc * nb;
    for (int q = threadIdx.x; q < 2048; q += 256) {
        const int kk = q >> 7, rr = q & 127, r = blk * 128 + rr, k = kc * 16 + kk;
        double2 z = make_double2(0.0, 0.0);
        if (r < N && k < N)
            z = A[(size_t)k * N + r];
        tile[kk][rr] = make_double2(z.x, -z.y);
    }
    __syncthreads();
    const int e = exp_of(bits_f(w->a_max));
    const float sc = ldexpf(1.0f, SCALE_BITS - e);
    const int s = BITS * SL_A - 1 - e;  // |n| < 2^55: the first digit stays within 64 too
    const int rr = (threadIdx.x >> 4) * 8 + (threadIdx.x & 7), ko = (threadIdx.x >> 3) & 1;
    float re[8], im[8];
    long long nr[8], ni[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const double2 z = tile[ko * 8 + i][rr];
        re[i] = (float)z.x * sc;
        im[i] = (float)z.y * sc;
        nr[i] = scaled_int(z.x, s);
        ni[i] = scaled_int(z.y, s);
    }
    store_octet(A16, nb, kc, blk, rr, ko, re, im);
    store_slices<SL_A>(ASL, 2 * SL_A, nb, kc, blk, rr, ko, nr, ni);
}

// Planes of X1 = 2 X0 - X0 A X0 (header comment), its rows and the rows of X1^H, and the exponents of the
// first step.
__global__ void __launch_bounds__(256) ns_init_kernel(const double2 *__restrict__ A, int N, int nb, int nkc,
                                                      const float *__restrict__ rs, uint16_t *__restrict__ X16,
                                                      Words *w)
{
    __shared__ float2 tile[16][129];
    const int kc = blockIdx.x, blk = blockIdx.y;
    const bool jac = w->d_bad == 0;
    const float c = 2.0f / (1.0f + bits_f(jac ? w->uj : w->u));
    const float x0 = jac ? c * bits_f(w->rs2_max) : c;  // max X0
    const int e = exp_of(2.0f * x0);
    if (kc == 0 && blk == 0 && threadIdx.x == 0) {
        w->ex[1] = e;
        const float spread = jac ? sqrtf(bits_f(w->d_max) * bits_f(w->rs2_max)) : 1.f;
        w->ey = exp_of(1.0f + spread * 1.001f);
    }
    // A[k][r] for the rows of X1^H
    for (int q = threadIdx.x; q < 2048; q += 256) {
        const int kk = q >> 7, rr = q & 127, r = blk * 128 + rr, k = kc * 16 + kk;
        double2 z = make_double2(0.0, 0.0);
        if (r < N && k < N)
            z = A[(size_t)k * N + r];
        tile[kk][rr] = make_float2((float)z.x, -(float)z.y);
    }
    __syncthreads();
    const float sc = ldexpf(1.0f, SCALE_BITS - e);
    const int rr = (threadIdx.x >> 4) * 8 + (threadIdx.x & 7), ko = (threadIdx.x >> 3) & 1;
    const int r = blk * 128 + rr;
    const float xr = r < N ? (jac ? c * rs[r] * rs[r] : c) : 0.f;
    float best = 0.f;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        float re[8], im[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = kc * 16 + ko * 8 + i;
            re[i] = im[i] = 0.f;
            if (r < N && k < N) {
                float2 a = tile[ko * 8 + i][rr];
                if (side == 0) {
                    const double2 z = A[(size_t)r * N + k];
                    a = make_float2((float)z.x, (float)z.y);
                }
                // (X0 a) X0: the product of two entries of X0 can overflow
                const float xk = jac ? c * rs[k] * rs[k] : c;
                re[i] = (r == k ? 2.f * xr : 0.f) - xr * a.x * xk;
                im[i] = -(xr * a.y) * xk;
                best = fmaxf(best, fmaxf(fabsf(re[i]), fabsf(im[i])));
            }
            re[i] *= sc;
            im[i] *= sc;
        }
        store_octet(X16 + (size_t)side * nkc * nb * 4 * 2048, nb, kc, blk, rr, ko, re, im);
    }
    block_max(best, &w->mx[1]);
}

// ------------------------------------------------------------------------------- FP16X3 products

constexpr int STAGES = 3;
constexpr uint32_t STAGE_BYTES = 8 * PL;  // four planes of each operand
constexpr uint32_t PIPE_BYTES = STAGES * STAGE_BYTES;  // 96 KB
constexpr uint32_t RECV_BYTES = 128 * 128 * 8;         // 128 KB: the parts of this CTA's rows
constexpr size_t GSMEM = PIPE_BYTES + RECV_BYTES + 128;
static_assert(GSMEM <= 227 * 1024, "shared memory of one CTA");
constexpr int GTHREADS = 320;  // warps 0..7 send the partial tile, warp 8 copies, warp 9 MMAs; all finish it
constexpr int G_COPY = 8, G_MMA = 9;
constexpr int MODE_Y = 0, MODE_X = 1, MODE_D = 2;
constexpr float LOSS_PER_CHUNK = 1.3e-7f;  // mean relative truncation loss of a TMEM sum, per 16-k chunk

// C = P Q^H over all k, one 128 x 128 tile per cluster of C CTAs, each taking a part of k, in two TMEM
// sums (half the truncation of one).  CTA `rank` finishes rows [rank 128/C, ...) of the tile: every CTA
// stores its partial rows asynchronously into the finisher's shared memory, which counts the bytes on a
// barrier -- no cluster-wide barrier or fence is waited for between the MMAs and the sum (a version that
// staged the partial tiles and read them through distributed shared memory spent 6000 clocks in each of
// two releasing cluster barriers: 22 us a product at N = 691, 14 us now).
//   MODE_Y  Y = 2I - C, P = X_it, Q = A^H; planes of Y, words.dev[it]
//   MODE_X  X_(it+1) = C, P = Y, Q = X_it^H; planes of X and of X^H, words.mx[it + 1]
//   MODE_D  dX = C, P = R_j, Q = X^H; D (complex128), words.md[j = it]
// X16 holds two buffers of xstride values, X_it in buffer it & 1: the rows of X, then those of X^H.
template <int MODE, int C>
__global__ void __launch_bounds__(GTHREADS, 1)
    ns_product_kernel(const uint16_t *__restrict__ A16, uint16_t *X16, size_t xstride, uint16_t *Y16, double2 *D,
                      int N, int nb, int nkc, int it, int max_steps, Words *w, uint32_t *err, uint64_t wait_ns)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int rank = C > 1 ? (int)cluster_ctarank() : 0, tile = blockIdx.x / C;
    const int ti = tile / nb, tj = tile - (tile / nb) * nb;
    float4 *recv = reinterpret_cast<float4 *>(smem + PIPE_BYTES);  // [part][column pair 64][row R]
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + PIPE_BYTES + RECV_BYTES);
    uint64_t *empty = full + STAGES;
    uint64_t *done = empty + STAGES;
    uint64_t *got = done + 1;  // every part of this CTA's rows has arrived
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(got + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *n_issued = abort_flag + 1;
    volatile int *n_consumed = abort_flag + 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per = (nkc + C - 1) / C;
    const int kc0 = min(nkc, rank * per), n = min(nkc, kc0 + per) - kc0;
    const int n0 = (n + 1) / 2;  // chunks of the first TMEM sum

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        mbar_init(got, 1);
        *abort_flag = 0;
        *n_issued = 0;
        *n_consumed = 0;
        fence_barrier_init();
        mbar_arrive_expect_tx(got, RECV_BYTES);
    }
    if (warp == G_MMA)
        tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // The same decision in every CTA: these words are not written by this launch, but for done, and that
    // to a value under which this launch still runs.
    bool run = true;
    if (MODE == MODE_D) {
        run = !refine_over(w, it);
    } else {
        const int dn = *reinterpret_cast<volatile int *>(&w->done);
        run = dn == 0 || dn > it + 1;
        if (run && MODE == MODE_X && blockIdx.x == 0 && threadIdx.x == 0 && bits_f(w->dev[it]) < (float)NS_TOL)
            w->done = it + 2;
    }
    if (!run) {
        if (warp == G_MMA)
            tmem_dealloc(tmem, 512);
        return;
    }
    if (C > 1)
        cluster_arrive_relaxed();  // this CTA's barriers are ready for its peers
    const int xi = MODE == MODE_D ? current_it(w, max_steps) : it;
    const uint16_t *Xc = X16 + (xi & 1) * xstride;
    const uint16_t *Pp = MODE == MODE_Y ? Xc : Y16;
    const uint16_t *Qp = MODE == MODE_Y ? A16 : Xc + xstride / 2;
    constexpr int R = 128 / C;
    const int row0 = rank * R;

    if (warp == G_COPY) {
        if (lane == 0) {
            for (int u = 0; u < n; ++u) {
                const int s = u % STAGES;
                if (u >= STAGES && !mbar_wait(&empty[s], (uint32_t)(u / STAGES - 1) & 1u, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                    *abort_flag = 1;
                    break;
                }
                if (*abort_flag)
                    break;
                uint8_t *st = smem + s * STAGE_BYTES;
                mbar_arrive_expect_tx(&full[s], STAGE_BYTES);
                bulk_g2s(st, Pp + plane_at(kc0 + u, nb, ti, 4), 4 * PL, &full[s]);
                bulk_g2s(st + 4 * PL, Qp + plane_at(kc0 + u, nb, tj, 4), 4 * PL, &full[s]);
                *n_issued = u + 1;
            }
        }
        __syncwarp();
        if (C > 1)
            cluster_wait();
    } else if (warp == G_MMA) {
        if (lane == 0) {
            constexpr uint32_t ID = mma_idesc(0u, 128, 256, false);
            constexpr uint32_t ID1 = mma_idesc(0u, 128, 128, false), ID1N = mma_idesc(0u, 128, 128, true);
            for (int u = 0; u < n; ++u) {
                const int s = u % STAGES;
                if (!mbar_wait(&full[s], (uint32_t)(u / STAGES) & 1u, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + (u < n0 ? 0 : 256);
                const uint32_t st = smem_u32(smem) + s * STAGE_BYTES;
                const uint64_t a_ih = smem_desc(st, LBO, SBO), a_rh = smem_desc(st + PL, LBO, SBO);
                const uint64_t a_il = smem_desc(st + 2 * PL, LBO, SBO), a_rl = smem_desc(st + 3 * PL, LBO, SBO);
                const uint64_t b_ih = smem_desc(st + 4 * PL, LBO, SBO), b_rh = smem_desc(st + 5 * PL, LBO, SBO);
                const uint64_t b_il = smem_desc(st + 6 * PL, LBO, SBO), b_rl = smem_desc(st + 7 * PL, LBO, SBO);
                mma_f16(d, a_ih, b_ih, ID, u > 0 && u != n0 ? 1u : 0u);  // Re += Pi Qi, Im += Pi Qr
                mma_f16(d, a_ih, b_il, ID, 1);
                mma_f16(d, a_il, b_ih, ID, 1);
                mma_f16(d, a_rh, b_rh, ID1, 1);               // Re += Pr Qr
                mma_f16(d, a_rh, b_rl, ID1, 1);
                mma_f16(d, a_rl, b_rh, ID1, 1);
                mma_f16(d + 128, a_rh, b_ih, ID1N, 1);        // Im -= Pr Qi
                mma_f16(d + 128, a_rh, b_il, ID1N, 1);
                mma_f16(d + 128, a_rl, b_ih, ID1N, 1);
                mma_commit(&empty[s]);
                *n_consumed = u + 1;
            }
            mma_commit(done);  // arrives once every MMA issued above has completed
        }
        __syncwarp();
        if (C > 1)
            cluster_wait();
    } else {
        // The partial tile to the CTAs that finish its rows: lane = row, two columns per store.  It is
        // sent whatever happened before, so that every CTA receives all its bytes and none leaves while
        // stores to it are in flight.
        const int q = warp & 3, owner = q * 32 / R, row = q * 32 - owner * R + lane;
        if (C > 1)
            cluster_wait();
        const uint32_t dst = mapa_shared(recv + (size_t)rank * 64 * R + row, owner);
        const uint32_t bar = mapa_shared(got, owner);
        if (!__all_sync(0xffffffffu, mbar_wait(done, 0, wait_ns)) && lane == 0)
            record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
        tc_fence_after();
        const uint32_t base = tmem + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
        for (int c0 = (warp >> 2) * 64, e = c0 + 64; c0 < e; c0 += 16) {
            float re[16], im[16];
#pragma unroll
            for (int i = 0; i < 16; ++i)
                re[i] = im[i] = 0.f;
            if (n > 0)
                tmem_ld16x2(base + c0, base + 128 + c0, re, im);
            if (n > n0) {
                float r2[16], i2[16];
                tmem_ld16x2(base + 256 + c0, base + 384 + c0, r2, i2);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    re[i] += r2[i];
                    im[i] += i2[i];
                }
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
                st_async16(dst + (uint32_t)((c0 / 2 + i) * R) * 16,
                           make_float4(re[2 * i], im[2 * i], re[2 * i + 1], im[2 * i + 1]), bar);
        }
        tc_fence_before();
    }

    // what the sums mean
    int ea, eb, eo = 0;
    if (MODE == MODE_Y) {
        ea = w->ex[it];
        eb = exp_of(bits_f(w->a_max));
        eo = w->ey;
    } else if (MODE == MODE_X) {
        ea = w->ey;
        eb = w->ex[it];
        eo = exp_of(2.0f * bits_f(w->mx[it]) * 1.001f);
        if (blockIdx.x == 0 && threadIdx.x == 0)
            w->ex[it + 1] = eo;
    } else {
        ea = w->er;
        eb = w->ex[xi];
    }
    const float sc = ldexpf(1.0f + LOSS_PER_CHUNK * (float)((per + 1) / 2), ea + eb - 2 * SCALE_BITS);
    const float so = ldexpf(1.0f, SCALE_BITS - eo);
    uint16_t *Out = MODE == MODE_Y ? Y16 : X16 + ((it + 1) & 1) * xstride;
    // the peers' MMA waits are bounded by wait_ns, and they send after them in any case
    if (!mbar_wait_cluster(got, 0, 2 * wait_ns + DRAIN_NS) && lane == 0)
        record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
    float best = 0.f;
    // items: (8-row group, chunk of 16 columns, octet, row of the group): sixteen consecutive threads write
    // the 256 contiguous bytes of a group's plane
    for (int t = threadIdx.x; t < R * 16; t += GTHREADS) {
        const int row = (t >> 7) * 8 + (t & 7), ko = (t >> 3) & 1, ch = (t >> 4) & 7;
        const int cp = ch * 8 + ko * 4;  // first of four column pairs
        float4 v[C][4];
#pragma unroll
        for (int p = 0; p < C; ++p)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                v[p][i] = recv[(size_t)(p * 64 + cp + i) * R + row];
        float re[8], im[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float4 a = v[0][i];
#pragma unroll
            for (int p = 1; p < C; ++p) {  // a fixed order: the same sum in every run
                a.x += v[p][i].x;
                a.y += v[p][i].y;
                a.z += v[p][i].z;
                a.w += v[p][i].w;
            }
            re[2 * i] = a.x;
            im[2 * i] = a.y;
            re[2 * i + 1] = a.z;
            im[2 * i + 1] = a.w;
        }
        const int gi = ti * 128 + row0 + row, gj0 = tj * 128 + cp * 2;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int gj = gj0 + i;
            const bool in = gi < N && gj < N;
            float x = re[i] * sc, y = im[i] * sc;
            if (MODE == MODE_Y) {
                const float d = gi == gj ? 1.f - x : -x;
                y = -y;
                if (in)
                    best = fmaxf(best, finite_or_inf(sqrtf(d * d + y * y)));
                x = gi == gj ? d + 1.f : d;
            } else if (in) {
                best = fmaxf(best, finite_or_inf(fmaxf(fabsf(x), fabsf(y))));
            }
            re[i] = in ? x : 0.f;
            im[i] = in ? y : 0.f;
        }
        if (MODE == MODE_D) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (gi < N && gj0 + i < N)
                    D[(size_t)gi * N + gj0 + i] = make_double2((double)re[i], (double)im[i]);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                re[i] *= so;
                im[i] *= so;
            }
            if (tj * 8 + ch < nkc)
                store_octet(Out, nb, tj * 8 + ch, ti, row0 + row, ko, re, im);
        }
        if (MODE == MODE_X) {  // kept for X^H, in the place of the first part
#pragma unroll
            for (int i = 0; i < 4; ++i)
                recv[(size_t)(cp + i) * R + row] = make_float4(re[2 * i], im[2 * i], re[2 * i + 1], im[2 * i + 1]);
        }
    }
    if (MODE == MODE_X) {
        // rows of X^H: the 128 rows of block tj, k = the R rows of this CTA (whole chunks: R >= 32)
        __syncthreads();
        constexpr int nch = R / 16;
        for (int t = threadIdx.x; t < R * 16; t += GTHREADS) {
            const int ko = (t >> 3) & 1, ch = (t >> 4) % nch, grp = (t >> 4) / nch;
            const int col = grp * 8 + (t & 7);  // column of the tile: the row of X^H
            const int k0 = ch * 16 + ko * 8;    // first of eight rows
            const int kc = ti * 8 + (row0 >> 4) + ch;
            float re[8], im[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 v = recv[(size_t)(col >> 1) * R + k0 + i];
                re[i] = col & 1 ? v.z : v.x;
                im[i] = col & 1 ? -v.w : -v.y;
            }
            if (kc < nkc)
                store_octet(Out + xstride / 2, nb, kc, tj, col, ko, re, im);
        }
    }
    block_max(best, MODE == MODE_Y ? &w->dev[it] : MODE == MODE_X ? &w->mx[it + 1] : &w->md[it]);
    // copies and MMAs still in flight after an early end
    if (threadIdx.x == 0) {
        bool ok = mbar_wait(done, 0, DRAIN_NS);
        const int issued = *n_issued, consumed = *n_consumed;
        for (int u = consumed; u < issued && ok; ++u)
            ok = mbar_wait(&full[u % STAGES], (uint32_t)(u / STAGES) & 1u, DRAIN_NS);
        if (!ok)
            record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == G_MMA) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------------------- slices

// X of phase 1 (hi + lo of its planes) rounded to 28 bits of the largest entry: four slices and X64.
__global__ void __launch_bounds__(256) ns_slice_x_kernel(const uint16_t *__restrict__ X16, size_t xstride, int N,
                                                         int nb, int max_steps, uint16_t *__restrict__ SL,
                                                         double2 *__restrict__ X64, const Words *w)
{
    const int kc = blockIdx.x, blk = blockIdx.y;
    const int it = current_it(w, max_steps);
    const uint16_t *p = X16 + (it & 1) * xstride + plane_at(kc, nb, blk, 4);
    const int rr = (threadIdx.x >> 4) * 8 + (threadIdx.x & 7), ko = (threadIdx.x >> 3) & 1;
    const int off = (rr >> 3) * 128 + ko * 64 + (rr & 7) * 8;
    const int e = exp_of(bits_f(w->mx[it])), ep = w->ex[it];
    const float sc = ldexpf(1.0f, ep - SCALE_BITS + BITS * SL_X - e);  // plane value -> units of 2^(e - 28)
    long long nr[8], ni[8];
    const uint4 raw[4] = {*reinterpret_cast<const uint4 *>(p + off), *reinterpret_cast<const uint4 *>(p + 2048 + off),
                          *reinterpret_cast<const uint4 *>(p + 2 * 2048 + off),
                          *reinterpret_cast<const uint4 *>(p + 3 * 2048 + off)};
    const double unit = ldexp(1.0, e - BITS * SL_X);
    const int r = blk * 128 + rr;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        auto val = [&](int q) { return __half2float(reinterpret_cast<const __half *>(&raw[q])[i]); };
        const int a = __float2int_rn((val(1) + val(3)) * sc), b = __float2int_rn((val(0) + val(2)) * sc);
        nr[i] = a;
        ni[i] = b;
        const int k = kc * 16 + ko * 8 + i;
        if (r < N && k < N)
            X64[(size_t)r * N + k] = make_double2((double)a * unit, (double)b * unit);
    }
    store_slices<SL_X>(SL, 2 * SL_XD, nb, kc, blk, rr, ko, nr, ni);
}

// dX_j rounded to 41 bits of its largest entry: six slices, added to X64 as rounded.
__global__ void __launch_bounds__(256) ns_slice_d_kernel(const double2 *__restrict__ D, int N, int nb, int j,
                                                         uint16_t *__restrict__ SL, double2 *__restrict__ X64,
                                                         const Words *w)
{
    if (refine_over(w, j + 1))  // R_j was the last residual: its dX is added unrounded at the end
        return;
    const int kc = blockIdx.x, blk = blockIdx.y;
    const int rr = (threadIdx.x >> 4) * 8 + (threadIdx.x & 7), ko = (threadIdx.x >> 3) & 1;
    const int e = exp_of(bits_f(w->md[j])), s = BITS * SL_D - 1 - e;
    const double unit = ldexp(1.0, -s);
    const int r = blk * 128 + rr;
    long long nr[8], ni[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int k = kc * 16 + ko * 8 + i;
        nr[i] = ni[i] = 0;
        if (r < N && k < N) {
            const size_t at = (size_t)r * N + k;
            const double2 d = D[at];
            nr[i] = scaled_int(d.x, s);
            ni[i] = scaled_int(d.y, s);
            double2 x = X64[at];
            x.x += (double)nr[i] * unit;
            x.y += (double)ni[i] * unit;
            X64[at] = x;
        }
    }
    store_slices<SL_D>(SL, 2 * SL_XD, nb, kc, blk, rr, ko, nr, ni);
}

// ------------------------------------------------------------------------------- residual products

// One group of the slice products: diagonals d0 and d0 + 1 (t + u = d) of the slices u in [u0, u0 + nu) of
// P and t in [t0, t0 + nt) of Q over the chunks [kc0, kc1), into slots slot and slot + 1.  At most `win`
// chunks are summed in TMEM before the sums (exact integers below 2^24) are added into the slots.
struct Group {
    int d0, nd, u0, nu, t0, nt, kc0, kc1, slot, win;
};
constexpr int MAX_GROUPS = 24;
struct Groups {
    Group g[MAX_GROUPS];
    int n, slots;
    int shift[2 * MAX_GROUPS];  // of a slot's integers, in the common unit
};

constexpr uint32_t RPIPE = 49152u * 4;  // 192 KB of stages
constexpr int RSTAGES = 8;              // at most
constexpr size_t RSMEM = RPIPE + 256;
constexpr int RTHREADS = 320;           // warps 0..7 read TMEM, warp 8 copies, warp 9 MMAs
constexpr int R_COPY = 8, R_MMA = 9;

// T[slot][tile][column pair][row]: the tile's Re, Im of two columns, as int4; rows along consecutive
// lanes, so the epilogue stores and the combine loads 512 contiguous bytes a warp.
__global__ void __launch_bounds__(RTHREADS, 1)
    ns_residual_kernel(const uint16_t *__restrict__ SP, int npP, const uint16_t *__restrict__ SQ, int npQ,
                       const __grid_constant__ Groups grp, int nb, int j, int4 *__restrict__ T, const Words *w,
                       uint32_t *err, uint64_t wait_ns)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const Group g = grp.g[blockIdx.y];
    const int tile = blockIdx.x, ti = tile / nb, tj = tile - (tile / nb) * nb;
    const uint32_t SB = (uint32_t)(g.nu + g.nt) * 2 * PL;
    const int NST = min(RSTAGES, (int)(RPIPE / SB));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + RPIPE);
    uint64_t *empty = full + RSTAGES;
    uint64_t *ready = empty + RSTAGES;  // window complete in TMEM
    uint64_t *freed = ready + 1;        // window read
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(freed + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *n_issued = abort_flag + 1;
    volatile int *n_consumed = abort_flag + 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = g.kc1 - g.kc0, nwin = (n + g.win - 1) / g.win;

    if (threadIdx.x == 0) {
        for (int s = 0; s < RSTAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(ready, 1);
        mbar_init(freed, 8);
        *abort_flag = 0;
        *n_issued = 0;
        *n_consumed = 0;
        fence_barrier_init();
    }
    if (warp == R_MMA)
        tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (refine_over(w, j)) {
        if (warp == R_MMA)
            tmem_dealloc(tmem, 512);
        return;
    }

    if (warp == R_COPY) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            for (int u = 0; u < n; ++u) {
                if (u >= NST && !mbar_wait(&empty[s], ph ^ 1u, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                    *abort_flag = 1;
                    break;
                }
                if (*abort_flag)
                    break;
                uint8_t *st = smem + s * SB;
                mbar_arrive_expect_tx(&full[s], SB);
                bulk_g2s(st, SP + plane_at(g.kc0 + u, nb, ti, npP) + (size_t)g.u0 * 2 * 2048, g.nu * 2 * PL, &full[s]);
                bulk_g2s(st + g.nu * 2 * PL, SQ + plane_at(g.kc0 + u, nb, tj, npQ) + (size_t)g.t0 * 2 * 2048,
                         g.nt * 2 * PL, &full[s]);
                *n_issued = u + 1;
                if (++s == NST) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        __syncwarp();
    } else if (warp == R_MMA) {
        if (lane == 0) {
            constexpr uint32_t ID = mma_idesc(0u, 128, 256, false);
            constexpr uint32_t ID1 = mma_idesc(0u, 128, 128, false), ID1N = mma_idesc(0u, 128, 128, true);
            int s = 0, u = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int win = 0; win < nwin && ok; ++win) {
                if (win > 0 && !mbar_wait(freed, (uint32_t)(win - 1) & 1u, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                const int end = min(n, u + g.win);
                uint32_t started = 0;  // bit a: accumulator a holds something of this window
                for (; u < end; ++u) {
                    if (!mbar_wait(&full[s], ph, wait_ns)) {
                        record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                        *abort_flag = 1;
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t st = smem_u32(smem) + s * SB;
                    for (int a = 0; a < g.nd; ++a)
                        for (int x = 0; x < g.nu; ++x) {
                            const int y = g.d0 + a - (g.u0 + x) - g.t0;
                            if (y < 0 || y >= g.nt)
                                continue;
                            const uint32_t d = tmem + a * 256;
                            const uint32_t pa = st + x * 2 * PL, pb = st + (g.nu + y) * 2 * PL;
                            const uint64_t ai = smem_desc(pa, LBO, SBO), ar = smem_desc(pa + PL, LBO, SBO);
                            const uint64_t bi = smem_desc(pb, LBO, SBO), br = smem_desc(pb + PL, LBO, SBO);
                            mma_f16(d, ai, bi, ID, (started >> a) & 1u);  // Re += Pi Qi, Im += Pi Qr
                            mma_f16(d, ar, br, ID1, 1);                   // Re += Pr Qr
                            mma_f16(d + 128, ar, bi, ID1N, 1);            // Im -= Pr Qi
                            started |= 1u << a;
                        }
                    mma_commit(&empty[s]);
                    *n_consumed = u + 1;
                    if (++s == NST) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                mma_commit(ready);
            }
        }
        __syncwarp();
    } else {
        const int q = warp & 3, row = q * 32 + lane;
        for (int win = 0; win < nwin; ++win) {
            if (!__all_sync(0xffffffffu, mbar_wait(ready, (uint32_t)win & 1u, wait_ns)) || *abort_flag) {
                if (lane == 0)
                    record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            for (int a = 0; a < g.nd; ++a) {
                int4 *out = T + ((size_t)(g.slot + a) * gridDim.x + tile) * (64 * 128) + row;
                const uint32_t base = tmem + ((uint32_t)(q * 32) << 16) + a * 256;
#pragma unroll 1
                for (int c0 = (warp >> 2) * 64; c0 < (warp >> 2) * 64 + 64; c0 += 16) {
                    float re[16], im[16];
                    tmem_ld16x2(base + c0, base + 128 + c0, re, im);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        int4 v = make_int4(__float2int_rn(re[2 * i]), __float2int_rn(im[2 * i]),
                                           __float2int_rn(re[2 * i + 1]), __float2int_rn(im[2 * i + 1]));
                        int4 *o = out + (size_t)(c0 / 2 + i) * 128;
                        if (win > 0) {  // fewer than 128 windows: the sums stay within 32 bits
                            const int4 p = *o;
                            v = make_int4(v.x + p.x, v.y + p.y, v.z + p.z, v.w + p.w);
                        }
                        *o = v;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(freed);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // the copies and MMAs still in flight after an early end
        const int issued = *n_issued, consumed = *n_consumed;
        bool ok = true;
        for (int u = consumed; u < issued && ok; ++u)
            ok = mbar_wait(&full[u % NST], (uint32_t)(u / NST) & 1u, DRAIN_NS);
        if (consumed > 0)
            ok = mbar_wait(&empty[(consumed - 1) % NST], (uint32_t)((consumed - 1) / NST) & 1u, DRAIN_NS) && ok;
        if (!ok)
            record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == R_MMA) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// R_0 = I - sum (j = 0) or R_j = R_(j-1) - sum (j > 0) of the slots' integers: R64, R's FP16X3 planes and
// max |R_j|.  The integers are added modulo 2^64 in units of 2^(e - width); R_0 is far below 2^(e - 1) after a
// phase 1 that converged, and an FP32 sum of the same slots tells where it is not: the entry of R_0 is then
// NaN and stays so in every later residual, whose maximum (infinite) fails the final check.  Thread: one row,
// eight columns.
__global__ void __launch_bounds__(256)
    ns_combine_kernel(const int4 *__restrict__ T, const __grid_constant__ Groups grp, int N, int nb, int nkc, int j,
                      int max_steps, double2 *__restrict__ R64, uint16_t *__restrict__ R16, Words *w)
{
    if (refine_over(w, j))
        return;
    const int tile = blockIdx.x, ti = tile / nb, tj = tile - (tile / nb) * nb;
    const int row = threadIdx.x & 127, oct = blockIdx.y * 2 + (threadIdx.x >> 7);
    const int it = current_it(w, max_steps);
    const int ea = exp_of(bits_f(w->a_max)) + 1;
    const int eb = j == 0 ? exp_of(bits_f(w->mx[it])) : exp_of(bits_f(w->md[j - 1])) + 1;
    const int width = j == 0 ? BITS * (SL_A + 1) : BITS * (SL_D + 1);  // unit 2^(ea + eb - width)
    // R's planes: a bound on max |R_j| (header comment on loose bounds)
    float bound;
    if (j == 0)
        bound = fmaxf(4.f * bits_f(w->dev[min(it, max_steps)]), ldexpf(1.0f, ea + eb - 14));
    else
        bound = 0.25f * bits_f(w->mr[j - 1]);
    const int er = exp_of(bound);
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0)
        w->er = er;
    const float so = ldexpf(1.0f, SCALE_BITS - er);
    const double unit = ldexp(1.0, ea + eb - width);
    const int gi = ti * 128 + row, gj0 = tj * 128 + oct * 8;
    long long sr[8], si[8];
    float fr[8], fi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        sr[i] = si[i] = 0;
        fr[i] = fi[i] = 0.f;
    }
    for (int s = 0; s < grp.slots; ++s) {
        const int4 *p = T + ((size_t)s * gridDim.x + tile) * (64 * 128) + (size_t)(oct * 4) * 128 + row;
        const int sh = grp.shift[s];
        const float fs = ldexpf(1.0f, sh - width);  // in units of 2^(ea + eb)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int4 v = p[i * 128];
            sr[2 * i] += (long long)((unsigned long long)(long long)v.x << sh);
            si[2 * i] += (long long)((unsigned long long)(long long)v.y << sh);
            sr[2 * i + 1] += (long long)((unsigned long long)(long long)v.z << sh);
            si[2 * i + 1] += (long long)((unsigned long long)(long long)v.w << sh);
            fr[2 * i] = fmaf((float)v.x, fs, fr[2 * i]);
            fi[2 * i] = fmaf((float)v.y, fs, fi[2 * i]);
            fr[2 * i + 1] = fmaf((float)v.z, fs, fr[2 * i + 1]);
            fi[2 * i + 1] = fmaf((float)v.w, fs, fi[2 * i + 1]);
        }
    }
    const int ish = width - (ea + eb);  // I in units
    float best = 0.f, re[8], im[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int gj = gj0 + i;
        re[i] = im[i] = 0.f;
        if (gi >= N || gj >= N)
            continue;
        double xr, xi;
        if (j == 0) {
            const unsigned long long one = gi == gj && ish >= 0 && ish < 64 ? 1ull << ish : 0ull;
            const float one_f = gi == gj ? ldexpf(1.0f, -(ea + eb)) : 0.f;
            xr = (double)(long long)(one - (unsigned long long)sr[i]) * unit;
            xi = (double)(long long)(0ull - (unsigned long long)si[i]) * unit;
            if (!(fabsf(one_f - fr[i]) < 0.4f) || !(fabsf(fi[i]) < 0.4f) || ish < 0 || (gi == gj && ish >= 64))
                xr = __longlong_as_double(0x7ff8000000000000ll);
        } else {
            const double2 r = R64[(size_t)gi * N + gj];
            xr = r.x - (double)sr[i] * unit;
            xi = r.y - (double)si[i] * unit;
        }
        R64[(size_t)gi * N + gj] = make_double2(xr, xi);
        re[i] = (float)xr;
        im[i] = (float)xi;
        best = fmaxf(best, finite_or_inf(sqrtf(re[i] * re[i] + im[i] * im[i])));
        re[i] *= so;
        im[i] *= so;
    }
    const int kc = tj * 8 + (oct >> 1);
    if (kc < nkc)
        store_octet(R16, nb, kc, ti, row, oct & 1, re, im);
    block_max(best, &w->mr[j]);
}

// Xout = X64 + the last dX, and the verdict: the last residual is small (each is exact for the X64 it was
// taken of) and the last dX, which no residual has seen, finite.  A failure after a phase 1 that ran out of steps is told
// apart (NS_DETAIL_CAP): the eager form, with more steps, may still converge.
__global__ void ns_final_kernel(const double2 *__restrict__ X64, const double2 *__restrict__ D, size_t n,
                                double2 *__restrict__ Xout, const Words *w, uint32_t *err)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double2 x = X64[i], d = D[i];
        Xout[i] = make_double2(x.x + d.x, x.y + d.y);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int last = 0;
        while (last + 1 < NS_REFINE && !refine_over(w, last + 1))
            ++last;
        if (!(bits_f(w->mr[last]) <= (float)NS_ACCEPT) || !isfinite(bits_f(w->md[last])))
            record_error(err, GW_E_NUMERIC, SITE_NS, w->done ? 0u : NS_DETAIL_CAP);
    }
}

// ------------------------------------------------------------------------------- host side

struct Carver {
    uint8_t *base;
    size_t used = 0;
    void *take(size_t bytes)
    {
        void *r = base ? base + used : nullptr;
        used += (bytes + 255) / 256 * 256;
        return r;
    }
};

// Slice groups of the residual with P in nsP slices of first digit m0 (64 or 128), Q in nsQ: the products
// with t + u <= dmax, two diagonals a group.  tiles < 64: each group's k range is cut into windows, one CTA
// each (N <= 1024: otherwise too few CTAs); else into two or one.
Groups make_groups(int nsP, int m0, int nsQ, int dmax, int nkc, int tiles)
{
    Groups r = {};
    for (int d0 = 0; d0 <= dmax; d0 += 2) {
        const int nd = std::min(2, dmax + 1 - d0);
        int umin = nsP, umax = -1, tmin = nsQ, tmax = -1, win = 1 << 20;
        for (int a = 0; a < nd; ++a) {
            int bound = 0;  // largest sum of |Re| or |Im| products per k, in units of 64 * 64
            for (int u = 0; u < nsP; ++u) {
                const int t = d0 + a - u;
                if (t < 0 || t >= nsQ)
                    continue;
                umin = std::min(umin, u);
                umax = std::max(umax, u);
                tmin = std::min(tmin, t);
                tmax = std::max(tmax, t);
                bound += 2 * (u == 0 ? m0 / 64 : 1);
            }
            if (bound > 0)
                win = std::min(win, (1 << 24) / (bound * 64 * 64 * 16));
        }
        const int parts = tiles <= 64 ? (nkc + win - 1) / win : tiles <= 256 ? std::min(2, nkc) : 1;
        const int per = (nkc + parts - 1) / parts;
        for (int p = 0; p * per < nkc; ++p) {
            Group &g = r.g[r.n++];
            g = {d0, nd, umin, umax - umin + 1, tmin, tmax - tmin + 1, p * per, std::min(nkc, (p + 1) * per), r.slots,
                 win};
            for (int a = 0; a < nd; ++a)
                r.shift[r.slots++] = BITS * (dmax - d0 - a);
        }
    }
    return r;
}

struct Work {
    int nb, nkc;
    Groups g0, g1;  // R_0, R_j
    size_t xstride;
    uint16_t *A16, *ASL, *X16, *Y16, *XSL;
    int4 *T;
    double2 *X64, *R64, *D;
    float *rs;
    Words *w;
    size_t bytes;
};

Work carve(void *base, int N)
{
    Work k = {};
    k.nb = (N + 127) / 128;
    k.nkc = (N + 15) / 16;
    k.g0 = make_groups(SL_X, 128, SL_A, SL_A - 1, k.nkc, k.nb * k.nb);
    k.g1 = make_groups(SL_D, 64, SL_D, SL_D - 1, k.nkc, k.nb * k.nb);
    const size_t plane = (size_t)k.nkc * k.nb * 2048;  // 16-bit values of one plane
    const size_t nn = (size_t)N * N;
    Carver c{static_cast<uint8_t *>(base)};
    k.xstride = 8 * plane;
    k.w = static_cast<Words *>(c.take(sizeof(Words)));
    k.rs = static_cast<float *>(c.take(N * sizeof(float)));
    k.A16 = static_cast<uint16_t *>(c.take(4 * plane * 2));
    k.ASL = static_cast<uint16_t *>(c.take(2 * SL_A * plane * 2));
    k.X16 = static_cast<uint16_t *>(c.take(16 * plane * 2));
    k.Y16 = static_cast<uint16_t *>(c.take(4 * plane * 2));
    k.XSL = static_cast<uint16_t *>(c.take(2 * SL_XD * plane * 2));
    k.T = static_cast<int4 *>(c.take((size_t)std::max(k.g0.slots, k.g1.slots) * k.nb * k.nb * 64 * 128 * sizeof(int4)));
    k.X64 = static_cast<double2 *>(c.take(nn * sizeof(double2)));
    k.R64 = static_cast<double2 *>(c.take(nn * sizeof(double2)));
    k.D = static_cast<double2 *>(c.take(nn * sizeof(double2)));
    k.bytes = c.used;
    return k;
}

// CTAs per tile, 1, 2 or 4: k split over a cluster while the launch still fits the GPU at one CTA per SM and
// each CTA keeps two chunks.  (Clusters of 8 are slower: 72 CTAs at N = 257 took 25 us more a product than
// 36 in clusters of 4.)
int cluster_size(int tiles, int nkc, int nsm)
{
    int c = 4;
    while (c > 1 && (tiles * c > nsm || nkc < 2 * c))
        c /= 2;
    return c;
}

template <typename... P, typename... Q>
cudaError_t launch(void (*kernel)(P...), dim3 grid, int threads, size_t smem, int cluster, cudaStream_t s, Q... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 0 ? 1 : 0;
    count_launches(1);
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

template <int MODE, int C>
cudaError_t launch_product_c(const Work &k, int N, int it, int max_steps, uint32_t *err, uint64_t wait_ns,
                             cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(ns_product_kernel<MODE, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)GSMEM);
    if (e != cudaSuccess)
        return e;
    return launch(ns_product_kernel<MODE, C>, dim3(k.nb * k.nb * C), GTHREADS, GSMEM, C, s, k.A16, k.X16,
                            k.xstride, k.Y16, k.D, N, k.nb, k.nkc, it, max_steps, k.w, err, wait_ns);
}

template <int MODE>
cudaError_t launch_product(const Work &k, int N, int it, int max_steps, int nsm, uint32_t *err, uint64_t wait_ns,
                           cudaStream_t s)
{
    switch (cluster_size(k.nb * k.nb, k.nkc, nsm)) {
    case 1: return launch_product_c<MODE, 1>(k, N, it, max_steps, err, wait_ns, s);
    case 2: return launch_product_c<MODE, 2>(k, N, it, max_steps, err, wait_ns, s);
    default: return launch_product_c<MODE, 4>(k, N, it, max_steps, err, wait_ns, s);
    }
}

// Host read of the phase-1 word (waits for the stream); a failed read counts as "not set".
bool phase1_done(const Words *w, cudaStream_t s)
{
    int h = 0;
    if (cudaMemcpyAsync(&h, &w->done, sizeof h, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return h != 0;
}

}  // namespace

size_t ns_work_bytes(int N)
{
    return carve(nullptr, N).bytes;
}

size_t ns_report_bytes()
{
    return sizeof(Words);
}

cudaError_t ns_report_copy(const void *work, int N, void *host, cudaStream_t s)
{
    return cudaMemcpyAsync(host, carve(const_cast<void *>(work), N).w, sizeof(Words), cudaMemcpyDeviceToHost, s);
}

// out4[0] FP16X3 steps of phase 1 until the tolerance was met, [1] residual max |I - X A| after phase 1, [2] the last measured
// residual, [3] refinements that ran.
void ns_report(const void *host, double *out4)
{
    const Words &h = *static_cast<const Words *>(host);
    auto f = [](unsigned b) { return (double)__builtin_bit_cast(float, b); };
    int last = 0;
    while (last + 1 < NS_REFINE && !(f(h.mr[last]) <= (double)(float)NS_LAST))
        ++last;
    out4[0] = h.done ? h.done - 2 : NS_MAX;
    out4[1] = f(h.mr[0]);
    out4[2] = f(h.mr[last]);
    out4[3] = last + 1;
}

// The kernels of every step check the device words, so the result does not depend on the host reads
// below: they only stop queuing steps that would return at once (after steps 4, 6, 8, ...), at the price
// of a stream synchronisation each.  With graph_safe every step is queued and nothing is read, so the
// whole inverse can be captured into a CUDA graph.
cudaError_t ns_inverse_enqueue(const double2 *A, int N, double2 *Xout, void *work, uint32_t *err, uint64_t wait_ns,
                               int nsm, cudaStream_t s, bool graph_safe, int max_steps)
{
    max_steps = std::max(1, std::min(max_steps, NS_MAX));
    const Work k = carve(work, N);
    const size_t nn = (size_t)N * N;
    const dim3 by_chunk(k.nkc, k.nb);
    const int flat = (int)std::max<size_t>(1, std::min<size_t>((nn + 255) / 256, (size_t)nsm * 8));
    cudaError_t e;
#define NS_TRY(x)                     \
    do {                              \
        if ((e = (x)) != cudaSuccess) \
            return e;                 \
    } while (0)
    NS_TRY(cudaMemsetAsync(k.w, 0, sizeof(Words), s));
    const int nslice = k.nkc * k.nb;
    NS_TRY(launch(ns_max_kernel, dim3(std::min(flat, nsm * 4)), 256, 0, 0, s, A, N, k.rs, k.w));
    NS_TRY(launch(ns_prep_kernel, dim3(nslice + std::max(1, std::min(nsm, (N + 7) / 8))), 256, 0, 0, s, A, N,
                            k.nb, k.nkc, k.rs, k.A16, k.ASL, k.w));
    NS_TRY(launch(ns_init_kernel, by_chunk, 256, 0, 0, s, A, N, k.nb, k.nkc, k.rs, k.X16 + k.xstride, k.w));
    for (int it = 1; it <= max_steps; ++it) {
        NS_TRY(launch_product<MODE_Y>(k, N, it, max_steps, nsm, err, wait_ns, s));
        NS_TRY(launch_product<MODE_X>(k, N, it, max_steps, nsm, err, wait_ns, s));
        if (!graph_safe && it >= 4 && !(it & 1) && phase1_done(k.w, s))
            break;
    }
    NS_TRY(launch(ns_slice_x_kernel, by_chunk, 256, 0, 0, s, k.X16, k.xstride, N, k.nb, max_steps, k.XSL, k.X64,
                            k.w));
    NS_TRY(cudaFuncSetAttribute(ns_residual_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RSMEM));
    for (int j = 0; j < NS_REFINE; ++j) {
        const Groups &g = j == 0 ? k.g0 : k.g1;
        NS_TRY(launch(ns_residual_kernel, dim3(k.nb * k.nb, g.n), RTHREADS, RSMEM, 0, s, k.XSL, 2 * SL_XD,
                                k.ASL, 2 * SL_A, g, k.nb, j, k.T, k.w, err, wait_ns));
        NS_TRY(launch(ns_combine_kernel, dim3(k.nb * k.nb, 8), 256, 0, 0, s, k.T, g, N, k.nb, k.nkc, j,
                                max_steps, k.R64, k.Y16, k.w));
        NS_TRY(launch_product<MODE_D>(k, N, j, max_steps, nsm, err, wait_ns, s));
        if (j + 1 < NS_REFINE)
            NS_TRY(launch(ns_slice_d_kernel, by_chunk, 256, 0, 0, s, k.D, N, k.nb, j, k.XSL, k.X64, k.w));
    }
    NS_TRY(launch(ns_final_kernel, dim3(flat), 256, 0, 0, s, k.X64, k.D, nn, Xout, k.w, err));
#undef NS_TRY
    return cudaSuccess;
}

}  // namespace gw
