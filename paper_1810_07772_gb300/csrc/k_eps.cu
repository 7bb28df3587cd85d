// eps_GG' = delta_GG' - sqrt(V(G)) P~_GG' sqrt(V(G')) and its FP64 inverse (Sec. 5.1).
//
// The inverse is a blocked Cholesky eps = L L^H (right-looking, 32-wide panels; each trailing update
// factors the next diagonal block beside it) followed by eps^-1 = Y^H Y with Y = L^-1, in triangular
// products whose work is dealt out evenly over the SMs.  N = 515: 1.9 -> 1.0 ms.  A general complex128 GEMM
// drives the paper's Newton iteration X <- X (2I - eps X) when that method is requested.
#include <algorithm>

#include "gw_internal.cuh"

namespace gw {

namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ double2 cconj(double2 a)
{
    return make_double2(a.x, -a.y);
}

__global__ void eps_build_kernel(const float2 *__restrict__ PG, const double *__restrict__ sv, int ng,
                                 double2 *__restrict__ eps)
{
    const size_t n = (size_t)ng * ng;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int g = static_cast<int>(i / ng), h = static_cast<int>(i - (size_t)g * ng);
        const float2 p = PG[i];
        const double s = sv[g] * sv[h];
        eps[i] = make_double2((g == h ? 1.0 : 0.0) - s * (double)p.x, -s * (double)p.y);
    }
}

// ---------------------------------------------------------------------------- zgemm
constexpr int ZT = 16;    // output tile (ZT x ZT, one complex output per thread)
constexpr int ZKC = 32;   // k chunk staged in shared memory

// C = alpha op(A) op(B) + beta C.
//
// FP64 on this GPU: each SM sub-partition retires about 0.42 lane-FMAs per clock, so one
// warp-wide DFMA holds its sub-partition for ~77 clocks and the kernel is bound by how many
// DFMAs each warp issues and on how many sub-partitions they run.  Each thread therefore owns a
// single output (4 DFMAs per k), a CTA is 8 warps (two per sub-partition) on a 16 x 16 tile, and
// even the small products of the factorisation spread over hundreds of warps.  Shared-memory and
// global traffic are minor next to that.  Batched products: problem blockIdx.z uses A + z sA,
// B + z sB, C + z sC.
__global__ void __launch_bounds__(256)
    zgemm_kernel(int M, int N, int K, double2 alpha, const double2 *__restrict__ A, int lda, int opA,
                 const double2 *__restrict__ B, int ldb, int opB, double2 beta, double2 *__restrict__ C, int ldc,
                 long sA, long sB, long sC)
{
    __shared__ double2 As[ZKC][ZT + 1];
    __shared__ double2 Bs[ZKC][ZT + 1];
    A += blockIdx.z * sA;
    B += blockIdx.z * sB;
    C += blockIdx.z * sC;
    const int i0 = blockIdx.y * ZT, j0 = blockIdx.x * ZT;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    double2 acc = make_double2(0.0, 0.0);
    for (int k0 = 0; k0 < K; k0 += ZKC) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int t = tid + 256 * e;
            int i, kk;
            if (opA == 0) {
                i = t / ZKC;
                kk = t % ZKC;
            } else {
                kk = t / ZT;
                i = t % ZT;
            }
            const int gi = i0 + i, gk = k0 + kk;
            double2 v = make_double2(0.0, 0.0);
            if (gi < M && gk < K)
                v = opA == 0 ? A[(size_t)gi * lda + gk] : cconj(A[(size_t)gk * lda + gi]);
            As[kk][i] = v;
            int j, kb;
            if (opB == 0) {
                kb = t / ZT;
                j = t % ZT;
            } else {
                j = t / ZKC;
                kb = t % ZKC;
            }
            const int gj = j0 + j, gk2 = k0 + kb;
            double2 w = make_double2(0.0, 0.0);
            if (gj < N && gk2 < K)
                w = opB == 0 ? B[(size_t)gk2 * ldb + gj] : cconj(B[(size_t)gj * ldb + gk2]);
            Bs[kb][j] = w;
        }
        __syncthreads();
        const int kn = min(ZKC, K - k0);
#pragma unroll 8
        for (int kk = 0; kk < kn; ++kk) {
            const double2 a = As[kk][ty], b = Bs[kk][tx];
            acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
            acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
        }
        __syncthreads();
    }
    const int gi = i0 + ty, gj = j0 + tx;
    if (gi < M && gj < N) {
        double2 v = cmul(alpha, acc);
        if (beta.x != 0.0 || beta.y != 0.0) {
            const double2 c = cmul(beta, C[(size_t)gi * ldc + gj]);
            v.x += c.x;
            v.y += c.y;
        }
        C[(size_t)gi * ldc + gj] = v;
    }
}

// ---------------------------------------------------------------------------- triangular products
// C = +-op(A) B where a known triangle of an operand is zero, the shapes of the triangular inverse:
//   TRI_RIGHT  B lower triangular (k >= j),   TRI_LEFT  A lower triangular (k <= i),
//   TRI_GRAM   C = A^H A of a lower triangular A (k >= max(i, j)): the lower half, mirrored.
// Tiles of 8 x 16 (one warp per sub-partition), of which a CTA per SM takes a fixed share: the tiles in
// descending order of their k range, dealt forwards and backwards in turn, so that every SM gets about
// the same number of DFMAs.  16 x 16 tiles one per CTA, in row order, left that to chance and the
// longest tiles to the end: at N = 515, A^H A 349 us, the 256-wide products 134 and 108, the three-row remainder
// 145; now 212, 79, 72 and 85.  The k terms of an output are added in ascending order, as in zgemm_kernel.
constexpr int TM = 8, TN = 16, TTHREADS = TM * TN;
enum { TRI_RIGHT = 0, TRI_LEFT = 1, TRI_GRAM = 2 };

template <int KIND>
__global__ void __launch_bounds__(TTHREADS)
    ztri_kernel(int M, int N, int K, double sign, const double2 *__restrict__ A, int lda, long sA,
                const double2 *__restrict__ B, int ldb, long sB, double2 *__restrict__ C, int ldc, long sC, int batch)
{
    __shared__ double2 As[ZKC][TM + 1];
    __shared__ double2 Bs[ZKC][TN + 1];
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int nti = (M + TM - 1) / TM, ntj = (N + TN - 1) / TN;
    // TRI_GRAM: rows 2p and 2p + 1 of tiles have p + 1 tiles each
    const int np = nti / 2, ntiles = KIND == TRI_GRAM ? np * (np + 1) + (nti & 1) * (np + 1) : nti * ntj * batch;
    for (int q = 0; q * (int)gridDim.x < ntiles; ++q) {
        const int t = q * gridDim.x + (q & 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
        if (t >= ntiles)
            continue;
        int ti, tj, z = 0;
        if (KIND == TRI_GRAM) {
            int p = (int)((sqrtf(4.f * t + 1.f) - 1.f) * 0.5f);
            while (p * (p + 1) > t)
                --p;
            while ((p + 1) * (p + 2) <= t)
                ++p;
            const int r = t - p * (p + 1);
            ti = 2 * p + r / (p + 1);
            tj = r % (p + 1);
        } else if (KIND == TRI_RIGHT) {
            tj = t / (nti * batch);
            ti = t % nti;
            z = t / nti % batch;
        } else {
            ti = nti - 1 - t / (ntj * batch);
            tj = t % ntj;
            z = t / ntj % batch;
        }
        const int i0 = ti * TM, j0 = tj * TN;
        const int kbeg = KIND == TRI_GRAM ? max(i0, j0) : KIND == TRI_RIGHT ? j0 : 0;
        const int kend = KIND == TRI_LEFT ? min(K, i0 + TM) : K;
        const double2 *a = A + z * sA, *b = B + z * sB;
        double2 ra[2], rb[4];
        auto fetch = [&](int k0) {  // one chunk of both operands
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int i = KIND == TRI_GRAM ? tid & 7 : (tid >> 5) + 4 * e;
                const int k = k0 + (KIND == TRI_GRAM ? (tid >> 3) + 16 * e : tid & 31);
                ra[e] = make_double2(0.0, 0.0);
                if (i0 + i < M && k < kend)
                    ra[e] = KIND == TRI_GRAM ? cconj(a[(size_t)k * lda + i0 + i]) : a[(size_t)(i0 + i) * lda + k];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int k = k0 + (tid >> 4) + 8 * e;
                rb[e] = make_double2(0.0, 0.0);
                if (j0 + tx < N && k < kend)
                    rb[e] = b[(size_t)k * ldb + j0 + tx];
            }
        };
        double2 acc = make_double2(0.0, 0.0);
        fetch(kbeg);
        for (int k0 = kbeg; k0 < kend; k0 += ZKC) {
#pragma unroll
            for (int e = 0; e < 2; ++e)
                As[KIND == TRI_GRAM ? (tid >> 3) + 16 * e : tid & 31][KIND == TRI_GRAM ? tid & 7 : (tid >> 5) + 4 * e] =
                    ra[e];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                Bs[(tid >> 4) + 8 * e][tx] = rb[e];
            __syncthreads();
            if (k0 + ZKC < kend)
                fetch(k0 + ZKC);  // behind this chunk's arithmetic
            const int kn = min(ZKC, kend - k0);
#pragma unroll 8
            for (int kk = 0; kk < kn; ++kk) {
                const double2 x = As[kk][ty], y = Bs[kk][tx];
                acc.x = fma(x.x, y.x, fma(-x.y, y.y, acc.x));
                acc.y = fma(x.x, y.y, fma(x.y, y.x, acc.y));
            }
            __syncthreads();
        }
        const int gi = i0 + ty, gj = j0 + tx;
        if (gi < M && gj < N && (KIND != TRI_GRAM || gj <= gi)) {
            const double2 v = make_double2(sign * acc.x, sign * acc.y);
            C[z * sC + (size_t)gi * ldc + gj] = v;
            if (KIND == TRI_GRAM && gj < gi)
                C[(size_t)gj * ldc + gi] = cconj(v);
        }
    }
}

// ---------------------------------------------------------------------------- diagonal block
// 1/sqrt(d) by the Newton-Raphson iteration y <- y (3 - d y^2) / 2 started from the FP32 estimate:
// each step doubles the number of correct bits (24 -> 48 -> FP64 rounding).  On this GPU an FP64
// FMA has a 64-cycle latency and a correctly rounded FP64 sqrt plus division cost more than 1000
// cycles, so two short Newton steps are the faster route to a pivot and its reciprocal.
__device__ __forceinline__ double rsqrt_newton(double d)
{
    const float df = static_cast<float>(d);
    if (!(df > 1e-30f) || !(df < 1e30f))
        return 1.0 / sqrt(d);
    double y = static_cast<double>(rsqrtf(df));
    const double hd = 0.5 * d;
    y = y * fma(-hd * y, y, 1.5);
    y = y * fma(-hd * y, y, 1.5);
    return y;
}

// 1/d by the Newton-Raphson iteration y <- y + y (1 - d y) from the FP32 reciprocal: each step
// doubles the number of correct bits (24 -> 48 -> FP64 rounding), two dependent FMAs per step.
__device__ __forceinline__ double rcp_newton(double d)
{
    const float df = static_cast<float>(d);
    if (!(fabsf(df) > 1e-30f) || !(fabsf(df) < 1e30f))
        return 1.0 / d;
    double y = static_cast<double>(__frcp_rn(df));
    y = fma(y, fma(-d, y, 1.0), y);
    y = fma(y, fma(-d, y, 1.0), y);
    return y;
}

// Factor the n x n (n <= 32) Hermitian block in m.S (lower triangle; zero elsewhere) as L L^H, L to A
// (the strict upper triangle zeroed) and Linv = L^-1 (lower, zero above).  256 threads.
//
// The block is factored as L~ D L~^H (L~ unit lower, D real), and L = L~ D^1/2 is formed at
// the end; the square roots and the column scalings are off the chain from one pivot to the next.
//  * pivot j (one barrier) subtracts S[i][j] r conj(S[l][j]), r = 1/d_j, from the entries (i, l), j < l <= i (column
//    j stays unscaled: it holds L~_ij d_j), and, for X = L~^-1, L~_kj X[j][c] from the entries (k, c), c <= j < k;
//  * warp 0 takes the next pivot's column, one entry a lane, and goes on to its reciprocal and the scaled
//    column L~_i,j+1, which the next step reads; the other warps take the rest of both lists, two products'
//    four DFMAs an entry;
//  * L = L~ diag(sqrt d), Linv = diag(1/sqrt d) X.
// Bound: FP64 issue of one SM (a warp's DFMA holds its sub-partition for 77 clocks).  With the scaling in every
// thread (two DMULs an entry more) and X in a loop of its own a block took 42 us, now 31.
constexpr int NB = 32;
struct DiagBlock {
    double2 S[NB][NB + 1], X[NB][NB + 1];
    double2 C[2][NB];  // the scaled column of pivot j, L~_ij, at [j & 1][i]
    double dv[NB], rdv[NB], qv[NB];
    unsigned short ent[NB * (NB - 1) / 2];
};

__device__ void factor_block(DiagBlock &m, int n, double2 *A, int lda, double2 *Linv, int pivot0, uint32_t *err)
{
    const int tid = threadIdx.x;
    for (int t = tid; t < NB * NB; t += 256) {
        const int i = t >> 5, l = t & 31;
        m.X[i][l] = make_double2(i == l && i < n ? 1.0 : 0.0, 0.0);
        if (l >= 1 && l <= i)  // position of (i, l): all entries of the columns right of l come first
            m.ent[(31 - l) * (32 - l) / 2 + (i - l)] = (unsigned short)((i << 8) | l);
    }
    // pivot l, of which lane 0 of warp 0 has the entry v and lane q that of row l + q: its reciprocal, scaled column
    auto pivot = [&](int l, double2 v) {
        double r = 0.0;
        if (tid == 0) {
            const bool ok = v.x > 0.0 && isfinite(v.x);
            if (!ok)
                record_error(err, GW_E_NUMERIC, SITE_CHOL_PIVOT, (uint32_t)(pivot0 + l));
            m.dv[l] = ok ? v.x : 1.0;
            r = ok ? rcp_newton(v.x) : 1.0;
            m.rdv[l] = r;
        }
        r = __shfl_sync(0xffffffffu, r, 0);
        if (tid > 0 && l + tid < NB)
            m.C[l & 1][l + tid] = make_double2(v.x * r, v.y * r);
    };
    __syncthreads();
    if (tid < 32 && n > 0)
        pivot(0, m.S[tid][0]);
    __syncthreads();
    for (int j = 0; j + 1 < n; ++j) {
        const double2 *c = m.C[j & 1];
        if (tid < 32) {
            const int i = j + 1 + tid;
            double2 v = make_double2(0.0, 0.0);
            if (i < NB) {
                const double2 a = c[i], b = m.S[j + 1][j];
                v = m.S[i][j + 1];
                v.x = fma(-a.x, b.x, fma(-a.y, b.y, v.x));
                v.y = fma(-a.y, b.x, fma(a.x, b.y, v.y));
                m.S[i][j + 1] = v;
            }
            pivot(j + 1, v);
        } else {
            const int cs = (30 - j) * (31 - j) / 2, cx = (31 - j) * (j + 1);  // columns right of the next pivot's; X
            const float inv = 1.f / (float)(j + 1);
            for (int p = tid - 32; p < cs + cx; p += 224) {
                if (p < cs) {
                    const int e = m.ent[p], i = e >> 8, l = e & 255;
                    const double2 a = c[i], b = m.S[l][j];
                    double2 v = m.S[i][l];
                    v.x = fma(-a.x, b.x, fma(-a.y, b.y, v.x));
                    v.y = fma(-a.y, b.x, fma(a.x, b.y, v.y));
                    m.S[i][l] = v;
                } else {
                    const int q = (int)(((float)(p - cs) + 0.5f) * inv), i = j + 1 + q, x = p - cs - q * (j + 1);
                    const double2 a = c[i], b = m.X[j][x];
                    double2 v = m.X[i][x];
                    v.x = fma(-a.x, b.x, fma(a.y, b.y, v.x));
                    v.y = fma(-a.x, b.y, fma(-a.y, b.x, v.y));
                    m.X[i][x] = v;
                }
            }
        }
        __syncthreads();
    }
    if (tid < n)
        m.qv[tid] = rsqrt_newton(m.dv[tid]);
    __syncthreads();
    for (int t = tid; t < n * n; t += 256) {
        const int i = t / n, j = t % n;
        double2 l = make_double2(0.0, 0.0), x = make_double2(0.0, 0.0);
        if (j < i) {
            const double r = m.rdv[j], sq = m.dv[j] * m.qv[j];
            l = make_double2(m.S[i][j].x * r * sq, m.S[i][j].y * r * sq);
        } else if (j == i) {
            l = make_double2(m.dv[j] * m.qv[j], 0.0);
        }
        if (j <= i)
            x = make_double2(m.X[i][j].x * m.qv[i], m.X[i][j].y * m.qv[i]);
        A[(size_t)i * lda + j] = l;
        Linv[i * NB + j] = x;
    }
}

__global__ void __launch_bounds__(256)
    chol_first_kernel(double2 *__restrict__ A, int lda, int n, double2 *__restrict__ Linv, uint32_t *err)
{
    __shared__ DiagBlock m;
    for (int t = threadIdx.x; t < NB * NB; t += 256) {
        const int i = t >> 5, l = t & 31;
        m.S[i][l] = (i < n && l <= i) ? A[(size_t)i * lda + l] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    factor_block(m, n, A, lda, Linv, 0, err);
}

// W = panel Linv^H (rest x 32) of the panel below a factored 32 x 32 block; 8 x 16 tiles, a warp per sub-partition.
__global__ void __launch_bounds__(128) chol_panel_kernel(const double2 *__restrict__ panel, int lda, int rest,
                                                         const double2 *__restrict__ Linv, double2 *__restrict__ W)
{
    __shared__ double2 Ps[NB][9], Ls[NB][17];
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, j0 = blockIdx.x * 16, i0 = blockIdx.y * 8;
    const int kend = j0 + 16;  // Linv is lower triangular
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int i = (tid >> 5) + 4 * e, k = tid & 31;
        Ps[k][i] = i0 + i < rest ? panel[(size_t)(i0 + i) * lda + k] : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int j = (tid >> 5) + 4 * e, k = tid & 31;
        Ls[k][j] = cconj(Linv[(j0 + j) * NB + k]);
    }
    __syncthreads();
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int k = 0; k < kend; ++k) {
        const double2 a = Ps[k][ty], b = Ls[k][tx];
        acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
        acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
    }
    if (i0 + ty < rest)
        W[(size_t)(i0 + ty) * NB + j0 + tx] = acc;
}

// The trailing update A -= W W^H (lower triangle) of a step, W also copied to its place in the panel, and the
// factorisation of the next diagonal block beside it.  CTAs 0..7 update four rows each of that block, and the one
// that finishes last factors it (no CTA waits for another), while the rest of the grid works on the other 16 x 16
// tiles.  The dynamic shared memory keeps the CTAs one per SM, so that one has its SM's FP64 units for itself.  As a
// launch per diagonal block, panel product, copy and update, a step at N = 515 took 42 + 13 + 3 + 12..48 us,
// now 8 + 40 (every step: 9 us of update and hand-over, 31 of factorisation).
constexpr int TRAIL_SMEM = 120 * 1024, TRAIL_HELPERS = 8;

__global__ void __launch_bounds__(256, 1)
    chol_trail_kernel(double2 *A, int lda, double2 *panel, const double2 *__restrict__ W, int rest, double2 *Linv,
                      int pivot0, unsigned *arrived, uint32_t *err)
{
    extern __shared__ __align__(16) uint8_t trail_smem[];
    const int tid = threadIdx.x, bid = blockIdx.x;
    if (bid < TRAIL_HELPERS) {
        const int n = min(NB, rest), r0 = 4 * bid;
        double2(*Ws)[NB + 1] = reinterpret_cast<double2(*)[NB + 1]>(trail_smem);
        for (int t = tid; t < NB * NB; t += 256) {
            const int i = t >> 5, k = t & 31;
            Ws[i][k] = i < n ? W[i * NB + k] : make_double2(0.0, 0.0);
        }
        __syncthreads();
        const int i = r0 + ((tid & 127) >> 5), l = tid & 31;
        if (i < n) {
            if (tid < 128) {
                if (l <= i) {
                    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 8
                    for (int k = 0; k < NB; ++k) {
                        const double2 a = Ws[i][k], b = cconj(Ws[l][k]);
                        acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
                        acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
                    }
                    double2 v = A[(size_t)i * lda + l];
                    v.x -= acc.x;
                    v.y -= acc.y;
                    A[(size_t)i * lda + l] = v;
                }
            } else {
                panel[(size_t)i * lda + l] = Ws[i][l];
            }
        }
        __shared__ int last;
        __threadfence();
        __syncthreads();  // every row of this CTA is written before it is counted
        if (tid == 0)
            last = atomicAdd(arrived, 1u) == TRAIL_HELPERS - 1;
        __syncthreads();
        if (!last)
            return;
        __threadfence();  // the other CTAs' rows, counted before this one
        DiagBlock &m = *reinterpret_cast<DiagBlock *>(trail_smem);
        for (int t = tid; t < NB * NB; t += 256) {
            const int ii = t >> 5, ll = t & 31;
            m.S[ii][ll] = (ii < n && ll <= ii) ? __ldcg(&A[(size_t)ii * lda + ll]) : make_double2(0.0, 0.0);
        }
        __syncthreads();
        factor_block(m, n, A, lda, Linv, pivot0, err);
        return;
    }
    // tile (ti, tj), tj <= ti, of the rows from 32 on: the lower triangle's tiles after the first three
    const int u = bid - TRAIL_HELPERS + 3;
    int ti = (int)((sqrtf(8.f * u + 1.f) - 1.f) * 0.5f);
    while (ti * (ti + 1) / 2 > u)
        --ti;
    while ((ti + 1) * (ti + 2) / 2 <= u)
        ++ti;
    const int tj = u - ti * (ti + 1) / 2, i0 = ti * ZT, j0 = tj * ZT, ty = tid >> 4, tx = tid & 15;
    double2(*Wi)[ZT + 1] = reinterpret_cast<double2(*)[ZT + 1]>(trail_smem);
    double2(*Wj)[ZT + 1] = Wi + NB;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int i = (tid >> 5) + 8 * e, k = tid & 31;
        const double2 x = i0 + i < rest ? W[(size_t)(i0 + i) * NB + k] : make_double2(0.0, 0.0);
        Wi[k][i] = x;
        if (tj == 0 && i0 + i < rest)
            panel[(size_t)(i0 + i) * lda + k] = x;
        Wj[k][i] = j0 + i < rest ? cconj(W[(size_t)(j0 + i) * NB + k]) : make_double2(0.0, 0.0);
    }
    __syncthreads();
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int k = 0; k < NB; ++k) {
        const double2 a = Wi[k][ty], b = Wj[k][tx];
        acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
        acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
    }
    const int gi = i0 + ty, gj = j0 + tx;
    if (gi < rest && gj <= gi) {  // the lower triangle is all that is read later
        double2 v = A[(size_t)gi * lda + gj];
        v.x -= acc.x;
        v.y -= acc.y;
        A[(size_t)gi * lda + gj] = v;
    }
}

__global__ void set_identity_kernel(double2 *A, int lda, int n, double scale)
{
    const size_t tot = (size_t)n * n;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < tot; t += (size_t)gridDim.x * blockDim.x) {
        const int i = static_cast<int>(t / n), j = static_cast<int>(t - (size_t)i * n);
        A[(size_t)i * lda + j] = make_double2(i == j ? scale : 0.0, 0.0);
    }
}

__global__ void two_minus_kernel(double2 *T, int n)
{
    const size_t tot = (size_t)n * n;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < tot; t += (size_t)gridDim.x * blockDim.x) {
        const int i = static_cast<int>(t / n), j = static_cast<int>(t - (size_t)i * n);
        double2 v = T[t];
        T[t] = make_double2((i == j ? 2.0 : 0.0) - v.x, -v.y);
    }
}

// X = A^H / den
__global__ void scaled_adjoint_kernel(const double2 *__restrict__ A, int n, const double *__restrict__ den,
                                      double2 *__restrict__ X)
{
    const double s = 1.0 / *den;
    const size_t tot = (size_t)n * n;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < tot; t += (size_t)gridDim.x * blockDim.x) {
        const int i = static_cast<int>(t / n), j = static_cast<int>(t - (size_t)i * n);
        const double2 a = A[(size_t)j * n + i];
        X[t] = make_double2(a.x * s, -a.y * s);
    }
}

// Single-CTA reductions (the matrices are at most a few thousand squared).
__global__ void max_absdiff_kernel(const double2 *__restrict__ A, const double2 *__restrict__ B, size_t n,
                                   double *out)
{
    __shared__ double red[256];
    double m = 0.0;
    for (size_t t = threadIdx.x; t < n; t += blockDim.x) {
        const double dx = A[t].x - B[t].x, dy = A[t].y - B[t].y;
        const double d = sqrt(dx * dx + dy * dy);
        m = d > m || d != d ? d : m;
    }
    red[threadIdx.x] = m;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            const double o = red[threadIdx.x + s];
            red[threadIdx.x] = o > red[threadIdx.x] || o != o ? o : red[threadIdx.x];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0)
        *out = red[0];
}

__global__ void row_abs_sum_max_kernel(const double2 *__restrict__ A, int n, double *out)
{
    __shared__ double red[256];
    double m = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double s = 0.0;
        for (int j = 0; j < n; ++j) {
            const double2 a = A[(size_t)i * n + j];
            s += sqrt(a.x * a.x + a.y * a.y);
        }
        m = s > m ? s : m;
    }
    red[threadIdx.x] = m;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            red[threadIdx.x] = red[threadIdx.x + s] > red[threadIdx.x] ? red[threadIdx.x + s] : red[threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        *out = red[0];
}

// The nblk inverses of the 32x32 diagonal blocks (Dinv, leading dimension 32) onto the diagonal of
// Y (leading dimension N); blockIdx.x = block.
__global__ void scatter_diag_blocks_kernel(const double2 *__restrict__ Dinv, int N, double2 *__restrict__ Y)
{
    const int b = blockIdx.x, n0 = 32 * b, nb = min(32, N - n0);
    for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
        const int i = t / nb, j = t % nb;
        Y[(size_t)(n0 + i) * N + n0 + j] = Dinv[(size_t)b * 32 * 32 + i * 32 + j];
    }
}

int grid_for(size_t n)
{
    size_t g = (n + 255) / 256;
    if (g > 152 * 8)
        g = 152 * 8;
    return g < 1 ? 1 : static_cast<int>(g);
}

}  // namespace

cudaError_t launch_eps_build(const float2 *PG, const double *sv, int ng, double2 *eps, cudaStream_t s)
{
    eps_build_kernel<<<grid_for((size_t)ng * ng), 256, 0, s>>>(PG, sv, ng, eps);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_zgemm(int M, int N, int K, double2 alpha, const double2 *A, int lda, int opA, const double2 *B,
                         int ldb, int opB, double2 beta, double2 *C, int ldc, cudaStream_t s)
{
    return launch_zgemm_batched(M, N, K, alpha, A, lda, opA, 0, B, ldb, opB, 0, beta, C, ldc, 0, 1, s);
}

cudaError_t launch_set_identity(double2 *A, int lda, int n, double scale, cudaStream_t s)
{
    set_identity_kernel<<<grid_for((size_t)n * n), 256, 0, s>>>(A, lda, n, scale);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_two_minus(double2 *T, int n, cudaStream_t s)
{
    two_minus_kernel<<<grid_for((size_t)n * n), 256, 0, s>>>(T, n);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_scaled_adjoint(const double2 *A, int n, const double *d_den, double2 *X, cudaStream_t s)
{
    scaled_adjoint_kernel<<<grid_for((size_t)n * n), 256, 0, s>>>(A, n, d_den, X);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_max_absdiff(const double2 *A, const double2 *B, size_t n, double *out, cudaStream_t s)
{
    max_absdiff_kernel<<<1, 256, 0, s>>>(A, B, n, out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_row_abs_sum_max(const double2 *A, int n, double *out, cudaStream_t s)
{
    row_abs_sum_max_kernel<<<1, 256, 0, s>>>(A, n, out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_zgemm_batched(int M, int N, int K, double2 alpha, const double2 *A, int lda, int opA, long sA,
                                 const double2 *B, int ldb, int opB, long sB, double2 beta, double2 *C, int ldc,
                                 long sC, int batch, cudaStream_t s)
{
    if (M <= 0 || N <= 0 || batch <= 0)
        return cudaSuccess;
    dim3 grid((N + ZT - 1) / ZT, (M + ZT - 1) / ZT, batch);
    zgemm_kernel<<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, opA, B, ldb, opB, beta, C, ldc, sA, sB, sC);
    count_launches(1);
    return cudaGetLastError();
}

template <int KIND>
static cudaError_t launch_ztri(int M, int N, int K, double sign, const double2 *A, int lda, long sA, const double2 *B,
                               int ldb, long sB, double2 *C, int ldc, long sC, int batch, cudaStream_t s)
{
    const int nti = (M + TM - 1) / TM, np = nti / 2;
    const long ntiles =
        KIND == TRI_GRAM ? (long)(np + (nti & 1)) * (np + 1) : (long)nti * ((N + TN - 1) / TN) * batch;
    ztri_kernel<KIND><<<(int)std::min(ntiles, 152L), TTHREADS, 0, s>>>(M, N, K, sign, A, lda, sA, B, ldb, sB, C, ldc,
                                                                       sC, batch);
    count_launches(1);
    return cudaGetLastError();
}

// eps^-1 of a Hermitian positive-definite N x N complex128 matrix, in FP64 (Sec. 5.1 asks for the
// inverse; the factorisation route is this library's):
//  1. blocked right-looking Cholesky eps = L L^H with 32-wide panels; the first diagonal block is
//     factored and inverted by itself, then each step is two launches: the panel below the block as a product
//     with its inverse, and the rank-32 update of the trailing lower triangle with the next block's factorisation;
//  2. Y = L^-1 by recursive doubling: with the inverted blocks of size b on the diagonal of Y,
//     each pair of neighbours becomes one block of size 2b through
//     [L11 0; L21 L22]^-1 = [Y11 0; -Y22 L21 Y11  Y22],
//     and all pairs of one size go in one batched product (a trailing pair with a short second
//     block in one more);
//  3. eps^-1 = Y^H Y, lower half computed and mirrored.
// Workspace: A, Y, T (N^2 each), W (N x 32), Dinv (ceil(N/32) x 32 x 32).  Status words for a
// non-positive pivot go to err.  T also holds the steps' arrival counters (4 bytes each) while 1. runs.
cudaError_t chol_inverse_enqueue(const double2 *eps, int N, double2 *epsinv, double2 *A, double2 *Y, double2 *T,
                                 double2 *W, double2 *Dinv, uint32_t *err, cudaStream_t s)
{
    const int nblk = (N + NB - 1) / NB;
    cudaError_t e;
#define ENQ(x)                         \
    do {                               \
        if ((e = (x)) != cudaSuccess)  \
            return e;                  \
    } while (0)
    ENQ(cudaMemcpyAsync(A, eps, (size_t)N * N * sizeof(double2), cudaMemcpyDeviceToDevice, s));
    unsigned *arrived = reinterpret_cast<unsigned *>(T);
    ENQ(cudaMemsetAsync(arrived, 0, nblk * sizeof(unsigned), s));
    ENQ(cudaFuncSetAttribute(chol_trail_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TRAIL_SMEM));
    chol_first_kernel<<<1, 256, 0, s>>>(A, N, std::min(NB, N), Dinv, err);
    count_launches(1);
    for (int kb = 0; kb + 1 < nblk; ++kb) {
        const int k0 = kb * NB, n0 = k0 + NB, rest = N - n0, nt = (rest + ZT - 1) / ZT;
        double2 *panel = A + (size_t)n0 * N + k0;
        const dim3 pgrid(2, (rest + 7) / 8);
        chol_panel_kernel<<<pgrid, 128, 0, s>>>(panel, N, rest, Dinv + (size_t)kb * NB * NB, W);
        const int tiles = nt > 2 ? nt * (nt + 1) / 2 - 3 : 0;
        chol_trail_kernel<<<TRAIL_HELPERS + tiles, 256, TRAIL_SMEM, s>>>(
            A + (size_t)n0 * N + n0, N, panel, W, rest, Dinv + (size_t)(kb + 1) * NB * NB, n0, arrived + kb, err);
        count_launches(2);
    }
    ENQ(cudaMemsetAsync(Y, 0, (size_t)N * N * sizeof(double2), s));
    scatter_diag_blocks_kernel<<<nblk, 256, 0, s>>>(Dinv, N, Y);
    count_launches(1);
    ENQ(cudaGetLastError());
    const long diag = (long)N + 1;
    for (int b = NB; b < N; b *= 2) {
        const int F = N / (2 * b);  // pairs of two full blocks
        if (F > 0) {
            // T_p = L21 Y11, then Y21 = -Y22 T_p, for the pairs starting at 2 p b
            ENQ(launch_ztri<TRI_RIGHT>(b, b, b, 1.0, A + (size_t)b * N, N, 2 * b * diag, Y, N, 2 * b * diag, T, b,
                                       (long)b * b, F, s));
            ENQ(launch_ztri<TRI_LEFT>(b, b, b, -1.0, Y + (size_t)b * diag, N, 2 * b * diag, T, b, (long)b * b,
                                      Y + (size_t)b * N, N, 2 * b * diag, F, s));
        }
        const int n0 = 2 * b * F, n2 = N - n0 - b;  // a last pair with a short second block
        if (n2 > 0) {
            ENQ(launch_ztri<TRI_RIGHT>(n2, b, b, 1.0, A + (size_t)(n0 + b) * N + n0, N, 0, Y + (size_t)n0 * diag, N, 0,
                                       T, b, 0, 1, s));
            ENQ(launch_ztri<TRI_LEFT>(n2, b, n2, -1.0, Y + (size_t)(n0 + b) * diag, N, 0, T, b, 0,
                                      Y + (size_t)(n0 + b) * N + n0, N, 0, 1, s));
        }
    }
    // (Y^H Y)[i][j] = sum_{k >= max(i, j)} conj(Y[k][i]) Y[k][j]; Hermitian, so the lower half is
    // computed and mirrored
    ENQ(launch_ztri<TRI_GRAM>(N, N, N, 1.0, Y, N, 0, Y, N, 0, epsinv, N, 0, 1, s));
#undef ENQ
    return cudaSuccess;
}

}  // namespace gw
