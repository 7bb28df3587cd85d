// Complex GEMM C = A B on the 16-bit tensor cores from sliced FP64 operands (gw_zgemm_tc).
//
// FP64 runs at about 1 TFLOP/s on this GPU and FP16 tensor MMAs at about 2 PFLOP/s.  Two splits:
//  * FP16X3 (22 significant bits): hi*hi + hi*lo + lo*hi accumulated in FP32;
//  * integer slices, to FP64 accuracy (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
//    Algorithms 59, 2012): every entry scaled into [-1, 1] is a sum of slices a_t 2^(-6(t+1))
//    with integer a_0 in [-64, 64] and a_t in [-32, 32] (t >= 1); nine slices keep 54 bits.  The
//    slice products a_t b_u are exact in FP16 and their sums over one work slot stay below 2^24,
//    so the FP32 tensor-core accumulation is exact; the slots are shifted and added in 128-bit integers.
//
// Operand planes (K-major, 8-row x 16-byte core matrices, as in the rank-k update): element
// (r, k) of plane p sits at 16-bit offset ((kc Rpad/128 + r/128) NP + p) 2048 + ((r%128)/8) 128 +
// ((k%16)/8) 64 + (r%8) 8 + k%8 with kc = k / 16: the NP planes of one chunk of one 128-row block
// are contiguous, so a stage arrives in one bulk copy per operand (large copies reach a higher
// per-SM ingress than 4 KB ones).  A operand (row i of A, k along the row): planes 2t (Re) and
// 2t + 1 (Im) of slice t.  B operand (row j = column j of B, k down the column): planes 2t (Re)
// and 2t + 1 (Im), so the 256 rows starting at Re are [Re; Im].  Then one M = 128, N = 256 MMA with
// A = Re(A) adds Re A Re B into the Re columns of the accumulator and Re A Im B into its Im
// columns, and two N = 128 MMAs with A = Im(A) add -Im A Im B (the A-negate bit of the instruction
// descriptor) into the Re columns and Im A Re B into the Im columns: C = A B with the tensor work of
// two N = 256 MMAs per slice pair and 16-wide chunk, and no negated plane in memory.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "gw_internal.cuh"
#include "ptx.cuh"

namespace gw {

namespace {

constexpr int ZT = 128;
constexpr uint32_t ZPL = ZT * 16 * 2;       // 4 KB: one plane of one 128-row block, one chunk
// A stage is one chunk of one slice pair (A Re, A Im, B Re, B Im: 16 KB, three MMAs) for the
// integer slices, and one chunk of all three FP16X3 pairs (A hi Re, Im, A lo Re, Im, B hi Re, Im,
// B lo Re, Im: 32 KB, nine MMAs, one commit) for the split, where each slice then loads once per
// chunk.
constexpr uint32_t ZSTAGE = 4 * ZPL;
constexpr int ZSTAGES = 6;                  // twelve stages in flight per SM cover the copy latency
constexpr uint32_t ZPIPE = ZSTAGES * ZSTAGE;  // 96 KB: two CTAs per SM
constexpr uint32_t ZSTAGE3 = 8 * ZPL;
constexpr int ZSTAGES3 = 3;
static_assert(ZSTAGES3 * ZSTAGE3 <= ZPIPE, "the fused stages share the pipeline buffers");
static_assert(128 * 65 * 8 <= ZPIPE, "epilogue staging must fit in the pipeline buffers");
constexpr size_t ZSMEM = ZPIPE + 128;
constexpr int ZTHREADS = 192;               // warp 0 copies, warp 1 MMAs, warps 2..5 epilogue
constexpr uint32_t LBO = 128, SBO = 256;
constexpr uint64_t DRAIN_NS = 2000000000ull;

constexpr int MODE_FP16X3 = 0, MODE_SLICES = 1;
constexpr int OZ_SLICES = 9;

// Scale exponent e of a matrix from the bits of max(|Re|, |Im|): m (1 + 2^-20) < 2^e, so a max
// taken in FP32 (relative error 2^-24) still bounds every entry (0 for an all-zero or non-finite
// matrix).
__device__ __forceinline__ int exp_of(const unsigned long long *w)
{
    const double m = __longlong_as_double((long long)*w);
    if (!(m > 0.0) || !isfinite(m))
        return 0;
    int e;
    frexp(m * (1.0 + 0x1p-20), &e);
    return e;
}

__device__ __forceinline__ void named_bar_sync(int id, int n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Named barrier over n threads that also ORs a predicate, so the participants agree on it.
__device__ __forceinline__ bool named_bar_or(int id, int n, bool pred)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"(pred ? 1u : 0u), "r"(id), "r"(n)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ uint16_t h16(float x)
{
    __half h = __float2half_rn(x);
    return *reinterpret_cast<uint16_t *>(&h);
}

// max(|Re|, |Im|) over a rows x cols complex128 matrix into *w (as the bits of a non-negative
// double, which order like unsigned integers).  *w must be zero (or smaller) beforehand.
__global__ void zmaxabs_kernel(const double2 *__restrict__ M, int rows, int cols, long ld, unsigned long long *w)
{
    __shared__ double red[32];
    double best = 0.0;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    for (int r = blockIdx.y; r < rows && c < cols; r += gridDim.y) {
        const double2 z = M[(size_t)r * ld + c];
        best = fmax(best, fmax(fabs(z.x), fabs(z.y)));
    }
    for (int o = 16; o > 0; o >>= 1)
        best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i)
            best = fmax(best, red[i]);
        atomicMax(w, (unsigned long long)__double_as_longlong(best));
    }
}

// Slice a complex128 matrix into operand planes (layouts above).  One block per (16-wide chunk
// kc, 128-row block rb of the operand): the 16 x 128 tile goes through shared memory, so both
// orientations read contiguous runs of M and every plane is written in 4 KB runs.  transpose = 0:
// operand row r is row r of M (A operand, element (r, k) = M[r][k]); transpose = 1: operand row r
// is column r of M (B operand, element (r, k) = M[k][r]).  npl = 2 planes (Re, Im) per slice for
// either operand.  Entries outside rows x K are zero.
//   FP16X3: y = float(x) 2^(14 - e), hi = rn16(y), lo = rn16(y - hi).
//   slices: n = rint(x 2^(6 ns - e)) (|n| <= 2^(6 ns)) written in balanced base 64,
//           n = sum_t a_t 2^(6 (ns - 1 - t)): a_(ns-1) .. a_1 in [-32, 31] from the low end, a_0 =
//           the rest, |a_0| <= 64; so x 2^-e = sum_t a_t 2^(-6 (t + 1)) up to 2^(-6 ns - 1).
__global__ void __launch_bounds__(512) zslice_kernel(const double2 *__restrict__ M, long ld, int rows, int K,
                                                     int transpose, int Rpad, int mode, int ns, int npl,
                                                     const unsigned long long *maxw, uint16_t *__restrict__ planes)
{
    __shared__ double2 tile[16][129];
    const int kc = blockIdx.x, rb = blockIdx.y;
    const int k0 = kc * 16, r0 = rb * 128;
    const double2 zero = make_double2(0.0, 0.0);
    if (transpose) {
        for (int q = threadIdx.x; q < 2048; q += blockDim.x) {
            const int kk = q >> 7, rr = q & 127, r = r0 + rr, k = k0 + kk;
            tile[kk][rr] = (r < rows && k < K) ? M[(size_t)k * ld + r] : zero;
        }
    } else {
        for (int q = threadIdx.x; q < 2048; q += blockDim.x) {
            const int rr = q >> 4, kk = q & 15, r = r0 + rr, k = k0 + kk;
            tile[kk][rr] = (r < rows && k < K) ? M[(size_t)r * ld + k] : zero;
        }
    }
    // the scales once per block: FP64 work per thread would rival the slicing itself here
    __shared__ float s_scf;
    __shared__ double s_scd;
    if (threadIdx.x == 0) {
        const int e = exp_of(maxw);
        s_scf = ldexpf(1.0f, 14 - e);
        s_scd = ldexp(1.0, 6 * ns - e);
    }
    __syncthreads();
    const int NP = ns * npl;
    constexpr size_t per = 2048;  // consecutive planes of one block and chunk
    uint16_t *base0 = planes + ((size_t)kc * (Rpad / ZT) + rb) * NP * per;
    const float scf = s_scf;
    const double scd = s_scd;
    for (int rem = threadIdx.x; rem < 2048; rem += blockDim.x) {
        const int rr = (rem >> 7) * 8 + ((rem & 63) >> 3);
        const int kk = ((rem & 127) >> 6) * 8 + (rem & 7);
        const double2 z = tile[kk][rr];
        uint16_t *b = base0 + rem;
        if (mode == MODE_FP16X3) {
            const float yr = (float)z.x * scf, yi = (float)z.y * scf;
            const uint16_t rh = h16(yr), ih = h16(yi);
            const uint16_t rl = h16(yr - __half2float(*reinterpret_cast<const __half *>(&rh)));
            const uint16_t il = h16(yi - __half2float(*reinterpret_cast<const __half *>(&ih)));
            const uint16_t re[2] = {rh, rl}, im[2] = {ih, il};
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                b[(size_t)(2 * t) * per] = re[t];
                b[(size_t)(2 * t + 1) * per] = im[t];
            }
        } else {
            long long nr = __double2ll_rn(z.x * scd), ni = __double2ll_rn(z.y * scd);
            for (int t = ns - 1; t >= 0; --t) {
                long long ar, ai;
                if (t > 0) {
                    ar = ((nr + 32) & 63) - 32;
                    ai = ((ni + 32) & 63) - 32;
                    nr = (nr - ar) >> 6;  // exact: nr - ar is a multiple of 64
                    ni = (ni - ai) >> 6;
                } else {
                    ar = nr;
                    ai = ni;
                }
                const uint16_t hr = h16((float)ar), hi = h16((float)ai);  // |a| <= 64: exact
                b[(size_t)(2 * t) * per] = hr;
                b[(size_t)(2 * t + 1) * per] = hi;
            }
        }
    }
}

// One work slot of the sliced product: slice pairs [p0, p1) of the pair list over chunks
// [kc0, kc1); the slot's result is one FP32 complex tile per output tile, T[slot][Mpad][Npad].
struct ZSlot {
    int p0, p1, kc0, kc1;
};

template <bool F3>  // true: FP16X3 slots, one stage per chunk with the pairs (0,0), (0,1), (1,0)
__global__ void __launch_bounds__(ZTHREADS, 2)
    zgemm16_kernel(const uint16_t *__restrict__ Ap, int npA, int Mpad, const uint16_t *__restrict__ Bp, int npB,
                   int Npad, const int2 *__restrict__ pairs, const ZSlot *__restrict__ slots, int ntj,
                   float2 *__restrict__ T, uint32_t *err, uint64_t wait_ns)
{
    constexpr uint32_t SB = F3 ? ZSTAGE3 : ZSTAGE;
    constexpr int NST = F3 ? ZSTAGES3 : ZSTAGES;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + ZPIPE);
    uint64_t *empty = full + NST;
    uint64_t *done = empty + NST;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *n_issued = abort_flag + 1;
    volatile int *n_consumed = abort_flag + 2;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ti = blockIdx.x / ntj, tj = blockIdx.x - (blockIdx.x / ntj) * ntj;
    const ZSlot sl = slots[blockIdx.y];
    const int np = sl.p1 - sl.p0;
    const int nunits = F3 ? sl.kc1 - sl.kc0 : np * (sl.kc1 - sl.kc0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        *n_issued = 0;
        *n_consumed = 0;
        fence_barrier_init();
    }
    if (warp == 1)
        tmem_alloc(tmem_slot, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            const int ntA = Mpad / ZT, ntB = Npad / ZT;  // 128-row blocks of each operand
            for (int u = 0; u < nunits; ++u) {
                const int s = u % NST;
                const uint32_t ph = (uint32_t)(u / NST) & 1u;
                if (u >= NST && !mbar_wait(&empty[s], ph ^ 1u, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                    *abort_flag = 1;
                    break;
                }
                if (*abort_flag)
                    break;
                uint8_t *st = smem + s * SB;
                mbar_arrive_expect_tx(&full[s], SB);
                if (F3) {  // A planes 0..3 (hi Re, hi Im, lo Re, lo Im), B planes 0..5 (hi, lo regions)
                    const int kc = sl.kc0 + u;
                    bulk_g2s(st, Ap + ((size_t)kc * ntA + ti) * npA * 2048, 4 * ZPL, &full[s]);
                    bulk_g2s(st + 4 * ZPL, Bp + ((size_t)kc * ntB + tj) * npB * 2048, 4 * ZPL, &full[s]);
                } else {
                    const int kc = sl.kc0 + u / np;  // chunk-major: every pair of a chunk in turn
                    const int2 pr = pairs[sl.p0 + u % np];
                    bulk_g2s(st, Ap + (((size_t)kc * ntA + ti) * npA + 2 * pr.x) * 2048, 2 * ZPL, &full[s]);
                    bulk_g2s(st + 2 * ZPL, Bp + (((size_t)kc * ntB + tj) * npB + 2 * pr.y) * 2048, 2 * ZPL,
                             &full[s]);
                }
                *n_issued = u + 1;
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t ID = mma_idesc(0u, ZT, 2 * ZT, false);  // FP16, N = 256: Re | Im
            constexpr uint32_t ID1 = mma_idesc(0u, ZT, ZT, false), ID1N = mma_idesc(0u, ZT, ZT, true);
            const uint32_t sbase = smem_u32(smem);
            for (int u = 0; u < nunits; ++u) {
                const int s = u % NST;
                if (!mbar_wait(&full[s], (uint32_t)(u / NST) & 1u, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t st = sbase + s * SB;
                // Re columns at tmem, Im columns at tmem + ZT
                if (F3) {
                    const uint64_t ahr = smem_desc(st, LBO, SBO), ahi = smem_desc(st + ZPL, LBO, SBO);
                    const uint64_t alr = smem_desc(st + 2 * ZPL, LBO, SBO), ali = smem_desc(st + 3 * ZPL, LBO, SBO);
                    const uint64_t bh_re = smem_desc(st + 4 * ZPL, LBO, SBO), bh_im = smem_desc(st + 5 * ZPL, LBO, SBO);
                    const uint64_t bl_re = smem_desc(st + 6 * ZPL, LBO, SBO), bl_im = smem_desc(st + 7 * ZPL, LBO, SBO);
                    mma_f16(tmem, ahr, bh_re, ID, u > 0 ? 1u : 0u);  // hi * hi
                    mma_f16(tmem, ahi, bh_im, ID1N, 1u);
                    mma_f16(tmem + ZT, ahi, bh_re, ID1, 1u);
                    mma_f16(tmem, ahr, bl_re, ID, 1u);               // hi * lo
                    mma_f16(tmem, ahi, bl_im, ID1N, 1u);
                    mma_f16(tmem + ZT, ahi, bl_re, ID1, 1u);
                    mma_f16(tmem, alr, bh_re, ID, 1u);               // lo * hi
                    mma_f16(tmem, ali, bh_im, ID1N, 1u);
                    mma_f16(tmem + ZT, ali, bh_re, ID1, 1u);
                } else {
                    const uint64_t a_re = smem_desc(st, LBO, SBO), a_im = smem_desc(st + ZPL, LBO, SBO);
                    const uint64_t b_re = smem_desc(st + 2 * ZPL, LBO, SBO);   // rows [Re B; Im B]
                    const uint64_t b_im = smem_desc(st + 3 * ZPL, LBO, SBO);
                    mma_f16(tmem, a_re, b_re, ID, u > 0 ? 1u : 0u);
                    mma_f16(tmem, a_im, b_im, ID1N, 1u);               // -Im A Im B into Re
                    mma_f16(tmem + ZT, a_im, b_re, ID1, 1u);           // Im A Re B into Im
                }
                mma_commit(&empty[s]);
                *n_consumed = u + 1;
            }
            mma_commit(done);  // arrives once every MMA issued above has completed
        }
        __syncwarp();
    } else {
        // epilogue warps 2..5: TMEM lane quarter warp % 4, one output row per thread
        const int q = warp & 3;
        const int row = q * 32 + lane;
        const bool waited = __all_sync(0xffffffffu, mbar_wait(done, 0, wait_ns));
        if (!waited) {
            if (lane == 0)
                record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
            *abort_flag = 1;
        }
        // one decision for the four epilogue warps (the staging below has barriers among them)
        if (!named_bar_or(1, 128, !waited || *abort_flag != 0)) {
            // every copy has landed and every MMA has read it, so the pipeline buffers stage the
            // tile: two halves of 64 columns, each written back as 512-byte row runs
            tc_fence_after();
            const uint32_t base = tmem + ((uint32_t)(q * 32) << 16);
            float2 *stage = reinterpret_cast<float2 *>(smem);  // [128][65]
            const int et = threadIdx.x - 64;                   // 0..127 over the epilogue warps
            for (int h = 0; h < 2; ++h) {
#pragma unroll 1
                for (int c0 = 0; c0 < 64; c0 += 16) {
                    float re[16], im[16];
                    tmem_ld16x2(base + h * 64 + c0, base + ZT + h * 64 + c0, re, im);
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        stage[row * 65 + c0 + i] = make_float2(re[i], im[i]);
                }
                named_bar_sync(1, 128);
                float2 *out = T + ((size_t)blockIdx.y * Mpad + (size_t)ti * ZT) * Npad + (size_t)tj * ZT + h * 64;
                for (int rr = et >> 5; rr < ZT; rr += 4) {
                    const int c = (et & 31) * 2;
                    const float2 a = stage[rr * 65 + c], b2 = stage[rr * 65 + c + 1];
                    *reinterpret_cast<float4 *>(out + (size_t)rr * Npad + c) = make_float4(a.x, a.y, b2.x, b2.y);
                }
                named_bar_sync(1, 128);
            }
        }
        tc_fence_before();
    }

    // ---------------- drain before releasing TMEM and shared memory
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!mbar_wait(done, 0, DRAIN_NS))
            record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
        const int issued = *n_issued, consumed = *n_consumed;
        for (int u = consumed; u < issued; ++u)
            if (!mbar_wait(&full[u % NST], (uint32_t)(u / NST) & 1u, DRAIN_NS)) {
                record_error(err, GW_E_TIMEOUT, SITE_ZGEMM, blockIdx.x);
                break;
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 256);
    }
}

// FP16X3 products: out = 2^(eA + eB - 28) sum_slot T[slot], the K-range slots summed in FP32 (their own
// rounding is below the split's 2^-22).
__global__ void zcombine16_kernel(const float2 *__restrict__ T, int nslots, int Mpad, int Npad,
                                  const unsigned long long *wA, const unsigned long long *wB, int M, int N,
                                  double2 *__restrict__ out)
{
    __shared__ float s_sc;
    if (threadIdx.x == 0)
        s_sc = (float)ldexp(1.0, exp_of(wA) + exp_of(wB) - 28);
    __syncthreads();
    const float sc = s_sc;
    const size_t plane = (size_t)Mpad * Npad;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    for (int r = blockIdx.y; r < M && c < N; r += gridDim.y) {
        const float2 *t = T + (size_t)r * Npad + c;
        float sr = 0.f, si = 0.f;
        for (int s = 0; s < nslots; ++s) {
            const float2 v = t[s * plane];
            sr += v.x;
            si += v.y;
        }
        out[(size_t)r * N + c] = make_double2((double)(sr * sc), (double)(si * sc));
    }
}

// Exact 128-bit integer -> double (one rounding in each half; the halves do not cancel).
__device__ __forceinline__ double i128_to_double(__int128 a)
{
    const bool neg = a < 0;
    const unsigned __int128 u = neg ? (unsigned __int128)(-a) : (unsigned __int128)a;
    const unsigned long long hi = (unsigned long long)(u >> 64), lo = (unsigned long long)u;
    const double v = hi ? fma((double)hi, 18446744073709551616.0, (double)lo) : (double)lo;
    return neg ? -v : v;
}

// Integer-slice products: every slot tile is an exact integer below 2^24 with weight
// 2^(wexp - 60 + 60) = 2^(-6(d + 2)); sum_slot T 2^(wexp + 60) is added up exactly in 128-bit
// integers, so out = 2^(eA + eB - 60) (that sum) is rounded once.
__global__ void zcombine_int_kernel(const float2 *__restrict__ T, int nslots, const int *__restrict__ wexp, int Mpad,
                                    int Npad, const unsigned long long *wA, const unsigned long long *wB, int M, int N,
                                    double2 *__restrict__ out)
{
    __shared__ int shift[256];
    __shared__ double s_sc;
    for (int s = threadIdx.x; s < nslots && s < 256; s += blockDim.x)
        shift[s] = wexp[s] + 60;  // 6 (8 - d) in [0, 48]
    if (threadIdx.x == 0)
        s_sc = ldexp(1.0, exp_of(wA) + exp_of(wB) - 60);
    __syncthreads();
    const double sc = s_sc;
    const size_t plane = (size_t)Mpad * Npad;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    for (int r = blockIdx.y; r < M && c < N; r += gridDim.y) {
        const float2 *t = T + (size_t)r * Npad + c;
        __int128 ar = 0, ai = 0;
        for (int s = 0; s < nslots; ++s) {
            const float2 v = t[s * plane];
            ar += (__int128)__float2int_rn(v.x) << shift[s];
            ai += (__int128)__float2int_rn(v.y) << shift[s];
        }
        out[(size_t)r * N + c] = make_double2(i128_to_double(ar) * sc, i128_to_double(ai) * sc);
    }
}

// Grid of the element-wise kernels over an M x N matrix: x covers the columns in 256-thread blocks,
// y strides over the rows, about eight blocks per SM in all.
dim3 grid2d(int M, int N)
{
    const int gx = std::max(1, (N + 255) / 256);
    const int gy = std::max(1, std::min(M, std::max(1, 152 * 8 / gx)));
    return dim3(gx, gy);
}

int round_up(int x, int m)
{
    return ((x + m - 1) / m) * m;
}

}  // namespace

// ---------------------------------------------------------------------------- host side

// Work slots of one product shape: FP16X3 = one slot of the three split pairs per K range (the
// K range split so that tiles x slots fills the GPU); slices = the pairs (t, u) with t + u <= 8,
// grouped by t + u into slots whose exact-sum bound sum 2 m_t m_u K_range stays below 2^24
// (m_0 = 64, m_t = 32) and that hold at most five pairs.
void ZPlan::build(int mode_, int M_, int N_, int K_, int nsm)
{
    mode = mode_;
    M = M_;
    N = N_;
    K = K_;
    Mpad = round_up(std::max(M, 1), ZT);
    Npad = round_up(std::max(N, 1), ZT);
    nkc = round_up(std::max(K, 1), 16) / 16;
    ntiles = (Mpad / ZT) * (Npad / ZT);
    ns = mode == MODE_FP16X3 ? 2 : OZ_SLICES;
    std::vector<int2> pr;
    std::vector<int> sl, we;  // slot: p0, p1, kc0, kc1
    auto add_slot = [&](int p0, int p1, int kc0, int kc1, int w) {
        sl.insert(sl.end(), {p0, p1, kc0, kc1});
        we.push_back(w);
    };
    if (mode == MODE_FP16X3) {
        pr = {make_int2(0, 0), make_int2(0, 1), make_int2(1, 0)};
        int ks = std::max(1, std::min(std::max(1, nkc / 4), (nsm + ntiles - 1) / ntiles));
        const int per = (nkc + ks - 1) / ks;
        ks = (nkc + per - 1) / per;
        for (int s = 0; s < ks; ++s)
            add_slot(0, 3, s * per, std::min(nkc, (s + 1) * per), -28);
    } else {
        const int ks = (nkc + 127) / 128;  // K range <= 2048: the pair (0, 0) alone stays exact
        const int per = (nkc + ks - 1) / ks;
        const double limit = 16777216.0;
        for (int s = 0; s < ks; ++s) {
            const int kc0 = s * per, kc1 = std::min(nkc, (s + 1) * per);
            const double krange = 16.0 * (kc1 - kc0);
            for (int d = 0; d < ns; ++d) {
                int p0 = static_cast<int>(pr.size());
                double bound = 0.0;
                for (int t = 0; t <= d; ++t) {
                    const int u = d - t;
                    const double b = 2.0 * (t == 0 ? 64 : 32) * (u == 0 ? 64 : 32) * krange;
                    const int cnt = static_cast<int>(pr.size()) - p0;
                    if (cnt > 0 && (bound + b >= limit || cnt == 5)) {
                        add_slot(p0, static_cast<int>(pr.size()), kc0, kc1, -6 * (d + 2));
                        p0 = static_cast<int>(pr.size());
                        bound = 0.0;
                    }
                    pr.push_back(make_int2(t, u));
                    bound += b;
                }
                add_slot(p0, static_cast<int>(pr.size()), kc0, kc1, -6 * (d + 2));
            }
        }
    }
    nslots = static_cast<int>(we.size());
    npairs = static_cast<int>(pr.size());
    host_pairs = pr;
    host_slots = sl;
    host_wexp = we;
}

size_t ZPlan::table_bytes() const
{
    return host_pairs.size() * sizeof(int2) + host_slots.size() * sizeof(int) + host_wexp.size() * sizeof(int);
}

size_t ZPlan::planes_bytes(bool a_operand) const
{
    const int npl = 2;  // Re, Im per slice for both operands
    return (size_t)nkc * ns * npl * (a_operand ? Mpad : Npad) * 16 * sizeof(uint16_t);
}

size_t ZPlan::T_bytes() const
{
    return (size_t)nslots * Mpad * Npad * sizeof(float2);
}

// Copy the slot tables into `tab` (device, table_bytes() long) on stream s.
cudaError_t ZPlan::upload(void *tab, cudaStream_t s)
{
    uint8_t *p = static_cast<uint8_t *>(tab);
    d_pairs = reinterpret_cast<int2 *>(p);
    d_slots = reinterpret_cast<int *>(p + host_pairs.size() * sizeof(int2));
    d_wexp = d_slots + host_slots.size();
    cudaError_t e = cudaMemcpyAsync(d_pairs, host_pairs.data(), host_pairs.size() * sizeof(int2),
                                    cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_slots, host_slots.data(), host_slots.size() * sizeof(int), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_wexp, host_wexp.data(), host_wexp.size() * sizeof(int), cudaMemcpyHostToDevice, s);
    return e;
}

cudaError_t launch_zmaxabs(const double2 *M, int rows, int cols, long ld, unsigned long long *w, cudaStream_t s)
{
    zmaxabs_kernel<<<grid2d(rows, cols), 256, 0, s>>>(M, rows, cols, ld, w);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_zslice(const ZPlan &p, bool a_operand, const double2 *Mx, long ld, const unsigned long long *maxw,
                          uint16_t *planes, cudaStream_t s)
{
    const int rows = a_operand ? p.M : p.N, Rpad = a_operand ? p.Mpad : p.Npad;
    zslice_kernel<<<dim3(p.nkc, Rpad / ZT), 512, 0, s>>>(Mx, ld, rows, p.K, a_operand ? 0 : 1, Rpad, p.mode, p.ns, 2,
                                                         maxw, planes);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_zgemm16(const ZPlan &p, const uint16_t *Ap, const uint16_t *Bp, float2 *T, uint32_t *err,
                           uint64_t wait_ns, cudaStream_t s)
{
    auto kernel = p.mode == MODE_FP16X3 ? zgemm16_kernel<true> : zgemm16_kernel<false>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ZSMEM);
    if (e != cudaSuccess)
        return e;
    kernel<<<dim3(p.ntiles, p.nslots), ZTHREADS, ZSMEM, s>>>(Ap, 2 * p.ns, p.Mpad, Bp, 2 * p.ns, p.Npad, p.d_pairs,
                                                             reinterpret_cast<const ZSlot *>(p.d_slots), p.Npad / ZT, T,
                                                             err, wait_ns);
    count_launches(1);
    return cudaGetLastError();
}

// out = A B from the slot tiles of plan p.
cudaError_t launch_zcombine(const ZPlan &p, const float2 *T, const unsigned long long *wA,
                            const unsigned long long *wB, double2 *out, cudaStream_t s)
{
    const dim3 grid(grid2d(p.M, p.N));
    if (p.mode == MODE_FP16X3) {
        zcombine16_kernel<<<grid, 256, 0, s>>>(T, p.nslots, p.Mpad, p.Npad, wA, wB, p.M, p.N, out);
    } else {
        if (p.nslots > 256)
            return cudaErrorInvalidValue;
        zcombine_int_kernel<<<grid, 256, 0, s>>>(T, p.nslots, p.d_wexp, p.Mpad, p.Npad, wA, wB, p.M, p.N, out);
    }
    count_launches(1);
    return cudaGetLastError();
}

namespace {
// Carves a workspace into 256-byte aligned pieces; with base == nullptr it only counts.
struct Carver {
    uint8_t *base;
    size_t used = 0;
    explicit Carver(void *b) : base(static_cast<uint8_t *>(b)) {}
    void *take(size_t bytes)
    {
        void *r = base ? base + used : nullptr;
        used += (bytes + 255) / 256 * 256;
        return r;
    }
};

struct GemmWork {
    uint16_t *Ap, *Bp;
    float2 *T;
    unsigned long long *words;
    void *tab;
};

GemmWork carve_gemm(const ZPlan &p, Carver &c)
{
    GemmWork g;
    g.Ap = static_cast<uint16_t *>(c.take(p.planes_bytes(true)));
    g.Bp = static_cast<uint16_t *>(c.take(p.planes_bytes(false)));
    g.T = static_cast<float2 *>(c.take(p.T_bytes()));
    g.words = static_cast<unsigned long long *>(c.take(64 * 8));
    g.tab = c.take(p.table_bytes());
    return g;
}
}  // namespace

// C = A B for M x K and K x N complex128 matrices (row-major, device), by the sliced tensor-core
// product of plan p (mode FP16X3 or integer slices); the workspace holds both operands' planes,
// the slot tiles T, the scalar words and the tables (zgemm_work_bytes).
size_t zgemm_work_bytes(const ZPlan &p)
{
    Carver c(nullptr);
    carve_gemm(p, c);
    return c.used;
}

cudaError_t zgemm_enqueue(ZPlan &p, const double2 *A, long lda, const double2 *B, long ldb, double2 *C, void *work,
                          uint32_t *err, uint64_t wait_ns, cudaStream_t s)
{
    Carver c(work);
    const GemmWork g = carve_gemm(p, c);
    uint16_t *Ap = g.Ap, *Bp = g.Bp;
    float2 *T = g.T;
    unsigned long long *words = g.words;
    cudaError_t e = p.upload(g.tab, s);
    if (e != cudaSuccess)
        return e;
    if ((e = cudaMemsetAsync(words, 0, 64 * 8, s)) != cudaSuccess)
        return e;
    // words[0], [1]: max of A and B
    if ((e = launch_zmaxabs(A, p.M, p.K, lda, &words[0], s)) != cudaSuccess)
        return e;
    if ((e = launch_zmaxabs(B, p.K, p.N, ldb, &words[1], s)) != cudaSuccess)
        return e;
    if ((e = launch_zslice(p, true, A, lda, &words[0], Ap, s)) != cudaSuccess)
        return e;
    if ((e = launch_zslice(p, false, B, ldb, &words[1], Bp, s)) != cudaSuccess)
        return e;
    if ((e = launch_zgemm16(p, Ap, Bp, T, err, wait_ns, s)) != cudaSuccess)
        return e;
    return launch_zcombine(p, T, &words[0], &words[1], C, s);
}

}  // namespace gw
