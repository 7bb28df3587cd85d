// Persistent Hermitian rank-k update of one or many systems (Eq. Pstatic; the outer product of
// Sec. 4.1) on the 16-bit tensor cores.  One CTA per SM walks a static list of (job, row block,
// column block) tiles (CTA b takes tiles b, b + grid, b + 2 grid, ...; the host orders them by
// decreasing work so the static schedule balances).
//
// A job is a system in one of two forms.
//  * Pair form (nvc = 0): P = -sum_k f_k(r) conj(f_k(r')) over all k = nv nc pair densities.  The
//    arithmetic per tile is that of herk16_kernel -- the FP16 / BF16 hi/lo split, W-chunk TMEM windows
//    promoted to FP32 registers, the registers added up every L windows -- bit for bit.
//  * Separable form (nvc > 0): with 2 / (E_c - E_v) = sum_t u_t(v) z_t(c) (sep_factors.h) the sum over
//    pairs splits, at every (r, r'), into products of two short sums,
//        P(r, r') = -sum_t V_t(r, r') C_t(r, r'),
//        C_t = sum_c z_t(c) psi_c(r) conj(psi_c(r')),   V_t = sum_v u_t(v) conj(psi_v(r)) psi_v(r'),
//    so the tensor cores contract T (nc + nv) states instead of nv nc pairs: 352 chunks of 16 against
//    960 at 24^3 (T = 11), 871 against 4000 at 36^3 with 64 / 1000 states.  Per term the C windows are
//    promoted into registers as above, then each V window is multiplied into them element by element
//    in FP32 and the products are added into the tile's sums.  The registers hold C_t (128 of the 168
//    a thread can have), so the sums over t live in global memory: 128 KB per CTA, written and read by
//    their own threads only (20 MB for the GPU, resident in L2), added with fire-and-forget vector
//    reductions so no thread waits for a load.
//
// Measured on one GB300 (update alone, FP16X3, W = 3): 24^3, 32 x 480 states: 24.2 -> 9.3 ms (0.95 of
// the sustained FP16 rate would be 6.9 ms for the issued MMAs); 36^3, 64 x 1000, BF16X3, W = 16: 0.97 ->
// 0.20 s.
//
// Bound: the tensor pipe and the shared memory that feeds it, as herk16_kernel (32 KB staged and 84 KB
// read per chunk).  Control: mbarrier phases and the two TMEM window buffers carry across tiles, so the
// producer streams the next tile's operands while the current tile is being written.
//
// Truncation.  tcgen05 adds into TMEM with truncation, so a window comes out smaller, and the product of two
// windowed sums loses twice.  How much depends on the states: elements of P whose terms have one sign
// lose most.  Measured loss, in 1e-7, for windows of n chunks together (C and V), FP16X3:
//                                n = 2          4         17 or 18     40 to 55
//   diagonal                 2.4 ..  4.8    3.8 .. 8.4    16 .. 40    49 .. 110
//   next to it               2.3 ..  5.4    3.7 .. 8.9    16 .. 22    48 ..  50
//   far from it              2.3 ..  3.2    3.7 .. 5.3     7 .. 16     7 ..  50
// (Haar-random states, band-structured ones, plane waves of equal size and states without a sign change,
// 12^3 to 20^3, up to 1600 unoccupied states); BF16X3 loses less.  The separable form adds a share of this
// back (loss_gain), at the low end of what was measured, so that no element is overcorrected by more
// than the pair form leaves it short.  Relative error of P against FP64 then, separable / pair form at the
// same W, in 1e-7: Haar, 14^3, 32 x 480: 1.5 / 2.8 (W = 1), 1.8 / 6.0 (3), 4.9 / 31 (16), 7 / 130 (64);
// band-structured, 14^3, 48 x 700: 1.4 / 2.4, 2.2 / 5.2, 7.4 / 28, 14 / 120; plane waves, 16^3, 19 x 600:
// 2.2 / 2.5, 4.7 / 4.7, 11 / 21, 24 / 89; BF16X3 the same three: 19 / 34, 11 / 25, 12 / 23 (W = 1), 21 / 49, 14 / 40,
// 15 / 30 (16).  Windows of 2 W chunks would take 8.5 ms instead of 9.3 at 24^3, but on the plane waves
// leave 6.8 where the pair form at W = 3 leaves 4.7.
//
// The occupied planes are FP16 in either precision (they are 1/16 of the work), so with BF16 operands
// only C_t carries the 8 + 8-bit split: both at 8 + 8 bits measured 5.7e-6 on the off-diagonal elements
// of P against 4.5e-6 in the pair form; now 4.1e-6.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "gw_internal.cuh"
#include "ptx.cuh"

namespace gw {

namespace {

constexpr int TM = 128, TN = 128;
constexpr uint32_t PL = TM * HERK16_KC * 2;  // 4 KB: one plane of one 128-row block
constexpr uint32_t NPL = HERK16_NPL;
// stage as in herk16_kernel: the A block's planes Im hi, Re hi, Im lo, Re lo (one bulk copy), then
// the B block's in the same order, i.e. regions [Im | Re] of the
// hi part and of the lo part, so one N = 256 MMA from A = Im fills the Re and Im columns of a window
constexpr uint32_t B_OFF = 4 * PL;
constexpr uint32_t CHUNK_BYTES = 8 * PL;  // 32 KB
// Chunks per pipeline stage, CPS (a stage holds chunks of one window only; six chunks are in flight):
// fewer barrier round trips and commits than one by one.  Two, or three where W is a multiple of three, so
// that the stages are full.  Measured, one / two / three chunks a stage, FP16X3: W = 3, 16^3 with 16 x 200
// states 0.497 / 0.506 / 0.485 ms, 24^3 9.40 / 9.39 / 9.25, 32^3 with 48 x 800 85.0 / 86.2 / 83.8; W = 4,
// 24^3 8.99 / 9.05 / 9.43; W = 16, 36^3, BF16X3, 204 / 200 / 202.
constexpr int RING_CHUNKS = 6;
constexpr uint32_t PIPE_BYTES = RING_CHUNKS * CHUNK_BYTES;  // 192 KB
constexpr int MAX_STAGES = 3;
constexpr uint32_t LBO = 128, SBO = 256;
constexpr int NPROMO_WARPS = 8;
constexpr int PRODUCER_WARP = 8, MMA_WARP = 9;
constexpr int NTHREADS = 320;
constexpr uint64_t DRAIN_NS = 2000000000ull;
// each promotion warp turns 32 rows x 16 columns of the result at a time, so that the rows of P are
// written in 128-byte runs (a row pitch of 17 values: conflict-free both ways)
constexpr int OUT_COLS = 16, OUT_PITCH = 17;
constexpr uint32_t BAR_BYTES = 256;
constexpr size_t SMEM = PIPE_BYTES + BAR_BYTES + NPROMO_WARPS * 32 * OUT_PITCH * sizeof(float2);
static_assert(SMEM <= 227 * 1024, "shared memory of one CTA");
constexpr int SUM_F4 = 32;  // float4 values per promotion thread: 64 complex sums
static_assert(HERK16P_SUMS == (size_t)SUM_F4 * NPROMO_WARPS * 32 * sizeof(float4), "sums per CTA");

// A thread's own running sums in global memory: a plain store starts them, reductions add, and the
// load at the tile's end bypasses L1, which may hold the previous tile's values.
__device__ __forceinline__ void sums_add(float4 *p, float4 v, bool first)
{
    if (first)
        asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z),
                     "f"(v.w)
                     : "memory");
    else
        asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y),
                     "f"(v.z), "f"(v.w)
                     : "memory");
}

__device__ __forceinline__ float4 sums_load(const float4 *p)
{
    float4 v;
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

// Position in the ring of stages: stage and phase parity of a stage counter.
template <int STAGES>
struct Ring {
    int s = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next()
    {
        if (++s == STAGES) {
            s = 0;
            ph ^= 1u;
        }
    }
};

// Windows of a job: each term has nwc windows of wc chunks over its ncc unoccupied (or pair) chunks, the
// last one shorter, then nwv windows of wv chunks over its nvc occupied ones; both at most W.
struct Windows {
    int wc, nwc, nwv, wv;
    __device__ __forceinline__ Windows(const HerkJob &j, int W)
    {
        wc = W;
        nwc = (j.ncc + wc - 1) / wc;
        nwv = (j.nvc + W - 1) / W;
        wv = nwv > 0 ? (j.nvc + nwv - 1) / nwv : 0;
    }
};

// Mean chunks per window of a sum over n chunks taken in windows of w (the last one shorter).
__device__ __forceinline__ float mean_window(int n, int w)
{
    if (n <= 0)
        return 0.f;
    const int full = n / w, rest = n - full * w;
    return (float)(full * w * w + rest * rest) / (float)n;
}

// The scales of the operands, 2^ec and 2^ev, come out of P = -sum_t V_t C_t 2^(-2 ec - 2 ev).  V is
// brought down to the size of its terms, so that the products with C stay in range, and the rest is
// applied to the sums in two factors, each a normal FP32 value.
constexpr int V_SHIFT = -28;

__device__ __forceinline__ void unscale(int ec, int ev, float &a, float &b)
{
    const int e = max(-252, min(252, -2 * ec - 2 * ev - V_SHIFT)), h = e / 2;
    a = ldexpf(1.0f, h);
    b = ldexpf(1.0f, e - h);
}

// Share of an element of P to add to it for what truncation took from a product of two sums over windows of n
// chunks together (header comment); the diagonal loses most and has its own.  It is added, not multiplied
// on: 1 + share has steps of 1.2e-7.
template <bool BF16>
__device__ __forceinline__ float loss_gain(float n, bool diagonal)
{
    if (BF16)
        return diagonal ? 1.5e-7f + 0.5e-7f * n : 1.2e-7f + 0.45e-7f * n;
    return diagonal ? 1.0e-7f + 1.5e-7f * n : 2.6e-7f + 0.3e-7f * n;
}

template <bool BF16, int CPS>
__global__ void __launch_bounds__(NTHREADS, 1)
    herk16p_kernel(const HerkJob *__restrict__ jobs, const int4 *__restrict__ tiles, int n_tiles, uint32_t *err,
                   uint64_t wait_ns, int W, int L, float4 *__restrict__ sums)
{
    constexpr int STAGES = RING_CHUNKS / CPS;
    static_assert(STAGES <= MAX_STAGES, "barriers");
    constexpr uint32_t STAGE_BYTES = CPS * CHUNK_BYTES;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + PIPE_BYTES);
    uint64_t *empty = full + STAGES;
    uint64_t *accf = empty + STAGES;
    uint64_t *acce = accf + 2;
    uint64_t *done = acce + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile long long *n_issued = reinterpret_cast<volatile long long *>(smem + PIPE_BYTES + 192);
    volatile long long *n_consumed = n_issued + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], NPROMO_WARPS);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        *n_issued = 0;
        *n_consumed = 0;
        fence_barrier_init();
    }
    if (warp == MMA_WARP)
        tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == PRODUCER_WARP) {
        if (lane == 0) {
            long long g = 0;  // stages issued by this CTA over all its tiles
            Ring<STAGES> ring;
            bool ok = true;
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
                const int4 tl = tiles[t];
                const HerkJob jb = jobs[tl.x];
                const Windows w(jb, W);
                const int nblk = jb.nr_pad / TM;  // block layout: one 16 KB copy per operand block
                const size_t step = plane16_block(1, 0, nblk, NPL, 0);
                const uint16_t *a = jb.A + plane16_block(0, tl.y, nblk, NPL, 0), *b = nullptr;
                auto window = [&](int n) {
                    for (int c = 0; c < n; c += CPS, ++g, ring.next()) {
                        if (g >= STAGES && !mbar_wait(&empty[ring.s], ring.ph ^ 1u, wait_ns)) {
                            record_error(err, GW_E_TIMEOUT, SITE_HERK_PRODUCER, blockIdx.x);
                            *abort_flag = 1;
                            return false;
                        }
                        if (*abort_flag)
                            return false;
                        uint8_t *st = smem + ring.s * STAGE_BYTES;
                        const int m = min(CPS, n - c);
                        mbar_arrive_expect_tx(&full[ring.s], m * CHUNK_BYTES);
                        for (int j = 0; j < m; ++j, a += step, b += step, st += CHUNK_BYTES) {
                            bulk_g2s(st, a, 4 * PL, &full[ring.s]);
                            bulk_g2s(st + B_OFF, b, 4 * PL, &full[ring.s]);
                        }
                        *n_issued = g + 1;
                    }
                    return true;
                };
                for (int term = 0; term < jb.T && ok; ++term) {
                    b = jb.B + plane16_block(0, tl.z, nblk, NPL, 0);  // the same for every term
                    for (int i = 0; i < w.nwc && ok; ++i)
                        ok = window(min(w.wc, jb.ncc - i * w.wc));
                    for (int i = 0; i < w.nwv && ok; ++i)
                        ok = window(min(w.wv, jb.nvc - i * w.wv));
                }
            }
        }
        __syncwarp();
    } else if (warp == MMA_WARP) {
        if (lane == 0) {
            constexpr uint32_t FMT = BF16 ? mma_idesc(1u, 0, 0, false) ^ mma_idesc(0u, 0, 0, false) : 0u;
            const uint32_t sbase = smem_u32(smem);
            long long g = 0;
            uint32_t gw = 0;  // windows issued by this CTA
            Ring<STAGES> ring;
            bool ok = true;
            // one window of n chunks into TMEM buffer gw & 1; the formats' bits of the descriptors: fmt
            auto window = [&](int n, uint32_t fmt) {
                const int b = (int)(gw & 1u);
                if (gw >= 2 && !mbar_wait(&acce[b], ((gw >> 1) - 1u) & 1u, wait_ns)) {
                    record_error(err, GW_E_TIMEOUT, SITE_HERK_MMA, blockIdx.x);
                    *abort_flag = 1;
                    return false;
                }
                tc_fence_after();
                const uint32_t d = tmem + b * 256;
                const uint32_t ID = mma_idesc(0u, TM, 2 * TN, false) | fmt;
                const uint32_t ID1 = mma_idesc(0u, TM, TN, false) | fmt, ID1N = mma_idesc(0u, TM, TN, true) | fmt;
                for (int c = 0; c < n; ++c) {
                    const int s = ring.s;
                    if (c % CPS == 0) {
                        if (!mbar_wait(&full[s], ring.ph, wait_ns)) {
                            record_error(err, GW_E_TIMEOUT, SITE_HERK_MMA, blockIdx.x);
                            *abort_flag = 1;
                            return false;
                        }
                        tc_fence_after();
                    }
                    const uint32_t st = sbase + s * STAGE_BYTES + (c % CPS) * CHUNK_BYTES;
                    const uint64_t a_ih = smem_desc(st, LBO, SBO), a_rh = smem_desc(st + PL, LBO, SBO);
                    const uint64_t a_il = smem_desc(st + 2 * PL, LBO, SBO);
                    const uint64_t a_rl = smem_desc(st + 3 * PL, LBO, SBO);
                    const uint64_t b_ih = smem_desc(st + B_OFF, LBO, SBO);
                    const uint64_t b_rh = smem_desc(st + B_OFF + PL, LBO, SBO);
                    const uint64_t b_il = smem_desc(st + B_OFF + 2 * PL, LBO, SBO);
                    const uint64_t b_rl = smem_desc(st + B_OFF + 3 * PL, LBO, SBO);
                    const uint32_t acc = c > 0 ? 1u : 0u;
                    mma_f16(d, a_ih, b_ih, ID, acc);       // Re += Ai Bi, Im += Ai Br
                    mma_f16(d, a_ih, b_il, ID, 1);
                    mma_f16(d, a_il, b_ih, ID, 1);
                    mma_f16(d, a_rh, b_rh, ID1, 1);        // Re += Ar Br
                    mma_f16(d, a_rh, b_rl, ID1, 1);
                    mma_f16(d, a_rl, b_rh, ID1, 1);
                    mma_f16(d + 128, a_rh, b_ih, ID1N, 1);  // Im -= Ar Bi
                    mma_f16(d + 128, a_rh, b_il, ID1N, 1);
                    mma_f16(d + 128, a_rl, b_ih, ID1N, 1);
                    if (c % CPS == CPS - 1 || c == n - 1) {
                        mma_commit(&empty[s]);
                        *n_consumed = ++g;
                        ring.next();
                    }
                }
                mma_commit(&accf[b]);
                ++gw;
                return true;
            };
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
                const HerkJob jb = jobs[tiles[t].x];
                const Windows w(jb, W);
                for (int term = 0; term < jb.T && ok; ++term) {
                    for (int i = 0; i < w.nwc && ok; ++i)
                        ok = window(min(w.wc, jb.ncc - i * w.wc), FMT);
                    for (int i = 0; i < w.nwv && ok; ++i)
                        ok = window(min(w.wv, jb.nvc - i * w.wv), 0u);
                }
            }
            mma_commit(done);  // arrives once every MMA issued above has completed
        }
        __syncwarp();
    } else {
        // ---------------- promotion warps 0..7
        const int q = warp & 3, h = warp >> 2;
        const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
        float4 *my = sums + (size_t)blockIdx.x * (SUM_F4 * NPROMO_WARPS * 32) + threadIdx.x;  // stride 256
        float2 *stage = reinterpret_cast<float2 *>(smem + PIPE_BYTES + BAR_BYTES) + warp * 32 * OUT_PITCH;
        uint32_t gw = 0;
        bool stop = false;
        float are[64], aim[64];
        // Wait for the next window; the outcome is the same in every lane, as the TMEM loads need.
        auto ready = [&]() {
            if (!__all_sync(0xffffffffu, mbar_wait(&accf[gw & 1u], (gw >> 1) & 1u, wait_ns))) {
                if (lane == 0)
                    record_error(err, GW_E_TIMEOUT, SITE_HERK_EPILOGUE, blockIdx.x);
                *abort_flag = 1;
                stop = true;
                return false;
            }
            tc_fence_after();
            return true;
        };
        auto release = [&]() {  // the window's TMEM buffer is free again
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&acce[gw & 1u]);
            ++gw;
        };
        for (int t = blockIdx.x; t < n_tiles && !stop; t += gridDim.x) {
            const int4 tl = tiles[t];
            const HerkJob &jb = jobs[tl.x];  // fields are read as needed: the registers hold the sums
            const bool sep = jb.nvc > 0;
            const Windows w(jb, W);
            // segments: the registers restart from zero in each (a fresh start rather than a conditional
            // reset keeps all 128 sums in registers)
            const int nseg = sep ? jb.T : (w.nwc + L - 1) / L;
            for (int seg = 0; seg < nseg && !stop; ++seg) {
#pragma unroll
                for (int i = 0; i < 64; ++i) {
                    are[i] = 0.f;
                    aim[i] = 0.f;
                }
                const int w0 = sep ? 0 : seg * L, w1 = sep ? w.nwc : min(w.nwc, w0 + L);
                for (int win = w0; win < w1; ++win) {
                    if (!ready())
                        break;
                    const uint32_t base = tmem + lane_addr + (gw & 1u) * 256 + h * 64;
#pragma unroll
                    for (int c0 = 0; c0 < 64; c0 += 16) {
                        float v[16];
                        tmem_ld16(base + c0, v);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            are[c0 + i] += v[i];
                        tmem_ld16(base + 128 + c0, v);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            aim[c0 + i] += v[i];
                    }
                    release();
                }
                if (stop)
                    break;
                if (!sep) {
#pragma unroll
                    for (int i = 0; i < SUM_F4; ++i)
                        sums_add(my + i * 256, make_float4(are[2 * i], aim[2 * i], are[2 * i + 1], aim[2 * i + 1]),
                                 seg == 0);
                    continue;
                }
                const float vs = jb.term_scale[seg] * ldexpf(1.0f, V_SHIFT);
                for (int win = 0; win < w.nwv; ++win) {
                    if (!ready())
                        break;
                    const uint32_t base = tmem + lane_addr + (gw & 1u) * 256 + h * 64;
                    const bool first = seg == 0 && win == 0;
#pragma unroll
                    for (int c0 = 0; c0 < 64; c0 += 8) {
                        float vr[8], vi[8];
                        tmem_ld8x2(base + c0, base + 128 + c0, vr, vi);
                        float4 o[4];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float x = vr[i] * vs, y = vi[i] * vs;
                            const float pr = fmaf(x, are[c0 + i], -(y * aim[c0 + i]));
                            const float pi = fmaf(x, aim[c0 + i], y * are[c0 + i]);
                            (i & 1 ? o[i / 2].z : o[i / 2].x) = pr;
                            (i & 1 ? o[i / 2].w : o[i / 2].y) = pi;
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            sums_add(my + (c0 / 2 + i) * 256, o[i], first);
                    }
                    release();
                }
            }
            if (stop)
                break;
            // the tile's sums -> P: entries c >= r (real diagonal) in 128-byte row runs through the
            // warp's stage, their mirror P[c][r] = conj(P[r][c]) straight from the lanes, which hold
            // consecutive r
            const int nr = jb.nr, r0 = tl.y * TM + q * 32, r = r0 + lane, cbase = tl.z * TN + h * 64;
            const float nw = mean_window(jb.ncc, w.wc) + mean_window(jb.nvc, w.wv);
            float s0 = 1.f, s1 = -ldexpf(1.0f, -2 * jb.scale_exp[0]);
            if (sep) {
                unscale(jb.scale_exp[0], jb.scale_exp[1], s0, s1);
                s1 = -s1;
            }
            const float gain = loss_gain<BF16>(nw, false), gain_d = loss_gain<BF16>(nw, true);
            auto out = [&](float v, bool diagonal) {
                const float x = v * s1 * s0;
                return sep ? fmaf(x, diagonal ? gain_d : gain, x) : x;
            };
            float2 *P = jb.P;
            for (int g0 = 0; g0 < 64; g0 += OUT_COLS) {
                float2 x[OUT_COLS];
#pragma unroll
                for (int i = 0; i < OUT_COLS / 2; ++i) {
                    const float4 v = sums_load(my + (g0 / 2 + i) * 256);
                    const int col = cbase + g0 + 2 * i;
                    x[2 * i] = make_float2(out(v.x, col == r), out(v.y, false));
                    x[2 * i + 1] = make_float2(out(v.z, col + 1 == r), out(v.w, false));
                }
#pragma unroll
                for (int i = 0; i < OUT_COLS; ++i) {
                    const int col = cbase + g0 + i;
                    if (r < nr && col < nr && col > r)
                        P[(size_t)col * nr + r] = make_float2(x[i].x, -x[i].y);
                    stage[lane * OUT_PITCH + i] = x[i];
                }
                __syncwarp();
#pragma unroll 4
                for (int p = 0; p < 16; ++p) {
                    const int row = 2 * p + (lane >> 4), i = lane & 15;
                    const int rr = r0 + row, col = cbase + g0 + i;
                    if (rr < nr && col < nr && col >= rr) {
                        const float2 v = stage[row * OUT_PITCH + i];
                        P[(size_t)rr * nr + col] = make_float2(v.x, col == rr ? 0.f : v.y);
                    }
                }
                __syncwarp();
            }
        }
    }

    __syncthreads();
    if (threadIdx.x == 0) {
        if (!mbar_wait(done, 0, DRAIN_NS))
            record_error(err, GW_E_TIMEOUT, SITE_HERK_DRAIN, blockIdx.x);
        const long long issued = *n_issued, consumed = *n_consumed;
        for (long long g = consumed; g < issued; ++g)
            if (!mbar_wait(&full[g % STAGES], (uint32_t)((g / STAGES) & 1), DRAIN_NS)) {
                record_error(err, GW_E_TIMEOUT, SITE_HERK_DRAIN, blockIdx.x);
                break;
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace

cudaError_t launch_herk16p(const HerkJob *jobs, const int4 *tiles, int n_tiles, int grid, bool bf16, uint32_t *err,
                           uint64_t wait_ns, int W, int L, float4 *sums, cudaStream_t s)
{
    if (n_tiles <= 0)
        return cudaSuccess;
    auto kernel = W % 3 == 0 ? (bf16 ? herk16p_kernel<true, 3> : herk16p_kernel<false, 3>)
                             : (bf16 ? herk16p_kernel<true, 2> : herk16p_kernel<false, 2>);
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
    if (e != cudaSuccess)
        return e;
    kernel<<<grid, NTHREADS, SMEM, s>>>(jobs, tiles, n_tiles, err, wait_ns, W, L, sums);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace gw
